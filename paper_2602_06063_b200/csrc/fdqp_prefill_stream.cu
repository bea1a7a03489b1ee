// Prefill-sized projection (M >= 9 token rows), the form every call takes unless a launch parameter asks for the tile kernels
// of fdqp_prefill.cu: pairs of SMs that stay for the whole call and share its work to the block.
//
//   D[n][tok] = sum_k w16[k][n] * x[tok][k],   w16 = RNE_bf16( d * q + m ), one rounding      (Eq. 3, then Eq. 14)
//
// Units of work are (tile of 256 output features x up to 256 tokens, block of 256 k); they lie tile by tile along one line that
// is cut into one range per pair, at tile boundaries where that costs less than an exchange of partial sums.  Inside a CTA
// (128 of the tile's rows) every part has its own warps and its own ring, so that nothing waits at a tile's end:
//   warp 0   x boxes (TMA, 64 k x half of the tile's tokens; where the whole K of one token tile fits, loaded once and kept)
//   warp 1   (CTA 0 of the pair) issues tcgen05.mma.cta_group::2, 256 rows x N tokens x 16 k
//   warps 2, 3   weights: whole packed blocks, cp.async.bulk into a ring, two strips each
//   warps 4..7   read finished accumulators and store y where there are two sets of them (up to 128 tokens); the last ones of a
//                range, and all where there is one set, are read by the four conversion warps of a strip
//   warps 8..23  convert: packed block -> bf16 pairs in registers -> tensor memory, where the MMA takes its A operand from;
//                the four of a strip take its half blocks (128 k) in turn
// A tile cut between pairs is finished by the last of them to arrive at its strip's counter: partial sums through global
// memory, added in K order whoever is last, so results do not depend on timing, and no CTA waits for another one's work.  Where
// there are so few tiles that every pair works on one tile only, the pairs of a tile can be one cluster instead (CLUSTER): they
// are resident together, write their sums into one another's shared memory and wait for them.
//
// What bounds it, and what that decided (B200, graph replays; the tile kernels this replaced in brackets):
//   - The tile kernels took 0.6 us per 64 k and CTA whatever the SM ran beside it: one thread waited, issued and committed for
//     every k-step, and every warp converted for every k-step.  Here a wait and a commit serve a block (256 k), issued by a warp
//     on uniform values with the next block's barriers tested ahead, and a conversion warp has every fourth half block.
//   - K = 2560, N = 262144: 88 us at 16 tokens, 99 at 48 (153), 112 at 64 (154), 150 at 128 (190), 541 at 512 with fp32 stores
//     (520-576 by the power cap).  Without conversion and tensor-memory stores the 48-token call takes 70, the HBM rate; the
//     stores (64 bytes a clock and SM) and the conversion's instructions do not overlap completely.
//   - One layer's calls at 37 tokens: 2560 x 4096 6.7 (10.2; 7.6 without clusters), 2048 x 2560 6.0 (8.7; 6.8), 2560 x 20480 13.3
//     (24.2), 10240 x 2560 10.9 (16.7); 200 tokens, 3840 x 30720, gated: 43 (47), 2560 x 4096 12.5 (14.2 without clusters).  The small ones are start-up (2.4 thousand cycles to the cluster's
//     barrier, a thousand more to the first weights) and, at the end, partial sums (counter and reading back: 2 us).
//   - No register of the conversion loop may go to local memory: 30 spilled ones made it 2.5 times slower, since with this much
//     shared memory no first-level cache is left.
#include "fdqp_tcgen05.cuh"

namespace fdqp {

constexpr int kStThreads = 24 * 32;

// ---- more tcgen05 wrappers ----------------------------------------------------------------------------------------

__device__ __forceinline__ void umma2_bf16_ta(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// The same for two k-steps at once: a map of [k / 64][token][64 k].
__device__ __forceinline__ void tma2_load_3d(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, uint32_t bar_cta0) {
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(dst), "l"(map), "r"(bar_cta0), "r"(c0), "r"(c1), "r"(c2)
        : "memory");
}

// Has the phase of this parity completed?  (No wait.)
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
    uint32_t is;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(is) : "r"(bar), "r"(parity) : "memory");
    return is != 0;
}

// Arrive on the barrier at this offset in the CTAs of the mask once every MMA issued so far by this thread has completed.
__device__ __forceinline__ void umma2_commit(uint32_t bar, uint16_t mask) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar), "h"(mask) : "memory");
}
// Another CTA's shared memory: 16 bytes, and an arrival that releases this warp's.
__device__ __forceinline__ void st_cluster(uint32_t addr, float a, float b, float c, float d) {
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}
__device__ __forceinline__ void mbar_arrive_release_cluster(uint32_t cluster_addr) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}

__device__ __forceinline__ bool elect_one() {
    uint32_t is;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(is));
    return is != 0;
}

// 16 registers to 16 columns of this thread's lane of tensor memory; tmem_st_wait before they are signalled.
__device__ __forceinline__ void tmem_st_16cols_async(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
          "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld_16cols(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}

// A whole warp waits for the phase of this parity; what it returns is the same in every lane.
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, int* status) {
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, status));
}

// Finished values of row `lane` of a 32-row strip, tokens [c, c + 16) of the tile, whose first row of y is tok0.
__device__ __forceinline__ void store_chunk(const StreamParams& p, const float (&v)[16], int64_t strip, int lane, int tok0, int c, int toks) {
    const int left = toks - c;
    if (p.epi == kEpiGegluBf16) {
        // lanes 0..15 hold gate rows, lanes 16..31 the up rows of the same outputs: the low half finishes the even tokens, the
        // high half the odd ones -- one exchange per token pair, every lane busy
        const bool low = lane < 16;
        const int64_t ld = p.N / 2;
        uint16_t* out = p.y16 + (int64_t)(tok0 + c + (low ? 0 : 1)) * ld + strip * 16 + (lane & 15);
#pragma unroll
        for (int jj = 0; jj < 8; ++jj, out += 2 * ld) {
            const float a = v[2 * jj], b = v[2 * jj + 1];
            const float got = __shfl_xor_sync(0xffffffffu, low ? b : a, 16);
            const float gate = low ? a : got, up = low ? got : b;
            if (2 * jj + (low ? 0 : 1) < left) *out = f32_to_bf16_rne(gelu_tanh(gate) * up);
        }
        return;
    }
    const int64_t at = (int64_t)(tok0 + c) * p.N + strip * kStripRows + lane;
    if (p.epi == kEpiBf16) {
        uint16_t* out = p.y16 + at;
#pragma unroll
        for (int j = 0; j < 16; ++j, out += p.N)
            if (j < left) *out = f32_to_bf16_rne(v[j]);
    } else {
        float* out = p.y + at;
#pragma unroll
        for (int j = 0; j < 16; ++j, out += p.N)
            if (j < left) *out = v[j];
    }
}

// A tile that pairs p0 .. p1 share.  The partial sums of pair r lie in slot 2 r (its range begins in the tile) or 2 r + 1 (it
// begins in an earlier one): [slot][CTA][strip][token / 4][32 rows][4 tokens].
struct SharedTile {
    int p0, p1;
    float4* base;         // this strip's and lane's part of slot 0
    int64_t slot_quads;   // from one slot to the next
    int first;            // 1: p0's range begins in an earlier tile
    __device__ __forceinline__ float4* slot(int r) const { return base + (2 * r + (r == p0 ? first : 0)) * slot_quads; }
};

__device__ __forceinline__ SharedTile shared_tile(const StreamParams& p, int tile, int strip8, int lane) {
    SharedTile s;
    s.p0 = st_owner(p, tile * p.nb);
    s.p1 = st_owner(p, (tile + 1) * p.nb - 1);
    s.slot_quads = (int64_t)2 * p.n_inst * kStripRows;  // 8 strips, 4 tokens per float4
    s.base = reinterpret_cast<float4*>(p.ws) + (int64_t)strip8 * (p.n_inst / 4) * kStripRows + lane;
    s.first = st_range_begin(p, s.p0) < tile * p.nb ? 1 : 0;
    return s;
}
// A piece's sums of 16 tokens from c on (`own`: they are still in the accumulators at acc).
__device__ __forceinline__ void piece16(const SharedTile& s, int r, bool own, uint32_t acc, int c, int toks, float (&v)[16]) {
    if (own) {
        tmem_ld_16cols(acc + (uint32_t)c, v);
        return;
    }
    const float4* at = s.slot(r) + (c / 4) * 32;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float4 f = c + 4 * i < toks ? __ldcg(at + 32 * i) : make_float4(0.f, 0.f, 0.f, 0.f);
        v[4 * i] = f.x, v[4 * i + 1] = f.y, v[4 * i + 2] = f.z, v[4 * i + 3] = f.w;
    }
}

// Adds the pieces of a shared tile's strip in pair order and stores the sums: part h of kStParts, i.e. tokens 16 i .. 16 i + 15
// for i = h, h + kStParts, ...; two pieces' loads in flight.  own >= 0: that pair's piece is still in the accumulators at acc.
__device__ __forceinline__ void sum_shared(const StreamParams& p, const SharedTile& s, int own, uint32_t acc, int strip, int lane, int tok0,
                                           int toks, int h) {
#pragma unroll 1
    for (int c = 16 * h; c < toks; c += 16 * kStParts) {
        float sum[16], v[16];
        if (s.p0 == own) {  // (the other one's loads first)
            piece16(s, s.p0 + 1, false, acc, c, toks, v);
            piece16(s, s.p0, true, acc, c, toks, sum);
        } else {
            piece16(s, s.p0, false, acc, c, toks, sum);
            piece16(s, s.p0 + 1, s.p0 + 1 == own, acc, c, toks, v);
        }
#pragma unroll
        for (int i = 0; i < 16; ++i) sum[i] += v[i];
#pragma unroll 1
        for (int r = s.p0 + 2; r <= s.p1; ++r) {
            piece16(s, r, r == own, acc, c, toks, v);
#pragma unroll
            for (int i = 0; i < 16; ++i) sum[i] += v[i];
        }
        store_chunk(p, sum, strip, lane, tok0, c, toks);
    }
}

__device__ __forceinline__ uint32_t lds_u16(uint32_t addr) {
    uint16_t v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(addr));
    return v;
}

// One group-tile of a packed block in shared memory: this lane's row (jb: groups of the block; the variants hold whole blocks).
template <int FMT>
__device__ __forceinline__ GroupRegs group_from_smem(uint32_t blk, int t, int jb, int lane) {
    using F = FmtTraits<FMT>;
    GroupRegs r;
    r.valid = true;
    r.codes = lds128(blk + (uint32_t)(t * 512 + lane * 16));
    r.m_bits = 0;
    if (F::kMx) {
        asm volatile("ld.shared.u8 %0, [%1];" : "=r"(r.d_bits) : "r"(blk + (uint32_t)(kCodeBytes + t * 32 + lane)));
    } else {
        const uint32_t at = 2u * (uint32_t)((t >> F::kShift) * 32 + lane);
        const uint32_t d = FMT == kFmtQ4nx ? 512u * (uint32_t)jb : (uint32_t)kCodeBytes;
        const uint32_t m = FMT == kFmtQ4nx ? 576u * (uint32_t)jb : (uint32_t)F::kOffSect;
        r.d_bits = lds_u16(blk + d + at);
        r.m_bits = lds_u16(blk + m + at);
    }
    return r;
}

// Eq. 3 on 32 codes, rounded once to bf16: fma.rn.bf16x2 of the exact codes, scale and offset.  A permute places codes 2 i and
// 2 i + 1 as the low bytes of a bf16 pair (its sign fill gives the zeros above them): the bf16 subnormals q 2^-133.  A
// multiplication by 2^127 and a scale of 64 d make that q d; both products are exact.  On this GPU logic and permute instructions
// and packed bf16 arithmetic are issued at half rate on pipes of their own: 28 and 32 per group here, against 44 and 16 with 64
// fp32 FMAs and conversions in the tile kernels.  BIG: for any finite scale (64 times one of 2^122 is not finite).
template <bool BIG>
__device__ __forceinline__ void convert32(const uint4& codes, uint32_t d_bits, uint32_t m_bits, uint32_t* out) {
    uint32_t d2 = pf_prmt(d_bits, 0, 0x1010u);
    const uint32_t m2 = pf_prmt(m_bits, 0, 0x1010u), words[4] = {codes.x, codes.y, codes.z, codes.w};
    if (!BIG) asm("mul.rn.bf16x2 %0, %0, %1;" : "+r"(d2) : "r"(0x42804280u));  // 64 d
#pragma unroll
    for (int wi = 0; wi < 4; ++wi) {
        const uint32_t e = words[wi] & 0x0F0F0F0Fu, o = (words[wi] >> 4) & 0x0F0F0F0Fu;
        uint32_t t[4] = {pf_prmt(e, o, 0xC480u), pf_prmt(e, o, 0xD591u), pf_prmt(e, o, 0xE6A2u), pf_prmt(e, o, 0xF7B3u)};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            asm("mul.rn.bf16x2 %0, %0, %1;" : "+r"(t[i]) : "r"(0x7F007F00u));          // 2^127: q / 64
            if (BIG) asm("mul.rn.bf16x2 %0, %0, %1;" : "+r"(t[i]) : "r"(0x42804280u));  // q
            asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(out[4 * wi + i]) : "r"(t[i]), "r"(d2), "r"(m2));
        }
    }
}

// A tile that the pairs of one cluster share, a K range each: part h is summed by pair h % split, the others write theirs into its
// shared memory.  All of them are resident, so it may wait for them: from the accumulators to y in about 2000 cycles, where the
// way through global memory and a counter takes 7000.
__device__ __forceinline__ void finish_cluster(const StreamParams& p, uint32_t exchange, uint32_t acc, int q, int h, uint32_t crank, int strip,
                                               bool rows, int toks, int lane) {
    const int sub = (int)(crank >> 1), owner = h % p.split, slots = kStParts / p.split, granules = (p.n_inst + 16 * kStParts - 1) / (16 * kStParts);
    const uint32_t bar = exchange + 8u * (uint32_t)(q * kStParts + h), piece_bytes = 2048u * (uint32_t)granules;
    const uint32_t mine = exchange + 128u + (uint32_t)((q * slots + h / p.split) * (p.split - 1)) * piece_bytes + 16u * (uint32_t)lane;
    if (owner != sub) {
        const uint32_t target = 2u * (uint32_t)owner + (crank & 1u);
        uint32_t to = mapa_shared(mine, target) + (uint32_t)(sub < owner ? sub : sub - 1) * piece_bytes;
        for (int c = 16 * h; rows && c < toks; c += 16 * kStParts, to += 2048u) {
            float v[16];
            tmem_ld_16cols(acc + (uint32_t)c, v);
#pragma unroll
            for (int i = 0; i < 4; ++i) st_cluster(to + 512u * (uint32_t)i, v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive_release_cluster(mapa_shared(bar, target));
        return;
    }
    if (!__all_sync(0xffffffffu, mbar_wait_cluster(bar, 0, p.status)) || !rows) return;
    uint32_t from = mine;
    for (int c = 16 * h; c < toks; c += 16 * kStParts, from += 2048u) {
        float sum[16];
        for (int r = 0; r < p.split; ++r) {
            float v[16];
            if (r == sub) {
                tmem_ld_16cols(acc + (uint32_t)c, v);
            } else {
                const uint32_t at = from + (uint32_t)(r < sub ? r : r - 1) * piece_bytes;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint4 w = lds128(at + 512u * (uint32_t)i);
                    v[4 * i] = __uint_as_float(w.x), v[4 * i + 1] = __uint_as_float(w.y), v[4 * i + 2] = __uint_as_float(w.z), v[4 * i + 3] = __uint_as_float(w.w);
                }
            }
#pragma unroll
            for (int i = 0; i < 16; ++i) sum[i] = r ? sum[i] + v[i] : v[i];
        }
        store_chunk(p, sum, strip, lane, 0, c, toks);
    }
}

// Reads the accumulators of the segment (a pair's part [u0, u1) of a tile, the one that ends before unit e), parts [h0, h1) of
// this warp's strip, and stores y or, where the tile is shared, partial sums.  The last pair at a part's counter adds them; one
// that finds all the others there before its own sums are complete leaves these where they are.
template <bool CLUSTER>
__device__ __forceinline__ bool st_finish(const StreamParams& p, uint32_t acc_bars, uint32_t acc_last, uint32_t exchange, int u0, int u1, int e, int h0, int h1) {
    const int lane = threadIdx.x & 31, q = (threadIdx.x >> 5) & 3, pair = (int)(blockIdx.x >> 1);
    const uint32_t crank = cluster_ctarank();
    const int strip8 = 4 * (int)(crank & 1u) + q;
    const int tile = (e - 1) / p.nb, idx = tile - u0 / p.nb;
    const int b = p.acc_sets == 2 ? idx & 1 : 0;
    const StAccWait full = st_acc_wait(p.acc_sets, idx, e == u1);
    const int n_tile = tile / p.tok_tiles, tok0 = (tile - n_tile * p.tok_tiles) * p.n_inst;
    const int toks = p.M - tok0 < p.n_inst ? p.M - tok0 : p.n_inst;
    const int strip = n_tile * 8 + strip8;
    const bool whole = tile * p.nb >= u0 && (tile + 1) * p.nb == e, rows = strip < p.N / kStripRows;
    const uint32_t acc = ((uint32_t)(q * 32) << 16) + (uint32_t)(b * p.n_inst);
    SharedTile s;
    int* tickets = nullptr;
    bool others = false;
    if (!CLUSTER && !whole) {
        s = shared_tile(p, tile, strip8, lane);
        tickets = p.tickets + s.p0 * kStTickets + strip8 * kStParts;
        if (h1 == h0 + 1) {
            int seen;
            asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(seen) : "l"(tickets + h0) : "memory");
            others = __all_sync(0xffffffffu, seen == s.p1 - s.p0);
        }
    }
    if (!warp_wait(full.bar == kStAccLast ? acc_last : acc_bars + 8u * (uint32_t)b, full.phase & 1u, p.status)) return false;
    tc_fence_after();
    if (CLUSTER) {
        finish_cluster(p, exchange, acc, q, h0, crank, strip, rows, toks, lane);
        return true;
    }
    if (rows && whole) {
        for (int h = h0; h < h1; ++h)
            for (int c = 16 * h; c < toks; c += 16 * kStParts) {
                float v[16];
                tmem_ld_16cols(acc + (uint32_t)c, v);
                store_chunk(p, v, strip, lane, tok0, c, toks);
            }
    } else if (rows && others) {
        sum_shared(p, s, pair, acc, strip, lane, tok0, toks, h0);
        if (lane == 0) tickets[h0] = 0;  // for the next launch
    } else if (rows) {
        float4* mine = s.slot(pair);
        for (int h = h0; h < h1; ++h)
            for (int c = 16 * h; c < toks; c += 16 * kStParts) {
                float v[16];
                tmem_ld_16cols(acc + (uint32_t)c, v);
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (c + 4 * i < toks) __stcg(mine + (c / 4 + i) * 32, make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]));
            }
    }
    if (e < u1) {  // (nobody waits for the last one)
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(mapa_shared(acc_bars + 8u * (uint32_t)(2 + b), crank & ~1u));
    }
    if (rows && !whole && !others) {
        // the warp's stores, then the arrival; and, at the last one, the others' stores behind their arrivals
        int seen = -1;
        __syncwarp();
        if (lane >= h0 && lane < h1) {
            asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], 1;" : "=r"(seen) : "l"(tickets + lane) : "memory");
            if (seen == s.p1 - s.p0) tickets[lane] = 0;  // for the next launch
        }
        const uint32_t last = __ballot_sync(0xffffffffu, seen == s.p1 - s.p0);
        __syncwarp();
        for (int h = h0; h < h1; ++h)
            if (last >> h & 1u) sum_shared(p, s, -1, 0, strip, lane, tok0, toks, h);
    }
    return true;
}

// ---- the kernel -------------------------------------------------------------------------------------------------------

// CLUSTER: p.split pairs share a tile and add their sums through shared memory.
template <int FMT, bool CLUSTER>
__global__ void __launch_bounds__(kStThreads, 1) fdqp_prefill_stream_kernel(const __grid_constant__ CUtensorMap x_map, const __grid_constant__ StreamParams p) {
    using F = FmtTraits<FMT>;
    extern __shared__ uint8_t smem_raw[];
    // (the broadcast tells the compiler that `warp` is uniform: the MMA issuer's descriptors then live in uniform registers)
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t x_ring = (raw + 1023u) & ~1023u;  // swizzle atoms; the same offset in both CTAs
    const uint32_t x_stage = (uint32_t)p.x_steps * p.x_box_bytes;
    const uint32_t w_ring = x_ring + (uint32_t)p.x_stages * x_stage;
    constexpr uint32_t kWStage = 4u * (uint32_t)F::kBlock;
    const uint32_t exchange = w_ring + (uint32_t)p.w_stages * kWStage;  // 16 barriers and sums of the cluster's other pairs
    const uint32_t bars = exchange + p.exchange_bytes;
    auto full_a = [&](int s) { return bars + 8u * (uint32_t)s; };                                  // CTA 0's: 16 warps
    auto empty_a = [&](int s) { return bars + 8u * (uint32_t)(4 + s); };                            // each its own, by commit
    auto acc_full = [&](int b) { return bars + 8u * (uint32_t)(8 + b); };                           // each its own, by commit (and acc_last)
    auto acc_empty = [&](int b) { return bars + 8u * (uint32_t)(10 + b); };                         // CTA 0's: the warps that read it
    auto full_w = [&](int s) { return bars + 8u * (uint32_t)(12 + s); };                            // each its own: 2 warps + bytes
    auto empty_w = [&](int s) { return bars + 8u * (uint32_t)(12 + kStMaxW + s); };                 // each its own: 8 warps
    const uint32_t tmem_slot = bars + 8u * (uint32_t)(12 + 2 * kStMaxW);
    const uint32_t acc_last = tmem_slot + 8u;
    const uint32_t x_bars = tmem_slot + 16u;
    auto full_x = [&](int s) { return x_bars + 8u * (uint32_t)s; };                                 // CTA 0's: 1 + both CTAs' bytes
    auto empty_x = [&](int s) { return x_bars + 8u * (uint32_t)(p.x_stages + s); };                 // each its own, by commit

    const uint32_t crank = cluster_ctarank(), rank = crank & 1u, leader_cta = crank & ~1u;  // CTA 0 of the pair, in its cluster
    const uint16_t pair_mask = (uint16_t)(3u << leader_cta);
    const int pair = (int)(blockIdx.x >> 1);
    // this pair's units: a part of its cluster's tile, or its range of the line of them all
    const int sub = (int)(crank >> 1), first_unit = CLUSTER ? pair / p.split * p.nb : 0;
    const int u0 = CLUSTER ? first_unit + p.nb * sub / p.split : st_range_begin(p, pair);
    const int u1 = CLUSTER ? first_unit + p.nb * (sub + 1) / p.split : st_range_begin(p, pair + 1);
    const int groups = p.K / kGroup;
    const int groups_last = groups - 8 * (p.nb - 1);        // groups of a strip's last block
    const int ksteps_last = (groups_last + 1) / 2;
    auto ksteps_of = [&](int kb) { return kb == p.nb - 1 ? ksteps_last : 4; };

    // Packed weights, warps 2 and 3: two strips' blocks of a unit each.  One elected lane issues; the loop is uniform.
    const int strips = p.N / kStripRows;
    const int64_t strip_bytes = FMT == kFmtQ4nx ? (int64_t)kGroupBytes * groups : (int64_t)F::kBlock * p.nb;
    const int tile0 = u0 / p.nb, kb0 = u0 % p.nb;
    const uint64_t policy = l2_policy_evict_first();
    int w_kb = kb0, w_tile = tile0;
    auto load_blocks = [&](int s) {
        const int half = 2 * (warp & 1);
        const int strip = (w_tile / p.tok_tiles) * 8 + 4 * (int)rank + half, left = strips - strip;
        const uint32_t bytes = FMT == kFmtQ4nx && w_kb == p.nb - 1 ? (uint32_t)(kGroupBytes * groups_last) : (uint32_t)F::kBlock;
        const uint8_t* src = p.W + strip * strip_bytes + (int64_t)w_kb * F::kBlock;
        const uint32_t dst = w_ring + (uint32_t)s * kWStage + (uint32_t)(half * F::kBlock), bar = full_w(s);
        if (elect_one()) {
            mbar_arrive_expect_tx(bar, left >= 2 ? 2 * bytes : (left == 1 ? bytes : 0u));
            if (p.tok_tiles == 1) {
                if (left >= 1) bulk_g2s_hint(dst, src, bytes, bar, policy);
                if (left >= 2) bulk_g2s_hint(dst + F::kBlock, src + strip_bytes, bytes, bar, policy);
            } else {  // (read again by the next token tile)
                if (left >= 1) bulk_g2s(dst, src, bytes, bar);
                if (left >= 2) bulk_g2s(dst + F::kBlock, src + strip_bytes, bytes, bar);
            }
        }
        __syncwarp();
        if (++w_kb == p.nb) {
            w_kb = 0;
            ++w_tile;
        }
    };
    // The first weights are on their way before anything else.
    const int w_first = u1 - u0 < p.w_stages ? u1 - u0 : p.w_stages, w_early = w_first < 2 ? w_first : 2;
    if (warp == 2 || warp == 3) {
        if (warp == 2) {
            if (lane < 2 * kStMaxW) mbar_init(full_w(lane), lane < kStMaxW ? 2u : 8u);
            mbar_fence_init();
        }
        asm volatile("bar.sync 1, 64;" ::: "memory");
        for (int s = 0; s < w_early; ++s) load_blocks(s);
    }
    // A thread per barrier: initialising them in a row took 2 us.  (Relaxed arrival: the fences have released them.)
    if (warp == 0) {
        tmem_alloc2(tmem_slot, 512);
        tmem_relinquish2();
    } else if (warp == 4) {
        if (lane < 13)
            mbar_init(lane == 12 ? acc_last : bars + 8u * (uint32_t)lane, lane < 4 ? 16u : (lane < 10 || lane == 12 ? 1u : (p.acc_sets == 1 ? 8u * kStParts : 8u)));
        mbar_fence_init();
    } else if (warp == 6) {
        if (CLUSTER && lane < 16) mbar_init(exchange + 8u * (uint32_t)lane, (uint32_t)p.split - 1u);
        mbar_fence_init();
    } else if (warp == 5) {
        for (int s = lane; s < 2 * p.x_stages; s += 32) mbar_init(full_x(s), 1);  // (and empty_x, behind them)
        mbar_fence_init();
    }
    tc_fence_before();
    __syncthreads();
    cluster_arrive_relaxed();
    if (warp == 2 || warp == 3)
        for (int s = w_early; s < w_first; ++s) load_blocks(s);
    cluster_wait();  // barriers of both CTAs initialised, tensor memory allocated in both
    tc_fence_after();
    // All 512 columns of tensor memory, so they begin at 0: accumulators (one or two sets of n_inst columns), and two or three
    // stages of converted weights, 128 columns to a block, at the end.
    const uint32_t tmem_a = 512u - 128u * (uint32_t)p.a_stages;
    bool ok = true;
    // Launch chaining: the launch behind this one may begin as SMs become free; weights are fetched ahead of the wait, x, y and
    // the workspace are touched after it.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    if (warp == 0) {
        // =============================== x boxes ============================================================
        asm volatile("griddepcontrol.wait;" ::: "memory");
        const int per_block = 4 / p.x_steps;  // stages
        int kb = kb0, tile = tile0, s = p.x_resident ? per_block * kb : 0;
        uint32_t ph = 0;
        const int u_end = p.x_resident && u1 - u0 > p.nb ? u0 + p.nb : u1;  // resident: every stage once
        const uint32_t bar0 = mapa_shared(full_x(0), leader_cta);
        for (int u = u0; u < u_end && ok; ++u) {
            const int n = ksteps_of(kb);
            const int row = (tile % p.tok_tiles) * p.n_inst + (int)rank * (p.n_inst / 2);
            for (int j = 0; j < n; j += p.x_steps) {
                if (!p.x_resident && !(ok = warp_wait(empty_x(s), ph ^ 1u, p.status))) break;
                const uint32_t dst = x_ring + (uint32_t)s * x_stage, bar = bar0 + 8u * (uint32_t)s;
                const int step = 4 * kb + j, here = n - j < p.x_steps ? n - j : p.x_steps;
                if (elect_one()) {
                    // both CTAs' boxes (the three-dimensional one comes whole: zeros past K)
                    if (rank == 0) mbar_arrive_expect_tx(full_x(s), 2u * (uint32_t)(p.x_3d ? p.x_steps : here) * p.x_box_bytes);
                    if (p.x_3d) tma2_load_3d(dst, &x_map, 0, row, step, bar);
                    else
                        for (int i = 0; i < here; ++i) tma2_load_2d(dst + (uint32_t)i * p.x_box_bytes, &x_map, (step + i) * kPfK, row, bar);
                }
                __syncwarp();
                if (++s == p.x_stages) {
                    s = 0;
                    ph ^= 1u;
                }
            }
            if (++kb == p.nb) {
                kb = 0;
                ++tile;
                if (p.x_resident) s = 0;
            }
        }
    } else if (warp == 1) {
        // =============================== MMA issuer (CTA 0 of the pair) ======================================
        // The warp runs the loop on uniform values and one elected lane issues; a block (up to sixteen MMAs) per wait and commit.
        // Waits are of CTA scope: the stages' data is ordered by the tensor-core fences and the async proxy.  (A single thread
        // with cluster-scope waits per k-step took 1040 cycles for each, whatever else there was to do; uniform code with the
        // next k-step's barriers tested ahead 540.)
        if (rank == 0) {
            // kind::f16: D fp32, A and B bf16, both K-major, M = 256 over the pair
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((256u >> 4) << 24) | ((uint32_t)(p.n_inst >> 3) << 17);
            const bool leader = elect_one();
            const int per_block = 4 / p.x_steps;
            int kb = kb0, sx = p.x_resident ? per_block * kb : 0, sa = 0, b = 0;
            uint32_t pha = 0, phx = 0, phb = 0;
            bool first = true, ready = false;  // ready: the next block's first stages have been seen full
            for (int u = u0; u < u1 && ok; ++u) {
                const bool wait_x = !p.x_resident || u - u0 < p.nb;  // (boxes that stay: full once and for all)
                if (first && !(ok = warp_wait(acc_empty(b), phb ^ 1u, p.status))) break;
                if (!ready) {
                    if (wait_x && !(ok = warp_wait(full_x(sx), phx, p.status))) break;
                    if (!(ok = warp_wait(full_a(sa), pha, p.status))) break;
                }
                tc_fence_after();
                const int n = ksteps_of(kb);
                const uint32_t d = (uint32_t)(b * p.n_inst), a = tmem_a + 128u * (uint32_t)sa, used_a = empty_a(sa);
                const bool tile_end = kb + 1 == p.nb, done = tile_end || u + 1 == u1;  // this pair's part of the tile
                if (++sa == p.a_stages) {
                    sa = 0;
                    pha ^= 1u;
                }
                bool peek = false;
                if (p.x_steps == 4) {
                    const uint64_t bdesc = umma_smem_desc(x_ring + (uint32_t)sx * x_stage), box = (uint64_t)(p.x_box_bytes >> 4);
                    const uint32_t used_x = empty_x(sx);
                    if (++sx == p.x_stages || (p.x_resident && tile_end)) {
                        sx = 0;
                        if (!p.x_resident) phx ^= 1u;
                    }
                    peek = mbar_test(full_a(sa), pha) & ((p.x_resident && u + 1 - u0 >= p.nb) || mbar_test(full_x(sx), phx));
                    if (leader) {
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (j < n) {
#pragma unroll
                                for (int k4 = 0; k4 < 4; ++k4)
                                    umma2_bf16_ta(d, a + (uint32_t)(32 * j + 8 * k4), bdesc + (uint64_t)j * box + 2 * k4, idesc, first && j + k4 == 0 ? 0u : 1u);
                            }
                        umma2_commit(used_a, pair_mask);
                        if (!p.x_resident) umma2_commit(used_x, pair_mask);
                        if (done) umma2_commit(u + 1 == u1 ? acc_last : acc_full(b), pair_mask);
                    }
                } else {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (2 * h >= n) break;
                        if (h && !(ok = warp_wait(full_x(sx), phx, p.status))) break;
                        const uint64_t bdesc = umma_smem_desc(x_ring + (uint32_t)sx * x_stage), box = (uint64_t)(p.x_box_bytes >> 4);
                        if (leader) {
#pragma unroll
                            for (int j = 0; j < 2; ++j)
                                if (2 * h + j < n) {
#pragma unroll
                                    for (int k4 = 0; k4 < 4; ++k4)
                                        umma2_bf16_ta(d, a + (uint32_t)(64 * h + 32 * j + 8 * k4), bdesc + (uint64_t)j * box + 2 * k4, idesc,
                                                      first && h + j + k4 == 0 ? 0u : 1u);
                                }
                            umma2_commit(empty_x(sx), pair_mask);
                        }
                        __syncwarp();
                        if (++sx == p.x_stages) {
                            sx = 0;
                            phx ^= 1u;
                        }
                    }
                    if (leader) {
                        umma2_commit(used_a, pair_mask);
                        if (done) umma2_commit(u + 1 == u1 ? acc_last : acc_full(b), pair_mask);
                    }
                }
                __syncwarp();
                ready = __all_sync(0xffffffffu, peek);
                first = done;
                if (done && ++b == p.acc_sets) {
                    b = 0;
                    phb ^= 1u;
                }
                kb = tile_end ? 0 : kb + 1;
            }
        }
    } else if (warp < 4) {
        // =============================== packed weights ======================================================
        int s = w_first == p.w_stages ? 0 : w_first;
        uint32_t ph = 0;  // (the first round is under way)
        for (int u = u0 + w_first; u < u1; ++u) {
            if (!(ok = warp_wait(empty_w(s), ph, p.status))) break;
            load_blocks(s);
            if (++s == p.w_stages) {
                s = 0;
                ph ^= 1u;
            }
        }
        // The last release of every stage of converted weights and of x has arrived (beside the read-out of the last sums; a lane a
        // barrier).
        if (warp == 2 && ok && warp_wait(acc_last, 0, p.status)) {
            const int x_loads = p.x_resident ? 0 : st_x_loads(u0, u1, p.nb, p.x_steps, ksteps_last);
            const bool of_a = lane < 4;
            const int s = of_a ? lane : lane - 4, stages = of_a ? p.a_stages : p.x_stages;
            const int uses = s < stages ? st_stage_uses(s, of_a ? u1 - u0 : x_loads, stages) : 0;
            if (uses) mbar_wait(of_a ? empty_a(s) : empty_x(s), (uint32_t)(uses - 1) & 1u, p.status);
        }
    } else {
        // =============================== conversion; accumulators -> y =======================================
        // Strip (= the warp's lane quarter of tensor memory) and place i among the strip's warps: half i % 2 of every second block.
        // (A wait tells a stage's phase from the next one only, not from that of two uses before.  When a warp comes round, the
        // block a_stages before its last one has been through the MMAs, which take the blocks in order: it waited for that stage of
        // converted weights.  So with four stages of packed weights or more, and two or three of converted ones, the use before the
        // one that it waits for is complete.  The accumulators of a range's last segment: st_acc_wait.)
        const bool converts = warp >= 8;
        const int q = warp & 3, i = converts ? (warp - 8) >> 2 : 0, t0 = 4 * (i & 1);
        const uint32_t full0 = mapa_shared(full_a(0), leader_cta);
        const uint32_t a_lane = tmem_a + ((uint32_t)(q * 32) << 16) + 64u * (uint32_t)(i & 1);
        const uint32_t blk0 = w_ring + (uint32_t)(q * F::kBlock);
        const uint32_t code0 = blk0 + (uint32_t)(512 * t0 + 16 * lane);
        const uint32_t meta0 = blk0 + (uint32_t)(kCodeBytes + (F::kMx ? 32 * t0 + lane : 64 * (t0 >> F::kShift) + 2 * lane));
        const bool ragged = FMT == kFmtQ4nx && groups_last < 8;
        int kb = kb0 + (i >> 1), sw = i >> 1, sa = i >> 1;
        uint32_t phw = 0, pha = 1;
        if (kb >= p.nb) kb -= p.nb;
        int u = u0 + (i >> 1);
        // Segments (parts of tiles) to read: all but the last one by the strip's warp of 4..7 where there are two sets of
        // accumulators, all parts; else, and the last one, a part each by the conversion warps.
        int seg_end = (tile0 + 1) * p.nb;
        if (converts && p.acc_sets == 2) seg_end = u1;
        if (seg_end > u1) seg_end = u1;
        bool waited = false;
        while (ok && (converts || (p.acc_sets == 2 && seg_end < u1))) {
            // (a segment's accumulators are read when the stages of converted weights are full again, two blocks into the next one)
            const int until = seg_end == u1 ? u1 : (p.nb < 2 ? seg_end + p.nb : seg_end + 2);
            while (converts && u < u1 && u < until) {
                if (!(ok = warp_wait(full_w(sw), phw, p.status))) break;
                const uint32_t at = (uint32_t)sw * kWStage;
                const uint32_t a_dst = a_lane + 128u * (uint32_t)sa;
                uint32_t d[4], m[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    m[k] = 0;
                    if (F::kMx) {
                        asm volatile("ld.shared.u8 %0, [%1];" : "=r"(d[k]) : "r"(meta0 + at + 32u * (uint32_t)k));
                    } else {
                        d[k] = lds_u16(meta0 + at + 64u * (uint32_t)(k >> F::kShift));
                        m[k] = lds_u16(meta0 + at + (uint32_t)(F::kOffSect - kCodeBytes) + 64u * (uint32_t)(k >> F::kShift));
                    }
                }
                uint4 codes[2] = {lds128(code0 + at), lds128(code0 + at + 512u)};
                if (!(ok = warp_wait(empty_a(sa), pha, p.status))) break;
                tc_fence_after();
                // (rows past N, rows of an absent strip: whatever shared memory holds, in lanes that nobody reads)
                const bool plain = F::kMx || !__any_sync(0xffffffffu, (d[0] | d[1] | d[2] | d[3]) & 0x4000u);  // no scale of 2 or more
                if (plain && !(ragged && kb == p.nb - 1)) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        uint32_t out[16];
                        if (F::kMx) {
                            GroupRegs g;
                            g.codes = codes[k & 1];
                            g.d_bits = d[k];
                            g.m_bits = 0;
                            g.valid = true;
                            group_convert<FMT>(g, out);
                        } else {
                            convert32<false>(codes[k & 1], d[k], m[k], out);
                        }
                        if (k < 2) codes[k] = lds128(code0 + at + 512u * (uint32_t)(k + 2));
                        tmem_st_16cols_async(a_dst + 16u * (uint32_t)k, out);
                    }
                } else {
                    const int jb = ragged && kb == p.nb - 1 ? groups_last : 8;
#pragma unroll 1
                    for (int k = 0; k < 4; ++k) {
                        uint32_t out[16];
#pragma unroll
                        for (int z = 0; z < 16; ++z) out[z] = 0;
                        if (t0 + k < jb) {
                            const GroupRegs g = group_from_smem<FMT>(blk0 + at, t0 + k, jb, lane);
                            convert32<true>(g.codes, g.d_bits, g.m_bits, out);
                        }
                        tmem_st_16cols_async(a_dst + 16u * (uint32_t)k, out);
                    }
                }
                if (lane == 0) mbar_arrive(empty_w(sw));  // (every lane's codes are in use)
                tmem_st_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    if (rank == 0) mbar_arrive(full_a(sa));
                    else mbar_arrive_cluster(full0 + 8u * (uint32_t)sa);
                }
                u += 2;
                sa += 2;
                if (sa >= p.a_stages) {
                    sa -= p.a_stages;
                    pha ^= 1u;
                }
                sw += 2;
                if (sw >= p.w_stages) {
                    sw -= p.w_stages;
                    phw ^= 1u;
                }
                kb += 2;
                while (kb >= p.nb) kb -= p.nb;
            }
            if (!ok) break;
            if (!waited) asm volatile("griddepcontrol.wait;" ::: "memory");
            waited = true;
            ok = st_finish<CLUSTER>(p, acc_full(0), acc_last, exchange, u0, u1, seg_end, converts ? i : 0, converts ? i + 1 : kStParts);
            if (seg_end == u1) break;
            seg_end = seg_end + p.nb < u1 ? seg_end + p.nb : u1;
        }
    }
    // =============================== teardown: every path of both CTAs releases tensor memory ================
    __syncwarp();
    tc_fence_before();
    cluster_sync_all();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc2(0, 512);
    }
}

// ---- host side ----------------------------------------------------------------------------------------------------

template <int FMT>
static cudaError_t stream_set_smem_limit(int bytes) {
    const cudaError_t e = cudaFuncSetAttribute(fdqp_prefill_stream_kernel<FMT, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    return e ? e : cudaFuncSetAttribute(fdqp_prefill_stream_kernel<FMT, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

cudaError_t prefill_stream_set_smem_limit(int bytes) {
    cudaError_t e;
    if ((e = stream_set_smem_limit<kFmtQ4nx>(bytes))) return e;
    if ((e = stream_set_smem_limit<kFmtG64>(bytes))) return e;
    if ((e = stream_set_smem_limit<kFmtG128>(bytes))) return e;
    return stream_set_smem_limit<kFmtMxfp4>(bytes);
}

// Clusters of `ctas` CTAs that can be resident at once (0: none).
int prefill_stream_max_clusters(int ctas, int smem_bytes) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3(kStThreads);
    cfg.dynamicSmemBytes = (size_t)smem_bytes;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)ctas;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, fdqp_prefill_stream_kernel<kFmtQ4nx, true>, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

template <int FMT>
static cudaError_t stream_launch(const CUtensorMap& map, const StreamParams& p, bool ahead, cudaStream_t stream) {
    return launch_chained(p.split > 1 ? fdqp_prefill_stream_kernel<FMT, true> : fdqp_prefill_stream_kernel<FMT, false>, 2 * (int64_t)p.pairs, kStThreads,
                          p.smem_bytes, 2 * p.split, ahead, stream, map, p);
}

cudaError_t prefill_stream_launch(const StreamParams& p, const uint16_t* x, int fmt, bool ahead, cudaStream_t stream) {
    EncodeTiledFn encode = encode_tiled_fn();
    if (!encode) return cudaErrorNotSupported;
    CUtensorMap map;
    cuuint32_t elem[3] = {1, 1, 1};
    CUresult r;
    if (p.x_3d) {
        const cuuint64_t dims[3] = {kPfK, (cuuint64_t)p.M, (cuuint64_t)(p.K / kPfK)}, strides[2] = {(cuuint64_t)p.K * 2, kPfK * 2};
        const cuuint32_t box[3] = {kPfK, (cuuint32_t)(p.n_inst / 2), (cuuint32_t)p.x_steps};
        r = encode(&map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<uint16_t*>(x), dims, strides, box, elem, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    } else {
        const cuuint64_t dims[2] = {(cuuint64_t)p.K, (cuuint64_t)p.M}, strides[1] = {(cuuint64_t)p.K * 2};  // innermost first
        const cuuint32_t box[2] = {kPfK, (cuuint32_t)(p.n_inst / 2)};
        r = encode(&map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<uint16_t*>(x), dims, strides, box, elem, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    }
    if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
    switch (fmt) {
        case kFmtQ4nx: return stream_launch<kFmtQ4nx>(map, p, ahead, stream);
        case kFmtG64: return stream_launch<kFmtG64>(map, p, ahead, stream);
        case kFmtG128: return stream_launch<kFmtG128>(map, p, ahead, stream);
        case kFmtMxfp4: return stream_launch<kFmtMxfp4>(map, p, ahead, stream);
    }
    return cudaErrorInvalidValue;
}

}  // namespace fdqp
