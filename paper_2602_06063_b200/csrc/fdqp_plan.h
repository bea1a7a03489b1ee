// Launch plan of the streaming GEMV kernels: the quantities the host fixes per call and the
// kernel re-derives per CTA.  Plain data, shared by the host dispatcher and the device code.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define FDQP_HD __host__ __device__
#else
#define FDQP_HD
#endif

namespace fdqp {

constexpr int kStripRows = 32;      // output features per strip
constexpr int kGroup = 32;          // quantisation group along K
constexpr int kBlockK = 256;        // input features per full Q4NX block
constexpr int kBlockBytes = 5120;   // bytes of a full block (Sec. "Dequantization Engine")
constexpr int kGroupBytes = 640;    // bytes a block spends per group: 512 codes + 64 scales + 64 offsets
constexpr int kMaxTokens = 8;       // token rows one GEMV launch handles
// What a kernel writes for a finished output value (values of fdqp_epilogue in fdqp.h).
constexpr int kEpiNone = 0;       // fp32 y [M][N]
constexpr int kEpiBf16 = 1;       // bf16 y [M][N]
constexpr int kEpiGegluBf16 = 2;  // bf16 [M][N/2]: gelu(row r) * (row r + 16) of every 32-row strip
// Up to this many tokens the GEMV lays the byte planes of a token out as MMA columns; above it, one MMA per plane.
constexpr int kColsMaxTokens = 2;
// Column modes hand three partial terms per (row, token) to the reducer (two column halves + the offset term).
constexpr int kColsPartTerms = 3;
// Prepared activations of the chained kernel, per group-tile (written by xprep_item, read by its tile loop):
//   column modes (M <= 2): one 136-byte record per (group-tile, token) -- four signed byte planes of the 31-bit fixed
//   point (4 x 32 bytes) and {sum of x, unit} at 128;
//   M >= 3: the bf16 activations themselves in MMA fragment order, 64 bytes per (group-tile, token), and the sums of x
//   of the (up to eight) tokens, 32 bytes per group-tile.
constexpr int kColsRecBytes = 136, kColsSumOff = 128, kColsUnitOff = 132;
constexpr int kPlaneRecBytes = 64, kPlaneSumBytes = 32;
// Prepared activations of the GEMV kernels: one record per block of 256 inputs (eight group-tiles t).
//   M <= 2: planes, 128 bytes per (t, token): four signed byte planes of the 31-bit fixed point, most significant first;
//     then 64 bytes per token: the units of the eight tiles times 65536, and the units;
//     then 128 bytes: the sums of x as a B fragment [8 tiles][8 columns], columns 4 token + {0, 1, 2} = its three bf16
//     parts (MXFP4: instead 16 bytes per (t, token), the four planes' MMA start values).
//   M >= 3: 64 bytes per (t, token), the bf16 activations in MMA fragment order; then 512 bytes: the sums of x as B
//     fragments [8 tiles][8 tokens], 16 bytes per lane: its word of the first, second and third parts (MXFP4: none).
FDQP_HD constexpr int gemv_rec_bytes(int M, bool mx) {
    return M <= kColsMaxTokens ? M * 1088 + (mx ? M * 128 : 128) : M * 512 + (mx ? 0 : 512);
}
constexpr int kMaxDepth = 16;       // blocks a warp's ring holds at most
constexpr int kMaxSplit = 8;        // K slices
constexpr int kMaxCtasPerSm = 2;

struct GemvPlan {
    const uint8_t* W;     // device, packed Q4NX
    const uint16_t* x;    // device, [M][K] bf16 bits
    const uint8_t* xq;    // device, records of a call whose x is prepared by fdqp_xprep_kernel (layout above)
    float* y;             // device, fp32 output [M][N] (epilogue kEpiNone)
    uint16_t* y16;        // device, bf16 output (other epilogues)
    int epi;
    const uint16_t* gamma;  // RMS normalisation of x fused into the in-kernel activation preparation (norm != 0):
    float eps;              //   x <- bf16(x * rsqrt(mean(x^2) + eps) * (1 + gamma)), per token row
    int norm;
    const uint16_t* residual;  // with norm: x + residual (bf16, one rounding) is what gets normalised ...
    uint16_t* h_out;           // ... and, when not null, is also written here by the grid's first CTA ([M][K] bf16)
    float* ws_edge;       // device, [grid][2][32*kMaxTokens] partial sums of strips shared between CTAs
    float* ws_full;       // device, [Z][S][32*kMaxTokens] partial sums of whole strip-slices (Z > 1)
    int* tickets;         // device, [S] arrival counters, zero between launches
    int* status;          // host-mapped sticky status word
    int fmt;              // container format (fdqp_format.h); 0 = Q4NX
    int M, K, N;
    int S;                // strips = N / 32
    int nb;               // blocks per strip = ceil(K / 256)
    int Z;                // K slices
    int nbz;              // blocks per slice = ceil(nb / Z); every slice is non-empty
    int Gz;               // CTAs per slice; grid = Z * Gz
    int warps;            // warps per CTA: 8, 12 or 16
    int active_warps;     // of which this many stream blocks (fewer only where the rings of all would not fit)
    int depth;            // blocks a warp's ring holds
    uint32_t gz_magic, len_magic;  // reciprocals of Gz and of a full slice's strip length (0: divide)
    int evict_first;      // weight copies carry an evict-first L2 hint
    int strip_aligned;    // 1: CTA ranges are cut at strip boundaries (no strip is shared between CTAs of a slice)
    int prep_inline;      // 1: every CTA prepares its K slice of x itself; 0: a preparation kernel ran before
    uint32_t off_xs;      // shared-memory offsets (bytes): activation records,
    uint32_t off_part;    //   head pieces, sums of a fused normalisation, barriers
    uint32_t off_norm;
    uint32_t off_bar;
    uint32_t smem_bytes;
};

// ---- prefill-sized calls, pairs of SMs that stay (fdqp_prefill_stream.cu) -------------------------------------------
constexpr int kStMaxX = 64, kStMaxW = 8;           // ring stages at most: half blocks of x, blocks of packed weights
constexpr int kStMinW = 4;                         // (the kernel's waits rely on it)
constexpr int kStMaxTokens = 256;                  // tokens of a tile
constexpr int kStBarBytes = 8 * (12 + 2 * kStMaxW) + 16;  // barriers of fixed number; and 16 per stage of x
constexpr int kStParts = 4;                        // warps that share a strip's accumulators at the end of a CTA's range
constexpr int kStTickets = 8 * kStParts;           // arrival counters per pair

struct StreamParams {
    const uint8_t* W;       // device, packed
    float* y;               // device, fp32 output [M][N] (epilogue kEpiNone)
    uint16_t* y16;          // device, bf16 output (other epilogues)
    float* ws;              // device, partial sums of tiles that pairs share: [pairs][2][8 strips][n_inst][32]
    int* tickets;           // device, [pairs][kStTickets] arrival counters, zero between launches
    int* status;            // host-mapped sticky status word
    int M, K, N, epi;
    int n_inst;             // tokens of a tile (a multiple of 16 up to 256)
    int tok_tiles, tiles;   // token tiles; tiles in all (token tiles of the same 256 output features adjacent)
    int nb;                 // blocks of 256 k
    int pairs;              // pairs of SMs; the line of tiles * nb units is cut into a range for each, in quanta of
    int quantum;            //   1 unit, or nb of them (then no tile is shared):
    int per_pair, one_more; //   per_pair quanta, and one more for the first one_more pairs
    int split;              // > 1: instead, a cluster of this many pairs per tile, each with a part of K
    uint32_t exchange_bytes;  // then: shared memory for the other pairs' sums
    int acc_sets, a_stages; // tensor memory: accumulator sets of n_inst columns, stages of a converted block
    int x_stages, x_resident, w_stages;  // shared memory: rings; x_resident: every stage of K, loaded once
    int x_steps;
    int x_3d;               // K is a multiple of 64: one copy brings a stage
    uint32_t x_box_bytes;   // 64 k x n_inst / 2 tokens; x_steps (2 or 4) to a stage
    uint32_t smem_bytes;
};

// First unit of a pair's range, and the pair whose range holds a unit (quantum 1).
FDQP_HD inline int st_range_begin(const StreamParams& p, int pair) {
    return (pair * p.per_pair + (pair < p.one_more ? pair : p.one_more)) * p.quantum;
}
FDQP_HD inline int st_owner(const StreamParams& p, int unit) {
    const int big = p.one_more * (p.per_pair + 1);
    return unit < big ? unit / (p.per_pair + 1) : p.one_more + (unit - big) / p.per_pair;
}

// Stages of x that a CTA loads for the units [u0, u1): a stage holds x_steps (2 or 4) of a block's four k-steps; a tile's last block
// may have fewer of them.
FDQP_HD inline int st_x_loads(int u0, int u1, int nb, int x_steps, int ksteps_last) {
    const int n = u1 - u0;
    return x_steps == 4 ? n : 2 * n - (ksteps_last <= 2 ? u1 / nb - u0 / nb : 0);
}
// How often a ring's stage is used, and so released, in `all` loads.  The releases go to both CTAs of the pair; no load waits for the last
// one of a stage, so the kernel does before a CTA leaves: it must not reach the barriers of a successor.  (Not signalling these instead
// cost 0.05 us a launch.)
FDQP_HD inline int st_stage_uses(int stage, int all, int stages) { return all > stage ? (all - stage - 1) / stages + 1 : 0; }

// The barrier (0, 1: of an accumulator set; kStAccLast) that tells that segment idx of a range, its idx-th part of a tile, is in the
// accumulators, and the number of that barrier's phase.  A wait sees a phase's parity only, so its warp has to know the phase
// before to be complete.  Warps that read every segment of a set do.  The last segment is read by the conversion warps, which
// where there are two sets have waited for no other one: it has a barrier of its own, used once.
constexpr int kStAccLast = 2;
struct StAccWait {
    int bar;
    uint32_t phase;
};
FDQP_HD inline StAccWait st_acc_wait(int acc_sets, int idx, bool last) {
    if (last) return {kStAccLast, 0u};
    return acc_sets == 2 ? StAccWait{idx & 1, (uint32_t)idx >> 1} : StAccWait{0, (uint32_t)idx};
}

// ---- a chain of projections in one persistent launch (fdqp_chain.cu) ---------------------------------------------
constexpr int kMaxChainSteps = 160;  // projections one launch walks (a longer chain is cut into several launches)
constexpr int kMaxChainUnits = 240;  // (step, K slice) pairs of one launch
constexpr int kChainEdgeSteps = 64;  // partial-row slots for strips shared between CTAs: two per CTA for this many steps

struct ChainStep {
    const uint8_t* W;          // device, packed Q4NX
    const uint16_t* x;         // device, [M][K] bf16 bits (may be written by the previous step: wait_prev)
    float* y;                  // device, fp32 output [M][N] (epilogue kEpiNone)
    uint16_t* y16;             // device, bf16 output (other epilogues)
    const uint16_t* gamma;     // RMS normalisation of x in the activation preparation (norm != 0)
    const uint16_t* residual;  // with norm: x + residual is what gets normalised ...
    uint16_t* h_out;           // ... and, when not null, is also written here by the grid's first CTA
    float eps;
    int epi, norm;
    int K, N;
    int S;                     // strips = N / 32
    int nb;                    // blocks per strip = ceil(K / 256)
    int Z, nbz;                // K slices and blocks per slice (the prepared x of a slice must fit shared memory)
    int Gz;                    // CTAs per slice (Z * Gz <= grid; the rest of the grid idles during this step)
    int strip_aligned;         // 1: CTA ranges are cut at strip boundaries
    uint32_t B;                // chain-wide cut: position of this step's first block in the chain's block sequence
    int wait_prev;             // 1: the step's input is the previous step's output: wait for all of its strips
    int signal;                // 1: the next step waits on this one: count the stored strips in done[step]
    uint32_t ticket_off;       // this step's arrival counters inside ChainPlan::tickets
    uint32_t edge_off;         // this step's slots inside ChainPlan::ws_edge (2 per CTA) ...
    uint32_t full_off;         // ... and inside ChainPlan::ws_full (Z * S, used when Z > 1)
};

struct ChainPlan {
    int nsteps, M;
    float* ws_edge;            // device, partial rows of strips shared between CTAs
    float* ws_full;            // device, partial rows of whole strip-slices (steps with K slices)
    int* tickets;              // device, arrival counters per (step, strip), zero between launches
    int* done;                 // device, [kMaxChainSteps] strips stored per step, zero between launches
    int* exit_count;           // device, CTAs that have finished (the last one resets `done`)
    int* status;               // host-mapped sticky status word
    int nstage, evict_first;
    int bpw;                   // blocks per consumer warp and ring stage (2 or 4; a stage holds twice as many blocks)
    int has_deps;              // 1: some step waits for the one before it (the completion counters are in use)
    int wide;                  // 1: chain-wide cut into CTA ranges (no step waits for another), 0: every step cut on its own
    uint32_t Wtot;             // chain-wide cut: blocks of all steps together
    int nunits;                // (step, K slice) pairs in processing order
    uint8_t unit_step[kMaxChainUnits], unit_slice[kMaxChainUnits];
    uint32_t off_xs, off_xsum, off_part, off_norm, off_geo, off_bar, smem_bytes;  // shared-memory carve-up (bytes)
    ChainStep step[kMaxChainSteps];
};

}  // namespace fdqp
