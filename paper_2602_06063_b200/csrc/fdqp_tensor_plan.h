// Which kernels a call of nine and more token rows takes, and the tensor-core kernels' plans: estimates of time and cuts of the
// work, on plain values.
#pragma once
#include <stddef.h>
#include <stdint.h>

#include <cstring>

#include "fdqp_format.h"
#include "fdqp_plan.h"

namespace fdqp {

// What the choice depends on beside a call's sizes: the device, the context's workspace, and launch parameters (-1 = automatic).
struct TensorSetup {
    int sm_count = 0;
    int smem_optin = 0;
    size_t pf_ws_bytes = 0;        // for partial results (0: no tensor-core kernels)
    int st_clusters[2] = {0, 0};   // streaming kernel: clusters of 2 and of 4 pairs that fit the device at once
    int64_t p_path = -1, p_pair = -1, p_pf_split = -1;
    int64_t p_atmem = 1;           // tile kernel up to 128 tokens: keep the converted weights in tensor memory
    int64_t p_st_tokens = -1, p_st_blocks = -1, p_st_cluster = -1;  // streaming kernel: most tokens of a tile, blocks of a pair, clusters
};

// Measured on B200: while all of x is smaller than 128 KB, the tensor-core kernels (every CTA re-reads the same few rows
// of x by TMA at every k-step) run 1.45x slower; with the same rows placed further apart, so that they cover at least
// 256 KB of addresses, the slow-down is gone.  Such an x is therefore copied into a spread-out staging buffer first.
constexpr int64_t kSpreadBelowBytes = 128 << 10;
constexpr int64_t kPrefillMinK = 256;          // shortest reduction the dispatch gives to the tensor-core kernels

// More than 256 token rows: a pair of SMs works on a 256 x 512 tile (every converted weight serves 512 tokens).
inline bool use_pair(const TensorSetup* ctx, int64_t M) { return ctx->p_pair >= 0 ? ctx->p_pair != 0 : M > 256; }

// Time model of a tensor-core call cut into Z K slices (microseconds, without the launch and the optional spreading
// copy; constants measured on B200).  A CTA (pair) costs about c per 64-wide k-step when its SM is full: c = 0.64 up to
// 64 tokens rising to 0.72 at 128 (128-row tiles, two CTAs per SM), 0.78 (256-row tiles, one CTA per SM), 0.95 (two-SM
// kernel).  The busiest SM runs n = ceil(CTAs / SMs) of them, two at a time where two fit; a CTA that has the SM to
// itself runs its k-steps in about 0.7 of that time.  Z > 1 adds the second kernel (2-3 us on the stream: it overlaps the first one's tail) and the partial results:
// written by the slices, read and summed by the second kernel.
inline double prefill_time_model(const TensorSetup* ctx, int64_t M, int64_t K, int64_t N, int64_t Z) {
    const bool pair = use_pair(ctx, M);
    const bool small = !pair && M <= 128;
    const int64_t tiles = pair ? ((N + 255) / 256) * ((M + 511) / 512)
                               : (small ? (N + 127) / 128 : ((N + 255) / 256) * ((M + 255) / 256));
    const int64_t units = pair ? ctx->sm_count / 2 : ctx->sm_count;
    const int64_t n = (tiles * Z + units - 1) / units;
    const double rounds = small ? (double)(n / 2) + ((n & 1) ? 0.7 : 0.0) : (double)n;
    const double c = pair ? 0.95 : (M <= 64 ? 0.64 : (M <= 128 ? 0.64 + 0.08 * (double)(M - 64) / 64.0 : 0.78));
    const int64_t kz = ((K + 63) / 64 + Z - 1) / Z;
    double t = rounds * (double)kz * c;
    if (Z > 1) t += 2.5 + (double)(2 * Z + 1) * (double)M * (double)N * 4.0 / 5.0e6;
    return t;
}

// K slices of a tensor-core call: the count the time model likes best (a larger count has to win by 8 %), while every
// slice keeps at least eight 64-wide k-steps and the partial results fit the context's workspace.  Few tiles (27B down:
// 42 of 128 rows) get as many slices as fill the SMs once; a tile count just above a multiple of the slots (12B-like
// K = 5376, N = 43008 at M = 32: 336 CTAs on 296 slots) gets the slices that even out the last round (85 -> 70 us).
inline int prefill_slices(const TensorSetup* ctx, int64_t M, int64_t K, int64_t N) {
    const int64_t ksteps = (K + 63) / 64;
    int64_t zmax = kMaxSplit;
    if (zmax > ksteps / 8) zmax = ksteps / 8;
    const int64_t fit = (int64_t)(ctx->pf_ws_bytes / ((size_t)M * (size_t)N * 4));
    if (zmax > fit) zmax = fit;
    if (zmax < 1) zmax = 1;
    if (ctx->p_pf_split > 0) return (int)(ctx->p_pf_split < zmax ? ctx->p_pf_split : zmax);
    int64_t best = 1;
    double t_best = prefill_time_model(ctx, M, K, N, 1);
    for (int64_t Z = 2; Z <= zmax; ++Z) {
        const double t = prefill_time_model(ctx, M, K, N, Z);
        if (t < 0.95 * t_best) {
            best = Z;
            t_best = t;
        }
    }
    return (int)best;
}

// Up to 128 tokens the one-SM kernel keeps the converted weights in tensor memory (mode 1, two CTAs per SM).  Up to 64
// tokens a variant with half the accumulator columns, two weight stages and a four-deep weight prefetch (64 registers)
// fits three CTAs per SM (mode 2): 6 % faster when the call has at least three CTAs per SM to run (LM head 181 -> 170 us),
// slower when it has not (12B gate|up at M = 32: 44 -> 47 us), so the automatic choice asks for that many.
inline int prefill_tmem_mode(const TensorSetup* ctx, int64_t M, int64_t K, int64_t N) {
    if (ctx->p_atmem != 1) return (int)ctx->p_atmem;
    if (M > 64) return 1;
    const int64_t ctas = ((N + 127) / 128) * prefill_slices(ctx, M, K, N);
    return ctas >= 3 * (int64_t)ctx->sm_count ? 2 : 1;
}

// ---- the streaming tensor-core kernel (fdqp_prefill_stream.cu) ----------------------------------------------------------
// Time of one unit (a block of 256 k of a tile of 256 output features x n tokens) on a pair of SMs, us.  Measured on B200: up to
// about 48 tokens the conversion of the weights sets the pace (K = 2560, N = 262144: 0.63 at 16 tokens, 0.70 at 48), then
// conversion and x together (0.80 at 64, 1.05 at 128), then the MMAs (1.4 at 208, 1.7 at 256).
inline double stream_unit_us(int n) { return n <= 128 ? 0.58 + 0.0035 * n : 1.03 + 0.0052 * (n - 128); }

// What a launch loses when its CTAs have to wait for those of the launch before it, one to an SM: those of a launch on half of the
// SMs or fewer find an SM, and have their barriers, tensor memory and first weights when the one before has ended.
inline double stream_crowd_us(int64_t pairs) { return pairs <= 37 ? 0.0 : (pairs <= 50 ? 0.8 : 1.6); }

// One way to cut a call: token tiles, and the range of units of a pair.
struct StreamCut {
    int64_t tok_tiles, per, pairs;  // per: units of the busiest pair
    bool aligned;                   // ranges of whole tiles
    int split;                      // pairs of a cluster that share a tile (1: ranges)
    double us;
};

// per: units wanted for a pair; whole tiles when it is a multiple of nb.
inline StreamCut stream_cut(int64_t M, int64_t nb, int64_t N, int64_t tok_tiles, int64_t per) {
    const int64_t n = ((M + tok_tiles - 1) / tok_tiles + 15) / 16 * 16;
    const int64_t units = (N + 255) / 256 * tok_tiles * nb;
    StreamCut c{tok_tiles, per, (units + per - 1) / per, per % nb == 0, 1, 0.0};
    c.us = (double)per * stream_unit_us((int)n);
    // More than 128 tokens: one set of accumulators, so the pair's MMAs wait while a tile is read out (about 2 us).
    const double reads = (double)((per + nb - 1) / nb);
    if (n > 128) c.us += 2.0 * (reads > 1 ? reads - 1 : 0);
    c.us += stream_crowd_us(c.pairs);
    if (c.aligned) {
        c.us += 0.004 * (double)n - 0.9;
    } else {
        // Tiles shared between pairs: partial sums out, a counter, and back in, by the piece; a range that begins in one tile and
        // ends in another leaves two.  Measured at 37 tokens (us beyond 0.7 a unit and 3 for the launch): K = 10240, N = 2560
        // 0.1 for 2 pieces, 2.1 for 4, 2.7 for 5, 4.6 for 7 or 8 with two to a range; K = 2560, N = 4096 1.1 for 2, 4.0 for 4 or 5.
        const bool even = nb % per == 0;
        const double pieces = (double)(even ? nb / per : nb / per + 2);
        // At 200 tokens K = 2560, N = 4096 4.2 for 2 pieces, 10.5 for 4 or 5.
        c.us += 0.2 + (0.12 + 0.0055 * (double)n) * pieces + (even ? 0.0 : 0.8) + 0.009 * (double)n;
    }
    return c;
}

// k-steps of x per stage: a block, so that the MMA issuer waits once per block; half of one where that would leave too few stages.
inline int64_t stream_x_steps(int64_t n) { return n <= 96 ? 4 : 2; }
inline int64_t stream_room(const TensorSetup* ctx) { return ctx->smem_optin - 1024 - kStBarBytes; }
// Shared memory in which a CTA receives the sums of its cluster's other pairs: its strips' parts, 2 KB per 16 tokens and piece.
inline int64_t stream_exchange_bytes(int64_t n, int split) {
    return split == 1 ? 0 : 128 + 4 * (kStParts / split) * (int64_t)(split - 1) * 2048 * ((n + 16 * kStParts - 1) / (16 * kStParts));
}

// Partial sums of one pair of SMs: of the tile that its range begins in and of one that it shares with the next pair.
inline size_t stream_slot_bytes(int64_t n) { return (size_t)2 * 8 * (size_t)n * kStripRows * 4; }
// Workspace with which every call of a context has room for its partial sums: no more pairs work than there are units, and a call of
// more token tiles has smaller ones.
inline size_t stream_ws_bytes(int sm_count, int64_t max_M, int64_t max_K, int64_t max_N) {
    const int64_t sms = sm_count / 2, units = (max_N + 255) / 256 * ((max_K + kBlockK - 1) / kBlockK);  // of one token tile
    size_t most = 0;
    for (int64_t tt = 1; tt <= (max_M + 15) / 16; ++tt) {
        const int64_t rows = ((max_M + tt - 1) / tt + 15) / 16 * 16, n = rows < kStMaxTokens ? rows : kStMaxTokens;
        const size_t bytes = (size_t)(units * tt < sms ? units * tt : sms) * stream_slot_bytes(n);
        if (most < bytes) most = bytes;
        if (units * tt >= sms) break;
    }
    return most;
}

// False: a launch parameter asks for one of the tile kernels, or the sizes are beyond this one's.
inline bool plan_stream(const TensorSetup* ctx, int64_t M, int64_t K, int64_t N, int fmt, StreamParams* p, double* us) {
    if (ctx->p_pair >= 0 || ctx->p_pf_split > 0 || (ctx->p_atmem != 1 && M <= 128) || !ctx->pf_ws_bytes) return false;
    const int64_t nb = (K + kBlockK - 1) / kBlockK, sms = ctx->sm_count / 2;
    const int64_t most = ctx->p_st_tokens > 0 ? ctx->p_st_tokens : kStMaxTokens;
    const int64_t fewest = (M + most - 1) / most;
    if (sms < 1 || (N + 255) / 256 * (fewest + 1) * nb > (int64_t)1 << 24) return false;
    StreamCut best{};
    for (int64_t tt = fewest; tt <= fewest + (M > 128 && ctx->p_st_tokens < 0 ? 1 : 0); ++tt) {
        const int64_t n = ((M + tt - 1) / tt + 15) / 16 * 16, units = (N + 255) / 256 * tt * nb;
        if (tt > fewest && (tt - 1) * n >= M) continue;  // (rounded up to 16, a tile fewer holds every token)
        const int64_t least = (units + sms - 1) / sms, whole = ((N + 255) / 256 * tt + sms - 1) / sms * nb;  // fewest units, whole tiles
        auto consider = [&](int64_t per) {
            const StreamCut c = stream_cut(M, nb, N, tt, per);
            if (!c.aligned && (size_t)c.pairs * stream_slot_bytes(n) > ctx->pf_ws_bytes) return;  // partial sums do not fit
            if (!best.tok_tiles || c.us < best.us) best = c;
        };
        if (ctx->p_st_blocks > 0) {
            const int64_t wanted = ctx->p_st_blocks < units ? ctx->p_st_blocks : units;  // (more than there are: one pair)
            consider(wanted > least ? wanted : least);
            if (!best.tok_tiles) consider(whole);
            continue;
        }
        // Few tiles: a cluster of two or four pairs for each, which add their sums through shared memory.
        for (int i = 1; i < 3; ++i) {
            const int64_t tiles = (N + 255) / 256 * tt, split = (int64_t)1 << i;
            if (tiles * split > sms || tiles > ctx->st_clusters[i - 1] || nb < split || tt > 1) continue;
            // (beside the exchange: the fewest stages of packed weights, and two of x)
            if (stream_exchange_bytes(n, (int)split) + kStMinW * 4 * (int64_t)fmt_block_bytes(fmt) + 2 * (stream_x_steps(n) * n * 64 + 16) > stream_room(ctx)) continue;
            StreamCut c{tt, (nb + split - 1) / split, tiles * split, false, (int)split, 0.0};
            // (measured as above: two pairs 0.1 at 48 tokens, 1.2 at 128, 2.6 when 32 clusters fill the device; four 1.4 and 3.3)
            c.us = (double)c.per * stream_unit_us((int)n) + (split == 2 ? -0.2 : 0.5) + 0.008 * (double)n + 1.5 * stream_crowd_us(c.pairs);
            if (ctx->p_st_cluster != 0 && (!best.tok_tiles || c.us < best.us)) best = c;
        }
        if (ctx->p_st_cluster == 1 && best.split > 1) continue;
        consider(whole);
        for (int64_t per = least; per < least + 64 && per < 2 * least + nb && per <= units; ++per) consider(per);
    }
    *us = best.us;
    std::memset(p, 0, sizeof(*p));
    p->M = (int)M;
    p->K = (int)K;
    p->N = (int)N;
    p->nb = (int)nb;
    p->tok_tiles = (int)best.tok_tiles;
    p->n_inst = (int)(((M + best.tok_tiles - 1) / best.tok_tiles + 15) / 16 * 16);
    p->tiles = (int)((N + 255) / 256 * best.tok_tiles);
    const int64_t quanta = best.aligned ? p->tiles : (int64_t)p->tiles * nb;
    p->quantum = (int)(best.aligned ? nb : 1);
    p->pairs = (int)best.pairs;
    p->split = best.split;
    p->exchange_bytes = (uint32_t)stream_exchange_bytes(p->n_inst, p->split);
    p->per_pair = (int)(quanta / best.pairs);
    p->one_more = (int)(quanta % best.pairs);
    // tensor memory: n_inst columns per set of accumulators, 128 per stage of converted weights
    p->acc_sets = p->n_inst <= 128 ? 2 : 1;
    p->a_stages = p->n_inst <= 64 ? 3 : 2;
    // shared memory: x once and for all where it fits beside four blocks of weights, else rings of both
    const int64_t x_steps = stream_x_steps(p->n_inst);
    const int64_t w_stage = 4 * (int64_t)fmt_block_bytes(fmt), x_box = (int64_t)p->n_inst / 2 * 128, x_stage = x_steps * x_box + 16;
    const int64_t room = stream_room(ctx) - (int64_t)p->exchange_bytes;
    p->x_steps = (int)x_steps;
    p->x_box_bytes = (uint32_t)x_box;
    p->x_3d = K % 64 == 0;
    p->x_stages = (int)((K + 64 * x_steps - 1) / (64 * x_steps));
    p->x_resident = best.tok_tiles == 1 && x_steps == 4 && p->x_stages <= kStMaxX && p->x_stages * x_stage + kStMinW * w_stage <= room;
    if (!p->x_resident) {
        p->x_stages = (int)((room - kStMinW * w_stage) / x_stage);
        if (p->x_stages > 12) p->x_stages = 12;
    }
    p->w_stages = (int)((room - p->x_stages * x_stage) / w_stage);
    if (p->w_stages > kStMaxW) p->w_stages = kStMaxW;
    p->smem_bytes = (uint32_t)(1024 + kStBarBytes + p->exchange_bytes + p->x_stages * x_stage + p->w_stages * w_stage);
    return (p->x_resident || p->x_stages >= 2) && p->w_stages >= kStMinW;
}

// M >= 9: the tensor-core kernels, or the GEMV kernel eight token rows at a time, by a small cost model (microseconds, constants
// measured on B200).
//   GEMV: every chunk streams the whole matrix, at about 5.5 TB/s for 1-2 rows, 3.9 for 3-4, 3.2 for 5-8, plus ~8 us
//   (back-to-back chunks of a small matrix: 2 x 15 us for 16 MB).
//   Tensor-core kernels: where their rounding of the weights to bf16 costs accuracy (1.5e-3 of y against 1e-7), prefill_time_model:
//   the line lies where the tile kernels overtake the GEMV chunks, and a faster tensor-core kernel does not move it, so that no call
//   loses accuracy to one.  (K = 21504, N = 1024, M = 9 / 16: 21.8 / 21.0 us, 19.9 / 24.6 by tiles, 11.5 / 11.6 by the streaming
//   kernel, which "path" = 3 gives every call to.)  MXFP4 weights are bf16 numbers: there the streaming kernel's own estimate decides
//   (the same sizes: 1.5e-7 against 0.75e-7, the fp32 sums').
inline bool use_prefill(const TensorSetup* ctx, int64_t M, int64_t K, int64_t N, int fmt = kFmtQ4nx) {
    if (M <= kMaxTokens || ctx->p_path == 2) return false;
    if (ctx->p_path == 3) return true;
    // The tensor-core kernels multiply by bf16-rounded weights (relative error up to 2^-8 per weight).  Against the
    // acceptance bound 2e-3 * sum|x w| that is safe only where the K terms' rounding errors average out: with K = 32 two
    // of 40,000 outputs were seen just outside it.  Short reductions therefore stay on the GEMV kernels (fp32 weights).
    if (K < kPrefillMinK) return false;
    const double mb = 0.625 * (double)K * (double)N / 1.0e6;  // packed weights, bytes per microsecond = TB/s * 1e6
    const int64_t last = M % kMaxTokens;                       // rows of the ragged last chunk (0: none)
    const double last_rate = last <= 2 ? 5.5 : (last <= 4 ? 3.9 : 3.2);
    const double t_gemv = (double)(M / kMaxTokens) * (8.0 + mb / 3.2) + (last ? 8.0 + mb / last_rate : 0.0);
    StreamParams stream;
    double t_stream;
    if (fmt == kFmtMxfp4 && plan_stream(ctx, M, K, N, fmt, &stream, &t_stream)) return 3.5 + t_stream < t_gemv;
    double t_tensor = 5.0 + prefill_time_model(ctx, M, K, N, prefill_slices(ctx, M, K, N));
    if (prefill_tmem_mode(ctx, M, K, N) == 2) t_tensor *= 0.94;  // three CTAs per SM
    if (M * K * 2 < kSpreadBelowBytes) t_tensor += 3.0;                                   // the spreading copy
    return t_tensor < t_gemv;
}

}  // namespace fdqp
