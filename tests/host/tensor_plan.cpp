// The library's own plans of prefill-sized calls (fdqp_tensor_plan.h) over a grid of sizes: what the kernel relies on.
#include <cstdio>
#include <cstring>
#include <map>
#include <set>
#include <vector>

#include "fdqp_tensor_plan.h"

using namespace fdqp;

static long failed = 0;

#define CHECK(what)                                                                       \
    do {                                                                                  \
        if (!(what) && ++failed <= 20) std::printf("M %lld K %lld N %lld: %s\n", (long long)M, (long long)K, (long long)N, #what); \
    } while (0)

static TensorSetup b200() {
    TensorSetup s;
    s.sm_count = 148;
    s.smem_optin = 227 * 1024;
    s.pf_ws_bytes = 128u << 20;
    s.st_clusters[0] = 32;
    s.st_clusters[1] = 14;
    return s;
}

// Every unit of work in one range, memory and counters within their bounds, no slot of partial sums used twice.
static void cut(const TensorSetup& setup, int64_t M, int64_t K, int64_t N, int fmt) {
    StreamParams p;
    double us;
    const bool planned = plan_stream(&setup, M, K, N, fmt, &p, &us);
    const int64_t most = setup.p_st_tokens > 0 ? setup.p_st_tokens : kStMaxTokens;
    CHECK(planned || (N + 255) / 256 * ((M + most - 1) / most + 1) * ((K + 255) / 256) > 1 << 24);  // (more units than it counts)
    if (failed || !planned) return;
    CHECK(p.n_inst % 16 == 0 && p.n_inst <= kStMaxTokens && (int64_t)p.n_inst * p.tok_tiles >= M && (int64_t)p.n_inst * (p.tok_tiles - 1) < M);
    CHECK(p.nb == (K + 255) / 256 && p.tiles == (N + 255) / 256 * p.tok_tiles);
    CHECK(p.acc_sets * p.n_inst + 128 * p.a_stages <= 512);
    CHECK(p.a_stages >= 2 && p.a_stages <= 3 && p.w_stages >= kStMinW && p.w_stages <= kStMaxW);
    CHECK(p.x_resident ? p.x_steps == 4 && p.x_stages == p.nb && p.tok_tiles == 1 : p.x_stages >= 2);
    CHECK(p.x_stages <= kStMaxX);
    CHECK((int64_t)p.smem_bytes <= setup.smem_optin);
    CHECK((int64_t)p.smem_bytes == 1024 + kStBarBytes + p.exchange_bytes + (int64_t)p.x_stages * (p.x_steps * p.x_box_bytes + 16) + (int64_t)p.w_stages * 4 * fmt_block_bytes(fmt));
    if (p.split > 1) {  // a cluster to a tile, a part of K to each of its pairs
        CHECK(p.pairs == p.tiles * p.split && p.pairs <= setup.sm_count / 2 && p.tok_tiles == 1 && p.nb >= p.split && kStParts % p.split == 0);
        return;
    }
    CHECK(p.pairs >= 1 && p.pairs <= setup.sm_count / 2 && p.per_pair >= 1 && (p.quantum == 1 || p.quantum == p.nb));
    if (failed) return;
    CHECK(st_range_begin(p, 0) == 0 && st_range_begin(p, p.pairs) == p.tiles * p.nb);
    std::map<int, int> slots;
    for (int r = 0; r < p.pairs; ++r) {
        const int u0 = st_range_begin(p, r), u1 = st_range_begin(p, r + 1);
        CHECK(u0 < u1);
        for (int u = u0; u < u1;) {
            const int tile = u / p.nb, end = u1 < (tile + 1) * p.nb ? u1 : (tile + 1) * p.nb;
            if (u != tile * p.nb || end != (tile + 1) * p.nb) {
                CHECK(p.quantum == 1 && st_owner(p, u) == r && st_owner(p, end - 1) == r);
                CHECK(slots.emplace(2 * r + (u0 >= tile * p.nb ? 0 : 1), tile).second);
            }
            u = end;
        }
    }
    if (slots.empty()) return;
    CHECK((size_t)p.pairs * 2 * 8 * p.n_inst * kStripRows * 4 <= setup.pf_ws_bytes);
    std::map<int, std::vector<int>> of_tile;
    for (const auto& s : slots) of_tile[s.second].push_back(s.first);  // (in order of the slots, so of the pairs)
    std::set<int> counters;
    for (const auto& t : of_tile) {
        const int p0 = st_owner(p, t.first * p.nb), p1 = st_owner(p, (t.first + 1) * p.nb - 1);
        CHECK(p0 < p1 && counters.insert(p0).second);  // the first pair's counters serve one tile
        // what the last arriver reads: the first pair's slot by where its range begins, the others' first ones
        std::vector<int> read;
        for (int r = p0; r <= p1; ++r) read.push_back(2 * r + (r == p0 && st_range_begin(p, p0) < t.first * p.nb ? 1 : 0));
        CHECK(read == t.second);
    }
}

static void cuts() {
    const int64_t Ks[] = {32, 256, 288, 544, 768, 1152, 2560, 3840, 5376, 6912, 10240, 15360, 21504};
    const int64_t Ns[] = {32, 64, 256, 288, 1024, 2560, 4096, 5376, 10240, 18944, 19200, 20480, 37888, 40960, 262144};
    const int64_t Ms[] = {9, 16, 17, 37, 48, 64, 65, 96, 97, 112, 128, 129, 144, 200, 208, 256, 257, 300, 511, 512, 1000, 4096};
    for (int64_t K : Ks)
        for (int64_t N : Ns)
            for (int64_t M : Ms) {
                TensorSetup s = b200();
                cut(s, M, K, N, kFmtQ4nx);
                if (K % kBlockK == 0) cut(s, M, K, N, kFmtMxfp4);
                for (int64_t blocks : {(int64_t)1, (int64_t)2, (int64_t)3, (int64_t)7, (int64_t)17, (int64_t)1000000, INT64_MAX - 3, INT64_MAX}) {
                    s.p_st_blocks = blocks;
                    cut(s, M, K, N, kFmtQ4nx);
                }
                s = b200();
                for (int64_t tokens : {16, 112, 256}) {
                    s.p_st_tokens = tokens;
                    cut(s, M, K, N, kFmtQ4nx);
                }
                for (int cluster = 0; cluster < 2; ++cluster) {
                    s = b200();
                    s.p_st_cluster = cluster;
                    cut(s, M, K, N, kFmtQ4nx);
                }
                s = b200();
                s.pf_ws_bytes = 1 << 20;  // little room for partial sums
                cut(s, M, K, N, kFmtQ4nx);
            }
}

// Calls whose weights would lose accuracy in bf16 and that the GEMV kernels serve about as fast as the tile kernels; and such that
// those serve faster.  MXFP4 weights lose nothing.
static void routes() {
    const struct { int64_t K, N, M; bool tensor, tensor_mx; } calls[] = {
        {6912, 32, 9, false, true}, {6912, 256, 9, false, true}, {10240, 128, 12, false, true}, {15360, 1024, 9, false, true}, {15360, 1024, 10, false, true},
        {21504, 1024, 9, false, true}, {21504, 1024, 16, false, true}, {21504, 1536, 9, false, true}, {21504, 1536, 10, false, true},
        {2560, 2560, 9, true, true}, {10240, 2560, 9, true, true}, {21504, 1024, 32, true, true}, {6912, 1152, 24, true, true}, {256, 4096, 512, true, true}};
    for (const auto& c : calls)
        for (int fmt : {kFmtQ4nx, kFmtG64, kFmtG128, kFmtMxfp4}) {
            const int64_t M = c.M, K = c.K, N = c.N;
            TensorSetup s = b200();
            CHECK(use_prefill(&s, M, K, N, fmt) == (fmt == kFmtMxfp4 ? c.tensor_mx : c.tensor));
            s.p_path = 2;
            CHECK(!use_prefill(&s, M, K, N, fmt));
            s.p_path = 3;
            CHECK(use_prefill(&s, M, K, N, fmt));
        }
}

// A context's workspace holds the partial sums of each of its calls, and is no larger than its largest calls can need.
static void workspaces() {
    const int64_t contexts[][3] = {{9, 2560, 64}, {16, 1152, 6912}, {40, 10240, 32}, {48, 21504, 5376}, {128, 512, 256}, {200, 3840, 30720}, {300, 1056, 288},
                                   {300, 256, 288}, {512, 21504, 262144}, {2000, 768, 1024}};
    for (const auto& c : contexts) {
        const int64_t M = c[0], K = c[1], N = c[2];
        TensorSetup roomy = b200(), own = roomy;
        own.pf_ws_bytes = stream_ws_bytes(roomy.sm_count, M, K, N);
        // no more pairs than units of work at the most token tiles (16 rows each) or SMs, no larger tiles than the largest
        const int64_t units = (N + 255) / 256 * ((K + 255) / 256) * ((M + 15) / 16), sms = roomy.sm_count / 2, rows = (M + 15) / 16 * 16;
        CHECK(own.pf_ws_bytes <= (size_t)(units < sms ? units : sms) * 2 * 8 * 32 * 4 * (size_t)(rows < 256 ? rows : 256));
        for (int64_t m = M; m > kMaxTokens; m = m * 7 / 8)
            for (int64_t k = K; k > 0; k = k * 3 / 4 / 32 * 32)
                for (int64_t n = N; n > 0; n = n * 2 / 3 / 32 * 32)
                    for (int64_t tokens : {-1, 16, 64}) {
                        roomy.p_st_tokens = own.p_st_tokens = tokens;
                        StreamParams a, b;
                        double us;
                        const bool planned = plan_stream(&roomy, m, k, n, kFmtQ4nx, &a, &us);
                        CHECK(plan_stream(&own, m, k, n, kFmtQ4nx, &b, &us) == planned && !std::memcmp(&a, &b, sizeof a));
                    }
    }
    const int64_t M = 300, K = 1056, N = 288;  // ten units to a token tile
    CHECK(stream_ws_bytes(148, M, K, N) <= 8 << 20);
}

// The parameters that ask for the tile kernels do so.
static void tile_kernels() {
    const int64_t K = 2560, N = 4096;
    for (int64_t M : {9, 64, 128, 129, 512}) {
        StreamParams p;
        double us;
        TensorSetup s = b200();
        CHECK(plan_stream(&s, M, K, N, kFmtQ4nx, &p, &us));
        for (int64_t v : {0, 1}) {
            s.p_pair = v;
            CHECK(!plan_stream(&s, M, K, N, kFmtQ4nx, &p, &us));
        }
        s = b200();
        s.p_pf_split = 1;
        CHECK(!plan_stream(&s, M, K, N, kFmtQ4nx, &p, &us));
        for (int64_t v : {0, 2}) {  // (a form of the one-SM kernel up to 128 rows)
            s = b200();
            s.p_atmem = v;
            CHECK(plan_stream(&s, M, K, N, kFmtQ4nx, &p, &us) == (M > 128));
        }
    }
}

int main(int argc, char** argv) {
    const char* what = argc > 1 ? argv[1] : "";
    if (!std::strcmp(what, "cuts")) cuts();
    else if (!std::strcmp(what, "routes")) routes();
    else if (!std::strcmp(what, "tile_kernels")) tile_kernels();
    else if (!std::strcmp(what, "workspaces")) workspaces();
    else return 2;
    std::printf("%ld wrong\n", failed);
    return failed ? 1 : 0;
}
