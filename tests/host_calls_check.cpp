// Host check of the library's device calls (compiled by tests/test_host_calls.py): api.cpp,
// plan.cpp and tune.cpp linked against a CUDA runtime and kernel launchers of this file.
// Device memory is host memory; a launcher only notes what it was asked for. Modes:
//   pruned    the fill of a pruned call gets the flags of its own tile grid, also when the
//             tuned tile edge changes while the call runs; fill_kernel = 1 gives every k that fill
//   ordering  no kernel is launched on a stream while a write of the default stream, which
//             that stream does not wait for, may still be on its way; host memory that an
//             asynchronous copy reads stays as it is until the copy's stream is waited for;
//             no result is read before that
//   choice    a pruned call's fill: the tile kernel where leaving cells out makes it the faster one
//   tuning    what the autotuner timed decides for the shapes it could time, and for no other
#include <cuda_runtime.h>
#include <malloc.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <string>
#include <vector>

#include "api_internal.h"

using namespace msadp;

static int g_bad = 0;
#define CHECK(cond, ...)                                            \
    do {                                                            \
        if (!(cond)) {                                              \
            printf("line %d: %s: ", __LINE__, #cond);               \
            printf(__VA_ARGS__);                                    \
            printf("\n");                                           \
            ++g_bad;                                                \
        }                                                           \
    } while (0)

// ---------------------------------------------------------------------------
// The runtime.

static float g_ms = 1;            // what events are apart
static int g_default_writes = 0;  // writes of the default stream that nothing has waited for
static bool g_busy = false;       // work on another stream that nothing has waited for
struct Source {
    const char *at;
    std::vector<char> bytes;
};
static std::vector<Source> g_sources;  // host memory of its copies

static void stream_work(const char *what) {
    CHECK(g_default_writes == 0, "%s with %d writes of the default stream on their way", what, g_default_writes);
    g_busy = true;
}
static void wait_streams() {
    for (const Source &s : g_sources)
        CHECK(memcmp(s.at, s.bytes.data(), s.bytes.size()) == 0, "a copy's source changed before the copy was waited for");
    g_sources.clear();
    g_busy = false;
}

extern "C" {
cudaError_t cudaGetDevice(int *d) { return *d = 0, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "error"; }
cudaError_t cudaMalloc(void **p, size_t n) { return (*p = calloc(n + 1, 1)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFree(void *p) { return free(p), cudaSuccess; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return cudaMalloc(p, n); }
cudaError_t cudaFreeHost(void *p) { return cudaFree(p); }
// A copy from pageable memory and a memset may return before the device has them; work on
// a non-blocking stream does not wait for the default stream's (every stream but it here).
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind kind) {
    if (kind == cudaMemcpyDeviceToHost) {
        CHECK(!g_busy, "results read before their stream is done");
        g_default_writes = 0;  // waits for the default stream
    } else {
        ++g_default_writes;
    }
    return memcpy(d, s, n), cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t s) {
    if (s) stream_work("memset");
    else ++g_default_writes;
    if (v || n < (64 << 20)) memset(d, v, n);  // (large ones: zero from calloc, and left to it)
    return cudaSuccess;
}
cudaError_t cudaMemset(void *d, int v, size_t n) { return cudaMemsetAsync(d, v, n, nullptr); }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind kind, cudaStream_t stream) {
    if (!stream) return cudaMemcpy(d, s, n, kind);
    stream_work("copy");
    if (kind == cudaMemcpyHostToDevice && n)
        g_sources.push_back({(const char *)s, std::vector<char>((const char *)s, (const char *)s + n)});
    return memcpy(d, s, n), cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
    if (s) wait_streams();
    else g_default_writes = 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() {
    wait_streams();
    g_default_writes = 0;
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { return *s = (cudaStream_t)0x10, cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { return *e = (cudaEvent_t)0x20, cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return wait_streams(), cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { return *ms = g_ms, cudaSuccess; }
}

// ---------------------------------------------------------------------------
// The kernel launchers.

static PruneDesc g_prune;           // of the last analysis
static double g_left_out = 0;       // share of the cells the analysis rules out
static int g_edge_after_prune = 0;  // tile edge another thread sets once the analysis is enqueued
static int g_tile_fills = 0, g_skipping_fills = 0;
static float g_cost[kKernelCount];  // ms of a fill by kernel, more the further a tile edge is from g_best_edge
static int g_best_edge = 0;

static cudaError_t kernel(cudaStream_t s) {
    if (s) stream_work("kernel");
    return cudaSuccess;
}

namespace msadp {
cudaError_t launch_encode(const ProblemDesc *, int, int, const IODesc *, IODesc, cudaStream_t s, int) { return kernel(s); }
cudaError_t launch_traceback(const ProblemDesc *, int, const int32_t *, const IODesc *, IODesc io, cudaStream_t s) {
    *io.result = msa_device_result{};
    return kernel(s);
}
cudaError_t launch_prune(const PruneDesc &D, bool, cudaStream_t s) {
    g_prune = D;
    double cells = 1;
    for (int i = 0; i < D.k; ++i) cells *= D.len[i] + 1;
    D.stats[1] = (int64_t)(g_left_out * cells);
    if (g_edge_after_prune) set_tile_edge(D.k, g_edge_after_prune);
    return kernel(s);
}
cudaError_t launch_fill_tiles(int k, int edge, const LaunchDesc &L, int, cudaStream_t s) {
    ++g_tile_fills;
    g_ms = g_cost[kKernelTiles] + 0.01f * (float)abs(edge - g_best_edge);
    const ProblemDesc &P = L.probs[0];
    if (P.skip) {
        ++g_skipping_fills;
        CHECK(P.skip == g_prune.skip, "flags of another call");
        CHECK(P.ntiles == g_prune.ntiles && L.ntickets == g_prune.ntiles, "k=%d: %lld tiles filled, flags of %lld", k,
              (long long)P.ntiles, (long long)g_prune.ntiles);
        for (int i = 0; i < k; ++i)
            CHECK(tile_ext(k, edge, i) == g_prune.E[i] && P.E[i] == g_prune.E[i], "k=%d axis %d: extent %d, flags for %d", k, i,
                  P.E[i], g_prune.E[i]);
    }
    return kernel(s);
}
cudaError_t launch_fill_col3(const LaunchDesc &, int, int, cudaStream_t s) { return g_ms = g_cost[kKernelCol3], kernel(s); }
cudaError_t launch_fill_band2(const LaunchDesc &, int, cudaStream_t s) { return g_ms = g_cost[kKernelBand2], kernel(s); }
cudaError_t launch_fill_lines(int, int, const LaunchDesc &, int, cudaStream_t s) { return g_ms = g_cost[kKernelLines], kernel(s); }
cudaError_t launch_fill_stream(int, const LaunchDesc &, int, cudaStream_t s, int) { return g_ms = g_cost[kKernelStream], kernel(s); }
size_t near_optimal_work_bytes(int, int64_t, int32_t) { return 0; }
cudaError_t launch_near_optimal(int, int64_t, const ProblemDesc *, IODesc, int64_t, int32_t, NearOut, cudaStream_t s) { return kernel(s); }
int fill_tiles_ctas_per_sm(int, int) { return 1; }
int fill_tiles_warps_per_cta(int, int) { return 1; }
int fill_col3_ctas_per_sm(int) { return 1; }
int fill_lines_ctas_per_sm(int, int) { return 1; }
int fill_lines_warps_per_cta(int, int) { return 1; }
int fill_stream_ctas_per_sm(int) { return 1; }
int fill_band2_ctas_per_sm() { return 1; }
int fill_band2_warps_per_cta() { return 2; }
int col3_smem_bytes(int) { return 1; }
}  // namespace msadp

// ---------------------------------------------------------------------------

struct Problem {
    int k;
    std::vector<std::string> text;
    std::vector<const char *> seqs;
    std::vector<int32_t> lens, table;
    std::string alphabet;
    Problem(std::vector<int32_t> lens_, int letters) : k((int)lens_.size()), lens(std::move(lens_)) {
        alphabet = std::string("ABCDEFGHIJKLMNOPQRSTUVWXYZ").substr(0, (size_t)letters);
        for (int32_t n : lens) text.push_back(std::string((size_t)n, 'A'));
        for (auto &t : text) seqs.push_back(t.c_str());
        table.assign((size_t)letters * letters, 1);
    }
};

static void pruned() {
    // k = 3 with 25 letters and k = 7, 8 with a long last axis take the tile kernel
    struct { std::vector<int32_t> lens; int letters, edge; } cases[] = {
        {{40, 41, 39}, 25, 8}, {{40, 41, 39}, 25, 16}, {{3, 4, 3, 2, 3, 4, 20}, 4, 3}};
    for (auto &c : cases) {
        Problem p(c.lens, c.letters);
        std::string out((size_t)p.k * 400, '\0');
        int32_t score = 0;
        g_tile_fills = 0;
        g_edge_after_prune = c.edge;
        const int rc = msa_align_pruned(p.k, p.seqs.data(), p.lens.data(), p.alphabet.c_str(), p.table.data(), -1, 0, 0, &score,
                                        &out[0], nullptr);
        CHECK(rc == MSA_OK, "%s", msa_last_error());
        CHECK(g_tile_fills == 1, "%d fills by the tile kernel", g_tile_fills);
        CHECK(tile_edge_for(p.k) == c.edge, "the edge did not change");
        g_edge_after_prune = 0;
        msa_set_tile_edge(p.k, 0);
    }
    for (int k = 2; k <= 8; ++k)
        for (int kernel : {0, 1}) {
            Problem p(std::vector<int32_t>((size_t)k, 4), 4);
            std::string out((size_t)k * 400, '\0');
            int32_t score = 0;
            g_skipping_fills = 0;
            msa_config("fill_kernel", kernel);
            CHECK(msa_align_pruned(k, p.seqs.data(), p.lens.data(), p.alphabet.c_str(), p.table.data(), -1, 0, 0, &score, &out[0],
                                   nullptr) == MSA_OK, "%s", msa_last_error());
            CHECK(g_skipping_fills == kernel, "k=%d: %d fills leave tiles out with fill_kernel = %d", k, g_skipping_fills, kernel);
        }
    msa_config("fill_kernel", 0);
}

static void ordering() {
    mallopt(M_PERTURB, 0xa5);  // freed memory changes at once
    for (int k = 2; k <= 8; ++k) {
        const int n = k == 2 ? 700 : k == 3 ? 40 : k < 6 ? 9 : 4;
        Problem p(std::vector<int32_t>((size_t)k, n), k == 3 ? 20 : 4);
        const int A = (int)p.alphabet.size();
        std::string out((size_t)k * (size_t)(k * n + 1), '\0');
        int32_t score = 0, ncols[4], count = 0, more = 0;
        int64_t scores[4];
        std::vector<uint8_t> masks((size_t)4 * k * n + 16);
        // plans of every kernel, executed on a stream of the caller's
        for (int kernel = 0; kernel <= 5; ++kernel) {
            msa_config("fill_kernel", kernel);
            msa_plan *plan = nullptr;
            CHECK(msa_plan_create(k, p.lens.data(), p.alphabet.c_str(), &plan) == MSA_OK, "%s", msa_last_error());
            msa_device_result res;
            msa_plan_execute(plan, p.seqs[0], p.table.data(), -1, &res, masks.data(), (void *)0x30);
            cudaStreamSynchronize((cudaStream_t)0x30);
            msa_plan_destroy(plan);
        }
        msa_config("fill_kernel", 0);
        CHECK(msa_align(k, p.seqs.data(), p.lens.data(), p.alphabet.c_str(), p.table.data(), -1, &score, &out[0]) == MSA_OK, "%s",
              msa_last_error());
        for (int given = 0; given < 2; ++given)
            CHECK(msa_align_pruned(k, p.seqs.data(), p.lens.data(), p.alphabet.c_str(), p.table.data(), -1, given, -5, &score,
                                   &out[0], nullptr) == MSA_OK, "%s", msa_last_error());
        const std::vector<int32_t> ext((size_t)k, 100);
        std::vector<int64_t> bounds(64);  // at most 7 x 7 tiles
        CHECK(msa_tile_bounds(k, p.seqs.data(), p.lens.data(), p.alphabet.c_str(), p.table.data(), -1, ext.data(),
                              bounds.data()) == MSA_OK, "%s", msa_last_error());
        CHECK(msa_near_optimal(k, p.seqs.data(), p.lens.data(), p.alphabet.c_str(), p.table.data(), -1, 1, 4, masks.data(), ncols,
                               scores, &count, &more) == MSA_OK, "%s", msa_last_error());
        msa_tuning t;
        CHECK(msa_autotune(k, p.lens.data(), A, 1, &t) == MSA_OK, "%s", msa_last_error());
    }
}

// Tunes on `lens` with the tile, line, column and streamed kernels' times, the tile kernel's
// best at `edge`.
static void tune(const std::vector<int32_t> &lens, float tiles, float lines, float column, float stream, int edge) {
    g_cost[kKernelTiles] = tiles;
    g_cost[kKernelLines] = lines;
    g_cost[kKernelCol3] = column;
    g_cost[kKernelStream] = stream;
    g_best_edge = edge;
    msa_tuning t;
    CHECK(msa_autotune((int)lens.size(), lens.data(), 20, 1, &t) == MSA_OK, "%s", msa_last_error());
}
static int chosen(const std::vector<int32_t> &lens, int A = 20) { return choose_kernel((int)lens.size(), lens.data(), A, kKernelAuto); }
static void defaults(int k) {
    msa_set_tile_edge(k, 0);
    msa_set_line_segment(k, 0);
}

static void tuning() {
    for (int k = 7; k <= 8; ++k) {
        std::vector<int32_t> shrt((size_t)k, 3), lng((size_t)k, 2);
        lng.back() = 20;  // beyond the whole-column form
        const int other = tile_edge_candidate(k, 1) > 0 ? tile_edge_candidate(k, 1) : tile_edge_candidate(k, 0);
        tune(lng, 5, 0, 0, 1, other);
        CHECK(chosen(shrt) == kKernelStream && chosen(lng) == kKernelTiles && tile_edge_for(k) == other, "k=%d", k);
        tune(shrt, 5, 0, 0, 1, other);
        CHECK(chosen(shrt) == kKernelStream && chosen(lng) == kKernelTiles && tile_edge_for(k) == other, "k=%d", k);
        tune(shrt, 1, 0, 0, 5, other);
        CHECK(chosen(shrt) == kKernelTiles, "k=%d", k);
        tune(lng, 1, 0, 0, 5, other);  // leaves that choice
        CHECK(chosen(shrt) == kKernelTiles, "k=%d", k);
        defaults(k);
        CHECK(chosen(shrt) == kKernelStream && tile_edge_for(k) == tile_edge_default(k), "k=%d", k);
        msa_set_tile_edge(k, tile_edge_candidate(k, 0));  // an edge of the caller's selects the tile kernel
        CHECK(chosen(shrt) == kKernelTiles, "k=%d", k);
        tune(lng, 5, 0, 0, 1, other);
        CHECK(chosen(shrt) == kKernelTiles, "k=%d", k);
        defaults(k);
    }
    const std::vector<int32_t> s6 = {3, 3, 3, 3, 3, 24}, l6 = {3, 3, 3, 3, 3, 25};
    for (float tiles : {5.f, 1.f}) {  // the last axis beyond the whole-column form, lines or tiles the fastest
        tune(l6, tiles, 2, 0, 3, 3);
        CHECK(chosen(s6) == kKernelStream && chosen(l6) == (tiles > 2 ? kKernelLines : kKernelTiles), "k=6");
        defaults(6);
    }
    tune(l6, 5, 2, 0, 1, 3);
    CHECK(chosen(s6) == kKernelStream && chosen(l6) == kKernelLines, "k=6");
    tune(s6, 5, 1, 0, 2, 3);
    CHECK(chosen(s6) == kKernelLines && chosen(l6) == kKernelLines, "k=6");
    tune(s6, 1, 5, 0, 2, 3);
    CHECK(chosen(s6) == kKernelTiles && chosen(l6) == kKernelTiles, "k=6");
    defaults(6);
    for (int k = 4; k <= 5; ++k) {
        const std::vector<int32_t> lens((size_t)k, 9);
        CHECK(chosen(lens) == kKernelStream, "k=%d", k);
        tune(lens, 5, 1, 0, 2, 4);
        CHECK(chosen(lens) == kKernelLines, "k=%d", k);
        tune(lens, 1, 2, 0, 2, 4);
        CHECK(chosen(lens) == kKernelTiles, "k=%d", k);
        tune(lens, 5, 2, 0, 1, 4);
        CHECK(chosen(lens) == kKernelStream, "k=%d", k);
        defaults(k);
    }
    const std::vector<int32_t> s3 = {9, 9, 9}, l3 = {1, 1, 5000};
    tune(l3, 1, 0, 0, 0, 8);  // a last axis the column kernel does not take
    CHECK(chosen(s3) == kKernelCol3 && chosen(l3) == kKernelTiles && tile_edge_for(3) == 8, "k=3");
    tune(s3, 1, 0, 2, 0, 8);
    CHECK(chosen(s3) == kKernelTiles, "k=3");
    tune(s3, 2, 0, 1, 0, 16);
    CHECK(chosen(s3) == kKernelCol3 && tile_edge_for(3) == 16, "k=3");
    defaults(3);
}

static void choice() {
    // both fills measured in one call, ms: the kernel that fills every cell, the tile kernel
    const struct { std::vector<int32_t> lens; double out; float fast, tiles; } cases[] = {
        {{60, 60, 60, 60}, 0.967, 0.65f, 1.14f},          {{200, 190, 200, 195}, 0.995, 11.4f, 14.2f},
        {{30, 30, 30, 30, 30}, 0.985, 1.08f, 1.36f},      {{40, 40, 40, 40, 40}, 0.987, 2.85f, 2.49f},
        {{40, 40, 40, 40, 40}, 0.356, 2.86f, 3.35f},      {{60, 60, 60, 60, 15}, 0.365, 7.05f, 5.26f},
        {{60, 60, 60, 60, 5}, 0.397, 4.68f, 3.09f},       {{25, 25, 25, 25, 100}, 0.97, 1.21f, 1.84f},
        {{14, 14, 14, 14, 14, 14}, 0.994, 0.86f, 1.05f},  {{20, 20, 20, 20, 20, 20}, 0.988, 3.01f, 2.16f},
        {{24, 24, 24, 24, 24, 24}, 0.699, 6.5f, 7.64f},   {{30, 30, 30, 30, 30, 5}, 0.732, 7.21f, 5.02f},
        {{26, 26, 26, 26, 26, 26}, 0.833, 25.6f, 7.18f},  {{20, 20, 20, 20, 20, 60}, 0.21, 12.4f, 9.62f},
        {{17, 17, 17, 17, 17, 26}, 0.57, 3.15f, 2.07f},   {{10, 10, 10, 10, 10, 60}, 0.452, 1.19f, 1.64f},
        {{12, 12, 12, 12, 12, 12, 12}, 1.0, 3.84f, 5.67f}, {{13, 13, 13, 13, 13, 13, 12}, 0.988, 4.0f, 6.2f},
        {{8, 8, 8, 8, 8, 8, 8, 8}, 0.996, 6.33f, 4.28f},  {{9, 9, 9, 9, 9, 9, 9, 4}, 0.983, 5.3f, 3.77f},
        {{10, 10, 10, 10, 10, 10, 10, 5}, 0.692, 18.3f, 21.f}};
    for (const auto &c : cases) {
        Problem p(c.lens, 4);
        std::string out((size_t)p.k * 1000, '\0');
        int32_t score = 0;
        g_left_out = c.out;
        g_skipping_fills = 0;
        CHECK(msa_align_pruned(p.k, p.seqs.data(), p.lens.data(), p.alphabet.c_str(), p.table.data(), -1, 0, 0, &score, &out[0],
                               nullptr) == MSA_OK, "%s", msa_last_error());
        CHECK(g_skipping_fills == (c.tiles < c.fast), "k=%d, last axis %d, %.3f left out", p.k, c.lens.back(), c.out);
    }
}

int main(int argc, char **argv) {
    const std::string mode = argc > 1 ? argv[1] : "";
    if (mode == "pruned") pruned();
    else if (mode == "ordering") ordering();
    else if (mode == "choice") choice();
    else if (mode == "tuning") tuning();
    else CHECK(false, "unknown mode");
    if (!g_bad) printf("ok\n");
    return g_bad != 0;
}
