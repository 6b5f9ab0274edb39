// Autotuner of the FP32 pass schedules (radix split and tile of P1-P5 of
// the mixed CG iteration), per grid size. Not part of the paper's method:
// it picks, by timing, among the schedule variants of schedule.cuh, all of
// which compute the same transforms.
//
// The choice is process-wide per grid size, kept in a small table that
// run_pass consults for the tuned pass kinds; the CUDA graph of a handle
// keeps the kernels it captured, so schedules are set before the handles
// that should use them are created. Tuned choices are kept in a text cache
// file keyed by device, grid size and library build, so a grid is timed
// once per machine.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cerrno>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <string>
#include <sys/stat.h>
#include <vector>

#include "../../include/fftg.h"
#include "host_common.h"
#include "schedule.cuh"

#ifndef FFTG_BUILD_ID
#define FFTG_BUILD_ID "dev"
#endif

namespace fftg {

#define FFTG_EXTERN_N(n)                                                                                \
    extern template cudaError_t run_variant_n<n>(int, int, const PassArgs&, int, cudaStream_t);        \
    extern template VariantShape variant_shape_n<n>(int, int);                                          \
    extern template cudaError_t run_pass_n<n>(PassKind, const PassArgs&, int, cudaStream_t);
FFTG_EXTERN_N(3)
FFTG_EXTERN_N(5)
FFTG_EXTERN_N(9)
FFTG_EXTERN_N(15)
FFTG_EXTERN_N(25)
FFTG_EXTERN_N(27)
FFTG_EXTERN_N(45)
FFTG_EXTERN_N(75)
FFTG_EXTERN_N(81)
FFTG_EXTERN_N(125)
FFTG_EXTERN_N(135)
FFTG_EXTERN_N(225)
FFTG_EXTERN_N(243)
#undef FFTG_EXTERN_N

namespace {

constexpr int kGrids[] = {3, 5, 9, 15, 25, 27, 45, 75, 81, 125, 135, 225, 243};
constexpr int kNumGrids = sizeof(kGrids) / sizeof(kGrids[0]);
std::atomic<int> g_sched[kNumGrids][TK_COUNT];

int grid_index(int N) {
    for (int i = 0; i < kNumGrids; ++i)
        if (kGrids[i] == N) return i;
    return -1;
}

// pass kinds of each tuned kind (the default launch of variant 0)
constexpr PassKind kDefaultKind[TK_COUNT] = {PK_ROWS_CG_F32, PK_P2_F32, PK_P3_F32, PK_P4_F32, PK_P5_USER_F32};
const char* const kTkName[TK_COUNT] = {"p1", "p2", "p3", "p4", "p5"};

std::mutex g_cache_mu;

std::string cache_path() {
    const char* p = std::getenv("FFTG_SCHEDULE_CACHE");
    if (p && *p) return p;
    const char* x = std::getenv("XDG_CACHE_HOME");
    std::string dir;
    if (x && *x) {
        dir = std::string(x) + "/fftg";
    } else {
        const char* home = std::getenv("HOME");
        if (!home || !*home) return "";
        mkdir((std::string(home) + "/.cache").c_str(), 0755);
        dir = std::string(home) + "/.cache/fftg";
    }
    mkdir(dir.c_str(), 0755);
    return dir + "/schedules.txt";
}

std::string cache_key(int N, int tk) {
    cudaDeviceProp prop{};
    int dev = 0;
    cudaGetDevice(&dev);
    cudaGetDeviceProperties(&prop, dev);
    std::string name = prop.name;
    std::replace(name.begin(), name.end(), ' ', '_');
    return name + " " + std::to_string(N) + " " + FFTG_BUILD_ID + " " + kTkName[tk];
}

// Variant recorded for (N, tk) in the cache, or -1.
int cache_lookup(const std::string& path, const std::string& key) {
    FILE* f = std::fopen(path.c_str(), "r");
    if (!f) return -1;
    char line[512];
    int found = -1;
    while (std::fgets(line, sizeof line, f)) {
        const size_t n = key.size();
        if (std::strncmp(line, key.c_str(), n) == 0 && line[n] == ' ') {
            const int v = std::atoi(line + n + 1);
            if (v >= 0 && v < kVariants) found = v;  // the last entry wins
        }
    }
    std::fclose(f);
    return found;
}

void cache_store(const std::string& path, const std::string& key, int v) {
    FILE* f = std::fopen(path.c_str(), "a");
    if (!f) return;
    std::fprintf(f, "%s %d\n", key.c_str(), v);
    std::fclose(f);
}

cudaError_t launch_schedule(int N, int tk, int v, const PassArgs& a, cudaStream_t s) {
    if (v > 0) return run_variant(N, tk, v, a, 1, s);
    switch (N) {
#define FFTG_CASE(n) case n: return run_pass_n<n>(kDefaultKind[tk], a, 1, s);
        FFTG_CASE(3) FFTG_CASE(5) FFTG_CASE(9) FFTG_CASE(15) FFTG_CASE(25) FFTG_CASE(27)
        FFTG_CASE(45) FFTG_CASE(75) FFTG_CASE(81) FFTG_CASE(125) FFTG_CASE(135) FFTG_CASE(225)
        FFTG_CASE(243)
#undef FFTG_CASE
        default: return cudaErrorInvalidValue;
    }
}

struct DeviceBuffer {
    void* p = nullptr;
    ~DeviceBuffer() {
        if (p) cudaFree(p);
    }
};

// Times every variant of every tuned kind on one field of scratch data and
// keeps the fastest (median of `reps` launches, each bracketed by events).
int tune(int N, cudaStream_t s, int reps, double* ms_out, int* chosen) {
    const size_t cs = (size_t)comp_stride(N);
    const size_t HP = (size_t)spec_pitch(N);
    const size_t field = 6 * cs * sizeof(float);
    const size_t spec = 6 * (size_t)N * N * HP * 2 * sizeof(float);
    int max_blocks = 0;
    for (int tk = 0; tk < TK_COUNT; ++tk)
        for (int v = 0; v < kVariants; ++v) max_blocks = std::max(max_blocks, variant_shape(N, tk, v).blocks);
    const size_t off_x = 0, off_t = off_x + field;
    const size_t off_s = off_t + ((7 * cs * sizeof(float) + 255) & ~size_t(255));
    const size_t off_part = off_s + ((spec + 255) & ~size_t(255));
    const size_t off_cg = off_part + (((size_t)max_blocks * 2 * sizeof(double) + 255) & ~size_t(255));
    const size_t off_tw = off_cg + 256;
    const size_t total = off_tw + (size_t)N * 8;
    DeviceBuffer buf;
    if (cudaMalloc(&buf.p, total) != cudaSuccess) {
        cudaGetLastError();
        return FFTG_ENOMEM;
    }
    char* b = (char*)buf.p;
    // positive finite data everywhere (bytes 0x3C: floats near 0.0115)
    if (cudaMemsetAsync(b, 0x3C, off_part, s) != cudaSuccess) return FFTG_ECUDA;
    std::vector<double> tw64(2 * N);
    std::vector<float> tw32(2 * N);
    twiddles(N, tw64.data(), tw32.data());
    if (cudaMemcpyAsync(b + off_tw, tw32.data(), (size_t)N * 8, cudaMemcpyHostToDevice, s) != cudaSuccess)
        return FFTG_ECUDA;
    CGState st{};
    st.rr = st.rr0 = 1.0;
    st.alpha = 1e-3;
    st.beta = 0.5;
    st.it = 1;
    st.max_it = 1 << 30;
    st.done = CG_RUNNING;
    CGState* cg = (CGState*)(b + off_cg);
    PassArgs a{};
    a.tw = b + off_tw;
    a.partials = (double*)(b + off_part);
    a.cs = (long long)cs;
    a.ucs = (long long)N * N * N;
    a.fstride = 6 * (long long)cs;
    a.sstride = 6LL * N * N * (long long)HP;
    a.tangent = b + off_t;
    a.scale = 1.0 / ((double)N * N * N);
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess) return FFTG_ECUDA;
    if (cudaEventCreate(&e1) != cudaSuccess) {
        cudaEventDestroy(e0);
        return FFTG_ECUDA;
    }
    int rc = FFTG_OK;
    for (int tk = 0; tk < TK_COUNT && rc == FFTG_OK; ++tk) {
        PassArgs k = a;
        k.out = b + off_s;
        if (tk == TK_P1) {
            k.cg = cg;
        } else if (tk == TK_P5) {
            k.in = b + off_s;
            k.out = b + off_x;
        }
        double best = 1e300;
        int best_v = 0;
        for (int v = 0; v < kVariants && rc == FFTG_OK; ++v) {
            std::vector<float> t;
            for (int r = 0; r <= reps; ++r) {
                if (k.cg && cudaMemcpyAsync(cg, &st, sizeof st, cudaMemcpyHostToDevice, s) != cudaSuccess) {
                    rc = FFTG_ECUDA;
                    break;
                }
                cudaEventRecord(e0, s);
                if (launch_schedule(N, tk, v, k, s) != cudaSuccess) {
                    rc = FFTG_ECUDA;
                    break;
                }
                cudaEventRecord(e1, s);
                float ms = 0.f;
                if (cudaEventSynchronize(e1) != cudaSuccess || cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) {
                    rc = FFTG_ECUDA;
                    break;
                }
                if (r > 0) t.push_back(ms);  // the first launch warms up
            }
            if (rc != FFTG_OK) break;
            std::sort(t.begin(), t.end());
            const double med = t[t.size() / 2];
            if (ms_out) ms_out[tk * kVariants + v] = med;
            // a variant replaces the default only when it is clearly faster
            if (med < (v == 0 ? best : 0.98 * best)) {
                best = med;
                best_v = v;
            }
        }
        if (rc == FFTG_OK) {
            chosen[tk] = best_v;
            g_sched[grid_index(N)][tk].store(best_v);
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (rc != FFTG_OK) cudaGetLastError();
    return rc;
}

}  // namespace

int tuned_kind(int pass_kind) {
    switch (pass_kind) {
        case PK_ROWS_CG_F32: return TK_P1;
        case PK_P2_F32: return TK_P2;
        case PK_P3_F32: return TK_P3;
        case PK_P4_F32: return TK_P4;
        case PK_P5_USER_F32: return TK_P5;
        default: return -1;
    }
}

int schedule_variant(int N, int tk) {
    const int g = grid_index(N);
    if (g < 0 || tk < 0 || tk >= TK_COUNT) return 0;
    return g_sched[g][tk].load(std::memory_order_relaxed);
}

cudaError_t run_variant(int N, int tk, int v, const PassArgs& a, int nf, cudaStream_t s) {
    switch (N) {
#define FFTG_CASE(n) case n: return run_variant_n<n>(tk, v, a, nf, s);
        FFTG_CASE(3) FFTG_CASE(5) FFTG_CASE(9) FFTG_CASE(15) FFTG_CASE(25) FFTG_CASE(27)
        FFTG_CASE(45) FFTG_CASE(75) FFTG_CASE(81) FFTG_CASE(125) FFTG_CASE(135) FFTG_CASE(225)
        FFTG_CASE(243)
#undef FFTG_CASE
        default: return cudaErrorInvalidValue;
    }
}

VariantShape variant_shape(int N, int tk, int v) {
    switch (N) {
#define FFTG_CASE(n) case n: return variant_shape_n<n>(tk, v);
        FFTG_CASE(3) FFTG_CASE(5) FFTG_CASE(9) FFTG_CASE(15) FFTG_CASE(25) FFTG_CASE(27)
        FFTG_CASE(45) FFTG_CASE(75) FFTG_CASE(81) FFTG_CASE(125) FFTG_CASE(135) FFTG_CASE(225)
        FFTG_CASE(243)
#undef FFTG_CASE
        default: return VariantShape{0, 0, 0, 0, 0};
    }
}

}  // namespace fftg

using namespace fftg;

extern "C" {

int fftg_schedule_set(int N, int kind, int variant) {
    const int g = grid_index(N);
    if (g < 0 || kind < 0 || kind >= TK_COUNT || variant < 0 || variant >= kVariants) return FFTG_EINVAL;
    g_sched[g][kind].store(variant);
    return FFTG_OK;
}

int fftg_schedule_get(int N, int kind) {
    const int g = grid_index(N);
    if (g < 0 || kind < 0 || kind >= TK_COUNT) return FFTG_EINVAL;
    return g_sched[g][kind].load();
}

int fftg_schedule_describe(int N, int kind, int variant, int shape[5]) {
    if (grid_index(N) < 0 || kind < 0 || kind >= TK_COUNT || variant < 0 || variant >= kVariants || !shape)
        return FFTG_EINVAL;
    const VariantShape sh = variant_shape(N, kind, variant);
    shape[0] = sh.n1;
    shape[1] = sh.n2;
    shape[2] = sh.rows;
    shape[3] = sh.cols;
    shape[4] = sh.blocks;
    return FFTG_OK;
}

int fftg_autotune(int N, int flags, void* stream, double* ms, int* chosen) {
    if (grid_index(N) < 0 || !chosen) return FFTG_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    std::lock_guard<std::mutex> lock(g_cache_mu);
    const std::string path = (flags & FFTG_TUNE_CACHE) ? cache_path() : std::string();
    if (ms)
        for (int i = 0; i < TK_COUNT * kVariants; ++i) ms[i] = -1.0;
    if (!path.empty() && !(flags & FFTG_TUNE_FORCE)) {
        int got[TK_COUNT];
        bool all = true;
        for (int tk = 0; tk < TK_COUNT; ++tk) {
            got[tk] = cache_lookup(path, cache_key(N, tk));
            all = all && got[tk] >= 0;
        }
        if (all) {
            for (int tk = 0; tk < TK_COUNT; ++tk) {
                chosen[tk] = got[tk];
                g_sched[grid_index(N)][tk].store(got[tk]);
            }
            return FFTG_OK;
        }
    }
    const long long V = (long long)N * N * N;
    const int reps = V >= 2000000 ? 5 : V >= 100000 ? 11 : 21;
    const int rc = tune(N, s, reps, ms, chosen);
    if (rc == FFTG_OK && !path.empty())
        for (int tk = 0; tk < TK_COUNT; ++tk) cache_store(path, cache_key(N, tk), chosen[tk]);
    return rc;
}

}  // extern "C"
