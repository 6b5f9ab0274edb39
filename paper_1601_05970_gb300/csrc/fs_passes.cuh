// Grid passes of the finite-strain extension (Section 6 names finite strain
// as the next step of the method): the projected matvec q = G (K : p) and
// the residual G P on real fields of nine components, the deformation-
// gradient-like tensor A_ij at component 3i + j, [9][cs], and a half
// spectrum [9][N][N][HP] (row pitch spec_pitch).
//
// The five passes are those of the small-strain path with three changes:
//  * nine real components share five complex FFTs per row (pairs (0,1),
//    (2,3), (4,5), (6,7) and component 8 alone);
//  * the projection onto gradient fields acts row by row: with n = xi/|xi|,
//    Ghat : A = (A n) (x) n, i.e. Ghat_ijlm = delta_il n_j n_m (the
//    finite-strain counterpart of Appendix A's operator; Ghat(0) = 0);
//  * the tangent is St. Venant-Kirchhoff's, applied on the fly from the
//    displacement gradient H = F - I (the only per-voxel tangent data) and
//    the phase's Lame constants: K : d = d S + F dS with
//    E = (H + H^T + H^T H)/2, S = lambda tr(E) I + 2 mu E, M = F^T d and
//    dS = lambda tr(M) I + mu (M + M^T).
// The mixed path's residual runs the plain passes in double-float
// arithmetic (dd.cuh) on the FP64 stress.
#pragma once

#include "common.cuh"
#include "fft_core.cuh"
#include "passes.cuh"

namespace fftg {

constexpr int kFsComp = 9;
constexpr int kFsPairs = 5;

enum : int { FS_P1_PLAIN = 0, FS_P1_TAN = 1, FS_P1_CG = 2, FS_P1_TANRHS = 3 };
enum : int { FS_P5_PLAIN = 0, FS_P5_DOT = 1, FS_P5_RHS = 2, FS_P5_NEWTON = 3 };
// FS_P5_NEWTON: F* += x for the solution x of a mixed inner solve, with its
// squared norm. The mixed path's CG iteration is that of fs_cg_passes.cuh.

struct FsArgs {
    const void* in;        // P1: real field; P5: spectrum
    void* out;             // P1: spectrum; P2-P4: spectrum (in place); P5: real field
    const void* aux;       // P1_CG: r; P5_DOT: p
    void* aux2;            // P1_CG: p (updated in place)
    void* aux3;            // P1_CG: x (gets the previous iteration's alpha p);
                           // P5_NEWTON: F* (FP64, updated in place)
    const void* hgrad;     // P1_TAN, P1_CG: H = F - I, [9][cs] in the FFT precision
    const uint8_t* phase;  // [cs]
    const double* lame;    // [nphase][2]: lambda, mu
    CGState* cg;
    double* partials;      // [row blocks][2]
    const void* tw;        // w_N^j, j < N, in the FFT precision
    double scale;          // P3: factor on Ghat (+-1/N^3)
    long long cs;          // component stride of the real fields (elements)
    long long ucs;         // that of in and out (and the p of P5_DOT): cs, or N^3 for a caller's fields
    int unit;              // P1_TANRHS: tau = K : E_unit, E_unit the unit tensor at component unit
    const double* red_in;  // P2 of the mixed CG iteration: the row pass's block partials of <p, K : p>
    int red_n;             // (reduced by P2's first block, which sets alpha)
};

// Tuning: shared-memory budgets (KB) of the row passes and of P3, and the
// minimum resident blocks per SM of the FP32 P1 and P5 (a bound on their
// registers; the FP64 ones take what they need: they are bound by FP64
// arithmetic, not by memory; the double-float P1 with two blocks per SM
// 2.08 ms at 243^3, with one 3.16). Set by timing variants at 243^3, FP32,
// with a P1 that also did the vector updates of a CG iteration (those are in
// k_x1i now): 40 KB of rows (R = 4) gave P1 0.66 ms (3 or 4 blocks per SM
// alike; 4 spills a little) and P5 0.34 ms with 4 blocks per SM (0.39 ms with
// 3); 80 KB of rows 0.76 ms; P3 with 100 or 64 KB of columns 0.44 and 0.71 ms
// against 0.39 ms with 150 KB. One voxel per lane: a caller's components start
// on any element (and two, on aligned fields, took P1 to 0.73-0.91 ms). P5 with the
// spectrum loads of two rounds issued together: 0.323 against 0.336 ms
// (with 3 blocks per SM 0.369 ms).
#ifndef FFTG_FS_ROW_KB
#define FFTG_FS_ROW_KB 40
#endif
#ifndef FFTG_FS_P3_KB
#define FFTG_FS_P3_KB 150
#endif
#ifndef FFTG_FS_P1_MINB
#define FFTG_FS_P1_MINB 3
#endif
#ifndef FFTG_FS_P5_MINB
#define FFTG_FS_P5_MINB 4
#endif
#ifndef FFTG_FS_P5_LDB
#define FFTG_FS_P5_LDB 2
#endif

template <int N, typename T>
struct FsCfg {
    static constexpr int H = (N + 1) / 2, HP = spec_pitch(N);
    static constexpr int CS = (int)sizeof(cplx<T>);
    static constexpr int fl2(int x) {
        return x >= 32 ? 32 : x >= 16 ? 16 : x >= 8 ? 8 : x >= 4 ? 4 : x >= 2 ? 2 : 1;
    }
    static constexpr int rup32(int x) { return ((x + 31) / 32) * 32; }
    static constexpr int cap(int x) { return x > 1024 ? 1024 : x; }
    // rows per block of P1/P5: five complex pencils per row; a power of two
    // >= 4, so a block's rows start on a 16-byte boundary of every component
    static constexpr int R0 = fl2(FFTG_FS_ROW_KB * 1024 / (kFsPairs * N * CS));
    static constexpr int R = R0 < 4 ? 4 : R0;
    // columns per block of P3: nine pencils per column
    static constexpr int W3 = fl2(FFTG_FS_P3_KB * 1024 / (kFsComp * N * CS));
    static constexpr int T3 = Plan<N>::N2 == 1 ? 256 : cap(rup32(kFsComp * W3 * Plan<N>::N2));
    static constexpr size_t smem_rows = (size_t)(kFsPairs * R * N + N) * CS;
    static constexpr size_t smem_p3 = (size_t)(kFsComp * W3 * N + N) * CS;
    static constexpr int row_blocks = (N * N + R - 1) / R;
    static_assert(smem_rows <= 227 * 1024 && smem_p3 <= 227 * 1024, "shared memory per block");
    static_assert(T3 <= 1024 && T3 % 32 == 0, "threads per block");
};

// tau = K(F) : d for St. Venant-Kirchhoff, from h = F - I.
template <typename T>
__device__ __forceinline__ void svk_tangent_apply(const T (&h)[9], T lam, T mu, const T (&d)[9], T (&tau)[9]) {
    T E[9];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            T hh = T(0);
#pragma unroll
            for (int k = 0; k < 3; ++k) hh += h[3 * k + i] * h[3 * k + j];
            E[3 * i + j] = T(0.5) * (h[3 * i + j] + h[3 * j + i] + hh);
        }
    const T le = lam * (E[0] + E[4] + E[8]);
    T M[9];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            T m = d[3 * i + j];  // (I + H)^T d
#pragma unroll
            for (int k = 0; k < 3; ++k) m += h[3 * k + i] * d[3 * k + j];
            M[3 * i + j] = m;
        }
    const T lm = lam * (M[0] + M[4] + M[8]);
    T S[9], dS[9];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            S[3 * i + j] = T(2) * mu * E[3 * i + j] + (i == j ? le : T(0));
            dS[3 * i + j] = mu * (M[3 * i + j] + M[3 * j + i]) + (i == j ? lm : T(0));
        }
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            T t = dS[3 * i + j];  // I dS
#pragma unroll
            for (int k = 0; k < 3; ++k) t += d[3 * i + k] * S[3 * k + j] + h[3 * i + k] * dS[3 * k + j];
            tau[3 * i + j] = t;
        }
}

// ----------------------------------------------------------------------- P1
// [x += alpha p; p = r + beta p]; tau = K : p or tau = input; x3 R2C FFT of
// R rows per block.
template <int N, typename T, int MODE>
__global__ void __launch_bounds__(kThreads, sizeof(T) == 4 ? FFTG_FS_P1_MINB : is_dd_v<T> ? 2 : 1) k_fs_p1(FsArgs a) {
    using C = FsCfg<N, T>;
    constexpr int R = C::R, H = C::H, HP = C::HP;
    constexpr int N1 = Plan<N>::N1, N2 = Plan<N>::N2;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cplx<T>* tw = reinterpret_cast<cplx<T>*>(smem_raw);
    cplx<T>* z = tw + N;  // [5][R][N]
    constexpr bool CGM = MODE == FS_P1_CG;
    if (CGM && a.cg->done) return;
    const int tid = threadIdx.x;
    load_tw<T>(tw, a.tw, N);
    const int row0 = blockIdx.x * R;
    const int nrows = min(R, N * N - row0);
    const long long base = (long long)row0 * N;
    const int nel = nrows * N;
    const long long cs = a.cs;
    T beta = T(0), alpha = T(0);
    bool first = true;
    if (CGM) {
        beta = (T)a.cg->beta;
        alpha = (T)a.cg->alpha;
        first = a.cg->it == 0;
    }
    // Elementwise phase, one voxel per lane. Every load of a voxel is issued
    // before its first store (the fields could alias as far as the compiler
    // knows, which would otherwise serialise one round trip per component).
    for (int i = tid; i < R * N; i += kThreads) {
        T s[9];
        if (i < nel) {
            const long long v = base + i;
            T p[9], h[9];
            if constexpr (CGM) {
                const T* r = (const T*)a.aux;
                T* pp = (T*)a.aux2;
                T* xx = (T*)a.aux3;
                T po[9], xo[9];
#pragma unroll
                for (int c = 0; c < 9; ++c) p[c] = r[c * cs + v];
                if (!first) {
#pragma unroll
                    for (int c = 0; c < 9; ++c) {
                        po[c] = pp[c * cs + v];
                        xo[c] = xx[c * cs + v];
                    }
                }
                const T* hg = (const T*)a.hgrad;
#pragma unroll
                for (int c = 0; c < 9; ++c) h[c] = hg[c * cs + v];
                const int ph = a.phase[v];
                if (!first) {
#pragma unroll
                    for (int c = 0; c < 9; ++c) {
                        xo[c] += alpha * po[c];
                        p[c] += beta * po[c];
                        xx[c * cs + v] = xo[c];
                    }
                }
#pragma unroll
                for (int c = 0; c < 9; ++c) pp[c * cs + v] = p[c];
                const double* m = a.lame + 2 * ph;
                svk_tangent_apply<T>(h, (T)m[0], (T)m[1], p, s);
            } else {
                using TIn = typename PlainIn<T>::type;
                const TIn* in = (const TIn*)a.in;
#pragma unroll
                for (int c = 0; c < 9; ++c)
                    p[c] = T(MODE == FS_P1_TANRHS ? TIn(c == a.unit ? 1 : 0) : in[c * a.ucs + v]);
                if constexpr (MODE == FS_P1_PLAIN) {
#pragma unroll
                    for (int c = 0; c < 9; ++c) s[c] = p[c];
                } else {
                    const T* hg = (const T*)a.hgrad;
#pragma unroll
                    for (int c = 0; c < 9; ++c) h[c] = hg[c * cs + v];
                    const double* m = a.lame + 2 * a.phase[v];
                    svk_tangent_apply<T>(h, (T)m[0], (T)m[1], p, s);
                }
            }
        } else {
#pragma unroll
            for (int c = 0; c < 9; ++c) s[c] = T(0);
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) z[c * R * N + i] = mk(s[2 * c], s[2 * c + 1]);
        z[4 * R * N + i] = mk(s[8], T(0));
    }
    __syncthreads();
    constexpr int NP = kFsPairs * R;
    for (int it = tid; it < NP * N2; it += kThreads) {
        const int pc = it % NP, t = it / NP;
        if (pc % R < nrows) fwdA<N, T>(z + pc * N, 1, z + pc * N, 1, t, tw);
    }
    __syncthreads();
    if (N2 > 1) {
        for (int it = tid; it < NP * N1; it += kThreads) {
            const int pc = it % NP, k1 = it / NP;
            if (pc % R < nrows) fwdB<N, false, T>(z + pc * N, 1, z + pc * N, 1, k1, tw);
        }
        __syncthreads();
    }
    // Split each packed transform Z = FFT(a + i b) into the half spectra
    // A_k = (Z_k + conj Z_{N-k})/2 and B_k = (Z_k - conj Z_{N-k})/(2i).
    cplx<T>* out = (cplx<T>*)a.out;
    const long long HS = (long long)N * N * HP;
    for (int it = tid; it < nrows * H; it += kThreads) {
        const int row = it / H, k = it - row * H;
        const int pk = perm_pos<N>(k), pn = perm_pos<N>(k == 0 ? 0 : N - k);
        const long long o = (long long)(row0 + row) * HP + k;
#pragma unroll
        for (int c = 0; c < kFsPairs; ++c) {
            const cplx<T> zk = z[(c * R + row) * N + pk];
            const cplx<T> zn = conj(z[(c * R + row) * N + pn]);
            out[(2 * c) * HS + o] = half_of(zk + zn);
            if (2 * c + 1 < kFsComp) {
                const cplx<T> d = zk - zn;
                out[(2 * c + 1) * HS + o] = half_of(mk(d.y, -d.x));
            }
        }
    }
}

// Ghat_fs : A at frequency (f1, f2, f3), times `scale`, in place on the nine
// complex components held at stride `cs`: row i becomes (A_i . n) n.
template <typename T>
__device__ __forceinline__ void ghat_fs_point(cplx<T>* b, int cs, int f1, int f2, int f3, T scale) {
    const T q2 = T(f1) * T(f1) + T(f2) * T(f2) + T(f3) * T(f3);
    const T inv = q2 > T(0) ? rsqrt_t(q2) : T(0);
    const T n0 = T(f1) * inv, n1 = T(f2) * inv, n2 = T(f3) * inv;
    const T m0 = scale * n0, m1 = scale * n1, m2 = scale * n2;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const cplx<T> t = n0 * b[(3 * i) * cs] + n1 * b[(3 * i + 1) * cs] + n2 * b[(3 * i + 2) * cs];
        b[(3 * i) * cs] = m0 * t;
        b[(3 * i + 1) * cs] = m1 * t;
        b[(3 * i + 2) * cs] = m2 * t;
    }
}

// ------------------------------------------------------------- P3 (x1 + Ghat)
// As the small-strain P3: stage A forward into shared memory, stage B
// forward in place, Ghat_fs with one thread per (column, frequency), stage B
// inverse, stage A inverse back to the spectrum; in FP32 with two-stage
// splits of N2 <= 9 the middle three phases are one (below).
template <int N, typename T>
__global__ void __launch_bounds__(FsCfg<N, T>::T3) k_fs_p3(FsArgs a) {
    using C = FsCfg<N, T>;
    constexpr int H = C::H, HP = C::HP, W = C::W3, NT = C::T3;
    constexpr int N1 = Plan<N>::N1, N2 = Plan<N>::N2;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cplx<T>* tw = reinterpret_cast<cplx<T>*>(smem_raw);
    cplx<T>* buf = tw + N;  // [9][N][W]
    if (a.cg && a.cg->done) return;
    const int tid = threadIdx.x;
    load_tw<T>(tw, a.tw, N);
    __syncthreads();
    const int col0 = blockIdx.x * W, k2g = blockIdx.y;
    cplx<T>* sp = (cplx<T>*)a.out;
    constexpr int P = kFsComp * W;
    const long long NH = (long long)N * HP;
    for (int it = tid; it < P * N2; it += NT) {
        const int pc = it % P, t = it / P;
        const int c = pc / W, w = pc - c * W, col = col0 + w;
        if (col < H) fwdA<N, T>(sp + c * N * NH + k2g * HP + col, (int)NH, buf + c * N * W + w, W, t, tw);
    }
    __syncthreads();
    const T scale = (T)a.scale;
    const int f2 = (k2g <= (N - 1) / 2) ? k2g : k2g - N;
    if constexpr (std::is_same<T, float>::value && N2 > 1 && N2 <= 9) {
        // Stage B, Ghat_fs and the inverse stage B in one phase: row i of
        // Ghat_fs : A is (A_i . n) n, which needs row i's three components
        // only. One thread per (column, k1, row) takes them through the
        // forward N2-point DFT, sums t = A_i . n for its N2 frequencies in
        // Ghat_fs's order, and writes scale n_j t back through the inverse
        // DFT and its twiddles: two shared-memory passes per point instead
        // of five, and two barriers fewer.
        for (int it = tid; it < W * N1 * 3; it += NT) {
            const int w = it % W, r = it / W;
            const int k1 = r % N1, row = r / N1, col = col0 + w;
            if (col >= H) continue;
            cplx<T>* base = buf + (3 * row * N + N2 * k1) * W + w;  // component 3 row + j at base[j N W]
            T n[N2][3];
#pragma unroll
            for (int k2 = 0; k2 < N2; ++k2) {
                const int kk = k1 + N1 * k2;
                const T f1 = T((kk <= (N - 1) / 2) ? kk : kk - N), g2 = T(f2), f3 = T(col);
                const T q2 = f1 * f1 + g2 * g2 + f3 * f3;
                const T inv = q2 > T(0) ? rsqrt_t(q2) : T(0);
                n[k2][0] = f1 * inv;
                n[k2][1] = g2 * inv;
                n[k2][2] = f3 * inv;
            }
            cplx<T> t[N2];
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                cplx<T> v[N2];
#pragma unroll
                for (int q = 0; q < N2; ++q) v[q] = base[j * N * W + q * W];
                RegDFT<N, N2, -1, T>::run(v, tw);
#pragma unroll
                for (int k2 = 0; k2 < N2; ++k2) t[k2] = j == 0 ? n[k2][0] * v[k2] : t[k2] + n[k2][j] * v[k2];
            }
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                cplx<T> v[N2];
#pragma unroll
                for (int k2 = 0; k2 < N2; ++k2) v[k2] = (scale * n[k2][j]) * t[k2];
                RegDFT<N, N2, +1, T>::run(v, tw);
#pragma unroll
                for (int q = 0; q < N2; ++q) {
                    cplx<T> z = v[q];
                    if (k1 > 0 && q > 0) z = twmul<+1>(z, tw[q * k1]);  // q*k1 < N
                    base[j * N * W + q * W] = z;
                }
            }
        }
    } else {
        if (N2 > 1) {
            for (int it = tid; it < P * N1; it += NT) {
                const int pc = it % P, k1 = it / P;
                const int c = pc / W, w = pc - c * W;
                if (col0 + w < H) fwdB<N, false, T>(buf + c * N * W + w, W, buf + c * N * W + w, W, k1, tw);
            }
            __syncthreads();
        }
        for (int it = tid; it < W * N; it += NT) {
            const int w = it % W, pos = it / W, col = col0 + w;
            const int k1 = pos / N2, k2 = pos - k1 * N2;
            const int kk = k1 + N1 * k2;  // frequency held at position N2*k1 + k2
            if (col < H)
                ghat_fs_point<T>(buf + pos * W + w, N * W, (kk <= (N - 1) / 2) ? kk : kk - N, f2, col, scale);
        }
        __syncthreads();
        if (N2 > 1) {
            for (int it = tid; it < P * N1; it += NT) {
                const int pc = it % P, k1 = it / P;
                const int c = pc / W, w = pc - c * W;
                if (col0 + w < H) invB<N, false, T>(buf + c * N * W + w, W, buf + c * N * W + w, W, k1, tw);
            }
        }
    }
    __syncthreads();
    for (int it = tid; it < P * N2; it += NT) {
        const int pc = it % P, t = it / P;
        const int c = pc / W, w = pc - c * W, col = col0 + w;
        if (col < H) invA<N, T>(buf + c * N * W + w, W, sp + c * N * NH + k2g * HP + col, (int)NH, t, tw);
    }
}

// ----------------------------------------------------------------------- P5
// x3 C2R inverse FFT of R rows per block; writes the real field (in TO) and,
// for DOT, the partials of <p, q> (then alpha), for RHS those of <r, r> in
// TO and of ||G P||^2 in T (then the start of the CG solve).
template <int N, typename T, int MODE, typename TO>
__global__ void __launch_bounds__(kThreads, sizeof(T) == 4 ? FFTG_FS_P5_MINB : 1) k_fs_p5(FsArgs a) {
    using C = FsCfg<N, T>;
    constexpr int R = C::R, H = C::H, HP = C::HP;
    constexpr int N1 = Plan<N>::N1, N2 = Plan<N>::N2;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cplx<T>* tw = reinterpret_cast<cplx<T>*>(smem_raw);
    cplx<T>* z = tw + N;  // [5][R][N]
    CGState* cg = a.cg;
    if (MODE == FS_P5_DOT && cg->done) return;
    const int tid = threadIdx.x;
    load_tw<T>(tw, a.tw, N);
    const int row0 = blockIdx.x * R;
    const int nrows = min(R, N * N - row0);
    const long long base = (long long)row0 * N;
    const int nel = nrows * N;
    const cplx<T>* in = (const cplx<T>*)a.in;
    const long long HS = (long long)N * N * HP;
    // Spectrum rows -> tile, the loads of FFTG_FS_P5_LDB rounds issued
    // before their stores.
    constexpr int NRL = (R * H + kThreads - 1) / kThreads;
    constexpr int LB = FFTG_FS_P5_LDB < NRL ? FFTG_FS_P5_LDB : NRL;
#pragma unroll
    for (int r0 = 0; r0 < NRL; r0 += LB) {
        cplx<T> A[LB][kFsPairs], B[LB][kFsPairs];
#pragma unroll
        for (int u = 0; u < LB; ++u) {
            const int it = tid + (r0 + u) * kThreads;
            if (r0 + u < NRL && it < nrows * H) {
                const int row = it / H, k = it - row * H;
                const long long o = (long long)(row0 + row) * HP + k;
#pragma unroll
                for (int c = 0; c < kFsPairs; ++c) {
                    A[u][c] = in[(2 * c) * HS + o];
                    B[u][c] = (2 * c + 1 < kFsComp) ? in[(2 * c + 1) * HS + o] : mk(T(0), T(0));
                }
            }
        }
#pragma unroll
        for (int u = 0; u < LB; ++u) {
            const int it = tid + (r0 + u) * kThreads;
            if (r0 + u < NRL && it < nrows * H) {
                const int row = it / H, k = it - row * H;
                const int pk = perm_pos<N>(k);
                const int pn = perm_pos<N>(k == 0 ? 0 : N - k);
#pragma unroll
                for (int c = 0; c < kFsPairs; ++c) {
                    const cplx<T> a0 = A[u][c], b0 = B[u][c];
                    // A + iB and conj(A) + i conj(B); A and B are real at k = 0
                    // (what their imaginary parts hold is rounding)
                    z[(c * R + row) * N + pk] = k > 0 ? mk(a0.x - b0.y, a0.y + b0.x) : mk(a0.x, b0.x);
                    if (k > 0) z[(c * R + row) * N + pn] = mk(a0.x + b0.y, b0.x - a0.y);
                }
            }
        }
    }
    __syncthreads();
    constexpr int NP = kFsPairs * R;
    if (N2 > 1) {
        for (int it = tid; it < NP * N1; it += kThreads) {
            const int pc = it % NP, k1 = it / NP;
            if (pc % R < nrows) invB<N, false, T>(z + pc * N, 1, z + pc * N, 1, k1, tw);
        }
        __syncthreads();
    }
    for (int it = tid; it < NP * N2; it += kThreads) {
        const int pc = it % NP, t = it / NP;
        if (pc % R < nrows) invA<N, T>(z + pc * N, 1, z + pc * N, 1, t, tw);
    }
    __syncthreads();
    const long long cs = a.cs;
    TO* out = (TO*)a.out;
    const TO* pin = (const TO*)a.aux;  // FS_P5_DOT: p
    double* Fw = MODE == FS_P5_NEWTON ? (double*)a.aux3 : nullptr;
    double accx = 0.0;  // FS_P5_NEWTON: squares of x
    T acc0 = T(0);
    double acc1 = 0.0;
    // One voxel per lane: p is loaded before q is stored. (Counted to R N: to nel
    // the loop is unrolled, and FP64 at 27^3 takes 130 registers instead of 122,
    // one block per SM instead of two.)
    for (int i = tid; i < R * N; i += kThreads) {
        if (i >= nel) continue;
        const long long v = base + i;
        TO pv[9];
        if (MODE == FS_P5_DOT) {
#pragma unroll
            for (int c = 0; c < 9; ++c) pv[c] = pin[c * a.ucs + v];
        }
        T qd[9];
        TO q[9];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const cplx<T> zz = z[c * R * N + i];
            qd[2 * c] = zz.x;
            qd[2 * c + 1] = zz.y;
        }
        qd[8] = z[4 * R * N + i].x;
#pragma unroll
        for (int c = 0; c < 9; ++c) q[c] = (TO)qd[c];
        if constexpr (MODE == FS_P5_NEWTON) {
            double fv[9];
#pragma unroll
            for (int c = 0; c < 9; ++c) fv[c] = Fw[c * cs + v];
#pragma unroll
            for (int c = 0; c < 9; ++c) {
                const double d = (double)q[c];
                Fw[c * cs + v] = fv[c] + d;
                accx += d * d;
            }
            continue;
        }
#pragma unroll
        for (int c = 0; c < 9; ++c) out[c * a.ucs + v] = q[c];
        if (MODE == FS_P5_PLAIN) continue;
#pragma unroll
        for (int c = 0; c < 9; ++c) {
            if (MODE == FS_P5_DOT) {
                acc0 += (T)(pv[c] * q[c]);
            } else {
                acc0 += (T)(q[c] * q[c]);
                acc1 += (double)(qd[c] * qd[c]);
            }
        }
    }
    if (MODE == FS_P5_PLAIN) return;
    const int nb = gridDim.x;
    double part[2];
    if (MODE == FS_P5_NEWTON) {
        // the block's part of ||x||^2 (k_fs_newton_norm sums the parts)
        part[0] = block_sum(accx);
        if (tid == 0) a.partials[blockIdx.x] = part[0];
        return;
    }
    part[0] = block_sum((double)acc0);
    part[1] = (MODE == FS_P5_RHS) ? block_sum(acc1) : 0.0;
    if (!publish_partials<2>(part, a.partials, blockIdx.x, nb, &cg->ticket)) return;
    double tot[2];
    reduce_partials<2>(a.partials, nb, &cg->ticket, tot);
    if (tid != 0) return;
    if (MODE == FS_P5_DOT)
        cg_after_dot(cg, tot[0]);
    else
        cg_start(cg, tot[0], tot[1]);
}

// ------------------------------------------------------------------ launcher
enum FsPassKind : int {
    FK_P1_PLAIN_F64, FK_P1_PLAIN_F32, FK_P1_TAN_F64, FK_P1_TAN_F32, FK_P1_CG_F64,
    FK_P2_F64, FK_P2_F32, FK_P3_F64, FK_P3_F32, FK_P4_F64, FK_P4_F32,
    FK_P5_PLAIN_F64, FK_P5_PLAIN_F32, FK_P5_DOT_F64, FK_P5_DOT_F32,
    FK_P5_RHS_F64_TO_F64,
    // double-float FFTs: FP64 field in and out
    FK_P1_PLAIN_DD, FK_P2_DD, FK_P3_DD, FK_P4_DD, FK_P5_PLAIN_DD_TO_F64,
    // right-hand sides of the macroscopic tangent
    FK_P1_TANRHS_F64, FK_P1_TANRHS_F32,
    // the mixed path's CG on coefficients (fs_cg_passes.cuh)
    FK_X1I_CG_F32, FK_P4_GRAD_F32, FK_ROWS_CG_F32, FK_P2_GRAD_F32, FK_X1F_CG_F32, FK_P2_GRAD_DD,
    FK_X1F_RHS_F32, FK_X1F_RHS_DD, FK_X1I_SOLUTION_F32, FK_P5_NEWTON_F32,
    FK_COUNT
};

int fs_row_blocks(int N, bool fp64);

cudaError_t run_fs_pass(int N, FsPassKind kind, const FsArgs& a, cudaStream_t s);

template <int N>
cudaError_t run_fs_pass_n(FsPassKind kind, const FsArgs& a, cudaStream_t s);

template <typename K>
static cudaError_t launch_fs(K kernel, dim3 grid, int threads, size_t smem, const FsArgs& a, cudaStream_t s) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kernel<<<grid, threads, smem, s>>>(a);
    return cudaGetLastError();
}

// The x2 passes are the small-strain kernels over nine components; they
// read the spectrum, the twiddles and (when set) the CG state.
template <int N, typename T, bool FWD>
static cudaError_t launch_fs_p24(const FsArgs& a, cudaStream_t s) {
    using C = Cfg<N, T>;
    PassArgs b{};
    b.out = a.out;
    b.cg = a.cg;
    b.tw = a.tw;
    b.red_in = a.red_in;
    b.red_n = a.red_n;
    const dim3 g((C::H + C::W2 - 1) / C::W2, (kFsComp * N + C::S2 - 1) / C::S2, 1);
    cudaError_t e = cudaFuncSetAttribute(k_p24<N, T, FWD, kFsComp>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)C::smem_p24);
    if (e != cudaSuccess) return e;
    k_p24<N, T, FWD, kFsComp><<<g, C::T2, C::smem_p24, s>>>(b);
    return cudaGetLastError();
}

}  // namespace fftg
