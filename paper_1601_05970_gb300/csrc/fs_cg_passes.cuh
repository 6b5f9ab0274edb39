// The FP32 CG iteration of the finite-strain mixed path on coefficients, as in
// cg_passes.cuh: every vector is a gradient field, a(x)f per frequency for one
// complex vector a, and r, p and x are held as a.
//
//   x1i   p = r + beta p, x += alpha p_old; inverse x1 of f1 a_i and a_i
//   P4g   inverse x2 of f1 a_i, f2 a_i and f3 a_i
//   rows  inverse x3, tau = K : p with <p, tau>, forward x3
//   P2g   forward x2; A_i1 and B_i = f2 A_i2 + f3 A_i3 go on (alpha is set)
//   x1f   forward x1, a of Ghat_fs : tau: a_i = (f1 A_i1 + B_i) / q;
//         r -= alpha a, <r, r>
//
// Six fields instead of nine pass x1, since f2 and f3 are known in the x2
// passes: 84.3 + 60.2 + 109.3 + 60.2 + 48.2 = 362 B per voxel at 243^3, where
// r, p and x as real fields of nine components moved 578 (an iteration 1.81 ->
// 1.28 ms there, 275 -> 190 us at 125^3).
#pragma once

#include "cg_passes.cuh"
#include "fs_passes.cuh"

namespace fftg {

// Columns of the x2 gradient passes: the three fields of one row i of the
// tensor and one x1 plane per block.
template <int N, typename T>
struct GradX2 {
    static constexpr int N1 = Plan<N>::N1, N2 = Plan<N>::N2, H = (N + 1) / 2;
    static constexpr int W = sizeof(T) == 4 ? 16 : 8;
    static constexpr size_t smem = (size_t)(3 * N * W + N) * sizeof(cplx<T>);
    static constexpr int items = ((3 * W * N2 + 31) / 32) * 32;
    static constexpr int NT = items < 64 ? 64 : items > 448 ? 448 : items;
    // registers: 72 in FP32 (at 111 and one block per SM P2g takes 205 instead
    // of 177 us at 243^3), 128 in double-float (at 178: 2.75 instead of 1.44 ms)
    static constexpr int MINB = (sizeof(T) == 4 ? 896 : 448) / NT;
    static constexpr int tiles = (H + W - 1) / W;
};

// a * f for an FP32 frequency f
__device__ __forceinline__ cplx<float> freq_mul(cplx<float> a, float f) { return f * a; }
__device__ __forceinline__ cplx<dd> freq_mul(cplx<dd> a, float f) { return dd_scale(a, f); }

// P2g: the three pencils (i, j) of a column; pencil (i, 1) is transformed,
// (i, 2) and (i, 3) are transformed and summed with f2 and f3, into the slots
// (i, 1) and (i, 3).
template <int N, typename T>
__global__ void __launch_bounds__(GradX2<N, T>::NT, GradX2<N, T>::MINB) k_p2_grad(PassArgs a) {
    using S = GradX2<N, T>;
    constexpr int N1 = S::N1, N2 = S::N2, H = S::H, HP = spec_pitch(N), W = S::W, NT = S::NT, P = 3 * W;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cplx<T>* tw = reinterpret_cast<cplx<T>*>(smem_raw);
    cplx<T>* buf = tw + N;  // [3][N][W]
    if (a.cg && a.cg->done) return;
    const int tid = threadIdx.x;
    if (a.red_in && blockIdx.x == 0 && blockIdx.y == 0) {
        // alpha from the block partials of <p, K : p> (as in k_p24)
        double acc = 0.0;
        for (int b = tid; b < a.red_n; b += NT) acc += a.red_in[b];
        acc = block_sum_any(acc);
        if (tid == 0) cg_after_dot(a.cg, acc);
    }
    load_tw<T>(tw, a.tw, N);
    __syncthreads();
    const int col0 = blockIdx.x * W, i = blockIdx.y / N, x1 = blockIdx.y - i * N;
    const long long plane = (long long)N * HP, comp = N * plane;
    cplx<T>* sp = (cplx<T>*)a.out + (3 * i) * comp + x1 * plane;
    for (int it = tid; it < P * N2; it += NT) {
        const int pc = it % P, t = it / P;
        const int s = pc / W, w = pc - s * W, col = col0 + w;
        if (col < H) fwdA<N, N1, T>(sp + s * comp + col, HP, buf + s * N * W + w, W, t, tw);
    }
    __syncthreads();
    for (int it = tid; it < 2 * W * N1; it += NT) {
        // the pencils of one kind first: a warp takes one branch below
        const int s = it / (W * N1), j = it - s * (W * N1);
        const int w = j % W, k1 = j / W, col = col0 + w;
        if (col >= H) continue;
        const cplx<T>* b = buf + s * N * W + w;
        cplx<T> v[N2];
#pragma unroll
        for (int q = 0; q < N2; ++q) v[q] = b[(N2 * k1 + q) * W];
        RegDFT<N, N2, -1, T>::run(v, tw);
        if (s == 1) {
            const float f3 = (float)col;
            cplx<T> u[N2];
#pragma unroll
            for (int q = 0; q < N2; ++q) u[q] = b[(N + N2 * k1 + q) * W];
            RegDFT<N, N2, -1, T>::run(u, tw);
#pragma unroll
            for (int k2 = 0; k2 < N2; ++k2)
                v[k2] = freq_mul(v[k2], (float)signed_freq(k1 + N1 * k2, N)) + freq_mul(u[k2], f3);
        }
        cplx<T>* o = sp + (2 * s) * comp + col;
#pragma unroll
        for (int k2 = 0; k2 < N2; ++k2) o[(long long)(k1 + N1 * k2) * HP] = v[k2];
    }
}

// P4g: from the slots (i, 1), holding f1 a_i, and (i, 3), holding a_i, the
// inverse x2 transforms of f1 a_i, f2 a_i and f3 a_i.
template <int N>
__global__ void __launch_bounds__(GradX2<N, float>::NT) k_p4_grad(PassArgs a) {
    using T = float;
    using S = GradX2<N, T>;
    constexpr int N1 = S::N1, N2 = S::N2, H = S::H, HP = spec_pitch(N), W = S::W, NT = S::NT, P = 3 * W;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cplx<T>* tw = reinterpret_cast<cplx<T>*>(smem_raw);
    cplx<T>* buf = tw + N;  // [3][N][W]
    if (a.cg && a.cg->done) return;
    const int tid = threadIdx.x;
    load_tw<T>(tw, a.tw, N);
    __syncthreads();
    const int col0 = blockIdx.x * W, i = blockIdx.y / N, x1 = blockIdx.y - i * N;
    const long long plane = (long long)N * HP, comp = N * plane;
    cplx<T>* sp = (cplx<T>*)a.out + (3 * i) * comp + x1 * plane;
    for (int it = tid; it < 2 * W * N1; it += NT) {
        // the pencils of one kind first: a warp takes one branch below
        const int s = it / (W * N1), j = it - s * (W * N1);
        const int w = j % W, k1 = j / W, col = col0 + w;
        if (col >= H) continue;
        const cplx<T>* in = sp + (2 * s) * comp + col;
        cplx<T> u[N2];
#pragma unroll
        for (int k2 = 0; k2 < N2; ++k2) u[k2] = in[(long long)(k1 + N1 * k2) * HP];
        // s = 0: f1 a as it is; s = 1: f2 a, then f3 a
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            if (g == 1 && s == 0) break;
            cplx<T> v[N2];
#pragma unroll
            for (int k2 = 0; k2 < N2; ++k2) {
                const T f = s == 0 ? T(1) : g == 0 ? (T)signed_freq(k1 + N1 * k2, N) : (T)col;
                v[k2] = f * u[k2];
            }
            RegDFT<N, N2, +1, T>::run(v, tw);
            cplx<T>* o = buf + (s + g) * N * W + w;
#pragma unroll
            for (int t = 0; t < N2; ++t) {
                cplx<T> z = v[t];
                if (k1 > 0 && t > 0) z = twmul<+1>(z, tw[t * k1]);  // t*k1 < N
                o[(N2 * k1 + t) * W] = z;
            }
        }
    }
    __syncthreads();
    for (int it = tid; it < P * N2; it += NT) {
        const int pc = it % P, t = it / P;
        const int s = pc / W, w = pc - s * W, col = col0 + w;
        if (col < H) invA<N, N1, T>(buf + s * N * W + w, W, sp + s * comp + col, HP, t, tw);
    }
}

// Row pass: inverse x3, tau = K : p (St. Venant-Kirchhoff), <p, tau>, forward
// x3 on R rows, in place on the nine components (five packed rows a row).
// Threads per SM that the registers leave room for, and rounds of spectrum
// loads issued together: 1024 and 1 take 473 us at 243^3 and 72 at 125^3, 768
// and 2 479 and 81, 768 and 3 469 and 80, 1024 and 2 484 and 72. (In the
// iteration on real fields P1 and P5 took 681 + 310 us.)
#ifndef FFTG_FS_ROWS_THREADS
#define FFTG_FS_ROWS_THREADS 1024
#endif
#ifndef FFTG_FS_ROWS_LDB
#define FFTG_FS_ROWS_LDB 1
#endif
template <int N>
struct FsRowCfg {
    static constexpr int fl2(int x) { return x >= 32 ? 32 : x >= 16 ? 16 : x >= 8 ? 8 : 4; }
    static constexpr int N1 = RowSplit<N>::N1, N2 = N / N1;
    static constexpr int R0 = FsCfg<N, float>::R;
    static constexpr int R = R0 < fl2(N * N / 152) ? R0 : fl2(N * N / 152);
    static constexpr int NT0 = ((kFsPairs * R * N2 + 31) / 32) * 32;
    static constexpr int NT = NT0 < 64 ? 64 : NT0 > 256 ? 256 : NT0;
    static constexpr int MINB = FFTG_FS_ROWS_THREADS / NT;
    static constexpr size_t smem = (size_t)(kFsPairs * R * N + N) * 8;
    static constexpr int blocks = (N * N + R - 1) / R;
};

template <int N>
__global__ void __launch_bounds__(FsRowCfg<N>::NT, FsRowCfg<N>::MINB) k_fs_rows_cg(FsArgs a) {
    using T = float;
    using S = FsRowCfg<N>;
    constexpr int R = S::R, H = (N + 1) / 2, HP = spec_pitch(N), NT = S::NT;
    constexpr int N1 = S::N1, N2 = S::N2;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cplx<T>* z = reinterpret_cast<cplx<T>*>(smem_raw);  // [5][R][N]
    cplx<T>* tw = z + kFsPairs * R * N;
    if (a.cg->done) return;
    const int tid = threadIdx.x;
    load_tw<T>(tw, a.tw, N);
    const int row0 = blockIdx.x * R;
    const int nrows = min(R, N * N - row0);
    const long long HS = (long long)N * N * HP;
    cplx<T>* sp = (cplx<T>*)a.out + (long long)row0 * HP;
    constexpr int NRL = (R * H + NT - 1) / NT;
    constexpr int LB = FFTG_FS_ROWS_LDB < NRL ? FFTG_FS_ROWS_LDB : NRL;
#pragma unroll
    for (int r0 = 0; r0 < NRL; r0 += LB) {
        cplx<T> A[LB][kFsComp];
#pragma unroll
        for (int u = 0; u < LB; ++u) {
            const int it = tid + (r0 + u) * NT;
            if (r0 + u < NRL && it < nrows * H) {
                const int row = it / H, o = it + row * (HP - H);
#pragma unroll
                for (int c = 0; c < kFsComp; ++c) A[u][c] = sp[c * HS + o];
            }
        }
#pragma unroll
        for (int u = 0; u < LB; ++u) {
            const int it = tid + (r0 + u) * NT;
            if (r0 + u < NRL && it < nrows * H) {
                const int row = it / H, k = it - row * H;
                const int pk = perm_pos<N, N1>(k);
                const int pn = perm_pos<N, N1>(k == 0 ? 0 : N - k);
#pragma unroll
                for (int c = 0; c < kFsPairs; ++c) {
                    const cplx<T> a0 = A[u][2 * c], b0 = 2 * c + 1 < kFsComp ? A[u][2 * c + 1] : mk(T(0), T(0));
                    cplx<T>* zr = z + (c * R + row) * N;
                    if (k == 0) {
                        zr[pk] = mk(a0.x, b0.x);
                    } else {
                        zr[pk] = mk(a0.x - b0.y, a0.y + b0.x);  // A + iB
                        zr[pn] = mk(a0.x + b0.y, b0.x - a0.y);  // conj(A) + i conj(B)
                    }
                }
            }
        }
    }
    __syncthreads();
    constexpr int NP = kFsPairs * R;
    if (N2 > 1) {
        for (int it = tid; it < NP * N1; it += NT) {
            const int pc = it % NP, k1 = it / NP;
            if (pc % R < nrows) invB<N, N1, false, T>(z + pc * N, 1, z + pc * N, 1, k1, tw);
        }
        __syncthreads();
    }
    for (int it = tid; it < NP * N2; it += NT) {
        const int pc = it % NP, t = it / NP;
        if (pc % R < nrows) invA<N, N1, T>(z + pc * N, 1, z + pc * N, 1, t, tw);
    }
    __syncthreads();
    const long long cs = a.cs, v0 = (long long)row0 * N;
    const T* hg = (const T*)a.hgrad;
    const int nel = nrows * N;
    T pkp = T(0);
    for (int i = tid; i < nel; i += NT) {
        T h[9], d[9], s[9];
#pragma unroll
        for (int c = 0; c < 9; ++c) h[c] = hg[c * cs + v0 + i];
        const double* m = a.lame + 2 * a.phase[v0 + i];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const cplx<T> zz = z[c * R * N + i];
            d[2 * c] = zz.x;
            d[2 * c + 1] = zz.y;
        }
        d[8] = z[4 * R * N + i].x;
        svk_tangent_apply<T>(h, (T)m[0], (T)m[1], d, s);
#pragma unroll
        for (int c = 0; c < 9; ++c) pkp += d[c] * s[c];
#pragma unroll
        for (int c = 0; c < 4; ++c) z[c * R * N + i] = mk(s[2 * c], s[2 * c + 1]);
        z[4 * R * N + i] = mk(s[8], T(0));
    }
    const double part = block_sum_any((double)pkp);  // its first barrier ends the phase
    if (tid == 0) a.partials[blockIdx.x] = part;
    for (int it = tid; it < NP * N2; it += NT) {
        const int pc = it % NP, t = it / NP;
        if (pc % R < nrows) fwdA<N, N1, T>(z + pc * N, 1, z + pc * N, 1, t, tw);
    }
    __syncthreads();
    if (N2 > 1) {
        for (int it = tid; it < NP * N1; it += NT) {
            const int pc = it % NP, k1 = it / NP;
            if (pc % R < nrows) fwdB<N, N1, false, T>(z + pc * N, 1, z + pc * N, 1, k1, tw);
        }
        __syncthreads();
    }
    for (int it = tid; it < nrows * H; it += NT) {
        const int row = it / H, k = it - row * H, o = row * HP + k;
        const int pk = perm_pos<N, N1>(k), pn = perm_pos<N, N1>(k == 0 ? 0 : N - k);
#pragma unroll
        for (int c = 0; c < kFsPairs; ++c) {
            const cplx<T> zk = z[(c * R + row) * N + pk];
            const cplx<T> zn = conj(z[(c * R + row) * N + pn]);
            sp[(2 * c) * HS + o] = half_of(zk + zn);
            if (2 * c + 1 < kFsComp) {
                const cplx<T> d = zk - zn;
                sp[(2 * c + 1) * HS + o] = half_of(mk(d.y, -d.x));
            }
        }
    }
}

// ------------------------------------------------------------------ launcher
// The kernels that the small-strain path has too, with their arguments.
template <typename K>
static cudaError_t launch_fs_x1(K kernel, dim3 grid, int threads, size_t smem, const FsArgs& a, cudaStream_t s) {
    PassArgs b{};
    b.in = a.in;
    b.out = a.out;
    b.aux = a.aux;
    b.aux2 = a.aux2;
    b.aux3 = a.aux3;
    b.cg = a.cg;
    b.partials = a.partials;
    b.tw = a.tw;
    b.scale = a.scale;
    b.red_in = a.red_in;
    b.red_n = a.red_n;
    return launch_k(kernel, grid, smem, b, s, threads);
}

template <int N>
cudaError_t run_fs_pass_n(FsPassKind kind, const FsArgs& a, cudaStream_t s) {
    using C32 = FsCfg<N, float>;
    using C64 = FsCfg<N, double>;
    using CDD = FsCfg<N, dd>;
    static_assert(CDD::row_blocks == C64::row_blocks && CDD::W3 == C64::W3,
                  "double-float passes share the FP64 geometry");
    const dim3 r32(C32::row_blocks), r64(C64::row_blocks);
    const dim3 g32((C32::H + C32::W3 - 1) / C32::W3, N), g64((C64::H + C64::W3 - 1) / C64::W3, N);
    const dim3 x32(X1<N>::tiles, N);
    const size_t m32 = C32::smem_rows, m64 = C64::smem_rows;
    switch (kind) {
        case FK_P1_PLAIN_F64: return launch_fs(k_fs_p1<N, double, FS_P1_PLAIN>, r64, kThreads, m64, a, s);
        case FK_P1_PLAIN_F32: return launch_fs(k_fs_p1<N, float, FS_P1_PLAIN>, r32, kThreads, m32, a, s);
        case FK_P1_TAN_F64: return launch_fs(k_fs_p1<N, double, FS_P1_TAN>, r64, kThreads, m64, a, s);
        case FK_P1_TAN_F32: return launch_fs(k_fs_p1<N, float, FS_P1_TAN>, r32, kThreads, m32, a, s);
        case FK_P1_CG_F64: return launch_fs(k_fs_p1<N, double, FS_P1_CG>, r64, kThreads, m64, a, s);
        case FK_P2_F64: return launch_fs_p24<N, double, true>(a, s);
        case FK_P2_F32: return launch_fs_p24<N, float, true>(a, s);
        case FK_P4_F64: return launch_fs_p24<N, double, false>(a, s);
        case FK_P4_F32: return launch_fs_p24<N, float, false>(a, s);
        case FK_P3_F64: return launch_fs(k_fs_p3<N, double>, g64, C64::T3, C64::smem_p3, a, s);
        case FK_P3_F32: return launch_fs(k_fs_p3<N, float>, g32, C32::T3, C32::smem_p3, a, s);
        case FK_P5_PLAIN_F64: return launch_fs(k_fs_p5<N, double, FS_P5_PLAIN, double>, r64, kThreads, m64, a, s);
        case FK_P5_PLAIN_F32: return launch_fs(k_fs_p5<N, float, FS_P5_PLAIN, float>, r32, kThreads, m32, a, s);
        case FK_P5_DOT_F64: return launch_fs(k_fs_p5<N, double, FS_P5_DOT, double>, r64, kThreads, m64, a, s);
        case FK_P5_DOT_F32: return launch_fs(k_fs_p5<N, float, FS_P5_DOT, float>, r32, kThreads, m32, a, s);
        case FK_P5_RHS_F64_TO_F64:
            return launch_fs(k_fs_p5<N, double, FS_P5_RHS, double>, r64, kThreads, m64, a, s);
        case FK_P1_PLAIN_DD: return launch_fs(k_fs_p1<N, dd, FS_P1_PLAIN>, r64, kThreads, m64, a, s);
        case FK_P2_DD: return launch_fs_p24<N, dd, true>(a, s);
        case FK_P4_DD: return launch_fs_p24<N, dd, false>(a, s);
        case FK_P3_DD: return launch_fs(k_fs_p3<N, dd>, g64, CDD::T3, CDD::smem_p3, a, s);
        case FK_P5_PLAIN_DD_TO_F64:
            return launch_fs(k_fs_p5<N, dd, FS_P5_PLAIN, double>, r64, kThreads, m64, a, s);
        case FK_P1_TANRHS_F64: return launch_fs(k_fs_p1<N, double, FS_P1_TANRHS>, r64, kThreads, m64, a, s);
        case FK_P1_TANRHS_F32: return launch_fs(k_fs_p1<N, float, FS_P1_TANRHS>, r32, kThreads, m32, a, s);
        case FK_P5_NEWTON_F32: return launch_fs(k_fs_p5<N, float, FS_P5_NEWTON, float>, r32, kThreads, m32, a, s);
        case FK_X1I_CG_F32: return launch_fs_x1(k_x1i<N, X1I_CG, true>, x32, X1<N>::NT, X1<N>::smem, a, s);
        case FK_X1I_SOLUTION_F32:
            return launch_fs_x1(k_x1i<N, X1I_SOLUTION, true>, x32, X1<N>::NT, X1<N>::smem, a, s);
        case FK_X1F_CG_F32: return launch_fs_x1(k_x1f<N, X1F_CG, true>, x32, X1<N>::NT, X1<N>::smem, a, s);
        case FK_X1F_RHS_F32: return launch_fs_x1(k_x1f<N, X1F_RHS, true>, x32, X1<N>::NT, X1<N>::smem, a, s);
        case FK_X1F_RHS_DD: {
            using X = X1dd<N>;
            return launch_fs_x1(k_x1f_dd<N, true>, dim3((X::H + X::W3 - 1) / X::W3, N), X::T3, X::smem_p3, a, s);
        }
        case FK_P4_GRAD_F32: {
            using G = GradX2<N, float>;
            return launch_fs_x1(k_p4_grad<N>, dim3(G::tiles, 3 * N), G::NT, G::smem, a, s);
        }
        case FK_P2_GRAD_F32: {
            using G = GradX2<N, float>;
            return launch_fs_x1(k_p2_grad<N, float>, dim3(G::tiles, 3 * N), G::NT, G::smem, a, s);
        }
        case FK_P2_GRAD_DD: {
            using G = GradX2<N, dd>;
            return launch_fs_x1(k_p2_grad<N, dd>, dim3(G::tiles, 3 * N), G::NT, G::smem, a, s);
        }
        case FK_ROWS_CG_F32: {
            using G = FsRowCfg<N>;
            return launch_fs(k_fs_rows_cg<N>, dim3(G::blocks), G::NT, G::smem, a, s);
        }
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace fftg
