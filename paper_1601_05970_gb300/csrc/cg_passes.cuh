// The FP32 CG iteration of the mixed path on displacement coefficients.
//
// Every vector of the projected CG is compatible, so at each frequency f it
// is f(x)w + w(x)f for one complex 3-vector w (the displacement coefficient,
// up to a constant factor). r, p and x are held as w on the half spectrum
// (tile by tile, below): half the bytes of a six-component real field and
// compatible whatever they hold, and only p is ever taken to real space, where
// C : p is formed. (On the plane f3 = 0 both f and -f are stored, and rounding
// can leave w there a little off the symmetry of a real field's; the row pass
// drops that part of p, <r, r> counts that of r. It is of the size of a few
// roundings, where the inner solves stop at 1e-5.)
//
//
//   x1i   p = r + beta p, x += alpha p_old; f(x)p + p(x)f; inverse x1
//   P4    inverse x2 (the column pass of passes.cuh)
//   rows  inverse x3, tau = C : p with <p, tau>, forward x3, in one pass
//   P2    forward x2 (its first block sets alpha = <r, r> / <p, tau>)
//   x1f   forward x1, w of Ghat : tau, r -= alpha w, <r, r>
//
// Ghat (Appendix A) in this form: with t = tau f and q = |f|^2,
//   w = (t - (f.t) / (2 q) f) / q,  Ghat : tau = f(x)w + w(x)f,
// which is n(x)u + u(x)n for n = f/|f|, u = |f| w. The Frobenius product of
// two fields is N^3 times the sum over frequencies of 2 (q a.b + (f.a)(f.b))
// (Parseval; the half spectrum counts f3 > 0 twice).
//
// An iteration moves 84.3 (x1i) + 2 x 48.2 (P4, P2) + 76.2 (rows) + 48.2
// (x1f) = 305 B per voxel at 243^3; with r, p and x as real fields it moved
// 388.8 (243^3: 1.12 -> 0.95 ms an iteration). The residual of a Newton
// iteration and a column's right-hand side stop at w (x1f), and the solution is
// taken to real space once (x1i, P4, P5), which makes a projection of it
// needless.
#pragma once

#include "passes.cuh"

namespace fftg {

enum : int { X1F_CG = 0, X1F_RHS = 1 };
enum : int { X1I_CG = 0, X1I_SOLUTION = 1 };

// x1 split N = N1 * N2 of the two passes: on small grids two stages rather
// than one, so that a column has more threads.
template <int N>
struct X1Split {
    static constexpr int N1 = N == 225 ? 25 : N == 27 ? 9 : N == 25 || N == 15 ? 5 : N == 9 ? 3 : Plan<N>::N1;
};

// Blocks of the x1 passes: W columns (64-byte runs of the spectrum), as many
// blocks per SM as shared memory allows up to four, about 1000 threads an SM
// among them and at most one stage-A item a thread. Stage B and the
// frequency points are phases of their own (28 warps an SM at 243^3): with a
// column's N2 frequencies in one thread's registers (14 warps) x1i and x1f
// took 282 and 210 us there, in this form 283 and 203 us, and with the
// vectors stored tile by tile (below) 234 and 179 us, 5.2 and 3.9 TB/s. Tiles
// of three components and twice the blocks: 303 and 228 us.
template <int N>
struct X1 {
    static constexpr int N1 = X1Split<N>::N1, N2 = N / N1, H = (N + 1) / 2, HP = spec_pitch(N), W = 8;
    static constexpr size_t smem = (size_t)(6 * N * W + N) * 8;
    static constexpr int NB0 = (int)(220 * 1024 / smem), NB = NB0 > 4 ? 4 : NB0;
    static constexpr int items = ((6 * W * N2 + 31) / 32) * 32, most = 1024 / NB;
    static constexpr int NT = items < most ? items : most;
    static constexpr int MINB = N1 > 15 && NB == 4 ? 3 : 1024 / NT;  // 64 registers; 25-point DFTs 85
    static constexpr int tiles = (H + W - 1) / W, blocks = tiles * N;
    static_assert(valid_split(N, N1) && W == kCoefTile, "x1 tiles of column pairs");
};

// Only the x1 passes touch the vectors, so these are laid out as their
// blocks take them: [nf][N (x2)][tiles][3][N (x1)][W], a block's part one run
// of 24 N W bytes (the columns past H in the last tile are never read back).
template <int N>
__device__ __forceinline__ long long coef_field() { return 3LL * N * N * X1<N>::tiles * X1<N>::W; }
template <int N>
__device__ __forceinline__ long long coef_tile(int tile, int k2) {
    return ((long long)k2 * X1<N>::tiles + tile) * (3 * N * X1<N>::W);
}

__device__ __forceinline__ void ld_pair(const cplx<float>* p, cplx<float> (&v)[2]) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    v[0] = mk(t.x, t.y);
    v[1] = mk(t.z, t.w);
}
__device__ __forceinline__ void st_pair(cplx<float>* p, const cplx<float> (&v)[2]) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
}

// Coefficients are stored times a power of two near N^(5/2) / 2, which
// brings those of a field of white noise to the size of the field's values:
// without it the FP32 squares of a converged residual's coefficients, smaller
// than its values by that factor, would underflow.
template <int N>
struct CoefScale {
    static constexpr int exponent() {
        double t = 0.25 * N * N * N * N * (double)N;
        int e = 0;
        for (; t >= 4.0; t *= 0.25) ++e;
        return e;
    }
    static constexpr float value = (float)(1 << exponent());
    static constexpr float inverse = 1.0f / value;
    // sum over voxels of a squared field from sum (q |w|^2 + |f.w|^2); half
    // of it from sum q |a|^2 of a gradient field
    static constexpr double square = 2.0 * N * N * (double)N / ((double)value * (double)value);
};

// Component of the nine of a finite-strain spectrum that holds field c of the
// six the x1 passes take: (i, 1) for the fields that f1 multiplies, (i, 3) for
// the others.
__device__ __forceinline__ int fs_slot(int c) { return c < 3 ? 3 * c : 3 * (c - 3) + 2; }

__device__ __forceinline__ int signed_freq(int k, int N) { return k <= (N - 1) / 2 ? k : k - N; }

// Rounds of spectrum loads of the row pass issued together: with 4 it takes
// 248 us at 243^3, with 2 261 us. Fetching the tangent to L2 ahead of its use
// (a bulk prefetch at the block's start) made it 16 us slower; C : p in the
// registers of the N1-point stage (9 points of all three packed rows, a
// shared-memory pass less, 80 registers) 290 us.
#ifndef FFTG_ROWS_LDB
#define FFTG_ROWS_LDB 4
#endif

// ---------------------------------------------------------------- x1 inverse
// aux = r (X1I_CG), aux2 = p, aux3 = x, out = spectrum; fields of 3 N N HP
// coefficients. X1I_CG updates p and x; X1I_SOLUTION takes x (+ the pending
// alpha p) to the spectrum. x holds a value once a step was added to it: the
// first step of a solve writes x = alpha p, so x needs no clearing.
//
// A thread takes column pairs (16-byte loads; the pair past an odd H is
// padding of the row pitch), then stage B and stage A of the inverse run on
// the tile in shared memory.
//
// FS (finite strain): the vectors are a_i of gradient fields a(x)f, and six
// fields go on: f1 a_i and a_i (the x2 pass applies f2 and f3 to the latter).
template <int N, int MODE, bool FS, int NT, bool GROUP>
__device__ __forceinline__ void x1i_tile(int tile, int k2g, int it, float alpha, float beta, bool pend,
                                         const cplx<float>* r, cplx<float>* p, cplx<float>* x, cplx<float>* sp,
                                         cplx<float>* buf, const cplx<float>* tw, int tid, int bar) {
    using T = float;
    using S = X1<N>;
    constexpr int N1 = S::N1, N2 = S::N2, H = S::H, HP = S::HP, W = S::W;
    const int col0 = tile * W;
    const long long NH = (long long)N * HP, vo = coef_tile<N>(tile, k2g);
    r += vo;
    p += vo;
    x += vo;
    sp += (long long)k2g * HP;
    // X1I_CG: iteration it adds step it - 1. X1I_SOLUTION: x holds a value
    // after step it - 1 was added, by the iteration that followed it.
    const bool has_x = MODE == X1I_CG ? it > 1 : (pend ? it > 1 : it > 0);
    constexpr T is = CoefScale<N>::inverse;
    const T g2 = is * (T)signed_freq(k2g, N);
    for (int j = tid; j < (W / 2) * N; j += NT) {
        const int w = 2 * (j % (W / 2)), kk = j / (W / 2), col = col0 + w;
        if (col >= H) continue;
        const int o = kk * W + w;
        cplx<T> d[3][2], po[3][2], xo[3][2];
        if (MODE == X1I_CG) {
#pragma unroll
            for (int i = 0; i < 3; ++i) ld_pair(r + o + i * N * W, d[i]);
            if (it > 0) {
#pragma unroll
                for (int i = 0; i < 3; ++i) ld_pair(p + o + i * N * W, po[i]);
                if (has_x) {
#pragma unroll
                    for (int i = 0; i < 3; ++i) ld_pair(x + o + i * N * W, xo[i]);
                }
#pragma unroll
                for (int i = 0; i < 3; ++i) {
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        xo[i][e] = has_x ? xo[i][e] + alpha * po[i][e] : alpha * po[i][e];
                        d[i][e] = d[i][e] + beta * po[i][e];
                    }
                    st_pair(x + o + i * N * W, xo[i]);
                }
            }
#pragma unroll
            for (int i = 0; i < 3; ++i) st_pair(p + o + i * N * W, d[i]);
        } else {
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                if (has_x) {
                    ld_pair(x + o + i * N * W, d[i]);
                } else {
                    d[i][0] = d[i][1] = mk(T(0), T(0));
                }
                if (pend) {
                    ld_pair(p + o + i * N * W, po[i]);
#pragma unroll
                    for (int e = 0; e < 2; ++e) d[i][e] = d[i][e] + alpha * po[i][e];
                }
            }
        }
        // f(x)d + d(x)f at the frequency's place in permuted order
        const T g1 = is * (T)signed_freq(kk, N);
        cplx<T>* b = buf + perm_pos<N, N1>(kk) * W + w;
        cplx<T> v[6][2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            if (FS) {
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    v[i][e] = g1 * d[i][e];
                    v[3 + i][e] = is * d[i][e];
                }
                continue;
            }
            const T g3 = is * (T)(col + e);
            v[0][e] = (g1 + g1) * d[0][e];
            v[1][e] = (g2 + g2) * d[1][e];
            v[2][e] = (g3 + g3) * d[2][e];
            v[3][e] = g2 * d[2][e] + g3 * d[1][e];
            v[4][e] = g1 * d[2][e] + g3 * d[0][e];
            v[5][e] = g1 * d[1][e] + g2 * d[0][e];
        }
#pragma unroll
        for (int c = 0; c < 6; ++c) st_pair(b + c * N * W, v[c]);
    }
    tile_sync<NT, GROUP>(bar);
    constexpr int P = 6 * W;
    if (N2 > 1) {
        for (int j = tid; j < P * N1; j += NT) {
            const int pc = j % P, k1 = j / P;
            const int c = pc / W, w = pc - c * W;
            if (col0 + w < H) invB<N, N1, false, T>(buf + c * N * W + w, W, buf + c * N * W + w, W, k1, tw);
        }
        tile_sync<NT, GROUP>(bar);
    }
    for (int j = tid; j < P * N2; j += NT) {
        const int pc = j % P, t = j / P;
        const int c = pc / W, w = pc - c * W, col = col0 + w;
        const int comp = FS ? fs_slot(c) : c;
        if (col < H) invA<N, N1, T>(buf + c * N * W + w, W, sp + comp * N * NH + col, (int)NH, t, tw);
    }
}

template <int N, int MODE, bool FS = false>
__global__ void __launch_bounds__(X1<N>::NT, X1<N>::MINB) k_x1i(PassArgs a) {
    using T = float;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cplx<T>* buf = reinterpret_cast<cplx<T>*>(smem_raw);  // [6][N][W]
    cplx<T>* tw = buf + 6 * N * X1<N>::W;
    const int f = blockIdx.z;
    if (a.active && !a.active[f]) return;
    const CGState* cg = a.cg + f;
    if (MODE == X1I_CG && cg->done) return;
    load_tw<T>(tw, a.tw, N);
    const long long vf = f * coef_field<N>();
    x1i_tile<N, MODE, FS, X1<N>::NT, false>(blockIdx.x, blockIdx.y, cg->it, (T)cg->alpha, (T)cg->beta, cg->pend != 0,
                                            (const cplx<T>*)a.aux + vf, (cplx<T>*)a.aux2 + vf,
                                            (cplx<T>*)a.aux3 + vf, (cplx<T>*)a.out + f * a.sstride, buf, tw,
                                            threadIdx.x, 0);
}

// Sum of in[0 .. n) by one warp in a fixed order, in every lane.
__device__ __forceinline__ double warp_total(const double* in, int n, int lane) {
    double acc = 0.0;
    for (int b = lane; b < n; b += 32) acc += __ldcg(in + b);
    return warp_sum(acc);
}

// ---------------------------------------------------------------- x1 forward
// in = spectrum of tau, aux3 = r. X1F_CG: r -= alpha w and the block's part
// of <r, r>; X1F_RHS: r = w with scale the sign and 1/N^3 of the right-hand
// side, and the parts of <r, r> and of ||G tau||^2.
// FS: t_i = f1 A_i1 + B_i of the six fields that the x2 pass leaves, w = t / q.
//
// A thread's part of the sum over its tile: in FP32 for <r, r>, and in FP64 for
// the norm of a right-hand side.
struct X1fSums {
    float rr;
    double norm;
};
template <int N, int MODE, bool FS, int NT, bool GROUP>
__device__ __forceinline__ X1fSums x1f_tile(int tile, int k2g, float step, const cplx<float>* sp, cplx<float>* r,
                                          cplx<float>* buf, const cplx<float>* tw, int tid, int bar) {
    using T = float;
    using S = X1<N>;
    constexpr int N1 = S::N1, N2 = S::N2, H = S::H, HP = S::HP, W = S::W;
    const int col0 = tile * W;
    const long long NH = (long long)N * HP;
    sp += (long long)k2g * HP;
    r += coef_tile<N>(tile, k2g);
    constexpr int P = 6 * W;
    for (int j = tid; j < P * N2; j += NT) {
        const int pc = j % P, t = j / P;
        const int c = pc / W, w = pc - c * W, col = col0 + w;
        const int comp = FS ? fs_slot(c) : c;
        if (col < H) fwdA<N, N1, T>(sp + comp * N * NH + col, (int)NH, buf + c * N * W + w, W, t, tw);
    }
    tile_sync<NT, GROUP>(bar);
    if (N2 > 1) {
        for (int j = tid; j < P * N1; j += NT) {
            const int pc = j % P, k1 = j / P;
            const int c = pc / W, w = pc - c * W;
            if (col0 + w < H) fwdB<N, N1, false, T>(buf + c * N * W + w, W, buf + c * N * W + w, W, k1, tw);
        }
        tile_sync<NT, GROUP>(bar);
    }
    const T f2 = (T)signed_freq(k2g, N);
    X1fSums sums{0.0f, 0.0};
    for (int j = tid; j < (W / 2) * N; j += NT) {
        const int w = 2 * (j % (W / 2)), kk = j / (W / 2), col = col0 + w;
        if (col >= H) continue;
        const int o = kk * W + w;
        cplx<T> z[3][2];
        if (MODE == X1F_CG) {
#pragma unroll
            for (int i = 0; i < 3; ++i) ld_pair(r + o + i * N * W, z[i]);
        }
        const cplx<T>* b = buf + perm_pos<N, N1>(kk) * W + w;
        cplx<T> c[6][2];
#pragma unroll
        for (int k = 0; k < 6; ++k) ld_pair(b + k * N * W, c[k]);
        const T f1 = (T)signed_freq(kk, N);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const T f3 = (T)(col + e);
            const T q = f1 * f1 + f2 * f2 + f3 * f3;
            const T iq = q > T(0) ? __frcp_rn(q) : T(0);  // the mean maps to zero
            const T m = step * iq;
            cplx<T> t0, t1, t2;
            if (FS) {
                t0 = m * (f1 * c[0][e] + c[3][e]);
                t1 = m * (f1 * c[1][e] + c[4][e]);
                t2 = m * (f1 * c[2][e] + c[5][e]);
            } else {
                t0 = f1 * c[0][e] + f2 * c[5][e] + f3 * c[4][e];
                t1 = f1 * c[5][e] + f2 * c[1][e] + f3 * c[3][e];
                t2 = f1 * c[4][e] + f2 * c[3][e] + f3 * c[2][e];
                const cplx<T> h = (T(-0.5) * iq) * (f1 * t0 + f2 * t1 + f3 * t2);
                t0 = m * (t0 + f1 * h);
                t1 = m * (t1 + f2 * h);
                t2 = m * (t2 + f3 * h);
            }
            z[0][e] = MODE == X1F_CG ? z[0][e] + t0 : t0;
            z[1][e] = MODE == X1F_CG ? z[1][e] + t1 : t1;
            z[2][e] = MODE == X1F_CG ? z[2][e] + t2 : t2;
            const cplx<T> fr = FS ? mk(T(0), T(0)) : f1 * z[0][e] + f2 * z[1][e] + f3 * z[2][e];
            const T s = z[0][e].x * z[0][e].x + z[0][e].y * z[0][e].y + z[1][e].x * z[1][e].x +
                        z[1][e].y * z[1][e].y + z[2][e].x * z[2][e].x + z[2][e].y * z[2][e].y;
            // f3 > 0 stands for -f3 too; the column past an odd H is padding
            const T part = q * s + fr.x * fr.x + fr.y * fr.y;
            if (col + e < H) {
                const T both = col + e == 0 ? part : T(2) * part;
                sums.rr += both;
                if (MODE == X1F_RHS) sums.norm += (double)both;
            }
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) st_pair(r + o + i * N * W, z[i]);
    }
    return sums;
}

template <int N, int MODE, bool FS = false>
__global__ void __launch_bounds__(X1<N>::NT, X1<N>::MINB) k_x1f(PassArgs a) {
    using T = float;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cplx<T>* buf = reinterpret_cast<cplx<T>*>(smem_raw);  // [6][N][W]
    cplx<T>* tw = buf + 6 * N * X1<N>::W;
    const int f = blockIdx.z;
    if (a.active && !a.active[f]) return;
    const CGState* cg = a.cg + f;
    if (MODE == X1F_CG && cg->done) return;
    load_tw<T>(tw, a.tw, N);
    __syncthreads();
    const double unit = (double)CoefScale<N>::value * a.scale;
    const X1fSums sums = x1f_tile<N, MODE, FS, X1<N>::NT, false>(
        blockIdx.x, blockIdx.y, MODE == X1F_CG ? (T)(-cg->alpha * unit) : (T)unit,
        (const cplx<T>*)a.in + f * a.sstride, (cplx<T>*)a.aux3 + f * coef_field<N>(), buf, tw, threadIdx.x, 0);
    const double square = (FS ? 0.5 : 1.0) * CoefScale<N>::square;
    const double s = block_sum_any((double)sums.rr) * square;
    const double norm = MODE == X1F_RHS ? block_sum_any(sums.norm) * square : 0.0;
    if (threadIdx.x == 0) {
        const size_t b = blockIdx.y * gridDim.x + blockIdx.x, nb = (size_t)gridDim.x * gridDim.y;
        if (MODE == X1F_CG) {
            a.partials[f * nb + b] = s;
        } else {
            a.partials[2 * (f * nb + b)] = s;
            a.partials[2 * (f * nb + b) + 1] = norm;
        }
    }
}

// 1/q of a positive integer q < 2^24 as a double-float: the remainder
// 1 - q y of the FP32 quotient y is exact in one fma, so y + y (1 - q y)
// leaves a relative error of (1 - q y)^2, about 2^-48.
__device__ __forceinline__ dd dd_recip(float q) {
    const float y = 1.0f / q;
    return dd(y, y * dd_fma(-q, y, 1.0f));
}

// a * f for an FP32 number f
__device__ __forceinline__ dd dd_scale(dd a, float f) {
    const dd p = dd_two_prod(a.hi, f);
    return dd_fast_two_sum(p.hi, dd_fma(a.lo, f, p.lo));
}
__device__ __forceinline__ cplx<dd> dd_scale(cplx<dd> a, float f) {
    return mk(dd_scale(a.x, f), dd_scale(a.y, f));
}

// The right-hand side of a Newton iteration, r = w of -G sigma, from the
// double-float spectrum of the FP64 stress: forward x1 in two stages, then
// one thread per frequency. The double-float inverse passes that a residual
// in real space needs (half of its work) are not run.
// Small grids take two stages (a double-float DFT of 27 points in one thread
// needs more registers than there are).
template <int N>
using X1dd = Cfg<N, dd, N <= 27 ? X1Split<N>::N1 : Plan<N>::N1>;

template <int N, bool FS = false>
__global__ void __launch_bounds__(X1dd<N>::T3) k_x1f_dd(PassArgs a) {
    using T = dd;
    using C = X1dd<N>;
    constexpr int H = C::H, HP = C::HP, W = C::W3, NT = C::T3;
    constexpr int N1 = C::PN1, N2 = C::PN2;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cplx<T>* tw = reinterpret_cast<cplx<T>*>(smem_raw);
    cplx<T>* buf = tw + N;  // [6][N][W]
    const int f = blockIdx.z;
    if (a.active && !a.active[f]) return;
    const int tid = threadIdx.x;
    load_tw<T>(tw, a.tw, N);
    __syncthreads();
    const int col0 = blockIdx.x * W, k2g = blockIdx.y;
    const long long NH = (long long)N * HP;
    const cplx<T>* sp = (const cplx<T>*)a.in + f * a.sstride + (long long)k2g * HP;
    cplx<float>* r = (cplx<float>*)a.aux3 + f * coef_field<N>();
    constexpr int P = 6 * W;
    for (int it = tid; it < P * N2; it += NT) {
        const int pc = it % P, t = it / P;
        const int c = pc / W, w = pc - c * W, col = col0 + w;
        const int comp = FS ? fs_slot(c) : c;
        if (col < H) fwdA<N, N1, T>(sp + comp * N * NH + col, (int)NH, buf + c * N * W + w, W, t, tw);
    }
    __syncthreads();
    if (N2 > 1) {
        for (int it = tid; it < P * N1; it += NT) {
            const int pc = it % P, k1 = it / P;
            const int c = pc / W, w = pc - c * W;
            if (col0 + w < H) fwdB<N, N1, false, T>(buf + c * N * W + w, W, buf + c * N * W + w, W, k1, tw);
        }
        __syncthreads();
    }
    const float f2 = (float)signed_freq(k2g, N);
    const dd scale((double)CoefScale<N>::value * a.scale);
    // <r0, r0> in double-float; the norm before rounding in FP64, a double-float a
    // frequency
    dd acc0(0.0f, 0.0f);
    double acc1 = 0.0;
    for (int it = tid; it < W * N; it += NT) {
        const int w = it % W, pos = it / W, col = col0 + w;
        const int k1 = pos / N2, k2 = pos - k1 * N2;
        const int kk = k1 + N1 * k2;  // frequency held at position N2*k1 + k2
        if (col >= H) continue;
        const float f1 = (float)signed_freq(kk, N), f3 = (float)col;
        const cplx<T>* b = buf + pos * W + w;
        cplx<T> c[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) c[k] = b[k * N * W];
        cplx<T> t[3];
        const float q = f1 * f1 + f2 * f2 + f3 * f3;  // an integer below 2^24: exact
        const dd iq = q > 0.0f ? dd_recip(q) : dd(0.0f, 0.0f);
        const dd m = scale * iq;
        if (FS) {
#pragma unroll
            for (int i = 0; i < 3; ++i) t[i] = m * (dd_scale(c[i], f1) + c[3 + i]);
        } else {
            t[0] = dd_scale(c[0], f1) + dd_scale(c[5], f2) + dd_scale(c[4], f3);
            t[1] = dd_scale(c[5], f1) + dd_scale(c[1], f2) + dd_scale(c[3], f3);
            t[2] = dd_scale(c[4], f1) + dd_scale(c[3], f2) + dd_scale(c[2], f3);
            const cplx<T> h = signed_by<-1>(
                half_of(iq * (dd_scale(t[0], f1) + dd_scale(t[1], f2) + dd_scale(t[2], f3))));
            t[0] = m * (t[0] + dd_scale(h, f1));
            t[1] = m * (t[1] + dd_scale(h, f2));
            t[2] = m * (t[2] + dd_scale(h, f3));
        }
        const float wt = col == 0 ? 1.0f : 2.0f;  // f3 > 0 stands for -f3 too
        constexpr int WX = X1<N>::W;
        const long long o = coef_tile<N>(col / WX, k2g) + kk * WX + col % WX;
        float s0 = 0.0f;
        cplx<float> fr = mk(0.0f, 0.0f);
        dd s1(0.0f, 0.0f);
        cplx<T> ft = mk(dd(0.0f, 0.0f), dd(0.0f, 0.0f));
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const float fi = i == 0 ? f1 : i == 1 ? f2 : f3;
            const cplx<float> z = mk((float)t[i].x, (float)t[i].y);
            r[o + i * N * WX] = z;
            s0 += z.x * z.x + z.y * z.y;
            fr = fr + fi * z;
            s1 += t[i].x * t[i].x + t[i].y * t[i].y;
            ft = ft + dd_scale(t[i], fi);
        }
        if (FS) {
            acc0 += dd(wt * q * s0, 0.0f);
            acc1 += (double)dd_scale(dd_scale(s1, q), wt);
        } else {
            acc0 += dd(wt * (q * s0 + fr.x * fr.x + fr.y * fr.y), 0.0f);
            acc1 += (double)dd_scale(dd_scale(s1, q) + ft.x * ft.x + ft.y * ft.y, wt);
        }
    }
    const double square = (FS ? 0.5 : 1.0) * CoefScale<N>::square;
    const double s0 = block_sum_any((double)acc0) * square;
    const double s1 = block_sum_any(acc1) * square;
    if (tid == 0) {
        const size_t b = blockIdx.y * gridDim.x + blockIdx.x, nb = (size_t)gridDim.x * gridDim.y;
        a.partials[2 * (f * nb + b)] = s0;
        a.partials[2 * (f * nb + b) + 1] = s1;
    }
}

// ---------------------------------------------------------------------- rows
// Radix split of the rows: the plan's, or two stages on the small grids,
// where a row of one stage has too few threads.
template <int N>
struct RowSplit {
    static constexpr int N1 = Plan<N>::N2 > 1 ? Plan<N>::N1 : X1Split<N>::N1;
    static constexpr int ALT = Plan<N>::N2 > 1 ? Plan<N>::N2 : Plan<N>::N1;
};

// Inverse x3, tau = C : p, forward x3 on R rows, in place on the spectrum.
// Rows per block: the row passes' rule, but enough blocks to fill the chip
// on small grids; threads: one stage-A item each.
template <int N, int NA, int TV>
struct RowCfg {
    using C = Cfg<N, float, NA, TV>;
    static constexpr int fl2(int x) {
        return x >= 64 ? 64 : x >= 32 ? 32 : x >= 16 ? 16 : x >= 8 ? 8 : 4;
    }
    static constexpr int R = C::R < fl2(N * N / 152) ? C::R : fl2(N * N / 152);
    static constexpr int N1 = NA, N2 = N / NA;
    static constexpr int NT0 = ((3 * R * N2 + 31) / 32) * 32;
    static constexpr int NT = NT0 < 64 ? 64 : NT0 > 448 ? 448 : NT0;
    static constexpr int MINB = 1024 / NT;  // 64 registers
    static constexpr size_t smem = (size_t)(3 * R * N + N) * 8;
    static constexpr int blocks = (N * N + R - 1) / R;
};

// `sp` and `tg` are those of the rows row0 .. row0 + R of `rows`; the spectrum
// has the pitch HP and component stride HS (global or shared memory), and the
// tangent is read VW voxels a lane (VW = 2: even offsets).
template <int N, int N1, int R, int NT, bool GROUP, int HP, int VW>
__device__ __forceinline__ void rows_tile(int row0, int rows, cplx<float>* sp, long long HS, const float* tg,
                                          long long cs, cplx<float>* z, const cplx<float>* tw, double* warp_part,
                                          int tid, int bar) {
    using T = float;
    constexpr int H = (N + 1) / 2, N2 = N / N1;
    const int nrows = min(R, rows - row0);
    sp += (long long)row0 * HP;
    tg += (long long)row0 * N;
    // the half spectra of two real components -> one complex row; the
    // imaginary parts at k = 0 are rounding and are dropped
    constexpr int NRL = (R * H + NT - 1) / NT;
    constexpr int LB = FFTG_ROWS_LDB < NRL ? FFTG_ROWS_LDB : NRL;
#pragma unroll
    for (int r0 = 0; r0 < NRL; r0 += LB) {
        cplx<T> A[LB][3], B[LB][3];
#pragma unroll
        for (int u = 0; u < LB; ++u) {
            const int it = tid + (r0 + u) * NT;
            if (r0 + u < NRL && it < nrows * H) {
                const int row = it / H, o = it + row * (HP - H);
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    A[u][c] = sp[(2 * c) * HS + o];
                    B[u][c] = sp[(2 * c + 1) * HS + o];
                }
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
                for (int c = 0; c < 3; ++c) {
                    const cplx<T> a0 = A[u][c], b0 = B[u][c];
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
    tile_sync<NT, GROUP>(bar);
    constexpr int NP = 3 * R;
    if (N2 > 1) {
        for (int it = tid; it < NP * N1; it += NT) {
            const int pc = it % NP, k1 = it / NP;
            if (pc % R < nrows) invB<N, N1, false, T>(z + pc * N, 1, z + pc * N, 1, k1, tw);
        }
        tile_sync<NT, GROUP>(bar);
    }
    for (int it = tid; it < NP * N2; it += NT) {
        const int pc = it % NP, t = it / NP;
        if (pc % R < nrows) invA<N, N1, T>(z + pc * N, 1, z + pc * N, 1, t, tw);
    }
    tile_sync<NT, GROUP>(bar);
    // tau = C : p (VW = 2: R N is even; in the last block the vector that
    // straddles the end of the grid reads the padding of the tangent and
    // changes rows that no stage reads)
    const int nel = nrows * N;
    T pcp = T(0);
    for (int j = tid; j < (R * N) / VW; j += NT) {
        const int i0 = j * VW;
        if (i0 >= nel) continue;
        T t7[7][VW];
#pragma unroll
        for (int k = 0; k < 7; ++k) ldv<VW, T>(tg + k * cs + i0, t7[k]);
        cplx<T> s[3][VW];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const cplx<T>* zc = z + c * R * N + i0;
            if constexpr (VW == 2)
                ld_pair(zc, s[c]);
            else
                s[c][0] = zc[0];
        }
#pragma unroll
        for (int e = 0; e < VW; ++e) {
            const T pe[6] = {s[0][e].x, s[0][e].y, s[1][e].x, s[1][e].y, s[2][e].x, s[2][e].y};
            T se[6];
            apply_tangent7<T>(t7[0][e], t7[1][e], t7[2][e], t7[3][e], t7[4][e], t7[5][e], t7[6][e], pe, se);
            if (i0 + e < nel) pcp += frob<T>(pe, se);
#pragma unroll
            for (int c = 0; c < 3; ++c) s[c][e] = mk(se[2 * c], se[2 * c + 1]);
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            cplx<T>* zc = z + c * R * N + i0;
            if constexpr (VW == 2)
                st_pair(zc, s[c]);
            else
                zc[0] = s[c][0];
        }
    }
    {
        const double wv = warp_sum((double)pcp);
        if ((tid & 31) == 0) warp_part[tid >> 5] = wv;
    }
    tile_sync<NT, GROUP>(bar);
    for (int it = tid; it < NP * N2; it += NT) {
        const int pc = it % NP, t = it / NP;
        if (pc % R < nrows) fwdA<N, N1, T>(z + pc * N, 1, z + pc * N, 1, t, tw);
    }
    tile_sync<NT, GROUP>(bar);
    if (N2 > 1) {
        for (int it = tid; it < NP * N1; it += NT) {
            const int pc = it % NP, k1 = it / NP;
            if (pc % R < nrows) fwdB<N, N1, false, T>(z + pc * N, 1, z + pc * N, 1, k1, tw);
        }
        tile_sync<NT, GROUP>(bar);
    }
    for (int it = tid; it < nrows * H; it += NT) {
        const int row = it / H, k = it - row * H, o = row * HP + k;
        const int pk = perm_pos<N, N1>(k), pn = perm_pos<N, N1>(k == 0 ? 0 : N - k);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const cplx<T> zk = z[(c * R + row) * N + pk];
            const cplx<T> zn = conj(z[(c * R + row) * N + pn]);
            const cplx<T> d = zk - zn;  // (zk - zn) / (2i) = (d.y, -d.x) / 2
            sp[(2 * c) * HS + o] = half_of(zk + zn);
            sp[(2 * c + 1) * HS + o] = half_of(mk(d.y, -d.x));
        }
    }
}

template <int N, int NA, int TV>
__global__ void __launch_bounds__(RowCfg<N, NA, TV>::NT, RowCfg<N, NA, TV>::MINB) k_rows_cg(PassArgs a) {
    using T = float;
    using S = RowCfg<N, NA, TV>;
    constexpr int R = S::R, NT = S::NT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double pcp_warp[NT / 32];
    cplx<T>* z = reinterpret_cast<cplx<T>*>(smem_raw);  // [3][R][N]
    cplx<T>* tw = z + 3 * R * N;
    const int f = blockIdx.z;
    if (a.cg[f].done) return;
    load_tw<T>(tw, a.tw, N);
    constexpr int HP = spec_pitch(N);
    rows_tile<N, NA, R, NT, false, HP, 2>(blockIdx.x * R, N * N, (cplx<T>*)a.out + f * a.sstride,
                                          (long long)N * N * HP, (const T*)a.tangent + f * a.tstride, a.cs, z, tw,
                                          pcp_warp, threadIdx.x, 0);
    // the block's part of <p, C : p> (written before the last barriers)
    if (threadIdx.x == 0) {
        double t = 0.0;
#pragma unroll
        for (int w = 0; w < NT / 32; ++w) t += pcp_warp[w];
        a.partials[(size_t)f * gridDim.x + blockIdx.x] = t;
    }
}

// -------------------------------------------------------------------- planes
// P4, the row pass and P2 act within one x1 plane. Where a plane's six
// components are small in shared memory one block takes it through all three:
// 77 B per voxel at 45^3 from and to global memory instead of 175, and two
// launches less an iteration. An iteration takes 39 instead of 50 us on one cell of
// 45^3 and 122 instead of 131 on sixteen. At 75^3 a plane takes 209 KB, one
// block of 20 warps an SM: 64 instead of 65 us on one cell but 508 instead of
// 481 on sixteen, so the line lies below it.
template <int N>
struct PlaneCfg {
    static constexpr bool ok = N <= 45;
    static constexpr int H = (N + 1) / 2, N1 = N == 3 || N == 5 ? N : X1Split<N>::N1, N2 = N / N1;
    // groups of GT threads share the rows, R a turn (R even)
    static constexpr int GT = 128, G = N <= 27 ? 4 : 3, R = 8, NT = GT * G, MINB = 2;
    static constexpr int row_tiles = (N + R - 1) / R;
    static constexpr int elems = 6 * N * H + (6 * N * H & 1) + G * 3 * R * N;  // plane, then the groups' rows
    static constexpr size_t smem = (size_t)(elems + N) * 8;
    static_assert(!ok || smem <= 227 * 1024, "shared memory per block");
};

// One x1 plane by the NT threads of the block: `sp` and `tg` are the plane's.
// The plane's <p, C : p> is left in group_part, one number a group.
template <int N>
__device__ __forceinline__ void plane_tile(cplx<float>* sp, const float* tg, long long cs, cplx<float>* buf,
                                           const cplx<float>* tw, double* warp_part, double* group_part) {
    using T = float;
    using S = PlaneCfg<N>;
    constexpr int H = S::H, HP = spec_pitch(N), N1 = S::N1, N2 = S::N2, NT = S::NT, GT = S::GT, P = 6 * H;
    const long long comp = (long long)N * N * HP;
    for (int it = threadIdx.x; it < P * N1; it += NT) {
        const int pc = it % P, k1 = it / P;
        const int c = pc / H, w = pc - c * H;
        invB<N, N1, true, T>(sp + c * comp + w, HP, buf + c * N * H + w, H, k1, tw);
    }
    __syncthreads();
    for (int it = threadIdx.x; it < P * N2; it += NT) {
        const int pc = it % P, t = it / P;
        cplx<T>* b = buf + (pc / H) * N * H + pc % H;
        invA<N, N1, T>(b, H, b, H, t, tw);
    }
    __syncthreads();
    {
        const int g = threadIdx.x / GT, tid = threadIdx.x - g * GT;
        cplx<T>* z = buf + 6 * N * H + (6 * N * H & 1) + g * 3 * S::R * N;
        double* wp = warp_part + g * (GT / 32);
        double sum = 0.0;
        for (int j = g; j < S::row_tiles; j += S::G) {
            rows_tile<N, RowSplit<N>::N1, S::R, GT, true, H, 1>(j * S::R, N, buf, N * H, tg, cs, z, tw, wp, tid, 1 + g);
            if (tid == 0)
                for (int w = 0; w < GT / 32; ++w) sum += wp[w];
            tile_sync<GT, true>(1 + g);
        }
        if (tid == 0) group_part[g] = sum;
    }
    __syncthreads();
    for (int it = threadIdx.x; it < P * N2; it += NT) {
        const int pc = it % P, t = it / P;
        cplx<T>* b = buf + (pc / H) * N * H + pc % H;
        fwdA<N, N1, T>(b, H, b, H, t, tw);
    }
    __syncthreads();
    for (int it = threadIdx.x; it < P * N1; it += NT) {
        const int pc = it % P, k1 = it / P;
        const int c = pc / H, w = pc - c * H;
        fwdB<N, N1, true, T>(buf + c * N * H + w, H, sp + c * comp + w, HP, k1, tw);
    }
}

// The plane's part of <p, C : p>, after a barrier (thread 0).
template <int N>
__device__ __forceinline__ double plane_part(const double* group_part) {
    double t = 0.0;
#pragma unroll
    for (int g = 0; g < PlaneCfg<N>::G; ++g) t += group_part[g];
    return t;
}

template <int N>
__global__ void __launch_bounds__(PlaneCfg<N>::NT, PlaneCfg<N>::MINB) k_plane_cg(PassArgs a) {
    using T = float;
    using S = PlaneCfg<N>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double warp_part[S::NT / 32], group_part[S::G];
    cplx<T>* buf = reinterpret_cast<cplx<T>*>(smem_raw);
    cplx<T>* tw = buf + S::elems;
    const int f = blockIdx.z;
    if (a.cg[f].done) return;
    load_tw<T>(tw, a.tw, N);
    __syncthreads();
    plane_tile<N>((cplx<T>*)a.out + f * a.sstride + (long long)blockIdx.x * N * spec_pitch(N),
                  (const T*)a.tangent + f * a.tstride + (long long)blockIdx.x * N * N, a.cs, buf, tw, warp_part,
                  group_part);
    // the field's last block sums the planes' parts of <p, C : p>: alpha
    __shared__ bool last;
    double* part = a.partials + (size_t)f * N;
    CGState* cg = a.cg + f;
    if (threadIdx.x == 0) {
        part[blockIdx.x] = plane_part<N>(group_part);
        __threadfence();
        last = atomicAdd(&cg->ticket, 1u) == N - 1;
    }
    __syncthreads();
    if (!last || threadIdx.x >= 32) return;
    __threadfence();
    const double pq = warp_total(part, N, threadIdx.x);
    if (threadIdx.x == 0) {
        cg->ticket = 0u;
        cg_after_dot(cg, pq);
    }
}

// --------------------------------------------------------------- small grids
// The whole CG solve of a field by one thread-block cluster: below 45^3 an
// iteration's six kernels do a few microseconds of work each, and launches
// and the loop's condition take most of the time. The phases are those above,
// x1 tiles over groups of GT threads and planes over the blocks, with the
// hardware's cluster barrier (which orders global memory within the cluster)
// between them; every block keeps the solve's scalars and takes the same
// steps, block 0 writes them back. The blocks of a cluster are resident together by construction, so no
// wait depends on another launch. An iteration takes 11 instead of 37 us on one
// cell of 15^3, 24 instead of 39 on one of 27^3 and 59 instead of 78 on
// thirty-two of them (cluster_blocks has the sizes of clusters).
template <int N>
struct ClusterCg {
    static constexpr bool ok = N <= 27;
    using PL = PlaneCfg<N>;
    static constexpr int GT = PL::GT, G = PL::G, NT = PL::NT;
    static constexpr int x1_elems = G * 6 * N * X1<N>::W;
    static constexpr int elems = x1_elems > PL::elems ? x1_elems : PL::elems;
    static constexpr size_t smem = (size_t)(elems + N) * 8;
    // partial sums of a field: one of each plane, then one of each x1 tile
    static constexpr int partials = N + X1<N>::blocks;
};

__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

template <int N>
__global__ void __launch_bounds__(ClusterCg<N>::NT, 2) k_cg_cluster(PassArgs a, int cl, unsigned int cap) {
    using T = float;
    using S = ClusterCg<N>;
    constexpr int GT = S::GT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ CGState st;
    __shared__ double warp_part[S::NT / 32], group_part[S::G];
    const int f = blockIdx.x / cl, rank = blockIdx.x - f * cl;
    if (a.cg[f].done) return;  // the same for every block of the cluster
    const int tid = threadIdx.x % GT, g = threadIdx.x / GT, bar = 1 + g;
    const int group = rank * S::G + g, groups = cl * S::G;
    cplx<T>* all = reinterpret_cast<cplx<T>*>(smem_raw);
    cplx<T>* buf = all + g * 6 * N * X1<N>::W;
    cplx<T>* tw = all + S::elems;
    double* wp = warp_part + g * (GT / 32);
    load_tw<T>(tw, a.tw, N);
    if (threadIdx.x == 0) st = a.cg[f];
    __syncthreads();
    const long long vf = f * coef_field<N>();
    cplx<T>* r = (cplx<T>*)a.aux + vf;
    cplx<T>* p = (cplx<T>*)a.aux2 + vf;
    cplx<T>* x = (cplx<T>*)a.aux3 + vf;
    cplx<T>* sp = (cplx<T>*)a.out + f * a.sstride;
    const T* tg = (const T*)a.tangent + f * a.tstride;
    double* part = a.partials + (size_t)f * S::partials;
    double* part_x1 = part + N;
    const double unit = (double)CoefScale<N>::value * a.scale;
    for (unsigned int pass = 0; pass < cap && st.done == CG_RUNNING; ++pass) {
        for (int j = group; j < X1<N>::blocks; j += groups) {
            x1i_tile<N, X1I_CG, false, GT, true>(j % X1<N>::tiles, j / X1<N>::tiles, st.it, (T)st.alpha, (T)st.beta,
                                                 st.pend != 0, r, p, x, sp, buf, tw, tid, bar);
            tile_sync<GT, true>(bar);  // the tile's buffer is free again
        }
        cluster_sync();
        for (int j = rank; j < N; j += cl) {
            plane_tile<N>(sp + (long long)j * N * spec_pitch(N), tg + (long long)j * N * N, a.cs, all, tw, warp_part,
                          group_part);
            if (threadIdx.x == 0) part[j] = plane_part<N>(group_part);
            __syncthreads();
        }
        cluster_sync();
        if (threadIdx.x < 32) {
            const double pq = warp_total(part, N, threadIdx.x);
            if (threadIdx.x == 0) cg_after_dot(&st, pq);
        }
        __syncthreads();
        if (st.done != CG_RUNNING) break;  // the same in every block
        for (int j = group; j < X1<N>::blocks; j += groups) {
            const X1fSums sums = x1f_tile<N, X1F_CG, false, GT, true>(
                j % X1<N>::tiles, j / X1<N>::tiles, (T)(-st.alpha * unit), sp, r, buf, tw, tid, bar);
            const double wv = warp_sum((double)sums.rr);
            if ((tid & 31) == 0) wp[tid >> 5] = wv;
            tile_sync<GT, true>(bar);
            if (tid == 0) {
                double t = 0.0;
#pragma unroll
                for (int w = 0; w < GT / 32; ++w) t += wp[w];
                part_x1[j] = t * CoefScale<N>::square;
            }
            tile_sync<GT, true>(bar);
        }
        cluster_sync();
        if (threadIdx.x < 32) {
            const double rr = warp_total(part_x1, X1<N>::blocks, threadIdx.x);
            if (threadIdx.x == 0) cg_after_update(&st, rr);
        }
        __syncthreads();
    }
    if (rank == 0 && threadIdx.x == 0) a.cg[f] = st;
}

// ------------------------------------------------------------------ launcher
template <int N>
cudaError_t run_pass_n(PassKind kind, const PassArgs& a, int nf, cudaStream_t s) {
    using C32 = Cfg<N, float>;
    using C64 = Cfg<N, double>;
    using CDD = Cfg<N, dd>;
    static_assert(CDD::row_blocks == C64::row_blocks && CDD::W2 == C64::W2 && CDD::S2 == C64::S2,
                  "double-float row and column passes share the FP64 geometry");
    using U32 = UserRows<N, float>;
    using U64 = UserRows<N, double>;
    const dim3 r32(C32::row_blocks, 1, nf), r64(C64::row_blocks, 1, nf);
    const dim3 u32(U32::row_blocks, 1, nf), u64(U64::row_blocks, 1, nf);
    const dim3 c32((C32::H + C32::W2 - 1) / C32::W2, (6 * N + C32::S2 - 1) / C32::S2, nf);
    const dim3 c64((C64::H + C64::W2 - 1) / C64::W2, (6 * N + C64::S2 - 1) / C64::S2, nf);
    const dim3 g64((C64::H + C64::W3 - 1) / C64::W3, N, nf);
    const dim3 x32(X1<N>::tiles, N, nf);
    const dim3 gdd((CDD::H + CDD::W3 - 1) / CDD::W3, N, nf);
    switch (kind) {
        case PK_P1_PLAIN_F64: return launch_k(k_p1<N, double, P1_PLAIN>, r64, C64::smem_rows, a, s, C64::TR);
        case PK_P1_PLAIN_F32: return launch_k(k_p1<N, float, P1_PLAIN, 1, Plan<N>::N1, 3>, u32, U32::smem_rows, a, s, U32::TR);
        case PK_P1_TAN_F64: return launch_k(k_p1<N, double, P1_TAN, 1, Plan<N>::N1, 3>, u64, U64::smem_rows, a, s, U64::TR);
        case PK_P1_TAN_F32: return launch_k(k_p1<N, float, P1_TAN, 1, Plan<N>::N1, 3>, u32, U32::smem_rows, a, s, U32::TR);
        case PK_P1_CG_F64: return launch_k(k_p1<N, double, P1_CG>, r64, C64::smem_rows, a, s, C64::TR);
        case PK_P1_TANRHS_F64: return launch_k(k_p1<N, double, P1_TANRHS>, r64, C64::smem_rows, a, s, C64::TR);
        case PK_P1_TANRHS_F32: return launch_k(k_p1<N, float, P1_TANRHS>, r32, C32::smem_rows, a, s, C32::TR);
        case PK_P2_F64: return launch_k(k_p24<N, double, true>, c64, C64::smem_p24, a, s, C64::T2);
        case PK_P2_F32: return launch_k(k_p24<N, float, true>, c32, C32::smem_p24, a, s, C32::T2);
        case PK_P4_F64: return launch_k(k_p24<N, double, false>, c64, C64::smem_p24, a, s, C64::T2);
        case PK_P4_F32: return launch_k(k_p24<N, float, false>, c32, C32::smem_p24, a, s, C32::T2);
        case PK_P3_F64: return launch_k(k_p3<N, double>, g64, C64::smem_p3, a, s, C64::T3);
        case PK_P3_F32: {
            using D = P3Default<N>;
            using C = Cfg<N, float, D::A>;
            const dim3 g((C::H + C::W3 - 1) / C::W3, N, nf);
            if constexpr (D::fused)
                return launch_k(k_p3f<N, D::A>, g, C::smem_p3, a, s, P3f<N, D::A>::NT);
            else
                return launch_k(k_p3<N, float, D::A>, g, C::smem_p3, a, s, C::T3);
        }
        case PK_P5_PLAIN_F64: return launch_k(k_p5<N, double, P5_PLAIN, double, 1, Plan<N>::N1, 3>, u64, U64::smem_rows, a, s);
        case PK_P5_PLAIN_F32: return launch_k(k_p5<N, float, P5_PLAIN, float>, r32, C32::smem_rows, a, s);
        case PK_P5_DOT_F64: return launch_k(k_p5<N, double, P5_DOT, double>, r64, C64::smem_rows, a, s);
        case PK_P5_DOT_F32: return launch_k(k_p5<N, float, P5_DOT, float, 1, Plan<N>::N1, 3>, u32, U32::smem_rows, a, s);
        case PK_P5_RHS_F64_TO_F64:
            return launch_k(k_p5<N, double, P5_RHS, double>, r64, C64::smem_rows, a, s);
        case PK_P1_PLAIN_DD: return launch_k(k_p1<N, dd, P1_PLAIN>, r64, CDD::smem_rows, a, s, CDD::TR);
        case PK_P2_DD: return launch_k(k_p24<N, dd, true>, c64, CDD::smem_p24, a, s, CDD::T2);
        case PK_P4_DD: return launch_k(k_p24<N, dd, false>, c64, CDD::smem_p24, a, s, CDD::T2);
        case PK_P3_DD: return launch_k(k_p3<N, dd>, gdd, CDD::smem_p3, a, s, CDD::T3);
        case PK_P5_PLAIN_DD_TO_F64:
            return launch_k(k_p5<N, dd, P5_PLAIN, double, 1, Plan<N>::N1, 3>, u64, U64::smem_rows, a, s);
        case PK_P1_USER_F64: return launch_k(k_p1<N, double, P1_PLAIN, 1, Plan<N>::N1, 3>, u64, U64::smem_rows, a, s, U64::TR);
        case PK_P1_USER_DD: return launch_k(k_p1<N, dd, P1_PLAIN, 1, Plan<N>::N1, 3>, u64, U64::smem_rows, a, s, Cfg<N, dd, Plan<N>::N1, 3>::TR);
        case PK_P5_USER_F32: return launch_k(k_p5<N, float, P5_PLAIN, float, 1, Plan<N>::N1, 3>, u32, U32::smem_rows, a, s);
        case PK_P5_DOT_USER_F64:
            return launch_k(k_p5<N, double, P5_DOT, double, 1, Plan<N>::N1, 3>, u64, U64::smem_rows, a, s);
        case PK_P5_NEWTON_F32: return launch_k(k_p5<N, float, P5_NEWTON, float>, r32, C32::smem_rows, a, s);
        case PK_X1I_CG_F32: return launch_k(k_x1i<N, X1I_CG>, x32, X1<N>::smem, a, s, X1<N>::NT);
        case PK_X1I_SOLUTION_F32: return launch_k(k_x1i<N, X1I_SOLUTION>, x32, X1<N>::smem, a, s, X1<N>::NT);
        case PK_X1F_CG_F32: return launch_k(k_x1f<N, X1F_CG>, x32, X1<N>::smem, a, s, X1<N>::NT);
        case PK_X1F_RHS_F32: return launch_k(k_x1f<N, X1F_RHS>, x32, X1<N>::smem, a, s, X1<N>::NT);
        case PK_X1F_RHS_DD: {
            using X = X1dd<N>;
            return launch_k(k_x1f_dd<N>, dim3((X::H + X::W3 - 1) / X::W3, N, nf), X::smem_p3, a, s, X::T3);
        }
        case PK_PLANE_CG_F32: {
            using S = PlaneCfg<N>;
            if constexpr (S::ok)
                return launch_k(k_plane_cg<N>, dim3(N, 1, nf), S::smem, a, s, S::NT);
            else
                return cudaErrorInvalidValue;
        }
        case PK_ROWS_CG_F32: {
            using R = RowCfg<N, RowSplit<N>::N1, 0>;
            return launch_k(k_rows_cg<N, RowSplit<N>::N1, 0>, dim3(R::blocks, 1, nf), R::smem, a, s, R::NT);
        }
        default: return cudaErrorInvalidValue;
    }
}

// The solve of nf fields by clusters of cl blocks (cl = 0: the largest size,
// 16 or 8, that the device takes, or 0, is written to *size and nothing runs).
template <int N>
cudaError_t run_cluster_n(const PassArgs& a, int nf, int cl, unsigned int cap, int* size, cudaStream_t s) {
    if constexpr (!ClusterCg<N>::ok) {
        if (size) *size = 0;
        return cl ? cudaErrorInvalidValue : cudaSuccess;
    } else {
        using S = ClusterCg<N>;
        cudaError_t e = cudaFuncSetAttribute(k_cg_cluster<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::smem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_cg_cluster<N>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cfg.blockDim = dim3(S::NT);
        cfg.dynamicSmemBytes = S::smem;
        cfg.stream = s;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        if (cl) {
            at.val.clusterDim.x = cl;
            cfg.gridDim = dim3(nf * cl);
            return cudaLaunchKernelEx(&cfg, k_cg_cluster<N>, a, cl, cap);
        }
        *size = 0;
        for (int c : {16, 8}) {
            int n = 0;
            at.val.clusterDim.x = c;
            cfg.gridDim = dim3(c);
            if (cudaOccupancyMaxActiveClusters(&n, k_cg_cluster<N>, &cfg) == cudaSuccess && n > 0) {
                *size = c;
                break;
            }
            cudaGetLastError();
        }
        return cudaSuccess;
    }
}

}  // namespace fftg
