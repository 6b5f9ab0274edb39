// Host-side helpers shared by the small- and finite-strain drivers.
#pragma once

#include <cmath>
#include <cstddef>
#include <cstdint>

namespace fftg {

// Grid sizes with a compiled plan: odd, 3^a 5^b, up to 243.
inline bool supported_grid(int N) {
    switch (N) {
        case 3: case 5: case 9: case 15: case 25: case 27: case 45: case 75: case 81: case 125:
        case 135: case 225: case 243:
            return true;
        default:
            return false;
    }
}

// Component stride of every field: N^3 rounded up past N^3 + 4 to a
// multiple of 32 elements, so each component starts 128-byte aligned and a
// 16-byte vector that straddles the end of the grid stays in the padding.
inline long long comp_stride(int N) {
    const long long V = (long long)N * N * N;
    return ((V + 4 + 31) / 32) * 32;
}

// Row pitch of the half spectra, in complex elements: (N + 1) / 2 rounded up
// to a multiple of 4, so that every row starts on a 32-byte sector and the
// runs of 8 and 16 columns that the x1 and x2 passes take touch no sector
// twice; on the grids whose spectrum is far larger than L2, of 16 (128-byte
// lines: an in-place copy in the x2 pattern 128 -> 120 us at 243^3).
constexpr int spec_pitch(int N) {
    const int H = (N + 1) / 2, u = N > 200 ? 16 : 4;
    return (H + u - 1) / u * u;
}

// The x1 passes of the mixed CG (cg_passes.cuh) take kCoefTile columns a
// block, and its vectors are stored tile by tile: complex elements a field.
constexpr int kCoefTile = 8;
constexpr long long coef_elements(int N) {
    return 3LL * N * N * (((N + 1) / 2 + kCoefTile - 1) / kCoefTile * kCoefTile);
}

// Passes after which a device loop over iterations stops whatever its solves
// report: the option's cap and some slack. Unsigned: caps up to INT_MAX are
// options ("no limit").
constexpr unsigned int pass_cap(int fixed, int most, unsigned int slack) {
    return (unsigned int)(fixed > 0 ? fixed : most) + slack;
}

// Memory that a caller's buffer starts in: the current device's or managed
// (here), and the allocation it belongs to (size 0: not known).
struct BufferRange {
    bool here = false;
    uintptr_t base = 0;
    size_t size = 0;
};

// Whether kernels can take a caller's field of `bytes` bytes where it is:
// memory they reach, aligned to its elements, and an allocation that holds all
// of the field. All else goes through cudaMemcpyAsync and a buffer of the
// handle: that reaches page-locked host memory, peers and fields over several
// mappings, and refuses with an error what a kernel would fault on.
inline bool usable_in_place(const BufferRange& r, const void* p, size_t bytes, size_t es) {
    const uintptr_t a = (uintptr_t)p;
    if (!r.here || (a & (es - 1)) || a < r.base) return false;
    return r.size >= a - r.base && r.size - (a - r.base) >= bytes;
}

// w_N^j = exp(-2 pi i j / N), evaluated in long double on the host: FP64,
// FP32 and (when twdd is not null) double-float (hi, lo) pairs, 4 floats
// per twiddle (re.hi, re.lo, im.hi, im.lo).
inline void twiddles(int N, double* tw64, float* tw32, float* twdd = nullptr) {
    const long double two_pi = 6.283185307179586476925286766559L;
    for (int j = 0; j < N; ++j) {
        const long double a = two_pi * (long double)j / (long double)N;
        const long double cl = cosl(a), sl = -sinl(a);
        const double c = (double)cl, s = (double)sl;
        tw64[2 * j] = c;
        tw64[2 * j + 1] = s;
        tw32[2 * j] = (float)c;
        tw32[2 * j + 1] = (float)s;
        if (twdd) {
            const float ch = (float)cl, sh = (float)sl;
            twdd[4 * j] = ch;
            twdd[4 * j + 1] = (float)(cl - (long double)ch);
            twdd[4 * j + 2] = sh;
            twdd[4 * j + 3] = (float)(sl - (long double)sh);
        }
    }
}

}  // namespace fftg
