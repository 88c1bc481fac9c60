// field_grid.cuh -- device helpers shared by the field's sample grid
// (field_grid.cu) and its adjoint (field_grid_adjoint.cu).
#pragma once

#include "internal.cuh"

namespace scm {

constexpr int kFgSlices = 16;            // slices of one x/z block

struct alignas(16) FgDouble4 {
    double x, y, z, w;
};
template <typename R> struct Fg;
template <> struct Fg<float> { using C = float2; using V4 = float4; };
template <> struct Fg<double> { using C = double2; using V4 = FgDouble4; };

// 1 / (x^2 - x_a^2) from the squares as pairs; the pole at a point itself is
// cut off far below the distances that arise, where the weights have long
// become 1 at that point and 0 elsewhere.
__device__ __forceinline__ float fg_recip(float xh, float xl, float nh, float nl) {
    float d = (xh - nh) + (xl - nl);
    d = fabsf(d) < 1e-12f ? 1e-12f : d;
    return __fdividef(1.0f, d);
}
// FP64: two Newton-Raphson steps r <- r + r (1 - d r) from the hardware's 2^-20
// approximation (2^-40, then within 2 ulp): four FP64 operations, which this part
// runs at 1/64 of its FP32 rate, and none of a division's special cases.
__device__ __forceinline__ double fg_recip(double xh, double, double nh, double) {
    double d = xh - nh, r;
    d = fabs(d) < 1e-30 ? 1e-30 : d;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
    r = fma(r, fma(-d, r, 1.0), r);
    return fma(r, fma(-d, r, 1.0), r);
}

// acc + low gains a b with twice the working precision (Ogita, Rump and Oishi's
// Dot2: the product's and the sum's rounding errors are collected in low).
__device__ __forceinline__ void fg_dot2(float a, float b, float &acc, float &low) {
    const float p = __fmul_rn(a, b), e = fmaf(a, b, -p);
    const float t = __fadd_rn(acc, p), z = __fsub_rn(t, acc);
    low += __fadd_rn(__fsub_rn(acc, __fsub_rn(t, z)), __fsub_rn(p, z)) + e;
    acc = t;
}
__device__ __forceinline__ void fg_dot2(double a, double b, double &acc, double &) { acc = fma(a, b, acc); }

// ---------------------------------------------------------------------------
// The folded sums.  A block of 256 threads computes two real products
//   out[row][col] = sum_k T[k][row] S[k][col]
// side by side: threads 0-127 the cosines with the even parts, 128-255 the
// sines with the odd parts.  64 columns, 8 kRpt rows; a thread holds rows
// bg + 8 i and columns 4 cg .. 4 cg + 3, K runs in tiles of kFgK staged in
// shared memory.  Per K value a warp reads 5 + kRpt shared-memory wavefronts
// for 4 kRpt FMAs per thread.
// ---------------------------------------------------------------------------
constexpr int kFgThreads = 256;
constexpr int kFgK = 32;
constexpr int kFgCols = 64;
constexpr int kFgColStride = kFgCols + 4;      // 16-byte stores of neighbouring K values fall in different banks

// kPad: rows of T one longer, for tiles filled along K.
template <typename R, int kRpt, int kPad = 0>
struct FgTile {
    alignas(32) R S[2][kFgK][kFgColStride];            // even, odd parts
    alignas(16) R T[2][kFgK][8 * kRpt + kPad];         // cosines, sines
};

template <typename R, int kRpt, int kPad>
__device__ __forceinline__ void fg_multiply(const FgTile<R, kRpt, kPad> &t, int grp, int bg, int cg, int kn, R (&acc)[kRpt][4]) {
    using V4 = typename Fg<R>::V4;
#pragma unroll 4
    for (int k = 0; k < kn; ++k) {
        const V4 s = *reinterpret_cast<const V4 *>(&t.S[grp][k][4 * cg]);
#pragma unroll
        for (int i = 0; i < kRpt; ++i) {
            const R w = t.T[grp][k][bg + 8 * i];
            acc[i][0] = fma(w, s.x, acc[i][0]);
            acc[i][1] = fma(w, s.y, acc[i][1]);
            acc[i][2] = fma(w, s.z, acc[i][2]);
            acc[i][3] = fma(w, s.w, acc[i][3]);
        }
    }
}

// The two mirror voxels of half-coordinate k on a side of n.
__device__ __forceinline__ int fg_plus(int k, int n) { return n / 2 + k; }
__device__ __forceinline__ int fg_minus(int k, int n) { return (n - 1) / 2 - k; }

// Opts a kernel in to `bytes` of dynamic shared memory where that needs it (beside at
// most 8 KB of static); always the same bytes per kernel or its plans' largest, so
// that launches of other threads stay valid.
template <typename K>
static cudaError_t fg_smem(K kernel, size_t bytes) {
    if (bytes <= (size_t)40 << 10) return cudaSuccess;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

}  // namespace scm
