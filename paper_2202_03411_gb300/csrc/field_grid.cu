// field_grid.cu -- Eq. 9 through the field's samples on a small grid of
// scattering directions.
//
// The field of a sample in a bounded box is a band-limited function of the
// direction k^ = (sqrt(1-s^2) t, s, sqrt(1-s^2) sqrt(1-t^2)) on the Ewald
// sphere, and a detector oversamples it many times over (128^3 voxels at a
// wavelength of 10 voxels and 60 degrees need about 80 x 74 directions, the
// 512^2 detector has 262144 pixels).  So the sums run over directions on a
// tensor grid of Chebyshev points s_a, t_b, where they separate,
//   H_a[j][x] = sum_y e^{-i k0 s_a y} s_j(x, y)
//   F_ab      = sum_j e^{-i q_z(a,b) z_j} sum_x e^{-i k0 sqrt(1-s_a^2) t_b x} H_a[j][x],
// and every pixel's field is the Chebyshev interpolant of F at its (s, t).
// On the flat detector t = X / sqrt(1 + X^2) depends on the pixel column only,
// on the uniform-q detector s = q_y / k0 on the row only: one direction is
// interpolated per column (row), the other per pixel.
//
// Everything is symmetric in the signs of s, t, x, y, so each sum runs over
// half the coordinates with the even and odd parts of its operand (cosines
// and sines are real: a quarter of the arithmetic), each interpolation over
// half the points (weights x_a K_a and x K_a, K_a = c_a / (x^2 - x_a^2)), and
// four mirrored pixels share their weights.
//
// The number of points per direction comes from a bound on the interpolation
// error over the whole box (plan_points below), not from the shape.
//
// Measured (forward pass with the voxeliser, against the direct sums): 128^3 on
// 512^2 to 60 degrees, BF16 split phases 74 us (1800); 96^3 on 256^2, by the size of the
// ellipsoid, FP32 27-32 us (4750-5800), FP64 160-196 us (73600-115000); 32^3 on 64^2, FP64
// 30 us (680-740); uniform-q 30^3 on 512^2, FP32 26-32 us (124, the separable sums
// per pixel row).
#include <algorithm>
#include <cmath>
#include <complex>

#include "internal.cuh"
#include "field_grid.cuh"

namespace scm {

// ---------------------------------------------------------------------------
// Host: plan
// ---------------------------------------------------------------------------

// Chebyshev points for functions exp(i k0 (x y + sqrt(1 - x^2) c)) with
// |y| <= along, |c| <= across on |x| <= top < 1.  On the Bernstein ellipse of
// parameter rho (about [-top, top]) the function is at most
// M = exp(k0 max(|Im x| along + |Im sqrt(1 - x^2)| across)), and its
// interpolant at N points is off by at most 4 M rho^-(N-1) / (rho - 1);
// the smallest N over the ellipses inside the branch points x = +-1.  The
// bound is loose by four to five decades for voxels anywhere in a filled box
// (it adds worst cases that do not meet) and more for a shape inside it, so
// tol = 1e-5 leaves 1e-9 to 1e-8 of a field that fills the box to its corners.
static int plan_points(double k0, double top, double along, double across, double tol) {
    const double inv = 1.0 / top;
    const double lmax = std::fmin(std::log(inv + std::sqrt(std::fmax(0.0, inv * inv - 1.0))), std::log(60.0));
    double best = 1e9;
    for (int i = 1; i <= 12; ++i) {
        const double l = lmax * i / 13.0, rho = std::exp(l);
        double e = 0.0;
        for (int p = 0; p <= 8; ++p) {
            const double ph = 0.5 * kPi * p / 8.0;
            const std::complex<double> x(top * 0.5 * (rho + 1.0 / rho) * std::cos(ph),
                                         top * 0.5 * (rho - 1.0 / rho) * std::sin(ph));
            const std::complex<double> c = std::sqrt(1.0 - x * x);
            e = std::fmax(e, std::fabs(x.imag()) * along + std::fabs(c.imag()) * across);
        }
        best = std::fmin(best, (k0 * e + std::log(4.0 / ((rho - 1.0) * tol))) / l + 1.0);
    }
    if (!(best < 4096.0)) return 4096;
    const int n = best < 2.0 ? 2 : (int)std::ceil(best);
    return n + (n & 1);
}

// Half the points of a direction at most (the per-pixel interpolation holds all
// points of 32 columns in shared memory: 131 KB in FP32, 200 KB in FP64).
static int fg_max_half(int elem) { return elem == 8 ? 96 : 128; }
constexpr int kFgMaxSide = 512;          // grid side in x and y
constexpr int kFgMaxRows = 65535;        // half the detector's rows: they are fg_pixels_kernel's grid.y

// elem: bytes of a real number in the sums.
bool plan_field_grid(const scatman_config &c, int elem, FieldGrid *f) {
    *f = FieldGrid();
    if (c.q_list || c.nx > kFgMaxSide || c.ny > kFgMaxSide || c.det_ny > 2 * kFgMaxRows) return false;
    const bool uniform = c.detector == SCATMAN_DETECTOR_UNIFORM_Q;
    const double k0 = 2.0 * kPi / c.wavelength;
    const double Lx = 0.5 * (c.nx - 1) * c.voxel, Ly = 0.5 * (c.ny - 1) * c.voxel, Lz = 0.5 * (c.nz - 1) * c.voxel;
    const double du = (double)(c.det_nx - 1) / c.det_nx, dv = (double)(c.det_ny - 1) / c.det_ny;
    const double th = c.theta_max_deg * kPi / 180.0;
    double sm, tm;
    if (!uniform) {
        const double h = std::tan(th), X = h * du, Y = h * dv, X0 = (c.det_nx & 1) ? 0.0 : h / c.det_nx;
        tm = X / std::sqrt(1.0 + X * X);
        sm = Y / std::sqrt(1.0 + Y * Y + X0 * X0);
    } else {
        const double h = std::sin(th);
        sm = h * dv;
        const double r = std::sqrt(std::fmax(0.0, 1.0 - sm * sm));
        tm = h * du < r ? h * du / r : 1.0;
    }
    // (an interval of zero width, a detector of one row or column, stays one)
    sm = std::fmax(sm, 1e-6);
    tm = std::fmax(tm, 1e-6);
    if (!(sm < 0.9995 && tm < 0.9995)) return false;
    const double hyp = std::hypot(Lx, Lz);
    // max over |t| <= tm of |t| Lx + sqrt(1 - t^2) Lz
    const double across = hyp > 0.0 && Lx / hyp <= tm ? hyp : tm * Lx + std::sqrt(1.0 - tm * tm) * Lz;
    const bool fp64 = c.precision == SCATMAN_FP64;
    const double tol = fp64 ? 1e-12 : 1e-5;
    const int Ns = plan_points(k0, sm, Ly, across, tol), Nt = plan_points(k0, tm, Lx, Lz, tol);
    if (Ns > 2 * fg_max_half(elem) || Nt > 2 * fg_max_half(elem)) return false;
    f->uniform = uniform;
    f->Hs = Ns / 2;
    f->Ht = Nt / 2;
    f->sm = sm;
    f->tm = tm;
    f->k0 = k0;
    f->voxel = c.voxel;
    f->top = uniform ? std::sin(th) : std::tan(th);
    f->nx = c.nx;
    f->ny = c.ny;
    f->nz = c.nz;
    f->det_nx = c.det_nx;
    f->det_ny = c.det_ny;
    f->Kx = (c.nx + 1) / 2;
    f->Ky = (c.ny + 1) / 2;
    f->U = (c.det_nx + 1) / 2;
    f->V = (c.det_ny + 1) / 2;
    f->H1 = uniform ? f->Hs : f->Ht;
    f->H2 = uniform ? f->Ht : f->Hs;
    f->n1 = uniform ? f->V : f->U;
    f->jc = (c.nz + kFgSlices - 1) / kFgSlices;
    f->elem = elem;
    f->io = fp64 ? 8 : 4;
    return true;
}

// Whether a handle of this configuration computes its field on the sample
// grid.  Not with a list of q (no detector), nor in the single-product modes
// and the tensor-core uniform-q detector (their 16-bit roundings belong to the
// pixel and to the row), nor where the direct sums are as fast.  FP32 and FP64:
// already at 16^3 voxels and 12^2 pixels.  Split phases on the tensor cores (45
// degrees, wavelength 8, ellipsoid, forward pass, grid / direct in us): 29 / 28 at
// 48^3 on 64^2, 29 / 32 on 96^2, 29 / 34 on 128^2; 35 / 36 at 64^3 on 64^2, 33 / 46 on
// 128^2; 48 / 47 at 96^3 on 64^2, 46 / 56 on 96^2; and where the grid has more points
// than the detector has pixels (60 degrees, wavelength 6) 58 / 47 at 96^3 on 64^2,
// 68 / 84 at 128^3 on 96^2.
// FP32 fits sum over the voxels and interpolate in FP64 (slices, field and pattern stay
// FP32).  A loss near its minimum shows the pattern's rounding many times larger: over
// 63 fits of 20^3 - 64^3 voxels the FP32 sums left the loss 7.0e-7 off (the direct
// FP32 sums 5.4e-7), these 3.4e-7, most of it the slices' own FP32; the pattern 2.1e-7
// (3.1e-7) and 6e-8.  The forward pass takes 40 us instead of 17 at 48^3 on 128^2 and 153
// instead of 25 at 96^3 on 256^2 (direct: 438 and 8660).  Where the points exceed the
// FP64 plan's limit the sums stay FP32.
// Patterns in FP32 keep FP32 sums: 2.1e-7 of the intensity off on the flat detector (the
// direct sums 2.9e-7), 2.0e-7 on the uniform-q one (its separable sums 1.3e-7: the
// alternating weights of the interpolation; 1.5e-7 at 67 us instead of 31 with only the
// pixels' own sums in FP32, 3e-8 at 153 us all in FP64, 30^3 on 512^2).
// Fits in the split phases sum over the pixels themselves, as their adjoint does:
// the 16-bit phase pairs round to 1e-6 of the intensity, and to another 1e-6 at the
// grid's directions.  A loss near its minimum, and more so a gradient that nearly
// cancels, shows that 25 to 100 times larger: with only the pattern's peak
// summed directly, served gradients of 96^3 and 128^3 still moved by up to 7e-5
// (by more than 2e-5 in 4 of 40 batches), and a 96^3 fit's on 256^2 by 1.9e-5.  The
// price: 8.5 ms instead of 2.8 for the 12 mixed server requests, 842 us instead of
// 614 for a fit step of 96^3 on 256^2 (forward and adjoint together).
bool use_field_grid(const scatman_config &c, FieldGrid *f) {
    const bool split = c.precision == SCATMAN_TC_F16_SPLIT || c.precision == SCATMAN_TC_BF16_SPLIT;
    const bool plain = c.precision == SCATMAN_FP64 || c.precision == SCATMAN_FP32;
    if (c.q_list || !(plain || (split && c.detector == SCATMAN_DETECTOR_FLAT))) return false;
    if (split && c.soft) return false;
    const double pixels = (double)c.det_nx * c.det_ny, terms = pixels * ((double)c.nx * c.ny * c.nz);
    if (plain ? pixels < 128.0 : terms < 5e8) return false;
    const bool fit = c.precision == SCATMAN_FP32 && c.soft;
    if (!(fit && plan_field_grid(c, 8, f)) && !plan_field_grid(c, c.precision == SCATMAN_FP64 ? 8 : 4, f)) return false;
    return !(split && terms < 8e9 && pixels < 2.4 * f->Hs * f->Ht);
}

// Whether the adjoint runs through the grid: FP32 and FP64, and tensor-core grids
// beyond the tensor-core adjoint's 128 voxels.  Within those the tensor-core modes
// sum over the pixels themselves.  A fit's upstream weight 2 (I - target) nearly
// cancels in some parameters, and a gradient there shows the operands' 16-bit
// roundings several hundred times larger: summed over the grid's directions, with
// three products, served gradients of 48^3 - 128^3 on 128^2 - 512^2 pixels moved by
// more than 2e-5 in 8 of 40 batches, by 4e-4 at most.  (Over the pixels 105 us of a
// 96^3 fit step on 256^2; over the directions 35.)
bool use_field_grid_adjoint(const scatman_config &c, FieldGrid *f) {
    const double pixels = (double)c.det_nx * c.det_ny;
    if (c.q_list || pixels < 128.0) return false;
    if (c.precision != SCATMAN_FP64 && c.precision != SCATMAN_FP32 && adjoint_tc_supported(c.nx, c.ny)) return false;
    return plan_field_grid(c, c.precision == SCATMAN_FP64 ? 8 : 4, f);
}

static size_t up256(size_t b) { return (b + 255) / 256 * 256; }

// Lays the grid's tables and, for the forward pass, its sums out from `base` (null:
// sizes only); returns the bytes.  Nxp: row of the tensor-core y-sums (0: none).
size_t field_grid_layout(FieldGrid *f, bool forward, int Nxp, unsigned char *base) {
    size_t at = 0;
    auto take = [&](size_t bytes) {
        unsigned char *p = base ? base + at : nullptr;
        at += up256(bytes);
        return (void *)p;
    };
    const size_t e = (size_t)f->elem;
    f->ty = take(2 * (size_t)f->Ky * f->Hs * e);
    f->tx = take(2 * (size_t)f->Hs * f->Kx * f->Ht * e);
    f->tz = take((size_t)f->Hs * f->Ht * f->nz * 2 * e);
    f->node2 = take((size_t)f->H2 * 4 * e);
    f->w1 = take(2 * (size_t)f->H1 * f->n1 * e);
    f->pix = take((size_t)f->U * f->V * 4 * e);
    f->qrow = (double *)take(2 * (size_t)f->Hs * 3 * sizeof(double));
    f->point_s = (double *)take(2 * (size_t)f->Hs * sizeof(double));
    f->point_t = (double *)take(2 * (size_t)f->Ht * sizeof(double));
    if (!forward) return at;
    const size_t row = (size_t)(Nxp > f->nx ? Nxp : f->nx);
    f->H = take(2 * (size_t)f->Hs * f->nz * row * 2 * e);
    f->Q = take((size_t)f->jc * f->Hs * f->Ht * 8 * e);
    f->B = take((size_t)f->H2 * 8 * ((f->n1 + 31) / 32 * 32) * e);
    return at;
}

// ---------------------------------------------------------------------------
// Tables (once per handle)
// ---------------------------------------------------------------------------

__device__ __forceinline__ double fg_angle(int a, int H) { return (2 * a + 1) * kPi / (4.0 * H); }   // N = 2H points

// cos and sin of a phase held in double; FP32 tables reduce it in FP64 first.
__device__ __forceinline__ float2 fg_cs(double ph, float) {
    ph -= 2.0 * kPi * rint(ph * (0.5 / kPi));
    float s, c;
    sincosf((float)ph, &s, &c);
    return make_float2(c, s);
}
__device__ __forceinline__ double2 fg_cs(double ph, double) {
    double s, c;
    sincos(ph, &s, &c);
    return make_double2(c, s);
}
__device__ __forceinline__ double fg_coord(int k, int n) { return (n & 1) ? (double)k : k + 0.5; }

template <typename R>
__device__ __forceinline__ typename Fg<R>::V4 fg_square(double x, R third, R fourth) {
    const double q = x * x;
    typename Fg<R>::V4 v;
    v.x = (R)q;
    v.y = (R)(q - (double)v.x);
    v.z = third;
    v.w = fourth;
    return v;
}

// The directions' points: s_a, sqrt(1 - s_a^2), then t_b, sqrt(1 - t_b^2), the
// rows' q_y (+s_a, then -s_a), and for the per-pixel direction x_a^2 (pair), c_a x_a, c_a.
template <typename R>
__global__ void fg_points_kernel(FieldGrid f) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < f.Hs) {
        const double s = f.sm * cos(fg_angle(k, f.Hs));
        f.point_s[2 * k] = s;
        f.point_s[2 * k + 1] = sqrt(1.0 - s * s);
        for (int m = 0; m < 2; ++m) {
            double *q = f.qrow + 3 * (size_t)(m * f.Hs + k);
            q[0] = q[2] = 0.0;
            q[1] = m ? -f.k0 * s : f.k0 * s;
        }
    }
    if (k < f.Ht) {
        const double x = f.tm * cos(fg_angle(k, f.Ht));
        f.point_t[2 * k] = x;
        f.point_t[2 * k + 1] = sqrt(1.0 - x * x);
    }
    if (k < f.H2) {
        double sn, x;
        sincos(fg_angle(k, f.H2), &sn, &x);
        const double c = (k & 1) ? -sn : sn;
        ((typename Fg<R>::V4 *)f.node2)[k] = fg_square<R>(x, (R)(c * x), (R)c);
    }
}

// The phases of the sums: cos, sin of q_y y' [y'][a] and of q_x x' [a][x'][b],
// and e^{-i q_z z_j} [a][b][j].
template <typename R>
__global__ void fg_tables_kernel(FieldGrid f) {
    using C = typename Fg<R>::C;
    R *cy = (R *)f.ty, *sy = cy + (size_t)f.Ky * f.Hs;
    R *cx = (R *)f.tx, *sx = cx + (size_t)f.Hs * f.Kx * f.Ht;
    C *tz = (C *)f.tz;
    const int n0 = f.Ky * f.Hs, n1 = f.Hs * f.Kx * f.Ht, n2 = f.Hs * f.Ht * f.nz;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n0 + n1 + n2; i += gridDim.x * blockDim.x) {
        if (i < n0) {
            const int a = i % f.Hs, y = i / f.Hs;
            const C e = fg_cs(f.k0 * f.point_s[2 * a] * (fg_coord(y, f.ny) * f.voxel), (R)0);
            cy[i] = e.x;
            sy[i] = e.y;
        } else if (i < n0 + n1) {
            const int k = i - n0, b = k % f.Ht, x = (k / f.Ht) % f.Kx, a = k / (f.Ht * f.Kx);
            const C e = fg_cs(f.k0 * f.point_s[2 * a + 1] * f.point_t[2 * b] * (fg_coord(x, f.nx) * f.voxel), (R)0);
            cx[k] = e.x;
            sx[k] = e.y;
        } else {
            const int k = i - n0 - n1, j = k % f.nz, b = (k / f.nz) % f.Ht, a = k / (f.nz * f.Ht);
            const double qz = f.k0 * (f.point_s[2 * a + 1] * f.point_t[2 * b + 1] - 1.0);
            const C e = fg_cs(qz * ((j - 0.5 * (f.nz - 1)) * f.voxel), (R)0);
            C v;
            v.x = e.x;
            v.y = -e.y;
            tz[k] = v;
        }
    }
}

// Normalised transverse coordinate of half-index i of n pixels (0 <= i < (n + 1) / 2).
__device__ __forceinline__ double fg_half_pixel(int i, int n) { return (double)(2 * (n / 2 + i) + 1 - n) / (double)n; }

// Interpolation weights of the per-column (per-row) direction, [even | odd][point][i]:
// one warp per i, its lanes over the points.
template <typename R>
__global__ void fg_weights_kernel(FieldGrid f) {
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (i >= f.n1) return;
    double x;
    if (f.uniform) {
        x = f.top * fg_half_pixel(i, f.det_ny) / f.sm;
    } else {
        const double X = f.top * fg_half_pixel(i, f.det_nx);
        x = X / sqrt(1.0 + X * X) / f.tm;
    }
    R *we = (R *)f.w1, *wo = we + (size_t)f.H1 * f.n1;
    constexpr int kMost = 4;                            // 32 kMost >= the points of a direction
    double w[kMost], xa[kMost], D = 0.0;
#pragma unroll
    for (int m = 0; m < kMost; ++m) {
        const int a = 32 * m + lane;
        w[m] = xa[m] = 0.0;
        if (a < f.H1) {
            double sn;
            sincos(fg_angle(a, f.H1), &sn, &xa[m]);
            double d = (x - xa[m]) * (x + xa[m]);
            d = fabs(d) < 1e-30 ? 1e-30 : d;
            w[m] = ((a & 1) ? -sn : sn) / d;
            D += w[m] * xa[m];
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) D += __shfl_xor_sync(0xffffffffu, D, o);
#pragma unroll
    for (int m = 0; m < kMost; ++m) {
        const int a = 32 * m + lane;
        if (a < f.H1) {
            we[(size_t)a * f.n1 + i] = (R)(w[m] * xa[m] / D);
            wo[(size_t)a * f.n1 + i] = (R)(w[m] * x / D);
        }
    }
}

// Per quadrant pixel: x^2 as a pair, x, and 1 / sum_a c_a x_a / (x^2 - x_a^2)
// (the weights' normalisation, with the reciprocals the interpolation forms);
// a quiet NaN in x marks pixels off the Ewald sphere.
template <typename R>
__global__ void fg_pixels_kernel(FieldGrid f) {
    using V4 = typename Fg<R>::V4;
    __shared__ double s_row;                             // uniform-q: top / sqrt(1 - (q_y / k0)^2) / tm of the row
    const int i = blockIdx.x * blockDim.x + threadIdx.x, v = blockIdx.y;
    const double pv = fg_half_pixel(v, f.det_ny);
    if (f.uniform) {
        if (threadIdx.x == 0) s_row = f.top / sqrt(1.0 - (f.top * pv) * (f.top * pv)) / f.tm;
        __syncthreads();
    }
    if (i >= f.U) return;
    double x;
    bool valid = true;
    const double pu = fg_half_pixel(i, f.det_nx);
    if (f.uniform) {
        // on the sphere: the FP64 operations that set the detector's q_z (the
        // quotient only where it could matter)
        const double qmax = f.k0 * f.top;
        const double qx = qmax * pu, qy = qmax * pv;
        const double q2 = __dadd_rn(__dmul_rn(qx, qx), __dmul_rn(qy, qy)), k2 = __dmul_rn(f.k0, f.k0);
        valid = q2 < 0.999 * k2 || __ddiv_rn(q2, k2) <= 1.0;
        x = valid ? s_row * pu : 0.0;
    } else {
        const double X = f.top * pu, Y = f.top * pv;
        x = Y / sqrt(1.0 + X * X + Y * Y) / f.sm;
    }
    V4 e = fg_square<R>(x, (R)x, (R)0);
    const V4 *nd = (const V4 *)f.node2;
    R D = (R)0, low = (R)0;
    for (int a = 0; a < f.H2; ++a) {
        const V4 n = nd[a];
        fg_dot2(n.z, fg_recip(e.x, e.y, n.x, n.y), D, low);
    }
    e.w = (R)1 / (D + low);
    if (!valid) e.z = (R)__longlong_as_double(0x7ff8000000000000ll);
    ((V4 *)f.pix)[(size_t)v * f.U + i] = e;
}

template <typename R>
static void fg_run_tables(const FieldGrid &f, cudaStream_t st) {
    const int most = f.Hs > f.Ht ? f.Hs : f.Ht;
    const long long n = (long long)f.Ky * f.Hs + (long long)f.Hs * f.Kx * f.Ht + (long long)f.Hs * f.Ht * f.nz;
    fg_points_kernel<R><<<(most + 31) / 32, 32, 0, st>>>(f);
    fg_tables_kernel<R><<<(unsigned)(n / 256 + 1), 256, 0, st>>>(f);
    fg_weights_kernel<R><<<(f.n1 + 3) / 4, 128, 0, st>>>(f);
    fg_pixels_kernel<R><<<dim3((f.U + 127) / 128, f.V), 128, 0, st>>>(f);
}

cudaError_t launch_field_grid_tables(const FieldGrid &f, cudaStream_t st) {
    if (f.elem == 8)
        fg_run_tables<double>(f, st);
    else
        fg_run_tables<float>(f, st);
    return cudaGetLastError();
}

// Rows per thread (tiles of 8 kRpt of n rows) on a grid of `others` blocks per row
// tile: the fewest rounds over the SMs times a block's work, its rows and the
// loads it makes whatever their number (worth three rows in FP32, half a row in
// FP64, whose arithmetic takes the time).  FP64 32^3 on 64^2: 36 blocks of 24 rows
// took 21 us, 108 of 8 rows take 8; larger grids keep five or six rows.
static int fg_rows_per_thread(int n, long long others, bool fp64, int sm_count) {
    int best = 3;
    double cost = 1e300;
    for (int r : {6, 5, 3, 2, 1}) {
        const long long blocks = others * ((n + 8 * r - 1) / (8 * r));
        const double c = (double)((blocks + sm_count - 1) / sm_count) * (r + (fp64 ? 0.5 : 3.0));
        if (c < 0.95 * cost) {
            cost = c;
            best = r;
        }
    }
    return best;
}

// Half-coordinates of a side of n that meet [lo, hi): above the middle up to hi - 1,
// below it down to lo; from the start of a tile of them.
struct FgFold {
    int beg, end;
};
__host__ __device__ __forceinline__ FgFold fg_fold(int lo, int hi, int n) {
    const int up = hi - n / 2, down = (n - 1) / 2 - lo + 1, most = (n + 1) / 2;
    const int far = up > down ? up : down, a = lo - n / 2, b = (n - 1) / 2 - (hi - 1), near = a > b ? a : b;
    return {(near > 0 ? near : 0) & ~(kFgK - 1), far < most ? far : most};
}

// H[a][even, odd][j][x] = sum over y' of cos (q_a y') even s, -i sin (q_a y') odd s.
// Block: 32 columns x of one slice.  Slices and columns outside the occupied
// box are not written (and not read later), y' beyond the box is skipped.
template <typename R, typename IO, int kRpt>
__global__ void __launch_bounds__(kFgThreads) fg_y_kernel(FieldGrid f, const typename Fg<IO>::C *__restrict__ s,
                                                          const int *__restrict__ bounds) {
    using C = typename Fg<R>::C;
    extern __shared__ __align__(32) unsigned char smem[];
    FgTile<R, kRpt> &t = *reinterpret_cast<FgTile<R, kRpt> *>(smem);
    const int j = blockIdx.y, x0 = blockIdx.x * 32, a0 = blockIdx.z * 8 * kRpt;
    pdl_wait();
    const int xlo = bounds[j], xhi = bounds[f.nz + j], ylo = bounds[2 * f.nz + j], yhi = bounds[3 * f.nz + j];
    if (xlo >= xhi || x0 >= xhi || x0 + 32 <= xlo) return;
    const int grp = threadIdx.x >> 7, tt = threadIdx.x & 127, cg = tt & 15, bg = tt >> 4;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const FgFold y = fg_fold(ylo, yhi, f.ny);
    const int kend = y.end, kbeg = y.beg;
    const R *cy = (const R *)f.ty, *sy = cy + (size_t)f.Ky * f.Hs;
    R acc[kRpt][4] = {};
    // one tile's operands on their way from memory
    R tc[kRpt], ts[kRpt];
    C sp[4], sm[4];
    auto load = [&](int k0) {
#pragma unroll
        for (int q = 0; q < kRpt; ++q) {
            const int i = threadIdx.x + q * kFgThreads, k = i / (8 * kRpt), a = i % (8 * kRpt);
            const bool in = k0 + k < kend && a0 + a < f.Hs;
            tc[q] = in ? cy[(size_t)(k0 + k) * f.Hs + a0 + a] : (R)0;
            ts[q] = in ? sy[(size_t)(k0 + k) * f.Hs + a0 + a] : (R)0;
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int x = x0 + warp * 4 + c, k = k0 + lane;
            sp[c].x = sp[c].y = sm[c].x = sm[c].y = (R)0;
            if (x < f.nx && k < kend) {
                const auto *line = s + ((size_t)j * f.nx + x) * f.ny;
                const int ip = fg_plus(k, f.ny), im = fg_minus(k, f.ny);
                sp[c].x = line[ip].x;
                sp[c].y = line[ip].y;
                if (im != ip) {
                    sm[c].x = line[im].x;
                    sm[c].y = line[im].y;
                }
            }
        }
    };
    auto store = [&]() {
#pragma unroll
        for (int q = 0; q < kRpt; ++q) {
            const int i = threadIdx.x + q * kFgThreads, k = i / (8 * kRpt), a = i % (8 * kRpt);
            t.T[0][k][a] = tc[q];
            t.T[1][k][a] = ts[q];
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int xl = warp * 4 + c;
            t.S[0][lane][2 * xl] = sp[c].x + sm[c].x;
            t.S[0][lane][2 * xl + 1] = sp[c].y + sm[c].y;
            t.S[1][lane][2 * xl] = sp[c].x - sm[c].x;
            t.S[1][lane][2 * xl + 1] = sp[c].y - sm[c].y;
        }
    };
    // (a tile's loads all in flight before the first is used; fetching the next
    // tile under this one's products as well gained nothing)
    for (int k0 = kbeg; k0 < kend; k0 += kFgK) {
        load(k0);
        __syncthreads();
        store();
        __syncthreads();
        fg_multiply<R, kRpt>(t, grp, bg, cg, min(kFgK, kend - k0), acc);
    }
#pragma unroll
    for (int i = 0; i < kRpt; ++i) {
        const int a = a0 + bg + 8 * i;
        if (a >= f.Hs) continue;
        C *out = (C *)f.H + (((size_t)a * 2 + grp) * f.nz + j) * f.nx;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int x = x0 + 2 * cg + c;
            if (x >= f.nx) continue;
            C v;
            v.x = acc[i][2 * c];
            v.y = acc[i][2 * c + 1];
            if (grp) {                                  // -i times
                const R r = v.x;
                v.x = v.y;
                v.y = -r;
            }
            out[x] = v;
        }
    }
}

// Q[chunk][a][b][even/odd in s x even/odd in t] over kFgSlices slices: the x
// sum with e^{-i q_x(a,b) x}, then the slice phases.  A column is one part of
// (even y, odd y) of one slice, so the thread that holds a row and a column
// group applies that slice's phase itself, and sixteen lanes add the slices.
// kPm: H holds the fields of the rows +s_a and -s_a (the tensor-core y-sum,
// rows of Nxp) instead of their even and odd parts.
template <typename R, int kRpt, bool kPm>
__global__ void __launch_bounds__(kFgThreads) fg_xz_kernel(FieldGrid f, int Nxp, const int *__restrict__ bounds,
                                                           const int *__restrict__ chunk_y) {
    using C = typename Fg<R>::C;
    using V4 = typename Fg<R>::V4;
    extern __shared__ __align__(32) unsigned char smem[];
    FgTile<R, kRpt> &t = *reinterpret_cast<FgTile<R, kRpt> *>(smem);
    __shared__ int s_lo[kFgSlices], s_hi[kFgSlices];
    __shared__ uint32_t s_live[kFgSlices];              // the occupied 8-column chunks, a bit each
    const int a = blockIdx.x, j0 = blockIdx.y * kFgSlices, b0 = blockIdx.z * 8 * kRpt;
    const int grp = threadIdx.x >> 7, tt = threadIdx.x & 127, cg = tt & 15, bg = tt >> 4;
    pdl_wait();
    if (threadIdx.x < kFgSlices) {
        const int j = j0 + threadIdx.x;
        s_lo[threadIdx.x] = j < f.nz ? bounds[j] : 0x7fffffff;
        s_hi[threadIdx.x] = j < f.nz ? bounds[f.nz + j] : 0;
    }
    if (kPm) {
        for (int jl = threadIdx.x >> 5; jl < kFgSlices; jl += kFgThreads / 32) {
            const int c = (j0 + jl) * kGeomChunks + (threadIdx.x & 31);
            const bool live = j0 + jl < f.nz && chunk_y[c] < chunk_y[kGeomChunks * f.nz + c];
            const uint32_t m = __ballot_sync(0xffffffffu, live);
            if ((threadIdx.x & 31) == 0) s_live[jl] = m;
        }
    }
    __syncthreads();
    int kend = 0;
#pragma unroll
    for (int j = 0; j < kFgSlices; ++j)
        if (s_lo[j] < s_hi[j]) kend = max(kend, fg_fold(s_lo[j], s_hi[j], f.nx).end);
    const R *cx = (const R *)f.tx + (size_t)a * f.Kx * f.Ht, *sx = cx + (size_t)f.Hs * f.Kx * f.Ht;
    const C *H = (const C *)f.H;
    R acc[kRpt][4] = {};
    // one tile's operands on their way from memory: the phases, and of two
    // (slice, x') the values of both parts at +x and -x
    R tc[kRpt], ts[kRpt];
    C he[2][2], ho[2][2];
    static_assert(kFgSlices * kFgK == 2 * kFgThreads, "two per thread");
    auto load = [&](int k0) {
#pragma unroll
        for (int q = 0; q < kRpt; ++q) {
            const int i = threadIdx.x + q * kFgThreads, k = i / (8 * kRpt), b = i % (8 * kRpt);
            const bool in = k0 + k < kend && b0 + b < f.Ht;
            tc[q] = in ? cx[(size_t)(k0 + k) * f.Ht + b0 + b] : (R)0;
            ts[q] = in ? sx[(size_t)(k0 + k) * f.Ht + b0 + b] : (R)0;
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int i = threadIdx.x + q * kFgThreads, jl = i / kFgK, k = i % kFgK, j = j0 + jl;
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                const int x = m == 0 ? fg_plus(k0 + k, f.nx) : fg_minus(k0 + k, f.nx);
                bool live = k0 + k < kend && x >= s_lo[jl] && x < s_hi[jl];
                // the tensor-core sum writes the occupied 8-column chunks only
                if (kPm && live) live = (s_live[jl] >> (x >> 3)) & 1u;
                if (m == 1 && x == fg_plus(k0 + k, f.nx)) live = false;        // the middle of an odd side counts once
                he[q][m].x = he[q][m].y = ho[q][m].x = ho[q][m].y = (R)0;
                if (live) {
                    he[q][m] = kPm ? H[((size_t)a * f.nz + j) * Nxp + x] : H[(((size_t)a * 2) * f.nz + j) * f.nx + x];
                    ho[q][m] = kPm ? H[((size_t)(f.Hs + a) * f.nz + j) * Nxp + x]
                                   : H[(((size_t)a * 2 + 1) * f.nz + j) * f.nx + x];
                }
            }
        }
    };
    auto store = [&]() {
#pragma unroll
        for (int q = 0; q < kRpt; ++q) {
            const int i = threadIdx.x + q * kFgThreads, k = i / (8 * kRpt), b = i % (8 * kRpt);
            t.T[0][k][b] = tc[q];
            t.T[1][k][b] = ts[q];
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int i = threadIdx.x + q * kFgThreads, jl = i / kFgK, k = i % kFgK;
            C e[2], o[2];                               // at +x, -x
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                e[m] = he[q][m];
                o[m] = ho[q][m];
                if (kPm) {
                    e[m].x = (R)0.5 * (he[q][m].x + ho[q][m].x);
                    e[m].y = (R)0.5 * (he[q][m].y + ho[q][m].y);
                    o[m].x = (R)0.5 * (he[q][m].x - ho[q][m].x);
                    o[m].y = (R)0.5 * (he[q][m].y - ho[q][m].y);
                }
            }
            V4 v;
            v.x = e[0].x + e[1].x;
            v.y = e[0].y + e[1].y;
            v.z = o[0].x + o[1].x;
            v.w = o[0].y + o[1].y;
            *reinterpret_cast<V4 *>(&t.S[0][k][4 * jl]) = v;
            v.x = e[0].x - e[1].x;
            v.y = e[0].y - e[1].y;
            v.z = o[0].x - o[1].x;
            v.w = o[0].y - o[1].y;
            *reinterpret_cast<V4 *>(&t.S[1][k][4 * jl]) = v;
        }
    };
    for (int k0 = 0; k0 < kend; k0 += kFgK) {
        load(k0);
        __syncthreads();
        store();
        __syncthreads();
        fg_multiply<R, kRpt>(t, grp, bg, cg, min(kFgK, kend - k0), acc);
    }
    const int j = j0 + cg;
    R *Q = (R *)f.Q + ((size_t)blockIdx.y * f.Hs + a) * f.Ht * 8;
#pragma unroll
    for (int i = 0; i < kRpt; ++i) {
        const int b = b0 + bg + 8 * i;
        C z;
        z.x = z.y = (R)0;
        if (b < f.Ht && j < f.nz && kend > 0) z = ((const C *)f.tz)[((size_t)a * f.Ht + b) * f.nz + j];
        R v[4] = {z.x * acc[i][0] - z.y * acc[i][1], z.x * acc[i][1] + z.y * acc[i][0],
                  z.x * acc[i][2] - z.y * acc[i][3], z.x * acc[i][3] + z.y * acc[i][2]};
#pragma unroll
        for (int o = 8; o > 0; o >>= 1)
#pragma unroll
            for (int c = 0; c < 4; ++c) v[c] += __shfl_xor_sync(0xffffffffu, v[c], o);
        if (cg == 0 && b < f.Ht) {
            // [ee, eo, oe, oo]; the odd x parts (sines) carry -i
            R *q = Q + (size_t)b * 8;
            if (grp == 0) {
                q[0] = v[0];
                q[1] = v[1];
                q[4] = v[2];
                q[5] = v[3];
            } else {
                q[2] = v[1];
                q[3] = -v[0];
                q[6] = v[3];
                q[7] = -v[2];
            }
        }
    }
}

// Place of value c (see fg_columns_kernel) of column (row) i at point p2 in B: the
// pixel kernel's shared-memory tile, in one piece per tile: 32 columns [point][8][32],
// on the uniform-q detector 4 rows [point][4][8].
__device__ __forceinline__ size_t fg_B_at(const FieldGrid &f, int p2, int c, int i) {
    return f.uniform ? ((size_t)(i >> 2) * f.H2 + p2) * 32 + (i & 3) * 8 + c
                     : ((size_t)(i >> 5) * f.H2 + p2) * 256 + c * 32 + (i & 31);
}

// Interpolation along the per-column (per-row) direction, after adding the
// slice chunks: B of 32 columns at one point of the per-pixel direction, values
// [2 parity 1 + parity 2] x (re, im), with the constants of the
// per-pixel direction's points folded in (c_a x_a on even parts, c_a on odd).
// The points are split over eight warps: the sums are short and wait for their
// loads, so the launch is as long as the longest chain of them.
template <typename R>
__global__ void __launch_bounds__(256) fg_columns_kernel(FieldGrid f) {
    using V4 = typename Fg<R>::V4;
    extern __shared__ __align__(32) unsigned char smem[];
    R *q = reinterpret_cast<R *>(smem);                 // [point 1][8]
    __shared__ R part[8][8][32];
    const int p2 = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
    const size_t chunk = (size_t)f.Hs * f.Ht * 8;
    pdl_wait();
    for (int k = threadIdx.x; k < f.H1 * 8; k += blockDim.x) {
        const int p1 = k >> 3, c = k & 7;
        const int a = f.uniform ? p1 : p2, b = f.uniform ? p2 : p1;
        const R *src = (const R *)f.Q + ((size_t)a * f.Ht + b) * 8 + c;
        R v = (R)0;
        for (int j0 = 0; j0 < f.jc; j0 += 8) {
            R t[8];                                     // eight chunks' loads in flight, added in order
#pragma unroll
            for (int j = 0; j < 8; ++j) t[j] = j0 + j < f.jc ? src[(j0 + j) * chunk] : (R)0;
#pragma unroll
            for (int j = 0; j < 8; ++j) v += t[j];
        }
        // first parity = that of direction 1: t on the flat detector, s on the uniform-q one
        const int pq = c >> 1, d = f.uniform ? pq : ((pq & 1) << 1) | (pq >> 1);
        q[p1 * 8 + 2 * d + (c & 1)] = v;
    }
    __syncthreads();
    const R *we = (const R *)f.w1, *wo = we + (size_t)f.H1 * f.n1;
    R acc[8] = {};
    if (i < f.n1) {
        for (int p0 = warp; p0 < f.H1; p0 += 32) {
            R e[4], o[4];                               // four points' weights in flight
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const int p = p0 + 8 * m;
                e[m] = p < f.H1 ? we[(size_t)p * f.n1 + i] : (R)0;
                o[m] = p < f.H1 ? wo[(size_t)p * f.n1 + i] : (R)0;
            }
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const int p = p0 + 8 * m;
                if (p >= f.H1) break;
                const V4 a = *reinterpret_cast<const V4 *>(q + p * 8), b = *reinterpret_cast<const V4 *>(q + p * 8 + 4);
                acc[0] = fma(e[m], a.x, acc[0]);
                acc[1] = fma(e[m], a.y, acc[1]);
                acc[2] = fma(e[m], a.z, acc[2]);
                acc[3] = fma(e[m], a.w, acc[3]);
                acc[4] = fma(o[m], b.x, acc[4]);
                acc[5] = fma(o[m], b.y, acc[5]);
                acc[6] = fma(o[m], b.z, acc[6]);
                acc[7] = fma(o[m], b.w, acc[7]);
            }
        }
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) part[warp][c][lane] = acc[c];
    __syncthreads();
    const int c = warp;                                 // this thread's value
    R v = part[0][c][lane];
#pragma unroll
    for (int w = 1; w < 8; ++w) v += part[w][c][lane];
    const V4 n = ((const V4 *)f.node2)[p2];
    // (columns past the last one are zero: the tiles are whole)
    ((R *)f.B)[fg_B_at(f, p2, c, i)] = v * (((c >> 1) & 1) ? n.w : n.z);
}

// Field and intensity of the pixels: a thread interpolates kPts quadruples of
// mirrored pixels, sharing the loads of B (flat: kPts rows of one column; uniform:
// kPts columns of one row).  A block's part of B (43 KB for 42 points) is one
// piece of memory, copied with all its loads in flight.
// kSplit (small detectors in FP64, of which a warp runs an operation in 64 cycles): the
// four warps share one row, each takes a quarter of the points, a quarter of the
// sums and one of the four mirrored pixels (32^3 on 64^2: 16 us with a warp per row).
template <typename R, typename IO, int kPts, bool kUniform, int kWarps, bool kSplit>
__global__ void __launch_bounds__(32 * kWarps) fg_pixels_out_kernel(FieldGrid f, double str_re, double str_im,
                                                            typename Fg<IO>::C *__restrict__ A, IO *__restrict__ I) {
    using C = typename Fg<IO>::C;
    using V4 = typename Fg<R>::V4;
    static_assert(!kUniform || kWarps == 4, "a warp per row");
    extern __shared__ __align__(32) unsigned char smem[];
    R *sB = reinterpret_cast<R *>(smem);
    V4 *sN = reinterpret_cast<V4 *>(sB + (size_t)f.H2 * 8 * (kUniform ? 4 : 32));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // flat: 32 columns x kWarps warps x kPts rows; uniform: 4 rows (one per warp) x 32 kPts columns
    const int tile = kUniform ? blockIdx.y : blockIdx.x;
    const int count = f.H2 * 8 * (kUniform ? 4 : 32);
    for (int k = threadIdx.x; k < f.H2; k += 32 * kWarps) sN[k] = ((const V4 *)f.node2)[k];
    pdl_wait();
    const R *src = (const R *)f.B + (size_t)tile * count;
    for (int k = threadIdx.x * (16 / sizeof(R)); k < count; k += 32 * kWarps * (16 / sizeof(R)))
        cp_async16(sB + k, src + k);
    cp_async_wait_all();
    __syncthreads();
    int u[kPts], v[kPts];
    V4 px[kPts];
    R acc[kPts][8];
#pragma unroll
    for (int p = 0; p < kPts; ++p) {
        u[p] = kUniform ? (blockIdx.x * kPts + p) * 32 + lane : blockIdx.x * 32 + lane;
        v[p] = kSplit ? blockIdx.y : kUniform ? blockIdx.y * 4 + warp : (blockIdx.y * kWarps + warp) * kPts + p;
        px[p].x = px[p].y = px[p].z = px[p].w = (R)0;
        if (u[p] < f.U && v[p] < f.V) px[p] = ((const V4 *)f.pix)[(size_t)v[p] * f.U + u[p]];
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[p][c] = (R)0;
    }
#pragma unroll 2
    for (int a = kSplit ? warp : 0; a < f.H2; a += kSplit ? kWarps : 1) {
        const V4 n = sN[a];
        R b[8];
        if (kUniform) {
            const V4 *q = reinterpret_cast<const V4 *>(sB + (a * 4 + warp) * 8);
            const V4 q0 = q[0], q1 = q[1];
            b[0] = q0.x;
            b[1] = q0.y;
            b[2] = q0.z;
            b[3] = q0.w;
            b[4] = q1.x;
            b[5] = q1.y;
            b[6] = q1.z;
            b[7] = q1.w;
        } else {
#pragma unroll
            for (int c = 0; c < 8; ++c) b[c] = sB[(a * 8 + c) * 32 + lane];
        }
#pragma unroll
        for (int p = 0; p < kPts; ++p) {
            const R r = fg_recip(px[p].x, px[p].y, n.x, n.y);
#pragma unroll
            for (int c = 0; c < 8; ++c) acc[p][c] = fma(r, b[c], acc[p][c]);
        }
    }
    if constexpr (kSplit) {
        static_assert(kPts == 1 && kWarps == 4 && !kUniform, "a quarter each");
        __shared__ R part[4][8][32];
#pragma unroll
        for (int c = 0; c < 8; ++c) part[warp][c][lane] = acc[0][c];
        __syncthreads();
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            R *q = &part[0][2 * warp + c][lane];
            q[0] = (q[0] + q[8 * 32]) + (q[2 * 8 * 32] + q[3 * 8 * 32]);
        }
        __syncthreads();
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[0][c] = part[0][c][lane];
    }
#pragma unroll
    for (int p = 0; p < kPts; ++p) {
        if (u[p] >= f.U || v[p] >= f.V) continue;
        const bool off = !(px[p].z == px[p].z);          // no scattering direction: A = 0
        const R we = px[p].w, wo = px[p].w * px[p].z;
        // [2 d1 + d2]: combine the per-pixel direction's parities, then the other's
        R g[2][4];                                       // [sign of direction 2][parity 1][re, im]
#pragma unroll
        for (int d1 = 0; d1 < 2; ++d1)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int k = 4 * d1 + c;
                const R e = we * acc[p][k], o = wo * acc[p][k + 2];
                g[0][2 * d1 + c] = e + o;
                g[1][2 * d1 + c] = e - o;
            }
#pragma unroll
        for (int m2 = 0; m2 < 2; ++m2)
#pragma unroll
            for (int m1 = 0; m1 < 2; ++m1) {
                if (kSplit && warp != 2 * m2 + m1) continue;
                const int mu = kUniform ? m2 : m1, mv = kUniform ? m1 : m2;
                const int iu = mu ? fg_minus(u[p], f.det_nx) : fg_plus(u[p], f.det_nx);
                const int iv = mv ? fg_minus(v[p], f.det_ny) : fg_plus(v[p], f.det_ny);
                const R re = m1 ? g[m2][0] - g[m2][2] : g[m2][0] + g[m2][2];
                const R im = m1 ? g[m2][1] - g[m2][3] : g[m2][1] + g[m2][3];
                const R ox = off ? (R)0 : (R)str_re * re - (R)str_im * im;
                const R oy = off ? (R)0 : (R)str_re * im + (R)str_im * re;
                const size_t at = (size_t)iv * f.det_nx + iu;
                C o;
                o.x = (IO)ox;
                o.y = (IO)oy;
                A[at] = o;
                I[at] = (IO)(ox * ox + oy * oy);
            }
    }
}

// ---------------------------------------------------------------------------
// Forward launches
// ---------------------------------------------------------------------------

template <typename R, typename IO, int kRpt>
static cudaError_t fg_run_y(const FieldGrid &f, const void *s, const int *bounds, cudaStream_t st) {
    const size_t smem = sizeof(FgTile<R, kRpt>);
    cudaError_t e = fg_smem(fg_y_kernel<R, IO, kRpt>, smem);
    if (e != cudaSuccess) return e;
    const dim3 grid((f.nx + 31) / 32, f.nz, (f.Hs + 8 * kRpt - 1) / (8 * kRpt));
    return launch_pdl(fg_y_kernel<R, IO, kRpt>, grid, dim3(kFgThreads), smem, st, f, (const typename Fg<IO>::C *)s, bounds);
}

template <typename R, int kRpt, bool kPm>
static cudaError_t fg_run_xz(const FieldGrid &f, int Nxp, const int *bounds, const int *chunk_y, cudaStream_t st) {
    const size_t smem = sizeof(FgTile<R, kRpt>);
    cudaError_t e = fg_smem(fg_xz_kernel<R, kRpt, kPm>, smem);
    if (e != cudaSuccess) return e;
    const dim3 grid(f.Hs, f.jc, (f.Ht + 8 * kRpt - 1) / (8 * kRpt));
    return launch_pdl(fg_xz_kernel<R, kRpt, kPm>, grid, dim3(kFgThreads), smem, st, f, Nxp, bounds, chunk_y);
}

template <typename R, typename IO, int kPts, bool kUniform, int kWarps, bool kSplit = false>
static cudaError_t fg_run_pixels(const FieldGrid &f, double str_re, double str_im, void *A, void *I, cudaStream_t st) {
    using V4 = typename Fg<R>::V4;
    const size_t smem = (size_t)f.H2 * 8 * (kUniform ? 4 : 32) * sizeof(R) + (size_t)f.H2 * sizeof(V4);
    // the largest size any plan uses, so concurrent launches of other handles stay valid
    const size_t most = (size_t)fg_max_half((int)sizeof(R)) * (8 * (kUniform ? 4 : 32) * sizeof(R) + sizeof(V4));
    const auto k = fg_pixels_out_kernel<R, IO, kPts, kUniform, kWarps, kSplit>;
    cudaError_t e = smem <= (size_t)40 << 10 ? cudaSuccess : fg_smem(k, most);
    if (e != cudaSuccess) return e;
    const dim3 grid = kUniform ? dim3((f.U + 32 * kPts - 1) / (32 * kPts), (f.V + 3) / 4)
                 : kSplit ? dim3((f.U + 31) / 32, f.V)
                          : dim3((f.U + 31) / 32, (f.V + kWarps * kPts - 1) / (kWarps * kPts));
    return launch_pdl(k, grid, dim3(32 * kWarps), smem, st, f, str_re, str_im, (typename Fg<IO>::C *)A, (IO *)I);
}

template <typename R, typename IO>
static cudaError_t fg_finish(const FieldGrid &f, double str_re, double str_im, void *A, void *I, int sm_count,
                             cudaStream_t st) {
    cudaError_t e = launch_pdl(fg_columns_kernel<R>, dim3((f.n1 + 31) / 32, f.H2), dim3(256),
                               (size_t)f.H1 * 8 * sizeof(R), st, f);
    if (e != cudaSuccess) return e;
    // more pixels per thread share the loads of B on large detectors; on small
    // ones fewer rows per block fill the SMs
    const long long blocks = (long long)f.U * f.V / 128;
    if (f.uniform)
        return blocks >= 8ll * sm_count   ? fg_run_pixels<R, IO, 4, true, 4>(f, str_re, str_im, A, I, st)
               : blocks >= 2ll * sm_count ? fg_run_pixels<R, IO, 2, true, 4>(f, str_re, str_im, A, I, st)
                                          : fg_run_pixels<R, IO, 1, true, 4>(f, str_re, str_im, A, I, st);
    return blocks >= 8ll * sm_count   ? fg_run_pixels<R, IO, 4, false, 4>(f, str_re, str_im, A, I, st)
           : blocks >= 2ll * sm_count ? fg_run_pixels<R, IO, 1, false, 8>(f, str_re, str_im, A, I, st)
           : 2 * blocks >= sm_count   ? fg_run_pixels<R, IO, 1, false, 4>(f, str_re, str_im, A, I, st)
           : sizeof(R) == 8           ? fg_run_pixels<R, IO, 1, false, 4, true>(f, str_re, str_im, A, I, st)
                                      : fg_run_pixels<R, IO, 1, false, 1>(f, str_re, str_im, A, I, st);
}

template <typename R, typename IO>
static cudaError_t fg_sum_y(const FieldGrid &f, const void *s, const int *bounds, int sm_count, cudaStream_t st) {
    switch (fg_rows_per_thread(f.Hs, (long long)((f.nx + 31) / 32) * f.nz, sizeof(R) == 8, sm_count)) {
        case 1: return fg_run_y<R, IO, 1>(f, s, bounds, st);
        case 2: return fg_run_y<R, IO, 2>(f, s, bounds, st);
        case 3: return fg_run_y<R, IO, 3>(f, s, bounds, st);
        case 5: return fg_run_y<R, IO, 5>(f, s, bounds, st);
        default: return fg_run_y<R, IO, 6>(f, s, bounds, st);
    }
}

template <typename R, bool kPm>
static cudaError_t fg_sum_xz(const FieldGrid &f, int Nxp, const int *bounds, const int *chunk_y, int sm_count,
                             cudaStream_t st) {
    switch (fg_rows_per_thread(f.Ht, (long long)f.Hs * f.jc, sizeof(R) == 8, sm_count)) {
        case 1: return fg_run_xz<R, 1, kPm>(f, Nxp, bounds, chunk_y, st);
        case 2: return fg_run_xz<R, 2, kPm>(f, Nxp, bounds, chunk_y, st);
        case 3: return fg_run_xz<R, 3, kPm>(f, Nxp, bounds, chunk_y, st);
        case 5: return fg_run_xz<R, 5, kPm>(f, Nxp, bounds, chunk_y, st);
        default: return fg_run_xz<R, 6, kPm>(f, Nxp, bounds, chunk_y, st);
    }
}

template <typename R, typename IO>
static cudaError_t fg_forward(const FieldGrid &f, const void *s, const int *bounds, double str_re, double str_im,
                              void *A, void *I, int sm_count, cudaStream_t st) {
    cudaError_t e = fg_sum_y<R, IO>(f, s, bounds, sm_count, st);
    if (e == cudaSuccess) e = fg_sum_xz<R, false>(f, f.nx, bounds, nullptr, sm_count, st);
    return e == cudaSuccess ? fg_finish<R, IO>(f, str_re, str_im, A, I, sm_count, st) : e;
}

double field_grid_issued_flops(const FieldGrid &f, const int *bounds) {
    // a folded term of either sum: an FMA each for even and odd parts, 64 columns a block
    constexpr double kTerm = 2.0 * 2.0 * kFgCols;
    double flops = 0.0;
    for (int j0 = 0; j0 < f.nz; j0 += kFgSlices) {
        int kx = 0;
        for (int j = j0; j < j0 + kFgSlices && j < f.nz; ++j) {
            const int xlo = bounds[j], xhi = bounds[f.nz + j], ylo = bounds[2 * f.nz + j], yhi = bounds[3 * f.nz + j];
            if (xlo >= xhi) continue;
            const FgFold y = fg_fold(ylo, yhi, f.ny);
            flops += kTerm * f.Hs * ((xhi + 31) / 32 - xlo / 32) * (y.end - y.beg);
            kx = std::max(kx, fg_fold(xlo, xhi, f.nx).end);
        }
        flops += kTerm * f.Hs * f.Ht * kx;
    }
    return flops;
}

cudaError_t launch_field_grid(const FieldGrid &f, const void *s, const int *bounds, double str_re, double str_im,
                              void *A, void *I, int sm_count, cudaStream_t st) {
    return f.io == 8     ? fg_forward<double, double>(f, s, bounds, str_re, str_im, A, I, sm_count, st)
           : f.elem == 8 ? fg_forward<double, float>(f, s, bounds, str_re, str_im, A, I, sm_count, st)
                         : fg_forward<float, float>(f, s, bounds, str_re, str_im, A, I, sm_count, st);
}

cudaError_t launch_field_grid_tc(const FieldGrid &f, int Nxp, const int *bounds, const int *chunk_y, double str_re,
                                 double str_im, float2 *A, float *I, int sm_count, cudaStream_t st) {
    const cudaError_t e = fg_sum_xz<float, true>(f, Nxp, bounds, chunk_y, sm_count, st);
    return e == cudaSuccess ? fg_finish<float, float>(f, str_re, str_im, A, I, sm_count, st) : e;
}

}  // namespace scm
