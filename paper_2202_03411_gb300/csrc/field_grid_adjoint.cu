// field_grid_adjoint.cu -- the adjoint field through the sample grid of
// scattering directions (field_grid.cu), its steps transposed.
//
// S_v = sum_p g_p e^{+i q_p r_v}, g = w A, is the transpose of the field's sum.
// Every pixel's phase is the interpolant W_p of the grid's phases, so the
// pixels' weights are first gathered onto the grid,
//   G_ab = sum_p W_p(a, b) g_p
// (along the per-pixel direction, then along the per-column one), and the sum
// over the few thousand grid directions separates over the box,
//   T_a[j][x] = sum_b e^{+i q_z(a,b) z_j} e^{+i q_x(a,b) x} G_ab
//   S[j][x][y] = sum_a e^{+i k0 s_a y} T_a[j][x],
// folded by the signs of s, t, x, y as in the forward sums: a parity of G
// meets only cosines or only sines, and two mirror voxels share a sum.
//
// Short kernels, bound by their launches and the latency of their loads: 48^3 on
// 128^2, FP32: pixels 6.2 us, columns 9.2, x/z 5.4, y 5.9 (the direct sums over pixels
// and voxels: 12.4 ms).
//
// All sums have a fixed order (chunks of pixels are added in order), so the
// gradient is the same bit for bit on every call.
#include "internal.cuh"
#include "field_grid.cuh"

namespace scm {

constexpr int kFaThreads = 256;
constexpr int kFaWarps = kFaThreads / 32;
constexpr int kFaPix = 16;             // pixels along the per-pixel direction per staged tile
constexpr int kFaPts = 4;              // grid points per thread
constexpr int kFaMaxChunks = 32;

// Chunks of the per-pixel direction: enough blocks for two per SM of a
// 152-SM part, no chunk shorter than one staged tile.
static int fa_chunks(const FieldGrid &f) {
    const int n2 = f.uniform ? f.U : f.V;
    const int blocks = ((f.n1 + 31) / 32) * ((f.H2 + kFaWarps * kFaPts - 1) / (kFaWarps * kFaPts));
    int c = (304 + blocks - 1) / blocks;
    const int most = (n2 + kFaPix - 1) / kFaPix;
    c = c > most ? most : c;
    return c < 1 ? 1 : c > kFaMaxChunks ? kFaMaxChunks : c;
}

size_t field_grid_adjoint_layout(FieldGrid *grid, const FieldGrid *fwd, FieldGridAdjoint *a, unsigned char *base) {
    FieldGrid &f = *grid;
    a->own = !(fwd && fwd->elem == f.elem);
    size_t at = 0;
    if (a->own)
        at = field_grid_layout(grid, false, 0, base);
    else
        f = *fwd;
    auto take = [&](size_t bytes) {
        unsigned char *p = base ? base + at : nullptr;
        at += (bytes + 255) / 256 * 256;
        return (void *)p;
    };
    const size_t e = (size_t)f.elem;
    a->chunks = fa_chunks(f);
    a->B = take((size_t)a->chunks * f.H2 * 8 * f.n1 * e);
    a->G = take((size_t)f.Hs * f.Ht * 8 * e);
    a->T = a->own ? take(2 * (size_t)f.Hs * f.nz * f.nx * 2 * e) : f.H;      // (the forward pass is done with H)
    return at;
}

// B[chunk][point 2][parity 1 x parity 2][i]: the pixels of one column (row) i
// and its mirror, gathered onto the points of the per-pixel direction.  A block
// stages the folded weights of 32 columns x kFaPix quadruples of mirrored pixels;
// a thread holds one column and kFaPts points, so a staged quadruple (10 loads)
// serves kFaPts reciprocals and 8 kFaPts FMAs.
template <typename R, bool kUniform>
__global__ void __launch_bounds__(kFaThreads) fa_pixels_kernel(FieldGrid f, FieldGridAdjoint ad,
                                                               const typename Fg<R>::C *__restrict__ A,
                                                               const R *__restrict__ w) {
    using C = typename Fg<R>::C;
    using V4 = typename Fg<R>::V4;
    __shared__ R sh[kFaPix][8][33];
    __shared__ R sx[kFaPix][2][33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i0 = blockIdx.x * 32, n2 = kUniform ? f.U : f.V;
    const int per = (n2 + ad.chunks - 1) / ad.chunks, lo = blockIdx.y * per, hi = min(n2, lo + per);
    const int a0 = blockIdx.z * kFaWarps * kFaPts + warp;
    R nh[kFaPts], nl[kFaPts], acc[kFaPts][8];
#pragma unroll
    for (int k = 0; k < kFaPts; ++k) {
        const int a = a0 + kFaWarps * k;
        nh[k] = nl[k] = (R)0;
        if (a < f.H2) {
            const V4 n = ((const V4 *)f.node2)[a];
            nh[k] = n.x;
            nl[k] = n.y;
        }
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[k][c] = (R)0;
    }
    for (int p0 = lo; p0 < hi; p0 += kFaPix) {
        __syncthreads();
        for (int t = threadIdx.x; t < 32 * kFaPix; t += kFaThreads) {
            // neighbouring threads hold neighbouring pixels of a detector row
            const int il = kUniform ? t / kFaPix : t & 31, pl = kUniform ? t % kFaPix : t >> 5;
            const int i = i0 + il, p = p0 + pl, u = kUniform ? p : i, v = kUniform ? i : p;
            R h[8] = {};
            V4 e;
            e.x = e.y = (R)0;
            if (i < f.n1 && p < hi) {
                e = ((const V4 *)f.pix)[(size_t)v * f.U + u];
                C g[2][2];                              // [sign of direction 1][sign of direction 2]
#pragma unroll
                for (int m1 = 0; m1 < 2; ++m1)
#pragma unroll
                    for (int m2 = 0; m2 < 2; ++m2) {
                        const int mu = kUniform ? m2 : m1, mv = kUniform ? m1 : m2;
                        const int iu = mu ? fg_minus(u, f.det_nx) : fg_plus(u, f.det_nx);
                        const int iv = mv ? fg_minus(v, f.det_ny) : fg_plus(v, f.det_ny);
                        g[m1][m2].x = g[m1][m2].y = (R)0;
                        // (the middle of an odd side counts once)
                        if (!(mu && iu == fg_plus(u, f.det_nx)) && !(mv && iv == fg_plus(v, f.det_ny))) {
                            const size_t at = (size_t)iv * f.det_nx + iu;
                            const C a = A[at];
                            const R wp = w[at];
                            g[m1][m2].x = a.x * wp;
                            g[m1][m2].y = a.y * wp;
                        }
                    }
                const R we = e.w, wo = e.z == e.z ? e.w * e.z : (R)0;     // (off the sphere x = 0)
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const R pp = c ? g[0][0].y : g[0][0].x, pm = c ? g[0][1].y : g[0][1].x;
                    const R mp = c ? g[1][0].y : g[1][0].x, mm = c ? g[1][1].y : g[1][1].x;
                    const R s0 = pp + mp, s1 = pm + mm, d0 = pp - mp, d1 = pm - mm;
                    h[c] = we * (s0 + s1);
                    h[2 + c] = wo * (s0 - s1);
                    h[4 + c] = we * (d0 + d1);
                    h[6 + c] = wo * (d0 - d1);
                }
            }
#pragma unroll
            for (int c = 0; c < 8; ++c) sh[pl][c][il] = h[c];
            sx[pl][0][il] = e.x;
            sx[pl][1][il] = e.y;
        }
        __syncthreads();
        const int n = min(kFaPix, hi - p0);
        for (int pl = 0; pl < n; ++pl) {
            const R xh = sx[pl][0][lane], xl = sx[pl][1][lane];
            R h[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) h[c] = sh[pl][c][lane];
#pragma unroll
            for (int k = 0; k < kFaPts; ++k) {
                const R r = fg_recip(xh, xl, nh[k], nl[k]);
#pragma unroll
                for (int c = 0; c < 8; ++c) acc[k][c] = fma(r, h[c], acc[k][c]);
            }
        }
    }
    if (i0 + lane >= f.n1) return;
#pragma unroll
    for (int k = 0; k < kFaPts; ++k) {
        const int a = a0 + kFaWarps * k;
        if (a >= f.H2) continue;
        R *out = (R *)ad.B + ((size_t)blockIdx.y * f.H2 + a) * 8 * f.n1 + i0 + lane;
#pragma unroll
        for (int c = 0; c < 8; ++c) out[(size_t)c * f.n1] = acc[k][c];
    }
}

// G[a][b][parity s x parity t]: the columns (rows) gathered onto the other
// direction's points.  Block: one point of the per-pixel direction; it adds the
// chunks of kFaCols columns in shared memory, then a warp sums kFaColPts points
// over them, its lanes along the columns.  (Five points per warp, so that one block
// adds the chunks for all: 11.7 us instead of 9.2 at 48^3 on 128^2 pixels, the
// points' sums are as long a chain as the chunks'.)
constexpr int kFaCols = 256;
constexpr int kFaColPts = 2;

template <typename R>
__global__ void __launch_bounds__(kFaThreads) fa_columns_kernel(FieldGrid f, FieldGridAdjoint ad) {
    using V4 = typename Fg<R>::V4;
    __shared__ R sb[8][kFaCols];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, p2 = blockIdx.x;
    const int q0 = (blockIdx.y * kFaWarps + warp) * kFaColPts;
    const V4 nd = ((const V4 *)f.node2)[p2];
    const R *we = (const R *)f.w1, *wo = we + (size_t)f.H1 * f.n1;
    const size_t chunk = (size_t)f.H2 * 8 * f.n1;
    R acc[kFaColPts][8];
#pragma unroll
    for (int k = 0; k < kFaColPts; ++k)
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[k][c] = (R)0;
    for (int i0 = 0; i0 < f.n1; i0 += kFaCols) {
        const int n = min(kFaCols, f.n1 - i0);
        __syncthreads();
        for (int t = threadIdx.x; t < 8 * kFaCols; t += kFaThreads) {
            const int c = t / kFaCols, i = t % kFaCols;
            R v = (R)0;
            if (i < n) {
                const R *src = (const R *)ad.B + ((size_t)p2 * 8 + c) * f.n1 + i0 + i;
                for (int k = 0; k < ad.chunks; k += 8) {
                    R part[8];                          // eight chunks' loads in flight, added in order
#pragma unroll
                    for (int q = 0; q < 8; ++q) part[q] = k + q < ad.chunks ? src[(k + q) * chunk] : (R)0;
#pragma unroll
                    for (int q = 0; q < 8; ++q) v += part[q];
                }
                v *= ((c >> 1) & 1) ? nd.w : nd.z;      // the per-pixel direction's constants: c_a x_a even, c_a odd
            }
            sb[c][i] = v;
        }
        __syncthreads();
#pragma unroll 2
        for (int i = lane; i < n; i += 32) {
            R b[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) b[c] = sb[c][i];
#pragma unroll
            for (int k = 0; k < kFaColPts; ++k) {
                if (q0 + k >= f.H1) break;
                const R e = we[(size_t)(q0 + k) * f.n1 + i0 + i], o = wo[(size_t)(q0 + k) * f.n1 + i0 + i];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    acc[k][c] = fma(e, b[c], acc[k][c]);
                    acc[k][4 + c] = fma(o, b[4 + c], acc[k][4 + c]);
                }
            }
        }
    }
#pragma unroll
    for (int k = 0; k < kFaColPts; ++k) {
        if (q0 + k >= f.H1) continue;
#pragma unroll
        for (int c = 0; c < 8; ++c)
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc[k][c] += __shfl_xor_sync(0xffffffffu, acc[k][c], o);
        if (lane == 0) {
            const int a = f.uniform ? q0 + k : p2, b = f.uniform ? p2 : q0 + k;
            // [2 d1 + d2] to [2 d_s + d_t]: direction 1 is t on the flat detector, s on the uniform-q one
            R g[8];
#pragma unroll
            for (int d = 0; d < 4; ++d) {
                const int e = ((d & 1) << 1) | (d >> 1);
                g[2 * d] = f.uniform ? acc[k][2 * d] : acc[k][2 * e];
                g[2 * d + 1] = f.uniform ? acc[k][2 * d + 1] : acc[k][2 * e + 1];
            }
            R *out = (R *)ad.G + ((size_t)a * f.Ht + b) * 8;
#pragma unroll
            for (int c = 0; c < 8; ++c) out[c] = g[c];
        }
    }
}

// The even (group 0) and odd (group 1) parts of a block's rows, exchanged
// through shared memory: E[group][row][column], row stride kFgCols + 2.
template <typename R, int kRpt>
__device__ __forceinline__ R *fa_exchange(R *E, int grp, int bg, int cg, const R (&acc)[kRpt][4]) {
    constexpr int kS = kFgCols + 2;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kRpt; ++i) {
        R *e = E + (size_t)(grp * 8 * kRpt + bg + 8 * i) * kS + 4 * cg;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            // the sines carry i
            e[2 * c] = grp ? -acc[i][2 * c + 1] : acc[i][2 * c];
            e[2 * c + 1] = grp ? acc[i][2 * c] : acc[i][2 * c + 1];
        }
    }
    __syncthreads();
    return E;
}

template <typename R, int kRpt>
union FaSmem {
    FgTile<R, kRpt, 1> t;
    R E[2 * 8 * kRpt * (kFgCols + 2)];
};

// T[a][even, odd in s][j][x] for one a, 16 slices and 8 kRpt half-coordinates x':
// K runs over the points t_b; a column is one part of (even, odd s) of one slice.
template <typename R, int kRpt>
__global__ void __launch_bounds__(kFgThreads) fa_xz_kernel(FieldGrid f, FieldGridAdjoint ad) {
    using C = typename Fg<R>::C;
    using V4 = typename Fg<R>::V4;
    extern __shared__ __align__(32) unsigned char smem[];
    FaSmem<R, kRpt> &sm = *reinterpret_cast<FaSmem<R, kRpt> *>(smem);
    const int a = blockIdx.x, j0 = blockIdx.y * kFgSlices, r0 = blockIdx.z * 8 * kRpt;
    const int grp = threadIdx.x >> 7, tt = threadIdx.x & 127, cg = tt & 15, bg = tt >> 4;
    const R *cx = (const R *)f.tx + (size_t)a * f.Kx * f.Ht, *sx = cx + (size_t)f.Hs * f.Kx * f.Ht;
    R acc[kRpt][4] = {};
    for (int k0 = 0; k0 < f.Ht; k0 += kFgK) {
        __syncthreads();
        for (int i = threadIdx.x; i < kFgK * 8 * kRpt; i += kFgThreads) {
            const int k = i % kFgK, r = i / kFgK;
            const bool in = k0 + k < f.Ht && r0 + r < f.Kx;
            sm.t.T[0][k][r] = in ? cx[(size_t)(r0 + r) * f.Ht + k0 + k] : (R)0;
            sm.t.T[1][k][r] = in ? sx[(size_t)(r0 + r) * f.Ht + k0 + k] : (R)0;
        }
        for (int i = threadIdx.x; i < kFgSlices * kFgK; i += kFgThreads) {
            const int jl = i % kFgSlices, k = i / kFgSlices, j = j0 + jl, b = k0 + k;
            V4 v0, v1;
            v0.x = v0.y = v0.z = v0.w = v1.x = v1.y = v1.z = v1.w = (R)0;
            if (b < f.Ht && j < f.nz) {
                const C z = ((const C *)f.tz)[((size_t)a * f.Ht + b) * f.nz + j];
                const V4 *g = (const V4 *)((const R *)ad.G + ((size_t)a * f.Ht + b) * 8);
                const V4 ge = g[0], go = g[1];          // even s: (even t, odd t); odd s
                // conj(z) times each
                v0.x = z.x * ge.x + z.y * ge.y;
                v0.y = z.x * ge.y - z.y * ge.x;
                v0.z = z.x * go.x + z.y * go.y;
                v0.w = z.x * go.y - z.y * go.x;
                v1.x = z.x * ge.z + z.y * ge.w;
                v1.y = z.x * ge.w - z.y * ge.z;
                v1.z = z.x * go.z + z.y * go.w;
                v1.w = z.x * go.w - z.y * go.z;
            }
            *reinterpret_cast<V4 *>(&sm.t.S[0][k][4 * jl]) = v0;
            *reinterpret_cast<V4 *>(&sm.t.S[1][k][4 * jl]) = v1;
        }
        __syncthreads();
        fg_multiply<R, kRpt, 1>(sm.t, grp, bg, cg, min(kFgK, f.Ht - k0), acc);
    }
    const R *E = fa_exchange<R, kRpt>(sm.E, grp, bg, cg, acc);
    constexpr int kS = kFgCols + 2, kRows = 8 * kRpt;
    for (int i = threadIdx.x; i < kRows * 2 * kFgSlices; i += kFgThreads) {
        const int r = i % kRows, ds = (i / kRows) & 1, jl = i / (2 * kRows), k = r0 + r, j = j0 + jl;
        if (k >= f.Kx || j >= f.nz) continue;
        const R *e = E + (size_t)r * kS + 4 * jl + 2 * ds, *o = e + (size_t)kRows * kS;
        C *out = (C *)ad.T + (((size_t)a * 2 + ds) * f.nz + j) * f.nx;
        const int ip = fg_plus(k, f.nx), im = fg_minus(k, f.nx);
        C v;
        v.x = e[0] + o[0];
        v.y = e[1] + o[1];
        out[ip] = v;
        if (im != ip) {
            v.x = e[0] - o[0];
            v.y = e[1] - o[1];
            out[im] = v;
        }
    }
}

// S[j][x][y] for one slice, 32 columns x and 8 kRpt half-coordinates y': K runs
// over the points s_a.
template <typename R, int kRpt>
__global__ void __launch_bounds__(kFgThreads) fa_y_kernel(FieldGrid f, FieldGridAdjoint ad,
                                                          typename Fg<R>::C *__restrict__ S) {
    using C = typename Fg<R>::C;
    extern __shared__ __align__(32) unsigned char smem[];
    FaSmem<R, kRpt> &sm = *reinterpret_cast<FaSmem<R, kRpt> *>(smem);
    const int j = blockIdx.y, x0 = blockIdx.x * 32, r0 = blockIdx.z * 8 * kRpt;
    const int grp = threadIdx.x >> 7, tt = threadIdx.x & 127, cg = tt & 15, bg = tt >> 4;
    const R *cy = (const R *)f.ty, *sy = cy + (size_t)f.Ky * f.Hs;
    R acc[kRpt][4] = {};
    for (int k0 = 0; k0 < f.Hs; k0 += kFgK) {
        __syncthreads();
        for (int i = threadIdx.x; i < kFgK * 8 * kRpt; i += kFgThreads) {
            const int k = i % kFgK, r = i / kFgK;
            const bool in = k0 + k < f.Hs && r0 + r < f.Ky;
            sm.t.T[0][k][r] = in ? cy[(size_t)(r0 + r) * f.Hs + k0 + k] : (R)0;
            sm.t.T[1][k][r] = in ? sy[(size_t)(r0 + r) * f.Hs + k0 + k] : (R)0;
        }
        for (int i = threadIdx.x; i < 2 * kFgK * 32; i += kFgThreads) {
            const int xl = i & 31, k = (i >> 5) % kFgK, g = i / (32 * kFgK);
            C v;
            v.x = v.y = (R)0;
            if (k0 + k < f.Hs && x0 + xl < f.nx)
                v = ((const C *)ad.T)[(((size_t)(k0 + k) * 2 + g) * f.nz + j) * f.nx + x0 + xl];
            *reinterpret_cast<C *>(&sm.t.S[g][k][2 * xl]) = v;
        }
        __syncthreads();
        fg_multiply<R, kRpt, 1>(sm.t, grp, bg, cg, min(kFgK, f.Hs - k0), acc);
    }
    const R *E = fa_exchange<R, kRpt>(sm.E, grp, bg, cg, acc);
    constexpr int kS = kFgCols + 2, kRows = 8 * kRpt;
    for (int i = threadIdx.x; i < kRows * 32; i += kFgThreads) {
        const int r = i % kRows, xl = i / kRows, k = r0 + r, x = x0 + xl;
        if (k >= f.Ky || x >= f.nx) continue;
        const R *e = E + (size_t)r * kS + 2 * xl, *o = e + (size_t)kRows * kS;
        C *out = S + ((size_t)j * f.nx + x) * f.ny;
        const int ip = fg_plus(k, f.ny), im = fg_minus(k, f.ny);
        C v;
        v.x = e[0] + o[0];
        v.y = e[1] + o[1];
        out[ip] = v;
        if (im != ip) {
            v.x = e[0] - o[0];
            v.y = e[1] - o[1];
            out[im] = v;
        }
    }
}

// ---------------------------------------------------------------------------
// Host
// ---------------------------------------------------------------------------

// Rows per thread whose tiles of 8 kRpt waste least on n rows.
static int fa_rows_per_thread(int n) {
    int best = 3, waste = 1 << 30;
    for (int r : {6, 4, 3}) {
        const int w = (n + 8 * r - 1) / (8 * r) * 8 * r;
        if (w < waste) {
            waste = w;
            best = r;
        }
    }
    return best;
}

template <typename R, int kRpt>
static cudaError_t fa_run_xz(const FieldGrid &f, const FieldGridAdjoint &ad, cudaStream_t st) {
    const size_t smem = sizeof(FaSmem<R, kRpt>);
    cudaError_t e = fg_smem(fa_xz_kernel<R, kRpt>, smem);
    if (e != cudaSuccess) return e;
    fa_xz_kernel<R, kRpt><<<dim3(f.Hs, f.jc, (f.Kx + 8 * kRpt - 1) / (8 * kRpt)), kFgThreads, smem, st>>>(f, ad);
    return cudaGetLastError();
}

template <typename R, int kRpt>
static cudaError_t fa_run_y(const FieldGrid &f, const FieldGridAdjoint &ad, void *S, cudaStream_t st) {
    const size_t smem = sizeof(FaSmem<R, kRpt>);
    cudaError_t e = fg_smem(fa_y_kernel<R, kRpt>, smem);
    if (e != cudaSuccess) return e;
    const dim3 grid((f.nx + 31) / 32, f.nz, (f.Ky + 8 * kRpt - 1) / (8 * kRpt));
    fa_y_kernel<R, kRpt><<<grid, kFgThreads, smem, st>>>(f, ad, (typename Fg<R>::C *)S);
    return cudaGetLastError();
}

template <typename R>
static cudaError_t fa_gather(const FieldGrid &f, const FieldGridAdjoint &ad, const void *A, const void *w,
                             cudaStream_t st) {
    using C = typename Fg<R>::C;
    const dim3 grid((f.n1 + 31) / 32, ad.chunks, (f.H2 + kFaWarps * kFaPts - 1) / (kFaWarps * kFaPts));
    if (f.uniform)
        fa_pixels_kernel<R, true><<<grid, kFaThreads, 0, st>>>(f, ad, (const C *)A, (const R *)w);
    else
        fa_pixels_kernel<R, false><<<grid, kFaThreads, 0, st>>>(f, ad, (const C *)A, (const R *)w);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const dim3 cols(f.H2, (f.H1 + kFaWarps * kFaColPts - 1) / (kFaWarps * kFaColPts));
    fa_columns_kernel<R><<<cols, kFaThreads, 0, st>>>(f, ad);
    return cudaGetLastError();
}

template <typename R>
static cudaError_t fa_run(const FieldGrid &f, const FieldGridAdjoint &ad, const void *A, const void *w, void *S,
                          cudaStream_t st) {
    cudaError_t e = fa_gather<R>(f, ad, A, w, st);
    if (e != cudaSuccess) return e;
    const int rx = fa_rows_per_thread(f.Kx), ry = fa_rows_per_thread(f.Ky);
    e = rx == 3   ? fa_run_xz<R, 3>(f, ad, st)
        : rx == 4 ? fa_run_xz<R, 4>(f, ad, st)
                  : fa_run_xz<R, 6>(f, ad, st);
    if (e != cudaSuccess) return e;
    return ry == 3   ? fa_run_y<R, 3>(f, ad, S, st)
           : ry == 4 ? fa_run_y<R, 4>(f, ad, S, st)
                     : fa_run_y<R, 6>(f, ad, S, st);
}

cudaError_t launch_field_grid_adjoint(const FieldGrid &f, const FieldGridAdjoint &ad, const void *A, const void *w,
                                      void *S, cudaStream_t st) {
    return f.elem == 8 ? fa_run<double>(f, ad, A, w, S, st) : fa_run<float>(f, ad, A, w, S, st);
}

}  // namespace scm
