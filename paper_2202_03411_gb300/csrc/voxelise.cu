// voxelise.cu -- detector q (Eq. 3) and the fused voxeliser + transmission
// scan (Block 5 + Block 9, Eq. 8 of arXiv 2202.03411).
//
// One CTA owns one x column-plane strip: a fixed x and 32 consecutive y lines.
// Each warp takes whole lines along z, 32 consecutive z per step (one per
// lane), and the exclusive prefix C_j = sum_{j'<j} chi is a warp-shuffle scan
// per step plus the running total of the earlier steps.  The slice strength
// s_j = chi_j exp(i k0 dz (n-1) C_j) is staged in shared memory and then
// written out so that consecutive threads store consecutive y -- the
// contraction's operand rows are y-contiguous.
#include "internal.cuh"
#include "shape_device.cuh"

namespace scm {

// ---------------------------------------------------------------------------
// a1: transfer momentum of every flat-detector pixel (Eq. 3).  The pixel sits
// at (X, Y, 1); k_out = k0 (X, Y, 1)/r and q = k_out - k0 z^.  q_z is written
// as -k0 (X^2+Y^2) / (r (1 + r)) to avoid cancellation near the axis.
// ---------------------------------------------------------------------------
__global__ void detector_q_kernel(int det_nx, int det_ny, double h, double k0, double *q) {
    long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    long long n = (long long)det_nx * det_ny;
    if (p >= n) return;
    int u = (int)(p % det_nx);
    int v = (int)(p / det_nx);
    double X = h * (double)(2 * u + 1 - det_nx) / (double)det_nx;
    double Y = h * (double)(2 * v + 1 - det_ny) / (double)det_ny;
    double rho2 = X * X + Y * Y;
    double r = sqrt(rho2 + 1.0);
    q[3 * p + 0] = k0 * X / r;
    q[3 * p + 1] = k0 * Y / r;
    q[3 * p + 2] = -k0 * rho2 / (r * (1.0 + r));
}

cudaError_t launch_detector_q(int det_nx, int det_ny, double theta_max_deg, double k0, double *q,
                              cudaStream_t st) {
    long long n = (long long)det_nx * det_ny;
    double h = tan(theta_max_deg * kPi / 180.0);
    int threads = 256;
    long long blocks = (n + threads - 1) / threads;
    detector_q_kernel<<<(unsigned)blocks, threads, 0, st>>>(det_nx, det_ny, h, k0, q);
    return cudaGetLastError();
}

constexpr int kLinesPerCta = 32;
constexpr int kVoxThreads = 256;
constexpr int kMaxRun = 16;         // z values per lane: nz <= 512 (256 in the FP64 mode)
constexpr int kVoxQueue = 512;      // binary voxels per CTA whose FP64 decision is batched

// s_j = chi_j T_j with T_j = exp(i k0 dz (n-1) C_j) = e^{-k0 dz beta C} e^{-i k0 dz delta C},
// for soft occupancy and for maps with an index per cell (binary shapes of one
// index: voxelise_binary_kernel below).
// A warp takes one (x, y) line at a time; its lanes take 32 consecutive z per
// step, so neighbouring lanes hold neighbouring voxels (and shapes with a radius
// band skip the surface radius where the whole step is clearly inside or outside).
// Pass 1 renders chi into shared memory for all of the CTA's lines.  Pass 2 forms
// the exclusive prefix C_j with a warp scan per step plus the running total
// of earlier steps, then T_j and s_j.  Tiles are [line][z] with a padded row,
// so both the z-walk and the line-fastest output loop are free of bank
// conflicts.
// Per-launch constants of the scan, formed on the host in FP64 and handed
// over in both precisions (no FP64 arithmetic in the kernel's prologue).
struct VoxConst {
    double att, ph, kdz, inv_scale;         // k0 dz beta, k0 dz delta, k0 dz, 1 / nscale
    float att_f, ph_f, kdz_f, inv_scale_f;
};
template <typename T> __device__ __forceinline__ T vc_pick(double d, float f);
template <> __device__ __forceinline__ double vc_pick<double>(double d, float) { return d; }
template <> __device__ __forceinline__ float vc_pick<float>(double, float f) { return f; }

template <bool kFp64, typename ScanT, bool kMaps>
__global__ void __launch_bounds__(kVoxThreads, 3) voxelise_scan_kernel(ShapeParams sp, GridParams gp,
                                                                    SliceOut out, VoxConst vc) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int nz = gp.nz;
    const int zs = nz + 1;                                                    // padded row
    using Cx = typename std::conditional<kFp64, double2, float2>::type;
    using Re = typename std::conditional<kFp64, double, float>::type;
    Cx *s_tile = reinterpret_cast<Cx *>(smem);                                // [32][zs]
    float *chi_tile = reinterpret_cast<float *>(smem + sizeof(Cx) * zs * kLinesPerCta);
    pdl_wait();

    const int ix = blockIdx.x;
    const int y0 = blockIdx.y * kLinesPerCta;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int steps = (nz + 31) / 32;
    const ScanT a_att = vc_pick<ScanT>(vc.att, vc.att_f);         // attenuation per unit C
    const ScanT a_ph = vc_pick<ScanT>(vc.ph, vc.ph_f);             // phase per unit C
    const bool varn = kMaps && sp.varn != 0;                      // per-cell index of a volume map
    const ScanT kdz = vc_pick<ScanT>(vc.kdz, vc.kdz_f);
    const Re inv_scale = vc_pick<Re>(vc.inv_scale, vc.inv_scale_f);
    // radius band (harmonics, radii maps, soft spheres and ellipsoids): inside below lo, outside above hi
    // (the host sets none for FP64 soft occupancy)
    const bool band = (!kFp64 || !sp.soft) && sp.band_hi > 0.f;
    const float vox = gp.voxf;
    const float xo = ((float)ix - 0.5f * (float)(gp.nx - 1)) * vox - sp.cxf;

    for (int yl = warp; yl < kLinesPerCta; yl += kVoxThreads / 32) {
        const int iy = y0 + yl;
        if (iy >= gp.ny) break;
        const float yo = ((float)iy - 0.5f * (float)(gp.ny - 1)) * vox - sp.cyf;
        const float r2xy = xo * xo + yo * yo;
        Cx *srow = s_tile + (size_t)yl * zs;
        float *crow = chi_tile + (size_t)yl * zs;
        // pass 1: occupancy (and, with a per-cell index, the cells' delta and beta)
#pragma unroll 1
        for (int st = 0; st < steps; ++st) {
            const int iz = 32 * st + lane;
            Re c = (Re)0;                       // FP32 in the FP32 modes: no FP64 on the common path
            if (iz < nz) {
                bool decided = false;
                if (band) {
                    // |p| = |d|: the rotation keeps lengths; margins cover FP32 rounding
                    const float zo = ((float)iz - 0.5f * (float)(nz - 1)) * vox - sp.czf;
                    const float d = sqrtf(r2xy + zo * zo);
                    const float m = 1e-3f * vox + 1e-5f * d;
                    if (d + m < sp.band_lo) {
                        c = (Re)1;
                        decided = true;
                    } else if (d - m > sp.band_hi) {
                        decided = true;
                    }
                }
                if (!decided) {
                    if (varn) {
                        const int cell = vmap_cell<kFp64>(sp, gp, ix, iy, iz);
                        c = (cell >= 0 && sp.vmap[cell] != 0) ? (Re)1 : (Re)0;
                    } else {
                        c = (Re)occupancy<kFp64, kMaps>(sp, gp, ix, iy, iz);
                    }
                }
                if (kFp64) srow[iz].x = c;                                // exact copy until pass 2
                crow[iz] = (float)c;
            }
        }
    }
    __syncthreads();
    for (int yl = warp; yl < kLinesPerCta; yl += kVoxThreads / 32) {
        const int iy = y0 + yl;
        if (iy >= gp.ny) break;
        Cx *srow = s_tile + (size_t)yl * zs;
        float *crow = chi_tile + (size_t)yl * zs;
        // pass 2: exclusive prefix along z, transmission, slice value
        ScanT carry = (ScanT)0, carry_d = (ScanT)0, carry_b = (ScanT)0;
#pragma unroll 1
        for (int st = 0; st < steps; ++st) {
            const int iz = 32 * st + lane;
            const Re chi = iz < nz ? (kFp64 ? (Re)srow[iz].x : (Re)crow[iz]) : (Re)0;
            if (varn) {
                // voxel-resolved index: T_j = exp(i k0 dz sum_{j'<j} chi (n_v - 1)),
                // s = chi (n_v^2 - 1) T / nscale (Eq. 8-9 with one n per voxel)
                double dl = 0.0, bt = 0.0;
                if (chi != (Re)0) {
                    const int cell = vmap_cell<kFp64>(sp, gp, ix, iy, iz);
                    dl = sp.mdelta[cell];
                    bt = sp.mbeta[cell];
                }
                const ScanT ed = (ScanT)(chi * (Re)dl), eb = (ScanT)(chi * (Re)bt);
                ScanT id = ed, ib = eb;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const ScanT a = __shfl_up_sync(0xffffffffu, id, o);
                    const ScanT b = __shfl_up_sync(0xffffffffu, ib, o);
                    if (lane >= o) {
                        id += a;
                        ib += b;
                    }
                }
                const ScanT Cd = carry_d + id - ed, Cb = carry_b + ib - eb;
                carry_d += __shfl_sync(0xffffffffu, id, 31);
                carry_b += __shfl_sync(0xffffffffu, ib, 31);
                if (iz < nz) {
                    Cx v;
                    v.x = v.y = (Re)0;
                    if (chi != (Re)0) {
                        const ScanT mag = exp(-kdz * Cb);
                        ScanT sn, cs;
                        sincos(kdz * Cd, &sn, &cs);
                        const Re sr = (Re)((-2.0 * dl + dl * dl - bt * bt)) * inv_scale;
                        const Re si = (Re)((2.0 * bt - 2.0 * dl * bt)) * inv_scale;
                        const Re tr = (Re)(mag * cs), ti = -(Re)(mag * sn);
                        v.x = chi * (sr * tr - si * ti);
                        v.y = chi * (sr * ti + si * tr);
                    }
                    srow[iz] = v;
                }
                continue;
            }
            ScanT incl = (ScanT)chi;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const ScanT nb = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += nb;
            }
            const ScanT C = carry + incl - (ScanT)chi;
            carry += __shfl_sync(0xffffffffu, incl, 31);
            if (iz < nz) {
                Cx v;
                v.x = v.y = (Re)0;                 // s = chi T vanishes with chi: no T needed
                if (chi != (Re)0) {
                    const ScanT mag = exp(-a_att * C);
                    ScanT sn, cs;
                    sincos(a_ph * C, &sn, &cs);
                    v.x = chi * (Re)(mag * cs);
                    v.y = -chi * (Re)(mag * sn);
                }
                srow[iz] = v;
            }
        }
    }
    __syncthreads();

    const int ny_here = min(kLinesPerCta, gp.ny - y0);
    const long long nxy = (long long)gp.nx * gp.ny;
    if (out.bounds) {
        // occupied box of each slice (order-independent min/max)
        for (int iz = threadIdx.x; iz < nz; iz += kVoxThreads) {
            int lo = kLinesPerCta, hi = -1;
            for (int yl = 0; yl < ny_here; ++yl)
                if (chi_tile[(size_t)yl * (nz + 1) + iz] != 0.f) {
                    lo = min(lo, yl);
                    hi = yl;
                }
            if (hi >= 0) {
                atomicMin(&out.bounds[iz], ix);
                atomicMax(&out.bounds[nz + iz], ix + 1);
                atomicMin(&out.bounds[2 * nz + iz], y0 + lo);
                atomicMax(&out.bounds[3 * nz + iz], y0 + hi + 1);
                if (out.chunk_y) {
                    // y range of this slice's 8-column chunk (tensor-core grids: ix < 8 kGeomChunks)
                    const int c = iz * kGeomChunks + (ix >> 3);
                    atomicMin(&out.chunk_y[c], y0 + lo);
                    atomicMax(&out.chunk_y[kGeomChunks * nz + c], y0 + hi + 1);
                }
            }
        }
    }
    for (int it = threadIdx.x; it < nz * kLinesPerCta; it += kVoxThreads) {
        const int iz = it / kLinesPerCta, yl = it % kLinesPerCta;
        if (yl >= ny_here) continue;
        const int iy = y0 + yl;
        const Cx v = s_tile[(size_t)yl * (nz + 1) + iz];
        const long long vidx = iz * nxy + (long long)ix * gp.ny + iy;
        out.chi[vidx] = chi_tile[(size_t)yl * (nz + 1) + iz];
        if (out.layout == kLayoutC64) {
            reinterpret_cast<double2 *>(out.s)[vidx] = make_double2((double)v.x, (double)v.y);
        } else if (out.layout == kLayoutC32) {
            reinterpret_cast<float2 *>(out.s)[vidx] = make_float2((float)v.x, (float)v.y);
        } else {
            // tensor-core slice operand: three planes per slice, rows
            // (3j + 0) Nxp + x = -Im s, (3j + 1) Nxp + x = Re s, (3j + 2) Nxp + x = Im s,
            // each row running over y (msft_tc.cu reads [Re | Im] and [-Im | Re] windows)
            const size_t row_n = (size_t)iz * 3 * out.Nxp + ix;
            const size_t row_r = row_n + out.Nxp;
            const size_t row_i = row_r + out.Nxp;
            const float sr = (float)v.x, si = (float)v.y;
            if (out.layout == kLayoutTcF16) {
                __half *B = reinterpret_cast<__half *>(out.s);
                B[row_n * out.Kp + iy] = __float2half_rn(-si);
                B[row_r * out.Kp + iy] = __float2half_rn(sr);
                B[row_i * out.Kp + iy] = __float2half_rn(si);
            } else {
                __nv_bfloat16 *B = reinterpret_cast<__nv_bfloat16 *>(out.s);
                B[row_n * out.Kp + iy] = __float2bfloat16_rn(-si);
                B[row_r * out.Kp + iy] = __float2bfloat16_rn(sr);
                B[row_i * out.Kp + iy] = __float2bfloat16_rn(si);
            }
        }
    }
}

// T after C full voxels of the beam's path, (Re, Im) in the slices' precision.
template <typename ScanT, typename Cx>
__device__ __forceinline__ Cx full_voxels_T(const VoxConst &vc, int C) {
    const ScanT mag = exp(-vc_pick<ScanT>(vc.att, vc.att_f) * (ScanT)C);
    ScanT sn, cs;
    sincos(vc_pick<ScanT>(vc.ph, vc.ph_f) * (ScanT)C, &sn, &cs);
    Cx v;
    v.x = mag * cs;
    v.y = -(mag * sn);
    return v;
}

// ---------------------------------------------------------------------------
// Binary shapes of one index.  A voxel is a bit, C_j is a count of bits, and T
// takes only the nz + 1 values of a table, so nothing of the scan runs per
// voxel: a line of 32 z is one ballot, its prefix a popcount, its transmission a
// load.  The FP64 modes settle a voxel in FP32 where the margin allows it, as
// the FP32 modes do (the decision is the FP64 one either way).
//
// A CTA owns kLines y lines at one x, a warp takes whole lines.  What is left
// is the surface radius near the surface: harmonics cost several hundred instructions
// a voxel, so first the radius band and then a table of radii over a cube of
// directions (6 x 64^2 for a radius of 48 voxels, good to the shape's steepest
// slope times half a cell, about 1.4 voxels there) settle what they can, and the
// voxels left are queued and evaluated by full warps.  Stores are 16 bytes per
// thread and plane.  Few lines per CTA keep the SMs evenly loaded (planes
// through the middle carry most of the surface): 16, and 8 where 16 would leave
// SMs without a CTA.
// ---------------------------------------------------------------------------
constexpr int kBitSteps = kMaxRun + 1;       // padded row of a line's bit words

// Coefficients staged in memory for the voxeliser: ShTerms, then the FP64 tables.
// (Kernel parameters serve one address at a time, so reading them by lane is slow:
// once per launch, not per CTA.)
static_assert(sizeof(ShTerms) + kShTabDoubles * sizeof(double) <= kShStageInts * sizeof(int) &&
                  sizeof(ShTerms) % 16 == 0,
              "staged coefficients");
__device__ __forceinline__ void block_copy(void *dst, const void *src, size_t bytes) {
    for (int k = threadIdx.x; k < (int)(bytes / 8); k += blockDim.x)
        reinterpret_cast<uint2 *>(dst)[k] = reinterpret_cast<const uint2 *>(src)[k];
}

// (relative error below 1e-6)
__device__ __forceinline__ float sqrt_approx(float x) {
    float r;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Cell of direction p in the radius table: cube face, then the two tangents.
__device__ __forceinline__ int rtab_cell(float px, float py, float pz, int n) {
    const float ax = fabsf(px), ay = fabsf(py), az = fabsf(pz);
    int face;
    float m, a, b;
    if (ax >= ay && ax >= az) {
        face = 0;
        m = px;
        a = py;
        b = pz;
    } else if (ay >= az) {
        face = 2;
        m = py;
        a = pz;
        b = px;
    } else {
        face = 4;
        m = pz;
        a = px;
        b = py;
    }
    if (m < 0.f) ++face;
    const float s = __fdividef(0.5f * (float)n, fabsf(m)), h = 0.5f * (float)n;
    const int i = min(n - 1, max(0, (int)fmaf(a, s, h))), j = min(n - 1, max(0, (int)fmaf(b, s, h)));
    return (face * n + i) * n + j;
}

// Radius at the centre of cell k (see rtab_cell).
__device__ __forceinline__ float rtab_radius(const ShapeParams &sp, const ShTerms &tab, int k) {
    const int n = sp.rtab_n, face = k / (n * n), i = (k / n) % n, j = k % n;
    const float m = (face & 1) ? -1.f : 1.f, a = (2 * i + 1) / (float)n - 1.f, b = (2 * j + 1) / (float)n - 1.f;
    const float px = face < 2 ? m : face < 4 ? b : a, py = face < 2 ? a : face < 4 ? m : b;
    const float pz = face < 2 ? b : face < 4 ? a : m;
    return sh_radius_f(sp, tab, px, py, pz, rsqrtf(px * px + py * py + pz * pz));
}

template <bool kFp64, typename ScanT, bool kMaps, int kLines>
__global__ void __launch_bounds__(kVoxThreads, 3) voxelise_binary_kernel(ShapeParams sp, GridParams gp, SliceOut out,
                                                                         VoxConst vc) {
    using Cx = typename std::conditional<kFp64, double2, float2>::type;
    extern __shared__ __align__(16) unsigned char smem[];
    Cx *T = reinterpret_cast<Cx *>(smem);                                     // [nz + 1]
    __shared__ __align__(16) double s_tab[kMaps ? 1 : kShTabDoubles];
    __shared__ uint32_t s_bits[kLines][kBitSteps];
    __shared__ int s_base[kLines][kBitSteps];
    uint16_t *near = reinterpret_cast<uint16_t *>(T + gp.nz + 1);             // [kLines nz]: (line << 9) | z
    __shared__ int s_queue[kVoxQueue];                                        // the same, for the FP64 test
    __shared__ int s_nn, s_qn;
    __shared__ ShTerms s_sh;
    if (threadIdx.x == 0) s_nn = s_qn = 0;
    pdl_wait();
    if (!kMaps && sp.kind == SCATMAN_SPHHARM) {
        if (out.stage)
            block_copy(&s_sh, out.stage, sizeof(ShTerms));
        else
            sh_stage_terms(sp, s_sh);
    }
    __syncthreads();
    const int nz = gp.nz, steps = (nz + 31) / 32, ix = blockIdx.x, y0 = blockIdx.y * kLines;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const float vox = gp.voxf;
    const float xo = ((float)ix - 0.5f * (float)(gp.nx - 1)) * vox - sp.cxf;
    const bool band = sp.band_hi > 0.f, rtab = !kMaps && sp.rtab_n > 0 && out.rtab != nullptr;
    const bool fp64_only = kFp64 && !sp.fp32_first;
    // shapes with a costly surface queue their undecided voxels
    const bool dense = sp.kind == SCATMAN_SPHHARM || sp.kind == SCATMAN_RADIALMAP || fp64_only;

    constexpr int kU = 4;                        // steps whose table loads are in flight together
    for (int yl = warp; yl < kLines; yl += kVoxThreads / 32) {
        const int iy = y0 + yl;
        const float yo = ((float)iy - 0.5f * (float)(gp.ny - 1)) * vox - sp.cyf;
        const float r2xy = xo * xo + yo * yo;
        const float rim = sp.band_hi * 1.0001f + 2e-3f * vox;
        if (iy >= gp.ny || (band && r2xy > rim * rim)) {
            // no voxel of the line (the band's margins are within the rim's)
            if (lane < steps) s_bits[yl][lane] = 0u;
            continue;
        }
#pragma unroll 1
        for (int st0 = 0; st0 < steps; st0 += kU) {
            bool in[kU], ask[kU];
            float d[kU], r[kU];
#pragma unroll
            for (int q = 0; q < kU; ++q) {
                const int iz = 32 * (st0 + q) + lane;
                in[q] = false;
                ask[q] = iz < nz;
                d[q] = r[q] = 0.f;
                if (ask[q] && band) {
                    // |p| = |d|: the rotation keeps lengths; margins cover FP32 rounding
                    const float zo = ((float)iz - 0.5f * (float)(nz - 1)) * vox - sp.czf;
                    d[q] = sqrt_approx(r2xy + zo * zo);
                    const float m = 1e-3f * vox + 1e-5f * d[q];
                    in[q] = d[q] + m < sp.band_lo;
                    ask[q] = !in[q] && d[q] - m <= sp.band_hi;
                    if (!kMaps && ask[q] && rtab) {
                        const float px = sp.Rf[0] * xo + sp.Rf[3] * yo + sp.Rf[6] * zo;
                        const float py = sp.Rf[1] * xo + sp.Rf[4] * yo + sp.Rf[7] * zo;
                        const float pz = sp.Rf[2] * xo + sp.Rf[5] * yo + sp.Rf[8] * zo;
                        r[q] = __ldg(&out.rtab[rtab_cell(px, py, pz, sp.rtab_n)]);
                    }
                }
            }
#pragma unroll
            for (int q = 0; q < kU; ++q) {
                const int st = st0 + q, iz = 32 * st + lane;
                if (st >= steps) break;
                if (!kMaps && rtab && ask[q]) {
                    const float over = r[q] - d[q];
                    in[q] = over > sp.rtab_slack;
                    ask[q] = fabsf(over) <= sp.rtab_slack;
                }
                if (!dense && ask[q]) {
                    // (a few instructions each: no queue)
                    const float c = occupancy_binary_f<kMaps>(sp, gp, s_sh, ix, iy, iz);
                    in[q] = c > 0.f;
                    if (c < 0.f) {
                        const int slot = atomicAdd(&s_qn, 1);
                        if (slot < kVoxQueue)
                            s_queue[slot] = (yl << 9) | iz;
                        else
                            in[q] = occupancy_binary_fp64(sp, gp, ix, iy, iz) != 0.0;
                    }
                }
                const uint32_t word = __ballot_sync(0xffffffffu, in[q]);
                if (lane == 0) s_bits[yl][st] = word;
                const uint32_t asking = __ballot_sync(0xffffffffu, dense && ask[q]);
                if (asking) {
                    int at = 0;
                    if (lane == 0) at = atomicAdd(&s_nn, __popc(asking));
                    at = __shfl_sync(0xffffffffu, at, 0);
                    if (dense && ask[q]) near[at + __popc(asking & ((1u << lane) - 1u))] = (uint16_t)((yl << 9) | iz);
                }
            }
        }
    }
    for (int k = threadIdx.x; k <= nz; k += kVoxThreads)
        T[k] = out.table ? reinterpret_cast<const Cx *>(out.table)[k] : full_voxels_T<ScanT, Cx>(vc, k);
    __syncthreads();
    if (dense) {
        for (int k = threadIdx.x; k < s_nn; k += kVoxThreads) {
            const int e = near[k], yl = e >> 9, iz = e & 511, iy = y0 + yl;
            bool in = false;
            if (fp64_only) {
                in = occupancy_binary_fp64(sp, gp, ix, iy, iz) != 0.0;
            } else {
                const float c = occupancy_binary_f<kMaps>(sp, gp, s_sh, ix, iy, iz);
                in = c > 0.f;
                if (c < 0.f) {
                    // too close to the surface for FP32: queue it (inline when full)
                    const int slot = atomicAdd(&s_qn, 1);
                    if (slot < kVoxQueue)
                        s_queue[slot] = e;
                    else
                        in = occupancy_binary_fp64(sp, gp, ix, iy, iz) != 0.0;
                }
            }
            if (in) atomicOr(&s_bits[yl][iz >> 5], 1u << (iz & 31));
        }
        __syncthreads();
    }
    const int qn = min(s_qn, kVoxQueue);
    if (qn > 0) {
        // the queued voxels' FP64 decisions: harmonics one voxel per warp, other kinds one per thread
        const bool warps = !kMaps && sp.kind == SCATMAN_SPHHARM;
        if (warps) {
            if (out.stage)
                block_copy(s_tab, reinterpret_cast<const unsigned char *>(out.stage) + sizeof(ShTerms), sizeof(s_tab));
            else
                sh_stage_tables(sp, s_tab);
            __syncthreads();
        }
        for (int k = warps ? warp : threadIdx.x; k < qn; k += warps ? kVoxThreads / 32 : kVoxThreads) {
            const int yl = s_queue[k] >> 9, iz = s_queue[k] & 511;
            const bool in = (warps ? sh_binary_fp64_warp(sp, gp, ix, y0 + yl, iz, s_tab)
                                   : occupancy_binary_fp64(sp, gp, ix, y0 + yl, iz)) != 0.0;
            if (in && !(warps && lane > 0)) atomicOr(&s_bits[yl][iz >> 5], 1u << (iz & 31));
        }
        __syncthreads();
    }
    if (threadIdx.x < kLines) {
        int n = 0;
        for (int st = 0; st < steps; ++st) {
            s_base[threadIdx.x][st] = n;
            n += __popc(s_bits[threadIdx.x][st]);
        }
    }
    if (out.bounds) {
        // occupied box of each slice (order-independent min/max): lane b of step
        // st collects slice 32 st + b's bits of all lines
        for (int st = kVoxThreads / 32 - 1 - warp; st < steps; st += kVoxThreads / 32) {
            const uint32_t w = lane < kLines ? s_bits[lane][st] : 0u;
            uint32_t mine = 0;
#pragma unroll
            for (int b = 0; b < 32; ++b) {
                const uint32_t m = __ballot_sync(0xffffffffu, (w >> b) & 1u);
                if (lane == b) mine = m;
            }
            const int iz = 32 * st + lane;
            if (mine) {
                const int lo = y0 + __ffs(mine) - 1, hi = y0 + 32 - __clz(mine);
                atomicMin(&out.bounds[iz], ix);
                atomicMax(&out.bounds[nz + iz], ix + 1);
                atomicMin(&out.bounds[2 * nz + iz], lo);
                atomicMax(&out.bounds[3 * nz + iz], hi);
                if (out.chunk_y) {
                    // y range of this slice's 8-column chunk (tensor-core grids: ix < 8 kGeomChunks)
                    const int c = iz * kGeomChunks + (ix >> 3);
                    atomicMin(&out.chunk_y[c], lo);
                    atomicMax(&out.chunk_y[kGeomChunks * nz + c], hi);
                }
            }
        }
    }
    __syncthreads();

    const long long nxy = (long long)gp.nx * gp.ny;
    if (out.layout == kLayoutC64 || out.layout == kLayoutC32) {
        for (int it = threadIdx.x; it < nz * kLines; it += kVoxThreads) {
            const int iz = it / kLines, yl = it % kLines, iy = y0 + yl;
            if (iy >= gp.ny) continue;
            const uint32_t w = s_bits[yl][iz >> 5], below = w & ((1u << (iz & 31)) - 1u);
            const bool in = (w >> (iz & 31)) & 1u;
            Cx v;
            v.x = v.y = 0;
            if (in) v = T[s_base[yl][iz >> 5] + __popc(below)];
            const long long at = iz * nxy + (long long)ix * gp.ny + iy;
            out.chi[at] = in ? 1.f : 0.f;
            reinterpret_cast<Cx *>(out.s)[at] = v;
        }
        return;
    }
    if constexpr (!kFp64) {
        // tensor-core slice operand (planes -Im, Re, Im; see voxelise_scan_kernel): a
        // thread packs 8 consecutive y of one slice.  Rows run to Kp, a multiple of
        // 16, so the store past ny falls into the padding, which stays zero.
        constexpr int kGroups = kLines / 8;
        const bool f16 = out.layout == kLayoutTcF16, wide = (gp.ny & 3) == 0;
        for (int it = threadIdx.x; it < nz * kGroups; it += kVoxThreads) {
            const int iz = it / kGroups, yg = 8 * (it % kGroups), iy = y0 + yg;
            if (iy >= gp.ny) continue;
            float re[8], im[8], chi[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const uint32_t w = s_bits[yg + k][iz >> 5], below = w & ((1u << (iz & 31)) - 1u);
                const bool in = (w >> (iz & 31)) & 1u;
                float2 v = make_float2(0.f, 0.f);
                if (in) v = T[s_base[yg + k][iz >> 5] + __popc(below)];
                re[k] = v.x;
                im[k] = v.y;
                chi[k] = in ? 1.f : 0.f;
            }
            uint32_t pr[4], pi[4], pn[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (f16) {
                    const __half2 a = __floats2half2_rn(re[2 * k], re[2 * k + 1]);
                    const __half2 b = __floats2half2_rn(im[2 * k], im[2 * k + 1]);
                    const __half2 c = __floats2half2_rn(-im[2 * k], -im[2 * k + 1]);
                    pr[k] = *reinterpret_cast<const uint32_t *>(&a);
                    pi[k] = *reinterpret_cast<const uint32_t *>(&b);
                    pn[k] = *reinterpret_cast<const uint32_t *>(&c);
                } else {
                    const __nv_bfloat162 a = __floats2bfloat162_rn(re[2 * k], re[2 * k + 1]);
                    const __nv_bfloat162 b = __floats2bfloat162_rn(im[2 * k], im[2 * k + 1]);
                    const __nv_bfloat162 c = __floats2bfloat162_rn(-im[2 * k], -im[2 * k + 1]);
                    pr[k] = *reinterpret_cast<const uint32_t *>(&a);
                    pi[k] = *reinterpret_cast<const uint32_t *>(&b);
                    pn[k] = *reinterpret_cast<const uint32_t *>(&c);
                }
            }
            uint16_t *row = reinterpret_cast<uint16_t *>(out.s) + ((size_t)iz * 3 * out.Nxp + ix) * out.Kp + iy;
            const size_t plane = (size_t)out.Nxp * out.Kp;
            *reinterpret_cast<uint4 *>(row) = make_uint4(pn[0], pn[1], pn[2], pn[3]);
            *reinterpret_cast<uint4 *>(row + plane) = make_uint4(pr[0], pr[1], pr[2], pr[3]);
            *reinterpret_cast<uint4 *>(row + 2 * plane) = make_uint4(pi[0], pi[1], pi[2], pi[3]);
            float *x = out.chi + iz * nxy + (long long)ix * gp.ny + iy;
#pragma unroll
            for (int g = 0; g < 2; ++g) {
                if (wide && iy + 4 * g + 4 <= gp.ny) {
                    *reinterpret_cast<float4 *>(x + 4 * g) =
                        make_float4(chi[4 * g], chi[4 * g + 1], chi[4 * g + 2], chi[4 * g + 3]);
                } else {
#pragma unroll
                    for (int k = 4 * g; k < 4 * g + 4; ++k)
                        if (iy + k < gp.ny) x[k] = chi[k];
                }
            }
        }
    }
}

// Empty bounds, the transmission table (table: the T of 0 .. nz full voxels, or
// null), and in the blocks from `first` on the radius table, after a block that
// stages the coefficients.
template <typename ScanT, typename Cx>
__global__ void voxelise_init_kernel(ShapeParams sp, int *b, int nz, int *cy, Cx *table, VoxConst vc, int first,
                                     void *stage, float *rtab) {
    pdl_wait();
    if ((int)blockIdx.x == first) {
        sh_stage_terms(sp, *reinterpret_cast<ShTerms *>(stage));
        sh_stage_tables(sp, reinterpret_cast<double *>(reinterpret_cast<unsigned char *>(stage) + sizeof(ShTerms)));
        return;
    }
    if ((int)blockIdx.x > first) {
        __shared__ ShTerms s_sh;
        sh_stage_terms(sp, s_sh);
        __syncthreads();
        const int k = (blockIdx.x - first - 1) * blockDim.x + threadIdx.x;
        if (k < 6 * sp.rtab_n * sp.rtab_n) rtab[k] = rtab_radius(sp, s_sh, k);
        return;
    }
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < 4 * nz) {
        const int part = i / nz;
        b[i] = (part == 0 || part == 2) ? 0x7fffffff : 0;     // lo parts start high, hi parts low
    }
    if (cy && i < 2 * kGeomChunks * nz) cy[i] = i < kGeomChunks * nz ? 0x7fffffff : 0;
    const int last = first * blockDim.x - 1 - i;          // the last threads: neither bounds nor many chunks
    if (table && last <= nz) table[last] = full_voxels_T<ScanT, Cx>(vc, last);
}

template <bool kFp64, typename ScanT>
static cudaError_t run_voxelise(const ShapeParams &sp, const GridParams &gp, const SliceOut &out, const VoxConst &vc,
                                cudaStream_t st) {
    using Cx = typename std::conditional<kFp64, double2, float2>::type;
    const bool maps = sp.kind == SCATMAN_RADIALMAP || sp.kind == SCATMAN_VOLUMEMAP;
    const bool binary = !sp.soft && !sp.varn;
    if (out.bounds) {
        const int first = (2 * kGeomChunks * gp.nz + 255) / 256;
        const int cells = binary ? 6 * sp.rtab_n * sp.rtab_n : 0;
        const int more = binary && sp.kind == SCATMAN_SPHHARM ? 1 + (cells + 255) / 256 : 0;
        const cudaError_t e = launch_pdl(voxelise_init_kernel<ScanT, Cx>, dim3(first + more), dim3(256), 0, st, sp,
                                         out.bounds, gp.nz, out.chunk_y, binary ? (Cx *)out.table : nullptr, vc, first,
                                         out.stage, out.rtab);
        if (e != cudaSuccess) return e;
    }
    if (binary) {
        // CTAs of 8 lines where 16 leave fewer than two per SM of a 152-SM part
        const bool small = (long long)gp.nx * ((gp.ny + 15) / 16) < 304;
        const int lines = small ? 8 : 16;
        const size_t smem = sizeof(Cx) * ((size_t)gp.nz + 1) + sizeof(uint16_t) * (size_t)lines * gp.nz;
        const dim3 grid(gp.nx, (gp.ny + lines - 1) / lines);
        auto k = small ? (maps ? voxelise_binary_kernel<kFp64, ScanT, true, 8> : voxelise_binary_kernel<kFp64, ScanT, false, 8>)
                       : (maps ? voxelise_binary_kernel<kFp64, ScanT, true, 16>
                               : voxelise_binary_kernel<kFp64, ScanT, false, 16>);
        return launch_pdl(k, grid, dim3(kVoxThreads), smem, st, sp, gp, out, vc);
    }
    const dim3 grid(gp.nx, (gp.ny + kLinesPerCta - 1) / kLinesPerCta);
    const size_t smem = (sizeof(Cx) + sizeof(float)) * (size_t)(gp.nz + 1) * kLinesPerCta;
    // per-function attribute shared by all threads: set it to the largest size
    // (nz = 256) so a concurrent launch from another thread is never rejected
    const int smem_max = (int)((sizeof(Cx) + sizeof(float)) * ((kFp64 ? 256 : 32 * kMaxRun) + 1) * kLinesPerCta);
    auto k = maps ? voxelise_scan_kernel<kFp64, ScanT, true> : voxelise_scan_kernel<kFp64, ScanT, false>;
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max);
    if (e != cudaSuccess) return e;
    return launch_pdl(k, grid, dim3(kVoxThreads), smem, st, sp, gp, out, vc);
}

cudaError_t launch_voxelise(const ShapeParams &sp, const GridParams &gp, const SliceOut &out, bool scan_fp64,
                            bool fp64_mode, cudaStream_t st) {
    if (gp.nz > 32 * kMaxRun || (fp64_mode && gp.nz > 256)) return cudaErrorInvalidValue;
    if (out.chunk_y && (out.bounds == nullptr || gp.nx > 8 * kGeomChunks)) return cudaErrorInvalidValue;
    VoxConst vc;
    vc.att = gp.k0 * gp.voxel * gp.beta;
    vc.ph = gp.k0 * gp.voxel * gp.delta;
    vc.kdz = gp.k0 * gp.voxel;
    vc.inv_scale = sp.nscale != 0.0 ? 1.0 / sp.nscale : 0.0;
    vc.att_f = (float)vc.att;
    vc.ph_f = (float)vc.ph;
    vc.kdz_f = (float)vc.kdz;
    vc.inv_scale_f = (float)vc.inv_scale;
    return fp64_mode   ? run_voxelise<true, double>(sp, gp, out, vc, st)
           : scan_fp64 ? run_voxelise<false, double>(sp, gp, out, vc, st)
                       : run_voxelise<false, float>(sp, gp, out, vc, st);
}

}  // namespace scm
