// internal.cuh -- declarations shared by the library's translation units.
// Not installed; the public surface is include/scatman.h.
#pragma once

#include <cuda_runtime.h>
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include <list>
#include <string>
#include <vector>

#include "../../include/scatman.h"

#include <nvtx3/nvToolsExt.h>

namespace scm {

constexpr double kPi = 3.14159265358979323846;

// An NVTX range around a stage of the host API (visible in Nsight timelines;
// a no-op unless a profiling tool is attached).
struct StageRange {
    explicit StageRange(const char *name) { nvtxRangePushA(name); }
    ~StageRange() { nvtxRangePop(); }
    StageRange(const StageRange &) = delete;
    StageRange &operator=(const StageRange &) = delete;
};

// Device allocation used by every buffer of the library; a test hook
// (scatman_debug_fail_allocation) can make one of them fail on the host.
cudaError_t device_malloc(void **p, size_t bytes);

// Status block of a handle on the device (kStatusBytes): the error word (int,
// byte 0) that kernels set; a test flag (int, byte 4) that makes the
// tensor-core kernels' MMA warps first wait on a barrier nothing arrives at,
// so that wait runs out and takes the abort path; and at byte 8 an optional
// shorter limit in ns for the kernels' work waits (unsigned long long; 0 =
// the default).
constexpr size_t kStatusBytes = 16;
constexpr unsigned long long kWaitLimitMaxNs = 2000000000ull;   // every bounded wait: 2 s at most

// Bits of the device error word written by kernels.
enum : int {
    kErrTimeoutProducer = 1,
    kErrTimeoutMma = 2,
    kErrTimeoutEpilogue = 4,
    kErrTimeoutDrain = 8,
    kErrBadLaunch = 16,
};

// Shape as the voxeliser kernels read it: body->lab rotation, centre, sizes
// and harmonic coefficients, everything in length units.
struct ShapeParams {
    int kind;
    int lmax;
    int soft;
    float inv_w_f;
    double inv_w;
    double r, a, b, c;
    double R0;
    double rmin, rmax;              // harmonics radius clip
    double R[9];                    // row-major body->lab rotation
    double cx, cy, cz;              // centre offset
    float Rf[9];                    // the rotation and the offsets in FP32 (fast path)
    float cxf, cyf, czf;
    float r2f, inv_af, inv_bf, inv_cf;   // r^2 and 1/a, 1/b, 1/c in FP32
    float R0f, rminf, rmaxf;             // harmonics radius scale and clip in FP32
    double alm[(SCATMAN_MAX_LMAX + 1) * (SCATMAN_MAX_LMAX + 1)];
    float almf[(SCATMAN_MAX_LMAX + 1) * (SCATMAN_MAX_LMAX + 1)];
    // normalised associated-Legendre recurrence coefficients, index l(l+1)/2 + m
    // (see real_sh_all): a_lm, b_lm, and the diagonal factors d_m, e_m
    double sh_a[(SCATMAN_MAX_LMAX + 1) * (SCATMAN_MAX_LMAX + 2) / 2];
    double sh_b[(SCATMAN_MAX_LMAX + 1) * (SCATMAN_MAX_LMAX + 2) / 2];
    double sh_d[SCATMAN_MAX_LMAX + 1];
    double sh_e[SCATMAN_MAX_LMAX + 1];
    float sh_af[(SCATMAN_MAX_LMAX + 1) * (SCATMAN_MAX_LMAX + 2) / 2];
    float sh_bf[(SCATMAN_MAX_LMAX + 1) * (SCATMAN_MAX_LMAX + 2) / 2];
    float sh_df[SCATMAN_MAX_LMAX + 1];
    float sh_ef[SCATMAN_MAX_LMAX + 1];
    // radii map (device copies, [ntheta][nphi])
    const double *rmap;
    const float *rmapf;
    int ntheta, nphi;
    double rm_tscale, rm_pscale;    // ntheta / pi, nphi / (2 pi)
    float rm_tscalef, rm_pscalef;
    float rm_slope;                 // max |dr/d angle| between neighbouring samples (FP32 decision margin)
    // volume map (device copies, [mx][my][mz])
    const unsigned char *vmap;
    int mx, my, mz;
    double mdx;
    float mdxf;
    const double *mdelta, *mbeta;   // per-cell index, or null
    int varn;                       // 1: voxel-resolved index (s carries (n_v^2 - 1) / nscale)
    double nscale;                  // max |n_v^2 - 1| over the map's cells
    // harmonics / radii map (and soft spheres / ellipsoids): a voxel centre with
    // |p| below band_lo is inside (soft: chi = 1), above band_hi outside
    // (chi = 0) (band_hi = 0: no band)
    float band_lo, band_hi;
    // FP64 mode, binary shapes: the FP32 test's margins hold for these sizes, so
    // it may settle voxels before the FP64 one
    int fp32_first;
    // binary harmonics: the voxeliser tabulates the radius at the centres of
    // rtab_n^2 cells on each face of a cube of directions; anywhere in a cell it
    // is within rtab_slack of that (rtab_n = 0: no table)
    int rtab_n;
    float rtab_slack;
    // binary harmonics: the FP32 test decides where the radius and the distance
    // differ by more than this (four times a bound on their FP32 error)
    float sh_margin;
};

// Soft occupancy cut of the FP32 modes: chi = 1 / (1 + e^{-t}) with
// t = (r_s - |p|) / w is taken as zero when chi < 2^-24, i.e. t < -kSoftCutT.
constexpr float kSoftCutT = 16.635532f;   // ln(2^24 - 1)
// Above this t the FP32 logistic is exactly 1.0f (e^{-t} below half an ulp of 1).
constexpr float kSoftOneT = 17.5f;

// Fills the FP32 copies and the harmonic recurrence tables of a ShapeParams
// whose double fields are set (api.cu).
void finish_shape_params(ShapeParams *sp);

// Number of geometric gradient parameters: sphere [r]; ellipsoid [a, b, c];
// harmonics [a_lm for l >= 1, R0].
#ifdef __CUDACC__
__host__ __device__
#endif
inline int n_geom_params(int kind, int lmax) {
    if (kind == SCATMAN_SPHERE) return 1;
    if (kind == SCATMAN_ELLIPSOID) return 3;
    if (kind == SCATMAN_RADIALMAP || kind == SCATMAN_VOLUMEMAP) return 0;
    return (lmax + 1) * (lmax + 1);
}

struct GridParams {
    int nx, ny, nz;
    double voxel;
    double k0;
    double delta, beta;
    float voxf;                     // voxel in FP32 (set by make_grid)
};

inline GridParams make_grid(int nx, int ny, int nz, double voxel, double k0, double delta, double beta) {
    GridParams g{nx, ny, nz, voxel, k0, delta, beta, (float)voxel};
    return g;
}

// Where the voxeliser writes s = chi*T.
enum SliceLayout { kLayoutC64 = 0, kLayoutC32 = 1, kLayoutTcF16 = 2, kLayoutTcBF16 = 3 };

// Tensor maps of the tensor-core slice operand, one per span width of 8k
// rows (k = 1 .. kTcMaxChunks): a box of 64 y x 8k rows x the three planes.
constexpr int kTcMaxChunks = 16;
struct TcMaps {
    CUtensorMap m[kTcMaxChunks];
};

// Per-slice geometry the voxeliser records for the contractions, in one
// device buffer of slice_geom_ints(nz) ints:
//   [0, 4 nz)            occupied box of every slice [x_lo | x_hi | y_lo | y_hi]
//   [4 nz, 68 nz)        occupied y range of every 8-column chunk of every slice,
//                        [y_lo | y_hi] x [nz][kGeomChunks] (tensor-core grids, nx <= 256)
//   then                 the tensor-core kernel's work-unit list (uint2, kMaxUnitsPerSlice nz + 1)
//   then                 T of 0 .. nz full voxels (16 bytes each), for binary shapes
//   then                 harmonics shapes: their coefficients as the voxeliser stages
//                        them (kShStageInts), and the radius table (floats)
constexpr int kRtabMax = 64;        // cells along a cube face's edge
constexpr int kShStageInts = 1536;
constexpr int kGeomChunks = 32;
constexpr int kMaxUnitsPerSlice = 4;
inline size_t geom_table_at(int nz) {
    return (4 * (size_t)nz + 2 * (size_t)kGeomChunks * nz + 2 * ((size_t)kMaxUnitsPerSlice * nz + 1) + 3) / 4 * 4;
}
inline size_t geom_stage_at(int nz) { return geom_table_at(nz) + 4 * ((size_t)nz + 1); }
inline size_t geom_rtab_at(int nz) { return geom_stage_at(nz) + kShStageInts; }
inline void *geom_stage(int *g, int nz) { return g + geom_stage_at(nz); }
inline size_t slice_geom_ints(int nz) { return geom_rtab_at(nz) + 6 * (size_t)kRtabMax * kRtabMax; }
inline void *geom_table(int *g, int nz) { return g + geom_table_at(nz); }
inline float *geom_rtab(int *g, int nz) { return reinterpret_cast<float *>(g + geom_rtab_at(nz)); }
inline int *geom_chunk_y(int *g, int nz) { return g + 4 * (size_t)nz; }
inline uint2 *geom_units(int *g, int nz) {
    return reinterpret_cast<uint2 *>(g + 4 * (size_t)nz + 2 * (size_t)kGeomChunks * nz);
}

struct SliceOut {
    int layout;
    int Nxp, Nyp, Kp;               // tensor-core operand: padded x and y; Kp = Nyp, the K extent of a row
    void *s;                        // C64: double2[nvox]; C32: float2[nvox]; TC: 16-bit [nz*3*Nxp][Kp]
    float *chi;                     // occupancy [z][x][y]
    int *bounds;                    // per slice [x_lo | x_hi | y_lo | y_hi] of chi != 0 (nz each), or null
    int *chunk_y;                   // per slice and 8-column chunk [y_lo | y_hi] (see above), or null
    void *table;                    // T of 0 .. nz full voxels (with bounds)
    void *stage;                    // staged coefficients of harmonics shapes (with bounds)
    float *rtab;                    // their radius table
};

// The field's sample grid on the Ewald sphere (field_grid.cu): sizes, then
// device buffers in one allocation.  Passed to its kernels by value.
struct FieldGrid {
    int uniform = 0;                // uniform-q detector (rows fix s) instead of the flat one (columns fix t)
    int elem = 4;                   // bytes of a real number in the sums and tables,
    int io = 4;                     // and in the slices, the field and the pattern
    int nx = 0, ny = 0, nz = 0, det_nx = 0, det_ny = 0;
    int Hs = 0, Ht = 0;             // half the points in s and t
    int H1 = 0, H2 = 0, n1 = 0;     // per-column (per-row) direction: its half points and half pixels; per-pixel direction
    int Kx = 0, Ky = 0, U = 0, V = 0;   // half sides of the grid and the detector, rounded up
    int jc = 0;                     // slice chunks of the x/z sum
    double sm = 0, tm = 0;          // largest |s|, |t|
    double k0 = 0, voxel = 0, top = 0;  // top: tan or sin of theta_max
    void *ty = nullptr, *tx = nullptr, *tz = nullptr;   // phases of the sums
    void *node2 = nullptr, *w1 = nullptr, *pix = nullptr;   // interpolation: points, weights, pixels
    double *qrow = nullptr, *point_s = nullptr, *point_t = nullptr;
    void *H = nullptr, *Q = nullptr, *B = nullptr;      // y-sums, samples, per-column interpolants
};

// Buffers of the adjoint through the grid (field_grid_adjoint.cu), one allocation.
struct FieldGridAdjoint {
    int chunks = 0;                 // of the per-pixel direction
    bool own = false;               // the grid's tables are its own (the forward pass has none of this type)
    void *B = nullptr, *G = nullptr, *T = nullptr;      // pixels gathered along it; onto the grid; x/z sums
};

}  // namespace scm

struct scatman_handle {
    scatman_config cfg;
    int device = 0;
    int sm_count = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    long long n_pix = 0;
    double k0 = 0;
    int precision = 0;
    bool tensor_core = false;
    bool split = false;
    bool bf16 = false;
    bool s_bf16 = false;            // 16-bit type of the tensor-core slice operand
    bool scan_fp64 = false;
    // tensor-core operand geometry
    int Nxp = 0, Nyp = 0, Kp = 0;
    size_t b_rows = 0;
    // device buffers
    double *d_q = nullptr;          // [n_pix][3]
    int *d_bounds = nullptr;        // per-slice occupied box [x_lo | x_hi | y_lo | y_hi], 4*nz ints,
                                    // then the tensor-core kernel's occupied-slice list (nz + 1 uint2)
    float *d_chi = nullptr;         // [nvox]
    void *d_s = nullptr;            // slices in the contraction's layout
    size_t s_bytes = 0;
    void *d_A = nullptr;            // field cache (double2 or float2)
    void *d_I = nullptr;            // intensity scratch for acquire
    void *d_I2 = nullptr;           // second intensity buffer of the batched acquire (on first use)
    cudaStream_t copy_stream = nullptr;   // batched acquire: device-to-host copies
    cudaEvent_t ev_fwd[2] = {nullptr, nullptr}, ev_copy[2] = {nullptr, nullptr};
    int *d_err = nullptr;
    double *d_part = nullptr;       // backward partial sums
    size_t part_count = 0;
    void *d_S = nullptr;            // backward adjoint field (complex, nvox)
    void *d_partial = nullptr;      // CUDA-core contraction: per-split partial fields
    float2 *d_tail = nullptr;       // tensor-core contraction: partial fields of the last wave's cut tiles
    void *d_H = nullptr;            // uniform-q detector: y-contracted slices [v][z][x], or in the
                                    // tensor-core modes 16-bit planes [row group][-Im | Re | Im][Rg Jp][Kx]
    bool uniform_q = false;
    bool uniform_tc = false;        // uniform-q detector with the x/z sum on the tensor cores
    int uq_Jp = 0, uq_Kx = 0, uq_Rg = 1;   // its operand geometry: nz padded to 16, nx padded to 64,
                                           // detector rows per GEMM column group
    float2 *d_uq_qz = nullptr;      // its per-pixel q_z (float pair; marker off the Ewald sphere)
    double *d_uq_qrow = nullptr;    // q of each detector row's first pixel (q_y of the row), tensor-core modes
    CUtensorMap tmap_H;
    bool from_q_list = false;       // q given by the caller: no pixel geometry
    float2 *d_adj_part = nullptr;   // tensor-core adjoint: per-pixel-range partial fields
    size_t adj_part_count = 0;
    unsigned *d_gmax = nullptr;     // tensor-core adjoint: max |w A| (float bits)
    int adj_orders = -1;            // tensor-core adjoint: Jacobi-Anger orders N (0: one GEMM per slice; -1: not chosen yet)
    float2 *d_adj_coef = nullptr;   // order mode: a[j][n] = e^{+i q_c z_j} eps_n i^n J_n(D z_j), [nz][N]
    float2 *d_adj_ord = nullptr;    // order mode: the orders' fields S~ [N][nx][ny]
    float4 *d_adj_tab = nullptr;    // tensor-core adjoint: per-pixel constants (built at the first backward)
    uint8_t *d_adj_rtile = nullptr; // tensor-core adjoint: y-phase operand tiles (built at the first backward)
    // map shapes: device copies of the last voxelised map (grown as needed)
    double *d_rmap = nullptr;
    float *d_rmapf = nullptr;
    size_t rmap_cap = 0;
    unsigned char *d_vmap = nullptr;
    size_t vmap_cap = 0;
    double *d_mdelta = nullptr, *d_mbeta = nullptr;
    size_t mindex_cap = 0;
    // pinned staging of the last two map uploads, each free again once its event has passed
    struct MapStage {
        unsigned char *p = nullptr;
        size_t cap = 0;
        cudaEvent_t ev = nullptr;
    } map_stage[2];
    int map_turn = 0;
    bool map_captured = false;      // the upload under way is being captured
    std::list<std::vector<double>> captured_maps;
    double str_re = 0, str_im = 0;  // global strength factor of s: n^2 - 1, or the map's index scale
    double map_index_max = 0;       // max |delta|, |beta| over a volume map's cells
    bool on_grid = false;           // the field goes through its sample grid
    scm::FieldGrid fg;
    unsigned char *d_fg = nullptr;  // its buffers
    bool adj_on_grid = false;       // the adjoint goes through the grid
    scm::FieldGrid fg_adj;
    scm::FieldGridAdjoint fga;
    unsigned char *d_fga = nullptr; // its buffers (from the first backward on)
    int splits = 1;
    long long device_bytes = 0;
    scm::TcMaps tmap_B;
    bool have_tmap = false;
    // state
    bool have_shape = false;
    bool have_forward = false;
    scatman_shape shape;
    std::vector<double> alm;
    scm::ShapeParams sp;
    std::string last_error;
};

namespace scm {

// ---- host helpers shared by the .cu files --------------------------------
int set_error(scatman_handle *h, int code, const std::string &msg);
int check_cuda(scatman_handle *h, cudaError_t e, const char *what);

// Voxeliser + exclusive scan (voxelise.cu).
cudaError_t launch_voxelise(const ShapeParams &sp, const GridParams &gp, const SliceOut &out,
                            bool scan_fp64, bool fp64_mode, cudaStream_t st);
// Detector q (voxelise.cu).
cudaError_t launch_detector_q(int det_nx, int det_ny, double theta_max_deg, double k0, double *q,
                              cudaStream_t st);
// Uniform-q virtual detector (msft_uniform.cu).
cudaError_t launch_detector_q_uniform(int det_nx, int det_ny, double theta_max_deg, double k0, double *q,
                                      cudaStream_t st);
// q_z table marker (a quiet-NaN bit pattern) of a pixel off the Ewald sphere.
constexpr uint32_t kUqOffSphereBits = 0x7fc00000u;
cudaError_t launch_msft_uniform(bool fp64, const void *s, int nx, int ny, int nz, int det_nx, int det_ny,
                                double theta_max_deg, double k0, double voxel, double str_re, double str_im,
                                const float2 *qz, void *H, void *A, void *I, cudaStream_t st);
// Uniform-q detector on the tensor cores (msft_tc.cu in store mode for U1,
// msft_uniform_tc.cu for the x/z contraction).
// Operand geometry: Kx = nx padded to its K block (16, 32 or 64), Jp = nz padded
// to 16, Rg rows per group.
void uq_tc_geometry(int nx, int nz, int *Kx, int *Jp, int *Rg);
size_t uq_tc_h_bytes(int nx, int nz, int det_ny);
int uq_tc_slots(int nx, int nz, bool split);
bool encode_tmap_uq(CUtensorMap *map, void *H, int nx, int nz, int det_ny, bool bf16, std::string *why);
double uq_tc_issued_flops(int nx, int nz, int det_nx, int det_ny, bool split);
// q_z per pixel as a float pair with a marker off the Ewald sphere (once per handle).
cudaError_t launch_uq_qz_table(const double *q, long long n, double k0, float2 *tab, cudaStream_t st);
cudaError_t launch_uq_tc(const CUtensorMap &map, const float2 *qz, int nx, int nz, int det_nx, int det_ny,
                         double theta_max_deg, double k0, double voxel, double str_re, double str_im, bool split,
                         bool bf16, float2 *A, float *I, int *err, int sm_count, cudaStream_t st);
// CUDA-core contraction (msft_simt.cu).
int simt_splits(long long n_pix, int nx, int nz, int sm_count);
// bounds: the voxeliser's per-slice occupied boxes (4 nz ints), or NULL for a dense sum.
cudaError_t launch_msft_simt(bool fp64, const void *s, const double *q, long long n_pix, int nx, int ny,
                             int nz, double voxel, double str_re, double str_im, void *A, void *I,
                             void *partial, int splits, cudaStream_t st, const int *bounds);
// Real flops the CUDA-core contraction executes with box skipping (host copy of the bounds).
double simt_issued_flops(const int *bounds, int nz, int ny, long long n_pix, bool fp64);
// Tensor-core contraction (msft_tc.cu).  Whether a padded grid fits its
// tensor-memory layout (phase operand and two accumulators) and unit masks.
bool tc_grid_ok(int Nxp, int Nyp, bool split);
// geom: the slice-geometry buffer (slice_geom_ints); tail_part: scratch of
// tc_tail_part_bytes for the partial fields of the last partial wave's tiles
// (null: every tile whole).
cudaError_t launch_msft_tc(const TcMaps &maps, const double *q, long long n_pix, int nx, int ny, int nz,
                           int Nxp, int Nyp, double voxel, double str_re, double str_im, bool split,
                           bool bf16, int *geom, float2 *A, float *I, int *err,
                           int sm_count, cudaStream_t st, float2 *tail_part);
size_t tc_tail_part_bytes(long long n_pix, int sm_count);
// The same kernel in store mode, the uniform-q detector's y-contraction on the
// tensor cores: rows are detector rows v (q_y(v) = qrow[3 v + 1]) and G is
// written to the x/z operand H as 16-bit planes.
struct UqStore {
    uint16_t *Ht;
    int Jp, Rg, Kx;
    bool bf16;                  // H's 16-bit type
    float2 *H32 = nullptr;      // FP32 sums instead of the planes (launch_rows_y_tc)
};
cudaError_t launch_uq_y_tc_mma(const TcMaps &maps, const double *qrow, int det_ny, int nx, int ny, int nz, int Nxp,
                               int Nyp, double voxel, bool split, bool bf16, int *geom,
                               const UqStore &store, int *err, int sm_count, cudaStream_t st);
// The same with the rows' sums kept in FP32: H[row][j][x], rows of Nxp, written
// in the occupied 8-column chunks.
cudaError_t launch_rows_y_tc(const TcMaps &maps, const double *qrow, int rows, int nx, int ny, int nz, int Nxp,
                             int Nyp, double voxel, bool split, bool bf16, int *geom, float2 *H, int *err,
                             int sm_count, cudaStream_t st);
// The field through its sample grid (field_grid.cu).  plan: whether the
// detector and box allow it, and its sizes; layout: buffer offsets from base.
bool plan_field_grid(const scatman_config &c, int elem, FieldGrid *f);
bool use_field_grid(const scatman_config &c, FieldGrid *f);
size_t field_grid_layout(FieldGrid *f, bool forward, int Nxp, unsigned char *base);
cudaError_t launch_field_grid_tables(const FieldGrid &f, cudaStream_t st);
// Forward from the slices (FP32 or FP64), or from the tensor-core y-sums in f.H.
cudaError_t launch_field_grid(const FieldGrid &f, const void *s, const int *bounds, double str_re, double str_im,
                              void *A, void *I, int sm_count, cudaStream_t st);
// Real flops of its folded sums over y and over x and z for the recorded slice
// geometry (a host copy of the first 4 nz ints of the buffer).
double field_grid_issued_flops(const FieldGrid &f, const int *bounds_host);
cudaError_t launch_field_grid_tc(const FieldGrid &f, int Nxp, const int *bounds, const int *chunk_y, double str_re,
                                 double str_im, float2 *A, float *I, int sm_count, cudaStream_t st);
// Whether a handle of this configuration runs its adjoint through the grid.
bool use_field_grid_adjoint(const scatman_config &c, FieldGrid *f);
// The adjoint field (field_grid_adjoint.cu).  layout: buffer offsets from base of the
// planned grid f, with the tables and sums of the forward pass's grid fwd (null: it has
// none) where that holds the same type; returns the bytes.
size_t field_grid_adjoint_layout(FieldGrid *f, const FieldGrid *fwd, FieldGridAdjoint *a, unsigned char *base);
cudaError_t launch_field_grid_adjoint(const FieldGrid &f, const FieldGridAdjoint &ad, const void *A, const void *w,
                                      void *S, cudaStream_t st);
// Real flops one contraction launch issues for the recorded slice geometry
// (a host copy of the first 4 nz + 2 kGeomChunks nz ints of the buffer).
double tc_issued_flops(const int *geom_host, int nz, int Nxp, int Nyp, long long n_pix, bool split);
bool encode_tmap_B(TcMaps *maps, void *base, int Kp, int Nxp, int nz, bool bf16, std::string *why);
// A 3D tiled tensor map over 16-bit elements with a 32-, 64- or 128-byte
// swizzle (dims innermost first; strides of dims 1 and 2 in bytes; the box's
// inner extent in bytes equals the swizzle width).
bool encode_tmap_3d_16bit(CUtensorMap *map, void *base, const uint64_t dims[3], const uint64_t strides[2],
                          const uint32_t box[3], bool bf16, std::string *why, int swizzle_bytes);
// Ideal detector (detector.cu): expected photons and Poisson counts per pixel.
cudaError_t launch_photon_counts(const void *I, bool fp64, long long n, int det_nx, int det_ny, bool uniform,
                                 double theta_max_deg, double wavelength, double voxel, double photon_density,
                                 uint64_t seed, double *lambda, long long *counts, cudaStream_t st);
// Backward (adjoint.cu).
cudaError_t launch_adjoint_field(bool fp64, const void *A, const void *dLdI, const double *q, long long n_pix,
                                 int nx, int ny, int nz, double voxel, void *S, cudaStream_t st);
int grad_param_count(const ShapeParams &sp);
cudaError_t launch_grad_voxels(bool fp64, const ShapeParams &sp, const GridParams &gp, const void *S,
                               double *partials, int n_blocks, cudaStream_t st);
int grad_voxel_blocks(bool fp64, const ShapeParams &sp, const GridParams &gp, int sm_count);
cudaError_t launch_grad_pixels(bool fp64, const void *A, const void *dLdI, long long n_pix,
                               double *partials, int n_blocks, cudaStream_t st);
int grad_pixel_blocks(long long n_pix);
// out: nv voxel sums over nvb blocks, the pixel sum over npb, the error word (nv + 2 doubles).
cudaError_t launch_grad_totals(const double *part, int nvb, int nv, int npb, const int *err, double *out,
                               cudaStream_t st);
// Tensor-core adjoint field (adjoint_tc.cu).
bool adjoint_tc_supported(int nx, int ny);
// nz: slices, or in order mode (orders != 0) the number N of Jacobi-Anger orders;
// S receives the slices' (or orders') fields [nz][nx][ny].
int adjoint_tc_splits(long long n_pix, int nz, int sm_count, bool orders);
cudaError_t launch_adjoint_tc(const float2 *A, const float *w, const float4 *tab, const uint8_t *rtile, long long n_pix,
                              int nx, int ny, int nz, int orders, double voxel, int splits, float2 *partial,
                              unsigned *gmax_bits, float2 *S, int *err, cudaStream_t st);
// Order mode: the slices' fields from the orders' (coef: [nz][N] complex).
cudaError_t launch_adj_orders_combine(const float2 *Sord, const float2 *coef, int N, int nz, int nx, int ny, float2 *S,
                                      cudaStream_t st);
// The adjoint's y-phase operand tiles (once per handle).
size_t adj_rtile_bytes(long long n_pix, int ny);
cudaError_t launch_adj_rtile(const float4 *tab, long long n_pix, int ny, double voxel, uint8_t *rt, cudaStream_t st);
// Per-pixel constants of the tensor-core adjoint (3 float4 per pixel), once per handle.
// orders != 0: order mode with theta = acos((q_z - qc) inv_d) in place of q_z.
cudaError_t launch_adj_pixel_table(const double *q, long long n, double voxel, int orders, double qc, double inv_d,
                                   float4 *tab, cudaStream_t st);
// Fit residual 2 (I - target) and partial sums of (I - target)^2 (adjoint.cu).
int l2_residual_blocks(long long n);
cudaError_t launch_l2_residual(bool fp64, const void *I, const float *target, long long n, void *w, double *partials,
                               int n_blocks, cudaStream_t st);

}  // namespace scm

// ---- device helpers ---------------------------------------------------------
#ifdef __CUDACC__
namespace scm {

// Programmatic dependent launch: the kernels of a pass are short, and each one's
// launch and prologue can run under the end of the one before.  A kernel launched
// so calls pdl_wait before it touches memory that other kernels use (reads or
// writes: everything before it in the stream is then behind it).  Forward passes in
// us, ordinary launches / this: 108 / 78 at 128^3 on 512^2 (BF16), 53 / 30 at 70 x 52 x
// 41 on 301 x 257, 50 / 31 at 30^3 on 512^2 (uniform-q, FP32).  No kernel lets the next
// one's blocks in early (launch_dependents): they would settle on the first SMs to
// have room and leave the grid lopsided (88 us for the first of these, and in FP64
// 275 instead of 190 at 96^3 on 256^2).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... P, typename... Q>
inline cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Q &&...args) {
    cudaLaunchAttribute a{};
    a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = st;
    c.attrs = &a;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
}

// 16-byte copies to shared memory, all of a thread's in flight until it waits.
__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}

// e^{-i q c} for a q held in double and a coordinate c that is a small
// multiple of the voxel: the argument q*c is formed as a float pair
// (FMA-exact product of the high part plus the low part's product) and
// reduced modulo 2 pi in two pieces (Cody-Waite), so the reduced angle is
// good to ~1e-7 rad even for |q c| of a few hundred radians.
__device__ __forceinline__ float2 expmi_fs(float qh, float ql, float cf) {
    const float kTwoPiHi = 6.28318548202514648f;
    const float kTwoPiLo = -1.7484555314695172e-07f;
    const float kInvTwoPi = 0.15915494309189535f;
    float p = qh * cf;
    float e = fmaf(qh, cf, -p);
    float lo = fmaf(ql, cf, e);
    float n = rintf(p * kInvTwoPi);
    float r = fmaf(-n, kTwoPiHi, p);
    r = r + fmaf(-n, kTwoPiLo, lo);
    float s, co;
    sincosf(r, &s, &co);
    return make_float2(co, -s);
}

__device__ __forceinline__ float2 expmi_f(double q, double c) {
    float qh = (float)q;
    float ql = (float)(q - (double)qh);
    return expmi_fs(qh, ql, (float)c);
}

__device__ __forceinline__ double2 expmi_d(double q, double c) {
    double s, co;
    sincos(q * c, &s, &co);
    return make_double2(co, -s);
}

}  // namespace scm
#endif
