"""The field through its sample grid on the Ewald sphere against the direct sums.

The same pixels as an explicit list of q take the direct sums, so the two paths
of one precision mode are compared on identical slices.  Tolerances (relative
L2 of I): FP64 1e-11 (the plan leaves 1e-12 of a box filled to its corners and
both sums round at 1e-14); FP32 3e-6 (each within the FP32 mode's ~1e-6); split
phases 1e-5 (FP16) and 1e-4 (BF16): the two paths round different phases, each
leaving u^2 = 2^-22 / 2^-16 per element, 2 sqrt(2) u^2 in I at worst.
"""
import numpy as np
import pytest

from gpu_helpers import rel_l2, run_gpu
from workloads import (DETECTOR_UNIFORM_Q, ELLIPSOID, SPHERE, VOLUMEMAP, Geometry, Shape)

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-11, "fp32": 3e-6, "tc_f16_split": 1e-5, "tc_bf16_split": 1e-4}


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _direct(g, s, prec, soft=False):
    import paper_2202_03411_gb300 as sm
    h = sm.scatman_create(g, "fp32")
    q = sm.scatman_get_q(h)
    h.close()
    flat = Geometry(g.nx, g.ny, g.nz, g.voxel, g.wavelength, g.theta_max_deg, g.det_nx, g.det_ny)
    I, A = run_gpu(flat, s, prec, q_list=q, soft=soft)
    if g.detector == DETECTOR_UNIFORM_Q:
        k0 = 2 * np.pi / g.wavelength
        off = (q[:, 0] ** 2 + q[:, 1] ** 2) / k0 ** 2 > 1.0
        I[off] = 0.0
    return I


def _solid(g, fill=1.0):
    """A volume map that fills the whole box to its corners."""
    n = max(g.nx, g.ny, g.nz)
    return Shape(VOLUMEMAP, volume_map=np.ones((4, 4, 4), dtype=bool), map_dx=fill * g.voxel * n / 4.0 + 1e-6,
                 delta=0.012, beta=0.002)


# grids and detectors off every tile: odd and even sides, one row, one column,
# more than 64 columns of half-coordinates, points beyond one row tile
PLAIN = [
    Geometry(21, 19, 23, 1.0, 7.0, 50.0, 45, 37),
    Geometry(64, 30, 17, 1.0, 6.0, 60.0, 33, 64),
    Geometry(9, 72, 1, 0.7, 5.0, 75.0, 131, 1),
    Geometry(35, 1, 40, 1.3, 9.0, 20.0, 1, 140),
    Geometry(140, 24, 33, 1.0, 5.0, 55.0, 40, 32),
    Geometry(24, 27, 30, 1.0, 5.0, 40.0, 70, 65, DETECTOR_UNIFORM_Q),
    Geometry(24, 24, 24, 1.0, 5.0, 60.0, 64, 64, DETECTOR_UNIFORM_Q),     # off-sphere corners: the separable sums
    Geometry(20, 18, 22, 1.0, 6.0, 44.5, 31, 40, DETECTOR_UNIFORM_Q),     # just inside the sphere's rim
    Geometry(30, 26, 28, 1.0, 8.0, 88.0, 24, 24),                          # too wide for the grid: direct
]


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("k", range(len(PLAIN)))
def test_plain_modes(k, prec):
    g = PLAIN[k]
    n = min(g.nx, g.ny, g.nz)
    shapes = [
        Shape(ELLIPSOID, a=0.3 * g.nx * g.voxel, b=0.2 * g.ny * g.voxel + 0.4, c=0.4 * g.nz * g.voxel + 0.4, delta=0.02,
              beta=0.004, latitude=-88, longitude=4, rotation=3, cx=0.15 * g.nx * g.voxel, cy=-0.2 * g.ny * g.voxel),
        _solid(g),
    ]
    for s in shapes:
        I, _ = run_gpu(g, s, prec)
        ref = _direct(g, s, prec)
        assert ref.max() > 0
        assert rel_l2(I, ref) < TOL[prec], (g, prec, s.kind, rel_l2(I, ref), n)


@pytest.mark.parametrize("prec", ["tc_f16_split", "tc_bf16_split"])
@pytest.mark.parametrize("g", [
    Geometry(96, 96, 96, 1.0, 10.0, 45.0, 70, 61),
    Geometry(160, 56, 48, 1.0, 9.0, 45.0, 140, 120),         # slices of two work units
    Geometry(100, 61, 90, 1.0, 4.5, 60.0, 128, 97),          # more than 128 rows: two row tiles
    Geometry(40, 128, 37, 1.0, 8.0, 50.0, 301, 200),
])
def test_split_phases(g, prec):
    from workloads import SPHHARM, random_alm
    shapes = [
        Shape(SPHERE, r=0.2 * min(g.nx, g.ny, g.nz), delta=0.02, beta=0.004, cx=0.28 * g.nx, cy=-0.25 * g.ny,
              cz=0.2 * g.nz),
        Shape(SPHHARM, R0=0.33 * min(g.nx, g.ny, g.nz), lmax=6, alm=random_alm(np.random.default_rng(2), 6),
              delta=0.01, beta=0.001, latitude=30, longitude=-60, rotation=40),
        _solid(g),
    ]
    for s in shapes:
        I, _ = run_gpu(g, s, prec)
        ref = _direct(g, s, prec)
        assert rel_l2(I, ref) < TOL[prec], (g, prec, s.kind, rel_l2(I, ref))


@pytest.mark.parametrize("prec", ["fp32", "tc_bf16_split"])
def test_empty_and_repeated_shapes(prec):
    """An empty shape gives exactly zero, also after a shape that filled the box."""
    import torch
    import paper_2202_03411_gb300 as sm
    g = Geometry(70, 64, 66, 1.0, 8.0, 45.0, 120, 120)
    empty = Shape(SPHERE, r=0.1, cx=0.25, cy=0.25, cz=0.25, delta=0.01, beta=0.001)
    body = Shape(SPHERE, r=9.0, cx=20.0, cy=-15.0, delta=0.01, beta=0.001)
    h = sm.scatman_create(g, prec)
    I = torch.empty(g.n_pix, device="cuda")
    out = []
    for s in (body, _solid(g), body, empty):
        sm.scatman_voxelise(h, s)
        sm.scatman_forward(h, I)
        sm.scatman_sync(h)
        out.append(I.cpu().numpy().copy())
    h.close()
    assert np.array_equal(out[0], out[2]) and out[0].max() > 0
    assert np.all(out[3] == 0.0)


@pytest.mark.parametrize("g", [
    Geometry(48, 48, 48, 1.0, 10.0, 45.0, 64, 64),
    Geometry(33, 41, 26, 1.0, 7.0, 55.0, 71, 58),
    Geometry(24, 27, 30, 1.0, 5.0, 40.0, 70, 65, DETECTOR_UNIFORM_Q),
])
def test_fp32_fit_sums_are_exact_to_the_stored_pattern(g):
    """A fit's loss is the difference of two nearly equal patterns, so an FP32 fit's
    sums over its (FP32) slices run in FP64.  I is rounded to FP32 once: 2^-24 = 6e-8 of it,
    and the plan leaves up to 1e-8 of a field; FP32 sums leave 2e-7."""
    import torch
    import oracle
    import paper_2202_03411_gb300 as sm
    s = Shape(ELLIPSOID, a=0.36 * g.nx, b=0.28 * g.ny, c=0.3 * g.nz, delta=0.012, beta=0.0012, latitude=30,
              longitude=70, rotation=-20)
    h = sm.scatman_create(g, "fp32", soft=True, soft_width=0.5)
    I = torch.empty(g.n_pix, device="cuda")
    sm.scatman_voxelise(h, s)
    sm.scatman_forward(h, I)
    rho = np.asarray(sm.scatman_get_slices(h, (g.nz, g.nx, g.ny)), dtype=np.complex128)
    q = sm.scatman_get_q(h)
    h.close()
    ref = np.abs(oracle.msft(rho * ((1 - s.delta + 1j * s.beta) ** 2 - 1), q, g.voxel)) ** 2
    assert rel_l2(I.cpu().double().numpy(), ref) < 8e-8


@pytest.mark.parametrize("prec,tol", [("fp32", 1e-5), ("tc_bf16_split", 1e-3)])
@pytest.mark.parametrize("rows", [131070, 140001])
def test_strip_detectors(rows, prec, tol):
    """A line of pixels up to the last row that the grid takes, and past it (direct sums)."""
    from gpu_helpers import oracle_field
    g = Geometry(17, 18, 16, 1.0, 7.0, 50.0, 1, rows)
    s = Shape(ELLIPSOID, a=6.0, b=5.0, c=6.5, delta=0.01, beta=0.001, latitude=20, longitude=50)
    at = np.concatenate([np.arange(40), rows // 2 + np.arange(-20, 20), rows - 1 - np.arange(40)])
    I, _ = run_gpu(g, s, prec)
    ref, _ = oracle_field(g, s, sample=at)
    assert rel_l2(I[at], ref) < tol


@pytest.mark.parametrize("rows", [131070, 140001])
def test_strip_detector_gradients(rows):
    """The same in the adjoint of an FP32 fit, against an FP64 fit of the weighted pixels."""
    import torch
    import oracle
    import paper_2202_03411_gb300 as sm
    g = Geometry(17, 18, 16, 1.0, 7.0, 50.0, 1, rows)
    s = Shape(ELLIPSOID, a=6.0, b=5.0, c=6.5, delta=0.01, beta=0.001, latitude=20, longitude=50)
    at = np.concatenate([np.arange(40), rows // 2 + np.arange(-20, 20), rows - 1 - np.arange(40)])
    w = torch.zeros(rows, device="cuda")
    w[torch.as_tensor(at, device="cuda")] = 1.0
    grads = []
    for prec, q, up in (("fp32", None, w), ("fp64", oracle.detector_q(g)[at], torch.ones(len(at), device="cuda").double())):
        h = sm.scatman_create(g, prec, soft=True, soft_width=0.5, q_list=q)
        sm.scatman_voxelise(h, s)
        sm.scatman_forward(h, torch.empty_like(up))
        grads.append(sm.scatman_backward(h, up))
        h.close()
    assert np.linalg.norm(grads[0] - grads[1]) / np.linalg.norm(grads[1]) < 2e-5


def _flops(g, s, prec, soft=False, q_list=None):
    import paper_2202_03411_gb300 as sm
    h = sm.scatman_create(g, prec, soft=soft, soft_width=0.5, q_list=q_list)
    sm.scatman_voxelise(h, s)
    out = sm.scatman_contraction_flops(h)
    h.close()
    return out


@pytest.mark.parametrize("prec", ["fp64", "fp32", "tc_bf16_split"])
def test_issued_flops_follow_the_box(prec):
    """The grid's sums skip what a shape leaves empty: a sphere of a quarter of the
    side in a corner counts well below the filled box (x/z sums: its half-coordinates reach
    the rim; y sums: a third of the slices, columns and y), and an empty shape nothing."""
    g = Geometry(96, 96, 96, 1.0, 10.0, 45.0, 200, 190)
    box, dense = _flops(g, _solid(g), prec)
    part, dense_part = _flops(g, Shape(SPHERE, r=12.0, cx=30, cy=-30, cz=20, delta=0.01, beta=0.001), prec)
    none, _ = _flops(g, Shape(SPHERE, r=0.1, cx=0.25, cy=0.25, cz=0.25, delta=0.01, beta=0.001), prec)
    assert none == 0 and 0 < part < 0.35 * box and dense == dense_part > 4 * box
    if prec != "tc_bf16_split":
        # Hs x (y: 96 slices, 3 tiles of columns, 48 half-coordinates; x/z: 6 chunks, 48, Ht), 256 flop each
        assert box % (256 * 48) == 0
        Hs_terms = box / (256 * 48)
        assert any(Hs_terms == Hs * (96 * 3 + 6 * Ht) for Hs in range(4, 97) for Ht in range(4, 97))


def test_issued_flops_of_a_fit_are_the_pixel_sums():
    """A split-phase fit sums over the pixels: what it reports is what the same pixels as a list of q report."""
    import paper_2202_03411_gb300 as sm
    g = Geometry(96, 96, 96, 1.0, 10.0, 45.0, 256, 256)
    h = sm.scatman_create(g, "fp32")
    q = sm.scatman_get_q(h)
    h.close()
    s = Shape(SPHERE, r=30.0, delta=0.01, beta=0.001)
    assert _flops(g, s, "tc_bf16_split", soft=True) == _flops(g, s, "tc_bf16_split", soft=True, q_list=q)


@pytest.mark.parametrize("prec,soft,tol", [("fp64", False, 1e-10), ("fp32", False, 1e-5), ("fp32", True, 1e-5)])
@pytest.mark.parametrize("g", [
    Geometry(12, 12, 12, 1.0, 6.0, 45.0, 401, 403),                       # flat: a row of pixels per warp, eight warps
    Geometry(12, 12, 12, 1.0, 6.0, 45.0, 801, 803),                       # flat: four rows a thread
    Geometry(12, 12, 12, 1.0, 6.0, 40.0, 431, 429, DETECTOR_UNIFORM_Q),   # uniform-q: two columns a thread
    Geometry(12, 12, 12, 1.0, 6.0, 40.0, 803, 801, DETECTOR_UNIFORM_Q),   # uniform-q: four
])
def test_large_odd_detectors(g, prec, soft, tol):
    """Each form of the interpolation to the pixels, past its last whole tile: the rim,
    the middle and a sample against the oracle (the modes' tolerances)."""
    from gpu_helpers import oracle_field
    s = Shape(ELLIPSOID, a=4.4, b=3.6, c=4.0, delta=0.01, beta=0.001, latitude=20, longitude=50, rotation=10, cx=0.3)
    I, _ = run_gpu(g, s, prec, soft=soft)
    v, u = np.divmod(np.arange(g.n_pix), g.det_nx)
    rim = (u < 2) | (u >= g.det_nx - 3) | (v < 2) | (v >= g.det_ny - 3) | ((u - g.det_nx // 2) ** 2 + (v - g.det_ny // 2) ** 2 < 30)
    at = np.union1d(np.flatnonzero(rim), np.random.default_rng(4).choice(g.n_pix, 2000, replace=False))
    ref, _ = oracle_field(g, s, sample=at, soft=soft)
    assert rel_l2(I[at], ref) < tol
    edge = np.flatnonzero(rim[at] & ((u[at] - g.det_nx // 2) ** 2 + (v[at] - g.det_ny // 2) ** 2 >= 30))
    assert rel_l2(I[at][edge], ref[edge]) < 100 * tol                     # (two to four decades below the peak)
