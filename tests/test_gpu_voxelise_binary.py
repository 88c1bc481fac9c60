"""Binary shapes through the bit voxeliser, at sizes off its tiles.

The occupancy must equal the FP64 oracle's voxel for voxel (the FP32 test only
settles voxels outside its error margin), and the slices the oracle's T within
rounding: 1e-14 (FP64), 1e-6 (FP32), 2^-10 and 2^-8 (FP16 and BF16 operands).
"""
import numpy as np
import pytest

import oracle
from workloads import ELLIPSOID, RADIALMAP, SPHERE, SPHHARM, Geometry, Shape, random_alm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


# one voxel, one line, odd and even sides, more than 32 and more than 256 slices,
# tails of 8 and 16 lines, CTAs of 8 lines (small grids) and of 16
GRIDS = [(1, 1, 1), (7, 1, 33), (24, 23, 65), (13, 41, 31), (40, 150, 96), (64, 77, 257)]


def _shapes(g, rng):
    n = max(4.0, float(min(g.nx, g.ny, g.nz))) * g.voxel
    rot = dict(latitude=33, longitude=-70, rotation=15)
    return [
        Shape(SPHERE, r=0.4 * n, delta=0.02, beta=0.003, cx=0.3 * g.voxel, cy=-0.5 * g.voxel, cz=0.5 * g.voxel),
        Shape(ELLIPSOID, a=0.45 * n, b=0.25 * n, c=0.35 * n, delta=0.02, beta=0.003, **rot),
        Shape(SPHHARM, R0=0.35 * n, lmax=5, alm=random_alm(rng, 5, 0.1), delta=0.02, beta=0.003, **rot),
        Shape(RADIALMAP, radial_map=0.3 * n * (1 + 0.2 * rng.random((9, 14))), delta=0.02, beta=0.003, **rot),
        Shape(SPHERE, r=9.0 * n, delta=0.01, beta=0.001),                   # every voxel
        Shape(SPHERE, r=1e-3 * g.voxel, delta=0.01, beta=0.001, cx=0.3 * g.voxel),   # none
    ]


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-14), ("fp32", 1e-6), ("tc_f16_split", 2 ** -10), ("tc_bf16_split", 2 ** -8)])
@pytest.mark.parametrize("k", range(len(GRIDS)))
def test_occupancy_and_slices(k, prec, tol):
    import paper_2202_03411_gb300 as sm
    nx, ny, nz = GRIDS[k]
    if prec == "fp64" and nz > 256:
        nz = 256
    if prec.startswith("tc") and ny > 128:
        ny = 121
    g = Geometry(nx, ny, nz, 0.8, 6.0, 40.0, 12, 12)
    h = sm.scatman_create(g, prec)
    for s in _shapes(g, np.random.default_rng(k)):
        sm.scatman_voxelise(h, s)
        chi, _ = oracle.voxelise(s, g, False, 0.5)
        got = sm.scatman_get_occupancy(h, (nz, nx, ny))
        assert np.array_equal(got, chi.reshape(nz, nx, ny)), (g, prec, s.kind, np.sum(got != chi.reshape(nz, nx, ny)))
        d = sm.scatman_get_slices(h, (nz, nx, ny))
        d = d if np.iscomplexobj(d) else d[..., 0] + 1j * d[..., 1]
        rho = oracle.slices(chi, g, s.delta, s.beta).reshape(nz, nx, ny)
        # n^2 - 1 without its cancellation
        c = -2 * s.delta + s.delta ** 2 - s.beta ** 2 + 1j * (2 * s.beta - 2 * s.delta * s.beta)
        assert np.abs(d - rho / c).max() <= tol, (g, prec, s.kind)
    h.close()


@pytest.mark.parametrize("far", [0.0, 3e5])
def test_fp64_mode_far_from_the_origin(far):
    """A shape whose centre is far from the grid's is out of the FP32 test's reach: the
    FP64 mode decides every voxel in FP64, as the oracle does."""
    import paper_2202_03411_gb300 as sm
    g = Geometry(24, 20, 22, 1.0, 6.0, 40.0, 12, 12)
    h = sm.scatman_create(g, "fp64")
    s = Shape(SPHERE, r=7.3 + far, cx=far, delta=0.01, beta=0.001)
    sm.scatman_voxelise(h, s)
    chi, _ = oracle.voxelise(s, g, False, 0.5)
    assert np.array_equal(sm.scatman_get_occupancy(h, (22, 24, 20)), chi.reshape(22, 24, 20))
    h.close()
