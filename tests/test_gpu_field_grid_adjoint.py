"""The adjoint through the sample grid of scattering directions against the direct sums.

The same pixels as an explicit list of q take the direct adjoint, so the two
paths of one precision mode are compared on the same shape.  The upstream
gradient is positive, so sum_p w_p I_p has no cancellation against a target;
tolerances (relative L2 of the gradient vector): FP64 1e-9 (the plan leaves
1e-12 of sum |w A|, a few hundred times |S|), FP32 2e-5 (field, adjoint and
voxel sums each within a few 1e-6 of 64 bits).
"""
import numpy as np
import pytest

from workloads import (DETECTOR_UNIFORM_Q, ELLIPSOID, SPHERE, SPHHARM, Geometry, Shape, random_alm)

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-9, "fp32": 2e-5}


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _grad(g, s, prec, w, q_list=None):
    import torch
    import paper_2202_03411_gb300 as sm
    h = sm.scatman_create(g, prec, soft=True, soft_width=0.6 * g.voxel, q_list=q_list)
    real = torch.float64 if prec == "fp64" else torch.float32
    I = torch.empty(sm.scatman_n_pix(h), dtype=real, device="cuda")
    sm.scatman_voxelise(h, s)
    sm.scatman_forward(h, I)
    up = torch.as_tensor(w, device="cuda").to(real)
    grad, again = sm.scatman_backward(h, up), sm.scatman_backward(h, up)
    q = sm.scatman_get_q(h)
    h.close()
    assert np.array_equal(grad, again, equal_nan=True)
    return grad, q


# grids and detectors off every tile: odd and even sides, one row, one column,
# one slice, more points than a thread's share, several chunks of pixels
GEOMETRIES = [
    Geometry(21, 19, 23, 1.0, 7.0, 50.0, 45, 37),
    Geometry(64, 30, 17, 1.0, 6.0, 60.0, 33, 64),
    Geometry(20, 72, 1, 0.7, 5.0, 75.0, 131, 1),
    Geometry(35, 3, 40, 1.3, 9.0, 20.0, 1, 140),
    Geometry(140, 24, 33, 1.0, 5.0, 55.0, 40, 600),
    Geometry(24, 27, 30, 1.0, 5.0, 40.0, 70, 65, DETECTOR_UNIFORM_Q),
    Geometry(22, 26, 20, 1.0, 6.0, 44.5, 631, 40, DETECTOR_UNIFORM_Q),    # just inside the sphere's rim
    Geometry(24, 24, 24, 1.0, 5.0, 60.0, 64, 64, DETECTOR_UNIFORM_Q),     # off-sphere corners: direct
]


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("k", range(len(GEOMETRIES)))
def test_plain_modes(k, prec):
    g = GEOMETRIES[k]
    rng = np.random.default_rng(k)
    lo = g.voxel * min(g.nx, g.ny, g.nz)
    shapes = [Shape(ELLIPSOID, a=0.3 * g.nx * g.voxel, b=0.25 * g.ny * g.voxel + 0.4, c=0.3 * g.nz * g.voxel + 0.4,
                    delta=0.02, beta=0.004, latitude=-88, longitude=4, rotation=3, cx=0.1 * g.nx * g.voxel,
                    cy=-0.1 * g.ny * g.voxel)]
    if lo > 12:
        shapes.append(Shape(SPHHARM, R0=0.3 * lo, lmax=3, alm=random_alm(rng, 3, 0.08), delta=0.02, beta=0.003,
                            latitude=20, longitude=70, rotation=-30))
    for s in shapes:
        w = 0.5 + rng.random(g.n_pix)
        got, q = _grad(g, s, prec, w)
        flat = Geometry(g.nx, g.ny, g.nz, g.voxel, g.wavelength, g.theta_max_deg, g.det_nx, g.det_ny)
        if g.detector == DETECTOR_UNIFORM_Q:
            k0 = 2 * np.pi / g.wavelength
            w = w * ((q[:, 0] ** 2 + q[:, 1] ** 2) / k0 ** 2 <= 1.0)
        ref, _ = _grad(flat, s, prec, w, q_list=q)
        err = np.linalg.norm(got - ref) / np.linalg.norm(ref)
        assert err < TOL[prec], (g, prec, s.kind, err)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_not_a_number_upstream_reaches_the_gradient(prec):
    g = Geometry(20, 22, 18, 1.0, 5.0, 45.0, 30, 26)
    w = np.ones(g.n_pix)
    w[77] = np.nan
    grad, _ = _grad(g, Shape(SPHERE, r=6.0, delta=0.02, beta=0.003), prec, w)
    assert np.all(np.isnan(grad))


@pytest.mark.parametrize("prec", ["tc_f16_split", "tc_bf16_split", "tc_f16"])
@pytest.mark.parametrize("g", [
    Geometry(40, 36, 44, 1.0, 7.0, 45.0, 150, 141),
    Geometry(96, 128, 3, 1.0, 9.0, 40.0, 256, 257),           # three slices: one product sum per slice
    Geometry(140, 40, 36, 1.0, 8.0, 45.0, 160, 130),          # wider than the tensor-core adjoint takes
])
def test_tensor_core_modes(g, prec):
    """The same slices on both sides.  5e-5: the direct tensor-core adjoint rounds
    its operands to FP16 (2^-12 each, independent over 20000 pixels and more), the
    fields of the two sides differ by a few 1e-6; the grid's split operands add less."""
    s = Shape(ELLIPSOID, a=0.3 * g.nx, b=0.3 * g.ny, c=0.3 * g.nz + 0.3, delta=0.02, beta=0.004, latitude=-80,
              longitude=4, rotation=3, cy=-0.05 * g.ny)
    w = 0.5 + np.random.default_rng(g.nx).random(g.n_pix)
    got, q = _grad(g, s, prec, w)
    ref, _ = _grad(g, s, prec, w, q_list=q)
    err = np.linalg.norm(got - ref) / np.linalg.norm(ref)
    assert err < 5e-5, (g, prec, err)


@pytest.mark.parametrize("shape,peak", [
    (Shape(SPHERE, r=30.0, delta=0.01, beta=0.001), 0.15),
    (Shape(ELLIPSOID, a=14.0, b=30.0, c=33.0, delta=0.01, beta=0.001, latitude=20, longitude=50), 0.3),
    (Shape(ELLIPSOID, a=3.0, b=30.0, c=33.0, delta=0.01, beta=0.001, latitude=20, longitude=50), 1.0),
])
def test_fit_handles_keep_the_peak_direct(shape, peak):
    """With soft occupancy the pixels around the forward direction carry the direct
    sums' values (up to the order of at most four partial sums, 4 x 2^-24 in the
    field), the others the grid's."""
    import torch
    import paper_2202_03411_gb300 as sm
    g = Geometry(96, 96, 80, 1.0, 10.0, 45.0, 201, 230)
    h = sm.scatman_create(g, "fp32")
    q = sm.scatman_get_q(h)
    h.close()
    out = []
    for ql in (None, q):
        h = sm.scatman_create(g, "tc_bf16_split", soft=True, soft_width=0.5, q_list=ql)
        I = torch.empty(g.n_pix, device="cuda")
        sm.scatman_voxelise(h, shape)
        sm.scatman_forward(h, I)
        sm.scatman_sync(h)
        out.append(I.cpu().double().numpy().reshape(g.det_ny, g.det_nx))
        h.close()
    x = np.abs((2 * np.arange(g.det_nx) + 1 - g.det_nx) / g.det_nx)
    y = np.abs((2 * np.arange(g.det_ny) + 1 - g.det_ny) / g.det_ny)
    at = np.ix_(y <= peak, x <= peak)
    d = np.linalg.norm(out[0][at] - out[1][at]) / np.linalg.norm(out[1][at])
    assert d < 5e-7, d
    assert np.linalg.norm(out[0] - out[1]) / np.linalg.norm(out[1]) < 1e-4


def _fit_gradient(g, s, target_shape, prec, q_list=None):
    """I and the gradient of sum (I - t)^2, with t the pattern of `target_shape` in FP32."""
    import torch
    import paper_2202_03411_gb300 as sm
    h = sm.scatman_create(g, "fp32")
    t = torch.empty(g.n_pix, device="cuda")
    sm.scatman_voxelise(h, target_shape)
    sm.scatman_forward(h, t)
    sm.scatman_sync(h)
    q = sm.scatman_get_q(h)
    h.close()
    h = sm.scatman_create(g, prec, soft=True, soft_width=0.5, q_list=q if q_list else None)
    I = torch.empty(g.n_pix, device="cuda")
    sm.scatman_voxelise(h, s)
    sm.scatman_forward(h, I)
    sm.scatman_sync(h)
    grad = sm.scatman_backward(h, 2 * (I - t))
    h.close()
    return I.cpu().numpy(), grad


@pytest.mark.parametrize("prec", ["tc_f16_split", "tc_bf16_split", "tc_bf16"])
def test_tensor_core_fit_gradient_is_the_pixel_sum(prec):
    """A served fit (48^3 on 128^2 pixels) near its target: the upstream weight cancels,
    so the gradient shows the adjoint's operand roundings (1e-4 of it between the sum
    over the pixels and one over the grid's directions).  The detector's pixels
    and the same pixels as a list of q take the same sums: bit for bit equal."""
    g = Geometry(48, 48, 48, 1.0, 10.0, 45.0, 128, 128)
    rng = np.random.default_rng(5)
    s = Shape(SPHHARM, R0=14.4, lmax=6, alm=random_alm(rng, 6), delta=0.012, beta=0.0012, latitude=25, longitude=-130,
              rotation=70)
    near = Shape(SPHERE, r=14.6, delta=0.012, beta=0.0012)
    I, grad = _fit_gradient(g, s, near, prec)
    I_q, grad_q = _fit_gradient(g, s, near, prec, q_list=True)
    assert np.array_equal(I, I_q)
    assert np.any(grad != 0) and np.array_equal(grad, grad_q)


@pytest.mark.parametrize("shape", [
    Shape(SPHERE, r=30.0, delta=0.01, beta=0.001),
    Shape(SPHHARM, R0=30.0, lmax=2, alm=np.array([0, 0, 0, 0, 0, 0, -0.35, 0, 0.25]), delta=0.01, beta=0.001,
          latitude=35, longitude=20, rotation=10),              # 0.75 R0 across its thinnest axis
])
@pytest.mark.parametrize("prec", ["tc_f16_split", "tc_bf16_split"])
def test_split_phase_fit_is_the_pixel_sum(shape, prec):
    """The pattern of a fit of 96^3 on 256^2, where a forward pass without soft occupancy
    goes through the grid: the phase pairs' roundings of every pixel are its
    own, and so are loss and gradient near the target (bit for bit)."""
    g = Geometry(96, 96, 96, 1.0, 10.0, 45.0, 256, 256)
    near = Shape(SPHERE, r=30.3, delta=0.01, beta=0.001)
    I, grad = _fit_gradient(g, shape, near, prec)
    I_q, grad_q = _fit_gradient(g, shape, near, prec, q_list=True)
    assert I.max() > 0 and np.array_equal(I, I_q)
    assert np.any(grad != 0) and np.array_equal(grad, grad_q)
