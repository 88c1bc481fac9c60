"""Passes captured in a CUDA graph, and map uploads that follow one another.

A captured pass launches what an uncaptured one does, so replays give its bits.  A
captured map upload reads its own copy of the map at every replay, whatever the handle
has voxelised since; uploads in a row reuse two staging buffers without waiting for the
stream.
"""
import numpy as np
import pytest

from workloads import RADIALMAP, SPHHARM, VOLUMEMAP, Geometry, Shape, random_alm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _volume(n, value, cells=7):
    v = np.ones((cells, cells, cells), dtype=bool)
    v[:2, 1:3] = False
    return Shape(VOLUMEMAP, volume_map=v, map_dx=0.6 * n / cells, map_delta=np.full(v.shape, value),
                 map_beta=np.full(v.shape, 0.1 * value), latitude=10, longitude=30, rotation=5)


def _radii(n, scale):
    r = scale * n * (1 + 0.1 * np.cos(np.arange(12)[:, None] * 0.5) * np.sin(np.arange(20)[None, :] * 0.6))
    return Shape(RADIALMAP, radial_map=r, delta=0.01, beta=0.001, latitude=10, longitude=30, rotation=5)


CASES = [("fp64", Geometry(24, 22, 26, 1.0, 8.0, 40.0, 40, 37)), ("fp32", Geometry(40, 40, 40, 1.0, 8.0, 40.0, 96, 96)),
         ("tc_bf16_split", Geometry(96, 96, 96, 1.0, 10.0, 45.0, 128, 128)),       # through the grid
         ("tc_f16", Geometry(40, 36, 44, 1.0, 8.0, 40.0, 70, 61))]                # over the pixels


@pytest.mark.parametrize("prec,g", CASES)
def test_captured_passes_replay_their_bits(prec, g):
    import torch
    import paper_2202_03411_gb300 as sm
    shapes = [Shape(SPHHARM, R0=0.35 * g.nx, lmax=4, alm=random_alm(np.random.default_rng(1), 4), delta=0.01, beta=0.001),
              _volume(g.nx, 0.01), _radii(g.nx, 0.3)]
    st = torch.cuda.Stream()
    h = sm.scatman_create(g, prec, stream=st.cuda_stream)
    I = torch.zeros(g.n_pix, dtype=torch.float64 if prec == "fp64" else torch.float32, device="cuda")
    torch.cuda.synchronize()
    want, graphs = [], []
    with torch.cuda.stream(st):
        for s in shapes:                            # (buffers grow here: an allocation cannot be captured)
            sm.scatman_voxelise(h, s)
            sm.scatman_forward(h, I)
            sm.scatman_sync(h)
            want.append(I.clone())
    torch.cuda.synchronize()
    for s in shapes:
        graphs.append(torch.cuda.CUDAGraph())
        with torch.cuda.graph(graphs[-1], stream=st):
            sm.scatman_voxelise(h, s)
            sm.scatman_forward(h, I)
    for order in ((0, 1, 2), (2, 1, 0), (1, 1, 2)):
        for k in order:
            I.zero_()
            torch.cuda.synchronize()
            with torch.cuda.stream(st):
                graphs[k].replay()
            torch.cuda.synchronize()
            assert want[k].max() > 0 and torch.equal(I, want[k]), (k, order)
    with torch.cuda.stream(st):                     # uncaptured again
        sm.scatman_voxelise(h, shapes[1])
        sm.scatman_forward(h, I)
        sm.scatman_sync(h)
    torch.cuda.synchronize()
    assert torch.equal(I, want[1])
    del graphs
    h.close()


@pytest.mark.parametrize("prec,g", CASES[1:3])
def test_map_uploads_in_a_row(prec, g):
    """Six passes over maps of two kinds and growing sizes, queued without a wait, and a
    refused map between them: each pattern is the one of a handle that waits."""
    import torch
    import paper_2202_03411_gb300 as sm
    shapes = [_volume(g.nx, 0.01), _volume(g.nx, 0.02), _radii(g.nx, 0.3), _volume(g.nx, 0.015, 19), _radii(g.nx, 0.2),
              _volume(g.nx, 0.005, 33)]
    bad = _volume(g.nx, 0.01)
    bad.map_beta = bad.map_beta.copy()
    bad.map_beta[-1, -1, -1] = np.inf
    h, one = sm.scatman_create(g, prec), sm.scatman_create(g, prec)
    out = torch.zeros(len(shapes), g.n_pix, device="cuda")
    ref = torch.zeros_like(out)
    torch.cuda.synchronize()
    for k, s in enumerate(shapes):
        sm.scatman_voxelise(h, s)
        with pytest.raises(sm.ScatmanError) as e:
            sm.scatman_voxelise(h, bad)
        assert e.value.code == -1                   # ERR_ARG, and the shape before it stays
        sm.scatman_forward(h, out[k])
    sm.scatman_sync(h)
    for k, s in enumerate(shapes):
        sm.scatman_voxelise(one, s)
        sm.scatman_sync(one)
        sm.scatman_forward(one, ref[k])
        sm.scatman_sync(one)
    h.close()
    one.close()
    assert ref.min(dim=1).values.min() >= 0 and (ref.max(dim=1).values > 0).all() and torch.equal(out, ref)
