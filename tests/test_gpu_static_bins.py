"""The binning without kept boxes (GPU only): the allocation-free entry point works out each region's box in
both passes, and a region next to a grid point must be kept by both or by neither.  On a mesh with thousands
of nearly flat edges and vertices (regions thin as needles) its field and winners must be the regular
call's, which keeps the boxes, bit for bit.  In the first case the two passes, compiled apart, once
disagreed and the call was refused."""
import ctypes

import numpy as np
import pytest
import torch

import meshgen
import paper_1903_00353_gb300 as sdf

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def agree(feats, grid, w):
    want, win = sdf.sdf_narrow_band(feats, grid, w, winner=True)
    d, wn = torch.empty_like(want), torch.empty_like(win)
    cg = grid.c()
    code = sdf.load_library().sdf_narrow_band_static(feats.handle, ctypes.byref(cg), w, d.data_ptr(), wn.data_ptr(),
                                                     torch.cuda.current_stream().cuda_stream)
    assert code == 0
    assert torch.isfinite(want).any() and torch.equal(d, want) and torch.equal(wn, win)


def noisy_union(rng):
    base = meshgen.box_union(2, 7550.0, seed=712)
    v = base.vertices - 0.5
    return meshgen.Mesh(v + 1e-6 * rng.standard_normal(v.shape), base.triangles)


def test_the_refused_call():
    rng = np.random.Generator(np.random.PCG64(11829))  # the draws of the random call that was refused
    for a, b in ((0, 10), (1, 1000), (2, 4), (100, 8000)):
        rng.integers(a, b)
    rng.random()
    m = noisy_union(rng)
    rng.choice(4), rng.random(), rng.random(), rng.random()
    scale = 10 ** rng.uniform(-3, 3)
    shift = 0.5 * rng.standard_normal(3)
    assert abs(scale - 0.5122760469) < 1e-9 and abs(shift[1] + 0.7730454) < 1e-6
    soup = meshgen.Mesh((m.vertices + shift) * scale, m.triangles).soup(seed=11829)
    feats = sdf.sdf_build_features(torch.from_numpy(soup).cuda())
    grid = sdf.Grid(83, 83, 83, (-0.19260190427303314, -0.5195608139038086, -0.1292906254529953), 0.0032885142136365175)
    agree(feats, grid, 0.007542196195572615)


@pytest.mark.parametrize("seed", range(8))
def test_static_equals_regular(seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    m = noisy_union(rng) if seed % 2 else meshgen.knot_tube(n_along=1200, n_around=24, seed=seed)
    v = m.vertices + rng.standard_normal(3)
    feats = sdf.sdf_build_features(torch.from_numpy(meshgen.Mesh(v, m.triangles).soup(seed=seed)).cuda())
    lo, ext = v.min(axis=0), float((v.max(axis=0) - v.min(axis=0)).max())
    for _ in range(12):
        n = int(rng.integers(40, 90))
        h = float(np.float32(ext * rng.uniform(0.6, 1.2) / n))
        origin = tuple(float(np.float32(x - h * rng.uniform(0, 4))) for x in lo)
        agree(feats, sdf.Grid(n, n, n, origin, h), float(np.float32(h * rng.uniform(0.7, 6.0))))
