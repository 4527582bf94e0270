"""Edge and vertex regions that pass between the grid points (GPU only).

The binning leaves out regions that hold no grid point.  Here the meshes are finer than the grid, so
that most edge and vertex regions are needles: the whole field must match the FP64 oracle on cubic,
ragged and shifted grids, far from the origin (a large inclusion tolerance) and on a slab, for bands
from below two cells to beyond the longest tested reach (16 cells).
"""
import numpy as np
import pytest
import torch

import meshgen
import oracle
import paper_1903_00353_gb300 as sdf
from tests import parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def f32(x):
    return float(np.float32(x))


MESHES = {
    "sphere": lambda: meshgen.icosphere(24, radius=0.3, displacement=0.02, seed=4),
    "knot": lambda: meshgen.knot_tube(n_along=1500, n_around=24, seed=5),
    "torus": lambda: meshgen.torus(nu=150, nv=60, jitter=5e-4, seed=6),
    "union": lambda: meshgen.box_union(3, 6000, seed=353_377),
}


@pytest.mark.parametrize("mesh", list(MESHES))
@pytest.mark.parametrize("dims,shift,cells", [((48, 48, 48), 0.0, 3.0), ((57, 41, 43), 0.0, 1.5),
                                              ((40, 52, 37), -7.3, 5.0), ((96, 96, 96), 0.0, 4.0),
                                              ((64, 64, 64), 0.0, 18.0)])
def test_needles_against_the_oracle(mesh, dims, shift, cells):
    base = MESHES[mesh]()
    soup = meshgen.Mesh(base.vertices + shift, base.triangles).soup(seed=3)
    h = f32(0.97 / max(dims))
    origin = tuple(f32(shift + 0.5 - 0.5 * n * h) for n in dims)
    w = f32(cells * h)
    grid = sdf.Grid(*dims, origin, h)
    feats = sdf.sdf_build_features(torch.from_numpy(soup).cuda())
    dist, win = sdf.sdf_narrow_band(feats, grid, w, winner=True)
    bound = feats.error_bound(grid, w)
    om = oracle.OracleMesh.from_soup(soup)
    st = parity.compare(dist.cpu().numpy(), om.narrow_band(dims, origin, h, w + 2 * h), w, h)
    assert st["mask_mismatch"] == 0 and st["sign_mismatch"] == 0, st
    assert st["max_abs_err"] <= bound["delta"], (st, bound)
    if mesh == "sphere" and cells <= 4.0 and max(dims) < 60:
        # fewer (tile, region) pairs than regions: most edges and vertices are left out
        assert feats.status()["pairs"] < feats.n_tri + feats.n_edge + feats.n_vert
    # a slab of the grid is bitwise its layers
    k0 = 16
    part = sdf.Grid(dims[0], dims[1], dims[2] - k0, origin, h, k0=k0)
    d2, w2 = sdf.sdf_narrow_band(feats, part, w, winner=True)
    assert torch.equal(d2, dist[k0:]) and torch.equal(w2, win[k0:])
