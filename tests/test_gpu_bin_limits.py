"""The binning at the limits of its size-dependent branches (GPU only): along each axis in turn, grids of
4096 points (thin regions tested for grid points) and 4097 (not tested), and of 65536 (boxes kept as 16-bit
indices between the binning's passes) and 65537 (worked out again).  A mesh finer than the grid, rich in
saddles, lies at the far end.  Field against the FP64 oracle there; both grids of a pair share their
origin and so their error windows, and agree bit for bit on their common points, winners included."""
import pytest
import torch

import meshgen
import oracle
import paper_1903_00353_gb300 as sdf
from tests import parity

pytestmark = pytest.mark.gpu

H, W, CROSS, TAIL = 2.0 ** -6, 3 * 2.0 ** -6, 28, 88


@pytest.fixture(scope="module")
def mesh():
    import __graft_entry__
    __graft_entry__.build()
    soup = meshgen.torus(nu=300, nv=120, jitter=5e-4, seed=6).soup(seed=3)
    return sdf.sdf_build_features(torch.from_numpy(soup).cuda()), oracle.OracleMesh.from_soup(soup)


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("n", [4096, 65536])
def test_either_side_of_the_limit(mesh, axis, n):
    feats, om = mesh
    origin = [28 * H, 28 * H, 18 * H]
    origin[axis] = (72 - n) * H  # multiples of H: exact in FP32
    fields = []
    for length in (n + 1, n):
        dims = [CROSS] * 3
        dims[axis] = length
        grid = sdf.Grid(*dims, tuple(origin), H)
        d, win = sdf.sdf_narrow_band(feats, grid, W, winner=True)
        fields.append((d.narrow(2 - axis, 0, n), win.narrow(2 - axis, 0, n)))
    assert torch.equal(fields[0][0], fields[1][0]) and torch.equal(fields[0][1], fields[1][1])
    dist = fields[1][0]
    assert not torch.isfinite(dist.narrow(2 - axis, 0, n - TAIL)).any()
    dims, start = [CROSS] * 3, list(origin)
    dims[axis], start[axis] = TAIL, (72 - TAIL) * H
    want = om.narrow_band(tuple(dims), tuple(start), H, W + 2 * H)
    st = parity.compare(dist.narrow(2 - axis, n - TAIL, TAIL).cpu().numpy(), want, W, H)
    assert st["band_gpu"] > 1000 and st["mask_mismatch"] == 0 and st["sign_mismatch"] == 0, st
    assert st["max_abs_err"] <= feats.error_bound(grid, W)["delta"], st
