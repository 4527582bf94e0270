"""The sign beyond the band on a row of nearly 2^31 points (GPU only), whose last step of 1024 points ends
beyond the largest 32-bit int: the row ends inside a sphere, and its last points must be those of a
short grid over the same layers, all before them outside."""
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


def test_a_row_of_nearly_two_to_the_31_points():
    h = 2.0 ** -12
    nx, tail = 2 ** 31 - 512, 4096
    base = meshgen.icosphere(4, radius=400 * h, center=(0.0, 0.0, 0.0))
    soup = meshgen.Mesh(base.vertices - np.array([511.5 * h, 0.0, 0.0]), base.triangles).soup(seed=1)
    feats = sdf.sdf_build_features(torch.from_numpy(soup).cuda())
    # points at (i + 1/2 - 2^31) h: the same as those of the short grid, in FP64
    long = sdf.Grid(nx, 1, 1, (-(2.0 ** 31) * h, -0.5 * h, -0.5 * h), h)
    short = sdf.Grid(tail, 1, 1, (-(512 + tail) * h, -0.5 * h, -0.5 * h), h)
    w = 3 * h
    want = sdf.sdf_narrow_band(feats, short, w, flags=sdf.FLAG_FILL_SIGN).reshape(-1)
    got = sdf.sdf_narrow_band(feats, long, w, flags=sdf.FLAG_FILL_SIGN).reshape(-1)
    assert torch.isneginf(want[-1]) and torch.isposinf(want[0]) and torch.isfinite(want).any()
    end = got[-tail:]
    assert torch.equal(torch.isfinite(end), torch.isfinite(want))
    assert torch.equal(torch.signbit(end), torch.signbit(want))
    band = torch.isfinite(want)
    assert float((end[band] - want[band]).abs().max()) <= feats.error_bound(short, w)["delta"]
    step = 1 << 28
    for a in range(0, nx - tail, step):
        assert bool(torch.isposinf(got[a:min(a + step, nx - tail)]).all())
