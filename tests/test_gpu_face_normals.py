"""Face normals on both sides of the filter that chooses how 1 / |n| is worked out (GPU only).

Faces clearly not degenerate and of a size within FP32's range take Newton's iteration from the FP32 value,
the others the FP64 square root and quotient; both end within FP64 rounding, so the FP32 normals are the
same.  The filter is absolute in size and everything else scales: a mesh and its grid scaled by a
power of two must give exactly the scaled field, for sizes below, across and above the filter's
limits (edges near 1e-6, squared doubled areas near 1e-30 and 1e30)."""
import numpy as np
import pytest
import torch

import meshgen
import paper_1903_00353_gb300 as sdf

pytestmark = pytest.mark.gpu

H = 2.0 ** -6
STRETCH = {"round": (1.0, 1.0, 1.0), "needle": (1.0, 2.0 ** -12, 2.0 ** -12)}
CASES = [("round", k) for k in (-20, -18, -17, -16, -15, 27, 28, 29, 30)] + \
        [("needle", k) for k in (-20, -17, -16, -15, -14, -13, 33, 34, 35)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def field(shape, k):
    m = meshgen.icosphere(4, radius=0.3, center=(0.0, 0.0, 0.0))
    soup = meshgen.Mesh(m.vertices * np.array(STRETCH[shape]), m.triangles).soup(seed=2)
    feats = sdf.sdf_build_features(torch.from_numpy(np.ldexp(soup, k).astype(np.float32)).cuda())
    dims = (48, 48, 48) if shape == "round" else (48, 8, 8)
    h = H * 2.0 ** k
    grid = sdf.Grid(*dims, tuple(-0.5 * n * h for n in dims), h)
    return sdf.sdf_narrow_band(feats, grid, 3 * h).cpu().numpy()


@pytest.mark.parametrize("shape,k", CASES)
def test_field_scales_with_the_mesh(shape, k):
    want, got = field(shape, 0), field(shape, k)
    assert np.isfinite(want).any()
    assert np.array_equal(got, np.ldexp(want, k))
