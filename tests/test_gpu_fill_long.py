"""The sign beyond the band on long axes (GPU only): grids of more than 1024 points along x, y or z that
start inside or outside a sphere, far from its surface, against the propagation written out in numpy."""
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


def propagate(sign, axis):
    """Unknown entries (0) take the sign of the nearest known entry before them, else after them."""
    s = np.moveaxis(sign, axis, -1).copy()
    pos = np.where(s != 0, np.arange(s.shape[-1]), -1)
    last = np.maximum.accumulate(pos, axis=-1)
    first = np.where((s != 0).any(axis=-1), (s != 0).argmax(axis=-1), 0)[..., None]
    idx = np.where(last >= 0, last, first)
    return np.moveaxis(np.take_along_axis(s, idx, axis=-1), -1, axis)


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("side", [-1, 1])
@pytest.mark.parametrize("length", [1023, 1025, 2500])
def test_long_axes(axis, side, length):
    dims = [37, 9, 11]
    dims[axis] = length
    h = float(np.float32(0.5 / length))
    centre = [0.5] * 3
    centre[axis] += 0.25 * side  # from the sphere's centre outward, or from outside to the centre
    origin = tuple(float(np.float32(c - 0.5 * n * h)) for c, n in zip(centre, dims))
    feats = sdf.sdf_build_features(torch.from_numpy(meshgen.icosphere(6, radius=0.3).soup(seed=1)).cuda())
    grid = sdf.Grid(*dims, origin, h)
    band = sdf.sdf_narrow_band(feats, grid, 3 * h).cpu().numpy()
    got = sdf.sdf_narrow_band(feats, grid, 3 * h, flags=sdf.FLAG_FILL_SIGN).cpu().numpy()
    sign = np.where(np.isfinite(band), np.where(np.signbit(band), -1, 1), 0)
    assert (sign == 1).any() and (sign == -1).any()
    for a in (2, 1, 0):
        sign = propagate(sign, a)
    want = np.where(np.isfinite(band), band, np.where(sign < 0, -np.inf, np.inf).astype(np.float32))
    assert np.array_equal(got, want)
    assert np.isneginf(got).any() and np.isposinf(got).any()
