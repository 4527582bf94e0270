"""The FP64 re-decision where many regions tie (GPU only).

The apex of a bipyramid of n sides sits on a grid point, and the band's width is the distance to
the grid point three cells above it, one FP32 step more, or one less.  Every face and edge of
the apex is exactly as far from that point as the apex itself: at n = 6 they fit a point's share of
the re-decision's queue, at 40 they exceed its list, at 400 and 1500 they exceed it several times
over, and at 1500 the tile's regions are shared by several warps.
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


@pytest.mark.parametrize("n", [6, 40, 400, 1500])
@pytest.mark.parametrize("step", [-1, 0, 1])
def test_apex_at_the_band_edge(n, step):
    N = 32
    h = 1.0 / N
    c = 16.5 * h  # a grid point, exact in FP32
    a = 2 * np.pi * np.arange(n) / n
    ring = np.stack([c + 0.2 * np.cos(a), c + 0.2 * np.sin(a), np.full(n, c - 0.05)], axis=1)
    verts = np.concatenate([[[c, c, c], [c, c, c - 0.15]], ring])
    i, j = 2 + np.arange(n), 2 + (np.arange(n) + 1) % n
    tris = np.concatenate([np.stack([np.zeros(n, int), i, j], 1), np.stack([np.ones(n, int), j, i], 1)])
    soup = meshgen.Mesh(verts, tris.astype(np.int32)).soup(seed=n)
    w = np.float32(3 * h)
    if step:
        w = np.nextafter(w, np.float32(step * np.inf))
    feats = sdf.sdf_build_features(torch.from_numpy(soup).cuda())
    dist, win = sdf.sdf_narrow_band(feats, sdf.Grid.cube(N), float(w), winner=True)
    dist, win = dist.cpu().numpy(), win.cpu().numpy()
    assert feats.status()["fp64_points"] >= 1
    om = oracle.OracleMesh.from_soup(soup)
    st = parity.compare(dist, om.narrow_band((N, N, N), (0, 0, 0), h, float(w) + 2 * h), float(w), h)
    parity.assert_parity(st)
    # the point above the apex: in the band only where w exceeds 3 h, and won by the apex
    apex = int(np.flatnonzero((feats.vertices().cpu().numpy() == np.float32(c)).all(axis=1))[0])
    k = 16 + 3
    if step > 0:
        assert dist[k, 16, 16] == np.float32(3 * h)
        assert win[k, 16, 16] == feats.n_tri + feats.n_edge + apex
    else:
        assert np.isinf(dist[k, 16, 16]) and win[k, 16, 16] == -1
