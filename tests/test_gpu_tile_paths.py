"""The tile kernel's two CTA sizes and its ways through a tile give the same field (GPU only).

A call on a small grid runs the tile kernel with 256 threads per CTA, a launch over more than 16384
tiles with 128; a tile of at most that many regions is set up in one pass, a larger one in chunks per
warp, a much larger one split.  The meshes below have tiles from a few to thousands of regions on
their grids; each is evaluated alone and in a batch whose large last grid takes the launch beyond the
line, densely with winners and with band lists: bit for bit the same.
"""
import pytest
import torch

import meshgen
import paper_1903_00353_gb300 as sdf

pytestmark = pytest.mark.gpu

CASES = [  # mesh, grid sides, band in cells
    (lambda: meshgen.icosphere(1, radius=0.3), (33, 9, 40), 2.0),
    (lambda: meshgen.icosphere(4, radius=0.3), (64, 64, 64), 3.0),
    (lambda: meshgen.icosphere(20, radius=0.3, displacement=0.02, seed=2), (45, 37, 61), 3.0),
    (lambda: meshgen.torus(nu=90, nv=36, seed=3), (96, 96, 40), 4.0),
    (lambda: meshgen.knot_tube(n_along=2400, n_around=32, seed=4), (72, 70, 35), 3.0),
    (lambda: meshgen.dense_cluster(freq_big=3, freq_small=40), (56, 56, 56), 3.0),
]


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _sorted(entries):
    e = entries.cpu().long()
    return e[torch.argsort(e[:, 0])]


def test_small_launches_equal_a_large_batch():
    feats, grids, ws = [], [], []
    for make, dims, cells in CASES + [(lambda: meshgen.icosphere(6, radius=0.3), (416, 416, 416), 2.0)]:
        h = 1.0 / max(dims)
        feats.append(sdf.sdf_build_features(torch.from_numpy(make().soup(seed=1)).cuda()))
        grids.append(sdf.Grid(*dims, tuple(0.5 - 0.5 * n * h for n in dims), h))
        ws.append(cells * h)
    tiles = [-(-g.nx // 32) * -(-g.ny // 8) * -(-g.nz // 8) for g in grids]
    assert max(tiles[:-1]) <= 16384 < sum(tiles)
    batch = sdf.sdf_narrow_band(feats, grids, ws, winner=True)
    outs, lists = sdf.sdf_narrow_band_lists(feats, grids, ws)
    for f, g, w, (d, win), d2, bl in zip(feats[:-1], grids, ws, batch, outs, lists):
        alone, win1 = sdf.sdf_narrow_band(f, g, w, winner=True)
        assert torch.equal(alone, d) and torch.equal(win1, win) and torch.equal(alone, d2)
        d3, bl1 = sdf.sdf_narrow_band_list(f, g, w)
        assert torch.equal(d3, alone)
        n = int(torch.isfinite(alone).sum())
        assert len(bl) == len(bl1) == n
        a, b = _sorted(bl.entries[:n]), _sorted(bl1.entries[:n])
        assert torch.equal(a, b)
        assert torch.equal(win1.reshape(-1).cpu().long()[a[:, 0]], a[:, 1])


@pytest.mark.parametrize("make", [lambda: meshgen.torus(nu=120, nv=48, seed=5),
                                  lambda: meshgen.dense_cluster(freq_big=3, freq_small=30)])
def test_work_list_in_one_block(make):
    """Launches over at most 8192 tiles list them in one block: 8192 tiles against the same layers of
    8448 (three launches), one problem and a batch (listed by cost class), down to a single tile."""
    feats = sdf.sdf_build_features(torch.from_numpy(make().soup(seed=2)).cuda())
    h = 1.0 / 512
    origin = (0.0, 0.5 - 64 * h, 0.5 - 128 * h)
    one = sdf.Grid(512, 128, 256, origin, h)
    more = sdf.Grid(512, 128, 264, origin, h)
    w = 3 * h
    d1, w1 = sdf.sdf_narrow_band(feats, one, w, winner=True)
    d2, w2 = sdf.sdf_narrow_band(feats, more, w, winner=True)
    assert torch.isfinite(d1).any()
    assert torch.equal(d1, d2[:256]) and torch.equal(w1, w2[:256])
    grids = [sdf.Grid(512, 128, 128, origin, h), sdf.Grid(512, 128, 100, origin, h, k0=128), sdf.Grid(20, 5, 3, origin, h)]
    d3 = sdf.sdf_narrow_band([feats] * 3, grids, [w] * 3)
    assert torch.equal(d3[0], d1[:128]) and torch.equal(d3[1], d1[128:228]) and torch.equal(d3[2], d1[:3, :5, :20])
    assert torch.equal(sdf.sdf_narrow_band(feats, grids[2], w), d1[:3, :5, :20])
