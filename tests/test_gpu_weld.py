"""The weld's vertices against numpy (GPU only): sorts on either side of the two-barrier limit (128 tiles,
65536 keys), and meshes whose vertices share Morton cells, with mixed runs of equal keys from a few
entries (put in order by a thread) to hundreds (by a block)."""
import numpy as np
import pytest
import torch

import meshgen
import paper_1903_00353_gb300 as sdf

pytestmark = pytest.mark.gpu

CASES = {
    "one_tile": lambda: meshgen.icosphere(2, radius=0.3),
    "torus_65532_corners": lambda: meshgen.torus(nu=127, nv=86, seed=3),
    "torus_65538_corners": lambda: meshgen.torus(nu=331, nv=33, seed=3),
    "cluster_short_runs": lambda: meshgen.dense_cluster(freq_big=2, freq_small=12),
    "cluster_mixed_runs": lambda: meshgen.dense_cluster(freq_big=2, freq_small=30),
    "cluster_long_runs": lambda: meshgen.dense_cluster(freq_big=2, freq_small=90),
}


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("case", list(CASES))
def test_weld_equals_unique(case):
    soup = CASES[case]().soup(seed=7)
    corners = soup.reshape(-1, 3)
    feats = sdf.sdf_build_features(torch.from_numpy(soup).cuda())
    vmap = feats.vertex_map().cpu().numpy()
    verts = feats.vertices().cpu().numpy()
    assert feats.n_vert == len(np.unique(corners, axis=0)) == len(np.unique(verts, axis=0))
    assert np.array_equal(verts[vmap], corners)
    # the library's faces are the soup's, and every edge joins two faces that share its end points
    fmap = feats.face_map().cpu().numpy()
    assert np.array_equal(np.sort(fmap), np.arange(feats.n_tri))
    tri = vmap.reshape(-1, 3)[fmap]
    e = feats.edges().cpu().numpy()
    for f in (e[:, 2], e[:, 3]):
        t = tri[f]
        assert np.all((t == e[:, :1]).any(axis=1) & (t == e[:, 1:2]).any(axis=1))
