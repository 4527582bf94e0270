"""Long mixed runs of equal weld keys (GPU only): hundreds of thousands of vertices in one Morton cell, so
that each of the 1024 hash values of the cell is a run of hundreds to thousands of different corners, on
either side of the 2048 entries that a block sorts in shared memory.  The vertices must be numpy's,
and the build must stay near one of the same size without such runs (one thread per run of more than
2048 entries took 1.3 s)."""
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


@pytest.mark.parametrize("freq", [150, 190, 270])  # runs of about 1320, 2115 and 4270 entries
def test_runs_of_thousands(freq):
    soup = meshgen.dense_cluster(freq_big=2, freq_small=freq).soup(seed=7)
    on_gpu = torch.from_numpy(soup).cuda()
    ms = []
    for _ in range(2):
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        t0.record()
        feats = sdf.sdf_build_features(on_gpu)
        t1.record()
        torch.cuda.synchronize()
        ms.append(t0.elapsed_time(t1))
    corners = soup.reshape(-1, 3)
    row = np.ascontiguousarray(corners).view([("", np.float32)] * 3).ravel()
    vmap = feats.vertex_map().cpu().numpy()
    verts = feats.vertices().cpu().numpy()
    assert feats.n_vert == len(np.unique(row)) == len(verts)
    assert np.array_equal(verts[vmap], corners)
    assert min(ms) < 100.0, ms
