"""The one-launch sort at the limit of its two-barrier passes, 65536 keys (GPU only): face sorts of 65532
and of exactly 65536 faces (128 tiles either way) give the tables of the launches per pass."""
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


@pytest.mark.parametrize("nu,nv", [(254, 129), (256, 128)])
def test_either_side_of_the_limit(nu, nv, monkeypatch):
    soup = meshgen.torus(nu=nu, nv=nv, seed=3).soup(seed=5)
    on_gpu = torch.from_numpy(soup).cuda()
    monkeypatch.delenv("SDF_RADIX_ONE_LAUNCH", raising=False)
    one = sdf.sdf_build_features(on_gpu)
    monkeypatch.setenv("SDF_RADIX_ONE_LAUNCH", "0")
    per_pass = sdf.sdf_build_features(on_gpu)
    assert one.counts == per_pass.counts
    for table in ("vertex_map", "face_map", "edges", "vertices"):
        assert torch.equal(getattr(one, table)(), getattr(per_pass, table)())
    assert np.array_equal(one.vertices().cpu().numpy()[one.vertex_map().cpu().numpy()], soup.reshape(-1, 3))
    assert one.n_vert == nu * nv
