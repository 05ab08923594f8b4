"""The launches a float32 shading call reports: one kernel while the outputs
fit on chip, two for each staged chunk of a network whose outputs do not."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,n,expect", [(32, 5000, 1), (256, 1024, 2), (256, 5000, 10)])
def test_float32_shading_counts_its_launches(L, n, expect):
    from paper_2506_05930_gb300 import nvc
    cache = nvc.VisibilityCache(dict(n_levels=16, n_features=2, log2_table_size=9, base_resolution=4,
                                     growth=1.3, hidden=(64, 64, 64), n_outputs=L))
    nvc.nvc_set_staging(cache.handle, 1024)
    r = np.random.default_rng(L)
    scene = nvc.Scene(np.hstack([r.uniform(0, 1, (L, 3)), r.uniform(0.5, 2.0, (L, 1))]))
    pos = torch.rand((n, 3), device="cuda")
    nvc.nvc_stage_times(cache.handle)            # starts the count again
    cache.shade(scene, pos, pos, seed=1, frame=1, fused=False)
    assert nvc.nvc_stage_times(cache.handle)[1] == expect
    cache.close()
