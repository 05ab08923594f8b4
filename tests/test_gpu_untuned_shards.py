"""Handles that chose no shading variant: a pixel's results do not depend on
what else is in its launch.  The layouts whose sums are added in another order
must not take turns by pixel count: shards below the lines of the rule, and
views alone, against one launch above them, bit for bit in every output."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

OUTS = ("idx", "pdf", "wsum", "radiance")


@pytest.mark.parametrize("L,precision", [(12, "fp16"), (16, "fp16"), (17, "bf16"), (21, "fp16"),
                                         (32, "fp16"), (32, "fp8"), (33, "fp16"), (40, "bf16"),
                                         (64, "fp16"), (65, "fp16"), (100, "fp8"), (130, "fp16")])
def test_shards_and_views_of_an_untuned_handle(L, precision):
    _check(L, precision, levels=5, log2=9)


@pytest.mark.parametrize("L", [4, 5, 16, 21, 32, 40])
def test_shards_and_views_with_a_large_table(L):
    """More than 2^22 rows: other layouts by default."""
    _check(L, "fp16", levels=9, log2=19)


def _check(L, precision, levels, log2):
    from paper_2506_05930_gb300 import nvc
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    cache = nvc.VisibilityCache(dict(n_levels=levels, n_features=2, log2_table_size=log2,
                                     base_resolution=4, growth=1.5, hidden=(32, 32), n_outputs=L,
                                     precision=precision, leaky_slope=0.01))
    g = torch.Generator(device="cuda").manual_seed(L)
    cache.set_params(0.3 * torch.randn(cache.n_params, device="cuda", generator=g))
    n = 4 * sms * 128 + 1000
    pos = torch.rand((n, 3), device="cuda", generator=g)
    nrm = torch.nn.functional.normalize(torch.randn((n, 3), device="cuda", generator=g), dim=1)
    if precision == "fp8":
        nvc.nvc_calibrate(cache.handle, pos[:512])
    r = np.random.default_rng(L)
    scene = nvc.Scene(np.hstack([r.uniform(0, 1, (L, 3)), r.uniform(0.5, 2.0, (L, 1))]))
    full = cache.shade(scene, pos, nrm, seed=5, frame=7, view=1)
    assert torch.equal(cache.infer(pos), torch.cat([cache.infer(pos[:900]), cache.infer(pos[900:])]))
    cuts = [0, 1, 1001, 1001 + sms * 128 // 2, 1001 + 2 * sms * 128, n]
    parts = [cache.shade(scene, pos[a:b], nrm[a:b], seed=5, frame=7, view=1, pixel_offset=a)
             for a, b in zip(cuts[:-1], cuts[1:])]
    for k in OUTS:
        assert torch.equal(full[k], torch.cat([q[k] for q in parts])), k
    views = [nvc.View(pos[:m], nrm[:m], v, idx=torch.empty(m, dtype=torch.int32, device="cuda"),
                      **{k: torch.empty(m, device="cuda") for k in OUTS[1:]})
             for v, m in ((0, 900), (1, n))]
    nvc.nvc_frame(cache.handle, scene, views, nvc.NO_TRAINING, 5, 7)
    alone = cache.shade(scene, pos[:900], nrm[:900], seed=5, frame=7, view=0)
    for k in OUTS:
        assert torch.equal(getattr(views[0], k), alone[k]), k
        assert torch.equal(getattr(views[1], k), full[k]), k
    cache.close()
