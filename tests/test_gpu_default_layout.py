"""Handles that chose no shading variant: the layout picked by light and
pixel count gives the monolithic kernel's visibilities and picks bit for bit,
at counts around each line of the rule and at ragged light groups."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [1, 3, 4, 21, 31, 32, 33, 64, 65])
@pytest.mark.parametrize("precision", ["fp16", "bf16", "fp8"])
def test_default_layout_equals_the_monolithic_kernel(L, precision):
    from paper_2506_05930_gb300 import nvc
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    cfg = dict(n_levels=5, n_features=2, log2_table_size=9, base_resolution=4, growth=1.5,
               hidden=(32, 32), n_outputs=L, precision=precision, leaky_slope=0.01)
    plain, chosen = nvc.VisibilityCache(cfg), nvc.VisibilityCache(cfg)
    g = torch.Generator(device="cuda").manual_seed(L)
    p = 0.3 * torch.randn(plain.n_params, device="cuda", generator=g)
    r = np.random.default_rng(L)
    scene = nvc.Scene(np.hstack([r.uniform(0, 1, (L, 3)), r.uniform(0.5, 2.0, (L, 1))]))
    n_max = (4 * sms + 1) * 128
    pos = torch.rand((n_max, 3), device="cuda", generator=g)
    nrm = torch.nn.functional.normalize(torch.randn((n_max, 3), device="cuda", generator=g), dim=1)
    for c in (plain, chosen):
        c.set_params(p)
        if precision == "fp8":
            nvc.nvc_calibrate(c.handle, pos[:512])
    nvc.nvc_set_shade_variant(chosen.handle, 0)
    tol = 2 * max(L - 1, 1) * 2.0 ** -24      # two half-sums against one
    for n in (1, 130, 3 * sms * 128, 3 * sms * 128 + 1, 4 * sms * 128, n_max):
        a = plain.shade(scene, pos[:n], nrm[:n], seed=5, frame=n)
        b = chosen.shade(scene, pos[:n], nrm[:n], seed=5, frame=n)
        assert torch.equal(plain.infer(pos[:n]), chosen.infer(pos[:n]))
        assert torch.equal(a["idx"], b["idx"])
        for k in ("wsum", "radiance"):
            assert torch.all((a[k] - b[k]).abs() <= tol * b[k].abs())
    plain.close()
    chosen.close()
