"""The two-threads-per-pixel kernel on scattered and neighbouring positions:
its encode reads a scattered warp's rows in x-pairs, and its light chunks run
past the last light.  Bit for bit the one-thread kernel's visibilities and
picks, at odd pixel and light counts, for both table precisions."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _positions(kind, n, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    if kind == "scattered":
        return torch.rand((n, 3), device="cuda", generator=g) * 1.1 - 0.05
    x = torch.linspace(0.0, 1.0, n, device="cuda") * min(1.0, n / 4000)
    p = torch.stack([x, 0.3 + 0.1 * x, 0.5 + 0.02 * torch.sin(9 * x)], 1)
    if kind == "both":                       # some warps either way, and a cell edge
        p[::97] = torch.rand((p[::97].shape[0], 3), device="cuda", generator=g)
        p[0] = 1.0
    return p.contiguous()


@pytest.mark.parametrize("kind", ["scattered", "line", "both"])
@pytest.mark.parametrize("table", ["fp32", "fp16"])
@pytest.mark.parametrize("precision,levels,L,n", [("fp16", 16, 33, 1), ("bf16", 15, 47, 127),
                                                  ("fp16", 9, 130, 129), ("fp16", 16, 256, 3000),
                                                  ("fp8", 16, 65, 1000)])
def test_pair_kernel_equals_the_one_thread_kernel(kind, table, precision, levels, L, n):
    from paper_2506_05930_gb300 import nvc
    cache = nvc.VisibilityCache(dict(n_levels=levels, n_features=2, log2_table_size=11,
                                     base_resolution=4, growth=1.4, hidden=(64, 64), n_outputs=L,
                                     leaky_slope=0.01, precision=precision),
                                table_precision=table)
    g = torch.Generator(device="cuda").manual_seed(L)
    cache.set_params(0.3 * torch.randn(cache.n_params, device="cuda", generator=g))
    pos = _positions(kind, n, seed=n)
    nrm = torch.nn.functional.normalize(torch.randn((n, 3), device="cuda", generator=g), dim=1)
    if precision == "fp8":
        nvc.nvc_calibrate(cache.handle, pos)
    r = np.random.default_rng(L)
    scene = nvc.Scene(np.hstack([r.uniform(0, 1, (L, 3)), r.uniform(0.5, 2.0, (L, 1))]))
    got = []
    for variant in (0, 5):
        nvc.nvc_set_shade_variant(cache.handle, variant)
        w = torch.empty((n, L), device="cuda")
        nvc.nvc_sampler_weights(cache.handle, scene, pos, nrm, w)
        got.append((cache.infer(pos), w, cache.shade(scene, pos, nrm, seed=2, frame=1)))
    (v0, w0, s0), (v5, w5, s5) = got
    assert torch.equal(v0, v5) and torch.equal(w0, w5)
    assert torch.equal(s0["idx"], s5["idx"])
    # two half-sums of positive terms against one sum: the order's rounding
    tol = 2 * (L - 1) * 2.0 ** -24
    for k in ("wsum", "radiance"):
        assert torch.all((s0[k] - s5[k]).abs() <= tol * s0[k].abs())
    cache.close()
