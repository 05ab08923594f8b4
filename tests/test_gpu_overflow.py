"""A last hidden unit whose 16-bit activation overflows to infinity gives
infinite logits and saturated visibilities; the accumulator's padding columns
(zero weights) then hold 0 x infinity.  They must not reach the results:
radiance, picks and sums stay finite at every light count and in every
layout."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U = 2.0 ** -24


@pytest.mark.parametrize("precision,big", [("fp16", 6e4), ("bf16", 3e38)])
@pytest.mark.parametrize("L", [1, 3, 4, 18, 21, 32, 33, 47, 64, 130, 250])
def test_padding_columns_stay_out_of_the_radiance(L, precision, big):
    from paper_2506_05930_gb300 import nvc
    n = 1500
    cache = nvc.VisibilityCache(dict(n_levels=4, n_features=2, log2_table_size=9, base_resolution=4,
                                     growth=1.5, hidden=(32, 32), n_outputs=L, leaky_slope=0.01,
                                     precision=precision))
    g = torch.Generator(device="cuda").manual_seed(L)
    p = torch.randn(cache.n_params, device="cuda", generator=g)
    w0 = 4 * 512 * 2
    w1, w2 = w0 + 32 * 8, w0 + 32 * 8 + 32 * 32
    p[w0:w1] *= 0.5
    p[w1:w2] *= 0.2
    p[w1 + 5 * 32:w1 + 6 * 32] = big           # unit 5 of the last hidden layer
    p[w2:] *= 0.2
    cache.set_params(p)
    pos = torch.rand((n, 3), device="cuda", generator=g)
    nrm = torch.nn.functional.normalize(torch.randn((n, 3), device="cuda", generator=g), dim=1)
    r = np.random.default_rng(L)
    lights = np.hstack([r.uniform(0, 1, (L, 3)), r.uniform(0.5, 2.0, (L, 1))]).astype(np.float32)
    scene = nvc.Scene(lights)
    vis = cache.infer(pos)
    assert torch.isfinite(vis).all()
    assert ((vis == 0) | (vis == 1)).all(1).sum() > n // 4       # the overflowed pixels
    c = torch.empty((n, L), device="cuda")
    nvc.nvc_light_weights(scene, pos, nrm, None, c)
    ref = (vis.double() * c.double()).sum(1)
    # the fused contribution is within 30 u of the normal-incidence value S of
    # the rounded one; L fused multiply-adds (and one sum of halves) follow
    d2 = ((torch.from_numpy(lights).cuda().double()[None, :, :3] - pos.double()[:, None]) ** 2).sum(-1)
    S = torch.from_numpy(lights).cuda().double()[:, 3] / (np.pi * d2.clamp(min=1e-6))
    tol = 31 * U * S.sum(1) + (L + 2) * U * ref
    got = {}
    for variant in (None, 0, 1, 2, 3, 4, 5, 6, 7):
        if L > 32 and variant not in (None, 0, 5):
            continue
        if variant is not None:
            nvc.nvc_set_shade_variant(cache.handle, variant)
        out = got[variant] = cache.shade(scene, pos, nrm, seed=3, frame=1)
        assert torch.isfinite(out["radiance"]).all() and torch.isfinite(out["wsum"]).all(), variant
        assert torch.all((out["radiance"].double() - ref).abs() <= tol), variant
        assert torch.equal(out["idx"], got[None]["idx"]), variant
    for variant, out in got.items():
        if variant not in (None, 0, 5):
            for k in ("radiance", "wsum", "pdf"):
                assert torch.equal(out[k], got[0][k]), (variant, k)
    cache.close()


@pytest.mark.parametrize("precision", ["fp16", "bf16"])
@pytest.mark.parametrize("L", [1, 21, 47])
def test_padding_rows_follow_the_training_step(L, precision):
    """The weight image after a step, padding included, is the one that a new
    handle makes from the same parameters: equal results bit for bit, with two
    units of the last hidden layer overflowing, whose weights the step changes."""
    from paper_2506_05930_gb300 import nvc
    n, big = 700, 6e4 if precision == "fp16" else 3e38
    cfg = dict(n_levels=4, n_features=2, log2_table_size=9, base_resolution=4, growth=1.5,
               hidden=(32, 32), n_outputs=L, leaky_slope=0.01, precision=precision,
               batch_positions=256, lr=0.05)
    a, b = nvc.VisibilityCache(cfg), nvc.VisibilityCache(cfg)
    g = torch.Generator(device="cuda").manual_seed(L)
    p = 0.3 * torch.randn(a.n_params, device="cuda", generator=g)
    a.set_params(p)
    r = np.random.default_rng(L)
    scene = nvc.Scene(np.hstack([r.uniform(0, 1, (L, 3)), r.uniform(0.5, 2.0, (L, 1))]),
                      np.array([[0.5, 0.5, 0.5, 0.3]]))
    for frame in range(3):
        a.train_step(scene, None, seed=1, frame=frame)
    assert a.counters()["step"] == 3
    q = torch.empty_like(p)
    nvc.nvc_get_state(a.handle, q)
    assert not torch.equal(p[-L * 32:], q[-L * 32:])
    b.set_params(q)
    pos = torch.rand((n, 3), device="cuda", generator=g)
    nrm = torch.nn.functional.normalize(torch.randn((n, 3), device="cuda", generator=g), dim=1)
    for variant in (0, 5) + ((6,) if L <= 32 else ()):
        outs = []
        for c in (a, b):
            nvc.nvc_set_shade_variant(c.handle, variant)
            outs.append(c.shade(scene, pos, nrm, seed=3, frame=1))
        for k in ("idx", "pdf", "wsum", "radiance"):
            assert torch.equal(outs[0][k], outs[1][k]), (variant, k)
    # one step from overflowing weights: +-infinite logits, a finite radiance
    w1 = 4 * 512 * 2 + 32 * 8
    q[w1 + 5 * 32:w1 + 6 * 32] = big
    a.set_params(q)
    a.train_step(scene, None, seed=1, frame=9)
    out = a.shade(scene, pos, nrm, seed=3, frame=1)
    assert torch.isfinite(a.infer(pos)).all() and torch.isfinite(out["radiance"]).all()
    a.close()
    b.close()
