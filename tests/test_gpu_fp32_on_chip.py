"""The float32 kernels that keep the network on chip, at the edges of their
tiles: 32 pixels or samples a tile, 8- and 32-wide output groups, one or two
activation areas, every feature count."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _scene(L, seed, box=1.0):
    from paper_2506_05930_gb300 import nvc
    r = np.random.default_rng(seed)
    lights = np.hstack([r.uniform(0, box, (L, 3)), r.uniform(0.5, 2.0, (L, 1))])
    spheres = np.hstack([r.uniform(0, box, (5, 3)), r.uniform(0.05, 0.2, (5, 1))])
    return nvc.Scene(lights, spheres, None, (0, 0, 0), (box, box, box))


def _cache(F, levels, hidden, L, seed, **kw):
    from paper_2506_05930_gb300 import nvc
    cache = nvc.VisibilityCache(dict(n_levels=levels, n_features=F, log2_table_size=10,
                                     base_resolution=3, growth=1.5, hidden=hidden, n_outputs=L,
                                     leaky_slope=0.01, **kw))
    g = torch.Generator(device="cuda").manual_seed(seed)
    p = 0.4 * torch.randn(cache.n_params, device="cuda", generator=g)
    cache.set_params(p)
    return cache, p


SHAPES = [(1, 1, (16,), 1), (2, 8, (32, 32), 4), (4, 10, (32, 32), 32), (8, 3, (48, 48), 33),
          (2, 16, (64, 64, 64), 100), (2, 16, (64, 64, 64), 256), (4, 4, (128,), 168),
          (1, 7, (32,) * 8, 8)]


@pytest.mark.parametrize("F,levels,hidden,L", SHAPES)
@pytest.mark.parametrize("n", [1, 31, 33, 5000])
def test_inference_and_shading_equal_the_separate_kernels(F, levels, hidden, L, n):
    """Bit for bit: the same operations in the same order."""
    from paper_2506_05930_gb300 import nvc
    cache, p = _cache(F, levels, hidden, L, seed=n + L)
    scene = _scene(L, seed=L)
    g = torch.Generator(device="cuda").manual_seed(n)
    pos = torch.rand((n, 3), device="cuda", generator=g) * 1.2 - 0.1
    nrm = torch.nn.functional.normalize(torch.randn((n, 3), device="cuda", generator=g), dim=1)
    vis = torch.full((n, L), -1.0, device="cuda")
    ref = torch.empty((n, L), device="cuda")
    nvc.nvc_infer(cache.handle, pos, vis)
    nvc.nvc_infer_noalloc(cache.cfg, p, pos, ref)      # separate encode and MLP kernels
    assert torch.equal(vis, ref)
    odd = torch.full((n * L + 1,), -1.0, device="cuda")[1:].view(n, L)   # 4-byte aligned rows
    nvc.nvc_infer(cache.handle, pos, odd)
    assert torch.equal(odd, ref)
    nvc.nvc_set_staging(cache.handle, 1024)     # the widest networks go through it in chunks
    out = cache.shade(scene, pos, nrm, seed=(3 << 32) + 9, frame=7, view=2, pixel_offset=11, fused=False)
    c, w = torch.empty((n, L), device="cuda"), torch.empty((n, L), device="cuda")
    nvc.nvc_light_weights(scene, pos, nrm, ref, c, w)
    idx = torch.empty(n, dtype=torch.int32, device="cuda")
    pdf, wsum = torch.empty(n, device="cuda"), torch.empty(n, device="cuda")
    nvc.nvc_wrs_from_weights(w, (3 << 32) + 9, 7, 2, 11, idx, pdf, wsum)
    assert torch.equal(out["idx"], idx) and torch.equal(out["pdf"], pdf)
    assert torch.equal(out["wsum"], wsum)
    # L products summed: (L + 1) roundings of at most the sum of magnitudes
    di = (ref.double() * c.double()).sum(1)
    assert torch.all((out["radiance"].double() - di).abs() <= (L + 1) * 2.0 ** -23 * di + 1e-30)
    cache.close()


@pytest.mark.parametrize("F,levels,hidden,L", SHAPES)
@pytest.mark.parametrize("loss", ["l2", "bce"])
@pytest.mark.parametrize("batch", [1, 33, 9000])
def test_training_gradient_equals_the_separate_kernels(F, levels, hidden, L, loss, batch):
    """Against nvc_mlp_forward / nvc_mlp_backward on the same batch with the
    loss gradient formed in float64.  Both sides round every product and add
    the same terms in another order: 1e-5 of the gradient's norm, as the
    oracle comparisons allow."""
    from paper_2506_05930_gb300 import nvc
    if L > 128:
        pytest.skip("this network does not fit on chip: the separate kernels run on both sides")
    cache, p = _cache(F, levels, hidden, L, seed=batch, loss=loss, batch_positions=batch,
                      loss_scale=16.0)
    scene = _scene(L, seed=L + 1)
    grad, loss_out = cache.train_gradient(scene, None, seed=5, frame=3)
    pos = torch.empty((batch, 3), device="cuda")
    y = torch.empty((batch, L), device="cuda")
    nvc.nvc_training_batch(cache.handle, pos, y)
    z = torch.empty((batch, L), device="cuda")
    nvc.nvc_mlp_forward(cache.handle, pos, z)
    z64, y64 = z.double().requires_grad_(True), y.double()
    ref_loss = (torch.nn.functional.binary_cross_entropy_with_logits(z64, y64) if loss == "bce"
                else ((torch.sigmoid(z64) - y64) ** 2).mean())
    dz, = torch.autograd.grad(ref_loss, z64)
    ref = torch.empty(cache.n_params, device="cuda")
    nvc.nvc_mlp_backward(cache.handle, pos, dz.float().contiguous(), ref)
    assert abs(loss_out.item() - ref_loss.item()) <= 1e-6 * abs(ref_loss.item())
    err = (grad.double() - ref.double()).norm().item()
    assert err <= 1e-5 * ref.double().norm().item()
    assert cache.counters()["error_flags"] == 0
    cache.close()
