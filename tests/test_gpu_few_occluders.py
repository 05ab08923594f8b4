"""Shadow rays on both sides of the lines between the kernels for few
occluders and the others (3 spheres + boxes at 36, exact DI at 12 occluders),
bit for bit: the visibilities against the oracle's float32 decisions, and every
call that casts a ray against those visibilities."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import nvc as O

COUNTS = [(0, 0), (1, 0), (0, 1), (2, 1), (6, 6), (12, 0), (13, 0), (0, 12), (0, 13), (0, 36), (0, 37),
          (9, 9), (9, 10), (10, 7), (31, 3), (300, 301)]


def _inputs(ns, nb, n, L, seed):
    r = np.random.default_rng(seed)
    pos = r.uniform(0, 10, (n, 3)).astype(np.float32)
    pos[: n // 2] = np.stack([np.linspace(1, 9, n // 2), np.full(n // 2, 4.0), np.full(n // 2, 2.0)], 1)
    nrm = r.normal(size=(n, 3))
    nrm = (nrm / np.linalg.norm(nrm, axis=1, keepdims=True)).astype(np.float32)
    lights = np.hstack([r.uniform(0, 10, (L, 3)), r.uniform(20, 100, (L, 1))]).astype(np.float32)
    lights[0, 1:3] = (4.0, 2.0)             # segments along x, and along no axis but two
    lights[1, 2] = 2.0
    lights[2, :3] = pos[0]                  # a segment of no length
    sp = np.hstack([r.uniform(0, 10, (ns, 3)), r.uniform(0.1, 1.0, (ns, 1))]).astype(np.float32)
    c, h = r.uniform(0, 10, (nb, 3)), r.uniform(0.05, 0.9, (nb, 3))
    bx = np.hstack([c - h, c + h]).astype(np.float32)
    if nb:
        bx[0] = (3.0, 3.5, 1.0, 3.5, 4.0, 2.0)     # touched by the row of pixels
    if ns > 1:
        sp[1, :3] = pos[3]                  # a pixel inside
    return pos, nrm, lights, sp, bx


@pytest.mark.parametrize("ns,nb", COUNTS)
@pytest.mark.parametrize("n,L", [(70, 5), (600, 9)])
def test_rays_with_few_and_many_occluders(ns, nb, n, L):
    from paper_2506_05930_gb300 import nvc
    pos, nrm, lights, sp, bx = _inputs(ns, nb, n, L, seed=100 * ns + nb)
    scene = nvc.Scene(lights, sp, bx, (0, 0, 0), (10, 10, 10))
    P, N = torch.from_numpy(pos).cuda(), torch.from_numpy(nrm).cuda()
    V = torch.empty((n, L), device="cuda")
    nvc.nvc_trace_visibility(scene, P, V)
    ref = O.visibility(pos, lights, sp, bx, np.float32)
    assert np.array_equal(V.cpu().numpy(), ref.astype(np.float32))
    c = torch.empty((n, L), device="cuda")
    nvc.nvc_light_weights(scene, P, N, None, c)
    rows = torch.arange(n, device="cuda")
    # the all-lights sum
    di, want = torch.empty(n, device="cuda"), torch.zeros(n, device="cuda")
    nvc.nvc_exact_di(scene, P, N, di)
    for i in range(L):
        want = torch.where((c[:, i] > 0) & (V[:, i] > 0), want + c[:, i], want)
    assert torch.equal(di, want)
    # the sampled light's ray, its estimate and the temporal reservoir's
    g = torch.Generator(device="cuda").manual_seed(n)
    idx = torch.randint(0, L, (n,), device="cuda", generator=g, dtype=torch.int32)
    pdf = 0.1 + torch.rand(n, device="cuda", generator=g)
    est = torch.empty(n, device="cuda")
    nvc.nvc_shade_estimate(scene, P, N, idx, pdf, est)
    ci, vi = c[rows, idx.long()], V[rows, idx.long()]
    assert torch.equal(est, torch.where((ci > 0) & (vi > 0), ci / pdf, torch.zeros_like(ci)))
    light, W = torch.empty_like(idx), torch.empty(n, device="cuda")
    nvc.nvc_temporal_merge(scene, P, N, idx, pdf, idx.roll(1), pdf, torch.full_like(idx, 7), 3, 1,
                           light=light, W=W, estimate=est)
    ci, vi = c[rows, light.clamp(min=0).long()], V[rows, light.clamp(min=0).long()]
    assert torch.equal(est, torch.where((light >= 0) & (vi > 0), ci * W, torch.zeros_like(ci)))
    # clustered: targets and both samplers
    assign = (np.arange(L) % 3).astype(np.int32)
    off, mem = O.cluster_table(assign, 3)
    for weights in ("sum", "visibility"):
        cl = nvc.Clusters(assign, 3, weights=weights)
        vis = torch.rand((n, 3), device="cuda", generator=g)
        nvc.nvc_sample_clustered(scene, cl, vis, P, N, 5, 2, light=light, weight=W, estimate=est)
        ci, vi = c[rows, light.clamp(min=0).long()], V[rows, light.clamp(min=0).long()]
        assert torch.equal(est, torch.where((light >= 0) & (vi > 0), ci * W, torch.zeros_like(ci)))
    tgt = torch.empty((n, 3), device="cuda")
    nvc.nvc_cluster_targets(scene, cl, P, 11, 4, tgt)
    want = O.cluster_targets(pos, lights, sp, bx, off, mem, np.arange(n), 11, 4)
    assert np.array_equal(tgt.cpu().numpy(), want.astype(np.float32))
