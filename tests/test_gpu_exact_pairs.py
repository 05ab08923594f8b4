"""The packed light contribution and the warp-wide shadow rays against the
kernels that take one light and one ray at a time: bit for bit, inside the
packed path's bounds and outside them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

L_CHUNK = 200


def _pixels(kind, n, seed):
    r = np.random.default_rng(seed)
    if kind == "line":                      # neighbours on a surface
        x = np.linspace(0.5, 9.5, n)
        pos = np.stack([x, np.full(n, 4.2), 2.0 + np.sin(x)], 1)
        nrm = np.stack([-np.cos(x), np.zeros(n), np.ones(n)], 1)
    else:
        pos, nrm = r.uniform(0, 10, (n, 3)), r.normal(size=(n, 3))
    nrm /= np.linalg.norm(nrm, axis=1, keepdims=True)
    pos, nrm = pos.astype(np.float32), nrm.astype(np.float32)
    if kind == "odd":                       # outside the packed bounds, one way each
        nrm[1 % n] *= 1e-30
        nrm[2 % n] = 0.0
        pos[3 % n] = (3e5, 1.0, 2.0)
        pos[4 % n] = (np.inf, 1.0, 2.0)
        nrm[5 % n] = (np.nan, 0.0, 1.0)
        pos[6 % n] = 0.0
        nrm[7 % n] *= 1e7
    return pos, nrm


def _lights(kind, L, pos, seed):
    r = np.random.default_rng(seed + 100)
    l = np.hstack([r.uniform(0, 10, (L, 3)), r.uniform(20, 100, (L, 1))]).astype(np.float32)
    if kind == "odd":
        l[0, :3] = pos[0]                                   # on a pixel
        l[1 % L, :3] = pos[min(8, len(pos) - 1)] + np.float32(1e-5)
        l[2 % L, 3] = 0.0
        l[3 % L, 3] = -4.0
        l[4 % L, :3] = (4e5, 0, 0)
        l[5 % L, 3] = 1e-30
        l[6 % L, 3] = 3e6
    return l


def _scene(lights, ns, nb, seed):
    from paper_2506_05930_gb300 import nvc
    r = np.random.default_rng(seed + 7)
    sp = np.hstack([r.uniform(0, 10, (ns, 3)), r.uniform(0.1, 0.8, (ns, 1))]).astype(np.float32)
    c, h = r.uniform(0, 10, (nb, 3)), r.uniform(0.05, 0.9, (nb, 3))
    bx = np.hstack([c - h, c + h]).astype(np.float32)
    if ns > 2:
        sp[1, 3] = -sp[1, 3]                # a negative radius blocks like a positive one
    if nb > 2:
        bx[1] = bx[1][[3, 4, 5, 0, 1, 2]]   # corners swapped
        bx[2, 2], bx[2, 5] = -np.inf, np.inf
    return nvc.Scene(lights, sp, bx, (0, 0, 0), (10, 10, 10))


def _per_light(lights, ns, nb, seed, pos, nrm):
    """Contributions and visibilities of every light, a chunk at a time."""
    from paper_2506_05930_gb300 import nvc
    cs, vs = [], []
    for i in range(0, len(lights), L_CHUNK):
        sc = _scene(lights[i:i + L_CHUNK], ns, nb, seed)
        m = min(L_CHUNK, len(lights) - i)
        c, v = torch.empty((len(pos), m), device="cuda"), torch.empty((len(pos), m), device="cuda")
        nvc.nvc_light_weights(sc, pos, nrm, None, c)
        nvc.nvc_trace_visibility(sc, pos, v)
        cs.append(c)
        vs.append(v)
    return torch.cat(cs, 1), torch.cat(vs, 1)


def _same(a, b):
    return torch.equal(torch.nan_to_num(a, nan=-7.0), torch.nan_to_num(b, nan=-7.0))


@pytest.mark.parametrize("kind", ["line", "random", "odd"])
@pytest.mark.parametrize("n,L,ns,nb", [(1, 1, 0, 0), (31, 3, 1, 0), (33, 4, 0, 1), (64, 9, 33, 31),
                                       (1000, 32, 32, 32), (257, 37, 65, 70), (300, 15000, 3, 2)])
def test_exact_di_equals_one_light_at_a_time(kind, n, L, ns, nb):
    from paper_2506_05930_gb300 import nvc
    pos, nrm = _pixels(kind, n, seed=n)
    lights = _lights(kind, L, pos, seed=L)
    P, N = torch.from_numpy(pos).cuda(), torch.from_numpy(nrm).cuda()
    c, v = _per_light(lights, ns, nb, n, P, N)
    ref = torch.zeros(n, device="cuda")
    for i in range(L):
        ref = torch.where((c[:, i] > 0) & (v[:, i] > 0), ref + c[:, i], ref)
    di = torch.empty(n, device="cuda")
    nvc.nvc_exact_di(_scene(lights, ns, nb, n), P, N, di)
    assert _same(di, ref)


@pytest.mark.parametrize("kind", ["line", "odd"])
@pytest.mark.parametrize("n,L,k", [(1, 1, 1), (33, 7, 3), (300, 37, 32), (700, 1021, 31),
                                   (500, 1025, 8), (70, 5000, 5)])
def test_cluster_sums_equal_one_light_at_a_time(kind, n, L, k):
    """The pick follows the clusters' summed contributions: both steps redone
    from each light's own contribution by the stand-alone sampler."""
    from paper_2506_05930_gb300 import nvc
    pos, nrm = _pixels(kind, n, seed=n + 1)
    lights = _lights(kind, L, pos, seed=L)
    lights[:, 3] = np.abs(lights[:, 3])     # a negative sum has no reservoir
    P, N = torch.from_numpy(pos).cuda(), torch.from_numpy(nrm).cuda()
    r = np.random.default_rng(L)
    assign = r.integers(0, k, L)
    if k > 2:
        assign[assign == 1] = 0             # an empty cluster
    c, _ = _per_light(lights, 0, 0, n, P, N)
    vis = torch.rand((n, k), device="cuda")
    w = torch.zeros((n, k), device="cuda")
    for y in range(k):
        s = torch.zeros(n, device="cuda")
        for i in np.nonzero(assign == y)[0]:
            s = s + c[:, i]
        w[:, y] = vis[:, y].clamp(min=0.001) * s
    idx = torch.empty(n, dtype=torch.int32, device="cuda")
    nvc.nvc_wrs_from_weights(w, 77, 5, 1, 3, idx=idx)
    light = torch.empty(n, dtype=torch.int32, device="cuda")
    W = torch.empty(n, device="cuda")
    nvc.nvc_sample_clustered(_scene(lights, 0, 0, n), nvc.Clusters(assign, k), vis, P, N, 77, 5, 1, 3,
                             light=light, weight=W)
    got = torch.from_numpy(assign).cuda()[light.clamp(min=0).long()]
    picked = light >= 0
    assert torch.equal(got[picked], idx.long()[picked])
    assert torch.all((idx[~picked] < 0) | (w.gather(1, idx.clamp(min=0).long().view(-1, 1)).view(-1)[~picked] > 0))
    assert picked.sum() > 0 or n == 1


@pytest.mark.parametrize("n,L", [(64, 9), (200, 32), (40, 250)])
def test_float32_shading_outside_the_packed_bounds(n, L):
    from paper_2506_05930_gb300 import nvc
    pos, nrm = _pixels("odd", n, seed=n)
    lights = _lights("odd", L, pos, seed=L)
    P, N = torch.from_numpy(pos).cuda(), torch.from_numpy(nrm).cuda()
    scene = _scene(lights, 0, 0, n)
    cache = nvc.VisibilityCache(dict(n_levels=2, n_features=2, log2_table_size=8, n_outputs=L,
                                     bounds_max=(10.0, 10.0, 10.0)))
    cache.set_params(0.3 * torch.randn(cache.n_params, device="cuda"))
    out = cache.shade(scene, P, N, seed=4, frame=2, fused=False)
    w, c = torch.empty((n, L), device="cuda"), torch.empty((n, L), device="cuda")
    nvc.nvc_light_weights(scene, P, N, cache.infer(P), c, w)
    idx = torch.empty(n, dtype=torch.int32, device="cuda")
    pdf, wsum = torch.empty(n, device="cuda"), torch.empty(n, device="cuda")
    nvc.nvc_wrs_from_weights(w, 4, 2, idx=idx, pdf=pdf, wsum=wsum)
    assert torch.equal(out["idx"], idx) and _same(out["pdf"], pdf) and _same(out["wsum"], wsum)
    cache.close()
