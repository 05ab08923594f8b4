"""Both steps of the clustered sampler redone from each light's own
contribution, as the kernels that take one light at a time give it: cluster,
member and contribution weight bit for bit, inside the packed contribution's
bounds and outside them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import nvc as O
from oracle import philox as ph


def _inputs(kind, n, L):
    r = np.random.default_rng(n + 31 * L)
    x = np.linspace(0.5, 9.5, n)
    pos = np.stack([x, np.full(n, 4.2), 2.0 + np.sin(x)], 1)
    nrm = np.stack([-np.cos(x), np.zeros(n), np.ones(n)], 1)
    nrm /= np.linalg.norm(nrm, axis=1, keepdims=True)
    pos, nrm = pos.astype(np.float32), nrm.astype(np.float32)
    lights = np.hstack([r.uniform(0, 10, (L, 3)), r.uniform(20, 100, (L, 1))]).astype(np.float32)
    if kind == "odd":      # every way out of the packed bounds, alone and together
        nrm[1::9] *= 1e-30
        nrm[2::9] = 0.0
        pos[3::9, 0] = 3e5
        pos[4::9, 0] = 3e10
        nrm[5::9, 0] = np.nan
        nrm[7::9] *= 1e7
        for q, l in enumerate(lights):
            if q % 11 == 1:
                l[:3] = pos[q % n]
            if q % 11 == 2:
                l[3] = 0.0
            if q % 11 == 5:
                l[:3] = (4e5, 0, 0)
            if q % 11 == 8:
                l[3] = 1e-30
            if q % 11 == 9:
                l[3] = 3e6
    return pos, nrm, lights


@pytest.mark.parametrize("weights", ["sum", "visibility"])
@pytest.mark.parametrize("kind", ["inside", "odd"])
@pytest.mark.parametrize("n,L,k", [(1, 1, 1), (33, 7, 3), (300, 37, 32), (700, 1021, 31), (300, 1025, 8),
                                   (70, 5000, 5)])
def test_cluster_member_and_weight_redone(n, L, k, kind, weights):
    from paper_2506_05930_gb300 import nvc
    pos, nrm, lights = _inputs(kind, n, L)
    P, N = torch.from_numpy(pos).cuda(), torch.from_numpy(nrm).cuda()
    c = []
    for i in range(0, L, 200):
        part = torch.empty((n, min(200, L - i)), device="cuda")
        nvc.nvc_light_weights(nvc.Scene(lights[i:i + 200]), P, N, None, part)
        c.append(part)
    c = torch.cat(c, 1).cpu().numpy()
    r = np.random.default_rng(L)
    assign = r.integers(0, k, L).astype(np.int32)
    if k > 2:
        assign[assign == 1] = 0             # an empty cluster
    off, mem = O.cluster_table(assign, k)
    off, mem = off.astype(np.int64), mem.astype(np.int64)
    vis = r.random((n, k)).astype(np.float32)
    seed, frame, view, first = 77, 5, 1, 3
    ids = first + np.arange(n)
    w = O.cluster_weights(vis, c, off, mem, weights)
    y, _, _ = O.wrs_select(w, ids, seed, frame, view)
    wsum = np.zeros(n, np.float32)
    for t in range(k):
        wsum = wsum + w[:, t]
    words = ph.stream_words(ids, frame, view, ph.TAG_RIS, 8, seed)
    light, W = np.full(n, -1, np.int32), np.zeros(n, np.float32)
    for p in np.nonzero(y >= 0)[0]:
        m = int(off[y[p] + 1] - off[y[p]])
        cand = mem[off[y[p]] + ((words[p, :4].astype(np.uint64) * np.uint64(m)) >> np.uint64(32)).astype(np.int64)]
        cc = c[p, cand]
        j = int(O.integer_pick(cc[None], words[p:p + 1, 4:8])[0])
        if j >= 0:
            light[p], W[p] = cand[j], O.ris_weight(cc, np.int64(j), w[p, y[p]], wsum[p], m)
    got, gw = torch.empty(n, dtype=torch.int32, device="cuda"), torch.empty(n, device="cuda")
    nvc.nvc_sample_clustered(nvc.Scene(lights), nvc.Clusters(assign, k, weights=weights),
                             torch.from_numpy(vis).cuda(), P, N, seed, frame, view, first, light=got,
                             weight=gw)
    assert np.array_equal(got.cpu().numpy(), light)
    assert np.array_equal(gw.cpu().numpy(), W, equal_nan=True)
    assert n < 100 or (light >= 0).mean() > 0.2
