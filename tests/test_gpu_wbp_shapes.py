"""Weighted BP on check shapes and slab widths that the ensemble of rate 0.1 at
width 16 does not have: the other rates, every width, several degree-1 VNs on a
check, checks of 7 to 16 terms.  Forward and gradients against the FP64 oracle
with the tolerances of the float kernels (posteriors 1e-4, gradients 1e-3 in the
norm; the float forward differs from FP64 by about 1e-6 a message)."""
import numpy as np
import pytest
from types import SimpleNamespace

import oracle
from synthetic import make_workload, preset_graph

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def mld():
    import paper_1711_01783_gb300 as m
    return m


def _relnorm(a, b):
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-30)


def _check(mld, g0, L, syn, x, W, T, k, n_types, seed):
    g = mld.Graph(g0.edge_vn, g0.edge_cn, g0.n_vn, g0.n_cn, g0.edge_type)
    dec = mld.Decoder(g, L.shape[0], msg_dtype="f32", slab_width=W)
    w = 1.0 + 0.2 * np.random.default_rng(seed).uniform(-1, 1, (T, n_types))
    llr = torch.from_numpy(L).cuda().requires_grad_(True)
    wt = torch.from_numpy(w.astype(np.float32)).cuda().requires_grad_(True)
    soft = mld.weighted_bp(dec, llr, torch.from_numpy(syn).cuda(), wt, ckpt_k=k)
    y = 1.0 - 2.0 * torch.from_numpy(x.astype(np.float32)).cuda()
    torch.nn.functional.softplus(-y * soft).mean().backward()
    ref = oracle.wbp(g0, L, syn, x, w.astype(np.float32).astype(np.float64))
    np.testing.assert_allclose(soft.detach().cpu().numpy(), ref["post"], rtol=1e-4, atol=1e-4)
    assert _relnorm(wt.grad.cpu().numpy(), ref["dw"]) < 1e-3
    assert _relnorm(llr.grad.cpu().numpy(), ref["dllr"]) < 1e-3


@pytest.mark.parametrize("rate", [0.1, 0.05, 0.02])
@pytest.mark.parametrize("W,B,k", [(8, 5, 2), (16, 20, 4), (32, 3, 1), (64, 66, 5)])
def test_rates_and_widths(mld, rate, W, B, k):
    g0 = preset_graph(rate, 2048, 3)
    w = make_workload(rate, 2048, B, 3, 70 + B, beta=0.5, graph=g0)
    L = (2.0 * w.y.astype(np.float64) / (w.sigma.astype(np.float64)[:, None] ** 2)).astype(np.float32)
    _check(mld, g0, L, w.s, w.x, W, 5, k, 3, W)


def _graph(shapes, per, nv, seed):
    """`per` checks of each shape (core edges, degree-1 VNs), mixed; core VNs of
    degree two and more; edge types 0 (core) and 1 (degree-1)."""
    rng = np.random.default_rng(seed)
    rows = [s for s in shapes for _ in range(per)]
    rng.shuffle(rows)
    total = sum(dc for dc, _ in rows)
    pool = np.concatenate([rng.permutation(nv) for _ in range(-(-total // nv))]).tolist()
    ev, ec, et, n = [], [], [], nv
    for c, (dc, dd) in enumerate(rows):
        row = []
        while len(row) < dc:
            v = pool.pop(0)
            (pool if v in row else row).append(v)
        ev += row + list(range(n, n + dd))
        ec += [c] * (dc + dd)
        et += [0] * dc + [1] * dd
        n += dd
    deg = np.bincount(ev, minlength=n)
    assert (deg[:nv] >= 2).all() and (deg[nv:] == 1).all()
    return SimpleNamespace(n_vn=n, n_cn=len(rows), edge_vn=np.array(ev, np.int32), edge_cn=np.array(ec, np.int32),
                           edge_type=np.array(et, np.uint8))


SHAPES = {
    "several degree-1 VNs": [(4, 2), (3, 3), (2, 2), (5, 1), (1, 2)],
    "seven and eight terms": [(7, 0), (8, 0), (6, 1), (7, 1), (5, 2), (6, 2)],
    "nine to sixteen terms": [(9, 0), (12, 0), (8, 1), (10, 4), (16, 0), (4, 1)],
    # more shapes than the table of one launch holds
    "eighteen shapes": [(d, 0) for d in range(1, 9)] + [(d, 1) for d in range(0, 8)] + [(3, 2), (9, 1)],
}


@pytest.mark.parametrize("name", list(SHAPES))
@pytest.mark.parametrize("W,B,k", [(8, 9, 2), (16, 16, 3), (32, 7, 1), (64, 65, 4)])
def test_check_shapes(mld, name, W, B, k):
    shapes = SHAPES[name]
    per = 12
    nv = sum(dc for dc, _ in shapes) * per // 3
    g0 = _graph(shapes, per, nv, len(name))
    rng = np.random.default_rng(B)
    x = rng.integers(0, 2, (B, g0.n_vn)).astype(np.uint8)
    syn = np.zeros((B, g0.n_cn), np.uint8)
    for v, c in zip(g0.edge_vn, g0.edge_cn):
        syn[:, c] ^= x[:, v]
    L = ((1.0 - 2.0 * x) * 1.0 + rng.normal(0, 1.4, x.shape)).astype(np.float32)
    _check(mld, g0, L, syn, x, W, 4, k, 2, W + 1)
