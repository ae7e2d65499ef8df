"""Codewords that have stopped keep their values: each codeword of an
early-terminated decode ends with the bits and posteriors of a fixed-iteration
decode of as many iterations, exactly, whatever its neighbours in the slab
do."""
import numpy as np
import pytest

from synthetic import make_workload, preset_graph

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def mld():
    import paper_1711_01783_gb300 as m
    return m


# fours and eights of lanes that are stopped, live, past the batch and mixed: one
# codeword, five, half a slab and one, all but one of a slab, a second slab of one
@pytest.mark.parametrize("B", [1, 5, 33, 63, 65])
@pytest.mark.parametrize("msg,W", [("f16", 64), ("f32", 32), ("f16", 8)])
@pytest.mark.parametrize("path", ["one_launch", "phases", "plan", "irregular"])
def test_outputs_are_those_of_the_last_iteration(mld, B, msg, W, path):
    rate, n, cap = 0.1, 4096, 25
    g0 = preset_graph(rate, n, 3)
    w = make_workload(rate, n, B, 3, 5100 + B, beta=0.42, graph=g0)
    ev, ec, nv, nc, syn = g0.edge_vn, g0.edge_cn, g0.n_vn, g0.n_cn, w.s
    if path == "irregular":  # the first checks merged in pairs: more than eight terms
        ec = np.where(ec < 400, ec // 2 * 2, ec).astype(np.int32)
        keep = np.unique(ev.astype(np.int64) * nc + ec, return_index=True)[1]
        ev, ec = ev[keep], ec[keep]
        x = w.x.astype(np.int64)
        syn = np.zeros_like(w.s)
        np.bitwise_xor.at(syn.T, ec, x.T[ev].astype(syn.dtype))
    g = mld.Graph(ev, ec, nv, nc)
    y, sig, s = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (w.y, w.sigma, syn))
    dec = mld.Decoder(g, B, msg_dtype=msg, slab_width=W)
    if path == "plan":
        out = mld.Plan([dict(decoder=dec, y=y, sigma=sig, syndrome=s, max_iters=cap)], early_term=True,
                       want_post=True).launch()[0]
    else:
        dec.timing(1 if path == "phases" else 0)
        out = dec.decode_y(y, sig, s, cap, early_term=True, want_post=True)
    torch.cuda.synchronize()
    its = out["iters_used"].cpu().numpy()
    if B > 5:
        assert its.min() < its.max()  # codewords stop at different iterations
    ref = mld.Decoder(g, B, msg_dtype=msg, slab_width=W)
    for l in np.unique(its):
        fixed = ref.decode_y(y, sig, s, int(l), want_post=True)
        torch.cuda.synchronize()
        rows = torch.from_numpy(np.flatnonzero(its == l)).cuda()
        for k in ("bits", "post", "converged"):
            assert torch.equal(out[k][rows], fixed[k][rows]), (k, l)
