"""The one-launch decode of small problems: graphs and batches at the edges of
its phases, against the launch-per-phase path (the same call with the kernel
timing hook on), exactly."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mld():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    import paper_1711_01783_gb300 as m
    return m


def _same(a, b):
    for k in a:
        if a[k] is not None:
            assert np.array_equal(a[k].cpu().numpy(), b[k].cpu().numpy()), k


def _decode(dec, llr, syn, iters, early, soft, timed):
    import torch
    dec.timing(1 if timed else 0)
    before = dec.one_launch_decodes()
    out = dec.decode(llr, syn, iters, early_term=early, want_post=soft)
    torch.cuda.synchronize()
    assert dec.status() == 0
    assert dec.one_launch_decodes() - before == (0 if timed else 1)
    return out


@pytest.mark.parametrize("msg,B", [("f16", 64), ("f16", 7), ("f32", 33)])
def test_many_checks_a_thread_in_the_syndrome_phase(mld, msg, B):
    """Eight checks with edges (rows and columns of a 4 x 3 array of VNs) and
    3000 without: the decode runs in one block of 512 threads, whose warps
    publish their first failures before they read the rest (more than four
    checks a thread).  The edgeless checks of some codewords ask for a 1, so
    those never converge."""
    import torch
    rng = np.random.default_rng(11)
    nv, c = 12, 8
    ev = np.array([[3 * j, 3 * j + 1, 3 * j + 2] for j in range(4)] + [[j, j + 4, j + 8] for j in range(4)],
                  np.int32).reshape(-1)
    ec = np.repeat(np.arange(c), 3).astype(np.int32)
    m = c + 3000
    g = mld.Graph(ev, ec, nv, m)
    x = rng.integers(0, 2, (B, nv))
    syn = np.zeros((B, m), np.uint8)
    for j in range(c):
        syn[:, j] = x[:, ev[3 * j:3 * j + 3]].sum(axis=1) & 1
    syn[::3, c + 17::500] = 1
    llr = ((1 - 2 * x) * 3.0 + rng.normal(0, 2, x.shape)).astype(np.float32)
    llr_d, syn_d = torch.from_numpy(llr).cuda(), torch.from_numpy(syn).cuda()
    dec = mld.Decoder(g, B, msg_dtype=msg)
    for early in (True, False):
        a = _decode(dec, llr_d, syn_d, 25, early, False, False)
        b = _decode(dec, llr_d, syn_d, 25, early, False, True)
        _same(a, b)
        conv = a["converged"].cpu().numpy()
        assert not conv[::3].any() and conv.any()


def _grid_graph(mld, rows, cols):
    """VNs in an array, a check per row and per column (every VN of degree 2)."""
    vn = np.arange(rows * cols, dtype=np.int32).reshape(rows, cols)
    ev = np.concatenate([vn.reshape(-1), vn.T.reshape(-1)])
    ec = np.concatenate([np.repeat(np.arange(rows), cols), rows + np.repeat(np.arange(cols), rows)]).astype(np.int32)
    return mld.Graph(ev, ec, rows * cols, rows + cols)


# 4 checks: one block of 16 warps with 17, 16 and 3 slabs of 8 (more slabs than
# warps, as many, and a share that leaves a warp over); the same with the most
# codewords of the path; 12 checks and 5 slabs of 32
@pytest.mark.parametrize("side,B,W,msg", [(2, 135, 8, "f16"), (2, 128, 8, "f32"), (2, 20, 8, "f16"),
                                          (2, 512, 64, "f16"), (6, 130, 32, "f32")])
@pytest.mark.parametrize("early", [False, True])
def test_batches_of_several_slabs(mld, side, B, W, msg, early):
    """The slabs' variables and checks are spread over all warps."""
    import torch
    rng = np.random.default_rng(side + B)
    g = _grid_graph(mld, side, side)
    llr = torch.from_numpy(rng.normal(0.5, 1.5, (B, g.n_vn)).astype(np.float32)).cuda()
    syn = torch.zeros((B, g.n_cn), dtype=torch.uint8, device="cuda")
    syn[::5, 0] = 1
    dec = mld.Decoder(g, B, msg_dtype=msg, slab_width=W)
    _same(_decode(dec, llr, syn, 11, early, True, False), _decode(dec, llr, syn, 11, early, True, True))


@pytest.mark.parametrize("early", [False, True])
def test_a_wait_that_runs_out_is_reported(mld, early):
    """A decode whose first barrier waits for an arrival that never comes
    (mld_decoder_test_stall) gives up after 2 s: no codeword counts as
    converged, whatever the output arrays held, in device and in host memory;
    the status says so, and later decodes of that decoder give up at once.  A
    new decoder is clean."""
    import time
    import torch
    from synthetic import make_workload
    w = make_workload(0.1, 4096, 8, 3, 4400, beta=0.3)
    g = mld.Graph.from_edges(w.graph)
    y, sig, s = (torch.from_numpy(v).cuda() for v in (w.y, w.sigma, w.s))
    dec = mld.Decoder(g, 8, msg_dtype="f16")
    ref = dec.decode_y(y, sig, s, 30, early_term=early)
    torch.cuda.synchronize()
    assert dec.status() == 0 and ref["converged"].all()

    def call(host):
        n = g.n_vn
        out = dict(bits=torch.zeros((8, n), dtype=torch.uint8), post=None,
                   converged=torch.full((8,), 1, dtype=torch.uint8), iters_used=torch.full((8,), 9, dtype=torch.int32))
        out = {k: v if v is None else (v.numpy() if host else v.cuda()) for k, v in out.items()}
        t0 = time.time()
        if host:
            dec.decode_y(w.y, w.sigma, w.s, 30, early_term=early, out=out)
        else:
            dec.decode_y(y, sig, s, 30, early_term=early, out=out)
        torch.cuda.synchronize()
        assert dec.status() == mld.MLD_ETIMEOUT
        for k in ("converged", "iters_used"):
            assert not np.asarray(out[k] if host else out[k].cpu()).any(), k
        return time.time() - t0

    dec.test_stall(1)
    dt = call(False)
    assert 1.9 < dt < 60, dt
    dec.test_stall(0)
    assert call(False) < 1.5 and call(True) < 1.5
    fresh = mld.Decoder(g, 8, msg_dtype="f16")
    got = fresh.decode_y(y, sig, s, 30, early_term=early)
    torch.cuda.synchronize()
    assert fresh.status() == 0
    _same(ref, got)


@pytest.mark.parametrize("msg", ["f32", "f16"])
@pytest.mark.parametrize("early,soft", [(False, False), (False, True), (True, False), (True, True)])
def test_every_check_shape_in_every_pass(mld, msg, early, soft):
    """Checks of one to six core edges, with and without a degree-1 VN: fixed
    iterations, the decisions-only pass and the soft early-terminated one.
    The channel values are strong enough for some codewords to stop early."""
    import torch
    rng = np.random.default_rng(6)
    nv, ev, ec, c = 160, [], [], 0
    order = np.concatenate([rng.permutation(160) for _ in range(4)]).tolist()
    for _ in range(10):
        for dc in range(1, 7):
            for dd in (0, 1):
                row = []
                while len(row) < dc:
                    v = order.pop(0)
                    (order if v in row else row).append(v)
                ev += row + ([nv] if dd else [])
                ec += [c] * (dc + dd)
                nv += dd
                c += 1
    g = mld.Graph(np.array(ev, np.int32), np.array(ec, np.int32), nv, c)
    B = 21
    x = rng.integers(0, 2, (B, nv)).astype(np.uint8)
    syn = np.zeros((B, c), np.uint8)
    for v, k in zip(ev, ec):
        syn[:, k] ^= x[:, v]
    scale = np.where(np.arange(B) % 2, 1.0, 4.0)[:, None]
    llr = (scale * (1 - 2.0 * x) + rng.normal(0, 1.2, x.shape)).astype(np.float32)
    llr, syn = torch.from_numpy(llr).cuda(), torch.from_numpy(syn).cuda()
    dec = mld.Decoder(g, B, msg_dtype=msg)
    one = _decode(dec, llr, syn, 12, early, soft, False)
    _same(one, _decode(dec, llr, syn, 12, early, soft, True))
    its = one["iters_used"].cpu().numpy()
    assert (its.min() < its.max()) if early else (its == 12).all()


@pytest.mark.parametrize("rate,n,B,msg,W,small", [
    (0.1, 4096, 1, "f32", 0, True), (0.05, 5001, 33, "f32", 0, True), (0.02, 5001, 65, "f16", 0, True),
    (0.1, 4096, 16, "f16", 64, True), (0.05, 3000, 140, "f32", 0, True),
    (0.1, 16384, 16, "f16", 0, True),     # a class of six core edges and a degree-1 VN
    (0.1, 65536, 64, "f16", 0, False),    # past the size limit
])
def test_which_decodes_run_in_one_launch(mld, rate, n, B, msg, W, small):
    import torch
    from synthetic import make_workload
    w = make_workload(rate, n, B, 3, 4200 + B, beta=0.35)
    g = mld.Graph.from_edges(w.graph)
    dec = mld.Decoder(g, B, msg_dtype=msg, slab_width=W)
    dec.decode_y(*(torch.from_numpy(v).cuda() for v in (w.y, w.sigma, w.s)), 3)
    torch.cuda.synchronize()
    assert dec.one_launch_decodes() == (1 if small else 0)


def test_checks_of_seven_core_edges_keep_a_launch_per_phase(mld):
    import torch
    g = _grid_graph(mld, 7, 7)
    dec = mld.Decoder(g, 4)
    dec.decode(torch.ones((4, 49), device="cuda"), torch.zeros((4, 14), dtype=torch.uint8, device="cuda"), 3)
    torch.cuda.synchronize()
    assert dec.one_launch_decodes() == 0 and dec.status() == 0
