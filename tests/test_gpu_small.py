"""Small problems are decoded in one cooperative launch; the same call with the
kernel timing hook on takes the launch-per-phase path.  Both, and the width
that a decoder chooses for a batch, give the same bits, posteriors, flags and
iteration counts, exactly."""
import numpy as np
import pytest

from synthetic import make_workload, preset_graph

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


# batches at the edges of every slab width and past one slab; n = 5001 has
# classes of one to four shapes that end inside a warp, n = 16384 one of seven
# terms; the last case is past the size limit of the one-launch path
@pytest.mark.parametrize("rate,n,B,msg,iters,early,soft", [
    (0.1, 4096, 1, "f32", 12, False, True),
    (0.1, 4096, 9, "f16", 30, True, False),
    (0.05, 5001, 33, "f32", 25, True, True),
    (0.02, 5001, 65, "f16", 40, True, False),
    (0.1, 16384, 16, "f16", 7, False, False),
    (0.05, 3000, 140, "f32", 1, False, True),
    (0.1, 65536, 64, "f16", 5, False, False),
])
def test_one_launch_equals_launch_per_phase(mld, rate, n, B, msg, iters, early, soft):
    import torch
    w = make_workload(rate, n, B, 3, 4200 + B, beta=0.35)
    g = mld.Graph.from_edges(w.graph)
    y, sig, s = (torch.from_numpy(v).cuda() for v in (w.y, w.sigma, w.s))

    def run(width, timed):
        dec = mld.Decoder(g, B, msg_dtype=msg, slab_width=width)
        if timed:
            dec.timing(1)
        out = [dec.decode_y(y, sig, s, iters, early_term=early, want_post=soft) for _ in range(2)]
        torch.cuda.synchronize()
        _same(out[0], out[1])
        if timed:
            assert dec.read_timing()["check_launches"] > 0
        assert dec.status() == 0
        return out[1]

    ref = run(32 if msg == "f32" else 64, True)
    _same(ref, run(0, False))
    _same(ref, run(0, True))
    _same(ref, run(8, False))


def test_all_check_shapes_in_one_launch(mld):
    """Checks of one to six core edges, with and without a degree-1 VN."""
    import torch
    rng = np.random.default_rng(5)
    ev, ec, nv, c = [], [], 60, 0
    core = np.arange(nv)
    for rep in range(12):
        for dc in range(1, 7):
            for dd in (0, 1):
                ev += list(rng.choice(core, dc, replace=False))
                ec += [c] * dc
                if dd:
                    ev.append(nv)
                    ec.append(c)
                    nv += 1
                c += 1
    g = mld.Graph(np.array(ev, np.int32), np.array(ec, np.int32), nv, c)
    B = 21
    llr = torch.from_numpy(rng.normal(0, 2, (B, nv)).astype(np.float32)).cuda()
    syn = torch.from_numpy(rng.integers(0, 2, (B, c)).astype(np.uint8)).cuda()
    for msg in ("f32", "f16"):
        outs = []
        for timed in (False, True):
            dec = mld.Decoder(g, B, msg_dtype=msg)
            if timed:
                dec.timing(1)
            outs.append(dec.decode(llr, syn, 9, want_post=True))
            torch.cuda.synchronize()
        _same(outs[0], outs[1])


def test_concurrent_streams(mld):
    """Decoders on their own threads and streams at the same time: each
    cooperative launch gets its blocks together, whatever else runs."""
    import threading
    import torch
    g0 = preset_graph(0.1, 16384, 3)
    g = mld.Graph.from_edges(g0)
    w = make_workload(0.1, 16384, 16, 3, 4300, beta=0.35, graph=g0)
    y, sig, s = (torch.from_numpy(v).cuda() for v in (w.y, w.sigma, w.s))
    ref = mld.Decoder(g, 16, msg_dtype="f16").decode_y(y, sig, s, 20, early_term=True, want_post=True)
    torch.cuda.synchronize()
    bad = []

    def work():
        try:
            st = torch.cuda.Stream()
            dec = mld.Decoder(g, 16, msg_dtype="f16")
            with torch.cuda.stream(st):
                for _ in range(40):
                    out = dec.decode_y(y, sig, s, 20, early_term=True, want_post=True)
                st.synchronize()
                assert dec.status() == 0
                _same(ref, out)
        except BaseException as e:  # noqa: BLE001 -- reported by the main thread
            bad.append(e)

    threads = [threading.Thread(target=work) for _ in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad, bad
