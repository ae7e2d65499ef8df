"""The loops of an early-terminated plan, split at the caps where the jobs past
them outweigh the others.  Each job gets what a decode of its own gives,
exactly."""
import numpy as np
import pytest

from synthetic import make_workload, preset_graph

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def mld():
    import paper_1711_01783_gb300 as m
    return m


# one job; caps that round up to the same end; odd, even and single iterations;
# a job of no iterations; a second loop for the last job; many caps
@pytest.mark.parametrize("caps", [(7,), (5, 6), (1, 2, 3), (0, 9, 4), (3, 3, 3, 3, 3, 8), tuple(range(1, 24, 2)) + (40,)])
@pytest.mark.parametrize("beta", [0.30, 0.9])
@pytest.mark.parametrize("soft", [False, True])
def test_each_job_equals_its_own_decode(mld, caps, beta, soft):
    g0 = preset_graph(0.1, 1024, 3)
    g = mld.Graph.from_edges(g0)
    jobs, want = [], []
    for k, cap in enumerate(caps):
        msg, B = ("f16", 3 + k) if k % 2 else ("f32", 9)
        w = make_workload(0.1, 1024, B, 3, 960 + k, beta=beta, graph=g0)
        y, sig, s = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (w.y, w.sigma, w.s))
        jobs.append(dict(decoder=mld.Decoder(g, B, msg_dtype=msg), y=y, sigma=sig, syndrome=s, max_iters=cap))
        want.append(mld.Decoder(g, B, msg_dtype=msg).decode_y(y, sig, s, cap, early_term=True, want_post=soft))
    plan = mld.Plan(jobs, early_term=True, want_post=soft)
    for _ in range(2):
        got = plan.launch()
        torch.cuda.synchronize()
        for a, b in zip(want, got):
            for k in ("bits", "converged", "iters_used") + (("post",) if soft else ()):
                assert torch.equal(a[k], b[k]), k
    last = max(int(o["iters_used"].max()) for o in got)
    if beta == 0.9:
        assert last == max(caps)
    # a body is run once at least, and once per two iterations after that
    runs = [plan.launched(i) for i in range(max(caps) + 1)]
    assert runs == sorted(runs) and runs[0] <= plan.launches + 1
    if len(caps) == 1:
        body = plan.launched(4) - plan.launched(2)
        assert plan.launched(max(caps)) == plan.launches + ((max(caps) + 1) // 2 - 1) * body


def test_launches_of_a_fixed_plan(mld):
    g0 = preset_graph(0.1, 1024, 3)
    g = mld.Graph.from_edges(g0)
    w = make_workload(0.1, 1024, 4, 3, 990, beta=0.5, graph=g0)
    y, sig, s = (torch.from_numpy(a).cuda() for a in (w.y, w.sigma, w.s))
    plan = mld.Plan([dict(decoder=mld.Decoder(g, 4), y=y, sigma=sig, syndrome=s, max_iters=6)])
    assert plan.launched(0) == plan.launched(6) == plan.launches
    with pytest.raises(mld.MldError):
        plan.launched(-1)
