"""The calls that a user of the decoder makes, as measurable cases.

A case names one pass through the public entry points: decoding a batch of
codewords of one code, decoding an uneven batch with a captured plan, one
weighted-BP training step, or the multidimensional-reconciliation front end.
``prepare`` makes what a user's program holds before the call (observations,
syndromes, the code's graph, its decoder or plan), ``run`` makes the call,
``exact`` restates it in 64 bits with torch alone.

Codes are the library's seeded MET ensemble at rates 0.1 / 0.05 / 0.02.
Operating points (``beta``, the reconciliation efficiency) are those at which
frames decode: 0.40 sits just under the ensemble's threshold at n = 10^6 and
0.30 decodes short codes too.  A program keeps its code for its whole life, so
graphs are built once per (rate, n).
"""
import functools
import math

import numpy as np
import torch
import torch.utils.checkpoint

import paper_1711_01783_gb300 as mld

D2 = {0.1: 20, 0.05: 22, 0.02: 32}      # type-2 edges per core node, by rate
CAP = {0.1: 100, 0.05: 150, 0.02: 200}  # iterations, by rate
# iterations that early-terminated frames take, by beta (largest of the batch)
TYPICAL = {0.3: 8, 0.4: 30}
LMAX = 25.0


def _decode(name, rate, n, batch, msg, *, iters, early, soft, beta, schedule="flooding", host=False):
    c = dict(kind="decode", rate=rate, n=n, batch=batch, msg=msg, iters=iters, early=early, soft=soft, beta=beta,
             schedule=schedule, host=host)
    return dict(c, name=name) if name else c


def listed():
    return [
        # A latency-bound call: a few short frames of a control channel,
        # stopped at their syndrome match, soft values kept.
        _decode("short_f32_b4_et_soft", 0.1, 4096, 4, "f32", iters=30, early=True, soft=True, beta=0.3),
        # A full slab of short frames at the paper's fixed iteration count.
        _decode("short_f16_b64_fixed", 0.1, 4096, 64, "f16", iters=100, early=False, soft=False, beta=0.3),
        # Mid-length frames, float messages, soft output for post-processing.
        _decode("mid_f32_b16_soft", 0.1, 65536, 16, "f32", iters=50, early=False, soft=True, beta=0.3),
        # The low-rate code (long distance) at an odd length with a ragged batch.
        _decode("lowrate_f16_b37_et", 0.02, 262145, 37, "f16", iters=200, early=True, soft=False, beta=0.3),
        # A raw key block in page-locked host memory, results back in host memory.
        _decode("host_f16_b64_et", 0.05, 262144, 64, "f16", iters=150, early=True, soft=False, beta=0.3, host=True),
        # The paper's mode at the benchmark's size: fixed iterations, no
        # decisions inside the loop.
        _decode("long_f16_b64_fixed", 0.1, 1000000, 64, "f16", iters=100, early=False, soft=False, beta=0.4),
        # The same block stopped codeword by codeword, close to the threshold.
        _decode("long_f16_b64_et", 0.1, 1000000, 64, "f16", iters=100, early=True, soft=False, beta=0.4),
        # The layered schedule, which halves the iterations of such a block.
        _decode("long_f16_b64_layered_et", 0.1, 1000000, 64, "f16", iters=100, early=True, soft=False, beta=0.4,
                schedule="layered"),
        # Float messages at full length with soft output.
        _decode("long_f32_b32_soft", 0.05, 1000000, 32, "f32", iters=30, early=False, soft=True, beta=0.3),
        # Codewords of three rates and three lengths in one captured plan, each
        # with its rate's iteration cap and early termination.
        dict(name="uneven_plan_b96", kind="plan", lengths="65536,262144,1000000", batches="9,16,9,15,6,13,11,12,5",
             msg="f16", beta=0.4),
        # One training step of the weighted decoder: forward, loss, adjoint.
        dict(name="train_f32_b16", kind="train", rate=0.1, n=100000, batch=16, iters=20, ckpt=5, beta=0.4),
        # Bob's and Alice's rotations of a 64-codeword block of raw key.
        dict(name="front_end_64x1e6", kind="front", rows=64, row_len=1000000),
    ]


def draw(rng):
    def log_int(lo, hi):
        return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    kind = rng.choice(["decode"] * 7 + ["plan", "train", "front"])
    if kind == "decode":
        rate = rng.choice([0.1, 0.05, 0.02])
        n = log_int(4096, 1000000)
        msg = rng.choice(["f16", "f32"])
        early = rng.random() < 0.5
        soft = rng.random() < 0.4
        batch = log_int(1, 64)
        schedule = rng.choice(["flooding", "flooding", "flooding", "layered"]) if early else "flooding"
        return _decode(None, rate, n, batch, msg, iters=CAP[rate] if early else rng.choice([20, 50, 100]), early=early,
                       soft=soft, beta=0.3, schedule=schedule, host=rng.random() < 0.15)
    if kind == "plan":
        return dict(kind="plan", lengths="%d,%d" % (log_int(4096, 65536), log_int(65536, 500000)),
                    batches=",".join(str(log_int(1, 32)) for _ in range(6)), msg=rng.choice(["f16", "f32"]), beta=0.3)
    if kind == "train":
        return dict(kind="train", rate=rng.choice([0.1, 0.05, 0.02]), n=log_int(4096, 100000), batch=log_int(1, 16),
                    iters=rng.choice([5, 10, 20]), ckpt=rng.choice([2, 5]), beta=0.4)
    return dict(kind="front", rows=log_int(1, 64), row_len=8 * log_int(512, 125000))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
class Code:
    """One code: the library's graph and its edge list on the GPU."""

    def __init__(self, rate, n):
        ev, ec, et, m = mld.ensemble_edges(rate, n, D2[rate], 2)
        self.n, self.m = n, m
        self.graph = mld.Graph(ev, ec, n, m, et)
        self.ev = torch.from_numpy(ev).cuda().long()
        self.ec = torch.from_numpy(ec).cuda().long()
        self.et = torch.from_numpy(et).cuda().long()

    def syndrome(self, x):
        s = torch.empty((x.shape[0], self.m), dtype=torch.uint8, device="cuda")
        for b in range(x.shape[0]):
            ones = torch.zeros(self.m, dtype=torch.int32, device="cuda")
            ones.index_add_(0, self.ec, x[b].to(torch.int32)[self.ev])
            s[b] = (ones & 1).to(torch.uint8)
        return s


@functools.lru_cache(maxsize=24)
def _code(rate, n):
    return Code(rate, n)


@functools.lru_cache(maxsize=64)
def _sigma(rate, beta):
    """Noise at which rate / C = beta on the binary-input AWGN channel."""
    t, w = np.polynomial.hermite.hermgauss(200)

    def capacity(s):
        z = 2.0 * (1.0 + math.sqrt(2.0) * s * t) / (s * s)
        return 1.0 - float(np.dot(w, np.logaddexp(0.0, -z) / math.log(2.0))) / math.sqrt(math.pi)

    lo, hi = 1e-2, 1e3
    for _ in range(100):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if capacity(mid) > rate / beta else (lo, mid)
    return 0.5 * (lo + hi)


def _frames(code, rate, batch, beta, seed):
    """Bob's bits, his syndrome and Alice's observation of the bits."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    sigma = torch.full((batch,), _sigma(rate, beta), dtype=torch.float32, device="cuda")
    x = torch.randint(0, 2, (batch, code.n), generator=g, dtype=torch.uint8, device="cuda")
    y = torch.randn((batch, code.n), generator=g, dtype=torch.float32, device="cuda")
    y.mul_(sigma[:, None]).add_(1.0 - 2.0 * x.float())
    return x, code.syndrome(x), y, sigma


def _plan_jobs(case):
    """(rate, n, batch) of the plan's jobs: every rate with every length."""
    lengths = [int(v) for v in case["lengths"].split(",")]
    batches = [int(v) for v in case["batches"].split(",")]
    pairs = [(r, n) for r in (0.1, 0.05, 0.02) for n in lengths]
    return [(r, n, b) for (r, n), b in zip(pairs, batches)]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "decode":
        code = _code(case["rate"], case["n"])
        _, syn, y, sigma = _frames(code, case["rate"], case["batch"], case["beta"], seed)
        dec = mld.Decoder(code.graph, case["batch"], msg_dtype=case["msg"], schedule=case["schedule"])
        out = None
        if case["host"]:
            y, syn, sigma = (t.cpu().pin_memory() for t in (y, syn, sigma))
            B, n = y.shape
            out = dict(bits=torch.empty((B, n), dtype=torch.uint8).pin_memory(),
                       post=torch.empty((B, n), dtype=torch.float32).pin_memory() if case["soft"] else None,
                       converged=torch.empty(B, dtype=torch.uint8).pin_memory(),
                       iters_used=torch.empty(B, dtype=torch.int32).pin_memory())
        return dict(case=case, dec=dec, y=y, sigma=sigma, syn=syn, out=out)
    if kind == "plan":
        jobs = []
        for k, (rate, n, batch) in enumerate(_plan_jobs(case)):
            code = _code(rate, n)
            _, syn, y, sigma = _frames(code, rate, batch, case["beta"], seed + 1000003 * k)
            width = next(w for w in (8, 16, 32) if batch <= w)
            dec = mld.Decoder(code.graph, batch, msg_dtype=case["msg"], slab_width=width)
            jobs.append(dict(decoder=dec, y=y, sigma=sigma, syndrome=syn, max_iters=CAP[rate]))
        return dict(case=case, plan=mld.Plan(jobs, early_term=True))
    if kind == "train":
        code = _code(case["rate"], case["n"])
        x, syn, y, sigma = _frames(code, case["rate"], case["batch"], case["beta"], seed)
        g = torch.Generator(device="cuda").manual_seed(seed + 1)
        w = 1.0 + 0.05 * torch.randn((case["iters"], 3), generator=g, device="cuda")
        llr = 2.0 * y / (sigma[:, None] * sigma[:, None])
        dec = mld.Decoder(code.graph, case["batch"], msg_dtype="f32", slab_width=8 if case["batch"] <= 8 else 16)
        return dict(case=case, dec=dec, llr=llr.requires_grad_(True), syn=syn, w=w.requires_grad_(True),
                    sign=1.0 - 2.0 * x.float())
    g = torch.Generator(device="cuda").manual_seed(seed)
    shape = (case["rows"], case["row_len"])
    x = 2.0 * torch.randn(shape, generator=g, device="cuda")
    var = 3.0 + 2.0 * torch.rand((case["rows"],), generator=g, device="cuda")
    y = x + var.sqrt()[:, None] * torch.randn(shape, generator=g, device="cuda")
    bits = torch.randint(0, 2, shape, generator=g, dtype=torch.uint8, device="cuda")
    return dict(case=case, x=x, y=y, bits=bits, var=var)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "decode":
        return state["dec"].decode_y(state["y"], state["sigma"], state["syn"], case["iters"], early_term=case["early"],
                                     want_post=case["soft"], out=state["out"])
    if kind == "plan":
        return state["plan"].launch()
    if kind == "train":
        llr, w = state["llr"], state["w"]
        llr.grad = w.grad = None
        soft = mld.weighted_bp(state["dec"], llr, state["syn"], w, ckpt_k=case["ckpt"])
        loss = torch.nn.functional.softplus(-state["sign"] * soft).mean()
        loss.backward()
        return dict(soft=soft.detach(), loss=loss.detach(), dw=w.grad, dllr=llr.grad)
    alpha, ynorm = mld.md_bob(state["y"], state["bits"])
    llr = mld.md_alice(state["x"], alpha, ynorm, state["var"])
    return dict(alpha=alpha, ynorm=ynorm, llr=llr)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _sizes(rate, n):
    """(edges, checks, core nodes, degree-1 nodes) of the ensemble."""
    nc = round({0.1: 0.20, 0.05: 0.12, 0.02: 0.06}[rate] * n)
    m2 = n - nc
    return int(nc * (2.6 + D2[rate])) + m2, n - round(rate * n), nc, m2


# arithmetic of one edge in one iteration: two evaluations of phi (about ten
# operations each) and the leave-one-out sum
EDGE_FLOPS = 25
ON_CHIP = 160e6  # L2 and shared memory: a larger message state has to pass through HBM


def _decode_work(rate, n, batch, msg, iters, soft, schedule="flooding"):
    e, m, nc, m2 = _sizes(rate, n)
    b = 2 if msg == "f16" else 4
    io = batch * (4.0 * n + m + n + (4.0 * n if soft else 0)) + 8.0 * (e + n)
    state = batch * (b * (e - m2) + 4.0 * nc)
    per_iter = batch * (2.0 * b * (e - m2) + b * m2 + nc * (b + 8.0) + m / 8)
    if schedule == "layered":
        per_iter = batch * (2.0 * b * (e - m2) + 8.0 * (e - m2) + b * m2 + m / 8)
    return io + (per_iter * iters if state > ON_CHIP else 0.0), float(EDGE_FLOPS) * e * batch * iters


def work(case):
    kind = case["kind"]
    if kind == "decode":
        it = case["iters"]
        if case["early"]:
            it = min(it, TYPICAL[case["beta"]])
            it = (it + 1) // 2 if case["schedule"] == "layered" else it
        by, fl = _decode_work(case["rate"], case["n"], case["batch"], case["msg"], it, case["soft"], case["schedule"])
    elif kind == "plan":
        parts = [_decode_work(r, n, b, case["msg"], min(CAP[r], TYPICAL[case["beta"]]), False)
                 for r, n, b in _plan_jobs(case)]
        by, fl = sum(p[0] for p in parts), sum(p[1] for p in parts)
    elif kind == "train":
        e, m, nc, m2 = _sizes(case["rate"], case["n"])
        B, T = case["batch"], case["iters"]
        by = B * (4.0 * 4 * case["n"] + m) + 8.0 * e
        if B * 4.0 * (e - m2) > ON_CHIP / 4:  # the adjoint needs every iteration's messages
            by += B * T * 4.0 * (e - m2) * 2
        fl = 4.0 * EDGE_FLOPS * e * B * T
    else:
        k = float(case["rows"]) * case["row_len"]
        by, fl = k * (4 + 1 + 4 + 0.5 + 4 + 4), k * 36  # y, bits, alpha, |y|, x, llr
    return {"bytes": by, "flops": fl}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
def _phi(x):
    return torch.log1p(2.0 / torch.expm1(x))


class _Bp64:
    """Flooding sum-product on the whole Tanner graph, codewords first.

    Checks are padded to the largest degree; padded terms carry phi = 0 and a
    positive sign, so they leave every other term's message as it is.
    """

    def __init__(self, code):
        order = torch.argsort(code.ec, stable=True)
        self.ev, self.ec, self.et = code.ev[order], code.ec[order], code.et[order]
        deg = torch.bincount(self.ec, minlength=code.m)
        first = torch.cumsum(deg, 0) - deg
        self.dmax = int(deg.max())
        at = torch.arange(len(order), device="cuda") - first[self.ec]
        self.slot = self.ec * self.dmax + at
        self.n, self.m = code.n, code.m
        self.amin = float(np.log1p(2.0 / np.expm1(LMAX)))

    def update(self, total, r, sgn, scale=None):
        """One check update from posteriors and old messages; new messages [B, E]."""
        q = total[:, self.ev] - r
        if scale is not None:
            q = q * scale
        q = q.clamp(-LMAX, LMAX)
        neg = (q < 0).double()
        f = _phi(q.abs().clamp(self.amin, LMAX))
        B = q.shape[0]
        pad = torch.zeros((B, self.m * self.dmax), dtype=torch.float64, device="cuda")
        F = pad.index_copy(1, self.slot, f).view(B, self.m, self.dmax)
        N = torch.zeros_like(pad).index_copy_(1, self.slot, neg).view(B, self.m, self.dmax)
        flip = sgn * (1.0 - 2.0 * (N.sum(2) % 2))
        pre, suf = [None] * self.dmax, [None] * self.dmax
        for i in range(1, self.dmax):
            pre[i] = F[..., i - 1] if i == 1 else pre[i - 1] + F[..., i - 1]
        for i in range(self.dmax - 2, -1, -1):
            suf[i] = F[..., i + 1] if i == self.dmax - 2 else suf[i + 1] + F[..., i + 1]
        o = torch.stack([suf[i] if i == 0 else pre[i] if i == self.dmax - 1 else pre[i] + suf[i]
                         for i in range(self.dmax)], 2).reshape(B, -1)[:, self.slot]
        mag = _phi(o.clamp(self.amin, LMAX)).clamp(max=LMAX)
        return mag * flip[:, self.ec] * (1.0 - 2.0 * neg)

    def totals(self, lch, r):
        return lch.index_add(1, self.ev, r)


def _exact_post(case, seed):
    code = _code(case["rate"], case["n"])
    _, syn, y, sigma = _frames(code, case["rate"], case["batch"], case["beta"], seed)
    bp = _Bp64(code)
    post = torch.empty(y.shape, dtype=torch.float64, device="cuda")
    step = max(1, int(1.5e8 // len(bp.ev)))
    for b in range(0, y.shape[0], step):
        s = sigma[b:b + step, None].double()
        lch = (2.0 * y[b:b + step].double() / (s * s)).clamp(-LMAX, LMAX)
        sgn = 1.0 - 2.0 * syn[b:b + step].double()
        r = torch.zeros((lch.shape[0], len(bp.ev)), dtype=torch.float64, device="cuda")
        total = lch
        for _ in range(case["iters"]):
            r = bp.update(total, r, sgn)
            total = bp.totals(lch, r)
        post[b:b + step] = total
    return dict(bits=None, post=post, converged=None, iters_used=None)


def _exact_train(case, seed):
    state = prepare(case, seed)
    bp = _Bp64(_code(case["rate"], case["n"]))
    llr = state["llr"].detach().double().requires_grad_(True)
    w = state["w"].detach().double().requires_grad_(True)
    sgn = 1.0 - 2.0 * state["syn"].double()

    def iterate(lch, total, r, row):
        r = bp.update(total, r, sgn, row[bp.et])
        return bp.totals(lch, r), r

    lch = llr.clamp(-LMAX, LMAX)
    total, r = lch, torch.zeros((llr.shape[0], len(bp.ev)), dtype=torch.float64, device="cuda")
    for t in range(case["iters"]):
        total, r = torch.utils.checkpoint.checkpoint(iterate, lch, total, r, w[t], use_reentrant=False)
    loss = torch.nn.functional.softplus(-state["sign"].double() * total).mean()
    loss.backward()
    return dict(soft=total.detach(), loss=loss.detach(), dw=w.grad, dllr=llr.grad)


def _octonions():
    """Signed permutations of left multiplication by the basis octonions:
    (A_i x)_k = sign[i, k] x[src[i, k]], by Cayley-Dickson doubling
    (a, b)(c, d) = (ac - conj(d) b, da + b conj(c))."""
    def mul(a, b):
        if len(a) == 1:
            return a * b
        h = len(a) // 2

        def conj(v):
            return np.concatenate([v[:1], -v[1:]])

        p, q, r, s = a[:h], a[h:], b[:h], b[h:]
        return np.concatenate([mul(p, r) - mul(conj(s), q), mul(s, p) + mul(q, conj(r))])

    eye = np.eye(8)
    a = np.stack([np.stack([mul(eye[i], eye[j]) for j in range(8)], 1) for i in range(8)])  # [i, k, j]
    src = np.abs(a).argmax(2)
    return src, np.take_along_axis(a, src[..., None], 2)[..., 0]


def _exact_front(case, seed):
    state = prepare(case, seed)
    src, sign = _octonions()
    y = state["y"].double().view(-1, 8)
    u = (1.0 - 2.0 * state["bits"].double().view(-1, 8)) / math.sqrt(8.0)
    norm = y.square().sum(1).sqrt()
    unit = y / norm[:, None]
    alpha = torch.stack([sum(float(sign[i, k]) * unit[:, int(src[i, k])] * u[:, k] for k in range(8))
                         for i in range(8)], 1)
    x = state["x"].double().view(-1, 8)
    mx = torch.stack([sum(float(sign[i, k]) * x[:, int(src[i, k])] * alpha[:, i] for i in range(8))
                      for k in range(8)], 1)
    shape = (case["rows"], case["row_len"])
    ynorm = norm.view(shape[0], -1)
    llr = mx.view(shape[0], -1, 8) * (2.0 * ynorm / (math.sqrt(8.0) * state["var"].double()[:, None]))[..., None]
    return dict(alpha=alpha.view(shape), ynorm=ynorm, llr=llr.reshape(shape))


def exact(case, seed):
    """64-bit outputs, or None where there is no floating output or no time
    (early termination is left out: its posteriors are those of each frame's
    own last iteration)."""
    if case["kind"] == "front":
        return _exact_front(case, seed)
    if case["kind"] == "train":
        return _exact_train(case, seed)
    if case["kind"] != "decode" or not case["soft"] or case["early"] or case["msg"] != "f32":
        return None
    if case["batch"] * case["n"] * case["iters"] > 1.2e9:
        return None
    return _exact_post(case, seed)
