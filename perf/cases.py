"""The performance cases of this library: what a decoding engine has it do, through the calls of
``paper_2512_11280_b200.Context``, from one sequence to a full batch.

``listed()`` are fixed cases, ``draw(rng)`` gives more from the same ranges.  ``prepare`` makes what an
engine holds before the call (logits of its draft and target model, uniforms, the context with each
sequence's history, output buffers, for some cases a captured CUDA graph), ``run`` makes the calls of one
pass, ``work`` counts the bytes and operations the pass cannot do without, ``tolerance`` says how far two
correct implementations may be apart.

A case:
  call      "round"    decode rounds: K draft steps, then verification with the fused threshold update
            "draft"    the K draft steps of a round
            "verify"   one verification call with the fused threshold update
            "vanilla"  one verification call of vanilla speculative sampling
            "greedy"   a round of greedy decoding: K draft steps that take the argmax, then verification
  B, K, V   sequences, window, vocabulary
  dtype     "bf16" or "fp32" logits
  history   entries of each of a sequence's three lists, which are then full (list_capacity): the state of
            a service that has run for a while.  0: the pass starts from adasd_reset, as a new request does
  rounds    decode rounds of a pass
  adaptive  the entropy stop check ends a sequence's window (on average in the middle of it); else fixed
  graph     the pass is a replay of a captured CUDA graph; else it is issued call by call
  temperature, top_k, top_p   the adjusted distribution (1, 0, 1: off)

Every sampled decision is settled: a uniform is drawn again when it lies within rounding distance of an
edge of the token's share of the cumulative distribution, so that results do not hang on the last bits.
"""
import math

import torch

import paper_2512_11280_b200 as adasd

MARGIN = 3e-6          # distance of a uniform from the edges of its token's share of the distribution
STOP_ENTROPY = 4.0     # T_G of the sequences of an adaptive case, nats


def _case(call, B, K, V, dtype="bf16", history=256, rounds=1, adaptive=False, graph=False, warp=(1.0, 0, 1.0), name=None):
    c = dict(call=call, B=B, K=K, V=V, dtype=dtype, history=history, rounds=rounds, adaptive=adaptive, graph=graph,
             temperature=warp[0], top_k=warp[1], top_p=warp[2])
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one user, a small model with fp32 logits, a new request: the lists fill from empty (workload C1)
        _case("round", 1, 5, 32000, "fp32", history=0, rounds=4, name="single stream fp32"),
        # one user, a large vocabulary, windows ended by the stop check (workload C2)
        _case("round", 1, 8, 128256, history=1024, adaptive=True, name="single stream bf16"),
        # a full service in steady state: adaptive windows, the whole round in one graph (workload C5)
        _case("round", 256, 16, 128256, history=1024, adaptive=True, graph=True, name="adaptive batch"),
        # verification of an ordinary batch (workload C3)
        _case("verify", 32, 8, 128256, name="verify batch"),
        # verification of the largest batch and vocabulary (workload C4)
        _case("verify", 128, 16, 151936, name="verify large"),
        # the draft steps of that batch
        _case("draft", 128, 16, 151936, name="draft large"),
        # the comparison mode on the ordinary batch
        _case("vanilla", 32, 8, 128256, name="vanilla batch"),
        # greedy decoding, the setting most evaluations use
        _case("greedy", 32, 8, 128256, name="greedy batch"),
        # sampling with temperature, top-k and top-p, window of 5
        _case("round", 16, 5, 128256, warp=(0.8, 50, 0.95), name="warped batch"),
        # an engine that hands over fp32 logits
        _case("verify", 16, 5, 128256, "fp32", name="verify fp32"),
        # a vocabulary that is no multiple of anything, rows packed one after the other
        _case("round", 8, 5, 50257, name="odd vocabulary"),
        # long-lived sequences: the KDE sums run over thousands of distances
        _case("verify", 32, 8, 128256, history=16384, name="long history"),
    ]


def draw(rng):
    def log_uniform(a, b):
        return math.exp(rng.uniform(math.log(a), math.log(b)))
    call = rng.choice(["round", "round", "round", "verify", "verify", "draft", "vanilla", "greedy"])
    B, K = int(round(log_uniform(1, 128))), rng.randint(2, 16)
    V = int(log_uniform(8192, 151936))
    pad = rng.choice([64, 64, 64, 8, 1])
    V = V // pad * pad
    dtype = rng.choice(["bf16", "bf16", "bf16", "fp32"])
    history = int(log_uniform(64, 16384))
    fresh = call == "round" and rng.random() < 0.2 and B * K * V < 4e7     # a few rounds of new requests
    adaptive = call == "round" and not fresh and rng.random() < 0.5
    graph = call == "round" and rng.random() < 0.3
    warp = (1.0, 0, 1.0)
    if call != "greedy" and rng.random() < 0.25:
        warp = rng.choice([(0.7, 0, 1.0), (1.0, 40, 1.0), (1.0, 0, 0.9), (0.8, 50, 0.95)])
    c = _case(call, B, K, V, dtype, history=0 if fresh else history, rounds=3 if fresh else 1, adaptive=adaptive,
              graph=graph, warp=warp)
    while c["B"] > 1 and work(c)["bytes"] > 6e8:
        c["B"] = c["B"] * 2 // 3
    return c


# ------------------------------------------------------------------------------------ preparation

def _logits(case, gen, windows):
    """Draft rows [B,K,V] and target rows [B,K+1,V] of one round.  A row is s N(0,1) - ln(rank): peaked
    (s = 4 .. 7, entropies of 1 to 4 nats) or flat (s = 1 .. 2, about 6 nats), the target row the draft row
    plus noise; one position in six is a near-copy.  Adaptive: the row that ends a window is flat, those
    before it are below the threshold."""
    B, K, V = case["B"], case["K"], case["V"]
    dev, dt = "cuda", torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    lnrank = torch.log(torch.randperm(V, generator=gen, device=dev).float() + 1.0)
    u = torch.rand((3, B, K + 1), generator=gen, device=dev)
    flat = u[0] < 0.25
    if windows is not None:
        step = torch.arange(K + 1, device=dev)
        flat = step[None, :] == windows[:, None] - 1
    s = torch.where(flat, 0.3 + 0.7 * u[1], 6.0 + 2.0 * u[1]) if windows is not None else torch.where(flat, 1.0 + u[1], 4.0 + 3.0 * u[1])
    tau = torch.where(u[2] < 1 / 6, 0.01, 0.1 + 1.5 * u[2])
    zd, zt = torch.empty((B, K, V), dtype=dt, device=dev), torch.empty((B, K + 1, V), dtype=dt, device=dev)
    for b in range(B):
        base = torch.randn((K + 1, V), generator=gen, device=dev) * s[b, :, None] - lnrank
        zd[b] = base[:K]
        zt[b] = base + torch.randn((K + 1, V), generator=gen, device=dev) * tau[b, :, None]
    return zd, zt


def _probabilities(z, case):
    """softmax of the adjusted rows in float64."""
    z = z.double() / case["temperature"]
    if 0 < case["top_k"] < z.shape[-1]:
        kth = torch.topk(z, case["top_k"], dim=-1).values[..., -1:]
        z = z.masked_fill(z < kth, -math.inf)
    p = torch.softmax(z, -1)
    if case["top_p"] < 1.0:
        down, order = torch.sort(p, dim=-1, descending=True)
        above = down.cumsum(-1) - down
        p = p.masked_fill(torch.zeros_like(p, dtype=torch.bool).scatter_(-1, order, above >= case["top_p"]), 0.0)
        p = p / p.sum(-1, keepdim=True)
    return p


def _settled(cdfs, gen):
    """A uniform per row (rows of all CDFs alike) that lies well inside a token's share of each CDF: the
    first of 24 draws that does.  Returns the uniforms [n] and the tokens of the first CDF [n]."""
    n = cdfs[0].shape[0]
    u = torch.rand((n, 24), generator=gen, device="cuda").clamp(max=1.0 - 1e-4)
    far = torch.full((n, 24), math.inf, dtype=torch.float64, device="cuda")
    tokens = None
    for c in cdfs:
        at = torch.searchsorted(c, u.double(), right=True).clamp(max=c.shape[1] - 1)
        below = torch.where(at > 0, c.gather(1, (at - 1).clamp(min=0)), torch.zeros_like(u, dtype=torch.float64))
        far = torch.minimum(far, torch.minimum(c.gather(1, at) - u, u - below))
        tokens = at if tokens is None else tokens
    first = torch.where((far > MARGIN).any(1), (far > MARGIN).float().argmax(1), far.argmax(1))[:, None]
    return u.gather(1, first)[:, 0], tokens.gather(1, first)[:, 0]


def _uniforms(case, zd, zt, gen):
    """Uniforms of one round and the draft tokens they give.  Draft and target share theirs, so that the
    tokens agree where the rows nearly do."""
    B, K = case["B"], case["K"]
    f = dict(dtype=torch.float32, device="cuda")
    ut, x = torch.empty((B, K + 1), **f), torch.empty((B, K), dtype=torch.int32, device="cuda")
    ua, ur = torch.rand((B, K), generator=gen, device="cuda"), torch.empty(B, **f)
    for b in range(B):
        p, q = _probabilities(zt[b], case), _probabilities(zd[b], case)
        cp, cq = p.cumsum(-1), q.cumsum(-1)
        ut[b, :K], tok = _settled([cq, cp[:K].contiguous()], gen)
        ut[b, K:], _ = _settled([cp[K:].contiguous()], gen)
        x[b] = tok.int()
        if case["call"] == "vanilla":
            alpha = (p[:K].gather(1, tok[:, None]) / q.gather(1, tok[:, None]))[:, 0].clamp(max=1.0)
            ua[b] = torch.where((ua[b] - alpha).abs() < 1e-4, (ua[b] + 0.01) % 1.0, ua[b])
            reject = (ua[b] >= alpha).nonzero()
            w = int(reject[0]) if len(reject) else K
            r = p[w] if w == K else (p[w] - q[w]).clamp(min=0.0)
            ur[b] = _settled([(r / r.sum()).cumsum(-1)[None, :]], gen)[0][0]
    return ut, ua, ur, x


def prepare(case, seed):
    gen = torch.Generator("cuda").manual_seed(int(seed))
    B, K, V, R, N = case["B"], case["K"], case["V"], case["rounds"], case["history"]
    cpu = torch.Generator().manual_seed(int(seed))
    ctx = adasd.Context(B, V, K, dtype=adasd.ADASD_BF16 if case["dtype"] == "bf16" else adasd.ADASD_FP32,
                        list_capacity=N if N > 0 else R * K + 8)
    ctx.set_warpers(case["temperature"], case["top_k"], case["top_p"])
    if N > 0 and case["call"] in ("round", "verify", "draft"):
        # accepted distances are small, rejected ones large, with some overlap
        LE = torch.full((B, N), STOP_ENTROPY).numpy()
        LA = (0.25 + 0.12 * torch.randn((B, N), generator=cpu)).clamp(0.01, 0.99).numpy()
        LR = (0.65 + 0.15 * torch.randn((B, N), generator=cpu)).clamp(0.01, 0.99).numpy()
        for b in range(B):
            ctx.state_import(b, 0.0, LE[b], LA[b], LR[b])
    windows = torch.randint(1, K + 1, (B,), generator=gen, device="cuda") if case["adaptive"] else None

    i32 = dict(dtype=torch.int32, device="cuda")
    st = dict(case=case, ctx=ctx, rounds=[])
    # one sequence: a step's token goes straight to its place; a batch: steps fill rows of [K,B]
    st["x"] = torch.zeros((B, K), **i32)
    st["tok"] = st["x"].view(K, 1) if B == 1 else torch.zeros((K, B), **i32)
    st["H"] = torch.zeros((K, B), device="cuda")
    st["stop"] = torch.zeros((K, B), dtype=torch.uint8, device="cuda")
    st["active"] = torch.ones(B, dtype=torch.uint8, device="cuda")
    st["dlen"] = torch.zeros(B, **i32)
    st["al"], st["nt"] = torch.zeros((R, B), **i32), torch.zeros((R, B), **i32)
    st["am"] = torch.zeros((B, K + 1), **i32)
    st["alpha"] = torch.zeros((B, K), device="cuda")
    st["rec"] = ctx.new_record()
    for r in range(R):
        zd, zt = _logits(case, gen, windows)
        if case["call"] == "greedy":
            # the candidates a draft model agrees with its target on for a while: its rows are the target's
            # up to a point of the window
            keep = torch.randint(0, K + 1, (B, 1), generator=gen, device="cuda") > torch.arange(K, device="cuda")[None, :]
            zd = torch.where(keep[:, :, None], zt[:, :K], zd)
            ut = ua = ur = x = None
        else:
            ut, ua, ur, x = _uniforms(case, zd, zt, gen)
        if case["call"] in ("verify", "vanilla"):
            st["x"].copy_(x)
        ud = ut[:, :K].T.contiguous() if ut is not None else None
        st["rounds"].append(dict(zd=zd, zt=zt, ut=ut, ua=ua, ur=ur, al=st["al"][r], nt=st["nt"][r],
                                 steps=[(zd[:, k, :], st["H"][k], ud[k] if ud is not None else None, st["tok"][k], st["stop"][k])
                                        for k in range(K)]))
    if case["graph"]:
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _pass(st)
        torch.cuda.synchronize()
        st["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(st["graph"], stream=side):
            st["out"] = _pass(st)
    torch.cuda.synchronize()
    return st


# ------------------------------------------------------------------------------------ the pass

def _pass(st):
    case, ctx, x, dlen = st["case"], st["ctx"], st["x"], st["dlen"]
    call = case["call"]
    if call == "verify":
        r = st["rounds"][0]
        ctx.verify(r["zd"], r["zt"], x, r["ut"], r["ua"], r["al"], r["nt"], record=st["rec"])
        return dict(st["rec"], al=r["al"], nt=r["nt"])
    if call == "vanilla":
        r = st["rounds"][0]
        ctx.vanilla_verify(r["zd"], r["zt"], x, r["ua"], r["ur"], r["al"], r["nt"], alpha_out=st["alpha"])
        return dict(al=r["al"], nt=r["nt"], alpha=st["alpha"])
    if call == "draft":
        for z, H, u, tok, stop in st["rounds"][0]["steps"]:
            ctx.draft_entropy(z, H, u=u, token_out=tok, stop_out=stop)
        return dict(H=st["H"], tok=st["tok"], stop=st["stop"])
    if call == "greedy":
        r = st["rounds"][0]
        for z, H, _, tok, stop in r["steps"]:
            ctx.draft_entropy(z, H, token_out=tok, stop_out=stop)
        if case["B"] > 1:
            x.copy_(st["tok"].T)
        ctx.greedy_verify(r["zt"], x, r["al"], r["nt"], argmax_out=st["am"])
        return dict(H=st["H"], tok=st["tok"], al=r["al"], nt=r["nt"], am=st["am"])
    if case["history"] == 0:
        ctx.reset()
    for r in st["rounds"]:
        if case["adaptive"]:
            dlen.zero_()
            st["active"].fill_(1)
        for z, H, u, tok, stop in r["steps"]:
            if case["adaptive"]:
                ctx.draft_entropy(z, H, u=u, token_out=tok, active=st["active"], stop_out=stop, draft_len=dlen)
            else:
                ctx.draft_entropy(z, H, u=u, token_out=tok, stop_out=stop)
        if case["B"] > 1:
            x.copy_(st["tok"].T)
        ctx.verify(r["zd"], r["zt"], x, r["ut"], r["ua"], r["al"], r["nt"], draft_len=dlen if case["adaptive"] else None,
                   record=st["rec"])
    out = dict(st["rec"], H=st["H"], tok=st["tok"], stop=st["stop"], dlen=dlen, al_rounds=st["al"], nt_rounds=st["nt"])
    if case["history"] == 0:
        out["T_G"], out["nE"], out["nA"], out["nR"] = ctx.get_thresholds()
    return out


def run(st):
    if "graph" in st:
        st["graph"].replay()
        return st["out"]
    return _pass(st)


# ------------------------------------------------------------------------------------ its cost and precision

def work(case):
    """Each needed logit row once (a window that the stop check ends has (K + 1) / 2 steps on average), the
    history's two distance lists once; per row pair two exponentials and one logarithm per logit with the
    handful of multiply-adds around them."""
    B, V, R = case["B"], case["V"], case["rounds"]
    K = (case["K"] + 1) / 2 if case["adaptive"] else case["K"]
    row = V * (2 if case["dtype"] == "bf16" else 4)
    draft, verify = B * K, B * (2 * K + 1)
    rows = {"round": draft + verify, "draft": draft, "verify": verify, "vanilla": verify, "greedy": draft + B * (K + 1)}[case["call"]]
    lists = 8 * B * case["history"] if case["call"] in ("round", "verify") else 0
    return {"bytes": R * (rows * row + lists), "flops": R * rows * V * 6.0}


def tolerance(case):
    """fp32 sums of V terms: 1e-6 of a log-sum-exp or entropy, 2.5e-7 of a divergence; the distance is a
    square root of it and P(A|d) a ratio of Gaussian sums in the distance, which magnify that.  Tokens are
    settled except for a few without a good uniform."""
    return {"rel": 5e-5, "max": 5e-3, "differ": 0.005}
