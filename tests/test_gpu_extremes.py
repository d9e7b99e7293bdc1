"""Rows at the ends of what the calls accept: logits with no probability (masks of the type's lowest value) where
only their order counts."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return torch


@pytest.fixture(scope="module")
def adasd():
    import paper_2512_11280_b200 as m
    m.lib()
    return m


def raw(t, torch):
    return t.view(torch.int16).cpu().numpy().view(np.uint16) if t.dtype == torch.bfloat16 else t.cpu().numpy()


# few rows (short chunks) and many (long ones); on and off 16-byte boundaries
@pytest.mark.parametrize("V,dtype,B", [(64, synth.FP32, 2), (1003, synth.FP32, 40), (8200, synth.BF16, 3), (4099, synth.BF16, 300),
                                       (32000, synth.FP32, 100), (50257, synth.FP32, 40)])
def test_the_largest_logit_is_chosen_however_low_it_is(torch, adasd, V, dtype, B):
    """Argmax drafting and greedy verification choose by the order of the logits alone: rows whose every logit is
    below -1e30, among them rows that are the type's lowest value throughout (first token) or but for a pair of
    equal ones, and rows with -inf beside them; only a row without a finite logit has no choice."""
    tdt = torch.bfloat16 if dtype == synth.BF16 else torch.float32
    low = torch.finfo(tdt).min
    K = 2
    rng = np.random.default_rng(V + B)
    z = torch.tensor(rng.uniform(-3.3e38, -2e30, size=(B, K + 1, V)).astype(np.float32), device="cuda").to(tdt)
    z[0, 0] = low
    z[0, 1] = low
    z[0, 1, [V // 2, V - 1]] = low / 2
    z[0, 2] = -np.inf
    z[1, 0, : V - 1] = -np.inf
    z[1, 0, V - 1] = low
    z[1, 1, 3:] = low
    z[1, 1, :3] = -np.inf
    i32 = dict(dtype=torch.int32, device="cuda")
    ctx = adasd.Context(B, V, K, dtype=dtype, list_capacity=8)
    zh = raw(z, torch)
    want = np.array([[oracle.argmax(zh[b, i]) for i in range(K + 1)] for b in range(B)])
    assert want[0, 0] == 0 and want[0, 1] == V // 2 and want[0, 2] == -1 and want[1, 0] == V - 1 and want[1, 1] == 3
    x = torch.tensor(want[:, :K].astype(np.int32), device="cuda").contiguous()
    al, nt, am = torch.full((B,), -9, **i32), torch.full((B,), -9, **i32), torch.full((B, K + 1), -9, **i32)
    ctx.greedy_verify(z, x, al, nt, argmax_out=am)
    assert ctx.status() == adasd.STATUS_NAN                     # the row without a finite logit
    assert (am.cpu().numpy() == want).all() and (al == K).all() and (nt.cpu().numpy() == want[:, K]).all()
    ctx.greedy_verify(z, x, al, nt, draft_len=torch.full((B,), 1, **i32), argmax_out=am)
    assert ctx.status() == 0
    for i in range(K + 1):
        H, tok = torch.zeros(B, device="cuda"), torch.full((B,), -9, **i32)
        ctx.draft_entropy(z[:, i], H, token_out=tok)            # no uniform: argmax
        assert (tok.cpu().numpy() == want[:, i]).all() and torch.isnan(H).all()
    assert ctx.status() == adasd.STATUS_NAN                     # (such rows have no distribution)


@pytest.mark.parametrize("V,dtype,B,pad", [(64, synth.FP32, 2, 0), (1003, synth.FP32, 3, 1), (32000, synth.FP32, 2, 0), (8200, synth.FP32, 150, 3),
                                           (128256, synth.FP32, 4, 0)])
@pytest.mark.parametrize("offset", [0.0, 300.0, -5000.0])
def test_vanilla_alpha_of_rows_with_a_large_offset(torch, adasd, V, dtype, B, pad, offset):
    """A constant added to a row's logits changes nothing: p(x) / q(x) has to come from differences of logits.  fp32
    logits around an offset o are multiples of ulp(o), exactly as both sides read them; what is left are the
    roundings of (z - m) log2 e and log2 S, of at most 2^5 here: 2 * 2^-19 each of p and q, under 1e-5 of alpha.  Tokens drawn
    from the residual agree with float64 where u lies further than that from an edge."""
    K = 3
    g = torch.Generator(device="cuda").manual_seed(V + B)
    buf_d = torch.empty(B * K * (V + pad) + pad, device="cuda")
    buf_t = torch.empty(B * (K + 1) * (V + pad) + pad, device="cuda")
    zd = buf_d.as_strided((B, K, V), (K * (V + pad), V + pad, 1), pad)
    zt = buf_t.as_strided((B, K + 1, V), ((K + 1) * (V + pad), V + pad, 1), pad)
    zt.copy_(torch.randn(B, K + 1, V, generator=g, device="cuda") * 2 + offset)
    zd.copy_(zt[:, :K] + torch.randn(B, K, V, generator=g, device="cuda") * 0.5)
    x = torch.multinomial(torch.softmax(zd.reshape(-1, V).double(), -1), 1, generator=g).view(B, K).to(torch.int32)
    u, ur = torch.full((B, K), 0.9, device="cuda"), torch.rand(B, generator=g, device="cuda")
    al, nt = torch.zeros(B, dtype=torch.int32, device="cuda"), torch.zeros(B, dtype=torch.int32, device="cuda")
    alpha = torch.zeros(B, K, device="cuda")
    ctx = adasd.Context(B, V, K, dtype=dtype, list_capacity=8)
    ctx.vanilla_verify(zd, zt, x, u, ur, al, nt, alpha_out=alpha)
    p, q = torch.softmax(zt.double(), -1), torch.softmax(zd.double(), -1)
    i = x.long()[..., None]
    want = (p[:, :K].gather(2, i) / q.gather(2, i))[..., 0].clamp(max=1.0)
    assert ctx.status() == 0
    assert (alpha.double() - want).abs().max() < 1e-5
    for b in range(B):
        w = int(al[b])
        r = (p[b, w] - q[b, w]).clamp(min=0) if w < K else p[b, w]
        c = torch.cumsum(r / r.sum(), 0)
        t = int(nt[b])
        assert float(c[t]) > float(ur[b]) - 1e-4 and (t == 0 or float(c[t - 1]) <= float(ur[b]) + 1e-4) and float(r[t]) > 0


# from a segment of several chunks to the most segments a position has (64), bf16 and fp32, on and off 16-byte boundaries
@pytest.mark.parametrize("V,dtype,B,pad", [(600, synth.FP32, 3, 0), (32000, synth.FP32, 1, 0), (32000, synth.FP32, 4, 1), (128256, synth.FP32, 1, 0),
                                           (128256, synth.FP32, 4, 3), (128256, synth.FP32, 16, 0), (128256, synth.BF16, 1, 1),
                                           (128256, synth.BF16, 5, 3), (128256, synth.BF16, 2, 0)])
def test_identical_rows_are_exactly_0_apart(torch, adasd, V, dtype, B, pad):
    """Sec. 4.4: a distance of exactly 0 stays out of the lists, so it has to be exactly 0."""
    K, tdt = 5, torch.bfloat16 if dtype == synth.BF16 else torch.float32
    g = torch.Generator(device="cuda").manual_seed(V + B)

    def rows(n):
        return torch.zeros(B * n * (V + pad) + 16, dtype=tdt, device="cuda").as_strided((B, n, V), (n * (V + pad), V + pad, 1), pad)
    zt, zd = rows(K + 1), rows(K)
    zt.copy_(torch.randn(B, K + 1, V, generator=g, device="cuda") * 2)
    zd.copy_(zt[:, :K])
    i32 = dict(dtype=torch.int32, device="cuda")
    ctx = adasd.Context(B, V, K, dtype=dtype, list_capacity=64)
    for warp in ((1.0, 0, 1.0), (0.7, 0, 0.9)):
        ctx.set_warpers(*warp)
        rec = ctx.new_record()
        ctx.verify(zd, zt, torch.zeros((B, K), **i32), torch.rand(B, K + 1, generator=g, device="cuda"), torch.zeros(B, K, device="cuda"),
                   torch.zeros(B, **i32), torch.zeros(B, **i32), record=rec)
        assert (rec["jsd"] == 0).all() and (rec["dist"] == 0).all() and torch.equal(rec["H_d"], rec["H_t"][:, :K])
    T, nE, nA, nR = ctx.get_thresholds()
    assert int(nA.max()) == 0 and int(nR.max()) == 0 and ctx.status() == 0


@pytest.mark.parametrize("V,dtype,B,pad", [(64, synth.FP32, 2, 0), (1003, synth.FP32, 5, 1), (32000, synth.FP32, 3, 0), (128256, synth.FP32, 2, 1), (5000, synth.BF16, 3, 1),
                                           (8200, synth.BF16, 2, 0), (32000, synth.BF16, 150, 0), (128256, synth.BF16, 3, 0)])
@pytest.mark.parametrize("T", [1e-3, 1e-9, 1e-10])
@pytest.mark.parametrize("mask", ["inf", "lowest"])
def test_temperatures_that_leave_only_the_largest_logits(torch, adasd, V, dtype, B, pad, T, mask):
    """Any positive temperature is accepted: for 1e-9, (z - max) log2 e / T of a masked logit is beyond fp32.  Rows
    whose every other token has no probability; entropies, distances and alphas are those of a few equal logits."""
    K, tdt = 2, torch.bfloat16 if dtype == synth.BF16 else torch.float32
    g = torch.Generator(device="cuda").manual_seed(V + B)

    def rows(n):
        return torch.zeros(B * n * (V + pad) + 16, dtype=tdt, device="cuda").as_strided((B, n, V), (n * (V + pad), V + pad, 1), pad)
    zt, zd = rows(K + 1), rows(K)
    z = torch.randn(B, K + 1, V, generator=g, device="cuda").round(decimals=1) * 8
    z[..., : V // 3] = -np.inf if mask == "inf" else torch.finfo(tdt).min
    zt.copy_(z)
    zd.copy_(z[:, :K])
    zd[:, 1] = zd[:, 1].roll(V // 2, -1)                        # another largest token
    T = float(np.float32(T))
    i32 = dict(dtype=torch.int32, device="cuda")
    ctx = adasd.Context(B, V, K, dtype=dtype, list_capacity=8)
    ctx.set_warpers(T, 0, 1.0)
    p, q = torch.softmax(zt.double() / T, -1), torch.softmax(zd.double() / T, -1)
    ent = lambda w: -(w * torch.log(w.clamp(min=1e-300))).sum(-1)
    H, tok = torch.zeros(B, device="cuda"), torch.zeros(B, **i32)
    lse = torch.zeros(B, device="cuda")
    x = torch.zeros((B, K), **i32)
    for i in range(K):
        ctx.draft_entropy(zd[:, i], H, u=torch.rand(B, generator=g, device="cuda"), token_out=tok, lse_out=lse)
        assert (H.double() - ent(q[:, i])).abs().max() < 1e-4
        want = torch.logsumexp(zd[:, i].double() / T, -1)
        assert ((lse.double() - want) / want.abs().clamp(min=1)).abs().max() < 1e-6
        x[:, i] = tok
    assert (x >= 0).all() and (q.gather(2, x.long()[..., None]) > 0).all()
    rec, al, nt = ctx.new_record(), torch.zeros(B, **i32), torch.zeros(B, **i32)
    ctx.verify(zd, zt, x, torch.rand(B, K + 1, generator=g, device="cuda"), torch.rand(B, K, generator=g, device="cuda"), al, nt, record=rec)
    assert (rec["H_d"].double() - ent(q)).abs().max() < 1e-4 and (rec["H_t"].double() - ent(p)).abs().max() < 1e-4
    m = 0.5 * (p[:, :K] + q)
    assert (rec["jsd"].double() - (ent(m) - 0.5 * (ent(p[:, :K]) + ent(q)))).abs().max() < 1e-4
    assert (rec["dist"][:, 0] == 0).all() and (p.gather(2, rec["y"].long()[..., None]) > 0).all()
    alpha = torch.zeros(B, K, device="cuda")
    ctx.vanilla_verify(zd, zt, x, torch.full((B, K), 0.5, device="cuda"), torch.rand(B, generator=g, device="cuda"), al, nt, alpha_out=alpha)
    want = (p[:, :K].gather(2, x.long()[..., None]) / q.gather(2, x.long()[..., None]))[..., 0].clamp(max=1.0)
    assert (alpha.double() - want).abs().max() < 1e-4
    assert all(float(p[b, int(al[b]), int(nt[b])]) > 0 for b in range(B))
    assert ctx.status() == 0
