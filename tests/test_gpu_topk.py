"""Top-k cutoffs by selection: rows where they can go wrong - many equal logits at the cut, large logits
piled into a few of the kernel's groups (neighbouring tokens), fewer finite logits than k, lengths off every
tile - against the k-th largest logit of the row."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return torch


@pytest.mark.parametrize("V,dtype", [(4096, synth.BF16), (4099, synth.FP32), (8200, synth.FP32), (50257, synth.BF16), (128256, synth.BF16)])
@pytest.mark.parametrize("k", [1, 2, 50, 512])
@pytest.mark.parametrize("B", [1, 3, 200])
def test_top_k_keeps_exactly_the_k_largest_and_their_ties(torch, V, dtype, k, B):
    import paper_2512_11280_b200 as adasd
    rng = np.random.default_rng(V + k + B)
    z = rng.normal(size=(B, V)).astype(np.float32) * 2
    kinds = np.arange(B) % 5
    for b in range(B):
        if kinds[b] == 1:
            z[b] = np.round(z[b])                              # ties everywhere
        elif kinds[b] == 2:
            z[b] = np.sort(z[b])[::-1]                         # the large ones side by side
        elif kinds[b] == 3:
            z[b, 7:] = -np.inf                                 # seven finite logits
        elif kinds[b] == 4:
            z[b] = -5.0 + 0.0 * z[b]                           # all equal
    t = torch.tensor(z, device="cuda").to(torch.bfloat16 if dtype == synth.BF16 else torch.float32)
    ctx = adasd.Context(B, V, 1, dtype=adasd.ADASD_BF16 if dtype == synth.BF16 else adasd.ADASD_FP32, list_capacity=8)
    ctx.set_warpers(1.0, k, 1.0)
    H, lse = torch.zeros(B, device="cuda"), torch.zeros(B, device="cuda")
    ctx.draft_entropy(t, H, lse_out=lse)
    f = t.double()
    kth = torch.topk(f, k, dim=-1).values[:, -1:]
    f = f.masked_fill(f < kth, -np.inf)
    want = torch.logsumexp(f, -1)
    q = torch.softmax(f, -1)
    ent = -(q * torch.log(q.clamp(min=1e-300))).sum(-1)
    assert (lse.double() - want).abs().max() < 1e-4 and (H.double() - ent).abs().max() < 1e-4
    assert ctx.status() == 0


# either side of the k where another kernel finds the cutoffs, on rows that keep to 16-byte boundaries and rows that do not
@pytest.mark.parametrize("V,dtype,ks", [(8200, synth.BF16, (64, 65, 200, 201)), (65536, synth.BF16, (200, 201)), (8200, synth.FP32, (448, 449, 512, 513))])
@pytest.mark.parametrize("top_p", [1.0, 0.9])
@pytest.mark.parametrize("B", [2, 250])
def test_every_route_to_a_cutoff_keeps_the_same_tokens(torch, V, dtype, ks, top_p, B):
    import oracle
    import paper_2512_11280_b200 as adasd
    tdt = torch.bfloat16 if dtype == synth.BF16 else torch.float32
    z = (torch.randn(B, V, generator=torch.Generator(device="cuda").manual_seed(V + B), device="cuda") * 2).to(tdt)
    z[1] = z[1].sort(descending=True).values
    off = torch.zeros(B * (V + 1) + 16, dtype=tdt, device="cuda").as_strided((B, V), (V + 1, 1), 1)
    off.copy_(z)
    ctx = adasd.Context(B, V, 1, dtype=dtype, list_capacity=8)
    for k in ks:
        ctx.set_warpers(1.0, k, top_p)
        out = []
        for rows in (z, off):
            H, lse = torch.zeros(B, device="cuda"), torch.zeros(B, device="cuda")
            ctx.draft_entropy(rows, H, lse_out=lse)
            out.append((H, lse))
        assert ctx.status() == 0
        for b in (0, 1, B - 1):
            row = z[b].view(torch.int16).cpu().numpy().view(np.uint16) if dtype == synth.BF16 else z[b].cpu().numpy()
            zw, _, band = oracle.warp(row, 1.0, k, float(np.float32(top_p)), band=5e-7)
            if band:                                           # a top-p decision too close to call
                continue
            o = oracle.draft_step(zw, 0.5, 0.0)
            for H, lse in out:
                assert abs(float(H[b]) - o["H"]) < 1e-4 and abs(float(lse[b]) - o["lse"]) < 1e-4, (k, b)
