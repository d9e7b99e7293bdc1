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
