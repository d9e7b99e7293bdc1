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
