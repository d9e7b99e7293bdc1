"""Several contexts side by side: what one sets up (limits of a kernel are kept per device, not per context)
leaves the calls of the others as they were."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return torch


# 128256 and 151936: one instantiation of the verify kernel, different shared memory a CTA; the others: neighbours on
# either side
@pytest.mark.parametrize("sizes", [(128256, 151936), (151936, 128256), (8200, 128256, 32000, 151936, 50264)])
@pytest.mark.parametrize("temperature", [1.0, 0.8])
def test_contexts_of_other_vocabularies_leave_a_context_usable(torch, sizes, temperature):
    import paper_2512_11280_b200 as adasd
    B, K = 2, 3

    def verify(ctx, V):
        g = torch.Generator(device="cuda").manual_seed(V)
        zd = (torch.randn(B, K, V, generator=g, device="cuda") * 2).bfloat16()
        zt = (torch.randn(B, K + 1, V, generator=g, device="cuda") * 2).bfloat16()
        i32 = dict(dtype=torch.int32, device="cuda")
        rec = ctx.new_record()
        ctx.verify(zd, zt, torch.zeros((B, K), **i32), torch.rand(B, K + 1, generator=g, device="cuda"),
                   torch.rand(B, K, generator=g, device="cuda"), torch.zeros(B, **i32), torch.zeros(B, **i32), record=rec)
        want = torch.logsumexp(zt.double() / temperature, -1)
        assert (rec["lse_t"].double() - want).abs().max() < 1e-4 and ctx.status() == 0

    ctxs = [adasd.Context(B, V, K, list_capacity=8) for V in sizes]
    for c in ctxs:
        c.set_warpers(temperature, 0, 1.0)
    for _ in range(2):
        for c, V in zip(ctxs, sizes):
            verify(c, V)
    again = adasd.Context(B, sizes[-1], K, list_capacity=8)          # ... and one that comes later
    for c, V in zip(ctxs, sizes):
        verify(c, V)
    again.close()
