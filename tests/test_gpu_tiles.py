"""The row kernels at the sizes where their tiling can go wrong: rows that end inside, at and just past a
16-byte unit, an iteration of a warp, a chunk and a warp's share; rows off every 16-byte boundary; a
single sequence and many.  Lockstep against the oracle."""
import pytest

import synth
from tests.test_gpu_parity import run_lockstep

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return torch


@pytest.mark.parametrize("V,dtype", [(1, synth.FP32), (7, synth.BF16), (255, synth.FP32), (2049, synth.BF16), (8191, synth.FP32),
                                     (8200, synth.BF16), (16391, synth.BF16)])
@pytest.mark.parametrize("B", [2, 40])
def test_rounds_at_tile_edges(torch, V, dtype, B):
    """Draft steps, adasd_verify and adasd_vanilla_verify: few rows (short chunks, many segments a row) and
    many, at any alignment."""
    run_lockstep(synth.WORKLOADS["C3"].scaled(name=f"tiles{V}_{B}", B=B, K=3, V=V, dtype=dtype, rounds=3), follow=range(min(B, 6)))
