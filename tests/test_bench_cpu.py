"""bench.py's own counts, without a GPU."""
import types

import pytest

import bench
import synth


@pytest.mark.parametrize("dtype,V,warpers,draft,rounds", [
    (synth.BF16, 128256, (0.8, 50, 0.95), 2, 3),       # selection, radix for the rest
    (synth.BF16, 128256, (1.0, 0, 0.9), 2, 4),         # histogram, radix
    (synth.BF16, 128256, (1.0, 600, 1.0), 2, 4),
    (synth.BF16, 2000, (1.0, 50, 1.0), 2, 4),
    (synth.FP32, 32000, (1.0, 0, 0.9), 1, 2),          # radix alone
    (synth.FP32, 32000, (1.0, 50, 1.0), 2, 3),
    (synth.FP32, 2000, (1.0, 50, 1.0), 1, 2),
    (synth.BF16, 50257, (1.0, 600, 0.9), 1, 2),
])
def test_cutoff_launches_follow_the_dispatch(dtype, V, warpers, draft, rounds):
    wl = synth.WORKLOADS["C3"].scaled(name="cuts", V=V, dtype=dtype)
    args = types.SimpleNamespace(warpers=warpers)
    assert bench.cuts_on(args, wl)
    assert (bench.cutoff_launches(args, wl, False), bench.cutoff_launches(args, wl, True)) == (draft, rounds)
