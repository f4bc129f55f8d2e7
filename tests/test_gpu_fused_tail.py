"""The fused recompute call with a handful of live keys, which the merge kernel attends itself (at most 8 per sequence) instead
of a streaming launch: around that limit, ragged batches, and windows that hide some or all of the recomputed keys.  Against
the oracle and the two-call path, with the tolerance of the other fused tests."""
import dataclasses

import pytest

from kvd_synth import GEMMA3_4B_GLOBAL, GEMMA3_4B_LOCAL, QWEN3_4B
from test_gpu_fused import attn_check, run_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [GEMMA3_4B_GLOBAL, QWEN3_4B], ids=lambda s: s.name)
@pytest.mark.parametrize("n_old,n_live", [([300], 1), ([300], 6), ([300], 7), ([300], 8), ([1, 700, 0], 3), ([260] * 20, 2)])
def test_live_keys_around_what_the_merge_kernel_takes(shape, n_old, n_live):
    fused, two, ref = run_case(shape, n_old, n_live, seed=n_live)
    attn_check(fused, ref, "fused vs oracle")
    attn_check(fused, two, "fused vs two-call")


@pytest.mark.parametrize("window", [1, 2, 4, 5, 300])  # n_live + 1 = 4 live keys: some of them, all of them, with recomputed ones
def test_windows_over_the_live_keys(window):
    shape = dataclasses.replace(GEMMA3_4B_LOCAL, sliding_window=window)
    fused, two, ref = run_case(shape, [290, 513], 3, seed=window)
    attn_check(fused, ref, "fused vs oracle")
    attn_check(fused, two, "fused vs two-call")
