"""The pooled readout at the edges of its block shapes (row groups, column
chunks, classes per pass) through sp_classify, against the fp64 oracle."""
import numpy as np
import pytest

from paper_2608_28099_gb300 import workloads as wl
from gpu_util import GpuRun, compare, oracle_logits

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,k,d,C,pool,lm_head", [
    (1, 1, 264, 1, wl.POOL_MEAN, False),      # one row: one group, a chunk of 264 of 1024 columns
    (1, 2, 1032, 5, wl.POOL_MEAN, True),      # two groups, eight columns in the last chunk
    (3, 7, 520, 21, wl.POOL_MEAN, False),     # four groups, more classes than one pass
    (2, 32, 256, 17, wl.POOL_LAST, True),     # one pooled row of many, classes past 4 x 4
    (2, 4, 264, 4, wl.POOL_LAST, False),      # one pooled row, one pass of classes: one group
    (2, 4, 1032, 5, wl.POOL_LAST, False),     # one pooled row, two groups by its classes
    (1, 1, 520, 9, wl.POOL_MEAN, True),       # one row, four groups by its classes
    (3, 1, 1032, 300, wl.POOL_MEAN, False),   # the same, many passes
    (160, 5, 128, 3, wl.POOL_MEAN, True),     # one group, rows past four
    (160, 16, 128, 33, wl.POOL_MEAN, False),  # one group, classes past a warp
])
def test_readout_block_shapes(B, k, d, C, pool, lm_head):
    sh = wl.Shape(d, 4, 2, 32, 64, k, C, pool=pool)
    rng = np.random.default_rng(B + k)
    w = wl.custom(sh, rng.integers(0, 40, size=B), wl.LAYOUT_PAGED, 501 + k, rows_per_seq=True,
                  head_bias=not lm_head)
    if lm_head:
        w = wl.with_lm_head(w)
    run = GpuRun(w)
    gpu, ref = run.logits(), oracle_logits(w)
    compare(gpu, ref, label="readout")
    assert np.array_equal(gpu, run.logits())  # counters are clear again, the sum order is fixed
    run.close()


@pytest.mark.parametrize("k,C,pool,groups", [
    (4, 4, wl.POOL_LAST, 1), (4, 5, wl.POOL_LAST, 2), (4, 9, wl.POOL_LAST, 4), (1, 300, wl.POOL_MEAN, 4),
    (4, 2, wl.POOL_MEAN, 4), (2, 2, wl.POOL_MEAN, 2),
])
def test_row_groups_follow_rows_and_classes(k, C, pool, groups):
    """A small batch: as many groups as the pooled rows or the classes can use."""
    import torch
    from torch.profiler import ProfilerActivity, profile
    w = wl.custom(wl.Shape(256, 4, 2, 32, 64, k, C, pool=pool), np.array([5, 9]), wl.LAYOUT_PAGED, 77,
                  rows_per_seq=True)
    run = GpuRun(w)
    for _ in range(3):  # (a process's first trace can be empty)
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            run.logits()
            torch.cuda.synchronize()
        names = " ".join(e.name for e in prof.events())
        if "readout_kernel" in names:
            break
    else:
        pytest.skip("no CUDA trace in this process (another profiler holds it)")
    run.close()
    assert f"readout_kernel<{groups}," in names, names
