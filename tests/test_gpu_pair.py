"""The two-CTA (cta_group::2) projection kernel at the edges of its work split:
fewer and more items than CTA pairs, fewer k-blocks than ring stages, ragged
last row tiles, every epilogue, and where the one-CTA kernel runs instead."""
import numpy as np
import pytest

import paper_2608_28099_gb300 as sp
from paper_2608_28099_gb300 import workloads as wl
from gpu_util import GpuRun, compare, oracle_logits
from test_gpu_project import run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [
    # (few k-blocks on few pairs: the one-CTA kernel, at the same edges)
    (65, 256, 64),        # one item, one k-block, half a row tile
    (128, 512, 1024),     # K split over several items
    (257, 256, 448),      # three row tiles, seven k-blocks
    # (the pair kernel)
    (65, 12288, 1280),    # 48 items on 76 pairs, half a row tile, the ring wraps
    (100, 2560, 9728),    # K split over several items
    (257, 4096, 1280),    # three row tiles, one row in the last
    (2500, 1024, 64),     # 80 items on 76 pairs, one k-block each
    (2500, 1024, 128),    # two k-blocks each
    (3001, 2048, 192),    # 192 items: both accumulators reused, ring across items
    (700, 4096, 640),
])
def test_pair_projection(M, N, K):
    y, ref = run(M, N, K, 2, M + N + K)
    # bf16 hi + lo activations: the bound of the other tensor-core shapes
    assert np.max(np.abs(y - ref)) <= 2e-5 * np.max(np.abs(ref)) * max(1.0, np.sqrt(K / 256))


@pytest.mark.parametrize("B,k,precision", [
    (128, 16, 0),  # hi + lo Q/K/V with the rotation, plain 256-row gate/up (SwiGLU) and down
    (110, 31, 3),  # every input plain, 3410 rows: a ragged last tile, rotation on 256-row tiles
    (67, 31, 3),   # the same on one-CTA tiles (2077 rows: fewer items than pairs)
    (67, 31, 1),   # every input hi + lo: SwiGLU on 128-row tiles
])
def test_pair_epilogues(B, k, precision):
    sh = wl.Shape(256, 8, 2, 128, 2048, k, 3)
    lens = np.random.default_rng(B).integers(0, 60, size=B)
    run_ = GpuRun(w := wl.custom(sh, lens, wl.LAYOUT_PAGED, 601 + B, rows_per_seq=True),
                  options={sp.SP_OPT_ACT_PRECISION: precision})
    compare(run_.logits(), oracle_logits(w), label=f"pair B={B} k={k}")
    run_.close()


def test_wait_timeout_is_reported_and_the_handle_recovers():
    # the failure path across the two CTAs: rank 0 of the first pair never loads its
    # first k-block, the MMA and every wait of both CTAs behind it give up after 1 ms,
    # both drain, free TMEM and return; nothing faults
    sh = wl.Shape(2048, 16, 2, 128, 512, 16, 3)
    run_ = GpuRun(w := wl.custom(sh, [20, 130, 64, 5] * 10, wl.LAYOUT_PAGED, 621, rows_per_seq=True))
    torch, h = run_.torch, run_.model.handle
    # output projection: 128-row hi + lo tiles, 40 items of 32 k-blocks
    plan = sp.sp_debug_gemm_plan(640, 2048, 2048, torch.cuda.get_device_properties(0).multi_processor_count, 1)
    assert plan["rows_per_tile"] == 128 and plan["kblocks_per_cta"] >= 20 and not plan["persistent"]
    out = torch.empty((40, 3), device="cuda")
    for _ in range(2):
        sp.sp_set_option(h, sp.SP_OPT_DEBUG_STALL, 1)
        sp.sp_classify(h, torch.cuda.current_stream(), 40, run_.ids, run_.cache.seq_lens, run_.cache.desc,
                       run_.rows, out)
        assert sp.sp_check_status(h) & sp.SP_DEV_TIMEOUT
        compare(run_.logits(), oracle_logits(w), label="after timeout")
    run_.close()


# Which kernel runs: pairs of CTAs from 20 k-blocks an item on, or with more items than
# pairs; below, the cluster's start costs more than it gives
@pytest.mark.parametrize("M,N,K,pair", [
    (128, 4096, 1024, False),   # 64 items of 4 k-blocks
    (128, 1024, 2048, False),   # 64 items of 2
    (256, 6144, 1024, False),   # 48 items of 16
    (300, 4096, 1024, False),   # 48 items of 16
    (100, 2560, 9728, True),    # 70 items of 22
    (640, 4096, 512, True),     # 80 items of 8 on 76 pairs
    (300, 512, 8192, False),    # 72 items of 11
    (128, 5120, 5120, True),    # 60 items of 27
    (16, 2560, 2560, False),    # other row tiles never
])
def test_which_kernel_runs(M, N, K, pair):
    import torch
    from torch.profiler import ProfilerActivity, profile
    p = sp.sp_debug_gemm_plan(M, N, K, torch.cuda.get_device_properties(0).multi_processor_count, 1)
    items = p["m_tiles"] * (p["n_tiles"] // 2) * p["splits"]
    for _ in range(3):  # (a process's first trace can be empty)
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            run(M, N, K, 2, M)
            torch.cuda.synchronize()
        names = " ".join(e.name for e in prof.events())
        if "gemm_" in names:
            break
    else:
        pytest.skip("no CUDA trace in this process (another profiler holds it)")
    assert ("gemm_pair_kernel" in names) == pair, (p, items, names)
