"""The two-CTA (cta_group::2) projection kernel at the edges of its work split:
fewer and more items than CTA pairs, fewer k-blocks than ring stages, ragged
last row tiles, and every epilogue."""
import numpy as np
import pytest

import paper_2608_28099_gb300 as sp
from paper_2608_28099_gb300 import workloads as wl
from gpu_util import GpuRun, compare, oracle_logits
from test_gpu_project import run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [
    (65, 256, 64),        # one item, one k-block, half a row tile
    (128, 512, 1024),     # K split over several items
    (257, 256, 448),      # three row tiles, seven k-blocks: the ring wraps once
    (2500, 1024, 128),    # 80 items on 76 pairs, two k-blocks each
    (3001, 2048, 192),    # 192 items: both accumulators reused, ring across items
    (700, 4096, 640),
])
def test_pair_projection(M, N, K):
    y, ref = run(M, N, K, 2, M + N + K)
    # bf16 hi + lo activations: the bound of the other tensor-core shapes
    assert np.max(np.abs(y - ref)) <= 2e-5 * np.max(np.abs(ref)) * max(1.0, np.sqrt(K / 256))


@pytest.mark.parametrize("B,k,precision", [
    (128, 16, 0),  # hi + lo Q/K/V with the rotation, plain 256-row gate/up (SwiGLU) and down
    (67, 31, 3),   # every input plain, 2077 rows: a ragged last tile, rotation on 256-row tiles
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
    sh = wl.Shape(256, 8, 2, 128, 512, 4, 3)
    run_ = GpuRun(w := wl.custom(sh, [20, 300, 64, 5] * 6, wl.LAYOUT_PAGED, 621, rows_per_seq=True))
    torch, h = run_.torch, run_.model.handle
    plan = sp.sp_debug_gemm_plan(96, 256, 1024, 152, 1)  # output projection: 128-row hi + lo tiles, eight items
    assert (plan["rows_per_tile"], plan["n_tiles"], plan["persistent"]) == (128, 2, 0)
    out = torch.empty((24, 3), device="cuda")
    for _ in range(2):
        sp.sp_set_option(h, sp.SP_OPT_DEBUG_STALL, 1)
        sp.sp_classify(h, torch.cuda.current_stream(), 24, run_.ids, run_.cache.seq_lens, run_.cache.desc,
                       run_.rows, out)
        assert sp.sp_check_status(h) & sp.SP_DEV_TIMEOUT
        compare(run_.logits(), oracle_logits(w), label="after timeout")
    run_.close()
