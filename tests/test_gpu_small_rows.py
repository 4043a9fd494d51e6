"""Kernels for few rows at the edges of their shapes: the warp-per-column
CUDA-core projection, the SwiGLU epilogue on 16-row tiles (parallel and
recursive), and the CUDA-core attention's vector loads."""
import numpy as np
import pytest

import oracle.sp_oracle as so
import paper_2608_28099_gb300 as sp
from paper_2608_28099_gb300 import workloads as wl
from gpu_util import GpuRun, compare, oracle_logits
from test_gpu_fusion import hidden_logits
from test_gpu_parity import _attend
from test_gpu_project import run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [(1, 1, 4), (3, 100, 90), (7, 13, 64), (8, 129, 132), (9, 64, 256),
                                   (32, 77, 128), (33, 64, 64)])
def test_cuda_core_projection_of_few_rows(M, N, K):
    # K = 90 (not a multiple of 4) and 33 rows take the tiled kernel
    y, ref = run(M, N, K, 1, M + N + K)
    assert np.max(np.abs(y - ref)) <= 1e-5 * np.max(np.abs(ref)) * max(1.0, np.sqrt(K / 256))


@pytest.mark.parametrize("B,k", [(2, 4), (2, 8), (3, 5), (1, 1)])
def test_swiglu_epilogue_on_sixteen_row_tiles(B, k):
    # 80 gate/up weight tiles: one CTA each, K not split
    sh = wl.Shape(256, 8, 2, 128, 5120, k, 3)
    w = wl.custom(sh, [50, 300, 7][:B], wl.LAYOUT_PAGED, 801 + k, rows_per_seq=True)
    r = GpuRun(w)
    compare(r.logits(), oracle_logits(w), label=f"B={B} k={k}")
    r.close()


def test_swiglu_epilogue_in_the_recursion():
    sh = wl.Shape(256, 8, 2, 128, 5120, 4, 3)
    w = wl.with_fusion(wl.custom(sh, [50, 300, 7], wl.LAYOUT_PAGED, 811))
    r = GpuRun(w, options={sp.SP_OPT_RECURSIVE: 1})
    ref = so.classify_recursive(so.Layer(w.shape, w.weights), w.cache, w.seq_ids, w.hidden)
    compare(hidden_logits(r, w.hidden), ref, label="recursive")
    r.close()


@pytest.mark.parametrize("dtype,dh,page", [(wl.F32, 32, 0), (wl.F32, 128, 16), (wl.BF16, 32, 64),
                                           (wl.BF16, 128, 0), (wl.F32, 64, 32)])
def test_cuda_core_attention_tile_edges(dtype, dh, page):
    shape = wl.Shape(256, 8, 2, dh, 256, 3, 2, kv_dtype=dtype, page_size=page or 16)
    lens = [0, 1, 29, 30, 31, 32, 33, 61, 64, 129]
    w = wl.custom(shape, lens, wl.LAYOUT_PAGED if page else wl.LAYOUT_CONTIGUOUS, 821)
    rng = np.random.default_rng(9)
    q = rng.standard_normal((len(lens), 3, 8, dh)).astype(np.float32)
    kn, vn = (rng.standard_normal((len(lens), 3, 2, dh)).astype(np.float32) for _ in range(2))
    ref = so.attention_step(shape, w.cache, w.seq_ids, *(t.astype(np.float64) for t in (q, kn, vn)))
    out, g = _attend(shape, w, q, kn, vn, 1, split=64)
    np.testing.assert_allclose(out, ref, rtol=1e-4, atol=1e-4)  # fp32 throughout
    if g is not None:
        for b, L in enumerate(lens):
            n = (L + page - 1) // page
            assert np.array_equal(g[b, :n], w.cache.page_table[b, :n]) and np.all(g[b, n:] == -7)
