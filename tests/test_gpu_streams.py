"""Calls on a stream of their own, several in a row without a wait between them:
there (not on the legacy default stream) the kernels are launched with
programmatic stream serialisation and overlap, so these are the calls in which a
kernel could run ahead of data it needs."""
import numpy as np
import pytest

import oracle.sp_oracle as so
import paper_2608_28099_gb300 as sp
from paper_2608_28099_gb300 import workloads as wl
from gpu_util import GpuRun, compare, rows_tensor

pytestmark = pytest.mark.gpu


def _row_sets(w, n):
    rng = np.random.default_rng(n)
    shape = (len(w.seq_ids), w.shape.k_rows, w.shape.d_model)
    return [wl.f32_to_bf16_bits((0.02 * rng.standard_normal(shape)).astype(np.float32)) for _ in range(n)]


def _classify_in_a_row(w, options=None, repeats=4):
    """Calls over three sets of input rows in turn, each checked."""
    run = GpuRun(w, options=options)
    torch = run.torch
    sets = _row_sets(w, 3)
    ref = [so.classify(so.Layer(w.shape, w.weights), w.cache, w.seq_ids, r) for r in sets]
    dev = [rows_tensor(torch, r) for r in sets]
    B = len(w.seq_ids)
    outs = [torch.empty((B, w.shape.n_classes), device="cuda") for _ in range(3 * repeats)]
    torch.cuda.synchronize()
    st = torch.cuda.Stream()
    for i, o in enumerate(outs):
        sp.sp_classify(run.model.handle, st, B, run.ids, run.cache.seq_lens, run.cache.desc, dev[i % 3], o)
    st.synchronize()
    assert sp.sp_check_status(run.model.handle) == 0, sp.sp_last_error()
    for i, o in enumerate(outs):
        compare(o.double().cpu().numpy(), ref[i % 3], label=f"call {i}")
        assert torch.equal(o, outs[i % 3])
    run.close()


# few short sequences, each whole in one share: the merge kernel has nothing to do;
# then pairs that it merges, and batches merged inside the attention
@pytest.mark.parametrize("lens", [[250], [200] * 4, [252, 0, 3], [300] * 3, [2500, 60], [700] * 12, [40] * 70])
@pytest.mark.parametrize("hq,k", [(4, 4), (6, 16)])
def test_classify(lens, hq, k):
    sh = wl.Shape(256, 2 * hq, 2, 128, 512, k, 3)
    _classify_in_a_row(wl.custom(sh, lens, wl.LAYOUT_PAGED, 900 + len(lens), rows_per_seq=True))
