"""Calls on a stream of their own, several in a row without a wait between them:
there (not on the legacy default stream) the kernels are launched with
programmatic stream serialisation and overlap, so these are the calls in which a
kernel could run ahead of data it needs."""
import numpy as np
import pytest

import oracle.sp_oracle as so
import paper_2608_28099_gb300 as sp
from paper_2608_28099_gb300 import workloads as wl
from gpu_util import GpuRun, compare, ensure_built, rows_tensor, torch_dev

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


@pytest.mark.parametrize("dh,kv", [(32, wl.BF16), (64, wl.F32), (128, wl.F32)])
def test_classify_with_cuda_core_attention(dh, kv):
    sh = wl.Shape(256, 8, 2, dh, 512, 5, 3, kv_dtype=kv)
    _classify_in_a_row(wl.custom(sh, [250, 31, 0, 700], wl.LAYOUT_CONTIGUOUS, 920 + dh, rows_per_seq=True))


@pytest.mark.parametrize("lens", [[24, 7], [40, 300, 1]])
def test_attend_reads_a_cache_that_the_call_before_it_writes(lens):
    # sp_project writes the fp32 values of a contiguous cache ([tokens][Hkv dh]) in
    # place, sp_attend reads them: other values in every turn
    ensure_built()
    torch = torch_dev()
    hkv, G, dh, k, K = 4, 2, 32, 3, 1024
    N, M = hkv * dh, sum(lens)
    rng = np.random.default_rng(M)
    shape = wl.Shape(256, hkv * G, hkv, dh, 256, k, 2, kv_dtype=wl.F32)
    w = wl.custom(shape, lens, wl.LAYOUT_CONTIGUOUS, 940)
    wbits = wl.f32_to_bf16_bits((0.05 * rng.standard_normal((N, K))).astype(np.float32))
    wt = torch.from_numpy(wbits.view(np.int16)).cuda()
    wf = wl.bf16_bits_to_f32(wbits).astype(np.float64)
    xs = [rng.standard_normal((M, K)).astype(np.float32) for _ in range(3)]
    q = rng.standard_normal((len(lens), k, hkv * G, dh)).astype(np.float32)
    kn, vn = (rng.standard_normal((len(lens), k, hkv, dh)).astype(np.float32) for _ in range(2))
    cache = sp.DeviceCache(w.cache)
    values = cache.v_flat
    assert tuple(values.shape) == (M, hkv, dh) and values.dtype == torch.float32
    refs = []
    for x in xs:
        w.cache.v_flat = (x.astype(np.float64) @ wf.T).reshape(M, hkv, dh).astype(np.float32)
        refs.append(so.attention_step(shape, w.cache, w.seq_ids, *(t.astype(np.float64) for t in (q, kn, vn))))
    dims = sp.sp_attn_dims(hkv * G, hkv, dh, k, sp.SP_F32, max(lens), 0, 0)
    ws = torch.empty(sp.sp_attend_workspace_bytes(dims, len(lens)), dtype=torch.uint8, device="cuda")
    pws = torch.empty(max(256, sp.sp_project_workspace_bytes(M, N, K)), dtype=torch.uint8, device="cuda")
    x_d = [torch.from_numpy(x).cuda() for x in xs]
    q_d, kn_d, vn_d = (torch.from_numpy(t).cuda() for t in (q, kn, vn))
    outs = [torch.empty(q.shape, device="cuda") for _ in range(60)]
    torch.cuda.synchronize()
    st = torch.cuda.Stream()
    for i, o in enumerate(outs):
        path = 1 + (i // 3) % 2  # the projection on CUDA cores and on tensor cores in turn
        sp.sp_project(st, M, N, K, x_d[i % 3], wt, values, path, pws, pws.numel())
        sp.sp_attend(st, dims, len(lens), None, cache.seq_lens, cache.desc, q_d, kn_d, vn_d, o, sp.SP_F32, ws, ws.numel())
    st.synchronize()
    for i, o in enumerate(outs):
        # values off by up to 4e-5 of the largest (hi + lo inputs, K = 1024), the rest fp32
        np.testing.assert_allclose(o.cpu().numpy(), refs[i % 3], rtol=1e-3, atol=1e-3)


@pytest.mark.parametrize("recursive", [0, 1])
def test_hidden_states(recursive):
    sh = wl.Shape(256, 8, 2, 128, 512, 4, 3)
    w = wl.with_fusion(wl.custom(sh, [120, 700, 3], wl.LAYOUT_PAGED, 950))
    run = GpuRun(w, options={sp.SP_OPT_RECURSIVE: recursive})
    torch, B = run.torch, 3
    rng = np.random.default_rng(3)
    states = [wl.f32_to_bf16_bits(rng.standard_normal((B, 256)).astype(np.float32)) for _ in range(3)]
    layer = so.Layer(w.shape, w.weights)
    ref = [so.classify_recursive(layer, w.cache, w.seq_ids, s) if recursive
           else so.classify(layer, w.cache, w.seq_ids, hidden=s) for s in states]
    dev = [rows_tensor(torch, s) for s in states]
    outs = [torch.empty((B, 3), device="cuda") for _ in range(12)]
    torch.cuda.synchronize()
    st = torch.cuda.Stream()
    for i, o in enumerate(outs):
        sp.sp_classify_hidden(run.model.handle, st, B, run.ids, run.cache.seq_lens, run.cache.desc, dev[i % 3], o)
    st.synchronize()
    for i, o in enumerate(outs):
        compare(o.double().cpu().numpy(), ref[i % 3], label=f"call {i}")
        assert torch.equal(o, outs[i % 3])
    run.close()


@pytest.mark.parametrize("M,N,K,path", [(7, 256, 192, 0), (300, 512, 256, 2), (40, 384, 128, 1)])
def test_project(M, N, K, path):
    ensure_built()
    torch = torch_dev()
    rng = np.random.default_rng(M)
    # the weights are an argument, too: another matrix in every turn, written in front
    # of the call on the same stream
    xs, ws = ([rng.standard_normal((r, K)).astype(np.float32) for _ in range(3)] for r in (M, N))
    bits = [wl.f32_to_bf16_bits(0.05 * w) for w in ws]
    ref = [x.astype(np.float64) @ wl.bf16_bits_to_f32(b).astype(np.float64).T for x, b in zip(xs, bits)]
    x_d = [torch.from_numpy(x).cuda() for x in xs]
    w_d = [torch.from_numpy(b.view(np.int16)).cuda() for b in bits]
    x, w = torch.empty_like(x_d[0]), torch.empty_like(w_d[0])
    n = max(256, sp.sp_project_workspace_bytes(M, N, K))
    scratch = torch.empty(n, dtype=torch.uint8, device="cuda")
    outs = [torch.empty((M, N), device="cuda") for _ in range(24)]
    torch.cuda.synchronize()
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        for i, o in enumerate(outs):
            x.copy_(x_d[i % 3])
            w.copy_(w_d[i % 3])
            sp.sp_project(st, M, N, K, x, w, o, path, scratch, n)
    st.synchronize()
    for i, o in enumerate(outs):
        # hi + lo activations and fp32 sums (the bound of the projection tests)
        assert np.max(np.abs(o.double().cpu().numpy() - ref[i % 3])) <= 2e-5 * np.max(np.abs(ref[i % 3]))


@pytest.mark.parametrize("lens", [[250, 30], [900, 0, 1500, 64], [100] * 40])
@pytest.mark.parametrize("k", [4, 24])
def test_attend_on_tensor_cores(lens, k):
    ensure_built()
    torch = torch_dev()
    shape, B = wl.Shape(256, 8, 2, 128, 256, k, 2), len(lens)
    w = wl.custom(shape, lens, wl.LAYOUT_PAGED, 960)
    rng = np.random.default_rng(k)
    qs = [rng.standard_normal((B, k, 8, 128)).astype(np.float32) for _ in range(3)]
    kn, vn = (rng.standard_normal((B, k, 2, 128)).astype(np.float32) for _ in range(2))
    ref = [so.attention_step(shape, w.cache, w.seq_ids, *(t.astype(np.float64) for t in (q, kn, vn))) for q in qs]
    cache = sp.DeviceCache(w.cache)
    dims = sp.sp_attn_dims(8, 2, 128, k, sp.SP_BF16, max(lens), 0, 2)
    ws = torch.empty(sp.sp_attend_workspace_bytes(dims, B), dtype=torch.uint8, device="cuda")
    q_d = [torch.from_numpy(q).cuda() for q in qs]
    kn_d, vn_d = torch.from_numpy(kn).cuda(), torch.from_numpy(vn).cuda()
    q = torch.empty_like(q_d[0])
    outs = [torch.empty(q.shape, device="cuda") for _ in range(24)]
    torch.cuda.synchronize()
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        for i, o in enumerate(outs):
            q.copy_(q_d[i % 3])
            sp.sp_attend(st, dims, B, None, cache.seq_lens, cache.desc, q, kn_d, vn_d, o, sp.SP_F32, ws, ws.numel())
    st.synchronize()
    for i, o in enumerate(outs):
        # bf16 new rows and probabilities (as in the other tests of this step)
        assert np.all(np.abs(o.cpu().numpy() - ref[i % 3]) <= 2e-2 * (1 + np.abs(ref[i % 3])))
        assert torch.equal(o, outs[i % 3])
