"""The attention kernel with tokens on the MMA's M side at the edges of its
work: query rows around the multiples of 16 it pads to, lengths around the
64-token tiles and 128-token steps, segments of one tile, pairs cut into many
segments, plain and hi + lo queries, every page size; against the fp64 oracle."""
import numpy as np
import pytest

import oracle.sp_oracle as so
import paper_2608_28099_gb300 as sp
from paper_2608_28099_gb300 import workloads as wl
from gpu_util import GpuRun, compare, ensure_built, oracle_logits, rows_tensor
from test_gpu_parity import _attend

pytestmark = pytest.mark.gpu

LENS = [0, 1, 63, 64, 65, 127, 128, 129, 191, 193, 700, 2100]


@pytest.mark.parametrize("hq,hkv,k,page", [
    (4, 2, 1, 16), (8, 2, 4, 0), (10, 2, 3, 32), (8, 2, 8, 64), (8, 2, 9, 16), (8, 2, 16, 0),
    (10, 2, 13, 16), (12, 2, 16, 32), (10, 2, 20, 0), (16, 2, 16, 16),
])
@pytest.mark.parametrize("split", [0, 64])
def test_rows_lengths_and_splits(hq, hkv, k, page, split):
    ensure_built()
    shape = wl.Shape(256, hq, hkv, 128, 256, k, 2, page_size=page or 16)
    w = wl.custom(shape, LENS, wl.LAYOUT_PAGED if page else wl.LAYOUT_CONTIGUOUS, 700 + k)
    rng = np.random.default_rng(k)
    B = len(LENS)
    q = (1.5 * rng.standard_normal((B, k, hq, 128))).astype(np.float32)
    kn, vn = (rng.standard_normal((B, k, hkv, 128)).astype(np.float32) for _ in range(2))
    q[0, 0, 0] *= 6.0  # rows whose maximum moves (scores of standard deviation 9)
    q[11, 0, 0] *= 6.0
    ref = so.attention_step(shape, w.cache, w.seq_ids, *(t.astype(np.float64) for t in (q, kn, vn)))
    out, g = _attend(shape, w, q, kn, vn, 2, split=split)
    # new values are bf16 (2^-9 of up to 4.5: 9e-3), a new key's score is off by
    # 1.5 * 2^-9 / sqrt(3) * N(0, 1) (up to 7e-3) and its weight by as much of
    # itself, times a spread of values of ~1.4: 2e-2 in all, seen 1.2e-2.  A sharp
    # row's scores are six times that off.
    err = np.abs(out - ref)
    sharp = np.zeros(out.shape, bool)
    sharp[[0, 11], 0, 0] = True
    assert np.all(err[~sharp] <= 2e-2 * (1 + np.abs(ref[~sharp])))
    assert np.all(err[sharp] <= 8e-2 * (1 + np.abs(ref[sharp])))
    if g is not None:
        for b, L in enumerate(LENS):
            n = (L + page - 1) // page
            assert np.array_equal(g[b, :n], w.cache.page_table[b, :n])


@pytest.mark.parametrize("hq,k", [(4, 4), (4, 16), (8, 16)])
@pytest.mark.parametrize("split", [0, 512])
def test_empty_share(hq, k, split):
    # four sequences of 15 tiles.  In shares of eight tiles and more the cuts are 0, 0,
    # 15, 15, 30, ...: every other group of CTAs, the first one too, has nothing to do.
    # In the default ones (four and more) two cuts meet in the middle, at 30.
    ensure_built()
    shape = wl.Shape(256, 2 * hq, 2, 128, 256, k, 2)
    w = wl.custom(shape, [900 - 4 * (k > 4)] * 4, wl.LAYOUT_PAGED, 710 + k)
    rng = np.random.default_rng(k)
    q = rng.standard_normal((4, k, 2 * hq, 128)).astype(np.float32)
    kn, vn = (rng.standard_normal((4, k, 2, 128)).astype(np.float32) for _ in range(2))
    ref = so.attention_step(shape, w.cache, w.seq_ids, *(t.astype(np.float64) for t in (q, kn, vn)))
    for _ in range(2):  # the merge counters are clear again after the first call
        out, _ = _attend(shape, w, q, kn, vn, 2, split=split)
        np.testing.assert_allclose(out, ref, rtol=1e-2, atol=1e-2)


@pytest.mark.parametrize("hq,k,T", [(4, 16, 1), (5, 16, 1), (3, 32, 1), (7, 16, 1), (4, 32, 1), (4, 16, 2)])
@pytest.mark.parametrize("layout", [wl.LAYOUT_PAGED, wl.LAYOUT_CONTIGUOUS])
def test_plain_queries_through_classify(hq, k, T, layout):
    sh = wl.Shape(256, 2 * hq, 2, 128, 512, k, 2)
    w = wl.custom(sh, [0, 60, 64, 65, 130, 900, 128, 3, 5, 1500], layout, 720 + k, rows_per_seq=True)
    if T > 1:
        w = wl.with_tasks(w, T)
        run = GpuRun(w)
        torch = run.torch
        out = torch.empty((len(w.seq_ids), T, 2), dtype=torch.float32, device="cuda")
        sp.sp_classify(run.model.handle, torch.cuda.current_stream(), len(w.seq_ids), run.ids,
                       run.cache.seq_lens, run.cache.desc, rows_tensor(torch, w.rows), out)
        torch.cuda.synchronize()
        prompts, heads, biases, rows = wl.task_views(w)
        ref = so.classify_tasks(so.Layer(w.shape, w.weights), w.cache, w.seq_ids, prompts, heads,
                                biases, rows)
        for t in range(T):
            compare(out[:, t].double().cpu().numpy(), ref[:, t], label=f"task {t}")
    else:
        run = GpuRun(w)
        compare(run.logits(), oracle_logits(w), label=f"plain R={hq * k}")
    run.close()


def _lens(B, longest):
    lens = np.random.default_rng(B).integers(0, 200, B)
    lens[B // 2] = longest
    return [int(x) for x in lens]


# 33 to 64 rows take this kernel from three (sequence, kv head) pairs per CTA on, 57
# sequences of 8 kv heads or 228 of 2 on 152 SMs; more rows never do
@pytest.mark.parametrize("hq,k,layout,B,longest,hkv", [
    (4, 16, wl.LAYOUT_PAGED, 120, 200, 2), (4, 15, wl.LAYOUT_CONTIGUOUS, 115, 129, 2),
    (4, 16, wl.LAYOUT_CONTIGUOUS, 25, 4200, 2), (5, 16, wl.LAYOUT_CONTIGUOUS, 25, 4200, 2),
    (4, 16, wl.LAYOUT_PAGED, 56, 700, 8), (4, 16, wl.LAYOUT_CONTIGUOUS, 57, 700, 8),
    (4, 16, wl.LAYOUT_PAGED, 300, 1100, 2), (7, 8, wl.LAYOUT_PAGED, 240, 500, 2), (3, 16, wl.LAYOUT_PAGED, 240, 300, 2),
])
def test_plain_queries_of_more_rows(hq, k, layout, B, longest, hkv):
    w = wl.custom(wl.Shape(256, hkv * hq, hkv, 128, 512, k, 2), _lens(B, longest), layout, 730 + k, rows_per_seq=True)
    run = GpuRun(w)
    compare(run.logits(), oracle_logits(w), label=f"plain R={hq * k}")
    run.close()


# (1900 sequences: the tables leave too little shared memory for 48 or 64 hi + lo rows)
@pytest.mark.parametrize("k,page,B,longest,hkv", [
    (12, 0, 8, 2100, 2), (16, 16, 16, 2100, 2), (16, 0, 25, 4200, 2),
    (12, 0, 56, 400, 8), (12, 16, 57, 1300, 8), (9, 0, 60, 1300, 8), (12, 64, 1900, 150, 2), (11, 32, 400, 700, 2),
    (16, 16, 240, 300, 2), (16, 0, 57, 900, 8), (15, 16, 1900, 150, 2),
])
def test_exact_queries_of_more_rows(k, page, B, longest, hkv):
    ensure_built()
    shape = wl.Shape(256, 4 * hkv, hkv, 128, 256, k, 2, page_size=page or 16)
    w = wl.custom(shape, _lens(B, longest), wl.LAYOUT_PAGED if page else wl.LAYOUT_CONTIGUOUS, 740 + k)
    rng = np.random.default_rng(k)
    q = rng.standard_normal((B, k, 4 * hkv, 128)).astype(np.float32)
    kn, vn = (rng.standard_normal((B, k, hkv, 128)).astype(np.float32) for _ in range(2))
    ref = so.attention_step(shape, w.cache, w.seq_ids, *(t.astype(np.float64) for t in (q, kn, vn)))
    out, _ = _attend(shape, w, q, kn, vn, 2)
    # as above: bf16 new values and scores, 2e-2 in all at 1.5 times these queries
    assert np.all(np.abs(out - ref) <= 2e-2 * (1 + np.abs(ref)))


# shares: whole sequences in a share each, more sequences than shares hold, one
# sequence over many shares, empty caches
@pytest.mark.parametrize("lens", [[500] * 16, [300] * 3, [1000] * 80 + [0] * 9, [0] * 30 + [5000], [2000, 70, 0, 70]])
@pytest.mark.parametrize("hq,k", [(4, 4), (6, 16)])
def test_shares(lens, hq, k):
    ensure_built()
    shape = wl.Shape(256, 4 * hq, 4, 128, 256, k, 2)
    w = wl.custom(shape, lens, wl.LAYOUT_PAGED, 750 + len(lens))
    rng = np.random.default_rng(len(lens))
    B = len(lens)
    q = rng.standard_normal((B, k, 4 * hq, 128)).astype(np.float32)
    kn, vn = (rng.standard_normal((B, k, 4, 128)).astype(np.float32) for _ in range(2))
    ref = so.attention_step(shape, w.cache, w.seq_ids, *(t.astype(np.float64) for t in (q, kn, vn)))
    for _ in range(2):  # the merge counters are clear again after the first call
        out, _ = _attend(shape, w, q, kn, vn, 2)
        assert np.all(np.abs(out - ref) <= 2e-2 * (1 + np.abs(ref)))


@pytest.mark.parametrize("hq,k,layout,B", [
    (4, 16, wl.LAYOUT_CONTIGUOUS, 16), (5, 16, wl.LAYOUT_CONTIGUOUS, 16), (3, 16, wl.LAYOUT_PAGED, 8),
    (4, 12, wl.LAYOUT_CONTIGUOUS, 4), (4, 15, wl.LAYOUT_PAGED, 8), (4, 8, wl.LAYOUT_PAGED, 3),
    (6, 16, wl.LAYOUT_CONTIGUOUS, 16),
])
def test_the_length_bound_chooses_nothing(hq, k, layout, B):
    # max_seq_len is a server's context limit and may be far above every length: the
    # kernel and its plan, and so the bits, do not depend on it
    w = wl.custom(wl.Shape(256, 2 * hq, 2, 128, 512, k, 2), _lens(B, 500), layout, 770 + k, rows_per_seq=True)
    got = []
    for bound in (500, 33000):
        run = GpuRun(w, max_seq_len=bound)
        got.append(run.logits())
        run.close()
    assert np.array_equal(got[0], got[1])


def _bf16(x):
    return wl.bf16_bits_to_f32(wl.f32_to_bf16_bits(x.astype(np.float32))).astype(np.float64)


@pytest.mark.parametrize("L,k,hq,layout", [
    (30, 4, 8, wl.LAYOUT_PAGED), (70, 4, 8, wl.LAYOUT_PAGED), (100, 1, 8, wl.LAYOUT_CONTIGUOUS),
    (100, 4, 8, wl.LAYOUT_PAGED), (128, 8, 8, wl.LAYOUT_PAGED), (200, 4, 8, wl.LAYOUT_PAGED),
    (250, 2, 8, wl.LAYOUT_CONTIGUOUS), (300, 4, 8, wl.LAYOUT_PAGED), (700, 8, 8, wl.LAYOUT_PAGED),
    (100, 12, 8, wl.LAYOUT_PAGED), (190, 16, 8, wl.LAYOUT_CONTIGUOUS),
])
def test_error_is_no_larger_than_that_of_the_kernel_with_queries_on_m(L, k, hq, layout):
    # The other kernel's error, from the same inputs: probabilities rounded to bf16
    # against a running maximum of its own in each of two pipelines (the even and the
    # odd 64-token tiles, the first tile's maximum: none here grows by 2^8), sums over
    # the unrounded ones, new rows rounded to bf16.  The 2-norm over 800 rows or more
    # of 128 varies by 2 % between such roundings.
    ensure_built()
    hkv, B = 2, 240 if k > 8 else 96  # (more than 32 rows take this kernel from 228 on)
    shape = wl.Shape(256, hq, hkv, 128, 256, k, 2)
    w = wl.custom(shape, [L] * B, layout, 760 + L + k)
    rng = np.random.default_rng(L + k)
    q = (1.28 * rng.standard_normal((B, k, hq, 128))).astype(np.float32)
    kn, vn = ((1.28 * rng.standard_normal((B, k, hkv, 128))).astype(np.float32) for _ in range(2))
    ref = so.attention_step(shape, w.cache, w.seq_ids, *(t.astype(np.float64) for t in (q, kn, vn)))
    other = np.empty_like(ref)
    t = np.arange(L + k)
    sees = t[None, :] <= L + np.arange(k)[:, None]
    for b in range(B):
        K, V = so.sequence_kv(w.cache, b)
        K = np.repeat(np.concatenate([K, _bf16(kn[b])]), hq // hkv, axis=1)
        V = np.repeat(np.concatenate([V, _bf16(vn[b])]), hq // hkv, axis=1)
        s = np.einsum("rhd,thd->hrt", q[b].astype(np.float64), K) / np.sqrt(128.0)
        s = np.where(sees[None], s, -np.inf)
        top = s.max(-1, keepdims=True)
        o, l = 0.0, 0.0
        for pipe in (0, 1):
            at = t[(t // 64) % 2 == pipe]
            if len(at) == 0:
                continue
            m = s[..., at[at // 64 == pipe]].max(-1, keepdims=True)
            m = np.where(np.isfinite(m), m, top)
            p = np.exp(s[..., at] - m)
            o = o + np.einsum("hrt,thd->rhd", _bf16(p) * np.exp(m - top), V[at])
            l = l + (p * np.exp(m - top)).sum(-1)
        other[b] = o / l.T[..., None]
    out, _ = _attend(shape, w, q, kn, vn, 2, split=0)
    err, want = np.linalg.norm(out - ref), np.linalg.norm(other - ref)
    assert err <= 1.02 * want, (err / np.linalg.norm(ref), want / np.linalg.norm(ref))


@pytest.mark.parametrize("k,lens", [
    (4, [160, 80, 143, 98, 105, 91]), (8, [187, 156, 154, 133, 117, 45, 116, 140]),
    (8, [54, 144, 133, 67, 82, 185, 72, 163, 117, 200, 175, 141, 131, 57, 108, 77]),
    (16, [105, 99, 62, 113, 185, 91, 59, 72, 50, 68, 48, 199]), (24, [60, 154, 125, 202, 203, 133, 174, 91]),
    (32, [184, 145, 91, 157, 195, 56, 81, 43, 126, 126]),
])
def test_short_sequences_stay_whole(k, lens):
    # a sequence that no share cut: the same bits as alone, where (up to 256 tokens
    # with the new ones) it is one share
    ensure_built()
    shape = wl.Shape(256, 32, 8, 128, 256, k, 2)
    w = wl.custom(shape, lens, wl.LAYOUT_CONTIGUOUS, 780 + k)
    rng = np.random.default_rng(k)
    B = len(lens)
    q = rng.standard_normal((B, k, 32, 128)).astype(np.float32)
    kn, vn = (rng.standard_normal((B, k, 8, 128)).astype(np.float32) for _ in range(2))
    out, _ = _attend(shape, w, q, kn, vn, 2, split=0)
    for b in range(B):
        o, n = int(w.cache.offsets[b]), lens[b]
        c = w.cache
        alone = wl.KVCache(c.layout, c.dtype, np.array([n], np.int32), c.k_flat[o:o + n], c.v_flat[o:o + n],
                           np.array([0], np.int64))
        one = wl.Workload(w.spec, w.weights, alone, np.array([0], np.int32), None)
        got, _ = _attend(shape, one, q[b:b + 1], kn[b:b + 1], vn[b:b + 1], 2, split=0)
        assert np.array_equal(got[0], out[b]), b
