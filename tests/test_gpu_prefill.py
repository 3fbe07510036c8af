"""GPU parity of the prefill attention against the CPU oracle, through the C-ABI."""
import numpy as np
import pytest
import torch

import oracle
from paper_2401_05391_b200 import segkv as sk
from paper_2401_05391_b200 import workloads as wl

from _harness import ATOL, RTOL

pytestmark = pytest.mark.gpu


def check_rows(w, q, kp, vp, out, slopes, rows):
    ref = oracle.prefill_sdpa(w.dtype, w.batch, w.heads, w.kv_heads, w.head_dim, wl.to_bits(q), wl.to_bits(kp),
                              wl.to_bits(vp), slopes=None if slopes is None else slopes.cpu().numpy(), rows=rows)
    got = np.stack([out[b, i, h].to(torch.float64).cpu().numpy() for b, i, h in rows])
    assert np.isfinite(got).all()
    err = np.abs(got - ref)
    # the path's stated tolerance for both storage types
    assert (err <= ATOL + RTOL * np.abs(ref)).all(), f"max err {err.max():.3e}"


def run_prefill(w, rows_fn, row_groups=0, prompt_layout=None):
    h = sk.SegKV(w.batch, w.beams, w.heads, w.kv_heads, w.head_dim, w.prompt_len, w.steps, w.torch_dtype)
    try:
        h.set_prefill_tuning(row_groups)
        if prompt_layout is not None:
            h.set_prompt_layout(prompt_layout)
        kp, vp = wl.make_prompt(w, "cuda")
        q = wl.make_prefill_query(w, "cuda")
        slopes = wl.alibi_slopes(w.heads).cuda() if w.alibi else None
        out = torch.full_like(q, float("nan"))
        h.prefill(kp, vp, q, out, slopes)
        torch.cuda.synchronize()
        assert not torch.isnan(out.float()).any(), "unwritten outputs"
        check_rows(w, q, kp, vp, out, slopes, rows_fn(w))
        assert h.get_error() == 0
        return h, q, kp, vp, out, slopes
    except Exception:
        h.destroy()
        raise


def all_rows(w):
    return [(b, i, h) for b in range(w.batch) for i in range(w.prompt_len) for h in range(w.heads)]


def sampled_rows(w, n=192, seed=0):
    rng = np.random.default_rng(w.seed + seed)
    rows = {(0, 0, 0), (w.batch - 1, w.prompt_len - 1, w.heads - 1), (0, 63, 0), (0, 64, 0), (0, w.prompt_len - 1, 0)}
    while len(rows) < n:
        rows.add((int(rng.integers(w.batch)), int(rng.integers(w.prompt_len)), int(rng.integers(w.heads))))
    return sorted(r for r in rows if r[1] < w.prompt_len)


@pytest.mark.parametrize("dtype", ["f16", "bf16"])
@pytest.mark.parametrize("D,P", [(64, 150), (128, 150), (128, 64), (128, 65), (64, 1), (256, 150), (256, 33), (128, 300)])
def test_prefill_ragged_small_shapes(dtype, D, P):
    # several tiles and a ragged tail, GQA, ALiBi on the bf16 variants
    w = wl.Workload("pf", 2, 3, 6, 2, D, P, 2, dtype, "uniform", dtype == "bf16", 80 + D // 64)
    h = run_prefill(w, all_rows)[0]
    h.destroy()


@pytest.mark.parametrize("dtype", ["f16", "bf16"])
@pytest.mark.parametrize("row_groups", [1, 2])
@pytest.mark.parametrize("P", [64, 128, 129, 150, 256, 257, 300, 520, 777])
def test_prefill_head_dim_128_row_groups(dtype, row_groups, P):
    # the tcgen05 kernel with one and with two 128-row groups per CTA: prompts that leave the
    # second group empty (64, 128), with one row (129), exact tiles (256), ragged (150, 257, 300, 777)
    # and spanning CTAs (520, 777)
    w = wl.Workload("pf", 2, 3, 4, 2, 128, P, 2, dtype, "uniform", dtype == "bf16", 90 + row_groups)
    h = run_prefill(w, all_rows if P <= 300 else (lambda w: sampled_rows(w, 400)), row_groups)[0]
    h.destroy()


@pytest.mark.parametrize("row_groups", [1, 2])
def test_prefill_llama2_7b_shape_row_groups_sampled(row_groups):
    h = run_prefill(wl.CONFIGS[1], lambda w: sampled_rows(w, 256), row_groups)[0]
    h.destroy()


@pytest.mark.parametrize("layout", ["token_major", "seq_first"])
@pytest.mark.parametrize("D,P", [(64, 150), (128, 300), (256, 150)])
def test_prefill_prompt_layouts(layout, D, P):
    w = wl.Workload("pf", 2, 3, 6, 2, D, P, 2, "f16", "uniform", False, 95)
    h = run_prefill(w, all_rows, prompt_layout=layout)[0]
    h.destroy()


@pytest.mark.parametrize("D,row_groups", [(256, 0), (128, 1), (64, 1), (64, 2)])
def test_prefill_many_items_per_cta(D, row_groups):
    # 768 or more work items on 148 persistent CTAs, tile counts 5 / 4 / 2 per item: every CTA walks
    # several items back to back (barrier phases, ring positions and tensor-memory buffers carry over)
    w = wl.Workload("pf", 16, 2, 16, 16, D, 300, 2, "f16", "uniform", False, 97)
    for _ in range(2):
        h = run_prefill(w, lambda w: sampled_rows(w, 300), row_groups)[0]
        h.destroy()


@pytest.mark.parametrize("dtype,D", [("f16", 128), ("bf16", 128), ("f16", 256), ("f16", 64)])
def test_prefill_per_request_prompt_lengths(dtype, D):
    # ragged prompts: each request is computed up to its own length (against the oracle run on that
    # request alone), the poisoned padding never leaks in, and the rows behind a request's length stay untouched
    lens = [300, 1, 129, 64, 257]
    w = wl.Workload("pf", len(lens), 2, 4, 2, D, 300, 2, dtype, "uniform", dtype == "bf16", 98)
    h = sk.SegKV(w.batch, w.beams, w.heads, w.kv_heads, w.head_dim, w.prompt_len, w.steps, w.torch_dtype)
    try:
        kp, vp = wl.make_prompt(w, "cuda")
        q = wl.make_prefill_query(w, "cuda")
        for b, n in enumerate(lens):
            kp[b, n:] = float("nan")
            vp[b, n:] = float("inf")
        slopes = wl.alibi_slopes(w.heads).cuda() if w.alibi else None
        for groups in (1, 2):
            if D == 256 and groups == 2:
                continue
            h.set_prefill_tuning(groups)
            h.prefill_write_ragged(kp, vp, lens)
            out = torch.full_like(q, 512.0)
            h.prefill_sdpa(q, out, slopes)
            torch.cuda.synchronize()
            assert h.get_error() == 0
            for b, n in enumerate(lens):
                assert bool((out[b, n:].float() == 512.0).all()), "rows behind the request's length were written"
                w1 = w.scaled(batch=1, prompt_len=n)
                rows = [(0, i, hd) for i in sorted({0, n - 1, n // 2, min(n - 1, 63), min(n - 1, 128)}) for hd in range(w.heads)]
                check_rows(w1, q[b:b + 1, :n].contiguous(), kp[b:b + 1, :n].contiguous(), vp[b:b + 1, :n].contiguous(),
                           out[b:b + 1, :n].contiguous(), slopes, rows)
    finally:
        h.destroy()


@pytest.mark.parametrize("layout", [None, "token_major", "seq_first"])
@pytest.mark.parametrize("dtype,D,heads,kv_heads,P", [("f16", 128, 8, 2, 300), ("bf16", 128, 4, 4, 129), ("f16", 256, 4, 2, 150),
                                                      ("f16", 64, 6, 3, 520)])
def test_fused_prefill_stores_the_same_segment_and_output_as_the_two_calls(layout, dtype, D, heads, kv_heads, P):
    # segkv_prefill (one launch: attention + prompt store) against segkv_prefill_write + segkv_prefill_sdpa:
    # same output bit for bit, and the decode attention over the stored segment agrees bit for bit too
    w = wl.Workload("pf", 3, 2, heads, kv_heads, D, P, 3, dtype, "uniform", dtype == "bf16", 99)
    kp, vp = wl.make_prompt(w, "cuda")
    q = wl.make_prefill_query(w, "cuda")
    slopes = wl.alibi_slopes(w.heads).cuda() if w.alibi else None
    qd, kd, vd = wl.make_step(w, 0, "cuda")
    results = []
    for fused in (False, True):
        h = sk.SegKV(w.batch, w.beams, w.heads, w.kv_heads, w.head_dim, w.prompt_len + 40, w.steps, w.torch_dtype)
        try:
            if layout is not None:
                h.set_prompt_layout(layout)
            out = torch.full_like(q, 512.0)
            if fused:
                h.prefill(kp, vp, q, out, slopes)
            else:
                h.prefill_write(kp, vp)
                h.prefill_sdpa(q, out, slopes)
            dec0 = h.decode_sdpa(qd, None, slopes)                 # prompt only
            h.append(0, None, kd, vd)
            dec1 = h.decode_sdpa(qd, None, slopes)
            torch.cuda.synchronize()
            assert h.get_error() == 0
            results.append((out.clone(), dec0.clone(), dec1.clone()))
        finally:
            h.destroy()
    for a, b in zip(*results):
        assert torch.equal(a.view(torch.int16), b.view(torch.int16))
    check_rows(w, q, kp, vp, results[1][0], slopes, sampled_rows(w, 96))


@pytest.mark.parametrize("D,H,Hkv,P,groups", [(256, 16, 16, 300, 0), (128, 16, 4, 300, 1), (128, 16, 16, 520, 2)])
def test_prefill_is_bit_reproducible_across_runs(D, H, Hkv, P, groups):
    # no atomics and a fixed schedule: repeated launches must give the same bits (a missed barrier phase
    # once showed up here as rows that changed from run to run)
    w = wl.Workload("pf", 16, 2, H, Hkv, D, P, 2, "f16", "uniform", False, 96)
    h = sk.SegKV(w.batch, w.beams, w.heads, w.kv_heads, w.head_dim, w.prompt_len, w.steps, w.torch_dtype)
    try:
        h.set_prefill_tuning(groups)
        kp, vp = wl.make_prompt(w, "cuda")
        q = wl.make_prefill_query(w, "cuda")
        ref = None
        for it in range(10):
            out = torch.full_like(q, 512.0)
            if it % 2:
                h.prefill(kp, vp, q, out)
            else:
                h.prefill_write(kp, vp)
                h.prefill_sdpa(q, out)
            torch.cuda.synchronize()
            assert not torch.isnan(out.float()).any()
            if ref is None:
                ref = out.clone()
            assert torch.equal(ref.view(torch.int16), out.view(torch.int16)), f"run {it} differs"
        assert h.get_error() == 0
    finally:
        h.destroy()


@pytest.mark.parametrize("D,H,Hkv,P", [(128, 8, 8, 4096), (256, 8, 2, 3000)])
def test_prefill_long_prompt_sampled(D, H, Hkv, P):
    # 32 or more key tiles per row group, items of very different lengths on every CTA
    w = wl.Workload("pf", 1, 2, H, Hkv, D, P, 2, "f16", "uniform", False, 94)
    h = run_prefill(w, lambda w: sampled_rows(w, 96))[0]
    h.destroy()


def test_prefill_llama2_7b_shape_sampled():
    h = run_prefill(wl.CONFIGS[1], lambda w: sampled_rows(w, 256))[0]
    h.destroy()


def test_prefill_gptj_shape_cut_to_batch_2_sampled():
    h = run_prefill(wl.CONFIGS[2].scaled(batch=2), lambda w: sampled_rows(w, 256))[0]
    h.destroy()


def test_prefill_bloom_shape_cut_to_batch_2_sampled():
    h = run_prefill(wl.CONFIGS[4].scaled(batch=2), lambda w: sampled_rows(w, 256))[0]
    h.destroy()


def test_prefill_last_row_agrees_with_the_decode_kernel_on_the_prompt():
    """The prefill kernel is the decode kernel's special case: its last row is what the decode
    kernel returns for a query that sees only the prompt."""
    w = wl.Workload("pfdec", 2, 4, 4, 2, 128, 200, 2, "f16", "uniform", True, 83)
    h, q, kp, vp, out, slopes = run_prefill(w, lambda w: sampled_rows(w, 64))
    try:
        qd = q[:, -1].repeat_interleave(w.beams, dim=0).contiguous()        # [rows, heads, D]
        od = h.decode_sdpa(qd, None, slopes)
        torch.cuda.synchronize()
        want = out[:, -1].repeat_interleave(w.beams, dim=0)
        assert torch.allclose(od.float(), want.float(), atol=2e-3, rtol=1e-2)
    finally:
        h.destroy()


def test_prefill_argument_and_state_errors():
    h = sk.SegKV(1, 2, 2, 2, 64, 16, 4, torch.float16)
    q = torch.zeros(1, 16, 2, 64, dtype=torch.float16, device="cuda")
    with pytest.raises(sk.SegKVError) as e:
        rc = sk.lib().segkv_prefill_sdpa(h._h, q.data_ptr(), q.data_ptr(), None, None)
        sk._check(rc, "segkv_prefill_sdpa")
    assert e.value.code == sk.SEGKV_ESTATE                   # no prompt stored yet
    rc = sk.lib().segkv_prefill_sdpa(h._h, None, q.data_ptr(), None, None)
    assert rc == sk.SEGKV_EINVAL
    h.destroy()


@pytest.mark.parametrize("dtype", ["f16", "bf16"])
@pytest.mark.parametrize("D,row_groups", [(64, 1), (64, 2), (128, 1), (128, 2), (256, 1)])
def test_prefill_scores_that_grow_from_tile_to_tile(dtype, D, row_groups):
    # no bias, keys 4, 10 and 25 times as long from the second, third and fifth tile on: rows whose maximum grows by more
    # than 2^8 of the reference they use, in full and in diagonal tiles, so that weights worked out in one pass are thrown
    # away, O is rescaled and the tile done again.  A few keys carry a row's weight then: besides the path's tolerance the
    # rounding of the weights (2^-9 of each in bf16, 2^-12 in fp16) times the largest value is allowed for.
    w = wl.Workload("grow", 2, 3, 4, 2, D, 700, 2, dtype, "uniform", False, 140)
    h = sk.SegKV(w.batch, w.beams, w.heads, w.kv_heads, w.head_dim, w.prompt_len, w.steps, w.torch_dtype)
    try:
        h.set_prefill_tuning(row_groups)
        kp, vp = wl.make_prompt(w, "cuda")
        for at, by in ((128, 4.0), (256, 2.5), (512, 2.5)):
            kp[:, at:] *= by
        q = wl.make_prefill_query(w, "cuda")
        h.prefill_write(kp, vp)
        out, fused = h.prefill_sdpa(q, None, None), torch.full_like(q, float("nan"))
        h.prefill(kp, vp, q, fused, None)
        torch.cuda.synchronize()
        assert h.get_error() == 0
        assert torch.equal(out, fused)
        rows = sampled_rows(w, 500)
        ref = oracle.prefill_sdpa(w.dtype, w.batch, w.heads, w.kv_heads, w.head_dim, wl.to_bits(q), wl.to_bits(kp), wl.to_bits(vp), rows=rows)
        got = np.stack([out[b, i, x].to(torch.float64).cpu().numpy() for b, i, x in rows])
        err = np.abs(got - ref)
        assert (err <= ATOL + RTOL * np.abs(ref) + float(vp.abs().max()) * 2.0 ** (-9 if dtype == "bf16" else -12)).all(), err.max()
    finally:
        h.destroy()


@pytest.mark.parametrize("dtype", ["f16", "bf16"])
@pytest.mark.parametrize("D,row_groups", [(64, 1), (64, 2), (128, 1), (128, 2), (256, 1)])
def test_prefill_references_that_fall_in_the_middle_of_a_tile(dtype, D, row_groups):
    # Single keys eight times as long at places that end a tile's one pass behind its first, second and last pieces of 16
    # keys (what is stored by then is scaled), at prompts that end in every part of a pair of row groups; and, in the
    # second half of the heads, slopes that favour OLDER keys, so that going back through the keys the maximum grows.  The
    # rounding of the weights is allowed for as above.
    for P in (129, 257, 390, 515):
        w = wl.Workload("spike", 1, 2, 4, 2, D, P, 2, dtype, "uniform", True, 150 + P)
        h = sk.SegKV(w.batch, w.beams, w.heads, w.kv_heads, w.head_dim, w.prompt_len, w.steps, w.torch_dtype)
        try:
            h.set_prefill_tuning(row_groups)
            kp, vp = wl.make_prompt(w, "cuda")
            for at in (20, 135, 128 + 40, 256 + 17, 256 + 63, 384 + 1, 512):
                kp[:, at:at + 1] *= 8.0
            q = wl.make_prefill_query(w, "cuda")
            for slopes in (None, torch.tensor([0.25, 0.01, -0.02, -0.25], device="cuda")):
                out, fused = torch.full_like(q, float("nan")), torch.full_like(q, float("nan"))
                h.prefill_write(kp, vp)
                h.prefill_sdpa(q, out, slopes)
                h.prefill(kp, vp, q, fused, slopes)
                torch.cuda.synchronize()
                assert h.get_error() == 0
                assert torch.equal(out, fused)
                rows = all_rows(w)[::3]
                ref = oracle.prefill_sdpa(w.dtype, w.batch, w.heads, w.kv_heads, w.head_dim, wl.to_bits(q), wl.to_bits(kp),
                                          wl.to_bits(vp), slopes=None if slopes is None else slopes.cpu().numpy(), rows=rows)
                got = np.stack([out[b, i, x].to(torch.float64).cpu().numpy() for b, i, x in rows])
                err = np.abs(got - ref)
                assert (err <= ATOL + RTOL * np.abs(ref) + float(vp.abs().max()) * 2.0 ** (-9 if dtype == "bf16" else -12)).all(), err.max()
        finally:
            h.destroy()


@pytest.mark.parametrize("dtype", ["f16", "bf16"])
@pytest.mark.parametrize("D,row_groups", [(64, 1), (64, 2), (128, 1), (128, 2), (256, 1)])
def test_prefill_rounds_no_weight_twice(dtype, D, row_groups):
    # Scores of 0 but in the third tile: weights of 2^-3 to 2^2 at keys 320 to 351, and behind them a key 2^9 to 2^11 times the
    # reference, which ends the tile's pass when those are stored.  Each of them is read off by an output element of its own.  Its
    # error is the rounding of the weight and that of the output: rounding to p bits is uniform within half a unit, 2^(1-p) of the
    # number's power of two, so with mantissas spread evenly over their logarithm its mean square is
    # r2 = 4^(1-p) / 12 * 3 / (8 ln 2), and the two together make 2 r2; a weight that is rounded again makes 3.
    H, P, keys = 8, 640, range(320, 352)
    w = wl.Workload("once", 1, 2, H, H, D, P, 2, dtype, "uniform", False, 160)
    g = torch.Generator().manual_seed(161)
    u = lambda *n: torch.rand(*n, generator=g, dtype=torch.float64)
    unit = np.log(2.0) * np.sqrt(D)                               # of q . k for a factor of two
    q, k, v = (torch.zeros(1, P, H, D, dtype=torch.float64) for _ in range(3))
    q[0, :, :, 0] = 1 + 0.25 * u(P, H)
    k[0, keys.start:keys.stop, :, 0] = (-2.4 + 4 * u(len(keys), H)) * unit
    k[0, 383, :, 0] = (9 + 0.2 * u(H)) * unit
    for i, j in enumerate(keys):
        v[0, j, :, i] = 64                                        # (keeps the outputs among the normal numbers)
    q, k, v = (x.to(w.torch_dtype) for x in (q, k, v))
    h = sk.SegKV(w.batch, w.beams, w.heads, w.kv_heads, w.head_dim, w.prompt_len, w.steps, w.torch_dtype)
    try:
        h.set_prefill_tuning(row_groups)
        h.prefill_write(k.cuda(), v.cuda())
        out = h.prefill_sdpa(q.cuda())
        torch.cuda.synchronize()
        assert h.get_error() == 0
        got = out[0, 512:, :, :len(keys)].double().cpu()          # [row, head, key]
        s = q[0, 512:, :, None, 0].double() * k[0, :, :, 0].double().T[None] / np.sqrt(D)      # [row, head, all keys]
        e = torch.exp(s) * (torch.arange(P)[None, None] <= torch.arange(512, P)[:, None, None])
        ref = 64 * e[:, :, keys.start:keys.stop] / e.sum(2, keepdim=True)
        r2 = 4.0 ** -(7 if dtype == "bf16" else 10) / 12 * 3 / (8 * np.log(2.0))
        mean = ((got / ref - 1) ** 2).mean().item()
        assert mean <= 2.4 * r2, mean / r2
    finally:
        h.destroy()


@pytest.mark.parametrize("D,kv_heads,P", [(64, 1, 1), (64, 3, 700), (128, 5, 77), (256, 7, 130), (256, 80, 3)])
def test_prompt_store_of_odd_shapes(D, kv_heads, P):
    # blocks of whole tokens: one head, odd heads, tokens that do not divide a block's, a token larger than a block; the fused
    # prefill, whose tiles go through the tensor maps, leaves the same segment
    w = wl.Workload("store", 3, 2, kv_heads, kv_heads, D, P, 2, "f16", "uniform", False, 160)
    outs = []
    for fused in (False, True):
        h = sk.SegKV(w.batch, w.beams, w.heads, w.kv_heads, w.head_dim, w.prompt_len, w.steps, w.torch_dtype)
        kp, vp = wl.make_prompt(w, "cuda")
        qp = wl.make_prefill_query(w, "cuda")
        q, k, v = wl.make_step(w, 0, "cuda")
        if fused:
            h.prefill(kp, vp, qp)
        else:
            h.prefill_write(kp, vp)
        h.append(0, None, k, v)
        outs.append(h.decode_sdpa(q))
        torch.cuda.synchronize()
        assert h.get_error() == 0
        h.destroy()
    assert torch.equal(outs[0], outs[1])


@pytest.mark.parametrize("dtype", ["f16", "bf16"])
@pytest.mark.parametrize("D,row_groups", [(64, 1), (64, 2), (128, 1), (128, 2), (256, 1)])
def test_prefill_under_negative_slopes_keeps_the_largest_weight_exact(dtype, D, row_groups):
    # Slopes that favour OLDER keys: keys of zeros, so that the weights are the bias alone and the oldest key's is the largest, and
    # values of zeros but the oldest key's ones.  The output is that key's weight over their sum, rounded once if the weight is exact;
    # a reference left up to 2^4 behind rounds the weight too, which moves about every third output by a unit in the last place.
    # The exponents' fp32 error (2^-24 of a bias of up to 22 in log2 units, times ln 2: 1e-6) can move a result that lies as near
    # to a rounding boundary: one in 2^9 (bf16: 2^12) is allowed for, twice over.
    P = 515
    slopes = torch.tensor([-0.01, -0.015, -0.02, -0.03], dtype=torch.float32)
    w = wl.Workload("neg", 1, 2, 4, 2, D, P, 2, dtype, "uniform", True, 170)
    h = sk.SegKV(w.batch, w.beams, w.heads, w.kv_heads, w.head_dim, w.prompt_len, w.steps, w.torch_dtype)
    try:
        h.set_prefill_tuning(row_groups)
        kp, vp = (torch.zeros_like(x) for x in wl.make_prompt(w, "cuda"))
        vp[:, 0] = 1
        q = wl.make_prefill_query(w, "cuda")
        h.prefill_write(kp, vp)
        out = h.prefill_sdpa(q, None, slopes.cuda())
        torch.cuda.synchronize()
        assert h.get_error() == 0
        i = torch.arange(P, dtype=torch.float64)
        s = slopes.to(torch.float64)
        weights = torch.exp(s[:, None] * i)                       # of a key i places behind the oldest, [heads, P]
        exact = 1.0 / weights.cumsum(1)                           # of row x: all keys up to x
        got = out[0].permute(1, 0, 2).cpu()                       # [heads, P, D]
        off = got != exact.to(w.torch_dtype)[:, :, None]
        assert off.double().mean() <= 2.0 ** (-11 if dtype == "bf16" else -8), off.double().mean()
    finally:
        h.destroy()


@pytest.mark.parametrize("D,B,heads,kv_heads,P,dtype,alibi", [
    (128, 8, 30, 30, 1300, "bf16", True), (128, 8, 30, 30, 1300, "f16", False), (128, 11, 32, 32, 549, "bf16", False), (256, 16, 37, 37, 500, "bf16", True),
    (256, 16, 37, 37, 500, "f16", True), (256, 6, 56, 28, 900, "bf16", False), (64, 9, 29, 29, 2400, "f16", False), (64, 9, 29, 29, 2400, "bf16", True),
    (256, 40, 16, 16, 130, "f16", False), (128, 40, 16, 16, 100, "bf16", True)])
def test_prefill_dealing_does_not_change_an_output(D, B, heads, kv_heads, P, dtype, alibi):
    # on both sides of the rule that deals items in pairs: many requests at once against one at a time (too few for pairs)
    w = wl.Workload("deal", B, 2, heads, kv_heads, D, P, 2, dtype, "uniform", alibi, 180)
    one = wl.Workload("deal", 1, 2, heads, kv_heads, D, P, 2, dtype, "uniform", alibi, 180)
    slopes = wl.alibi_slopes(heads).cuda() if alibi else None
    h, h1 = (sk.SegKV(x.batch, x.beams, x.heads, x.kv_heads, x.head_dim, x.prompt_len, x.steps, x.torch_dtype) for x in (w, one))
    try:
        kp, vp = wl.make_prompt(w, "cuda")
        q = wl.make_prefill_query(w, "cuda")
        out, fused, ragged = (torch.full_like(q, float("nan")) for _ in range(3))
        h.prefill(kp, vp, q, fused, slopes)
        h.prefill_sdpa(q, out, slopes)
        lens = [P - (37 * b) % (P // 2) for b in range(B)]
        lens[B // 2] = P
        h.prefill_write_ragged(kp, vp, lens)
        h.prefill_sdpa(q, ragged, slopes)
        h1.set_prefill_tuning(1 if D == 256 else 2)
        for b in range(B):
            ref = torch.empty_like(q[b:b + 1])
            h1.prefill(kp[b:b + 1], vp[b:b + 1], q[b:b + 1], ref, slopes)
            assert torch.equal(out[b:b + 1], ref) and torch.equal(fused[b:b + 1], ref)
            assert torch.equal(ragged[b, :lens[b]], ref[0, :lens[b]])
        assert h.get_error() == 0 and h1.get_error() == 0
    finally:
        h.destroy()
        h1.destroy()
