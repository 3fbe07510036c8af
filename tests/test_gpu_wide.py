"""Decode attention for work groups of many query columns (the tcgen05 kernel): beams x query heads per kv
head beyond what the tiled kernel takes, against the CPU oracle."""
import numpy as np
import pytest
import torch

from paper_2401_05391_b200 import segkv as sk
from paper_2401_05391_b200 import workloads as wl

from _harness import Run, all_pairs, sampled_pairs
from test_gpu_parity import run_workload, run_workload_fused

pytestmark = pytest.mark.gpu


def _w(name, batch, beams, group, hkv, D, P, steps, dtype="f16", parents="uniform", alibi=False, seed=0):
    return wl.Workload(name, batch, beams, hkv * group, hkv, D, P, steps, dtype, parents, alibi, 300 + seed)


# prompts at the edges of a key tile (64 keys; 32 at head_dim 256), responses of none, one and several tiles,
# column counts from the smallest to the full 32, one and several splits
@pytest.mark.parametrize("dtype", ["f16", "bf16"])
@pytest.mark.parametrize("D,beams,group,P,splits", [
    (64, 4, 8, 63, 0), (64, 32, 1, 129, 3), (64, 3, 7, 1, 1),
    (128, 4, 8, 64, 0), (128, 8, 4, 200, 3), (128, 17, 1, 65, 1), (128, 5, 5, 520, 0),
    (256, 4, 8, 33, 0), (256, 9, 1, 31, 1), (256, 4, 4, 150, 3)])
def test_wide_small_shapes(dtype, D, beams, group, P, splits):
    w = _w("wide", 2, beams, group, 2, D, P, 40, dtype, alibi=group == 4, seed=D + beams)
    run_workload(w, all_pairs, check_steps=(0, 1, 15, 39), splits=splits, every_step_ancestry=False)


@pytest.mark.parametrize("D,dtype", [(64, "bf16"), (128, "f16"), (256, "bf16")])
def test_wide_many_items_per_cta(D, dtype):
    # more work groups than SMs: every CTA walks several items, with rings and phases carried across them
    w = _w("many", 50, 4, 5, 8, D, 70, 9, dtype, alibi=True, seed=1)
    run_workload(w, sampled_pairs, check_steps=(0, 8), every_step_ancestry=False)
    run_workload(w, sampled_pairs, check_steps=(8,), splits=2, every_step_ancestry=False)


@pytest.mark.parametrize("layout", [None, "token_major", "seq_first"])
def test_wide_ragged_prompts_growing_cache_and_layouts(layout):
    for D, dtype in ((64, "f16"), (128, "bf16"), (256, "f16")):
        w = _w("ragged", 4, 6, 3, 2, D, 140, 21, dtype, seed=2)
        run_workload(w, all_pairs, check_steps=(0, 16, 20), prompt_lens=[140, 1, 64, 97], chunk_steps=8,
                     prompt_layout=layout, every_step_ancestry=False)


def test_wide_no_prompt_fused_call_and_redone_step():
    run_workload(_w("none", 2, 8, 4, 2, 128, 0, 30, seed=3), all_pairs, check_steps=(0, 1, 29))
    w = _w("fused", 1, 4, 8, 2, 128, 100, 12, "bf16", seed=4)
    run_workload_fused(w, all_pairs, check_steps=(0, 5, 11))
    r = Run(w)
    try:
        r.advance_to(6)
        for t in (6, 5):                           # the step before the dropped one is attended to again
            q = r.q_steps[t]
            out, _ = r.decode(q)
            r.check(out, q, t, all_pairs(w))
            r.h.truncate_last() if t == 6 else None
    finally:
        r.close()


@pytest.mark.parametrize("splits", [1, 3])
def test_wide_wait_runs_out_and_the_handle_recovers(splits):
    w = _w("wait", 2, 4, 8, 2, 128, 200, 6, "bf16", seed=5)
    r = Run(w, splits=splits)
    try:
        r.advance_to(3)
        q = r.q_steps[-1]
        out = torch.full((w.rows, w.heads, w.head_dim), float("nan"), dtype=w.torch_dtype, device="cuda")
        r.h.debug_inject(1_000_000, True)
        r.h.decode_sdpa(q, out)
        torch.cuda.synchronize()
        assert r.h.get_error() & sk.SEGKV_DEV_WAIT_LIMIT
        assert torch.isnan(out.float()).all()
        for _ in range(2):
            out2, q2 = r.decode()
            r.check(out2, q2, 3, all_pairs(w))
        assert r.h.get_error() == 0
        assert np.array_equal(r.h.get_ancestry(), r.oracle_ancestry(3))
    finally:
        r.close()


@pytest.mark.parametrize("dtype,beams,group", [("f16", 3, 3), ("bf16", 4, 4)])
def test_nine_to_sixteen_columns_on_both_sides_of_the_dispatch(dtype, beams, group):
    # head_dim 128: from 16384 prompt keys over all work groups on, these columns run on the wide kernel (which form runs
    # is asserted by test_form_of_a_step_with_nine_to_sixteen_columns)
    for P in (511, 512):
        w = _w("nt2", 4, beams, group, 8, 128, P, 20, dtype, alibi=group == 4, seed=6)
        run_workload(w, sampled_pairs, check_steps=(0, 19), every_step_ancestry=False)
        run_workload_fused(w, sampled_pairs, check_steps=(0, 7, 19))


def test_more_forced_splits_than_the_merge_has_room_for():
    w = _w("cap", 1, 4, 8, 1, 256, 100, 4, "bf16", seed=7)
    r = Run(w, splits=64)
    try:
        r.advance_to(3)
        assert r.h.get_splits() == 32                  # the most that this shape takes
        out, q = r.decode()
        r.check(out, q, 3, all_pairs(w))
    finally:
        r.close()


def _float64(r, q, t):
    """decode attention of every row in float64 on the device, from the tensors the run holds"""
    w = r.w
    W, G, D = w.beams, w.heads // w.kv_heads, w.head_dim
    anc = torch.from_numpy(r.oracle_ancestry(t)).long().cuda()
    step = torch.arange(t + 1, device="cuda")
    K, V = torch.stack(r.k_steps[:t + 1])[step, anc].double(), torch.stack(r.v_steps[:t + 1])[step, anc].double()
    out = torch.empty(w.rows, w.heads, D, dtype=torch.float64, device="cuda")
    for row in range(w.rows):
        k, v = (torch.cat([p[row // W].double(), x[row]]).transpose(0, 1) for p, x in ((r.kp, K), (r.vp, V)))
        p = torch.softmax(q[row].double().view(w.kv_heads, G, D) @ k.transpose(1, 2) / D ** 0.5, -1)
        out[row] = (p @ v).reshape(w.heads, D)
    return out


@pytest.mark.parametrize("dtype", ["f16", "bf16"])
@pytest.mark.parametrize("D,beams,group", [(64, 4, 8), (128, 5, 4), (128, 4, 8), (256, 3, 4)])
@pytest.mark.parametrize("splits", [1, 4])
@pytest.mark.parametrize("cancel", [False, True])
def test_weights_as_precise_as_the_per_beam_kernels(dtype, D, beams, group, splits, cancel):
    # The per-beam kernel works in fp32 throughout.  Ordinary values show a weight of 11 bits beside the 11 of an fp16
    # output, values that cancel nearly all of what they weigh one of 16.  Both errors end in the same rounding of the
    # output: 2 % is for the few numbers that fall on its other side.
    w = _w("precise", 2, beams, group, 2, D, 500, 8, dtype, seed=9)
    r = Run(w, splits=splits)
    try:
        if cancel:
            r.vp = r.vp[:, :1].abs().repeat(1, w.prompt_len, 1, 1).contiguous()
            r.vp[:, 1::2] *= -1
            r.h.prefill_write(r.kp, r.vp)
        r.advance_to(7)
        if cancel:
            r.v_steps = [torch.zeros_like(v) for v in r.v_steps]
            r.h.reset(keep_prompt=True)
            for t in range(8):
                r.h.append(t, r.parents_dev[t] if t else None, r.k_steps[t], r.v_steps[t])
        q = r.q_steps[-1] * (1e-3 if cancel else 1.0)
        ref = _float64(r, q, 7)
        err = {}
        for f in (r.h.decode_sdpa, r.h.decode_sdpa_rowwise):
            out = torch.empty_like(q)
            f(q, out)
            err[f.__name__] = ((out.double() - ref).norm() / ref.norm()).item()
        print(f"{dtype} D {D} {beams}x{group} S {splits} cancel {cancel}: {err}")
        assert err["decode_sdpa"] <= 1.02 * err["decode_sdpa_rowwise"], err
    finally:
        r.close()


@pytest.mark.parametrize("dtype", ["f16", "bf16"])
@pytest.mark.parametrize("D,beams,group,batch,hkv,splits", [
    (64, 4, 8, 2, 2, 1), (128, 4, 8, 2, 2, 3), (128, 4, 8, 50, 8, 1), (128, 5, 4, 2, 2, 1), (256, 4, 4, 2, 2, 1),
    (256, 4, 8, 40, 4, 2)])
def test_values_that_are_not_finite_stay_with_the_beams_that_read_them(dtype, D, beams, group, batch, hkv, splits):
    # one beam's value rows hold Inf, -Inf, NaN or numbers whose weighted sum leaves the range; parents keep the beams
    # apart.  Every column of a group that holds such a row is the per-beam kernel's, bit by bit, the others' as ever
    w = _w("apart", batch, beams, group, hkv, D, 70, 6, dtype, seed=10)
    par = np.tile(np.arange(beams, dtype=np.int32), (6, batch))
    r = Run(w, parents=par, splits=splits)
    try:
        r.advance_to(4)
        q, k, v = wl.make_step(w, 5, "cuda")
        ref = v.clone()
        bad = [(b, h) for b in range(0, batch, 3) for h in range(hkv) if (b + h) % 2 == 0]
        huge = torch.finfo(w.torch_dtype).max
        for i, (b, h) in enumerate(bad):
            v[b * beams + 1, h, i % D] = [float("inf"), float("-inf"), float("nan"), huge][i % 4]
        r.h.append(5, r.parents_dev[5], k, v)
        out, row = torch.empty_like(q), torch.empty_like(q)
        r.h.decode_sdpa(q, out)
        r.h.decode_sdpa_rowwise(q, row)
        r.h.truncate_last()
        r.h.append(5, r.parents_dev[5], k, ref)
        clean = torch.empty_like(q)
        r.h.decode_sdpa(q, clean)
        torch.cuda.synchronize()
        assert r.h.get_error() == 0 and torch.isfinite(clean.float()).all()
        nonfinite = ~torch.isfinite(row.float())
        for b in range(batch):
            for h in range(hkv):
                a, e, c = (t[b * beams:(b + 1) * beams, h * group:(h + 1) * group] for t in (out, row, clean))
                hit = (b, h) in bad and bool((~torch.isfinite(e.float())).any())
                if hit:
                    assert torch.equal(a.view(torch.int16), e.view(torch.int16)), (b, h)
                    others = [j for j in range(beams) if j != 1]
                    assert torch.isfinite(a[others].float()).all()
                elif (b, h) not in bad:
                    assert torch.equal(a, c), (b, h)
        assert bool(nonfinite.any())
    finally:
        r.close()


@pytest.mark.parametrize("D,beams", [(64, 32), (128, 32), (256, 16)])
def test_rows_of_beams_that_stay_apart_are_shared_out_evenly(D, beams):
    # Beams that never merge have beams * steps distinct rows; a share of the splits that counts on merged beams leaves
    # nearly all of them to the last one (2.5 times the per-beam kernel's time at 32 beams; evenly shared, half of it).
    w = _w("shares", 1, beams, 1, 4, D, 128, 256, "f16", seed=11)
    par = np.tile(np.arange(beams, dtype=np.int32), (256, 1))
    r = Run(w, parents=par, splits=8)
    try:
        r.advance_to(255)
        q = r.q_steps[-1]
        out, _ = r.decode(q)
        r.check(out, q, 255, [(0, 0), (0, 3)])
        t = {}
        for f in (r.h.decode_sdpa, r.h.decode_sdpa_rowwise):
            f(q, out)
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            torch.cuda._sleep(1000000)
            e[0].record()
            for _ in range(20):
                f(q, out)
            e[1].record()
            torch.cuda.synchronize()
            t[f.__name__] = e[0].elapsed_time(e[1])
        assert t["decode_sdpa"] < t["decode_sdpa_rowwise"], t
    finally:
        r.close()


@pytest.mark.parametrize("dtype,beams,group", [("f16", 3, 3), ("bf16", 4, 4)])
def test_overlap_does_not_choose_the_kernel(dtype, beams, group):
    # nine to 16 columns at head_dim 128: with dependent launch off the same kernel runs, and every bit is the same
    w = _w("overlap", 4, beams, group, 8, 128, 600, 6, dtype, alibi=group == 4, seed=12)
    r = Run(w)
    try:
        r.advance_to(5)
        out, q = r.decode()
        r.h.set_overlap(False)
        off, _ = r.decode(q)
        assert torch.equal(out.view(torch.int16), off.view(torch.int16))
    finally:
        r.close()


@pytest.mark.parametrize("batch,hkv,beams,group,P,launches", [
    (4, 8, 3, 3, 511, 1),          # too few keys for the wide kernel: the tiled kernel's fused step
    (4, 8, 3, 3, 512, 2),          # the wide kernel, behind an append of its own
    (4, 8, 4, 4, 512, 2),
    (4, 8, 16, 1, 511, 1), (4, 8, 16, 1, 512, 1),      # many beams: fused although the wide kernel could
    (4, 8, 9, 1, 1137, 2), (4, 8, 9, 1, 1138, 1),
    (37, 4, 4, 4, 128, 2), (149, 1, 4, 4, 128, 2)])    # at and above one work group per SM (tiled: unsplit, two launches)
def test_form_of_a_step_with_nine_to_sixteen_columns(batch, hkv, beams, group, P, launches):
    w = _w("forms", batch, beams, group, hkv, 128, P, 4, "f16", seed=13)
    r = Run(w)
    try:
        for t in range(3):
            n = r.h.launch_count
            _, out, q = r.step_fused()
            assert r.h.launch_count - n == launches
        r.check(out, q, 2, sampled_pairs(w, 16))
        again, _ = r.decode(q)                     # and the attention call by itself
        r.check(again, q, 2, sampled_pairs(w, 16))
    finally:
        r.close()


@pytest.mark.parametrize("dtype", ["f16", "bf16"])
@pytest.mark.parametrize("D,keys", [(64, (36, 40)), (128, (46, 54)), (256, (64, 80))])
@pytest.mark.parametrize("batch", [1, 5, 10])
def test_few_keys_run_on_the_per_beam_kernel(D, keys, dtype, batch):
    # 32 columns, 4 kv heads: 128, 640 (over four CTAs an SM) and 1280 (over eight) rows and heads; on both sides of the
    # last key count that the per-beam kernel takes: its bits up to there, the oracle's values always
    last = keys[dtype == "bf16"] if batch == 1 else keys[dtype == "bf16"] * 2 // 3
    w = _w("few", batch, 4, 8, 4, D, last - 4, 8, dtype, seed=14)
    r = Run(w)
    try:
        for t in range(6):
            _, out, q = r.step_fused()
            ref = torch.empty_like(q)
            r.h.decode_sdpa_rowwise(q, ref)
            same = torch.equal(out.view(torch.int16), ref.view(torch.int16))
            assert same == (batch < 10 and w.prompt_len + t + 1 <= last), (t, same)
            if t in (3, 4):
                r.check(out, q, t, sampled_pairs(w, 8))
    finally:
        r.close()


@pytest.mark.parametrize("dtype", ["f16", "bf16"])
@pytest.mark.parametrize("D,beams,group,P", [(64, 4, 8, 0), (128, 4, 8, 0), (256, 4, 4, 0), (128, 32, 1, 3), (64, 4, 8, 64), (256, 4, 8, 32)])
def test_wide_kernel_on_a_few_keys(dtype, D, beams, group, P):
    # a forced split count keeps the wide kernel: no prompt, hardly any keys, a prompt without a step
    w = _w("smallest", 3, beams, group, 2, D, P, 12, dtype, seed=15)
    run_workload(w, all_pairs, check_steps=(0, 1, 11), splits=1, every_step_ancestry=False)
    run_workload(w, all_pairs, check_steps=(11,), splits=2, every_step_ancestry=False)
    if P:
        r = Run(w, splits=1)
        try:
            out, q = r.decode()
            r.check(out, q, -1, all_pairs(w))
        finally:
            r.close()


@pytest.mark.parametrize("dtype", ["f16", "bf16"])
@pytest.mark.parametrize("D,beams,group", [(64, 4, 8), (128, 3, 4), (256, 3, 4)])
@pytest.mark.parametrize("splits", [1, 3])
def test_wide_scores_that_grow_from_tile_to_tile(dtype, D, beams, group, splits):
    # no bias, longer keys from tile to tile: the reference is renewed and O rescaled behind weights already worked out
    w = _w("grow", 2, beams, group, 2, D, 400, 9, dtype, seed=16)
    r = Run(w, splits=splits)
    try:
        for at, by in ((64, 4.0), (192, 2.5), (300, 2.5)):
            r.kp[:, at:] *= by
        r.h.prefill_write(r.kp, r.vp)
        r.advance_to(8)
        out, q = r.decode()
        r.check(out, q, 8, all_pairs(w))
        assert r.h.get_error() == 0
    finally:
        r.close()


@pytest.mark.parametrize("dtype", ["f16", "bf16"])
@pytest.mark.parametrize("D,batch,beams,group,hkv,P,splits", [
    (64, 3, 4, 8, 4, 130, 0), (128, 2, 4, 8, 4, 700, 0), (128, 40, 4, 8, 4, 90, 0), (128, 4, 4, 4, 8, 600, 0), (256, 3, 3, 4, 2, 300, 4)])
def test_wide_layers_queued_without_waiting(dtype, D, batch, beams, group, hkv, P, splits):
    # Three layers stepped in turn, nothing waited for on the host: a launch starts, and asks for its prompt, while the one
    # before drains.  Against the oracle, and bit by bit against plain stream order, a second run, a captured step that is
    # replayed, and layers that share one beam-index table.
    w = _w("queued", batch, beams, group, hkv, D, P, 12, dtype, alibi=group == 8, seed=17)
    par = wl.make_parents(w)
    runs = {}
    try:
        for name in ("plain", "again", "order", "shared"):
            rs = runs[name] = [Run(w.scaled(index=170 + i), parents=par, splits=splits) for i in range(3)]
            if name == "shared":
                for r in rs[1:]:
                    r.h.share_index(rs[0].h)
            for r in rs:
                r.h.set_overlap(name != "order")
        steps = [[wl.make_step(r.w, t, "cuda") for r in runs["plain"]] for t in range(w.steps)]
        torch.cuda.synchronize()
        outs = {}
        for name, rs in runs.items():
            outs[name] = torch.full((w.steps, 3, w.rows, w.heads, D), float("nan"), dtype=w.torch_dtype, device="cuda")
            torch.cuda.synchronize()
            for t in range(w.steps):
                for i, r in enumerate(rs):
                    q, k, v = steps[t][i]
                    r.h.decode_step(t, r.parents_dev[t] if t else None, k, v, q, outs[name][t, i], r.slopes)
            torch.cuda.synchronize()
            assert all(r.h.get_error() == 0 for r in rs)
        for name in ("again", "order", "shared"):
            assert torch.equal(outs[name], outs["plain"]), name
        rs, last = runs["plain"], w.steps - 1
        for r, i in ((rs[0], 0), (rs[2], 2)):
            r.q_steps, r.k_steps, r.v_steps = (list(x) for x in zip(*[steps[t][i] for t in range(w.steps)]))
            for t in (0, 5, last):
                r.check(outs["plain"][t, i], r.q_steps[t], t, sampled_pairs(r.w, 8))
        again = torch.empty_like(outs["plain"][last])

        def redo():
            for i, r in enumerate(rs):
                if r.h.steps > last:
                    r.h.truncate_last()
                r.h.decode_step(last, r.parents_dev[last], steps[last][i][1], steps[last][i][2], steps[last][i][0], again[i], r.slopes)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            redo()
        for _ in range(3):
            again.fill_(float("nan"))
            g.replay()
            g.replay()
            torch.cuda.synchronize()
            assert torch.equal(again, outs["plain"][last])
        assert all(r.h.get_error() == 0 for r in rs)
    finally:
        for rs in runs.values():
            for r in reversed(rs):
                r.close()


# the partials of a work group land in the prompt ring (128 KB) at once where they fit and the CTA has no further items: the
# largest counts that fit, one more, columns that do not fill the padding, and CTAs with and without further items
@pytest.mark.parametrize("D,beams,group,B,kv_heads,splits", [
    (128, 4, 8, 1, 2, 8), (128, 4, 8, 1, 2, 9), (128, 3, 6, 1, 1, 14), (128, 3, 6, 1, 1, 15), (128, 3, 6, 1, 1, 40), (64, 4, 8, 1, 2, 16), (64, 4, 8, 1, 2, 17),
    (256, 4, 8, 1, 1, 4), (256, 4, 8, 1, 1, 5), (128, 4, 8, 20, 4, 3)])
def test_split_merge_in_the_prompt_ring(D, beams, group, B, kv_heads, splits):
    w = wl.Workload("land", B, beams, kv_heads * group, kv_heads, D, 700, 4, "f16", "uniform", False, 620 + splits)
    run_workload(w, sampled_pairs, check_steps=(0, 3), splits=splits, every_step_ancestry=False)
