"""Several layers' caches driven in turn on one stream, as a model does: by the time a layer's
attention is launched, the launches that wrote its rows, tables and lists are older than its
predecessor in the stream, so the kernel fetches them ahead of its grid-dependency wait (into the
stage set aside for the first response tile).  Single-handle tests never reach those paths; the
results must be the same bits either way and must match the oracle."""
import numpy as np
import pytest
import torch

from paper_2401_05391_b200 import segkv as sk
from paper_2401_05391_b200 import workloads as wl

from _harness import Run, all_pairs, sampled_pairs

pytestmark = pytest.mark.gpu


def layers_of(w, n, **kw):
    par = wl.make_parents(w)
    return [Run(w.scaled(index=w.index + 11 * i), parents=par, **kw) for i in range(n)]


@pytest.mark.parametrize("tile,splits,combine", [(0, 0, 0), (64, 3, 1), (64, 4, 2), (32, 8, 2), (32, 4, 2), (32, 2, 1),
                                                 (32, 5, 0), (64, 1, 0)])
def test_separate_calls_over_three_layers(tile, splits, combine):
    w = wl.Workload("il", 2, 4, 8, 4, 128, 200, 40, "f16", "uniform", False, 300)
    ls = layers_of(w, 3, tile=tile, splits=splits, combine=combine)
    # the first layer once more, alone and without dependent launch: nothing is fetched ahead there
    ref = Run(w.scaled(index=w.index), parents=ls[0].parents, tile=tile, splits=splits, combine=combine)
    forced = tile != 0 and splits != 0 and combine != 0
    if forced:
        ref.h.set_overlap(False)
    try:
        for t in range(w.steps):
            for r in ls:
                r.append_next()
            outs = [r.decode() for r in ls]          # each attention follows another layer's launch
            if t in (0, 1, 7, 20, 39):
                for r, (out, q) in zip(ls, outs):
                    r.check(out, q, t, all_pairs(w))
            # the same layer driven alone (its append is the attention's predecessor): same bits
            ref.append_next()
            out_ref, _ = ref.decode()
            if forced:
                assert torch.equal(out_ref.view(torch.int16), outs[0][0].view(torch.int16)), f"step {t}"
        for r in ls + [ref]:
            assert r.h.get_error() == 0
    finally:
        for r in ls + [ref]:
            r.close()


@pytest.mark.parametrize("dtype,D,B,W,steps,tile,splits,combine", [
    ("f16", 128, 1, 4, 40, 0, 0, 0),        # automatic: the small clustered form
    ("f16", 128, 2, 4, 70, 32, 4, 2),       # a response share of several 32-key tiles
    ("f16", 128, 2, 4, 40, 32, 8, 2),
    ("bf16", 64, 2, 3, 40, 32, 2, 2),       # three beams: four lanes per step, one idle
    ("f16", 128, 1, 8, 40, 32, 4, 1),       # eight beams, workspace merge
    ("bf16", 128, 2, 4, 40, 64, 4, 1),
    ("f16", 256, 1, 4, 40, 0, 4, 0),
    ("f16", 128, 1, 4, 150, 64, 1, 0),      # one CTA per work group: many windows, many tiles
])
def test_fused_steps_over_three_layers(dtype, D, B, W, steps, tile, splits, combine):
    w = wl.Workload("ilf", B, W, 4, 4, D, 260, steps, dtype, "uniform", dtype == "bf16", 310 + D)
    ls = layers_of(w, 3, tile=tile, splits=splits, combine=combine)
    ref = Run(w.scaled(index=w.index), parents=ls[0].parents, tile=tile, splits=splits, combine=combine)
    forced = tile != 0 and splits != 0 and combine != 0
    if forced:
        ref.h.set_overlap(False)
    try:
        for t in range(w.steps):
            outs = [r.step_fused() for r in ls]
            if t in (0, 1, 2, 17, 39, 69, 149):
                for r, (_, out, q) in zip(ls, outs):
                    r.check(out, q, t, all_pairs(w))
                    assert np.array_equal(r.h.get_ancestry(), r.oracle_ancestry(t))
            # (alone, the rows come after the wait in the new parents' order, so the low bits may differ:
            # both are compared with the oracle only)
            _, out_ref, q_ref = ref.step_fused()
            if t in (0, 1, 2, 17, 39, 69, 149):
                ref.check(out_ref, q_ref, t, all_pairs(w))
        for r in ls + [ref]:
            assert r.h.get_error() == 0
    finally:
        for r in ls + [ref]:
            r.close()


@pytest.mark.parametrize("B,heads,kv_heads,P", [(2, 8, 4, 200), (5, 64, 64, 300), (2, 32, 4, 512)])
def test_appends_in_a_row_and_attention_behind_them(B, heads, kv_heads, P):
    # Appends let their successors go at once, so behind several of them only what was complete before the first may be read
    # ahead: the small form, more work groups than SMs and the wide kernel, against the same calls with a wait after each.
    w = wl.Workload("chain", B, 4, heads, kv_heads, 128, P, 24, "f16", "uniform", False, 310)
    ls, refs = layers_of(w, 3), layers_of(w, 3)
    try:
        for t in range(w.steps):
            for r in ls:
                r.append_next()
            outs = [r.decode()[0] for r in (ls if t % 2 else ls[::-1])]
            for r in refs:
                r.append_next()
                torch.cuda.synchronize()
            for r, out in zip(refs if t % 2 else refs[::-1], outs):
                ref = r.decode()[0]
                torch.cuda.synchronize()
                assert torch.equal(out.view(torch.int16), ref.view(torch.int16)), f"step {t}"
        for r in ls + refs:
            assert r.h.get_error() == 0
    finally:
        for r in ls + refs:
            r.close()


@pytest.mark.parametrize("D,B,W,heads,kv_heads,P,ragged", [
    (64, 3, 4, 8, 8, 300, False), (64, 3, 4, 8, 8, 300, True), (64, 3, 8, 8, 8, 300, True), (128, 5, 4, 8, 4, 300, True),
    (128, 6, 4, 40, 40, 813, False), (128, 6, 4, 40, 40, 814, False)])          # 99.9 and 100.02 MB of prompt
def test_appends_that_release_at_once_and_after_their_wait(D, B, W, heads, kv_heads, P, ragged):
    # three layers' appends in a row, then their attentions, and layer by layer: the bits of calls that are each waited for
    w = wl.Workload("rel", B, W, heads, kv_heads, D, P, 4, "f16", "uniform", False, 340)
    par = torch.from_numpy(wl.make_parents(w)).cuda()
    kp, vp = wl.make_prompt(w, "cuda")
    steps = [[wl.make_step(w.scaled(index=w.index + 11 * i), t, "cuda") for i in range(3)] for t in range(w.steps)]
    outs = {}
    for mode in ("plain", "rows", "layers"):
        hs = [sk.SegKV(B, W, heads, kv_heads, D, P, w.steps, w.torch_dtype) for _ in range(3)]
        outs[mode] = []
        for h in hs:
            if ragged:
                h.prefill_write_ragged(kp, vp, [P - (61 * b) % (P // 2) for b in range(B)])
            else:
                h.prefill_write(kp, vp)
        for t in range(w.steps):
            if mode == "rows":
                for h, (q, k, v) in zip(hs, steps[t]):
                    h.append(t, par[t] if t else None, k, v)
                outs[mode] += [h.decode_sdpa(q) for h, (q, k, v) in zip(hs, steps[t])]
            else:
                for h, (q, k, v) in zip(hs, steps[t]):
                    h.append(t, par[t] if t else None, k, v)
                    if mode == "plain":
                        torch.cuda.synchronize()
                    outs[mode].append(h.decode_sdpa(q))
                    if mode == "plain":
                        torch.cuda.synchronize()
        torch.cuda.synchronize()
        assert all(h.get_error() == 0 for h in hs)
        for h in hs:
            h.destroy()
    for x, y, z in zip(*(outs[m] for m in ("plain", "rows", "layers"))):
        assert torch.equal(x, y) and torch.equal(x, z)
