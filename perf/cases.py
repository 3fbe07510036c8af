"""Performance cases of the segment-KV attention library: what a decoder's attention layers ask of it.

A case describes a stack of equal attention layers and one piece of a model's work on it:

  decode    one decode step of every layer from device tensors (``SegKV.decode_step``): the inner loop of
            generation, with the cache as it is after ``steps - 1`` steps;
  rope      the same step for a model with rotary embeddings whose layers share one beam-index table:
            ``append_rope`` and ``decode_sdpa`` per layer, the first layer leading (``share_index``);
  host      the same step for a program that keeps its activations in pinned host memory
            (``LayerStack.step`` and a wait for the stream, as the outputs are read on the host);
  prefill   the prompt of every layer (``prefill``, or ``prefill_write_ragged`` + ``prefill_sdpa`` when the
            requests' lengths differ), then the first decode step, which reads what was stored;
  generate  a whole short generation: prefill, then ``steps`` decode steps, layer by layer.

Activations are N(0,1) values in the storage type (rotary embedding already applied unless the case
applies it), beam parents uniform draws, or, for ``half_identity``, kept as they are in every other step.
"""
import math
import random

import numpy as np
import torch

from paper_2401_05391_b200 import workloads
from paper_2401_05391_b200.segkv import LayerStack, SegKV


def _case(kind, batch, beams, heads, kv_heads, head_dim, prompt, steps, layers, dtype="f16", alibi=False,
          ragged=False, chunk=0, rope="", parents="uniform", name=None):
    c = dict(kind=kind, batch=batch, beams=beams, heads=heads, kv_heads=kv_heads, head_dim=head_dim, prompt=prompt,
             steps=steps, layers=layers, dtype=dtype, alibi=alibi, ragged=ragged, chunk=chunk, rope=rope,
             parents=parents)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest use: a toy model (the "tiny" workload's layer) generating eight tokens; all calls and launches
        _case("generate", 1, 4, 4, 4, 64, 32, 8, 2, name="generate_tiny"),
        # one token of one request on a 7B model: 32 Llama2-7B layers, the interactive case
        _case("decode", 1, 4, 32, 32, 128, 1024, 128, 32, name="decode_llama2_7b"),
        # the same token when the rest of the model lives on the host side
        _case("host", 1, 4, 32, 32, 128, 1024, 128, 32, name="host_llama2_7b"),
        # a small serving batch of unequal, odd prompts on Llama2-13B layers with the cache growing in chunks
        _case("decode", 6, 4, 40, 40, 128, 1237, 77, 8, ragged=True, chunk=16, name="decode_13b_ragged"),
        # a rotary model with 256-wide heads, one beam-index table for all layers
        _case("rope", 16, 4, 16, 16, 256, 1024, 128, 4, rope="interleaved", name="rope_gptj_6b"),
        # the large serving batch: 4.3 GB of keys and values read in one step of one layer
        _case("decode", 64, 4, 56, 56, 128, 2048, 256, 1, parents="half_identity", name="decode_opt_30b"),
        # many heads, bf16, ALiBi
        _case("decode", 32, 4, 112, 112, 128, 1024, 128, 1, dtype="bf16", alibi=True, name="decode_bloom_176b"),
        # grouped-query attention under beam search: eight query heads per kv head times four beams
        _case("decode", 8, 4, 32, 4, 128, 2048, 64, 4, dtype="bf16", name="decode_gqa_8x4"),
        # the prompt of one interactive request
        _case("prefill", 1, 4, 32, 32, 128, 1024, 1, 8, name="prefill_llama2_7b"),
        # the prompts of the large batch
        _case("prefill", 64, 4, 56, 56, 128, 2048, 1, 1, name="prefill_opt_30b"),
        # bf16 and ALiBi prompts
        _case("prefill", 32, 4, 112, 112, 128, 1024, 1, 1, dtype="bf16", alibi=True, name="prefill_bloom_176b"),
        # prompts of unequal, odd lengths, 256-wide heads
        _case("prefill", 16, 4, 16, 16, 256, 1003, 1, 2, ragged=True, name="prefill_gptj_ragged"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    """One more case of the ranges above: every size between the smallest and the largest listed."""
    kind = rng.choice(["decode"] * 4 + ["rope"] * 2 + ["host"] + ["prefill"] * 4 + ["generate"])
    head_dim = rng.choice([64, 128, 128, 256])
    group = rng.choice([1, 1, 1, 2, 4, 8])
    kv_heads = _log(rng, 4, 112 if group == 1 else 16)
    beams = min(rng.choice([1, 2, 3, 4, 4, 5, 8]), 32 // group)
    batch, prompt = _log(rng, 1, 64), _log(rng, 32, 4096)
    steps = 1 if kind == "prefill" else _log(rng, 2, 24 if kind == "generate" else 256)
    layers = _log(rng, 1, 32)
    dtype = rng.choice(["f16", "bf16"])
    alibi = kind not in ("rope", "host") and rng.random() < 0.25
    ragged = kind in ("decode", "prefill") and batch > 1 and rng.random() < 0.4
    chunk = 16 if kind == "decode" and rng.random() < 0.3 else 0
    rope = rng.choice(["half", "interleaved"]) if kind == "rope" else ""

    def made():
        return _case(kind, batch, beams, kv_heads * group, kv_heads, head_dim, prompt, steps, layers, dtype, alibi,
                     ragged, chunk, rope)

    # no more than the largest listed cases: about a third of their bytes, operations and outputs
    while True:
        w = work(made())
        wide = group if beams * group > 16 or (head_dim == 256 and beams * group > 8) else 1
        if w["bytes"] * wide <= (1.5e9 if kind != "host" else 3e8) and w["flops"] <= 1.2e12:
            return made()
        if layers > 1:
            layers = layers // 2
        elif batch > 1:
            batch = batch * 2 // 3
        else:
            prompt = prompt * 2 // 3


def _lens(case):
    """Prompt lengths of a ragged batch: spread evenly between a quarter of the longest and the longest."""
    p = case["prompt"]
    if not case["ragged"]:
        return [p] * case["batch"]
    out = [max(1, int(p * (0.25 + 0.75 * ((b + 1) * 0.6180339887 % 1.0)))) for b in range(case["batch"])]
    out[case["batch"] // 2] = p
    return out


def _parents(case, seed):
    w = workloads.Workload("case", case["batch"], case["beams"], case["heads"], case["kv_heads"], case["head_dim"],
                           case["prompt"], case["steps"], case["dtype"], case["parents"], case["alibi"], 0)
    return workloads.make_parents(w, seed)


def _distinct_rows(case):
    """Distinct response rows that one request's beams read at the last step (a typical draw of the parents)."""
    W, T = case["beams"], case["steps"]
    par = _parents(dict(case, batch=1), 7)
    path, n = np.arange(W), W
    for s in range(T - 1, 0, -1):
        path = par[s][path]
        n += len(set(path.tolist()))
    return n


def _seen_keys(case, step):
    """Prompt and response rows one layer reads at `step` (0-based), summed over the requests."""
    return sum(_lens(case)) + case["batch"] * min(_distinct_rows(case), (step + 1) * case["beams"])


def work(case):
    B, W, H, Hkv, D, L = (case[k] for k in ("batch", "beams", "heads", "kv_heads", "head_dim", "layers"))
    lens, rows = _lens(case), B * W
    token, qtok = 2 * Hkv * D * 2, H * D * 2                     # K and V of one token; one query (or output) row

    def step(t):
        keys = sum(lens) + B * (t + 1)
        # keys and values once, the query and the new rows in, the new rows and the output back
        return _seen_keys(case, t) * token + rows * (2 * token + 2 * qtok), 4.0 * D * H * W * keys

    def prompt():
        n = sum(lens)
        return n * (2 * token + 2 * qtok), 4.0 * D * H * sum(p * (p + 1) / 2 for p in lens)

    parts = []
    if case["kind"] in ("prefill", "generate"):
        parts.append(prompt())
    if case["kind"] == "generate":
        parts += [step(t) for t in range(case["steps"])]
    else:
        parts.append(step(case["steps"] - 1))
    return {"bytes": L * sum(b for b, _ in parts), "flops": L * sum(f for _, f in parts)}


def tolerance(case):
    # Measured against a float64 evaluation of the same 16-bit inputs (head_dim 64 to 256, prompts of 33 to 4096,
    # with and without ALiBi): fp16 up to 2.7e-4 (2-norm) and 4.2e-3 (largest element), bf16 up to 2.0e-3 and
    # 1.5e-2, all of it the rounding of the softmax weights and of the outputs.  Stated: four times that.
    return {"rel": 1.1e-3, "max": 1.7e-2} if case["dtype"] == "f16" else {"rel": 8e-3, "max": 6e-2}


class _State:
    pass


def prepare(case, seed):
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    dt = torch.float16 if case["dtype"] == "f16" else torch.bfloat16
    B, W, H, Hkv, D = (case[k] for k in ("batch", "beams", "heads", "kv_heads", "head_dim"))
    P, T, L, kind = case["prompt"], case["steps"], case["layers"], case["kind"]
    rows = B * W

    def normal(*shape):
        return torch.randn(shape, generator=g, device=dev, dtype=dt)

    s = _State()
    s.kind, s.T, s.L, s.ragged = kind, T, L, case["ragged"]
    s.lens = _lens(case)
    s.slopes = workloads.alibi_slopes(H).to(dev) if case["alibi"] else None
    par = torch.from_numpy(_parents(case, seed))
    s.parents = [None] + [par[t].to(dev) for t in range(1, T)]
    if case["rope"]:
        s.style = case["rope"]
        s.cos, s.sin = (t.to(dev) for t in workloads.rope_tables(P + T, D))
    s.layers = [SegKV(B, W, H, Hkv, D, P, T, dt, chunk_steps=case["chunk"]) for _ in range(L)]
    if kind == "rope":
        for h in s.layers[1:]:
            h.share_index(s.layers[0])

    if kind in ("prefill", "generate"):
        s.k, s.v = [normal(B, P, Hkv, D) for _ in range(L)], [normal(B, P, Hkv, D) for _ in range(L)]
        s.q = [normal(B, P, H, D) for _ in range(L)]
        s.out = [torch.zeros(B, P, H, D, device=dev, dtype=dt) for _ in range(L)]
        s.kn, s.vn = normal(T, L, rows, Hkv, D), normal(T, L, rows, Hkv, D)
        s.qn, s.outn = normal(T, L, rows, H, D), torch.zeros(T, L, rows, H, D, device=dev, dtype=dt)
        return s

    # the cache as it stands before the step that is timed: the prompt and T - 1 steps
    for h in s.layers:
        k, v = normal(B, P, Hkv, D), normal(B, P, Hkv, D)
        if s.ragged:
            h.prefill_write_ragged(k, v, s.lens)
        else:
            h.prefill_write(k, v)
        del k, v
    for t in range(T - 1):
        k, v = normal(L, rows, Hkv, D), normal(L, rows, Hkv, D)
        for h, kl, vl in zip(s.layers, k, v):
            h.append(t, s.parents[t], kl, vl)
    s.k, s.v, s.q = normal(L, rows, Hkv, D), normal(L, rows, Hkv, D), normal(L, rows, H, D)
    s.out = torch.zeros(L, rows, H, D, device=dev, dtype=dt)
    if kind == "host":
        total, off = s.layers[0].host_pack_layout()
        block = torch.zeros(L, total, dtype=torch.uint8).pin_memory()
        s.out = torch.zeros(L, rows, H, D, dtype=dt).pin_memory()

        def put(layer, at, t):
            b = t.detach().contiguous().cpu().view(-1).view(torch.uint8)
            block[layer, at:at + b.numel()] = b

        for i in range(L):
            if T > 1:
                put(i, off[0], s.parents[T - 1])
            put(i, off[2], s.k[i])
            put(i, off[3], s.v[i])
            put(i, off[4], s.q[i])
        s.block = block
        s.stack = LayerStack(s.layers, [block[i] for i in range(L)], [s.out[i] for i in range(L)])
    # per-layer views, as a model holds its layers' activations
    s.kl, s.vl, s.ql, s.outl = (list(t.unbind(0)) for t in (s.k, s.v, s.q, s.out))
    return s


def run(s):
    t = s.T - 1
    if s.kind == "host":
        s.stack.step(t, redo=True)
        torch.cuda.current_stream().synchronize()                 # the outputs are read on the host
        return s.out
    if s.kind == "decode":
        for h, k, v, q, out in zip(s.layers, s.kl, s.vl, s.ql, s.outl):
            if h.steps > t:
                h.truncate_last()                                 # the step again
            h.decode_step(t, s.parents[t], k, v, q, out, s.slopes)
        return s.out
    if s.kind == "rope":
        for h in s.layers:
            if h.steps > t:
                h.truncate_last()
        for h, k, v, q, out in zip(s.layers, s.kl, s.vl, s.ql, s.outl):
            h.append_rope(t, s.parents[t], k, v, s.cos, s.sin, s.style)
            h.decode_sdpa(q, out)
        return s.out
    for i, h in enumerate(s.layers):
        if s.ragged:
            h.prefill_write_ragged(s.k[i], s.v[i], s.lens)
            h.prefill_sdpa(s.q[i], s.out[i], s.slopes)
        else:
            h.prefill(s.k[i], s.v[i], s.q[i], s.out[i], s.slopes)
    for t in range(s.T):
        for i, h in enumerate(s.layers):
            h.decode_step(t, s.parents[t], s.kn[t, i], s.vn[t, i], s.qn[t, i], s.outn[t, i], s.slopes)
    return s.out + [s.outn]
