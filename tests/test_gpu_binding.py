"""The decode loop's calls through the extension module: what it takes runs as the general path does, what it does not take
is refused by that path as before."""
import threading

import pytest
import torch

from paper_2401_05391_b200 import segkv as sk
from paper_2401_05391_b200 import workloads as wl

pytestmark = pytest.mark.gpu


def handle(w):
    h = sk.SegKV(w.batch, w.beams, w.heads, w.kv_heads, w.head_dim, w.prompt_len, w.steps, w.torch_dtype)
    h.prefill_write(*wl.make_prompt(w, "cuda"))
    return h


@pytest.mark.parametrize("dtype", ["f16", "bf16"])
def test_same_results_with_and_without_a_stream_argument(dtype):
    w = wl.Workload("hot", 2, 4, 8, 4, 64, 50, 4, dtype, "uniform", True, 400)
    par = torch.from_numpy(wl.make_parents(w)).cuda()
    slopes = wl.alibi_slopes(w.heads).cuda()
    a, b = handle(w), handle(w)
    st = torch.cuda.current_stream()
    for t in range(w.steps):
        q, k, v = wl.make_step(w, t, "cuda")
        p = par[t] if t else None
        if t % 2:
            x, y = a.decode_step(t, p, k, v, q, None, slopes), b.decode_step(t, p, k, v, q, None, slopes, stream=st)
        else:
            a.append(t, p, k, v)
            b.append(t, p, k, v, stream=st)
            x, y = a.decode_sdpa(q, None, slopes), b.decode_sdpa(q, None, slopes, stream=st)
        torch.cuda.synchronize()
        assert torch.equal(x, y) and a.steps == b.steps == t + 1
    a.destroy()
    b.destroy()


def test_refused_arguments():
    w = wl.Workload("hot", 2, 4, 8, 4, 64, 50, 4, "f16", "uniform", False, 401)
    h = handle(w)
    q, k, v = wl.make_step(w, 0, "cuda")
    for bad in (q[:, :4], q.float(), q.cpu(), q.transpose(0, 1), torch.zeros(8, 8, 128, dtype=q.dtype, device="cuda")[..., ::2]):
        with pytest.raises(ValueError):
            h.decode_step(0, None, k, v, bad)
    with pytest.raises(ValueError):
        h.append(0, None, k[..., :32], v)
    for step in (1, -1):
        with pytest.raises(sk.SegKVError):
            h.append(step, torch.zeros(8, dtype=torch.int32, device="cuda"), k, v)
    assert h.steps == 0
    h.decode_step(0, None, k, v, torch.nn.Parameter(q, requires_grad=False))     # (plain to torch's exact-type test)
    assert h.steps == 1
    h.truncate_last()
    assert h.steps == 0
    h.destroy()
    with pytest.raises(sk.SegKVError):
        h.append(0, None, k, v)


class Marked(torch.Tensor):
    """A tensor subclass of the caller's own."""


def test_what_the_extension_takes_and_what_it_leaves():
    w = wl.Workload("hot", 2, 4, 8, 4, 64, 50, 4, "f16", "uniform", True, 402)
    h, ref = handle(w), handle(w)
    slopes = wl.alibi_slopes(w.heads).cuda()
    q, k, v = wl.make_step(w, 0, "cuda")
    out = torch.empty_like(q)
    hot = h._hot
    assert hot is not None                        # built with the library
    mk = q.as_subclass(Marked)
    assert hot.decode_step(0, None, k, v, mk, out, slopes) is None and hot.decode_sdpa(q, out.as_subclass(Marked), slopes) is None
    assert hot.append(0, None, k.as_subclass(Marked), v) is None and hot.append(0.0, None, k, v) is None
    assert hot.append(True, None, k, v) is None and hot.append(2 ** 40, None, k, v) is None
    assert hot.decode_step(0, None, k, v, q[:, :4], out, slopes) is None and hot.decode_sdpa(q, out, slopes.double()) is None
    assert hot.decode_sdpa(torch.empty(q.shape, dtype=q.dtype, device="meta"), out, slopes) is None
    assert h.steps == hot.steps() == 0
    assert hot.append(0, None, k, v) == 0 and hot.decode_sdpa(q, out, slopes) == 0 and hot.steps() == 1
    assert hot.truncate_last() == 0
    assert hot.decode_step(0, None, k, v, q, out, slopes) == 0
    y = ref.decode_step(0, None, k.as_subclass(Marked), v, mk, None, slopes)      # the general path takes them as ever
    torch.cuda.synchronize()
    assert torch.equal(out, y) and h.steps == ref.steps == 1
    h.destroy()
    ref.destroy()


def test_without_the_extension(monkeypatch):
    w = wl.Workload("hot", 2, 4, 8, 4, 64, 50, 3, "bf16", "uniform", False, 403)
    par = torch.from_numpy(wl.make_parents(w)).cuda()
    a = handle(w)
    monkeypatch.setattr(sk, "_hot_module", lambda: None)
    b = handle(w)
    assert b._hot is None
    for t in range(w.steps):
        q, k, v = wl.make_step(w, t, "cuda")
        x, y = (h.decode_step(t, par[t] if t else None, k, v, q) for h in (a, b))
        torch.cuda.synchronize()
        assert torch.equal(x, y) and a.steps == b.steps == t + 1
    b.truncate_last()
    assert b.steps == w.steps - 1
    a.destroy()
    b.destroy()


def test_side_streams_and_threads():
    # calls on the current stream of the thread that makes them: a side stream behind a slow kernel, and two threads at once
    w = wl.Workload("hot", 2, 4, 8, 4, 128, 300, 24, "f16", "uniform", False, 404)
    par = torch.from_numpy(wl.make_parents(w)).cuda()
    steps = [wl.make_step(w, t, "cuda") for t in range(w.steps)]
    prompt = wl.make_prompt(w, "cuda")

    def run(h, outs):
        h.prefill_write(*prompt)
        for t, (q, k, v) in enumerate(steps):
            if t % 2:
                outs.append(h.decode_step(t, par[t], k, v, q))
            else:
                h.append(t, par[t] if t else None, k, v)
                outs.append(h.decode_sdpa(q))

    hs = [sk.SegKV(w.batch, w.beams, w.heads, w.kv_heads, w.head_dim, w.prompt_len, w.steps, w.torch_dtype) for _ in range(4)]
    results = [[] for _ in hs]
    torch.cuda.synchronize()
    run(hs[0], results[0])
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        torch.cuda._sleep(400_000_000)
        run(hs[1], results[1])
        done = torch.cuda.Event()
        done.record()
        assert not done.query()                   # queued on the side stream, behind the sleep

    def worker(i):
        with torch.cuda.stream(torch.cuda.Stream()):
            run(hs[i], results[i])

    threads = [threading.Thread(target=worker, args=(i,)) for i in (2, 3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    for r in results[1:]:
        assert len(r) == w.steps and all(torch.equal(x, y) for x, y in zip(r, results[0]))
    assert all(h.get_error() == 0 for h in hs)
    for h in hs:
        h.destroy()
