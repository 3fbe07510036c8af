"""The decode loop's calls through the extension module: what it takes runs as the general path does, what it does not take
is refused by that path as before."""
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
    h.decode_step(0, None, k, v, torch.nn.Parameter(q, requires_grad=False))     # a subclass takes the general path
    assert h.steps == 1
    h.truncate_last()
    assert h.steps == 0
    h.destroy()
    with pytest.raises(sk.SegKVError):
        h.append(0, None, k, v)
