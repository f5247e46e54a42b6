"""The Python binding's outputs where a program watches or changes torch's allocations."""
import pytest

import synth
from tests.gpu_util import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def loom():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2609_29219_gb300 as m
    return m


def _qkv(seed, sq):
    return [to_dev(synth.bf16_normal(seed, s, (1, 2, n, 64)))
            for s, n in ((synth.STREAM_Q, sq), (synth.STREAM_K, 200), (synth.STREAM_V, 200))]


def _calls(loom):
    """One call per entry point that allocates outputs, and how many it allocates."""
    import torch
    q, k, v = _qkv(1, 100)
    q1 = _qkv(2, 1)[0]
    flat = [x.transpose(1, 2).reshape(-1, 2, 64).contiguous() for x in (k, k, v)]
    cu = torch.tensor([0, 200], dtype=torch.int32, device="cuda")
    table = torch.zeros((1, 2), dtype=torch.int32, device="cuda")
    table[0, 1] = 1
    pages = [x.reshape(1, 2, 200, 64)[:, :, :128].reshape(2, 2, 64, 64).contiguous() for x in (k, v)]
    lens = torch.tensor([100], dtype=torch.int32, device="cuda")
    b = v[0, 0].t().contiguous()
    ws = torch.empty(1 << 20, dtype=torch.uint8, device="cuda")
    return [(lambda: loom.loom_attn_fwd(q, k, v, return_lse=True), 2),
            (lambda: loom.loom_attn_fwd_varlen(*flat, cu, cu, 200, return_lse=True), 2),
            (lambda: loom.loom_attn_decode(q1, k, v, lens, workspace=ws, return_lse=True), 2),
            (lambda: loom.loom_attn_decode_paged(q1, *pages, table, lens, workspace=ws, return_lse=True,
                                                 layout="hnd"), 2),
            (lambda: (loom.loom_gemm_bf16(k[0, 0], b),), 1)]


def test_outputs_are_the_same_whichever_way_they_are_allocated(loom, monkeypatch):
    import torch
    calls = _calls(loom)
    direct = [f() for f, _ in calls]
    monkeypatch.setattr(loom, "_empty_strided_cuda", None)
    for (f, _), a in zip(calls, direct):
        for x, y in zip(a, f()):
            assert x.shape == y.shape and x.stride() == y.stride() and x.dtype == y.dtype and torch.equal(x, y)
    loom.loom_attn_check_error()


def test_a_dispatch_mode_sees_the_outputs(loom):
    import torch
    from torch.utils._python_dispatch import TorchDispatchMode

    class Watch(TorchDispatchMode):
        def __init__(self):
            super().__init__()
            self.seen = []

        def __torch_dispatch__(self, func, types, args=(), kwargs=None):
            out = func(*args, **(kwargs or {}))
            if "empty" in str(func):
                self.seen.append(out.data_ptr())
            return out

    for f, n in _calls(loom):
        with Watch() as w:
            out = f()
        assert len(w.seen) == n and all(x.data_ptr() in w.seen for x in out)


def test_deterministic_mode_and_subclasses_take_torchs_way(loom, monkeypatch):
    import torch
    used = []
    call = loom._empty_strided_cuda
    if call is None:
        pytest.skip("this torch has no direct allocation")
    monkeypatch.setattr(loom, "_empty_strided_cuda", lambda *a: used.append(a) or call(*a))
    q, k, v = _qkv(3, 64)
    loom.loom_attn_fwd(q, k, v)
    assert len(used) == 1
    torch.use_deterministic_algorithms(True)
    try:
        loom.loom_attn_fwd(q, k, v)
    finally:
        torch.use_deterministic_algorithms(False)

    class Tagged(torch.Tensor):
        pass

    assert isinstance(loom.loom_attn_fwd(q.as_subclass(Tagged), k, v), Tagged)
    assert len(used) == 1
    loom.loom_attn_check_error()
