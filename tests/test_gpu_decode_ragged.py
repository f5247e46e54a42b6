"""GPU parity of Flash Decode where the kernels choose between two split counts by the
lengths of the batch: equal lengths take the model's, unequal ones a larger one."""
import numpy as np
import pytest

import oracle
import synth
from tests.gpu_util import assert_parity, o_to_f64, to_dev

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


def _lens(kind, B, Skv):
    lens = np.full(B, Skv, np.int64)
    if kind == "one_long":      # one sequence takes nearly all of the partials
        lens[:] = 1
        lens[B // 2] = Skv
    elif kind == "empties":
        lens[:] = np.arange(B) % 3 * (Skv // 2)
    elif kind == "ramp":
        lens = np.linspace(1, Skv, B).astype(np.int64)
    elif kind == "past":        # beyond the cache (clamped) and negative (empty)
        lens[0], lens[-1] = Skv + 1000, -5
    elif kind == "near":        # either side of the rule's line between the counts
        lens[0] -= Skv * B // 25
    elif kind == "none":
        lens[:] = 0
    return lens.astype(np.int32)


@pytest.mark.parametrize("kind", ["equal", "one_long", "empties", "ramp", "past", "near", "none"])
@pytest.mark.parametrize("B,Hq,Hkv,Skv,D,splits", [
    (2, 8, 2, 1000, 128, 0), (5, 64, 2, 3000, 64, 0), (33, 16, 16, 700, 128, 0), (32, 8, 1, 1025, 64, 0),
    (256, 4, 4, 600, 128, 0), (257, 2, 1, 300, 64, 0), (2, 1, 1, 40000, 64, 0), (16, 8, 8, 2048, 128, 0),
    (5, 4, 1, 3000, 64, 3)])
def test_ragged_splits(loom, kind, B, Hq, Hkv, Skv, D, splits):
    import torch
    q = synth.bf16_normal(4, synth.STREAM_Q, (B, Hq, 1, D))
    k = synth.bf16_normal(4, synth.STREAM_K, (B, Hkv, Skv, D))
    v = synth.bf16_normal(4, synth.STREAM_V, (B, Hkv, Skv, D))
    lens = _lens(kind, B, Skv)
    need = loom.loom_attn_decode_workspace_bytes(B, Hq, Hkv, Skv, D, splits)
    ws = torch.full((need + 256,), 0x7F, dtype=torch.uint8, device="cuda")  # bytes behind it stay as they are
    out = torch.full((B, Hq, 1, D), float("nan"), dtype=torch.bfloat16, device="cuda")
    lse = torch.full((B, Hq), float("nan"), device="cuda")
    qd, kd, vd, ld = to_dev(q), to_dev(k), to_dev(v), torch.from_numpy(lens).cuda()
    o_ref, lse_ref = oracle.attention(q, k, v, seqlens_k=np.clip(lens, 0, Skv).astype(np.int32))
    for _ in range(2):  # the first call on a workspace deals its items statically
        loom.loom_attn_decode(qd, kd, vd, ld, out, lse, ws[:need], num_splits=splits)
        loom.loom_attn_check_error()
        assert_parity(o_to_f64(out), o_ref, lse.cpu().numpy().reshape(lse_ref.shape), lse_ref, f"{kind} B={B}")
    assert bool((ws[need:] == 0x7F).all())


@pytest.mark.parametrize("B,Hkv,Skv,lo,larger", [
    (16, 8, 8192, 1.0, False), (16, 8, 8192, 0.98, False),  # one length, nearly
    (16, 8, 8192, 0.5, True), (11, 16, 5211, 0.9, True),    # uneven; too few items of one length each
    (28, 8, 2567, 0.9, False), (16, 8, 2048, 0.5, False),   # a last round with few items in it
    (16, 8, 8192, 0.0, True)])
def test_count_taken(loom, B, Hkv, Skv, lo, larger):
    """The count that the split kernel leaves behind the item counter for the merge kernel."""
    import torch
    D = 128
    n = loom.loom_attn_decode_num_splits(B, 2 * Hkv, Hkv, Skv, D)
    need = loom.loom_attn_decode_workspace_bytes(B, 2 * Hkv, Hkv, Skv, D, 0)
    ws = torch.zeros(need, dtype=torch.uint8, device="cuda")
    q = torch.randn((B, 2 * Hkv, 1, D), device="cuda", dtype=torch.bfloat16)
    kv = torch.randn((B, Hkv, Skv, D), device="cuda", dtype=torch.bfloat16)
    lens = torch.linspace(lo * Skv, Skv, B).round().int().cuda()
    loom.loom_attn_decode(q, kv, kv, lens, workspace=ws)
    loom.loom_attn_check_error()
    count = int(ws[need - 256:].view(torch.int64)[1])
    assert (n < count <= 64) if larger else count == n


def test_smaller_workspace_keeps_the_models_count(loom):
    """A workspace of the model's own count, as num_splits names it, is still enough."""
    import torch
    B, Hq, Hkv, Skv, D = 16, 8, 8, 2048, 128
    q = synth.bf16_normal(5, synth.STREAM_Q, (B, Hq, 1, D))
    k = synth.bf16_normal(5, synth.STREAM_K, (B, Hkv, Skv, D))
    v = synth.bf16_normal(5, synth.STREAM_V, (B, Hkv, Skv, D))
    lens = _lens("ramp", B, Skv)
    n = loom.loom_attn_decode_num_splits(B, Hq, Hkv, Skv, D)
    need = loom.loom_attn_decode_workspace_bytes(B, Hq, Hkv, Skv, D, n)
    assert need < loom.loom_attn_decode_workspace_bytes(B, Hq, Hkv, Skv, D, 0)
    ws = torch.full((need + 256,), 0x7F, dtype=torch.uint8, device="cuda")
    o, lse = loom.loom_attn_decode(to_dev(q), to_dev(k), to_dev(v), torch.from_numpy(lens).cuda(), workspace=ws[:need],
                                   return_lse=True)
    loom.loom_attn_check_error()
    o_ref, lse_ref = oracle.attention(q, k, v, seqlens_k=lens)
    assert_parity(o_to_f64(o), o_ref, lse.cpu().numpy().reshape(lse_ref.shape), lse_ref, "small workspace")
    assert bool((ws[need:] == 0x7F).all())


@pytest.mark.parametrize("what", ["plan 32x2x2", "plan 128x3x1", "CUDA cores", "one CTA per split", "persistent", "cluster"])
def test_other_kernels_keep_the_models_count(loom, what):
    """Kernels that do not count splits by the lengths take the model's, on the same workspace."""
    import torch
    B, Hq, Hkv, Skv, D = 16, 32, 8, 2048, 128
    n = loom.loom_attn_decode_num_splits(B, Hq, Hkv, Skv, D)
    assert (loom.loom_attn_decode_workspace_bytes(B, Hq, Hkv, Skv, D, 0) >
            loom.loom_attn_decode_workspace_bytes(B, Hq, Hkv, Skv, D, n))  # a batch that has two counts
    q = synth.bf16_normal(6, synth.STREAM_Q, (B, Hq, 1, D))
    k = synth.bf16_normal(6, synth.STREAM_K, (B, Hkv, Skv, D))
    v = synth.bf16_normal(6, synth.STREAM_V, (B, Hkv, Skv, D))
    lens = _lens("ramp", B, Skv)
    o_ref, lse_ref = oracle.attention(q, k, v, seqlens_k=lens)
    qd, kd, vd, ld = to_dev(q), to_dev(k), to_dev(v), torch.from_numpy(lens).cuda()
    try:
        if what.startswith("plan"):
            assert loom.loom_debug_decode_stage_plan(*map(int, what.split()[1].split("x")))
        elif what in ("persistent", "cluster"):
            loom.loom_debug_decode_form(2 if what == "persistent" else 3)
        else:
            loom.loom_debug_decode_tensor_cores(0 if what == "CUDA cores" else 2)
        need = loom.loom_attn_decode_workspace_bytes(B, Hq, Hkv, Skv, D, 0)
        ws = torch.zeros(need, dtype=torch.uint8, device="cuda")
        o, lse = loom.loom_attn_decode(qd, kd, vd, ld, workspace=ws, return_lse=True)
        loom.loom_attn_check_error()
    finally:
        loom.loom_debug_decode_stage_plan(0)
        loom.loom_debug_decode_form(0)
        loom.loom_debug_decode_tensor_cores(1)
    assert_parity(o_to_f64(o), o_ref, lse.cpu().numpy().reshape(lse_ref.shape), lse_ref, what)
