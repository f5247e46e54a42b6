"""GPU parity of the prefill paths that few work items take: heads packed into planes of
query rows, items of one query tile, and clusters of CTAs that share an item's KV tiles."""
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


# B, Hq, Hkv, Sq, Skv, D, causal.  CLUSTERED, one item per cluster: of 2 with a one-tile item last
# in its plane; of 2 or 4 with 1400 rows of G = 2; of 8 with a handful of rows; a share that ends
# before tile 0's diagonal; groups that are no power of two; no causal mask
CLUSTERED = [
    (1, 32, 8, 515, 3001, 128, True), (2, 6, 3, 700, 2000, 128, True), (1, 8, 1, 3, 4100, 128, True),
    (1, 8, 1, 300, 2049, 64, True), (1, 8, 8, 2048, 2048, 128, True), (1, 4, 4, 1500, 1500, 64, True),
    (1, 6, 1, 130, 2300, 128, False), (2, 4, 4, 129, 5000, 64, False), (1, 12, 1, 129, 4096, 64, True),
    (3, 16, 4, 257, 2600, 128, False),
]
SHAPES = CLUSTERED + [
    # a last item of one tile: run as one in a causal launch of one round and where it is all of
    # its plane, computed as two in more rounds and without a causal mask
    (1, 32, 1, 65, 1025, 128, True), (3, 6, 3, 288, 288, 128, True), (10, 12, 1, 280, 280, 64, True),
    (7, 32, 32, 128, 128, 64, True), (40, 8, 8, 50, 170, 128, False), (9, 16, 2, 300, 300, 64, True),
    (2, 4, 4, 3400, 300, 128, False), (3, 16, 2, 128, 128, 128, False),
]


@pytest.mark.parametrize("B,Hq,Hkv,Sq,Skv,D,causal", SHAPES)
def test_few_items(loom, B, Hq, Hkv, Sq, Skv, D, causal):
    import torch
    clustered = (B, Hq, Hkv, Sq, Skv, D, causal) in CLUSTERED
    assert (loom.loom_attn_fwd_cluster(B, Hq, Hkv, Sq, Skv, D, causal) > 1) == clustered
    q = synth.bf16_normal(1, synth.STREAM_Q, (B, Hq, Sq, D))
    k = synth.bf16_normal(1, synth.STREAM_K, (B, Hkv, Skv, D))
    v = synth.bf16_normal(1, synth.STREAM_V, (B, Hkv, Skv, D))
    o = torch.full((B, Hq, Sq, D), float("nan"), dtype=torch.bfloat16, device="cuda")
    lse = torch.full((B, Hq, Sq), float("nan"), device="cuda")
    # a second call on the same buffers gives the same bits: nothing depends on timing
    loom.loom_attn_fwd(to_dev(q), to_dev(k), to_dev(v), o, lse, causal=causal)
    first = o.clone(), lse.clone()
    loom.loom_attn_fwd(to_dev(q), to_dev(k), to_dev(v), o, lse, causal=causal)
    loom.loom_attn_check_error()
    assert torch.equal(o.view(torch.int16), first[0].view(torch.int16)) and torch.equal(lse, first[1])
    o_ref, lse_ref = oracle.attention(q, k, v, causal=causal)
    assert_parity(o_to_f64(o), o_ref, lse.cpu().numpy(), lse_ref, f"{(B, Hq, Hkv, Sq, Skv, D, causal)}")


# Clusters that take several items in turn (more items than the SMs hold clusters at once)
# of 2 and 4: the last item of a plane has one tile; causal items so short that a CTA of the
# cluster has no keys of them; both; neither
ROUNDS = [
    (1, 12, 1, 1673, 1799, 64, True, 2), (1, 12, 1, 1779, 1827, 128, True, 2), (1, 8, 1, 2503, 2595, 64, True, 2),
    (1, 16, 2, 1636, 1698, 128, True, 2), (3, 32, 32, 259, 5340, 64, False, 2), (1, 4, 4, 3392, 5663, 64, True, 4),
    (1, 4, 4, 3253, 3715, 128, True, 4),
]


@pytest.mark.parametrize("B,Hq,Hkv,Sq,Skv,D,causal,cluster", ROUNDS)
def test_several_items_per_cluster(loom, B, Hq, Hkv, Sq, Skv, D, causal, cluster):
    import torch
    assert loom.loom_attn_fwd_cluster(B, Hq, Hkv, Sq, Skv, D, causal) == cluster
    group = Hq // Hkv
    packed = group & -group  # heads whose rows share query tiles: the group's power of two
    items = B * Hq // packed * -(-Sq * packed // 256)
    assert items * cluster > torch.cuda.get_device_properties(0).multi_processor_count
    q = synth.bf16_normal(7, synth.STREAM_Q, (B, Hq, Sq, D))
    k = synth.bf16_normal(7, synth.STREAM_K, (B, Hkv, Skv, D))
    v = synth.bf16_normal(7, synth.STREAM_V, (B, Hkv, Skv, D))
    qd, kd, vd = to_dev(q), to_dev(k), to_dev(v)
    first = None
    for _ in range(30):  # the same bits each time: nothing depends on the order the CTAs run in
        o = torch.full((B, Hq, Sq, D), float("nan"), dtype=torch.bfloat16, device="cuda")
        lse = torch.full((B, Hq, Sq), float("nan"), device="cuda")
        loom.loom_attn_fwd(qd, kd, vd, o, lse, causal=causal)
        if first is None:
            first = o, lse
        assert torch.equal(o.view(torch.int16), first[0].view(torch.int16)) and torch.equal(lse, first[1])
    loom.loom_attn_check_error()
    o_ref, lse_ref = oracle.attention(q, k, v, causal=causal)
    assert_parity(o_to_f64(o), o_ref, lse.cpu().numpy(), lse_ref, f"{(B, Hq, Hkv, Sq, Skv, D, causal)}")


def test_extreme_scores_across_shares(loom):
    """Rows whose largest scores lie in one CTA's share: the other shares' weights underflow
    to zero (their partials must not bring in NaN or infinity)."""
    B, Hq, Hkv, Sq, Skv, D = 1, 4, 1, 64, 4096, 64
    q = synth.bf16_normal(2, synth.STREAM_Q, (B, Hq, Sq, D))
    k = synth.bf16_normal(2, synth.STREAM_K, (B, Hkv, Skv, D))
    v = synth.bf16_normal(2, synth.STREAM_V, (B, Hkv, Skv, D))
    kf = (k.astype(np.uint32) << 16).view(np.float32).copy()
    kf[:, :, :700] *= 60.0
    k = synth.f32_to_bf16(kf)
    assert loom.loom_attn_fwd_cluster(B, Hq, Hkv, Sq, Skv, D) > 1
    o, lse = loom.loom_attn_fwd(to_dev(q), to_dev(k), to_dev(v), return_lse=True)
    loom.loom_attn_check_error()
    o_ref, lse_ref = oracle.attention(q, k, v)
    assert_parity(o_to_f64(o), o_ref, lse.cpu().numpy(), lse_ref, "scores of one share dominate")


NAN, INF = 0x7FC0, 0x7F80  # bf16 bits


# Clusters of 2 with a first item whose tile 0 falls to one CTA, of 4, of 4
@pytest.mark.parametrize("tensor,pos,bits", [
    ("q", 5, NAN), ("q", -1, NAN), ("k", 0, NAN), ("k", 777, NAN), ("k", -1, NAN), ("k", 300, INF), ("v", 0, NAN),
    ("v", 900, INF), ("v", -1, NAN)])
@pytest.mark.parametrize("B,Hq,Hkv,Sq,Skv,D,causal", [
    (1, 8, 8, 2048, 2048, 128, True), (1, 4, 4, 1500, 1500, 64, True), (1, 8, 1, 300, 2049, 64, False)])
@pytest.mark.parametrize("steep", [False, True])
def test_nan_and_infinity(loom, steep, tensor, pos, bits, B, Hq, Hkv, Sq, Skv, D, causal):
    """NaN and infinity reach the same elements as where one CTA walks all keys of an item.
    steep: the last keys' scores are so large that the other shares' weights are 0."""
    q = synth.bf16_normal(6, synth.STREAM_Q, (B, Hq, Sq, D))
    k = synth.bf16_normal(6, synth.STREAM_K, (B, Hkv, Skv, D))
    v = synth.bf16_normal(6, synth.STREAM_V, (B, Hkv, Skv, D))
    if steep:
        kf = (k.astype(np.uint32) << 16).view(np.float32).copy()
        kf[:, :, -Skv // 16:] *= 200.0
        k = synth.f32_to_bf16(kf)
    {"q": q, "k": k, "v": v}[tensor][0, 0, pos, 3] = bits
    qd, kd, vd = to_dev(q), to_dev(k), to_dev(v)
    assert loom.loom_attn_fwd_cluster(B, Hq, Hkv, Sq, Skv, D, causal) > 1
    o, lse = loom.loom_attn_fwd(qd, kd, vd, causal=causal, return_lse=True)
    loom.loom_debug_prefill_slots(D, 2 if D == 128 else 9)  # a pinned ring depth runs one CTA per item
    try:
        o1, lse1 = loom.loom_attn_fwd(qd, kd, vd, causal=causal, return_lse=True)
    finally:
        loom.loom_debug_prefill_slots(D, 0)
    loom.loom_attn_check_error()
    a, b = o_to_f64(o), o_to_f64(o1)
    assert not np.isfinite(b).all()
    assert np.array_equal(np.isnan(a), np.isnan(b)), "elements that are NaN"
    assert np.array_equal(np.isinf(a), np.isinf(b)), "elements that are infinite"
    fin = np.isfinite(b)
    # either side rounds P and O to bf16 (2^-9 each, of at most the largest value)
    vf = (v.astype(np.uint32) << 16).view(np.float32)
    assert np.abs(a[fin] - b[fin]).max(initial=0.0) <= 2.0 ** -7 * np.abs(vf[np.isfinite(vf)]).max()
    assert np.allclose(lse.cpu().numpy(), lse1.cpu().numpy(), rtol=1e-5, atol=1e-4, equal_nan=True)


@pytest.mark.parametrize("D", [64, 128])
def test_timeout_in_a_cluster_is_reported(loom, D):
    """A K/V tile that never arrives in any CTA of a cluster: every wait runs out, the call
    reports it, and the next call is right."""
    B, Hq, Hkv, Sq, Skv = 1, 8, 2, 200, 4000
    q = synth.bf16_normal(3, synth.STREAM_Q, (B, Hq, Sq, D))
    k = synth.bf16_normal(3, synth.STREAM_K, (B, Hkv, Skv, D))
    v = synth.bf16_normal(3, synth.STREAM_V, (B, Hkv, Skv, D))
    assert loom.loom_attn_fwd_cluster(B, Hq, Hkv, Sq, Skv, D) > 1
    qd, kd, vd = to_dev(q), to_dev(k), to_dev(v)
    loom.loom_attn_check_error()
    loom.loom_debug_set_timeout_ns(50_000_000)
    try:
        loom.loom_debug_inject(2)
        loom.loom_attn_fwd(qd, kd, vd)
        with pytest.raises(loom.LoomError) as e:
            loom.loom_attn_check_error()
        assert e.value.status == 6
    finally:
        loom.loom_debug_inject(0)
        loom.loom_debug_set_timeout_ns(0)
    o, lse = loom.loom_attn_fwd(qd, kd, vd, return_lse=True)
    loom.loom_attn_check_error()
    o_ref, lse_ref = oracle.attention(q, k, v)
    assert_parity(o_to_f64(o), o_ref, lse.cpu().numpy(), lse_ref, f"after timeout D={D}")
