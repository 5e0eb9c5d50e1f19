"""The one-launch segmenter (calls of few layers) against the separate launches, which the parity tests hold to the oracle.

A context created with clusters of at most eight CTAs segments in separate launches and runs the map pass as one; everything
in between is integer arithmetic, so maps, thresholds, spans, votes, representatives and outputs have to agree to the bit."""
import os

import numpy as np
import pytest
import torch

from oracle import ltri_oracle as orc
from paper_2412_04757_b200 import binding
from tests.test_gpu_segmenter import GOLDEN, block_map

pytestmark = pytest.mark.gpu

# call sizes around the edges of the row blocks (32 per call), of the 128-entry row groups and of the rounds' key counts
# (a context of this window and chunk keeps nine regions pending; eight of the last sequence leave the window in one call)
EDGES = [[1024, 1023, 1, 512, 2, 993, 17], [513, 700, 511, 16, 257, 481, 31], [256, 1024, 255, 32, 129, 128, 33],
         [640, 65, 64, 1000, 127, 15, 416], [64, 40, 33, 32, 31, 17, 16, 8, 1024, 300, 128]]


def pair(monkeypatch, **kw):
    p = dict(n_layers=2, n_q_heads=8, n_kv_heads=2, max_tokens=4096, chunk=1024, window=600, n_sink=16, top_k=8)
    p.update(kw)
    one = binding.Ltri(binding.make_params(**p))
    monkeypatch.setenv("LTRI_MAX_CLUSTER", "8")
    return p, one, binding.Ltri(binding.make_params(**p))


def check(one, two, layers, votes):
    for l in range(layers):
        assert np.array_equal(one.ltri_get_pending_spans(0, l), two.ltri_get_pending_spans(0, l))
        assert np.array_equal(one.ltri_get_spans(0, l), two.ltri_get_spans(0, l))
        assert np.array_equal(one.ltri_get_selected(0, l), two.ltri_get_selected(0, l))
        for what in (binding.BUF_MAP, binding.BUF_THETA):
            assert np.array_equal(one.ltri_debug_read(what, 0, l), two.ltri_debug_read(what, 0, l)), what
        n = one.ltri_get_stats(0, l).last_call_spans  # (what lies behind the call's spans is stale)
        assert np.array_equal(*(x.ltri_debug_read(binding.BUF_NREPS, 0, l)[:n] for x in (one, two)))
        assert np.array_equal(*(x.ltri_debug_read(binding.BUF_QREPS, 0, l)[:, :n] for x in (one, two)))
        if votes:
            t = one.ltri_get_stats(0, l).tokens
            assert np.array_equal(*(x.ltri_debug_read(binding.BUF_VOTES, 0, l)[:t] for x in (one, two)))


def splits_map_pass(lt, layer, n, per_call):
    """Whether the call of n tokens that is just behind `layer` had a launch of its own for the keys before it: three products of
    a key tile with a query block per two SMs, or more, and a third of the SMs beside the segmenter or an early end."""
    p, s = lt.params, lt.ltri_get_stats(0, layer)
    t0 = s.tokens - n
    if s.evicted_end < p.n_sink or t0 <= s.evicted_end:
        return False
    products = -(-(t0 - s.evicted_end) // 128) * -(-n * p.n_q_heads // p.n_kv_heads // 128) * p.n_kv_heads * per_call
    sms, busy = torch.cuda.get_device_properties(0).multi_processor_count, 16 * per_call
    return 2 * products >= 3 * sms and (3 * busy <= 2 * sms or products * 66 <= (sms - busy) * 10 * (150 + n * 2 // 5))


@pytest.mark.parametrize("per_call,kw", [
    (1, dict()),
    (2, dict(theta=0.5)),
    (7, dict(n_layers=7, n_q_heads=8, n_kv_heads=1)),                # the segmenter on three quarters of the SMs
    (1, dict(theta=0.0)), (1, dict(theta=1.0)),                    # first and last rank
    (2, dict(theta_mode=0, theta=0.002)),                          # a given threshold
    (2, dict(layer_theta=[0.8, 0.97], layer_nms_iou_milli=[0, 200], layer_rep_lambda=[1.0, 2.0], rep_mode=1)),
    (1, dict(rep_mode=1, nms_iou_milli=100, ratio_kind=0, rep_lambda=3.0)),
    (2, dict(unit_tokens=64, max_spans_per_region=3, flags=binding.FLAG_SEGMENT_PER_UNIT)),
    (2, dict(retrieval_head=[5, -1])),
    (1, dict(n_q_heads=72, n_kv_heads=9)),                          # column sums of a block beyond 32 bits
    (4, dict(n_layers=4, unit_tokens=64, cache_units=8, flags=binding.FLAG_HOST_KV)),   # pager: a group per layer
])
def test_same_as_the_separate_launches(per_call, kw, monkeypatch):
    p, one, two = pair(monkeypatch, **kw)
    gen = torch.Generator(device="cuda").manual_seed(7)
    L, hq, hkv = p["n_layers"], p["n_q_heads"], p["n_kv_heads"]
    paged = p.get("flags") == binding.FLAG_HOST_KV
    split = 0
    for i, n in enumerate(sum(EDGES, [])):
        if i % 7 == 0 and i < 35:
            one.ltri_reset_sequence(0)
            two.ltri_reset_sequence(0)
        centre = torch.randn(L, 1, hkv, 128, device="cuda", generator=gen)
        k = centre + torch.randn(L, n, hkv, 128, device="cuda", generator=gen)
        q = centre.repeat_interleave(hq // hkv, dim=2) + torch.randn(L, n, hq, 128, device="cuda", generator=gen)
        q, k, v = (t.to(torch.bfloat16) for t in (q, k, torch.randn(L, n, hkv, 128, device="cuda", generator=gen)))
        for lo in range(0, L, per_call):
            hi = lo + per_call
            before = [x.ltri_launch_count() for x in (one, two)]
            outs = [x.ltri_prefill_chunk(0, lo, per_call, q[lo:hi], k[lo:hi], v[lo:hi]) for x in (one, two)]
            assert torch.equal(*outs), f"call {i} of {n} tokens"
            if not paged:  # four launches of the segmenter in one, and one more of the map pass where it splits
                saved = two.ltri_launch_count() - before[1] - (one.ltri_launch_count() - before[0])
                splits = splits_map_pass(one, lo, n, per_call)
                assert saved == (2 if splits else 3), f"call {i} of {n} tokens"
                split += splits
        check(one, two, L, votes=i % 7 == 6)
    assert paged or split > 0
    for x in (one, two):
        assert x.ltri_sync_status() == 0
        x.close()


def test_calls_of_few_and_of_many_layers_in_turn(monkeypatch):
    # the one-launch segmenter finds the scratch it adds up in clear, whatever ran on the layer before
    p, one, two = pair(monkeypatch, n_layers=9, chunk=256, window=600, max_tokens=4096)
    gen = torch.Generator(device="cuda").manual_seed(3)
    for i, n in enumerate([256, 200, 256, 77, 256]):
        q, k, v = (torch.randn(9, n, h, 128, device="cuda", generator=gen).to(torch.bfloat16) for h in (8, 2, 2))
        per = 9 if i % 2 else 3
        for lo in range(0, 9, per):
            outs = [x.ltri_prefill_chunk(0, lo, per, q[lo:lo + per], k[lo:lo + per], v[lo:lo + per]) for x in (one, two)]
            assert torch.equal(*outs)
        check(one, two, 9, votes=True)
    for x in (one, two):
        x.close()


def hand_built(m, seed, bound):
    """Maps of non-negative entries whose rows sum up to at most `bound`: dense, sparse with large entries, of a few values
    only (many equal scores), and planted blocks with noise."""
    rng = np.random.default_rng(seed)
    top = bound // m
    yield np.tril(rng.integers(0, top, size=(m, m)))
    yield np.tril(rng.integers(0, top * 8, size=(m, m)) * (rng.random((m, m)) < 0.1))
    yield np.tril(rng.integers(0, 3, size=(m, m)))
    lens = []
    while sum(lens) < m:
        lens.append(min(int(rng.integers(1, max(2, m // 6))), m - sum(lens)))
    yield block_map(top // 2, lens) + np.tril(rng.integers(0, top // 8 + 1, size=(m, m)))


@pytest.mark.parametrize("phi_milli", [0, 300])
@pytest.mark.parametrize("heads", [(64, 8), (72, 9)])   # column sums of a row block in 32 bits, and in 64
def test_hand_built_maps_against_the_oracle(heads, phi_milli, monkeypatch):
    monkeypatch.setenv("LTRI_DEBUG_SEGMENT", "one")
    lt = binding.Ltri(binding.make_params(1, *heads, 4096, 1024, 1024, 64, 4, max_spans_per_region=16, nms_iou_milli=phi_milli))
    bound = heads[0] << 20
    with pytest.raises(binding.LtriError):   # (only the one-launch segmenter refuses such a map)
        lt.ltri_debug_segment_map(np.full((1, 1), 2 * bound, dtype=np.int32), theta_mode=2)
    for m in (1, 2, 31, 32, 33, 100, 257, 512, 513, 1024):
        for Mq in hand_built(m, m, bound):
            Mq = np.minimum(Mq, 2**31 - 1).astype(np.int32)
            rows = Mq.sum(axis=1, dtype=np.int64)
            Mq[rows > bound] = 0
            for theta in (0.0, 0.5, 0.95, 1.0):
                thq = orc.theta_q(Mq, 1, theta, heads[0])
                want, _ = orc.segment_map(Mq, thq, 16, phi_milli)
                assert lt.ltri_debug_segment_map(Mq, theta_mode=1, theta=theta).tolist() == want.tolist(), (m, theta)
                assert int(lt.ltri_debug_read(binding.BUF_THETA, 0, 0)[0]) == thq
            for thq, spans in ((bound // m // 3, 5), (1, 16)):
                want, _ = orc.segment_map(Mq, thq, spans, phi_milli)
                got = lt.ltri_debug_segment_map(Mq, theta_mode=2, theta_q=thq, max_spans=spans)
                assert got.tolist() == want.tolist(), (m, thq, spans)
    with open(os.path.join(GOLDEN, "block_maps.txt")) as f:
        for line in f:
            if line.strip() and not line.startswith("#") and phi_milli == 0:
                (c, thq, spans), lens = ([int(v) for v in part.split()] for part in line.split("|"))
                if c * max(lens) > bound:
                    continue
                got = lt.ltri_debug_segment_map(block_map(c, lens), theta_mode=2, theta_q=thq, max_spans=spans)
                assert got[:, 1].tolist() == lens and got[0, 0] == 0
    assert lt.ltri_sync_status() == 0
    lt.close()
