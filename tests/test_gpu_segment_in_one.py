"""The one-launch segmenter (calls of few layers) against the separate launches, which the parity tests hold to the oracle.

A context created with clusters of at most eight CTAs segments in separate launches and runs the map pass as one; everything
in between is integer arithmetic, so maps, thresholds, spans, votes, representatives and outputs have to agree to the bit."""
import numpy as np
import pytest
import torch

from paper_2412_04757_b200 import binding

pytestmark = pytest.mark.gpu

# call sizes around the edges of the row blocks (32 per call), of the 128-entry row groups and of the rounds' key counts
# (seven to a sequence: a context of this window and chunk keeps eight regions pending)
EDGES = [[1024, 1023, 1, 512, 2, 993, 17], [513, 700, 511, 16, 257, 481, 31], [256, 1024, 255, 32, 129, 128, 33],
         [640, 65, 64, 1000, 127, 15, 416]]


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


@pytest.mark.parametrize("per_call,kw", [
    (1, dict()),
    (2, dict(theta=0.5)),
    (1, dict(theta=0.0)), (1, dict(theta=1.0)),                    # first and last rank
    (2, dict(theta_mode=0, theta=0.002)),                          # a given threshold
    (2, dict(layer_theta=[0.8, 0.97], layer_nms_iou_milli=[0, 200], layer_rep_lambda=[1.0, 2.0], rep_mode=1)),
    (1, dict(rep_mode=1, nms_iou_milli=100, ratio_kind=0, rep_lambda=3.0)),
    (2, dict(unit_tokens=64, max_spans_per_region=3, flags=binding.FLAG_SEGMENT_PER_UNIT)),
    (2, dict(retrieval_head=[5, -1])),
    (1, dict(n_q_heads=72, n_kv_heads=9)),                          # column sums of a block beyond 32 bits
])
def test_same_as_the_separate_launches(per_call, kw, monkeypatch):
    p, one, two = pair(monkeypatch, **kw)
    gen = torch.Generator(device="cuda").manual_seed(7)
    L, hq, hkv = p["n_layers"], p["n_q_heads"], p["n_kv_heads"]
    for i, n in enumerate(sum(EDGES, [])):
        if i % 7 == 0:
            one.ltri_reset_sequence(0)
            two.ltri_reset_sequence(0)
        centre = torch.randn(L, 1, hkv, 128, device="cuda", generator=gen)
        k = centre + torch.randn(L, n, hkv, 128, device="cuda", generator=gen)
        q = centre.repeat_interleave(hq // hkv, dim=2) + torch.randn(L, n, hq, 128, device="cuda", generator=gen)
        q, k, v = (t.to(torch.bfloat16) for t in (q, k, torch.randn(L, n, hkv, 128, device="cuda", generator=gen)))
        for lo in range(0, L, per_call):
            hi = lo + per_call
            outs = [x.ltri_prefill_chunk(0, lo, per_call, q[lo:hi], k[lo:hi], v[lo:hi]) for x in (one, two)]
            assert torch.equal(*outs), f"call {i} of {n} tokens"
        check(one, two, L, votes=i % 7 == 6)
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
