"""The one-launch decode step against the oracle, at the sizes where its splits and short cuts change."""
import pytest
import torch

from paper_2412_04757_b200 import binding, inputs
from tests import parity_harness as ph
from tests.test_gpu_parity import small_cfg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cluster", [2, 4, 8, 16])
@pytest.mark.parametrize("extra", [
    dict(context=40, n_sink=64),                                   # inside the sink, no index, most CTAs without tokens
    dict(context=1280, top_k=64),                                  # fewer spans than top_k at first, lists of 64
    dict(context=3000, top_k=6, max_spans_per_region=16, seg_min=8, seg_max=24),   # uneven slices, the histogram cut
    dict(context=1536, top_k=5, unit_tokens=40, persist_decode=True),              # units ranked, two selections united
    dict(context=1536, top_k=6, nms_iou_milli=300),                # overlapping spans: every token once
])
def test_one_launch_step(cluster, extra, monkeypatch):
    monkeypatch.setenv("LTRI_DEC_CLUSTER", str(cluster))
    kw = dict(n_layers=2, decode_steps=5)
    kw.update(extra)
    rep = ph.run_stream(small_cfg(**kw), layers=[0, 1], deep=False)
    print(rep)


@pytest.mark.parametrize("shared,heads,one_launch", [
    ("q", None, True),            # every cluster overwrites the queries that it alone has read
    ("q", (5, 2), False),         # a retrieval head's queries are read by the clusters of all KV heads
    ("k", None, False),           # the outputs of some heads lie over the new rows of others
])
def test_outputs_written_over_the_inputs(shared, heads, one_launch, monkeypatch):
    cfg = small_cfg(n_layers=2, context=1280, decode_steps=4, retrieval_head=heads)
    st = inputs.SyntheticStream(cfg)
    lt = binding.Ltri(ph.params_of(cfg))
    if not one_launch:
        monkeypatch.setenv("LTRI_DEC_FUSED", "0")   # the twin takes the same launches with buffers of its own
    twin = binding.Ltri(ph.params_of(cfg))
    for t0, n in st.prefill_chunks():
        q, k, v = (x.cuda() for x in st.tokens(t0, n))
        lt.ltri_prefill_chunk(0, 0, 2, q, k, v)
        twin.ltri_prefill_chunk(0, 0, 2, q, k, v)
    for s in range(cfg.decode_steps):
        q, k, v = (x.permute(1, 0, 2, 3).contiguous().cuda() for x in st.tokens(cfg.context + s, 1, kind=1))
        want = twin.ltri_decode_step([0], 0, 2, q, k, v)
        out = torch.empty_like(q)
        if shared == "q":
            out.copy_(q)
            q = out
        else:                     # k inside the output's memory, 256 bytes from its start
            k = out.view(-1)[128:128 + k.numel()].view(k.shape).copy_(k)
        before = lt.ltri_launch_count()
        lt.ltri_decode_step([0], 0, 2, q, k, v, out=out)
        assert (lt.ltri_launch_count() - before == 1) == one_launch
        assert torch.equal(out, want), f"step {s}"
    assert lt.ltri_sync_status() == 0
    lt.close()
    twin.close()
