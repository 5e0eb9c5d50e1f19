"""The one-launch decode step against the oracle, at the sizes where its splits and short cuts change."""
import pytest

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
