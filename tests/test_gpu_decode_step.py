"""The one-launch decode step against the oracle, at the sizes where its splits and short cuts change."""
import numpy as np
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
    assert rep.step_launches == {1}
    print(rep)


@pytest.mark.parametrize("cluster", [2, 4, 8, 16])
@pytest.mark.parametrize("kind", ["thirds", "all", "one_slice", "far"])
def test_selection_of_equal_and_of_distant_scores(kind, cluster, monkeypatch):
    # The short cut of the cluster's select lists candidates near the largest score, 512 / cluster per CTA and 256 in all;
    # beyond that the general select takes over.  700 loaded spans, ties go to the lower span:
    #   thirds     three groups of 233 equal scores that cross all slices, the cut inside the first: the short cut
    #   all        700 equal scores
    #   one_slice  the last CTA's whole slice equal and on top: more than its list holds
    #   far        three scores more than 255 steps of the histogram above the others
    monkeypatch.setenv("LTRI_DEC_CLUSTER", str(cluster))
    L, hq, hkv, topk, N = 2, 8, 2, 5, 700
    cfg = small_cfg(n_layers=L, n_q_heads=hq, n_kv_heads=hkv, context=1536, window=128, n_sink=16, top_k=topk,
                    max_spans_per_region=64, decode_steps=1)
    st = inputs.SyntheticStream(cfg, device="cuda:0")
    lts = [binding.Ltri(ph.params_of(cfg))]
    monkeypatch.setenv("LTRI_DEC_FUSED", "0")
    lts.append(binding.Ltri(ph.params_of(cfg)))
    for t0, n in st.prefill_chunks():
        for lt in lts:
            lt.ltri_prefill_chunk(0, 0, L, *st.tokens(t0, n))
    q, k, v = (x.permute(1, 0, 2, 3).contiguous() for x in st.tokens(cfg.context, 1, kind=1))
    want = []
    for layer in range(L):
        E = lts[0].ltri_get_stats(0, layer).evicted_end
        lens = np.full(N, (E - cfg.n_sink) // N)
        lens[:(E - cfg.n_sink) % N] += 1
        spans = np.stack([cfg.n_sink + np.concatenate([[0], np.cumsum(lens)[:-1]]), lens], axis=1).astype(np.int32)
        u = q[0, layer].double().view(hkv, hq // hkv, 128).sum(1).cpu()       # the summed queries of every KV head
        rng = torch.Generator().manual_seed(layer)
        top = u[:, None].expand(hkv, N, 128)
        low = 0.05 * torch.randn(hkv, N, 128, generator=rng, dtype=torch.float64)
        if kind == "thirds":
            idx = torch.randn(hkv, 3, 128, generator=rng, dtype=torch.float64)[:, torch.arange(N) % 3]
        elif kind == "all":
            idx = top.clone()
        else:
            on_top = torch.zeros(N, dtype=torch.bool)
            if kind == "one_slice":
                on_top[-(-N // cluster) * (cluster - 1):] = True
            else:
                on_top[[3, 350, 699]] = True
            idx = torch.where(on_top[:, None], top, low)
        idx = idx.to(torch.bfloat16)
        sc = torch.einsum("gnd,gd->gn", idx.double(), u).numpy()
        want.append([sorted(np.argsort(-sc[g], kind="stable")[:topk].tolist()) for g in range(hkv)])
        for lt in lts:
            lt.ltri_debug_load_index(0, layer, E, spans, inputs.bf16_bits(idx))
    outs, launched = [], []
    for lt in lts:
        before = lt.ltri_launch_count()
        outs.append(lt.ltri_decode_step([0], 0, L, q, k, v))
        launched.append(lt.ltri_launch_count() - before)
        for layer in range(L):
            assert lt.ltri_get_selected(0, layer).tolist() == want[layer]
        assert lt.ltri_sync_status() == 0
    assert launched[0] == 1 and launched[1] > 1
    assert float((outs[0].float() - outs[1].float()).abs().max()) <= ph.MAX_ABS
    for lt in lts:
        lt.close()


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
