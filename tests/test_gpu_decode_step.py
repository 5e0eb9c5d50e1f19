"""The one-launch decode step against the oracle, at the sizes where its splits and short cuts change."""
import os
import re

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


STEP = open(os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2412_04757_b200", "csrc",
                         "kernels_dec_step.cu")).read()


def step_constant(name):
    return int(re.search(rf"constexpr int {name} = (\d+);", STEP).group(1))


@pytest.mark.parametrize("cluster", [2, 4, 8, 16])
@pytest.mark.parametrize("kind", ["thirds", "all", "brim", "over", "one_slice", "far"])
def test_selection_of_equal_and_of_distant_scores(kind, cluster, monkeypatch):
    # The short cut of the cluster's select lists candidates near the largest score, kStList / cluster per CTA and one per
    # thread in all; beyond that the general select takes over.  Ties go to the lower span:
    #   thirds     three groups of 233 equal scores that cross all slices, the cut inside the first: the short cut
    #   all        700 equal scores
    #   brim       as many equal scores on top as the last CTA's list holds, or as are ranked in all: the short cut
    #   over       one more
    #   one_slice  the last CTA's whole slice equal and on top
    #   far        three scores further above the others than the histogram reaches
    limit = min(step_constant("kStList") // cluster, step_constant("kStThreads"))
    N = 700 if kind in ("thirds", "all") else 1600
    per = -(-N // cluster)
    assert "kStCand = kStThreads;" in STEP and (kind != "one_slice" or per > step_constant("kStList") // cluster)
    monkeypatch.setenv("LTRI_DEC_CLUSTER", str(cluster))
    L, hq, hkv, topk = 2, 8, 2, 5
    cfg = small_cfg(n_layers=L, n_q_heads=hq, n_kv_heads=hkv, context=1536 if N == 700 else 2048, window=128, n_sink=16,
                    top_k=topk, max_spans_per_region=64, decode_steps=1)
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
            first = per * (cluster - 1)                # of the last CTA's slice
            if kind == "far":
                on_top[[3, 350, 699]] = True
                low *= 2.0 ** -24
            else:
                on_top[first:first + {"brim": limit, "over": limit + 1, "one_slice": N}[kind]] = True
            idx = torch.where(on_top[:, None], top, low)
        idx = idx.to(torch.bfloat16)
        sc = torch.einsum("gnd,gd->gn", idx.double(), u).numpy()
        if kind == "far":                              # the histogram ends 22.5 octaves below the largest score
            assert all(np.log2(sc[g].max() / np.sort(sc[g])[-topk]) > 23 for g in range(hkv))
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


@pytest.mark.parametrize("seqs,context,one_launch", [
    (6, 4096, True), (6, 5120, False),      # 48 units as clusters of four: 1088 tokens per CTA are the line
    (12, 1920, True), (12, 2560, False),    # 96 units as clusters of two
    (2, 6656, True), (2, 7680, False),      # 16 units as clusters of eight: 864 tokens per CTA
    (4, 7680, True),                        # 32 units as clusters of eight
])
def test_route_of_steps_that_fetch_every_unit(seqs, context, one_launch, monkeypatch):
    # a small index of units, all of them fetched: either route attends over every token
    cfg = small_cfg(n_layers=1, n_q_heads=16, n_kv_heads=8, context=context, chunk=512, window=512, n_seqs=seqs,
                    unit_tokens=128, top_k=64, decode_steps=1)
    st = inputs.SyntheticStream(cfg, device="cuda:0")
    lts = [binding.Ltri(ph.params_of(cfg))]
    monkeypatch.setenv("LTRI_DEC_FUSED", "0")
    lts.append(binding.Ltri(ph.params_of(cfg)))
    K, V = [], []
    for t0, n in st.prefill_chunks():
        q, k, v = st.tokens(t0, n)
        K.append(k[0])
        V.append(v[0])
        for lt in lts:
            for s in range(seqs):
                lt.ltri_prefill_chunk(s, 0, 1, q, k, v)
    q, k, v = (x.permute(1, 0, 2, 3).expand(seqs, -1, -1, -1).contiguous() for x in st.tokens(context, 1, kind=1))
    K, V = torch.cat(K + [k[0]]).double(), torch.cat(V + [v[0]]).double()
    p = torch.softmax(torch.einsum("gjd,tgd->gjt", q[0, 0].double().view(8, 2, 128), K) / 128 ** 0.5, dim=-1)
    want = torch.einsum("gjt,tgd->gjd", p, V).reshape(16, 128).cpu().numpy()
    rep = ph.Report()
    for lt, one in zip(lts, (one_launch, False)):
        before = lt.ltri_launch_count()
        out = lt.ltri_decode_step(list(range(seqs)), 0, 1, q, k, v)
        assert (lt.ltri_launch_count() - before == 1) == one
        for s in range(seqs):
            ph.check_output(out[s, 0], want, rep, f"sequence {s}")
        assert lt.ltri_sync_status() == 0
        lt.close()


@pytest.mark.parametrize("seqs,layers,top_k,window,persist,one_launch", [
    (1, 8, 64, 3072, True, True),      # 64 units as clusters of four: 16384 fetched and 3.6K known tokens a unit
    (1, 8, 64, 4608, True, False),     # 20480 are the line
    (2, 8, 8, 896, False, True),       # 128 units as clusters of two: 1024 fetched and 1.6K known tokens a unit
    (2, 8, 8, 2496, False, False),     # 3072 are the line
])
def test_route_of_steps_that_fetch_some_units(seqs, layers, top_k, window, persist, one_launch, monkeypatch):
    # an index of more units than are fetched, with and without the selection kept from the last prefill call
    chunk = 512
    context = 2 * 64 * 128 + window + 2 * chunk if top_k == 64 else 4096 + window
    context += -context % chunk
    cfg = small_cfg(n_layers=layers, n_q_heads=16, n_kv_heads=8, context=context, chunk=chunk, window=window, n_seqs=seqs,
                    unit_tokens=128, top_k=top_k, decode_steps=2, persist_decode=persist, max_spans_per_region=8)
    st = inputs.SyntheticStream(cfg, device="cuda:0")
    lts = [binding.Ltri(ph.params_of(cfg))]
    monkeypatch.setenv("LTRI_DEC_FUSED", "0")
    lts.append(binding.Ltri(ph.params_of(cfg)))
    for t0, n in st.prefill_chunks():
        q, k, v = st.tokens(t0, n)
        for lt in lts:
            for s in range(seqs):
                lt.ltri_prefill_chunk(s, 0, layers, q, k, v)
    E = lts[0].ltri_get_stats(0, 0).evicted_end
    known = cfg.n_sink + context + 1 - E
    tokens = known + min(E, top_k * 128 * (2 if persist else 1))
    assert (E - 1) // 128 >= top_k and (tokens <= (20480 if layers * seqs == 8 else 3072)) == one_launch
    for step in range(cfg.decode_steps):
        q, k, v = (x.permute(1, 0, 2, 3).expand(seqs, -1, -1, -1).contiguous() for x in st.tokens(context + step, 1, kind=1))
        outs = []
        for lt, one in zip(lts, (one_launch, False)):
            before = lt.ltri_launch_count()
            outs.append(lt.ltri_decode_step(list(range(seqs)), 0, layers, q, k, v))
            assert (lt.ltri_launch_count() - before == 1) == one
        for s in range(seqs):
            for l in range(layers):
                assert (lts[0].ltri_get_selected(s, l) == lts[1].ltri_get_selected(s, l)).all()
        assert float((outs[0].float() - outs[1].float()).abs().max()) <= ph.MAX_ABS
    for lt in lts:
        assert lt.ltri_sync_status() == 0
        lt.close()


@pytest.mark.parametrize("seqs,one_launch", [(3, True), (4, False)])
def test_route_of_steps_over_a_large_index(seqs, one_launch, monkeypatch):
    # 18K spans and 4.3K known tokens: 24 units read 639K rows, 32 read 851K; the line lies at 768K
    N, window = 18000, 4096
    context = (N + window + 300) // 128 * 128
    cfg = small_cfg(n_layers=1, n_q_heads=16, n_kv_heads=8, context=context, window=window, n_sink=16, n_seqs=seqs,
                    top_k=32, max_spans_per_region=64, decode_steps=1)
    lts = [binding.Ltri(ph.params_of(cfg))]
    monkeypatch.setenv("LTRI_DEC_FUSED", "1")
    lts.append(binding.Ltri(ph.params_of(cfg)))
    g = torch.Generator(device="cuda").manual_seed(4)
    q, k, v = (torch.randn(1, 128, h, 128, generator=g, device="cuda").to(torch.bfloat16) for h in (16, 8, 8))
    for _ in range(context // 128):
        for lt in lts:
            for s in range(seqs):
                lt.ltri_prefill_chunk(s, 0, 1, q, k, v)
    E = lts[0].ltri_get_stats(0, 0).evicted_end
    lens = np.full(N, (E - 16) // N)
    lens[:(E - 16) % N] += 1
    spans = np.stack([16 + np.concatenate([[0], np.cumsum(lens)[:-1]]), lens], axis=1).astype(np.int32)
    idx = torch.randn(8, N, 128, generator=torch.Generator().manual_seed(5)).to(torch.bfloat16)
    for lt in lts:
        for s in range(seqs):
            lt.ltri_debug_load_index(s, 0, E, spans, inputs.bf16_bits(idx))
    q, k, v = (torch.randn(seqs, 1, h, 128, generator=g, device="cuda").to(torch.bfloat16) for h in (16, 8, 8))
    outs = []
    for lt, one in zip(lts, (one_launch, False)):
        before = lt.ltri_launch_count()
        outs.append(lt.ltri_decode_step(list(range(seqs)), 0, 1, q, k, v))
        assert (lt.ltri_launch_count() - before == 1) == one
        assert lt.ltri_sync_status() == 0
    for s in range(seqs):
        assert (lts[0].ltri_get_selected(s, 0) == lts[1].ltri_get_selected(s, 0)).all()
    assert float((outs[0].float() - outs[1].float()).abs().max()) <= ph.MAX_ABS
    for lt in lts:
        lt.close()
