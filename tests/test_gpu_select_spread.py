"""Selection when the best scores lie far apart: one test per step width of the histogram that finds the cut, and one beyond it.

The K best of 700 loaded spans fall by `octaves` powers of two from the first to the K-th, the rest lie below.  The histogram
has one step of 1/128 octave per bin for the first octave, then 4, 16 and 64 steps, and ends after 22.5 octaves."""
import numpy as np
import pytest
import torch

from paper_2412_04757_b200 import binding, inputs
from tests import parity_harness as ph
from tests.test_gpu_parity import small_cfg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("route", ["c2", "c16", "0", "1", "2"])   # one launch in clusters of 2 and 16, the separate retrievers
@pytest.mark.parametrize("octaves,topk", [(0.4, 5), (0.9, 40), (1.1, 5), (2.5, 40), (4.0, 5), (6.5, 40), (9.0, 12), (21.0, 64),
                                          (30.0, 12)])
def test_cut_at_every_step_width(octaves, topk, route, monkeypatch):
    monkeypatch.setenv(*(("LTRI_DEC_CLUSTER", route[1:]) if route[0] == "c" else ("LTRI_DEC_FUSED", route)))
    hq, hkv, N = 8, 2, 700
    cfg = small_cfg(n_layers=1, n_q_heads=hq, n_kv_heads=hkv, context=1536, window=128, n_sink=16, top_k=topk,
                    max_spans_per_region=64, decode_steps=1)
    st = inputs.SyntheticStream(cfg, device="cuda:0")
    lt = binding.Ltri(ph.params_of(cfg))
    for t0, n in st.prefill_chunks():
        lt.ltri_prefill_chunk(0, 0, 1, *st.tokens(t0, n))
    q, k, v = (x.permute(1, 0, 2, 3).contiguous() for x in st.tokens(cfg.context, 1, kind=1))
    E = lt.ltri_get_stats(0, 0).evicted_end
    lens = np.full(N, (E - cfg.n_sink) // N)
    lens[:(E - cfg.n_sink) % N] += 1
    spans = np.stack([cfg.n_sink + np.concatenate([[0], np.cumsum(lens)[:-1]]), lens], axis=1).astype(np.int32)
    u = q[0, 0].double().view(hkv, hq // hkv, 128).sum(1).cpu()
    rng = torch.Generator().manual_seed(int(10 * octaves) + topk)
    fall = torch.arange(N, dtype=torch.float64) * (octaves / topk)          # in octaves below the best, by rank
    fall[topk:] = octaves + 0.3 + 2.0 * torch.rand(N - topk, generator=rng, dtype=torch.float64)
    perm = torch.randperm(N, generator=rng)
    scale = torch.empty(N, dtype=torch.float64)
    scale[perm] = 2.0 ** -fall
    idx = (u[:, None] * scale[None, :, None]).to(torch.bfloat16)            # rows along u: the scores fall as said
    sc = torch.einsum("gnd,gd->gn", idx.double(), u).numpy()
    want = [sorted(np.argsort(-sc[g], kind="stable")[:topk].tolist()) for g in range(hkv)]
    lt.ltri_debug_load_index(0, 0, E, spans, inputs.bf16_bits(idx))
    before = lt.ltri_launch_count()
    lt.ltri_decode_step([0], 0, 1, q, k, v)
    assert (lt.ltri_launch_count() - before == 1) == (route[0] == "c")
    assert lt.ltri_get_selected(0, 0).tolist() == want
    assert lt.ltri_sync_status() == 0
    lt.close()
