"""Every index size that the dispatch sends to a one-launch decode retriever is within the kernel's limit of shared memory."""
import pytest
import torch

from paper_2412_04757_b200 import binding

pytestmark = pytest.mark.gpu


def _params(tokens, **kw):
    # 64 spans kept per region: a region of 128 tokens counts 128 possible spans, so a short stream has a large index
    p = dict(n_layers=1, n_q_heads=1, n_kv_heads=1, max_tokens=tokens, chunk=128, window=64, n_sink=16, top_k=8,
             max_spans_per_region=64)
    p.update(kw)
    return binding.make_params(**p)


@pytest.mark.parametrize("layers,heads,calls", [(19, 8, 92), (1, 1, 720)])
def test_decode_of_an_index_that_fills_the_shared_memory_of_its_retriever(layers, heads, calls, monkeypatch):
    # 11.6K possible spans in one CTA per KV head (152 of them: a CTA for every SM) and 92K in a cluster of eight: 45 KB of
    # order keys beside the kernel's static arrays, more than a kernel may use without asking
    lts = [binding.Ltri(_params(128 * calls + 4, n_layers=layers, n_q_heads=heads, n_kv_heads=heads))]
    monkeypatch.setenv("LTRI_DEC_FUSED", "0")
    lts.append(binding.Ltri(lts[0]._params_src))
    g = torch.Generator(device="cuda").manual_seed(3)
    for _ in range(calls):
        q, k, v = (torch.randn(layers, 128, heads, 128, generator=g, device="cuda").to(torch.bfloat16) for _ in range(3))
        for lt in lts:
            lt.ltri_prefill_chunk(0, 0, layers, q, k, v)
    q, k, v = (torch.randn(1, layers, heads, 128, generator=g, device="cuda").to(torch.bfloat16) for _ in range(3))
    outs = [lt.ltri_decode_step([0], 0, layers, q, k, v) for lt in lts]
    for l in range(layers):
        assert (lts[0].ltri_get_selected(0, l) == lts[1].ltri_get_selected(0, l)).all()
    # (the two retrievers lead to the same attention kernel over the same ranges)
    assert torch.equal(outs[0], outs[1])
    assert all(lt.ltri_sync_status() == 0 for lt in lts)
    for lt in lts:
        lt.close()
