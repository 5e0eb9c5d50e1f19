"""Host-buffer entry: layer ranges that cut its groups, calls of several sizes, outputs over the inputs."""
import pytest
import torch

from paper_2412_04757_b200 import binding, inputs
from tests import parity_harness as ph
from tests.test_gpu_parity import small_cfg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layers,ranges", [
    (7, [(0, 7)]),                       # groups of 1, 2, 2 and 2 layers, all of them in flight
    (7, [(0, 2), (2, 4), (6, 1)]),       # ranges that start and end inside a group, and one of a single group
    (3, [(0, 3)]),                       # fewer layers than groups
])
@pytest.mark.parametrize("in_place", [False, True])
def test_groups_and_ranges(layers, ranges, in_place):
    # Staging sets alternate from call to call and a group's bytes in them are its own, so a call's copies run beside the
    # kernels and the copies of the one before it: nothing waits on the host in between.  Same bits as the device entry.
    cfg = small_cfg(n_layers=layers, context=1536, decode_steps=0)
    st = inputs.SyntheticStream(cfg)
    p = ph.params_of(cfg)
    p.flags |= binding.FLAG_HOST_STAGING
    dev, host = binding.Ltri(ph.params_of(cfg)), binding.Ltri(p)
    t0, pairs = 0, []
    for n in [128, 128, 77, 128, 16, 128, 128, 51, 128, 1, 128, 128, 128, 128, 111]:
        q, k, v = st.tokens(t0, n)
        t0 += n
        for lo, cnt in ranges:
            part = [x[lo:lo + cnt].contiguous() for x in (q, k, v)]
            want = dev.ltri_prefill_chunk(0, lo, cnt, *(x.cuda() for x in part))
            hq, hk, hv = (x.pin_memory() for x in part)
            out = hq if in_place else torch.empty_like(hq).pin_memory()
            host.ltri_prefill_chunk_host(0, lo, cnt, hq, hk, hv, out)
            pairs.append((want, out, hk, hv))
    assert t0 == cfg.context
    host.ltri_host_outputs_ready()
    torch.cuda.synchronize()
    for i, (want, out, _, _) in enumerate(pairs):
        assert torch.equal(want.cpu(), out), f"call {i}"
    assert dev.ltri_sync_status() == 0 and host.ltri_sync_status() == 0
    dev.close()
    host.close()
