"""Calls that take device arrays are ordered against the caller's stream, the
default one included: what it has queued on the array before the call is
done before the library reads or writes it."""
import numpy as np
import pytest

from paper_1910_01031_gb300 import iewpf, synth
from gpu_common import ensemble, start_state

pytestmark = pytest.mark.gpu


@pytest.fixture(params=["default", "side"])
def busy(request):
    """A stream, and a function that queues some tens of milliseconds of work on it."""
    import torch
    a = torch.zeros(1 << 28, dtype=torch.float32, device="cuda")      # 1 GB: 2 GB of traffic per pass

    def queue():
        for _ in range(100):
            a.add_(1.0)
    stream = torch.cuda.default_stream() if request.param == "default" else torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        yield queue
    torch.cuda.synchronize()


def test_states_wait_for_the_callers_stream(busy):
    import torch
    cfg = synth.Config("edge", 64, 64, n_particles=5)
    U32, _ = start_state(cfg, 5)
    ens = ensemble(cfg)
    src, want = torch.full(U32.shape, 7.0, device="cuda"), torch.from_numpy(U32).cuda()
    torch.cuda.synchronize()
    busy()
    src.copy_(want)                          # still to come when set_state is called
    ens.set_state(src)
    assert np.array_equal(ens.get_state(), U32)
    out = torch.full(U32.shape, 3.0, device="cuda")
    torch.cuda.synchronize()
    busy()
    before = out.clone()                     # reads the array before get_state writes it
    out.fill_(-1.0)
    ens.get_state(out)
    torch.cuda.synchronize()
    assert bool((before == 3.0).all())
    assert torch.equal(out, want)


@pytest.mark.parametrize("in_place", [False, True])
def test_network_calls_wait_for_the_callers_stream(busy, in_place):
    import torch
    cfg = synth.Config("edge", 64, 32, n_particles=2)
    net = iewpf.Surrogate(64, 32)
    U32, _ = start_state(cfg, 2)
    want = net.apply(U32)
    src, U = torch.full(U32.shape, 7.0, device="cuda"), torch.from_numpy(U32).cuda()
    out = src if in_place else torch.empty_like(src)
    torch.cuda.synchronize()
    busy()
    src.copy_(U)
    got = net.apply_device(src, out)
    torch.cuda.synchronize()
    assert np.array_equal(got.cpu().numpy(), want)
