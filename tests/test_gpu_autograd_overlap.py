"""Two calls of the autograd wrappers that share a kept context and would overlap on the GPU:
the second one's stream reaches its work while the first one's is in the middle of its steps,
and both give the bits of calls that are waited for one by one."""
import pytest

import workloads

pytestmark = pytest.mark.gpu

STEPS = 60    # tens of milliseconds of steps, few enough launches to be queued behind a delay
DELAY = 400_000_000   # about 0.2 s: longer than the host takes to queue both calls


def test_overlapping_calls_share_a_context():
    import torch

    from paper_1301_3389_gb300.autograd import UnrolledDNAH
    p = workloads.custom(2000, 8000, 64, seed=9)
    inputs = []
    for k in range(2):
        g = torch.Generator(device="cuda")
        g.manual_seed(k)
        inputs.append([torch.from_numpy(p.V).cuda() * (1.0 + k),
                       torch.rand(p.W.shape, generator=g, device="cuda") + 0.1,
                       torch.rand(p.H.shape, generator=g, device="cuda") + 0.1])
    ref = []
    for x in inputs:
        ref.append(UnrolledDNAH.apply(*x, STEPS, STEPS).clone())
        torch.cuda.synchronize()
    assert not torch.equal(ref[0], ref[1])
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    got = []
    for s, x in zip(streams, inputs):
        # both delays run at the same time, the second one started later by the time that the
        # host takes to queue the first call
        with torch.cuda.stream(s):
            torch.cuda._sleep(DELAY)
            got.append(UnrolledDNAH.apply(*x, STEPS, STEPS))
    assert not streams[0].query()
    torch.cuda.synchronize()
    for a, b in zip(ref, got):
        assert torch.equal(a, b)
