"""The autograd wrappers queue their work without waiting for it: calls on alternating streams
that share a kept context, and inputs released right after the call, give the bits of calls
that are waited for one by one; a call under graph capture is refused."""
import pytest

import workloads

pytestmark = pytest.mark.gpu


def _inputs(p, seed):
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    V = torch.from_numpy(p.V).cuda()
    return [V.clone(), torch.rand(p.W.shape, generator=g, device="cuda") + 0.1,
            torch.rand(p.H.shape, generator=g, device="cuda") + 0.1,
            torch.randn(p.H.shape, generator=g, device="cuda")]


def _call(V, W, H, G):
    import torch

    from paper_1301_3389_gb300.autograd import KLDiv, UnrolledDNAH
    for t in (V, W, H):
        t.requires_grad_()
    HK = UnrolledDNAH.apply(V, W, H, 3, 2)
    out = [HK.detach(), *torch.autograd.grad(HK, (V, W, H), G)]
    return out + list(torch.autograd.grad(KLDiv.apply(V, W, H), (V, W, H)))


def test_streams_share_a_context():
    import torch
    p = workloads.custom(300, 900, 24, seed=5)
    ref = []
    for k in range(6):
        x = _inputs(p, k)
        torch.cuda.synchronize()
        ref.append([t.clone() for t in _call(*x)])
        torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    got = []
    for k in range(6):
        x = _inputs(p, k)                       # made on the default stream
        s = streams[k % 2]
        s.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(s):
            got.append(_call(*x))
        del x                                   # their memory may be handed out again at once
        junk = [torch.full((300, 900), float("nan"), device="cuda") for _ in range(4)]
        del junk
    torch.cuda.synchronize()
    for a, b in zip(ref, got):
        for s, t in zip(a, b):
            assert torch.equal(s, t)


def test_capture_is_refused():
    import torch

    from paper_1301_3389_gb300.autograd import UnrolledDNAH
    p = workloads.custom(40, 60, 8, seed=6)
    V, W, H, _ = _inputs(p, 0)
    UnrolledDNAH.apply(V, W, H, 2, 2)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        graph.capture_begin()
        try:
            with pytest.raises(RuntimeError, match="captured"):
                UnrolledDNAH.apply(V, W, H, 2, 2)
        finally:
            graph.capture_end()
    torch.cuda.synchronize()
