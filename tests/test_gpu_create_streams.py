"""A context made while the default stream is busy, bound and stepped at once on a stream of its
own: what creation clears (status, selections, costs) is clear before the first call, and is not
cleared later, behind the work that was queued on the default stream."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def _run(form, fault, busy):
    import torch

    import paper_1301_3389_gb300 as dna
    p = workloads.custom(130, 201, 16, seed=3)
    W = p.W.copy()
    if fault:
        W[7] = 0.0                       # z = 0 where v > 0
    V, W, H = (torch.from_numpy(np.ascontiguousarray(x)).to("cuda", torch.float32)
               for x in (p.V, W, p.H))
    N, T = V.shape
    csr = [torch.arange(0, N * T + 1, T, device="cuda"),
           torch.arange(T, dtype=torch.int32, device="cuda").repeat(N), V.flatten()]
    side = torch.cuda.Stream()
    opts = dna.make_opts(dtype=dna.DNA_F32)

    def state():
        """What the context holds; the calls wait for the side stream only."""
        choice, dm, dd = np.zeros(T, np.uint8), np.zeros(T), np.zeros(T)
        code = dna.LIB.dna_get_choice(ctx, 0, choice.ctypes.data, T)
        dna.LIB.dna_get_costs(ctx, 0, dm.ctypes.data, dd.ctypes.data, T)
        return code, choice, dm, dd

    torch.cuda.synchronize()
    if busy:
        torch.cuda._sleep(1_000_000_000)   # about 0.5 s on the default stream
    if form == "sparse":
        ctx = dna.dna_create_sparse(N, T, 16, N * T, opts)
        dna.dna_set_stream(ctx, side)
        dna.dna_bind_csr(ctx, *csr, W, H)
        dna.dna_step_H(ctx)
    else:
        ctx = dna.dna_create(N, T, 16, opts)
        dna.dna_set_stream(ctx, side)
        dna.dna_bind(ctx, V, W, H)
        (dna.dna_step_H_fixed if form == "fixed" else dna.dna_step_H)(ctx)
    first = state()
    assert torch.cuda.default_stream().query() != busy
    torch.cuda.synchronize()
    second = state()
    dna.dna_destroy(ctx)
    return first, second


@pytest.mark.parametrize("fault", [False, True])
@pytest.mark.parametrize("form", ["dense", "fixed", "sparse"])
def test_create_beside_a_busy_default_stream(form, fault):
    import paper_1301_3389_gb300 as dna
    ref = _run(form, fault, False)
    assert ref[0][0] == (dna.DNA_ERR_NONFINITE if fault else dna.DNA_OK)
    assert fault or ref[0][1].any()
    for got in _run(form, fault, True):
        for a, b in zip(ref[0], got):
            assert np.array_equal(a, b, equal_nan=True)


def _run_group(bf16, fault, busy):
    import torch

    import paper_1301_3389_gb300 as dna
    probs = [workloads.custom(n, t, r, seed=n) for n, t, r in ((130, 201, 16), (65, 700, 40))]
    if fault:
        probs[1].W[7] = 0.0
    V, W, H = ([torch.from_numpy(np.ascontiguousarray(getattr(p, k))).to("cuda", torch.float32)
                for p in probs] for k in "VWH")
    sizes = [[x.shape[d] for x in m] for m, d in ((V, 0), (V, 1), (W, 1))]
    side = torch.cuda.Stream()

    def state():
        out = []
        for q in range(2):
            choice = np.zeros(sizes[1][q], np.uint8)
            out += [dna.LIB.dna_group_get_choice(g, q, 0, choice.ctypes.data, len(choice)), choice]
        return out

    torch.cuda.synchronize()
    if busy:
        torch.cuda._sleep(1_000_000_000)
    g = dna.dna_group_create(*sizes, dna.make_opts(dtype=dna.DNA_BF16 if bf16 else dna.DNA_F32))
    dna.dna_group_set_stream(g, side)
    dna.dna_group_bind(g, V, W, H)
    dna.dna_group_step_H(g)
    first = state()
    assert torch.cuda.default_stream().query() != busy
    torch.cuda.synchronize()
    second = state()
    dna.dna_group_destroy(g)
    return first, second


@pytest.mark.parametrize("fault", [False, True])
@pytest.mark.parametrize("bf16", [False, True])
def test_group_beside_a_busy_default_stream(bf16, fault):
    """As above for a group; its tables reach the device in the group's own order too."""
    import paper_1301_3389_gb300 as dna
    ref = _run_group(bf16, fault, False)[0]
    assert ref[0] == (dna.DNA_ERR_NONFINITE if fault else dna.DNA_OK) and ref[1].any()
    for got in _run_group(bf16, fault, True):
        assert all(np.array_equal(a, b) for a, b in zip(ref, got))
