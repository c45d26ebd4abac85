"""A context made and bound on a stream of its own while the default stream is busy: what the
library clears before it copies V must be ordered with the copies, not behind the work queued
on the default stream."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def _run(form, N, T, R, busy):
    import torch

    import paper_1301_3389_gb300 as dna
    p = workloads.custom(N, T, R, seed=N + T)
    V, W, H = (torch.from_numpy(np.ascontiguousarray(x)).to("cuda", torch.float32)
               for x in (p.V, p.W, p.H))
    side = torch.cuda.Stream()
    opts = dna.make_opts(dtype=dna.DNA_BF16 if form == "bf16" else dna.DNA_F32)
    torch.cuda.synchronize()
    if busy:
        torch.cuda._sleep(200_000_000)   # about 0.1 s on the default stream
    ctx = dna.dna_create(N, T, R, opts)
    dna.dna_set_stream(ctx, side)
    dna.dna_bind(ctx, V, W, H)
    torch.cuda.synchronize()             # the default stream's work ends after the binding
    dna.dna_normalize(ctx, 1)
    dna.dna_iterate(ctx, 2)
    torch.cuda.synchronize()
    out = W.cpu().numpy(), H.cpu().numpy()
    dna.dna_destroy(ctx)
    return out


@pytest.mark.parametrize("form,N,T", [("f32", 130, 201), ("f32", 128, 200), ("bf16", 130, 201)])
def test_bind_beside_a_busy_default_stream(form, N, T):
    for a, b in zip(_run(form, N, T, 16, False), _run(form, N, T, 16, True)):
        assert np.array_equal(a, b)
