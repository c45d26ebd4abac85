"""The float32 passes on the CUDA cores at ranks up to 128, at the sizes where their layout
changes: every multiple of 16 of the rank (padding, single rows, groups of s), chunks and
o-blocks of 64 with remainders, one and many splits, rows that cannot be copied 16 bytes at a
time.  Tolerances are the FP32 form's (1e-4 relative Frobenius per half-step from the GPU's
own state, d_KL 1e-6: its terms are float32 sums of a few entries, added exactly beyond)."""
import numpy as np
import pytest

import workloads
from gpu_helpers import GpuProblem, rel_fro, step_pair
from oracle import dna as o

pytestmark = pytest.mark.gpu

TOL = 1e-4
KL_TOL = 1e-6


def _half_steps(N, T, R, mu=False, kl=False, **opts):
    p = workloads.custom(N, T, R, seed=N + 7 * T + 13 * R)
    oopts = {"eps": o.EPS, "alpha": o.ALPHA, "rho": opts.get("rho", 0.0), "lam": opts.get("lam", 0.0)}
    with GpuProblem(p.V, p.W, p.H, "f32", **opts) as gp:
        gp.dna.dna_normalize(gp.ctx, 1)
        W, H = o.normalize_w_columns(p.W, p.H, oopts["lam"])
        for which in (0, 1):
            W, H, _ = step_pair(gp, W, H, which, mu=mu, opts=oopts)
            Wg, Hg = gp.WH()
            assert rel_fro(Wg, W) < TOL and rel_fro(Hg, H) < TOL, which
        if kl:   # not where W H can be exact: d_KL is then rounding alone
            ref = o.kl_divergence(p.V.astype(np.float64), Wg @ Hg)
            assert abs(gp.dna.dna_kl(gp.ctx) - ref) <= KL_TOL * abs(ref)


@pytest.mark.parametrize("R", [1, 15, 16, 17, 32, 33, 48, 49, 64, 65, 80, 81, 96, 97, 112, 113,
                               127, 128])
def test_rank_classes(R):
    _half_steps(131, 200, R, kl=True)


@pytest.mark.parametrize("R", [3, 16, 40, 80, 128])
def test_mu_rank_classes(R):
    _half_steps(131, 200, R, mu=True)


@pytest.mark.parametrize("N,T,R", [(1, 1, 1), (1, 130, 5), (63, 65, 16), (64, 64, 32), (65, 63, 20),
                                   (128, 193, 8), (5000, 3, 24), (3, 5000, 70), (700, 2501, 80)])
def test_chunk_and_block_edges(N, T, R):
    _half_steps(N, T, R)


def test_regularised():
    _half_steps(190, 77, 52, rho=0.4, lam=0.7)


@pytest.mark.parametrize("R", [16, 80, 128])
def test_unaligned_buffers(R):
    """Factors and V that start 4 bytes past a 16-byte boundary (V's rows 3 values longer than
    T): the same bits as from aligned buffers (only the width of the copies differs)."""
    import torch
    p = workloads.custom(130, 141, R, seed=R)
    outs = []
    for shift in (0, 1):
        with GpuProblem(p.V, p.W, p.H, "f32") as gp:
            buf = {}
            for name, x, ld in (("V", gp.V, gp.T + 3 * shift), ("W", gp.W, gp.R), ("H", gp.H, gp.T)):
                flat = torch.zeros(x.shape[0] * ld + 4, device="cuda")
                view = flat[shift:shift + x.shape[0] * ld].view(x.shape[0], ld)[:, :x.shape[1]]
                view.copy_(x)
                buf[name] = view
            gp.dna.dna_bind(gp.ctx, buf["V"], buf["W"], buf["H"])
            gp.dna.dna_normalize(gp.ctx, 1)
            gp.dna.dna_iterate(gp.ctx, 2)
            outs.append((gp.dna.dna_kl(gp.ctx), buf["W"].cpu().numpy(), buf["H"].cpu().numpy()))
    assert outs[0][0] == outs[1][0]
    assert np.array_equal(outs[0][1], outs[1][1]) and np.array_equal(outs[0][2], outs[1][2])
