"""The float32 adjoint kernel at the edges of its tiles (ranks around multiples of 16, o-blocks
and chunks of 64 with remainders, several o-blocks per W partial, V and Vbar rows that are not
16-byte aligned): one adjoint step against the FP64 vector-Jacobian product of the same step at
the same state and selections (oracle/unrolled.step_vjp).  Tolerance: the sums of the adjoint
carry float32 rounding of up to ~1e4 terms (1e-5), and Abar, Bbar divide by b and by a
difference, which magnifies the 1e-6 of A and B by up to a hundred: 1e-3 relative Frobenius."""
import numpy as np
import pytest

import workloads
from gpu_helpers import GpuProblem, rel_fro
from oracle import unrolled as u

pytestmark = pytest.mark.gpu

TOL = 1e-3


@pytest.mark.parametrize("N,T,R", [(64, 64, 16), (65, 63, 17), (131, 200, 33), (40, 2100, 48),
                                   (700, 130, 64), (150, 141, 80), (70, 65, 112), (190, 333, 128),
                                   (30, 300, 3)])
def test_adjoint_step(N, T, R):
    import torch
    p = workloads.custom(N, T, R, seed=N + 3 * T + 5 * R)
    rng = np.random.default_rng(R)
    Hb = rng.normal(size=(R, T)).astype(np.float32)
    with GpuProblem(p.V, p.W, p.H, "f32") as gp:
        dna = gp.dna
        Hk = gp.H.clone()
        choice = torch.empty(T, dtype=torch.uint8, device="cuda")
        dna.dna_step_H_fixed(gp.ctx, choice)
        Hbar = torch.from_numpy(Hb).cuda()
        out = torch.empty_like(Hbar)
        Vbar, Wbar = torch.zeros_like(gp.V), torch.zeros_like(gp.W)
        dna.dna_step_H_adjoint_w(gp.ctx, Hk, choice, Hbar, out, Vbar, Wbar)
        out2 = torch.empty_like(Hbar)
        dna.dna_step_H_adjoint(gp.ctx, Hk, choice, Hbar, out2, Vbar)   # no W; adds into Vbar
        torch.cuda.synchronize()
        ch = choice.bool().cpu().numpy()
        dH, dV, dW = u.step_vjp(p.V.astype(np.float64), p.W.astype(np.float64),
                                p.H.astype(np.float64), ch, Hb.astype(np.float64))
        assert torch.equal(out, out2)
        assert rel_fro(out.cpu().numpy(), dH) < TOL
        assert rel_fro(Vbar.cpu().numpy() / 2, dV) < TOL
        assert rel_fro(Wbar.cpu().numpy(), dW) < TOL
