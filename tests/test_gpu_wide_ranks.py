"""Ranks above 128, where the tensor-core forms take only the 64-wide slices of a padded rank
that hold values and cut r into equal blocks; and ranks above 256 in float32, where the candidates kernel walks r in groups of 32 and
writes the bf16 rows of the tensor-core forms: the edges of its rank range, column counts
that leave a partial CTA, one and several splits of the sums.  Each half-step starts from
the GPU's own state and is held to the element-wise one-step bounds of gpu_helpers; the FP32
forms also to their Frobenius tolerances (1e-4, split FP32 above rank 300 2e-4).  BF16 has
none here: with fewer columns than a thirtieth of the rank the Newton step a / b magnifies
the operands' rounding (N=517 T=16 R=511: 4e-2), which the element-wise bound follows."""
import numpy as np
import pytest

import workloads
from gpu_helpers import GpuProblem, one_step_check, rel_fro, replay_choice
from oracle import dna as o

pytestmark = pytest.mark.gpu

TOL = {"f32": 1e-4, "f32t": 2e-4}


def one_iteration(form, N, T, R):
    p = workloads.custom(N, T, R, seed=N + 3 * T + 7 * R)
    V = p.V.astype(np.float64)
    with GpuProblem(p.V, p.W, p.H, form) as gp:
        gp.dna.dna_normalize(gp.ctx, 1)
        for which in (0, 1):
            W0, H0 = gp.WH()
            (gp.dna.dna_step_H if which == 0 else gp.dna.dna_step_W)(gp.ctx)
            assert one_step_check(gp, which, W0, H0, label=form) <= 1.0
            if form not in TOL:
                continue
            half = (o.h_half_step if which == 0 else o.w_half_step)(V, W0, H0)
            mask, _ = replay_choice(half, gp.choice(which), form)
            W, H, _ = (o.dna_step_h if which == 0 else o.dna_step_w)(V, W0, H0, choice=mask)
            Wg, Hg = gp.WH()
            assert rel_fro(Wg, W) < TOL[form] and rel_fro(Hg, H) < TOL[form], which


@pytest.mark.parametrize("form", ["f32t", "bf16"])
@pytest.mark.parametrize("R", [129, 144, 145, 192, 193, 256, 300, 320, 400, 448, 449])
def test_rank_slices(form, R):
    one_iteration(form, 700, 1300, R)


@pytest.mark.parametrize("form", ["f32", "f32t", "bf16"])
@pytest.mark.parametrize("N,T,R", [(33, 47, 257), (130, 65, 288), (300, 4100, 289), (517, 16, 511),
                                   (640, 1, 512), (2100, 401, 384)])
def test_half_steps(form, N, T, R):
    one_iteration(form, N, T, R)
