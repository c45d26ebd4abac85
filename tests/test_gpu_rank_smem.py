"""Ranks 311 to 371 on the tensor cores: the selection's dynamic shared memory (128 bytes per
rank) lies under 48 KB there, but not together with its static arrays, so the launch needs
the opt-in.  Each case runs in a process of its own: the opt-in of a larger rank would last."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CODE = """
import sys
import numpy as np
sys.path[:0] = [{root!r}, {tests!r}]
import workloads
from gpu_helpers import GpuProblem
p = workloads.custom(200, 300, {R}, seed=1)
with GpuProblem(p.V, p.W, p.H, {form!r}) as gp:
    gp.dna.dna_normalize(gp.ctx, 1)
    first = gp.dna.dna_kl(gp.ctx)
    gp.dna.dna_iterate(gp.ctx, 3)
    W, H = gp.WH()
    assert np.isfinite(W).all() and np.isfinite(H).all()
    assert gp.dna.dna_kl(gp.ctx) < first
"""


@pytest.mark.parametrize("form", ["f32", "f32t", "bf16"])
@pytest.mark.parametrize("R", [311, 340, 371])
def test_first_rank_of_a_process(form, R):
    tests = os.path.dirname(os.path.abspath(__file__))
    code = CODE.format(root=os.path.dirname(tests), tests=tests, R=R, form=form)
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
