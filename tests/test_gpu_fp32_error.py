"""The FP32 error of ACE energies and forces against FP64 (needs a GPU).

Both row builds (cell groups for the ascending queue, a warp per row for the descending one) on
67,200 atoms of a thermal slab and 74,400 of a thermal crystal.  The bars are what an evaluation
with normalised harmonics and the rows of a warp measured on such structures, of energies of
about -3.4 eV: rms 2.81e-5 and 2.85e-5 eV, mean 4.3e-6 and 4.1e-6 eV, forces 5.44e-6 and 5.33e-6
relative, each with two standard errors of its estimate (0.55 % of an rms, 2.1e-7 eV)."""
import numpy as np
import pytest
import torch

import ap_inputs as I
from test_gpu_kernel_paths import A, PERIODIC, context, crystal

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2411_03002_gb300 as ap


@pytest.mark.parametrize("name", ["slab", "bulk"])
def test_fp32_error_against_fp64(name):
    if name == "slab":
        x, box = crystal(20, 21, 40, 0.06), ((0, 0, -10.0), (20 * A, 21 * A, 39.5 * A + 10.0), (True, True, False))
    else:
        x, box = crystal(24, 25, 31, 0.06), ((0, 0, 0), (24 * A, 25 * A, 31 * A), PERIODIC)
    bar_rms, bar_mean, bar_f = (2.83e-5, 4.5e-6, 5.47e-6) if name == "slab" else (2.87e-5, 4.3e-6, 5.36e-6)
    n = x.shape[0]
    lam = torch.zeros(n, dtype=torch.float64, device="cuda")
    every = torch.arange(n, dtype=torch.int32, device="cuda")
    count = torch.tensor([n], dtype=torch.int64, device="cuda")
    ref, xt = context(x, box, ap.PREC_FP64)
    e0, f0 = ref.eval_ace(xt, lam, every, count)
    ref.close()
    ctx, xt = context(x, box)
    for q in (every, every.flip(0).contiguous()):
        e, f = ctx.eval_ace(xt, lam, q, count)
        d = e - e0
        assert float(d.pow(2).mean().sqrt()) <= bar_rms
        assert abs(float(d.mean())) <= bar_mean
        assert float((f - f0).norm() / f0.norm()) <= bar_f
    ctx.close()
