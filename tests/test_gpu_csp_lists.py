"""CSP of structures in which most atoms have no clear shells, on both sides of the list length from
which they are sorted by threads (140 per SM), against the definition (needs a GPU).

Bit for bit on the exported rows, with row capacities that are and are not multiples of 4 (16-byte
row loads), from rows built at the positions (ap_step walks the in-range part first) and from
kept rows."""
import dataclasses

import numpy as np
import pytest
import torch

import ap_inputs as I
from test_gpu_kernel_paths import A, PERIODIC, context, crystal, csp_of_rows, gas

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2411_03002_gb300 as ap


@pytest.mark.parametrize("cap", [240, 241])
@pytest.mark.parametrize("per_sm", [120, 190])
def test_gas_on_both_sides_of_the_limit(per_sm, cap):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    x, box = gas(per_sm * sms)
    ctx, xt = context(x, box, cap_eam=cap)
    ctx.classify(xt)
    assert torch.equal(ctx.get_lambda_state()["csp"], csp_of_rows(ctx, xt, box))
    ctx.close()


def run(x, box, rebuild_every):
    hyb = dataclasses.replace(I.SINGLE_EVAL, dlam_min=0.0)
    ctx = ap.Context(ap.make_config(I.eam_params(0), I.ace_params_anchored(), hyb, dt=0.02, lambda_every=2,
                                    rebuild_every=rebuild_every))
    s = {k: torch.zeros(x.shape[0], 3, dtype=torch.float64, device="cuda") for k in "vf"}
    xt = torch.as_tensor(x, device="cuda").clone()
    m = torch.full((x.shape[0],), I.MASS_CU, dtype=torch.float64, device="cuda")
    lam = torch.empty_like(m)
    ctx.build_neighbors(xt, ap.make_box(*box))

    def step(k):
        return ctx.step(xt, s["v"], s["f"], m, None, lam, k)
    return ctx, xt, step


@pytest.mark.parametrize("cells", [(14, 14, 14), (24, 25, 26)])
def test_disordered_crystal_in_a_run(cells):
    """sigma = 0.25 A: most atoms are handed on, to the sort in the larger crystal."""
    box = ((0, 0, 0), tuple(A * c for c in cells), PERIODIC)
    ctx, x, step = run(crystal(*cells, 0.25), box, ap.REBUILD_SKIN)
    step(0)
    assert torch.equal(ctx.get_lambda_state()["csp"], csp_of_rows(ctx, x, box))
    s = step(4)
    assert s.kept == 2 and s.error_bits == 0
    ref, _ = context(x.cpu().numpy(), box)
    ref.classify(x)
    assert torch.equal(ctx.get_lambda_state()["csp"], ref.get_lambda_state()["csp"])
    ctx.close(), ref.close()
