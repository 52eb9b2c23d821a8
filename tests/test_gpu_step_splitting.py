"""One ap_step call of n steps and n calls of one step are the same run, bit for bit (needs a GPU).

Inside a call the ACE forces, the indenter and the second half kick of a step join the next
drift; at the end of a call they are kernels of their own, in the same order and rounding.  The
forces are fixed-point (the reduction order of the float ones varies), the indenter moves and
touches the surface, the bottom layers are fixed, and the run crosses rebuilds and a lambda update."""
import dataclasses

import numpy as np
import pytest
import torch

import ap_inputs as I

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2411_03002_gb300 as ap


def run(precision, thermostat, rebuild_every, calls):
    nx, nz = 10, 12
    x = I.fcc_lattice(nx, nx, nz)
    n, edge, top = x.shape[0], nx * I.A_CU, (nz - 0.5) * I.A_CU
    g = np.random.Generator(np.random.PCG64(11))
    fixed = x[:, 2] < 1.25 * I.A_CU
    x[~fixed] += 0.06 * g.standard_normal((int((~fixed).sum()), 3))
    v = np.where(fixed[:, None], 0.0, 2e-3 * g.standard_normal(x.shape))
    ind = I.Indenter(center0=np.array([edge / 2, edge / 2, top + 19.0]), velocity=np.array([1e-3, 0.0, -2e-2]), radius=20.0)
    hyb = dataclasses.replace(I.HYB1, n_csp_avg=1, n_lam_avg=1, dlam_min=0.0)
    ctx = ap.Context(ap.make_config(I.eam_params(0), I.ace_params_anchored(), hyb, precision=precision, dt=1.0, indenter=ind,
                                    lambda_every=6, rebuild_every=rebuild_every, thermostat=thermostat, deterministic=True))
    s = {"x": torch.as_tensor(x, device="cuda"), "v": torch.as_tensor(v, device="cuda")}
    s["f"] = torch.zeros_like(s["x"])
    m = torch.full((n,), I.MASS_CU, dtype=torch.float64, device="cuda")
    s["lam"] = torch.empty(n, dtype=torch.float64, device="cuda")
    fx = torch.as_tensor(fixed.astype(np.uint8), device="cuda")
    ctx.build_neighbors(s["x"], ap.make_box((0, 0, -5.0), (edge, edge, top + 15.0), (True, True, False)))
    for k in calls:
        st = ctx.step(s["x"], s["v"], s["f"], m, fx, s["lam"], k)
    ctx.close()
    return s, st


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("thermostat,rebuild_every", [(False, 4), (False, -1), (True, 4)])
def test_one_call_and_many(precision, thermostat, rebuild_every):
    prec = ap.PREC_MIXED if precision == "mixed" else ap.PREC_FP64
    a, sa = run(prec, thermostat, rebuild_every, [14])
    b, sb = run(prec, thermostat, rebuild_every, [1] * 14)
    for k in a:
        assert torch.equal(a[k], b[k]), k
    assert sa.error_bits == sb.error_bits == 0 and sa.n_precise == sb.n_precise > 0
    assert sa.e_pot == sb.e_pot and sa.e_kin == sb.e_kin
    assert sa.th_corrected == sb.th_corrected
