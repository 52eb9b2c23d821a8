"""Thermostat corrections from rows beyond the 192 entries that the sweep holds in registers, with
and without repeated atoms in the rows, against the oracle (needs a GPU).

A skin of 3 A makes rows of 185 to 220 entries; the 4-cell box (14.5 A) holds images of one atom in
a row, the 7-cell box (25.3 A) does not.  One lambda-update step in FP64 as in the other thermostat
tests, with their bar (1e-9 relative)."""
import dataclasses

import numpy as np
import pytest
import torch

import ap_inputs as I
import oracle as O
import oracle.thermostat as TH
from test_gpu_thermostat import fresh_hyb

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2411_03002_gb300 as ap

SKIN = 3.0


def oracle_step(x, box, hyb, v0, m, dt):
    eam, ace, n = I.eam_params(0), O.ACE(I.ace_params(0)), x.shape[0]
    st = O.LambdaState(n, hyb.n_csp_avg, hyb.n_lam_avg)
    r_row = float(eam.rc) + SKIN
    lam0, *_ = O.classify(st, x, box, hyb, r_search=r_row)
    _, f0, _, _ = O.hybrid(x, box, lam0, eam, ace)
    vh = v0 + 0.5 * dt * f0 * O.ACC / m[:, None]
    x1 = x + dt * vh
    lam1, *_ = O.classify(st, x1, box, hyb, r_search=r_row)
    _, fd, ef, _ = O.hybrid(x1, box, lam1, eam, ace)
    _, fc, _, _ = O.hybrid(x1, box, lam0, eam, ace)
    ep, _ = ace.eval(x1, box)
    dE = TH.delta_v(lam0, lam1, ef, ep) + TH.delta_t(fc, fd, vh, m, dt)
    v1 = vh + 0.5 * dt * fd * O.ACC / m[:, None]
    return v1, *TH.correct(x1, box, v1, m, dE, r_row, SKIN)


@pytest.mark.parametrize("cells", [4, 7])
def test_long_rows(cells):
    L = cells * I.A_CU
    g = np.random.Generator(np.random.PCG64(21))
    x = I.fcc_lattice(cells, cells, cells)
    x = x[np.linalg.norm(x - np.round(cells / 2) * I.A_CU, axis=1) >= 4.0]   # a void: lambda < 1 around it
    x = x + 0.05 * g.standard_normal(x.shape)
    n, dt = x.shape[0], 1.0
    m = np.full(n, I.MASS_CU)
    v0 = I.maxwell_boltzmann(m, np.ones(n, bool), 900.0, g)
    box = I.Box(np.zeros(3), np.full(3, L), np.ones(3, bool))
    hyb = dataclasses.replace(fresh_hyb(I.SINGLE_EVAL), csp_lo=1.0, csp_hi=4.0)
    v1, v1c, n_ok, n_bad = oracle_step(x, box, hyb, v0, m, dt)
    assert n_ok > 0 and n_bad == 0 and np.abs(v1 - v1c).max() > 0
    ctx = ap.Context(ap.make_config(I.eam_params(0), I.ace_params(0), hyb, precision=ap.PREC_FP64, dt=dt, lambda_every=1,
                                    thermostat=True, skin=SKIN))
    s = [torch.as_tensor(a, device="cuda").clone() for a in (x, v0, np.zeros_like(x), m)]
    lam = torch.empty(n, dtype=torch.float64, device="cuda")
    ctx.build_neighbors(s[0], box)
    ctx.step(*s, None, lam, 0)
    st = ctx.step(*s, None, lam, 1)
    rows = ctx.get_neighbors(0, 320)[0]
    assert int(rows.max()) <= 320 and int((rows > 192).sum()) > n // 2   # the sweep meets both kinds
    assert st.th_refused == 0 and st.th_corrected == n_ok
    scale = np.abs(v1c).max()
    assert np.abs(s[1].cpu().numpy() - v1c).max() <= 1e-9 * scale
    ctx.close()
