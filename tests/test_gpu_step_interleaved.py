"""Evaluations on a context between two ap_step calls (needs a GPU).

ap_eval_ace and ap_classify use the context's precise queue and ACE rows.  The run goes on with
its own: positions, velocities, lambda and energies are those of a run without them.  Both runs
are FP64; a rebuild only reorders rows, so that forces differ by some 1e-13 eV/A and positions
after some steps of 1 fs by less (bars 1e-10 A and 1e-11 A/fs; 1e-7 eV of 2e5 eV for the energy)."""
import dataclasses

import numpy as np
import pytest
import torch

import ap_inputs as I

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2411_03002_gb300 as ap


class Run:
    def __init__(self, nxy, nz, rebuild_every):
        x = I.fcc_lattice(nxy, nxy, nz)
        g = np.random.Generator(np.random.PCG64(7))
        n = x.shape[0]
        lo, hi = (0, 0, -10.0), (nxy * I.A_CU, nxy * I.A_CU, nz * I.A_CU + 10.0)
        hyb = dataclasses.replace(I.HYB1, n_csp_avg=2, n_lam_avg=2)
        self.ctx = ap.Context(ap.make_config(I.eam_params(0), I.ace_params_anchored(), hyb, precision=ap.PREC_FP64, dt=1.0,
                                             lambda_every=10, rebuild_every=rebuild_every))
        self.x = torch.as_tensor(x + 0.06 * g.standard_normal(x.shape), device="cuda")
        self.v = torch.as_tensor(2e-3 * g.standard_normal(x.shape), device="cuda")
        self.f = torch.zeros_like(self.x)
        self.lam = torch.empty(n, dtype=torch.float64, device="cuda")
        self.m = torch.full((n,), I.MASS_CU, dtype=torch.float64, device="cuda")
        self.ctx.build_neighbors(self.x, ap.make_box(lo, hi, (True, True, False)))
        self.L = torch.as_tensor(np.asarray(hi) - np.asarray(lo), device="cuda")
        self.step(0)

    def step(self, k):
        return self.ctx.step(self.x, self.v, self.f, self.m, None, self.lam, k)

    def eval(self, queue):
        self.ctx.eval_ace(self.x, self.lam, queue, torch.tensor([queue.numel()], dtype=torch.int64, device="cuda"))


def subset(r):
    r.eval(torch.arange(0, r.x.shape[0], 3, dtype=torch.int32, device="cuda"))


def repeats(r):   # more than 400 entries per SM, every atom twice
    n = r.x.shape[0]
    r.eval(torch.arange(n, dtype=torch.int32, device="cuda") // 2)


def classify(r):
    r.ctx.classify(r.x)


# (what happens in between, cells of the slab, steps before and after): rebuilds between lambda
# updates (every 2 steps, or by the skin rule), and a lambda update at step 10 where the
# histories hold the run's own samples
@pytest.mark.parametrize("rebuild_every", [2, 0, -1])
@pytest.mark.parametrize("between,nxy,nz,before,after", [(subset, 14, 16, 7, 8), (repeats, 25, 25, 3, 4), (classify, 14, 16, 3, 4)],
                         ids=["subset", "repeats", "classify"])
def test_run_goes_on_with_its_own_queue(between, nxy, nz, before, after, rebuild_every):
    a, b = Run(nxy, nz, rebuild_every), Run(nxy, nz, rebuild_every)
    a.step(before), b.step(before)
    between(a)
    s0, t0 = a.step(0), b.step(0)
    assert s0.n_precise == t0.n_precise and abs(s0.e_pot - t0.e_pot) < 1e-7
    sa, sb = a.step(after), b.step(after)
    assert sa.error_bits == 0 and sa.n_precise == sb.n_precise > 0
    d = a.x - b.x
    d -= a.L * torch.round(d / a.L)
    assert d.abs().max() < 1e-10 and (a.v - b.v).abs().max() < 1e-11
    assert (a.lam - b.lam).abs().max() < 1e-9
    assert abs(sa.e_pot - sb.e_pot) < 1e-7
    a.ctx.close(), b.ctx.close()


def test_only_built_rows_are_exported():
    """A classification makes a new queue; until its ACE rows are built there are none to export."""
    r = Run(8, 10, 0)
    s = r.step(2)
    assert r.ctx.get_neighbors(1)[0].shape[0] == s.n_precise
    fresh = ap.Context(r.ctx.cfg)
    fresh.build_neighbors(r.x, ap.make_box((0, 0, -10.0), (8 * I.A_CU, 8 * I.A_CU, 10 * I.A_CU + 10.0), (True, True, False)))
    lam, queue, count = fresh.classify(r.x)
    assert int(count) > 0 and fresh.get_neighbors(1)[0].shape[0] == 0 and fresh.neighbor_total(1) == 0
    fresh.eval_ace(r.x, lam, queue, count)
    cnt = fresh.get_neighbors(1)[0]
    assert cnt.shape[0] == int(count) and fresh.neighbor_total(1) == int(cnt.sum()) > 0
    for c in (r.ctx, fresh):
        c.close()
