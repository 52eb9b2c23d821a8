"""The kernels chosen by size, against the general paths or plain FP64 torch (needs a GPU).

* EAM rows (a block per cell, a block per 2 x 2 x 2 cells, narrow boxes, crowded cells that
  need several rounds) against all pairs and images.
* ACE rows of a long ascending queue (cell groups) against the same atoms in descending order
  (a warp per row).
* CSP by thresholds, by sorting and by a warp per atom: bit for bit the definition on the
  exported rows.
* nu = 3 with queues at the edges of its blocks and of its two kernels.
* ACE adjoint with 8 and with 32 lanes per atom, for queue lengths that fill no warp.
"""
import numpy as np
import pytest
import torch

import ap_inputs as I

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2411_03002_gb300 as ap


def crystal(nx, ny, nz, sigma, seed=3):
    g = np.random.Generator(np.random.PCG64(seed))
    x = I.fcc_lattice(nx, ny, nz)
    return x + sigma * g.standard_normal(x.shape)


def context(x, box, precision=None, hyb=I.SINGLE_EVAL, **kw):
    ctx = ap.Context(ap.make_config(I.eam_params(0), I.ace_params_anchored(), hyb,
                                    precision=ap.PREC_MIXED if precision is None else precision, **kw))
    xt = torch.as_tensor(x, device="cuda")
    ctx.build_neighbors(xt, ap.make_box(*box))
    return ctx, xt


def all_pairs(x, box, rc):
    """Sorted keys (i, j, image) of every pair within rc, FP64, the defining expression."""
    lo, hi, per = (np.asarray(v, dtype=np.float64) for v in box)
    L, n, keys = hi - lo, x.shape[0], []
    xt = torch.as_tensor(x, device="cuda")
    m = [int(np.ceil(rc / L[d])) + 1 if per[d] else 0 for d in range(3)]
    for sz in range(-m[2], m[2] + 1):
        for sy in range(-m[1], m[1] + 1):
            for sx in range(-m[0], m[0] + 1):
                s = torch.as_tensor(np.array([sx, sy, sz]) * L, device="cuda")
                code = ((sz + 16) * 32 + sy + 16) * 32 + sx + 16
                for a in range(0, n, 2048):
                    d = (xt[None] + s) - xt[a:a + 2048, None]
                    r2 = d[..., 0] * d[..., 0] + d[..., 1] * d[..., 1] + d[..., 2] * d[..., 2]
                    ok = r2 < rc * rc
                    if sx == sy == sz == 0:
                        ok &= torch.arange(n, device="cuda")[None] != torch.arange(a, min(a + 2048, n), device="cuda")[:, None]
                    i, j = torch.nonzero(ok, as_tuple=True)
                    keys.append(((i + a) * n + j) * 32768 + code)
    return torch.sort(torch.cat(keys)).values


def row_keys(ctx, which, atoms, n, cap=320):
    cnt, idx, sh = ctx.get_neighbors(which, cap)
    ok = torch.arange(cap, device="cuda")[None] < cnt[:, None]
    code = ((sh[..., 2].long() + 16) * 32 + sh[..., 1].long() + 16) * 32 + sh[..., 0].long() + 16
    return torch.sort((((atoms[:, None].long() * n) + idx.long()) * 32768 + code)[ok]).values


A = I.A_CU
PERIODIC = (True, True, True)
ROW_CASES = {
    # one, two, three and five search cells per dimension, a free surface, a single pencil of cells
    "1x2x3": (crystal(2, 3, 4, 0.1), ((0, 0, 0), (2 * A, 3 * A, 4 * A), PERIODIC)),
    "5x6x7": (crystal(6, 7, 8, 0.1), ((0, 0, 0), (6 * A, 7 * A, 8 * A), PERIODIC)),
    "1x1x40": (crystal(1, 2, 44, 0.1), ((0, 0, -3.0), (A, 2 * A, 44 * A + 3.0), (True, True, False))),
    "slab": (crystal(9, 8, 5, 0.1), ((0, 0, -10.0), (9 * A, 8 * A, 5 * A + 10.0), (True, True, False))),
    # 50 atoms in a cell's volume: more atoms than lanes, more candidates than one stage
    "crowded": (np.random.Generator(np.random.PCG64(5)).uniform(0, 26.0, (1400, 3)) * np.array([1.0, 0.4, 0.4]) + 1.0,
                ((0, 0, 0), (28.0, 28.0, 28.0), PERIODIC)),
    # just below and above the number of cells from which a block takes 2 x 2 x 2 of them
    "13^3 cells": (crystal(14, 14, 15, 0.1), ((0, 0, 0), (14 * A, 14 * A, 15 * A), PERIODIC)),
    "15x14x13 cells": (crystal(16, 16, 15, 0.1), ((0, 0, 0), (16.8 * A, 15.8 * A, 15 * A), PERIODIC)),
}


@pytest.mark.parametrize("name", ROW_CASES)
def test_eam_rows_hold_every_pair(name):
    x, box = ROW_CASES[name]
    lo, hi = np.asarray(box[0], float), np.asarray(box[1], float)
    per = np.asarray(box[2])
    x = np.where(per, lo + np.mod(x - lo, hi - lo), x)
    ctx, xt = context(x, box)
    n = x.shape[0]
    assert torch.equal(row_keys(ctx, 0, torch.arange(n, device="cuda"), n, 960 if name == "crowded" else 320),
                       all_pairs(x, box, 6.5))
    ctx.close()


def test_ace_rows_of_long_queues():
    """62,500 atoms, above 400 per SM on any part with up to 156 SMs."""
    x = crystal(25, 25, 25, 0.08)
    ctx, xt = context(x, ((0, 0, -5.0), (25 * A, 25 * A, 25 * A + 5.0), (True, True, False)))
    n = x.shape[0]
    every = torch.arange(n, dtype=torch.int32, device="cuda")
    lam = torch.zeros(n, dtype=torch.float64, device="cuda")
    got = {}
    for name, q in (("groups", every), ("rows", every.flip(0).contiguous())):
        ctx.eval_ace(xt, lam, q, torch.tensor([q.numel()], dtype=torch.int64, device="cuda"))
        got[name] = row_keys(ctx, 1, q, n)
    assert torch.equal(got["groups"], got["rows"])
    ctx.close()


def csp_of_rows(ctx, x, box):
    """The definition on the exported rows: 12 nearest, six smallest |r_a + r_b|^2, ascending sum."""
    cnt, idx, sh = ctx.get_neighbors(0, 320)
    L = torch.as_tensor(np.asarray(box[1], float) - np.asarray(box[0], float), device="cuda")
    n = x.shape[0]
    out = torch.full((n,), float("inf"), dtype=torch.float64, device="cuda")
    ia, ib = np.triu_indices(12, 1)
    for a in range(0, n, 4096):
        s = slice(a, min(a + 4096, n))
        d = (x[idx[s].long()] + sh[s].double() * L) - x[s][:, None]
        r2 = d[..., 0] * d[..., 0] + d[..., 1] * d[..., 1] + d[..., 2] * d[..., 2]
        r2 = torch.where(torch.arange(320, device="cuda")[None] < cnt[s][:, None], r2, torch.full_like(r2, float("inf")))
        near = torch.topk(r2, 12, dim=1, largest=False).indices
        dn = torch.gather(d, 1, near[..., None].expand(-1, -1, 3))
        t = dn[:, ia] + dn[:, ib]
        v = torch.sort(t[..., 0] * t[..., 0] + t[..., 1] * t[..., 1] + t[..., 2] * t[..., 2], dim=1).values[:, :6]
        c = v[:, 0]
        for k in range(1, 6):
            c = c + v[:, k]
        out[s] = torch.where(cnt[s] >= 12, c, torch.full_like(c, float("inf")))
    return out


def gas(n, seed=9):
    edge = (n * A ** 3 / 4) ** (1 / 3)
    return np.random.Generator(np.random.PCG64(seed)).uniform(0, edge, (n, 3)), ((0, 0, 0), (edge,) * 3, PERIODIC)


@pytest.mark.parametrize("name", ["gas 1,000", "gas 20,000", "gas 70,000", "crystal", "hot crystal", "slab"])
def test_csp_by_every_path(name):
    """A gas has no shells: all its atoms are handed on, to a warp each (20,000) or, beyond the
    sort's limit (70,000), to the sort; 1,000 atoms take the warps at once.  The crystals are
    decided by thresholds but for a few atoms, the slab's surfaces are handed on."""
    if name.startswith("gas"):
        x, box = gas(int(name.split()[1].replace(",", "")))
    else:
        x = crystal(17, 18, 19, {"crystal": 0.05, "hot crystal": 0.13, "slab": 0.06}[name])
        box = ((0, 0, 0), (17 * A, 18 * A, 19 * A), PERIODIC)
        if name == "slab":
            box = ((0, 0, -10.0), (17 * A, 18 * A, 19 * A + 10.0), (True, True, False))
    lo, hi = np.asarray(box[0], float), np.asarray(box[1], float)
    x = np.where(np.asarray(box[2]), lo + np.mod(x - lo, hi - lo), x)
    ctx, xt = context(x, box)
    ctx.classify(xt)
    assert torch.equal(ctx.get_lambda_state()["csp"], csp_of_rows(ctx, xt, box))
    ctx.close()


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_ace_queue_lengths(precision):
    """Queues of 1 to 33 atoms (blocks of 32) and on both sides of the nu = 3 and adjoint rules,
    against FP64."""
    x = crystal(15, 15, 15, 0.08)
    box = ((0, 0, 0), (15 * A,) * 3, PERIODIC)
    ctx, xt = context(x, box, ap.PREC_MIXED if precision == "mixed" else ap.PREC_FP64)
    ref, _ = context(x, box, ap.PREC_FP64)
    n = x.shape[0]
    lam = torch.zeros(n, dtype=torch.float64, device="cuda")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    # FP32 energies of this potential scatter by 8e-6 of 3.4 eV (one standard deviation) about FP64,
    # forces have the library's mixed-precision bar of 1 meV/A
    tol_e, tol_f = (5e-4, 1e-3) if precision == "mixed" else (1e-10, 1e-10)

    def run(c, q):
        return c.eval_ace(xt, lam, q, torch.tensor([q.numel()], dtype=torch.int64, device="cuda"))

    lengths = [1, 3, 31, 32, 33] + ([64 * sms - 1, 64 * sms] if 64 * sms <= n else [n])
    for m in lengths:
        q = torch.randperm(n, generator=torch.Generator().manual_seed(m))[:m].sort().values.to(torch.int32).cuda()
        e, f = run(ctx, q)
        er, fr = run(ref, q)
        assert (e - er).abs().max() < tol_e, m
        assert (f - fr).abs().max() < tol_f, m
        assert e[q.long()].abs().min() > 0
    ctx.close()
    ref.close()


def test_adjoint_lanes_agree():
    """The same atoms as one long queue (8 lanes each) and as short ones (a warp each)."""
    x = crystal(21, 21, 20, 0.08)
    ctx, xt = context(x, ((0, 0, 0), (21 * A, 21 * A, 20 * A), PERIODIC))
    n = x.shape[0]
    lam = torch.zeros(n, dtype=torch.float64, device="cuda")
    every = torch.arange(n, dtype=torch.int32, device="cuda")
    _, f = ctx.eval_ace(xt, lam, every, torch.tensor([n], dtype=torch.int64, device="cuda"))
    g = torch.zeros_like(f)
    for q in every.split(4099):
        ctx.eval_ace(xt, lam, q.contiguous(), torch.tensor([q.numel()], dtype=torch.int64, device="cuda"), f=g)
    assert (f - g).abs().max() < 1e-3      # two FP32 results, each within the mixed-precision bar of 1 meV/A
    ctx.close()
