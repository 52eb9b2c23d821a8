"""ACE of long queues: the kernels taken from 64, 192 and 400 atoms per SM on, against the oracle;
their rows against a warp per row (needs a GPU).

* The structure repeats a small periodic cell, so the oracle needs only that cell.
* Linear and Finnis-Sinclair form, FP64 and mixed precision (bars: 1e-10 eV and 1e-9 eV/A; the
  mixed-precision bar of 1 meV/A, and seven standard deviations, 2e-4 eV, of the linear form's FP32
  energies).
* ACE rows by groups of cells: narrow boxes (stored offsets) of several systems, a random part
  of the atoms, crowded cells that need several rounds, and cells older than the positions."""
import dataclasses

import numpy as np
import pytest
import torch

import ap_inputs as I
import oracle as O
from test_gpu_kernel_paths import A, PERIODIC, context, crystal, row_keys

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2411_03002_gb300 as ap


def per_sm(k):
    return k * torch.cuda.get_device_properties(0).multi_processor_count


def count(q):
    return torch.tensor([q.numel()], dtype=torch.int64, device="cuda")


ORACLE = {}


def cell(form):
    """A periodic cell of 864 atoms: positions, edge, parameters, E and F of the oracle."""
    if form not in ORACLE:
        p = I.ace_params_anchored() if form == "linear" else I.ace_params_fs(0)
        x, L = crystal(6, 6, 6, 0.1), 6 * A
        box = I.Box(np.zeros(3), np.full(3, L), np.ones(3, bool))
        e, f = O.ace_for(p).eval(np.mod(x, L), box)
        ORACLE[form] = np.mod(x, L), L, p, e, f
    return ORACLE[form]


@pytest.mark.parametrize("form", ["linear", "fs"])
@pytest.mark.parametrize("precision,atoms_per_sm", [("fp64", 65), ("mixed", 65), ("mixed", 193), ("mixed", 401)])
def test_long_queues_match_the_oracle(precision, atoms_per_sm, form):
    x, L, p, e0, f0 = cell(form)
    tiles = (3, 4, -(-per_sm(atoms_per_sm) // (12 * x.shape[0])))
    k = np.stack(np.meshgrid(*(np.arange(t) for t in tiles), indexing="ij"), -1).reshape(-1, 1, 3) * L
    xt = torch.as_tensor((x[None] + k).reshape(-1, 3), device="cuda")
    prec = ap.PREC_FP64 if precision == "fp64" else ap.PREC_MIXED
    ctx = ap.Context(ap.make_config(I.eam_params(0), p, I.SINGLE_EVAL, precision=prec))
    ctx.build_neighbors(xt, ap.make_box((0, 0, 0), [t * L for t in tiles], PERIODIC))
    q = torch.arange(xt.shape[0], dtype=torch.int32, device="cuda")
    e, f = ctx.eval_ace(xt, torch.zeros(xt.shape[0], dtype=torch.float64, device="cuda"), q, count(q))
    de = e.cpu().numpy().reshape(-1, x.shape[0]) - e0
    df = f.cpu().numpy().reshape(-1, x.shape[0], 3) - f0
    if precision == "fp64":
        assert np.abs(de).max() < 1e-10 and np.abs(df).max() < 1e-9
    else:
        assert np.linalg.norm(df, axis=-1).max() <= 1e-3
        assert np.abs(de).max() < 2e-4 if form == "linear" else abs(de.mean()) <= 1e-6
    ctx.close()


def both_builds(ctx, x, q, cap=320):
    """Row keys of an ascending queue (cell groups) and of the descending one (a warp per row)."""
    assert q.numel() >= per_sm(400)
    lam = torch.zeros(x.shape[0], dtype=torch.float64, device="cuda")
    got = []
    for qq in (q, q.flip(0).contiguous()):
        ctx.eval_ace(x, lam, qq, count(qq), forces=False)
        assert ctx.neighbor_total(1) == int(ctx.get_neighbors(1, cap)[0].sum())   # nothing cut off by cap
        got.append(row_keys(ctx, 1, qq, x.shape[0], cap))
    return got


def test_rows_by_groups_in_narrow_boxes_of_several_systems():
    dims = [(2, 3, 40), (3, 3, 30), (2, 2, 50), (40, 3, 2)]
    parts, boxes, n, k = [], [], 0, 0
    while n < per_sm(401):
        d = dims[k % 4]
        parts.append(crystal(*d, 0.08, seed=k))
        boxes.append(ap.make_box((0, 0, 0), [c * A for c in d], PERIODIC))
        n, k = n + parts[-1].shape[0], k + 1
    x = torch.as_tensor(np.concatenate(parts), device="cuda")
    ctx = ap.Context(ap.make_config(I.eam_params(0), I.ace_params_anchored(), I.SINGLE_EVAL))
    ctx.build_neighbors_batch(x, np.cumsum([0] + [p.shape[0] for p in parts]).tolist(), boxes)
    a, b = both_builds(ctx, x, torch.arange(n, dtype=torch.int32, device="cuda"))
    assert torch.equal(a, b)
    ctx.close()


@pytest.mark.parametrize("name", ["part", "scattered", "crowded", "crowded part"])
def test_rows_by_groups(name):
    m = per_sm(401)
    if name in ("part", "scattered"):   # 22 of a group's 44 atoms, or 6 (a warp per row after all)
        c = int(np.ceil(((2.0 if name == "part" else 7.0) * m / 4) ** (1 / 3)))
        x, box = crystal(c, c, c, 0.08), ((0, 0, -4.0), (c * A, c * A, c * A + 4.0), (True, True, False))
    else:   # about five times the crystal's density; a block per cell, or per 2 x 2 x 2 cells
        n = m if name == "crowded" else 2 * m
        edge = (n / 0.42) ** (1 / 3)
        x, box = np.random.Generator(np.random.PCG64(6)).uniform(0, edge, (n, 3)), ((0, 0, 0), (edge,) * 3, PERIODIC)
    ctx, xt = context(x, box)
    n = x.shape[0]
    q = torch.randperm(n, generator=torch.Generator().manual_seed(2))[:m].sort().values.to(torch.int32).cuda()
    a, b = both_builds(ctx, xt, q, 1400 if "crowded" in name else 320)
    assert torch.equal(a, b)
    ctx.close()


def test_rows_by_groups_from_kept_cells():
    """A kept lambda update builds the queue's rows from cells older than the positions."""
    c = int(np.ceil((per_sm(401) / 4) ** (1 / 3)))
    x = torch.as_tensor(crystal(c, c, c, 0.06), device="cuda")
    n, box = x.shape[0], ap.make_box((0, 0, 0), (c * A,) * 3, PERIODIC)
    # every atom is detected
    hyb = dataclasses.replace(I.SINGLE_EVAL, csp_lo=1e-9, csp_hi=2e-9)
    ctx = ap.Context(ap.make_config(I.eam_params(0), I.ace_params_anchored(), hyb, dt=1.0, lambda_every=20,
                                    rebuild_every=ap.REBUILD_SKIN))
    v = 2.5e-3 * torch.randn(n, 3, generator=torch.Generator().manual_seed(3), dtype=torch.float64).cuda()
    f, m = torch.zeros_like(x), torch.full((n,), I.MASS_CU, dtype=torch.float64, device="cuda")
    lam = torch.empty_like(m)
    ctx.build_neighbors(x, box)
    ctx.step(x, v, f, m, None, lam, 0)
    s = ctx.step(x, v, f, m, None, lam, 20)
    assert s.kept == 1 and s.n_precise == n and s.max_disp > 0.1
    every = torch.arange(n, dtype=torch.int32, device="cuda")
    got = row_keys(ctx, 1, every, n)
    ref = ap.Context(ap.make_config(I.eam_params(0), I.ace_params_anchored(), hyb))
    ref.build_neighbors(x, box)
    ref.eval_ace(x, torch.zeros_like(m), every, count(every), forces=False)
    assert torch.equal(got, row_keys(ref, 1, every, n))
    ctx.close(), ref.close()
