"""Pairs at the lower bound of the FP32 guard band around the list radius (needs a GPU).

A pair whose FP32 r^2 equals the rounded bound fl(r_list^2 - band) is neither surely inside
nor, at list radii where that bound rounds down, within the band of r_list^2: it still belongs
to the row.  All coordinates are multiples of 2^-18 or 2^-20 A and the cell origins are exact
in FP32, so the kernels' r^2 is known here."""
import dataclasses

import numpy as np
import pytest
import torch

import ap_inputs as I

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2411_03002_gb300 as ap

f32 = np.float32
BAND = f32(1e-3)


def fp32_r2(d):
    """The kernels' r^2 of exactly representable differences: x^2, then two fused products."""
    r2 = (d[:, 0] * d[:, 0]).astype(f32)
    for a in (1, 2):
        r2 = (r2.astype(np.float64) + d[:, a] * d[:, a]).astype(f32)
    return r2


def at_bound(radius, grid, count, g):
    """`count` difference vectors with FP32 r^2 == fl(radius^2 - band)."""
    sure = f32(f32(radius * radius) - BAND)
    out = []
    while sum(map(len, out)) < count:
        d = np.round(g.uniform(-0.5, 0.5, (200000, 3)) * radius / grid) * grid
        d[:, 2] = np.round(np.sqrt(np.maximum(float(sure) - d[:, 0] ** 2 - d[:, 1] ** 2, 0.0)) / grid) * grid
        out.append(d[fp32_r2(d) == sure])
    return np.concatenate(out)[:count]


def workload(radius, n, edge, pairs):
    grid = 2.0 ** -20 if radius < 4 else 2.0 ** -18
    g = np.random.Generator(np.random.PCG64(41))
    d = at_bound(radius, grid, pairs, g)
    a = np.round(g.uniform(0.5 * radius, edge - radius - 1.0, (pairs, 3)) / grid) * grid
    a[:, 2] = np.minimum(a[:, 2], edge - radius - 1.0)
    rest = np.round(g.uniform(0.0, edge - 0.5, (n - 2 * pairs, 3)) / grid) * grid
    return np.concatenate([a, a + d, rest]), pairs


def context(radius):
    eam = dataclasses.replace(I.eam_params(0), rc=radius - 1.0)
    ace = dataclasses.replace(I.ace_params_anchored(), rc=radius - 1.0)
    return ap.Context(ap.make_config(eam, ace, I.SINGLE_EVAL, skin=1.0))


def row_sets(ctx, which, cap):
    cnt, idx, _ = ctx.get_neighbors(which, cap)
    assert int(cnt.max()) <= cap
    ok = torch.arange(cap, device="cuda")[None] < cnt[:, None]
    i = torch.arange(cnt.shape[0], device="cuda")[:, None].expand(-1, cap)
    return torch.sort(i[ok] * cnt.shape[0] + idx[ok].long()).values


def pair_sets(x, radius):
    n, keys = x.shape[0], []
    for a in range(0, n, 2048):
        d = x[None] - x[a:a + 2048, None]
        ok = d[..., 0] * d[..., 0] + d[..., 1] * d[..., 1] + d[..., 2] * d[..., 2] < radius * radius
        i, j = torch.nonzero(ok, as_tuple=True)
        k = (i + a) * n + j
        keys.append(k[i + a != j])
    return torch.sort(torch.cat(keys)).values


# (list radius, atoms, box edge): a block per cell, a block per 2 x 2 x 2 cells, enough atoms for
# the ACE rows by groups of cells (400 per SM), and a gas dilute enough for a thread per row
@pytest.mark.parametrize("radius,n,edge", [(3.0, 2000, 15.0), (12.0, 1500, 60.0), (12.0, 20000, 120.0),
                                           (12.0, 64000, 120.0), (12.0, 20000, 480.0)])
def test_pairs_at_the_lower_bound_are_in_the_rows(radius, n, edge):
    x, pairs = workload(radius, n, edge, 64)
    r2 = f32(radius * radius)
    assert r2 - f32(r2 - BAND) > BAND          # the bound rounds down at these radii
    xt = torch.as_tensor(x, device="cuda")
    ctx = context(radius)
    ctx.build_neighbors(xt, ap.make_box((0, 0, 0), (edge,) * 3, (False,) * 3))
    want = pair_sets(xt, radius)
    assert torch.equal(row_sets(ctx, 0, 768), want)
    if n >= 64000:
        every = torch.arange(n, dtype=torch.int32, device="cuda")
        ctx.eval_ace(xt, torch.zeros(n, dtype=torch.float64, device="cuda"), every,
                     torch.tensor([n], dtype=torch.int64, device="cuda"), forces=False)
        assert torch.equal(row_sets(ctx, 1, 768), want)
    ctx.close()
