"""EAM rows of bodies in boxes that are mostly vacuum, built from a list of the cell groups that
hold atoms, and of dilute gases, built by a thread per row, against all pairs (needs a GPU)."""
import numpy as np
import pytest
import torch

import ap_inputs as I
from test_gpu_kernel_paths import A, PERIODIC, all_pairs, context, crystal, row_keys

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import paper_2411_03002_gb300 as ap


def body(cells, at):
    return crystal(*cells, 0.1) + np.asarray(at)


# the body inside, across the periodic corner (unwrapped positions), in a box of three cells in x
# (stored offsets), and as two far clusters with a lone atom in a free box
CASES = {
    "inside": (body((6, 6, 6), (40, 70, 99)), ((0, 0, 0), (160, 160, 160), PERIODIC)),
    "corner": (body((6, 5, 7), (-9, -8, -12)), ((0, 0, 0), (160, 165, 158), PERIODIC)),
    "narrow": (body((3, 6, 5), (1, 395, 180)), ((0, 0, 0), (3.4 * A, 400, 404), PERIODIC)),
    "clusters": (np.concatenate([body((4, 4, 4), (3, 3, 3)), body((5, 4, 3), (140, 141, 142)), [[80.0, 20.0, 50.0]]]),
                 ((0, 0, 0), (164, 164, 164), (False, False, False))),
}


@pytest.mark.parametrize("name", CASES)
def test_rows_of_a_body_in_vacuum(name):
    x, box = CASES[name]
    ctx, xt = context(x, box)
    n = x.shape[0]
    assert torch.equal(row_keys(ctx, 0, torch.arange(n, device="cuda"), n), all_pairs(x, box, 6.5))
    ctx.close()


def test_rows_of_bodies_in_several_boxes():
    parts = [CASES["inside"], CASES["clusters"], CASES["corner"]]
    x = np.concatenate([p[0] for p in parts])
    off = np.cumsum([0] + [p[0].shape[0] for p in parts])
    ctx = ap.Context(ap.make_config(I.eam_params(0), I.ace_params_anchored(), I.SINGLE_EVAL))
    ctx.build_neighbors_batch(torch.as_tensor(x, device="cuda"), off.tolist(), [ap.make_box(*p[1]) for p in parts])
    n = x.shape[0]
    got = row_keys(ctx, 0, torch.arange(n, device="cuda"), n)
    want = []
    for (y, box), a in zip(parts, off):
        k, m = all_pairs(y, box, 6.5), y.shape[0]
        i, j, code = k // 32768 // m, k // 32768 % m, k % 32768
        want.append(((i + int(a)) * n + j + int(a)) * 32768 + code)
    assert torch.equal(got, torch.sort(torch.cat(want)).values)
    ctx.close()


def dilute(n, box, seed, cluster=0):
    lo, hi = np.asarray(box[0], float), np.asarray(box[1], float)
    g = np.random.Generator(np.random.PCG64(seed))
    x = g.uniform(lo, hi, (n, 3))
    if cluster:   # rows beyond the default capacity
        x[:cluster] = 0.5 * (lo + hi) + g.uniform(-3.0, 3.0, (cluster, 3))
    return x, box


GASES = {
    "periodic": dilute(20000, ((0, 0, 0), (168, 170, 166), PERIODIC), 1),
    "free": dilute(20000, ((-5, -5, -5), (163, 165, 161), (False, False, False)), 2, 300),
    "narrow": dilute(20000, ((0, 0, 0), (3.4 * A, 620, 610), PERIODIC), 3),
    "outside": (lambda x, b: (x + np.array([168.0, -170.0, 332.0]), b))(*dilute(20000, ((0, 0, 0), (168, 170, 166), PERIODIC), 4)),
}


@pytest.mark.parametrize("name", GASES)
def test_rows_of_a_dilute_gas(name):
    x, box = GASES[name]
    ctx, xt = context(x, box)
    n = x.shape[0]
    assert torch.equal(row_keys(ctx, 0, torch.arange(n, device="cuda"), n), all_pairs(x, box, 6.5))
    ctx.close()
