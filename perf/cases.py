"""What a user of this library has it do, as cases that can be timed and checked.

kind "forces"    one adaptive force evaluation of a structure: neighbour build, classification
                 (or a given lambda), EAM, ACE, blend.  Sampling, relaxation and labelling do this.
kind "gradient"  the autograd function: energy, then its gradient through the adjoint kernels.
kind "lambda"    neighbour build and one lambda update, without forces (analysis of a snapshot).
kind "md"        `steps` velocity-Verlet steps of a running simulation through Context.step.
kind "scores"    neighbour build, selector features and selector scores of a structure.
kind "train"     `steps` Adam steps of the selector on batches of a resident data set.

In mixed precision the potentials are FP32, and the arrays that a program keeps of a pass (the
trajectory frame, the forces of a sample) are single precision too: `run` returns them so.  In
FP64 the library's own FP64 arrays are returned.  A lambda that is computed from given positions
is FP64 in both.  All inputs are made on the GPU from the seed.
"""
import dataclasses
import math

import numpy as np
import torch

import ap_inputs as I
import paper_2411_03002_gb300 as ap
from paper_2411_03002_gb300 import autograd as ap_autograd

A0 = I.A_CU
PAD = 10.0            # vacuum above and below a slab (A)
DENSITY = 4.0 / A0 ** 3


# --------------------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest call: a 237-atom periodic cell with a void (narrower than five search cells)
        dict(name="cell_forces", kind="forces", shape="void", nx=4, ny=4, nz=4, sigma=0.05, precision="mixed",
             lam="classify", zone="single", ace="seeded", eam="analytic"),
        # finite-difference checks, relaxations and phonons of small cells want FP64 gradients
        dict(name="cell_gradient_fp64", kind="gradient", cells=1, nx=8, ny=8, nz=8, sigma=0.1, precision="fp64"),
        # a training or screening batch: 64 independent cells of 500 to 4,000 atoms in one launch
        dict(name="batch_gradient", kind="gradient", cells=64, lo=5, hi=10, sizes=1, sigma=0.1, precision="mixed"),
        # the parity mode: one adaptive evaluation of the 32,000-atom slab with a disordered hemisphere
        dict(name="slab_forces_fp64", kind="forces", shape="slab", nx=20, ny=20, nz=20, sigma=0.05, disorder=0.3,
             precision="fp64", lam="classify", zone="hyb1", ace="anchored", eam="analytic"),
        # molecular dynamics of a small system: launches and host round trips count
        dict(name="slab_md", kind="md", nx=20, ny=20, nz=20, steps=10, precision="mixed", zone="hyb1", rebuild=5,
             skin=1.0, fixed=False, indenter=False, thermostat=False, fixed_point=False),
        # production MD as the paper runs it, with the local thermostat; odd sizes
        dict(name="thermostat_md", kind="md", nx=37, ny=41, nz=59, steps=10, precision="mixed", zone="hyb2",
             rebuild=0, skin=0.7, fixed=True, indenter=True, thermostat=True, fixed_point=False),
        # the 4,000,000-atom nanoindentation run, lists on the skin criterion (the benchmark's workload)
        dict(name="indent_md_4m", kind="md", nx=100, ny=100, nz=100, steps=10, precision="mixed", zone="hyb2",
             rebuild=-1, skin=0.7, fixed=True, indenter=True, thermostat=False, fixed_point=False),
        # every atom precise: the reference forces that adaptive runs are judged against
        dict(name="full_ace_forces", kind="forces", shape="slab", nx=39, ny=40, nz=41, sigma=0.06, precision="mixed",
             lam="zero", zone="hyb1", ace="anchored", eam="analytic"),
        # every atom fast, with the paper's copper EAM: bulk screening of large cells
        dict(name="mishin_forces", kind="forces", shape="bulk", nx=61, ny=63, nz=65, sigma=0.07, precision="mixed",
             lam="one", zone="hyb1", ace="anchored", eam="mishin"),
        # classification of a large defected snapshot
        dict(name="lambda_update", kind="lambda", shape="slab", nx=59, ny=61, nz=67, sigma=0.06, vacancy=2e-4,
             zone="hyb1", precision="mixed", ace="anchored", eam="analytic"),
        # the learned detector on a slab: features and scores of every atom
        dict(name="selector_scores", kind="scores", shape="slab", nx=31, ny=32, nz=33, sigma=0.07, disorder=0.2,
             precision="mixed", zone="hyb1", ace="anchored", eam="analytic"),
        # selector training: eight Adam steps on batches of the size that the training driver uses
        dict(name="selector_train", kind="train", samples=131072, batch=8192, steps=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _dims(rng, lo, hi, cap):
    """Three edge lengths in cells, each lo..hi, with at most `cap` cells in all."""
    while True:
        m = _log_int(rng, lo, hi)
        d = [max(lo, min(hi, m + rng.randint(-max(1, m // 5), max(1, m // 5)))) for _ in range(3)]
        if d[0] * d[1] * d[2] <= cap:
            return dict(nx=d[0], ny=d[1], nz=d[2])


def draw(rng):
    kind = rng.choice(["forces", "forces", "forces", "md", "md", "gradient", "lambda", "scores", "train"])
    if kind == "train":
        batch = rng.choice([1024, 4096, 8192, 8192, 16384, rng.randint(300, 20000)])
        return dict(kind=kind, samples=batch * rng.randint(4, 24) + rng.randint(0, batch), batch=batch,
                    steps=rng.randint(1, 12))
    if kind == "gradient":
        fp64 = rng.random() < 0.5
        if rng.random() < 0.5:
            return dict(kind=kind, cells=1, sigma=round(rng.uniform(0.03, 0.15), 3), precision="fp64" if fp64 else "mixed",
                        **_dims(rng, 3, 12 if fp64 else 24, 1000 if fp64 else 12000))
        return dict(kind=kind, cells=rng.randint(2, 6 if fp64 else 90), lo=rng.randint(3, 5), hi=rng.randint(6, 11 if not fp64 else 7),
                    sizes=rng.randint(2, 10 ** 6), sigma=round(rng.uniform(0.03, 0.15), 3),
                    precision="fp64" if fp64 else "mixed")
    fp64 = rng.random() < 0.25
    if kind == "md":
        skin = rng.choice([0.6, 0.7, 0.8, 1.0])
        rebuild = rng.choice([-1, -1, 0, 5])
        thermostat = rng.random() < 0.2
        d = _dims(rng, 8, 20 if fp64 else 90, 3000 if fp64 else 600000)
        return dict(kind=kind, steps=rng.choice([10, 10, 10, 20]), precision="fp64" if fp64 else "mixed",
                    zone=rng.choice(["hyb1", "hyb2"]), rebuild=0 if thermostat else rebuild, skin=skin,
                    fixed=rng.random() < 0.5, indenter=rng.random() < 0.5, thermostat=thermostat,
                    fixed_point=rng.random() < 0.25, **d)
    if kind == "scores":
        return dict(kind=kind, shape=rng.choice(["slab", "bulk"]), sigma=round(rng.uniform(0.04, 0.12), 3),
                    disorder=rng.choice([0.0, 0.2, 0.4]), precision="mixed", zone="hyb1", ace="anchored",
                    eam="analytic", **_dims(rng, 7, 60, 150000))
    if kind == "lambda":
        return dict(kind=kind, shape=rng.choice(["slab", "slab", "bulk"]), sigma=round(rng.uniform(0.03, 0.09), 3),
                    vacancy=rng.choice([1e-4, 2e-4, 1e-3]), zone=rng.choice(["hyb1", "hyb2"]), precision="mixed",
                    ace="anchored", eam="analytic", **_dims(rng, 9, 80, 300000))
    lam = rng.choice(["classify", "classify", "zero", "one", "mix"])
    cap = 5000 if fp64 else 250000 if lam in ("one", "classify") else 60000
    return dict(kind=kind, shape=rng.choice(["slab", "bulk", "void"]), sigma=round(rng.uniform(0.03, 0.12), 3),
                precision="fp64" if fp64 else "mixed", lam=lam, zone=rng.choice(["single", "hyb1", "hyb2"]),
                ace=rng.choice(["seeded", "anchored", "anchored", "fs"]),
                eam=rng.choice(["analytic", "analytic", "mishin"]), **_dims(rng, 4, 17 if fp64 else 62, cap))


# --------------------------------------------------------------------------- inputs
def _gen(seed, k=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 16 + k)
    return g


def _randn(shape, g):
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)


def _rand(n, g):
    return torch.rand(n, generator=g, device="cuda", dtype=torch.float64)


def _fcc(nx, ny, nz):
    """FCC sites, z layers outermost (the order of ap_inputs.fcc_lattice), on the GPU."""
    k, j, i = torch.meshgrid(*(torch.arange(m, device="cuda", dtype=torch.float64) for m in (nz, ny, nx)), indexing="ij")
    cells = torch.stack([i.reshape(-1), j.reshape(-1), k.reshape(-1)], 1)
    basis = torch.tensor([[0.0, 0.0, 0.0], [0.5, 0.5, 0.0], [0.5, 0.0, 0.5], [0.0, 0.5, 0.5]], device="cuda",
                         dtype=torch.float64)
    return ((cells[:, None, :] + basis[None]) * A0).reshape(-1, 3)


def _sites(case):
    """(sites, box lo, box hi, periodic) of a case's structure; the number of atoms depends on the case alone."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    x = _fcc(nx, ny, nz)
    if case.get("shape", "slab") == "slab":
        return x, (0.0, 0.0, -PAD), (nx * A0, ny * A0, (nz - 0.5) * A0 + PAD), (True, True, False)
    if case["shape"] == "void":
        c = torch.tensor([nx // 2, ny // 2, nz // 2], device="cuda", dtype=torch.float64) * A0
        x = x[torch.linalg.vector_norm(x - c, dim=1) >= 4.0]
    return x, (0.0, 0.0, 0.0), (nx * A0, ny * A0, nz * A0), (True, True, True)


def _structure(case, seed):
    """Positions of a case with its vacancies, its thermal noise and its disordered hemisphere."""
    x, lo, hi, per = _sites(case)
    g = _gen(seed)
    if case.get("vacancy"):
        keep = torch.ones(x.shape[0], dtype=torch.bool, device="cuda")
        keep[torch.randperm(x.shape[0], generator=g, device="cuda")[:max(1, round(case["vacancy"] * x.shape[0]))]] = False
        x = x[keep]
    sig = torch.full((x.shape[0], 1), float(case["sigma"]), device="cuda", dtype=torch.float64)
    if case.get("disorder"):
        top = torch.tensor([hi[0] / 2, hi[1] / 2, (case["nz"] - 0.5) * A0], device="cuda", dtype=torch.float64)
        inside = torch.linalg.vector_norm(x - top, dim=1) < min(15.0, 0.4 * hi[0])
        sig[inside] = float(case["disorder"])
    return (x + sig * _randn(x.shape, g)).contiguous(), lo, hi, per


def _batch(case, seed):
    """Independent periodic cells: positions, offsets and box lengths, with a lambda of thirds 0, 1 and U(0, 1)."""
    if case["cells"] == 1:
        dims = [(case["nx"], case["ny"], case["nz"])]
    else:
        dims = np.random.RandomState(case["sizes"]).randint(case["lo"], case["hi"] + 1, (case["cells"], 3)).tolist()
    g = _gen(seed)
    xs = [_fcc(*d) for d in dims]
    off = np.concatenate([[0], np.cumsum([x.shape[0] for x in xs])]).tolist()
    x = torch.cat(xs)
    x = (x + case["sigma"] * _randn(x.shape, g)).contiguous()
    return x, off, [[m * A0 for m in d] for d in dims], _mix(x.shape[0], seed)


def _mix(n, seed):
    cat = torch.randint(0, 3, (n,), generator=_gen(seed, 1), device="cuda")
    u = _rand(n, _gen(seed, 2))
    return torch.where(cat == 0, 0.0, torch.where(cat == 1, 1.0, u)).contiguous()


def _eam(case):
    return I.MISHIN_ORIGINAL if case.get("eam") == "mishin" else I.eam_params(0)


def _ace(case):
    kind = case.get("ace", "anchored")
    return I.ace_params_anchored() if kind == "anchored" else I.ace_params_fs() if kind == "fs" else I.ace_params(0)


def _zone(case):
    z = {"single": I.SINGLE_EVAL, "hyb1": I.HYB1, "hyb2": I.HYB2}[case.get("zone", "hyb1")]
    # one evaluation of one structure has one sample; a snapshot's update and MD keep their windows
    return dataclasses.replace(z, n_csp_avg=1, n_lam_avg=1) if case["kind"] in ("forces", "scores") else z


def _prec(case):
    return ap.PREC_FP64 if case["precision"] == "fp64" else ap.PREC_MIXED


def _selector_model():
    import os
    d = np.load(os.path.join(os.path.dirname(ap.__file__), "selector_cu.npz"))
    return d["params"], d["mu"], d["inv_sigma"]


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind == "train":
        g = _gen(seed)
        params, mu, inv = _selector_model()
        n, b = case["samples"], case["batch"]
        noise = torch.randn((n, 24), generator=g, device="cuda")
        mu_t, sd_t = torch.as_tensor(mu, device="cuda"), 1.0 / torch.as_tensor(inv, device="cuda")
        y = (torch.rand(n, generator=g, device="cuda") < 0.3).float()
        st["feat"] = (mu_t + sd_t * (noise + 0.4 * y[:, None])).contiguous()
        st["label"] = y
        st["weight"] = torch.where(y > 0.5, 0.5 / 0.3, 0.5 / 0.7) / b
        st["batches"] = [torch.randint(0, n, (b,), generator=g, device="cuda").to(torch.int32) for _ in range(case["steps"])]
        w0 = np.random.RandomState(seed % (1 << 31)).standard_normal(ap.SEL_NPARAMS).astype(np.float32) * 0.02
        st["ctx"] = ap.Context(ap.make_config(I.eam_params(0), I.ace_params(0), I.HYB1))
        st["ctx"].sel_set_model(params + w0, mu, inv)
        st["loss"] = torch.zeros(case["steps"], device="cuda")
        return st
    if kind == "gradient":
        x, off, lengths, lam = _batch(case, seed)
        hyb = I.SINGLE_EVAL
        st["ctx"] = ap.Context(ap.make_config(I.eam_params(0), I.ace_params(0), hyb, precision=_prec(case)))
        boxes = [ap.make_box((0.0, 0.0, 0.0), L, (True, True, True)) for L in lengths]
        st.update(x=x, lam=lam, box=boxes[0], batch=(off, boxes) if case["cells"] > 1 else None)
        return st
    if kind == "md":
        x, lo, hi, per = _sites(case)
        n = x.shape[0]
        g = _gen(seed)
        fixed = (x[:, 2] < 1.25 * A0) if case["fixed"] else torch.zeros(n, dtype=torch.bool, device="cuda")
        mobile = (~fixed)[:, None].to(torch.float64)
        x = (x + 0.06 * mobile * _randn(x.shape, g)).contiguous()   # a thermal start, as in the middle of a run
        v = mobile * _randn(x.shape, g) * math.sqrt(I.KB_EV * 300.0 * I.ACC_EV_A_AMU / I.MASS_CU)
        v = v - mobile * (v.sum(0) / mobile.sum())
        ztop = (case["nz"] - 0.5) * A0
        ind = I.Indenter(center0=np.array([hi[0] / 2, hi[1] / 2, ztop + 50.0]), velocity=np.array([0.0, 0.0, -2.0e-4]),
                         radius=50.0, k=10.0) if case["indenter"] else None
        cfg = ap.make_config(I.eam_params(0), I.ace_params_anchored(), _zone(case), precision=_prec(case), skin=case["skin"],
                             dt=1.0, indenter=ind, lambda_every=10, rebuild_every=case["rebuild"],
                             thermostat=case["thermostat"], deterministic=case["fixed_point"])
        ctx = ap.Context(cfg)
        st.update(ctx=ctx, x=x, v=v.contiguous(), f=torch.zeros_like(x), lam=torch.empty(n, dtype=torch.float64, device="cuda"),
                  mass=torch.full((n,), I.MASS_CU, dtype=torch.float64, device="cuda"),
                  fixed=fixed.to(torch.uint8) if case["fixed"] else None)
        ctx.build_neighbors(x, ap.make_box(lo, hi, per))
        ctx.step(st["x"], st["v"], st["f"], st["mass"], st["fixed"], st["lam"], 0)   # the simulation is running
        return st
    x, lo, hi, per = _structure(case, seed)
    n = x.shape[0]
    ctx = ap.Context(ap.make_config(_eam(case), _ace(case), _zone(case), precision=_prec(case)))
    st.update(ctx=ctx, x=x, box=ap.make_box(lo, hi, per))
    if kind == "scores":
        ctx.sel_set_model(*_selector_model())
    elif kind == "forces" and case["lam"] != "classify":
        st["lam"] = (_mix(n, seed) if case["lam"] == "mix" else
                     torch.full((n,), 0.0 if case["lam"] == "zero" else 1.0, dtype=torch.float64, device="cuda"))
    return st


def run(state):
    case, ctx = state["case"], state["ctx"]
    kind = case["kind"]
    keep = (lambda t: t) if case.get("precision") == "fp64" else (lambda t: t.float())
    if kind == "train":
        for k, idx in enumerate(state["batches"]):
            ctx.sel_train_step(state["feat"], state["label"], state["weight"], idx=idx, lr=1e-3, loss=state["loss"][k:k + 1])
        return {"params": ctx.sel_get_model()[0], "loss": state["loss"]}
    if kind == "gradient":
        x = state["x"].detach().requires_grad_()
        e = ap_autograd.energy(x, state["lam"], ctx, box=state["box"], batch=state["batch"])
        (g,) = torch.autograd.grad(e, x)
        return {"energy": keep(e), "grad": keep(g)}
    if kind == "md":
        s = ctx.step(state["x"], state["v"], state["f"], state["mass"], state["fixed"], state["lam"], case["steps"])
        return {"x": keep(state["x"]), "v": keep(state["v"]), "f": keep(state["f"]), "lam": keep(state["lam"]),
                "e_pot": s.e_pot, "e_kin": s.e_kin}
    x = state["x"]
    ctx.build_neighbors(x, state["box"])
    if kind == "lambda":
        lam, _, count = ctx.classify(x)
        return {"lam": lam, "count": count}
    if kind == "scores":
        feat = ctx.sel_features(x)
        p, logit = ctx.sel_predict(feat)
        return {"feat": feat, "p": p, "logit": logit}
    if case["lam"] == "classify":
        lam, queue, count = ctx.classify(x)
    else:
        lam = state["lam"]
        queue, count = ctx.precise_queue(lam)
    e_fast, f = ctx.eval_eam(x, lam)
    e_prec, f = ctx.eval_ace(x, lam, queue, count, f=f)
    e_atom, e_tot = ctx.blend_forces(lam, e_fast, e_prec)
    out = {"f": keep(f), "e_atom": keep(e_atom), "e_tot": keep(e_tot), "count": count}
    if case["lam"] == "classify":
        out["lam"] = lam
    return out


# --------------------------------------------------------------------------- what a pass cannot do without
PAIRS_EAM, PAIRS_ACE = 54.0, 134.0           # FCC neighbours inside 5.5 and 7 A
FLOP_EAM = 80.0                              # per ordered pair and evaluation: zeta, Phi, their derivatives, the force
FLOP_ACE_PAIR = 510.0 + 1580.0               # per pair inside the ACE cutoff: A-basis, then the adjoint
FLOP_ACE_ATOM = 7000.0 + 11400.0 + 3300.0    # per precise atom: A, B (nu <= 3) and the gradient


def _atoms(case):
    if case["kind"] == "gradient" and case["cells"] > 1:
        d = np.random.RandomState(case["sizes"]).randint(case["lo"], case["hi"] + 1, (case["cells"], 3))
        return int(4 * d.prod(1).sum())
    n = 4 * case["nx"] * case["ny"] * case["nz"]
    if case.get("shape") == "void":
        n -= 19
    return n


def _precise(case, n):
    """Atoms with lambda < 1, from the geometry: layers within the outer radius of a free surface."""
    lam = case.get("lam", "mix" if case["kind"] == "gradient" else "classify")
    if lam != "classify":
        return {"zero": n, "one": 0, "mix": 2 * n // 3}[lam]
    r_hi = _zone(case).r_hi
    if case.get("shape", "slab") == "slab":
        surfaces = 1 if case.get("fixed") else 2
        return int(min(1.0, surfaces * (r_hi + A0 / 2) / (case["nz"] * A0)) * n)
    if case["shape"] == "void":
        return int(min(n, DENSITY * 4.0 / 3.0 * math.pi * (4.0 + r_hi) ** 3))
    return 0


def work(case):
    kind = case["kind"]
    if kind == "train":
        b, steps = case["batch"], case["steps"]
        return {"bytes": steps * (b * (24 * 4 + 4 + 4 + 4) + 7 * 4 * ap.SEL_NPARAMS), "flops": steps * b * 6.0 * (24 * 64 + 64 * 64 + 64)}
    n = _atoms(case)
    if kind == "scores":
        return {"bytes": n * (24 + 96 + 8), "flops": n * (PAIRS_EAM * 60.0 + 66 * 8.0 + 2.0 * (24 * 64 + 64 * 64 + 64))}
    if kind == "lambda":
        return {"bytes": n * (24 + 8), "flops": n * (PAIRS_EAM * 10.0 + 66 * 8.0)}
    ace = _precise(case, n) * (PAIRS_ACE * FLOP_ACE_PAIR + FLOP_ACE_ATOM)
    eam = n * PAIRS_EAM * FLOP_EAM
    if kind == "md":
        return {"bytes": n * (24 * 6 + 8 + 8), "flops": case["steps"] * (eam + ace)}
    if kind == "gradient":
        return {"bytes": n * (24 + 8 + 24), "flops": 2.0 * eam + ace * 1.3}
    return {"bytes": n * (24 + 8 + 24 + 8), "flops": eam + ace}


# --------------------------------------------------------------------------- the same in plain torch, 64 bits
def _pair_chunks(x, lo, hi, per, rc, centers, chunk):
    """For chunks of `centers`: (centers of the chunk, j [c, K], d [c, K, 3], mask [c, K]) with d = x_j + s L - x_i
    over every image within rc; a cell list over the atoms and their ghosts."""
    dev = x.device
    lo_t, L = torch.tensor(lo, device=dev, dtype=torch.float64), torch.tensor([h - l for h, l in zip(hi, lo)], device=dev, dtype=torch.float64)
    per_t = torch.tensor(per, device=dev)
    nw = torch.where(per_t, torch.floor((x - lo_t) / L), torch.zeros_like(x))
    xw = x - nw * L
    gx, gj = [xw], [torch.arange(x.shape[0], device=dev)]
    for d in range(3):      # ghosts dimension by dimension, from what is there already
        if not per[d]:
            continue
        bx, bj = torch.cat(gx), torch.cat(gj)
        m = int(math.ceil((rc + 1e-9) / float(L[d])))
        for s in range(-m, m + 1):
            if s == 0:
                continue
            y = bx.clone()
            y[:, d] += s * L[d]
            k = (y[:, d] > lo_t[d] - rc) & (y[:, d] < lo_t[d] + L[d] + rc)
            gx.append(y[k])
            gj.append(bj[k])
    ax, aj = torch.cat(gx), torch.cat(gj)
    o = ax.amin(0) - 1e-6
    c3 = torch.floor((ax - o) / rc).long()
    nc = [int(v) + 3 for v in c3.amax(0)]
    cid = ((c3[:, 2] + 1) * nc[1] + c3[:, 1] + 1) * nc[0] + c3[:, 0] + 1
    order = torch.argsort(cid)
    cnt = torch.bincount(cid, minlength=nc[0] * nc[1] * nc[2])
    start = torch.cumsum(cnt, 0) - cnt
    most = int(cnt.max())
    sx, sj = ax[order], aj[order]
    own = torch.empty(ax.shape[0], dtype=torch.long, device=dev)
    own[order] = torch.arange(ax.shape[0], device=dev)
    steps = torch.tensor([(dz * nc[1] + dy) * nc[0] + dx for dz in (-1, 0, 1) for dy in (-1, 0, 1) for dx in (-1, 0, 1)], device=dev)
    slot = torch.arange(most, device=dev)
    for b in range(0, centers.shape[0], chunk):
        c = centers[b:b + chunk]
        cells = cid[c][:, None] + steps
        p = (start[cells][:, :, None] + slot).reshape(c.shape[0], -1)
        ok = (slot < cnt[cells][:, :, None]).reshape(c.shape[0], -1) & (p != own[c][:, None])
        p = torch.where(ok, p, torch.zeros_like(p))
        d = sx[p] - xw[c][:, None, :]
        r2 = (d * d).sum(-1)
        ok &= r2 < rc * rc
        num = ok.sum(1)
        K = max(1, int(num.max()))
        at = torch.argsort(ok.to(torch.int8), dim=1, descending=True, stable=True)[:, :K]
        mask = torch.arange(K, device=dev) < num[:, None]
        yield c, sj[torch.gather(p, 1, at)], torch.gather(d, 1, at[..., None].expand(-1, -1, 3)), mask


def _fcut(t):
    v = 1.0 - 1.875 * t + 1.25 * t ** 3 - 0.375 * t ** 5
    return torch.where(t < 0, torch.ones_like(t), torch.where(t > 1, torch.zeros_like(t), v))


def _exact_lambda(x, lo, hi, per, hyb, r_search):
    n = x.shape[0]
    csp = torch.full((n,), math.inf, dtype=torch.float64, device=x.device)
    ia, ib = (torch.as_tensor(v, device=x.device) for v in np.triu_indices(12, 1))
    for c, _, d, mask in _pair_chunks(x, lo, hi, per, r_search, torch.arange(n, device=x.device), 20000):
        if d.shape[1] < 12:
            continue
        r2 = torch.where(mask, (d * d).sum(-1), torch.full_like(d[..., 0], math.inf))
        near = torch.topk(r2, 12, dim=1, largest=False).indices
        dn = torch.gather(d, 1, near[..., None].expand(-1, -1, 3))
        s = dn[:, ia] + dn[:, ib]
        v = torch.topk((s * s).sum(-1), 6, dim=1, largest=False).values.sum(1)
        csp[c] = torch.where(mask.sum(1) >= 12, v, torch.full_like(v, math.inf))
    lam0 = 1.0 - _fcut((hyb.csp_hi - csp) / (hyb.csp_hi - hyb.csp_lo))
    lam0 = torch.where(torch.isinf(csp), torch.zeros_like(lam0), lam0)
    lam = lam0.clone()
    det = torch.nonzero(lam0 < 1.0).flatten()
    step = max(16, int(4e7 / (27 * DENSITY * hyb.r_hi ** 3 + 1)))
    if det.numel():
        for c, j, d, mask in _pair_chunks(x, lo, hi, per, hyb.r_hi, det, step):
            r = torch.sqrt((d * d).sum(-1))
            v = 1.0 - (1.0 - lam0[c])[:, None] * _fcut((r - hyb.r_lo) / (hyb.r_hi - hyb.r_lo))
            lam.scatter_reduce_(0, j[mask], v[mask], reduce="amin")
    return lam


def _psi(r, rc, h):
    u4 = ((r - rc) / h) ** 4
    return torch.where(r < rc, u4 / (1 + u4), torch.zeros_like(r))


def _eam_forms(p):
    if hasattr(p, "E1"):
        def morse(r, r0, a):
            e = torch.exp(-a * (r - r0))
            return e * e - 2 * e

        def phi(r):
            v = (p.E1 * morse(r, p.r01, p.a1) + p.E2 * morse(r, p.r02, p.a2) + p.delta) * _psi(r, p.rc, p.h)
            for s, S in ((p.rs1, p.S1), (p.rs2, p.S2), (p.rs3, p.S3)):
                v = v - torch.where(r <= s, S * (s - r) ** 4, torch.zeros_like(r))
            return v

        def zeta(r):
            return (p.a * torch.exp(-p.b1 * (r - p.r03) ** 2) + torch.exp(-p.b2 * (r - p.r04))) * _psi(r, p.rc, p.h)

        def embed(x):
            y = x - 1
            low = p.xi0 + 0.5 * p.xi2 * y ** 2 + p.q1 * y ** 3 + p.q2 * y ** 4 + p.q3 * y ** 5 + p.q4 * y ** 6
            high = (p.xi0 + 0.5 * p.xi2 * y ** 2 + p.q1 * y ** 3 + p.Q1 * y ** 4) / (1 + p.Q2 * y ** 3)
            return p.F0 + torch.where(x <= 1, low, high)
        return phi, zeta, embed

    def phi(r):
        e = torch.exp(-p.alpha * (r - p.rp))
        return p.D * (e * e - 2 * e) * _psi(r, p.rc, p.h)

    def zeta(r):
        return torch.exp(-p.beta * (r / p.r0 - 1)) * _psi(r, p.rc, p.h)

    def embed(x):
        return -p.A * torch.sqrt(torch.clamp(x, min=1e-300))
    return phi, zeta, embed


def _exact_eam(x, lo, hi, per, p, lam):
    n, dev = x.shape[0], x.device
    phi, zeta, embed = _eam_forms(p)
    every = torch.arange(n, device=dev)
    rho, pair = torch.zeros(n, dtype=torch.float64, device=dev), torch.zeros(n, dtype=torch.float64, device=dev)
    for c, j, d, mask in _pair_chunks(x, lo, hi, per, p.rc, every, 20000):
        r = torch.where(mask, torch.sqrt((d * d).sum(-1)), torch.full_like(d[..., 0], 2.0 * p.rc))
        rho[c] = (zeta(r) * mask).sum(1)
        pair[c] = 0.5 * (phi(r) * mask).sum(1)
    with torch.enable_grad():
        rg = rho.clone().requires_grad_()
        xi = embed(rg)
        (dxi,) = torch.autograd.grad(xi.sum(), rg)
    dxi = torch.where(rho > 0, dxi, torch.zeros_like(dxi))
    f = torch.zeros_like(x)
    for c, j, d, mask in _pair_chunks(x, lo, hi, per, p.rc, every, 20000):
        r = torch.where(mask, torch.sqrt((d * d).sum(-1)), torch.full_like(d[..., 0], 2.0 * p.rc))
        with torch.enable_grad():
            rg = r.clone().requires_grad_()
            (dz,) = torch.autograd.grad(zeta(rg).sum(), rg)
            rg = r.clone().requires_grad_()
            (dp,) = torch.autograd.grad(phi(rg).sum(), rg)
        q = lam * dxi
        g = (q[c][:, None] + q[j]) * dz + 0.5 * (lam[c][:, None] + lam[j]) * dp
        f[c] = ((g * mask / r)[..., None] * d).sum(1)
    return xi.detach() + pair, f


def _real_sh(u):
    """Real orthonormal spherical harmonics, l <= 4, of unit vectors [..., 3] -> [..., 25] (index l^2 + l + m)."""
    x, y, z = u.unbind(-1)
    A, B = [torch.ones_like(x)], [torch.zeros_like(x)]
    for _ in range(4):      # (x + i y)^m
        A, B = A + [A[-1] * x - B[-1] * y], B + [A[-1] * y + B[-1] * x]
    out = [None] * 25
    for m in range(5):
        P = {m: torch.full_like(z, float(np.prod(np.arange(2 * m - 1, 0, -2)) if m else 1.0))}
        if m < 4:
            P[m + 1] = (2 * m + 1) * z * P[m]
        for l in range(m + 2, 5):
            P[l] = ((2 * l - 1) * z * P[l - 1] - (l + m - 1) * P[l - 2]) / (l - m)
        for l in range(m, 5):
            N = math.sqrt((2 * l + 1) / (4 * math.pi) * math.factorial(l - m) / math.factorial(l + m)) * (math.sqrt(2.0) if m else 1.0)
            out[l * l + l + m] = N * P[l] * A[m]
            if m:
                out[l * l + l - m] = N * P[l] * B[m]
    return torch.stack(out, -1)


def _ace_terms(c):
    """Coefficients c [325+] as: c1 [8], symmetric m2 [5, 8, 8], and the nu = 3 terms (three indices n * 25 + lm, value)."""
    c = np.asarray(c, np.float64)
    m2, v = np.zeros((5, 8, 8)), 8
    for n1 in range(8):
        for n2 in range(n1, 8):
            for l in range(5):
                m2[l, n1, n2] += 0.5 * c[v]
                m2[l, n2, n1] += 0.5 * c[v]
                v += 1
    t, w = np.polynomial.legendre.leggauss(12)
    ph = 2 * np.pi * np.arange(24) / 24
    T, Ph = np.meshgrid(t, ph, indexing="ij")
    s = np.sqrt(1 - T * T)
    Y = _real_sh(torch.as_tensor(np.stack([s * np.cos(Ph), s * np.sin(Ph), T], -1).reshape(-1, 3))).numpy()
    wt = (w[:, None] * np.full(24, 2 * np.pi / 24)).reshape(-1)
    G = np.einsum("q,qa,qb,qc->abc", wt, Y[:, :16], Y[:, :16], Y[:, :16])
    idx, val = [], []
    for p1 in range(12):
        for p2 in range(p1, 12):
            for p3 in range(p2, 12):
                (n1, l1), (n2, l2), (n3, l3) = divmod(p1, 4), divmod(p2, 4), divmod(p3, 4)
                if l3 > l1 + l2 or l3 < abs(l1 - l2) or (l1 + l2 + l3) % 2:
                    continue
                for a in range(l1 * l1, (l1 + 1) ** 2):
                    for b in range(l2 * l2, (l2 + 1) ** 2):
                        for e in range(l3 * l3, (l3 + 1) ** 2):
                            if abs(G[a, b, e]) > 1e-12:
                                idx.append((n1 * 25 + a, n2 * 25 + b, n3 * 25 + e))
                                val.append(c[v] * G[a, b, e])
                v += 1
    dev = "cuda"
    return (torch.as_tensor(c[:8], device=dev), torch.as_tensor(m2, device=dev), torch.as_tensor(np.array(idx), device=dev).T,
            torch.as_tensor(np.array(val), device=dev))


def _exact_ace(x, lo, hi, per, p, w, queue):
    """E_i of the queue's atoms (0 elsewhere) and -grad sum_i w_i E_i."""
    n, dev = x.shape[0], x.device
    e_out, f = torch.zeros(n, dtype=torch.float64, device=dev), torch.zeros_like(x)
    W = torch.as_tensor(np.ascontiguousarray(p.W, np.float64).reshape(5, 8, 8), device=dev)
    sets = [_ace_terms(p.c)] + ([_ace_terms(p.c2)] if p.c2 is not None else [])
    l_of = torch.tensor([0] + [1] * 3 + [2] * 5 + [3] * 7 + [4] * 9, device=dev)
    for c, j, d, mask in _pair_chunks(x, lo, hi, per, p.rc, queue, 3000):
        with torch.enable_grad():
            dg = torch.where(mask[..., None], d, torch.ones_like(d)).requires_grad_()
            r = torch.sqrt((dg * dg).sum(-1))
            t = r / p.rc
            cut = (1.0 - 1.875 * t + 1.25 * t ** 3 - 0.375 * t ** 5) * mask
            T = [torch.ones_like(t), 2 * t - 1]
            for _ in range(6):
                T.append(2 * (2 * t - 1) * T[-1] - T[-2])
            g = torch.stack(T, 1) * cut[:, None, :]                      # [c, 8, K]
            G = g @ _real_sh(dg / r[..., None])                          # [c, 8, 25]
            A = torch.einsum("lnk,ckl->cnl", W[l_of], G) / p.n0
            Af = A.reshape(A.shape[0], 200)
            phis = []
            for c1, m2, idx, val in sets:
                e = (A[:, :, 0] * c1).sum(1) + (A * torch.einsum("lnm,cml->cnl", m2[l_of], A)).sum((1, 2))
                phis.append(e + (Af[:, idx[0]] * Af[:, idx[1]] * Af[:, idx[2]]) @ val)
            e = phis[0]
            if len(phis) > 1:
                q = phis[1]
                e = e + torch.sign(q) * (torch.sqrt(q.abs() + p.fs_eps ** 2) - p.fs_eps)
            (gr,) = torch.autograd.grad((w[c] * e).sum(), dg)
        gr = gr * mask[..., None]
        e_out[c] = e.detach()
        f.index_add_(0, c, gr.sum(1))
        f.index_add_(0, j.reshape(-1), -gr.reshape(-1, 3))
    return e_out, f


def _exact_forces(x, lo, hi, per, eam, ace, lam):
    e_f, f = _exact_eam(x, lo, hi, per, eam, lam)
    queue = torch.nonzero(lam < 1.0).flatten()
    if queue.numel():
        e_p, fp = _exact_ace(x, lo, hi, per, ace, 1.0 - lam, queue)
    else:
        e_p, fp = torch.zeros_like(e_f), torch.zeros_like(f)
    return lam * e_f + (1.0 - lam) * e_p, f + fp


@torch.no_grad()
def exact(case, seed):
    kind = case["kind"]
    if kind in ("md", "scores", "train"):
        return None        # a trajectory, and a network with bf16 operands by definition
    if kind == "gradient":
        x, off, lengths, lam = _batch(case, seed)
        total, grad = 0.0, torch.empty_like(x)
        for a, b, L in zip(off[:-1], off[1:], lengths):
            e, f = _exact_forces(x[a:b], (0.0, 0.0, 0.0), L, (True, True, True), I.eam_params(0), I.ace_params(0), lam[a:b])
            total = total + e.sum()
            grad[a:b] = -f
        return {"energy": total, "grad": grad}
    x, lo, hi, per = _structure(case, seed)
    hyb, eam = _zone(case), _eam(case)
    if kind == "lambda" or case["lam"] == "classify":
        lam = _exact_lambda(x, lo, hi, per, hyb, eam.rc + 1.0)
        if kind == "lambda":
            return {"lam": lam, "count": None}
    elif case["lam"] == "mix":
        lam = _mix(x.shape[0], seed)
    else:
        lam = torch.full((x.shape[0],), 0.0 if case["lam"] == "zero" else 1.0, dtype=torch.float64, device="cuda")
    e, f = _exact_forces(x, lo, hi, per, eam, _ace(case), lam)
    out = {"f": f, "e_atom": e, "e_tot": e.sum().reshape(1), "count": None}
    if case["lam"] == "classify":
        out["lam"] = lam
    return out
