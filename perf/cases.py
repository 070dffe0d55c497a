"""The workloads whose speed counts, as a program that uses this library runs them.

A case is a plain dict; ``prepare`` makes what the program has in hand before the call
(fields, dt, the pre-scaled coefficient it keeps, a batch), ``run`` is one pass through the
public entry points, ``exact`` the same pass in plain FP64 torch.  Kinds of pass:

* ``solve``: a whole FP64 problem with its field on the device: dt from maximum(Ci), the
  pre-scaled coefficient, nt steps replayed from the library's graph cache;
* ``run``: the time loop alone with a given dt (FP32 plain, in fused pairs or compensated;
  FP64 on the pre-scaled coefficient, or on Ci as given where the spacings differ);
* ``run2d``: the 2-D time loop;
* ``grad``: loss and gradient of the inverse problem (``loss_and_grad``);
* ``autograd``: the time loop inside a torch program (``Diffusion3DFn`` and its backward);
* ``batch``: many problems of different sizes stepped together.

Loops start every pass from T0 (one device copy), so that a pass does not depend on how
many came before it.
"""
from __future__ import annotations

import math

import torch

from paper_2211_15634_gb300 import api
from paper_2211_15634_gb300 import autograd as ag
from paper_2211_15634_gb300 import inputs

DEVICE = "cuda"
BASE = 1.7  # constant part of the initial temperature; FP32 fields store T - BASE


def listed():
    return [
        # the library's benchmark configuration: 512^3 FP64, 100 steps, whole problem on the device
        dict(name="solve_fp64_512", kind="solve", nx=512, ny=512, nz=512, nt=100),
        # the smallest problem in earnest use (a test or tuning run, one of many): latency counts
        dict(name="solve_fp64_64", kind="solve", nx=64, ny=64, nz=64, nt=100),
        # FP32 production loop in the fused-pair form
        dict(name="run_fp32_pairs_512", kind="run", dtype="f32", option="pairs", field="gauss",
             spacing="equal", nx=512, ny=512, nz=512, nt=50),
        # FP32 loop as called by default on a grid with 2^k - 1 nodes per axis
        dict(name="run_fp32_odd_255", kind="run", dtype="f32", option="plain", field="gauss",
             spacing="equal", nx=255, ny=255, nz=255, nt=50),
        # FP64 loop on a grid with 2^k + 1 nodes per axis (2^k cells)
        dict(name="run_fp64_odd_257", kind="run", dtype="f64", option="scaled", field="gauss",
             spacing="equal", nx=257, ny=257, nz=257, nt=30),
        # FP64 loop on a box with another number of nodes per axis: unequal spacings, Ci as given
        dict(name="run_fp64_unequal_512x384x256", kind="run", dtype="f64", option="plain", field="gauss",
             spacing="unequal", nx=512, ny=384, nz=256, nt=20),
        # FP64 loop on a temperature that changes sign (a deviation from a reference)
        dict(name="run_fp64_signed_320", kind="run", dtype="f64", option="scaled", field="sine",
             spacing="equal", nx=320, ny=320, nz=320, nt=30),
        # 2-D FP64 loop on a rectangle gridded with unequal spacings
        dict(name="run2d_fp64_unequal_8192x6000", kind="run2d", dtype="f64", option="plain",
             spacing="unequal", nx=8192, ny=6000, nt=20),
        # the inverse problem: loss and gradient at 256^3 FP64, every state kept
        dict(name="grad_fp64_256", kind="grad", dtype="f64", spacing="equal", nx=256, ny=256, nz=256,
             nt=40, every=1),
        # the inverse problem in FP32 with checkpoints every sqrt(nt) steps
        dict(name="grad_fp32_ckpt_192", kind="grad", dtype="f32", spacing="equal", nx=192, ny=192, nz=192,
             nt=64, every=8),
        # forward and backward inside a torch program, FP64, odd rows and unequal spacings
        dict(name="autograd_fp64_161x128x96", kind="autograd", dtype="f64", spacing="unequal",
             nx=161, ny=128, nz=96, nt=24),
        # an ensemble of problems of different sizes, FP64
        dict(name="batch_fp64_128", kind="batch", dtype="f64", nprob=128, lo=32, hi=160, nt=10),
    ]


def _size(rng, lo, hi):
    """A size spread over the logarithm of [lo, hi]: a multiple of 16, even or odd alike."""
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    how = rng.randrange(3)
    if how == 0:
        n = 16 * max(1, round(n / 16))
    elif how == 1:
        n |= 1
    return max(lo, min(hi, n))


def draw(rng):
    kind = rng.choice(["solve", "run", "run", "run", "run2d", "grad", "autograd", "batch"])
    if kind == "batch":
        lo = rng.randint(32, 64)
        return dict(kind=kind, dtype=rng.choice(["f64", "f32"]), nprob=rng.randint(16, 128), lo=lo,
                    hi=rng.randint(lo + 16, 160), nt=rng.randint(5, 20))
    if kind == "run2d":
        c = dict(kind=kind, dtype=rng.choice(["f64", "f64", "f32"]), spacing=rng.choice(["equal", "unequal"]),
                 nx=_size(rng, 256, 8192), ny=_size(rng, 256, 8192), nt=rng.randint(10, 40))
        c["option"] = "scaled" if c["dtype"] == "f64" and c["spacing"] == "equal" else "plain"
        return c
    if kind in ("grad", "autograd"):
        nt = rng.randint(16, 64)
        c = dict(kind=kind, dtype=rng.choice(["f64", "f32"]), spacing=rng.choice(["equal", "unequal"]),
                 nx=_size(rng, 48, 256), ny=_size(rng, 48, 256), nz=_size(rng, 48, 256), nt=nt)
        if kind == "grad":
            c["every"] = rng.choice([1, int(math.ceil(math.sqrt(nt)))])
        return c
    c = dict(kind=kind, nx=_size(rng, 48, 512), ny=_size(rng, 48, 512), nz=_size(rng, 48, 512),
             nt=rng.randint(20, 100))
    if kind == "run":
        c.update(dtype=rng.choice(["f64", "f32"]), field=rng.choice(["gauss", "gauss", "sine"]),
                 spacing=rng.choice(["equal", "equal", "unequal"]))
        if c["dtype"] == "f32":
            c["option"] = rng.choice(["plain", "pairs", "comp"])
        else:
            c["option"] = "scaled" if c["spacing"] == "equal" else "plain"
    return c


# ---------------------------------------------------------------- inputs
def _dtype(case):
    return torch.float32 if case.get("dtype", "f64") == "f32" else torch.float64


def _grid(case):
    """(nz, ny, nx), inverse spacings and lengths: the unit cube with its own spacing per
    axis, or one spacing on all axes (the box's lengths follow)."""
    shape = tuple(case[k] for k in ("nz", "ny", "nx") if k in case)
    n = tuple(reversed(shape))
    if case.get("spacing", "equal") == "unequal":
        return shape, tuple(float(m - 1) for m in n), (1.0,) * len(n)
    inv = float(max(n) - 1)
    return shape, (inv,) * len(n), tuple((m - 1) / inv for m in n)


def _generator(seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed)
    return g


def _axes(shape, lengths):
    """Node coordinates per axis of ``shape``, each ready to broadcast."""
    out = []
    for d, (n, length) in enumerate(zip(shape, reversed(lengths))):
        x = torch.arange(n, dtype=torch.float64, device=DEVICE) * (length / (n - 1))
        out.append(x.view([-1 if e == d else 1 for e in range(len(shape))]))
    return out


def _field(case, shape, lengths, g):
    """Initial temperature (FP64): a warm Gaussian spot on the constant base, or a product
    of half sine waves about zero; where the spot sits and how warm it is come from the seed."""
    u = torch.rand(5, generator=g, device=DEVICE, dtype=torch.float64)
    axes = _axes(shape, lengths)
    if case.get("field", "gauss") == "sine":
        s = 1.0 + 0.2 * u[4]
        for x, length in zip(axes, reversed(lengths)):
            s = s * torch.sin(math.pi * x / length)
        return s - 0.5
    r2 = 0.0
    for d, (x, length) in enumerate(zip(axes, reversed(lengths))):
        r2 = r2 + (x - length * (0.4 + 0.2 * u[d])) ** 2
    return BASE + (0.8 + 0.4 * u[4]) * torch.exp(-r2 / 0.01)


def _coefficient(shape, g):
    """Ci = (1/c0) (1 + 0.5 U), c0 = 2: the variable coefficient of the forward workloads."""
    return torch.rand(shape, generator=g, device=DEVICE, dtype=torch.float64).mul_(0.5).add_(1.0).mul_(0.5)


def _as_stored(T, dtype):
    """FP32 fields hold the deviation from BASE (rounded once)."""
    return T if dtype == torch.float64 else (T - BASE).float()


def _dt(inv):
    """The step of ``api.stable_dt`` for the bound Ci <= 0.75 of these coefficients."""
    d = min(1.0 / v for v in inv)
    return d * d / 0.75 / (6.1 if len(inv) == 3 else 4.1)


def _batch_layout(case):
    """Sizes of the problems, their row pitches (16-byte rows) and offsets in one block."""
    per = 16 // torch.empty((), dtype=_dtype(case)).element_size()
    sizes = [int(n) for n in inputs.batch_sizes(case["nprob"], case["lo"], case["hi"])]
    pitches = [-(-n // per) * per for n in sizes]
    offsets, total = [], 0
    for n, pitch in zip(sizes, pitches):
        offsets.append(total)
        total += -(-n * n * pitch // 32) * 32
    return sizes, pitches, offsets, total


def _batch_views(flat, layout):
    sizes, pitches, offsets, _ = layout
    return [flat[o:o + n * n * p].view(n, n, p)[:, :, :n] for n, p, o in zip(sizes, pitches, offsets)]


def _batch_fields(case, seed):
    """T0 and Ci of every problem in one block each, and the layout."""
    layout, dtype, g = _batch_layout(case), _dtype(case), _generator(seed)
    T0 = torch.zeros(layout[3], dtype=dtype, device=DEVICE)
    Ci = torch.full((layout[3],), 0.5, dtype=dtype, device=DEVICE)
    for t, c in zip(_batch_views(T0, layout), _batch_views(Ci, layout)):
        shape = tuple(t.shape)
        t.copy_(_as_stored(_field(case, shape, (1.0,) * 3, g), dtype))
        c.copy_(_coefficient(shape, g))
    return T0, Ci, layout


def _fields(case, seed):
    """(T0, Ci, shape, inv, lengths, third field) as stored, from the seed alone: the third
    field is the observed state of ``grad`` or the cotangent of ``autograd``."""
    shape, inv, lengths = _grid(case)
    dtype, g = _dtype(case), _generator(seed)
    T0 = _as_stored(_field(case, shape, lengths, g), dtype)
    Ci = _coefficient(shape, g).to(dtype)
    third = None
    if case["kind"] == "grad":
        third = _as_stored(_field(case, shape, lengths, g), dtype)
    elif case["kind"] == "autograd":
        third = (torch.rand(shape, generator=g, device=DEVICE, dtype=torch.float64) - 0.5).to(dtype)
    return T0, Ci, shape, inv, lengths, third


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        T0, Ci, layout = _batch_fields(case, seed)
        T, T2 = T0.clone(), T0.clone()
        views = zip(*(_batch_views(f, layout) for f in (T, T2, Ci)), layout[0])
        probs = [dict(T=t, T2=t2, Ci=c, lam=1.0, dt=_dt((n - 1.0,) * 3), inv_spacing=(n - 1.0,) * 3)
                 for t, t2, c, n in views]
        return dict(case=case, T0=T0, T=T, T2=T2, batch=api.Batch(probs))
    T0, Ci, shape, inv, lengths, third = _fields(case, seed)
    state = dict(case=case, T0=T0, Ci=Ci, inv=inv, lengths=lengths, dt=_dt(inv))
    if kind in ("solve", "run", "run2d"):
        state.update(T=torch.empty_like(T0), T2=torch.empty_like(T0))
        if kind == "solve":
            state["Cs"] = torch.empty_like(Ci)
        elif case["option"] == "scaled":
            state["Ci"] = api.scale_ci(Ci, 1.0, state["dt"], inv)
        elif case["option"] == "comp":
            state["comp"] = api.compensation_fields(T0)
    elif kind == "grad":
        state["Tobs"] = third
    else:
        state.update(T0=T0.requires_grad_(), Ci=Ci.requires_grad_(), cotangent=third)
    return state


def run(state):
    case = state["case"]
    kind, nt = case["kind"], case["nt"]
    if kind == "batch":
        state["T"].copy_(state["T0"])
        state["batch"].run(nt)
        return state["T2"] if nt & 1 else state["T"]
    T0, Ci, inv, dt = state["T0"], state["Ci"], state["inv"], state["dt"]
    if kind == "grad":
        return list(ag.loss_and_grad(T0, Ci, state["Tobs"], 1.0, dt, inv, nt, every=case["every"]))
    if kind == "autograd":
        out = ag.Diffusion3DFn.apply(T0, Ci, 1.0, dt, inv, nt)
        return [out] + list(torch.autograd.grad(out, (T0, Ci), state["cotangent"]))
    T, T2 = state["T"], state["T2"]
    T.copy_(T0)
    if kind == "solve":
        dt = api.stable_dt(Ci, 1.0, state["lengths"])
        Cs = api.scale_ci(Ci, 1.0, dt, inv, out=state["Cs"])
        return [dt, api.run(T, T2, Cs, 1.0, dt, inv, nt, graph=True, ci_scaled=True)]
    if kind == "run2d":
        return api.run2d(T, T2, Ci, 1.0, dt, inv, nt, graph=True, ci_scaled=case["option"] == "scaled")
    if case["option"] == "comp":
        comp = state["comp"]
        comp.zero_()
        return [api.run(T, T2, Ci, 1.0, dt, inv, nt, comp=comp, graph=True), comp[nt % 2]]
    return api.run(T, T2, Ci, 1.0, dt, inv, nt, graph=True, ci_scaled=case["option"] == "scaled",
                   temporal2=case["option"] == "pairs")


def work(case):
    """Bytes: per step T and Ci read and the new state written once (the library's T_eff
    convention, whole arrays), twice that per transposed step; the compensated state is a
    pair.  Operations: Fig. 1's step as printed has 19 per node, its transpose about 30."""
    kind, nt = case["kind"], case["nt"]
    size = 4 if case.get("dtype", "f64") == "f32" else 8
    if kind == "batch":
        nodes = sum(n ** 3 for n in _batch_layout(case)[0])
    else:
        nodes = case["nx"] * case["ny"] * case.get("nz", 1)
    arrays, flops = 3.0 * nt, 19.0 * nt
    if kind == "run2d":
        flops = 14.0 * nt
    if case.get("option") == "comp":
        arrays, flops = 5.0 * nt, 36.0 * nt
    if kind in ("grad", "autograd"):
        arrays, flops = 9.0 * nt, 49.0 * nt
    if kind == "solve":
        arrays += 3.0  # maximum(Ci), the scaled copy
    return {"bytes": arrays * nodes * size, "flops": flops * nodes}


# ---------------------------------------------------------------- plain FP64
def _laplacian(T, a, out=None):
    """Fig. 1's weighted second differences on the interior nodes of a 2-D or 3-D field."""
    inner = (slice(1, -1),) * T.dim()
    out = torch.zeros_like(T) if out is None else out
    acc = out[inner]
    acc.zero_()
    for d in range(T.dim()):
        lo, hi = list(inner), list(inner)
        lo[d], hi[d] = slice(0, -2), slice(2, None)
        acc.add_((T[tuple(hi)] - T[inner]) - (T[inner] - T[tuple(lo)]), alpha=a[T.dim() - 1 - d])
    return out


def _forward(T0, C, a, nt, keep=False):
    """T(nt) with C = dt*lam*Ci; every state T(0) .. T(nt-1) too where asked."""
    T, states, work = T0.clone(), [], torch.zeros_like(T0)
    for _ in range(nt):
        if keep:
            states.append(T.clone())
        T.add_(_laplacian(T, a, work).mul_(C))
    return T, states


def _reverse(ybar, states, C, a, scale):
    """(dL/dT0, dL/dCi) of nt steps: the transposed steps in reverse order."""
    y, cbar, work = ybar.clone(), torch.zeros_like(ybar), torch.zeros_like(ybar)
    inner = (slice(1, -1),) * y.dim()
    for T in reversed(states):
        cbar.add_(_laplacian(T, a, work).mul_(y), alpha=scale)
        w = C * y
        wi = torch.zeros_like(w)
        wi[inner] = w[inner]  # the step writes interior nodes only
        wp = torch.nn.functional.pad(wi, (1, 1) * y.dim())
        y = y + _laplacian(wp, a)[inner]
    return y, cbar


def exact(case, seed):
    kind, nt = case["kind"], case["nt"]
    if kind == "batch":
        T0, Ci, layout = _batch_fields(case, seed)
        out = T0.double()
        for t, c, n in zip(_batch_views(out, layout), _batch_views(Ci, layout), layout[0]):
            inv = (n - 1.0,) * 3
            t.copy_(_forward(t.clone(), c.double() * _dt(inv), [v * v for v in inv], nt)[0])
        return out
    T0, Ci, shape, inv, lengths, third = _fields(case, seed)
    T0, Ci, a = T0.double(), Ci.double(), [v * v for v in inv]
    dt = _dt(inv)
    if kind == "solve":
        d = min(length / (n - 1) for length, n in zip(lengths, reversed(shape)))
        dt = d * d / float(Ci.max()) / 6.1
        return [dt, _forward(T0, Ci * dt, a, nt)[0]]
    C = Ci * dt
    T, states = _forward(T0, C, a, nt, keep=kind in ("grad", "autograd"))
    if kind == "grad":
        resid = T - third.double()
        return [0.5 * (resid * resid).sum()] + list(_reverse(resid, states, C, a, dt))
    if kind == "autograd":
        return [T] + list(_reverse(third.double(), states, C, a, dt))
    if case["option"] == "comp":
        return [T, None]  # the correction field alone has no value of its own
    return T
