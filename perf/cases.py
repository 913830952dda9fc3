"""What a user of the library has it do, as measurable cases.

A case is one pass of a user's program through the public entry points:

* ``sweep``: an initial field that is on the device goes in, T steps run, u_T comes out
  (``Stencil.set_field`` / ``run`` / ``get_field``), with the schedule that
  ``set_tuning("auto")`` selects, or (``tuned`` false) with what a grid has when the
  program never calls ``set_tuning``. The grid and its coefficients are kept.
* ``adjoint``: one training step's gradients through ``autograd.sweep``: the loss
  0.5 ||u_T - target||^2, differentiated with respect to u_0 and every coefficient array.
* ``batch``: many uneven grids get new fields, advance in one persistent launch
  (``batch.Batch``) and are read back. The plan is kept. T is even for every grid, so
  each launch starts from the array that ``set_field`` writes.

Sizes, step counts and distributions are those of the library's benchmark and tests:
cubes of 64 (FP64, T = 8), 512 and 1024 (constant coefficients, T = 100), 384 (variable,
T = 50) and 256 (25 points, T = 40), 64 uneven grids with sides 32..192 and T 10..200,
and small and odd shapes as a program with its own domain has them.
"""
import math

import torch

from paper_1410_5561_gb300.autograd import sweep
from paper_1410_5561_gb300.batch import Batch
from paper_1410_5561_gb300.stencil import Stencil, Tuning

RADIUS = {"7pt_const": 1, "7pt_var": 1, "25pt_var": 4}
NCOEF = {"7pt_const": 0, "7pt_var": 7, "25pt_var": 13}
FLOPS = {"7pt_const": 10, "7pt_var": 13, "25pt_var": 37}  # per update, as the listings write them
DTYPE = {"f32": torch.float32, "f64": torch.float64, "bf16": torch.bfloat16}
BYTES = {"f32": 4, "f64": 8, "bf16": 2}
C0, C1 = 0.4, 0.1
ROW_SUM = 0.95


def _sweep(name, kind, nx, ny, nz, T, field="f32", coef=None, tuned=True):
    return {"name": name, "do": "sweep", "kind": kind, "nx": nx, "ny": ny, "nz": nz, "T": T, "field": field,
            "coef": coef or field, "tuned": tuned}


def _adjoint(name, kind, nx, ny, nz, T, field="f32", coef=None):
    return {**_sweep(name, kind, nx, ny, nz, T, field, coef), "do": "adjoint"}


def _batch(name, kind, grids, lo, hi, field="f32", coef=None):
    return {"name": name, "do": "batch", "kind": kind, "grids": grids, "lo": lo, "hi": hi, "field": field,
            "coef": coef or field}


def listed():
    return [
        # the smallest call: a few FP64 steps of a small cube, the check that a user starts with
        _sweep("const_f64_64_T8", "7pt_const", 64, 64, 64, 8, "f64"),
        # a small odd domain inside a larger program: launches and latency
        _sweep("const_f32_small_odd", "7pt_const", 101, 75, 62, 50),
        # an ordinary odd domain, larger than one SM's share, smaller than L2
        _sweep("const_f32_mid_odd", "7pt_const", 301, 257, 199, 60),
        # the benchmark's headline workload, the largest
        _sweep("const_f32_1024", "7pt_const", 1024, 1024, 1024, 100),
        # the benchmark's double-precision workload
        _sweep("const_f64_512", "7pt_const", 512, 512, 512, 100, "f64"),
        # the benchmark's variable-coefficient workload, single precision
        _sweep("var7_f32_384", "7pt_var", 384, 384, 384, 50),
        # coefficients stored in 16 bits, an odd domain
        _sweep("var7_bf16_odd", "7pt_var", 250, 333, 195, 50, "f32", "bf16"),
        # the benchmark's high-order workload
        _sweep("var25_f32_256", "25pt_var", 256, 256, 256, 40),
        # high order, 16-bit coefficients, a few steps between other work, a grid used as it comes
        _sweep("var25_bf16_odd_T10", "25pt_var", 203, 250, 141, 10, "f32", "bf16", tuned=False),
        # the benchmark's training step: gradients for the field and all 13 coefficient arrays
        _adjoint("adjoint25_f32_256", "25pt_var", 256, 256, 256, 40),
        # a training step on a small odd domain
        _adjoint("adjoint7_f32_small", "7pt_var", 96, 70, 83, 24),
        # the benchmark's batch of uneven grids
        _batch("batch64_var7_f32", "7pt_var", 64, 32, 192),
    ]


# ns per update at the rates these sweeps run at; drawn work stays below the largest listed case
_NS = {("7pt_const", "f32", "f32"): 0.0015, ("7pt_const", "f64", "f64"): 0.014, ("7pt_var", "f32", "f32"): 0.006,
       ("7pt_var", "f32", "bf16"): 0.005, ("7pt_var", "f64", "f64"): 0.014, ("25pt_var", "f32", "f32"): 0.011,
       ("25pt_var", "f32", "bf16"): 0.008, ("25pt_var", "f64", "f64"): 0.05}


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _unnamed(case):
    return {k: v for k, v in case.items() if k != "name"}


def draw(rng):
    what = rng.choice(["sweep", "sweep", "sweep", "sweep", "adjoint", "batch"])
    kind, field, coef = rng.choice(sorted(_NS))
    if what == "batch":
        while kind == "25pt_var":  # the batch serves the 7-point stencils in earnest
            kind, field, coef = rng.choice(sorted(_NS))
        lo = _log(rng, 16, 64)
        hi = rng.randint(lo + 16, 192 if field == "f32" else 128)
        return _unnamed(_batch("", kind, _log(rng, 4, 64), lo, hi, field, coef))
    if what == "adjoint":
        while kind == "7pt_const" or field == "f64":  # gradients are for coefficient arrays
            kind, field, coef = rng.choice(sorted(_NS))
    top = 20.0 if what == "adjoint" else 80.0  # ms of forward work
    while True:
        nx, ny, nz = (_log(rng, 24, 256 if what == "adjoint" else 640) for _ in range(3))
        T = _log(rng, 2 if what == "adjoint" else 1, 100)
        if nx * ny * nz * T * _NS[kind, field, coef] * 1e-6 <= top and nx * ny * nz * (13 if kind == "25pt_var" else 7) <= 6e8:
            break
    c = (_adjoint if what == "adjoint" else _sweep)("", kind, nx, ny, nz, T, field, coef)
    if what == "sweep":
        c["tuned"] = rng.random() < 0.8
    return _unnamed(c)


# ------------------------------------------------------------------ inputs
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _field(g, shape, dtype):
    """Uniform on [-1, 1)."""
    return torch.rand(shape, generator=g, device="cuda", dtype=dtype).mul_(2).sub_(1)


def _coefs(g, kind, shape, dtype):
    """Positive weights whose sum over a point's neighbours is ROW_SUM: a list of arrays, [] for constant ones."""
    if kind == "7pt_const":
        return []
    work = torch.float64 if dtype == torch.float64 else torch.float32
    r = [torch.rand(shape, generator=g, device="cuda", dtype=work) for _ in range(NCOEF[kind])]
    s = r[1].clone()
    for x in r[2:]:
        s += x
    s = (2 * s if kind == "25pt_var" else s) + r[0]
    return [(ROW_SUM * x / s).to(dtype) for x in r]


def _problem(case, seed):
    """(u_0, coefficients, target) of a single grid, from the seed alone."""
    g = _generator(seed)
    shape = (case["nz"], case["ny"], case["nx"])
    u0 = _field(g, shape, DTYPE[case["field"]])
    c = _coefs(g, case["kind"], shape, DTYPE[case["coef"]])
    target = _field(g, shape, DTYPE[case["field"]]) if case["do"] == "adjoint" else None
    return u0, c, target


def _batch_shapes(case):
    """(nx, ny, nz, T) of every grid: a property of the case, the same for every seed."""
    g = torch.Generator().manual_seed(1000 * case["lo"] + case["hi"])
    out = []
    for _ in range(case["grids"]):
        n = torch.randint(case["lo"], case["hi"] + 1, (3,), generator=g).tolist()
        out.append((*n, 2 * int(torch.randint(5, 101, (1,), generator=g))))
    return out


def _grid(case, nx, ny, nz, coefs):
    s = Stencil(case["kind"], nx, ny, nz, dtype=DTYPE[case["field"]], coef_dtype=DTYPE[case["coef"]])
    if coefs:
        s.set_coeffs(arrays=coefs)
    else:
        s.set_coeffs(scalars=(C0, C1))
    return s


def prepare(case, seed):
    if case["do"] == "batch":
        grids, u0, T = [], [], []
        for q, (nx, ny, nz, t) in enumerate(_batch_shapes(case)):
            g = _generator(1000003 * seed + q)
            u0.append(_field(g, (nz, ny, nx), DTYPE[case["field"]]))
            s = _grid(case, nx, ny, nz, _coefs(g, case["kind"], (nz, ny, nx), DTYPE[case["coef"]]))
            s.set_field(u0[-1])
            grids.append(s)
            T.append(t)
        # the first candidate of the batch tuner, within 3 % of the fastest one for grids of these sizes
        return {"do": "batch", "grids": grids, "u0": u0, "batch": Batch(grids, T, Tuning(4, 1, 8, 0))}
    u0, c, target = _problem(case, seed)
    s = _grid(case, case["nx"], case["ny"], case["nz"], c)
    if case["tuned"]:
        s.set_tuning("auto")
    state = {"do": case["do"], "grid": s, "u0": u0, "T": case["T"]}
    if case["do"] == "adjoint":
        state.update(u0=u0.requires_grad_(), coefs=torch.stack(c).requires_grad_(), target=target)
    return state


def run(state):
    if state["do"] == "sweep":
        s = state["grid"]
        s.set_field(state["u0"])
        s.run(state["T"])
        return s.get_field()
    if state["do"] == "adjoint":
        uT = sweep(state["u0"], state["coefs"], state["grid"], state["T"])
        loss = 0.5 * ((uT - state["target"]) ** 2).sum()
        return (uT.detach(), *torch.autograd.grad(loss, (state["u0"], state["coefs"])))
    for s, u in zip(state["grids"], state["u0"]):
        s.set_field(u)
    state["batch"].launch()
    return [s.get_field() for s in state["grids"]]


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    kind, f = case["kind"], BYTES[case["field"]]
    if case["do"] == "batch":
        sizes = [(nx * ny * nz, t) for nx, ny, nz, t in _batch_shapes(case)]
    else:
        sizes = [(case["nx"] * case["ny"] * case["nz"], case["T"])]
    n, lups = sum(p for p, _ in sizes), sum(p * t for p, t in sizes)
    coef = NCOEF[kind] * BYTES[case["coef"]]
    if case["do"] != "adjoint":  # u_0 and the coefficients in, u_T out
        return {"bytes": n * (2 * f + coef), "flops": lups * FLOPS[kind]}
    # u_0, target and coefficients in; u_T and the gradients out; per step the forward update, the
    # transposed one (a product and a sum for every point read) and one product and sum for each
    # coefficient's gradient (25 points: and the pair sums that it multiplies)
    points = 25 if kind == "25pt_var" else 7
    back = 2 * points + 2 * NCOEF[kind] + (12 if kind == "25pt_var" else 0)
    return {"bytes": n * (4 * f + 2 * coef), "flops": lups * (FLOPS[kind] + back)}


# ------------------------------------------------------------------ the same in 64 bits, with plain torch
def _neighbours(kind):
    """(coefficient array, axis, offset) of every neighbour; axes of a (z, y, x) tensor."""
    if kind == "25pt_var":
        return [(3 * (d - 1) + a + 1, 2 - a, o) for d in range(1, 5) for a in range(3) for o in (d, -d)]
    return [(1 + 2 * a + i, 2 - a, o) for a in range(3) for i, o in enumerate((1, -1))]


def _inside(p, r):
    return p[r:-r, r:-r, r:-r]


def _moved(p, r, axis, o):
    """The interior of the padded p, moved by o along an axis: the value at x + o for every x."""
    at = [slice(r, n - r) for n in p.shape]
    at[axis] = slice(r + o, p.shape[axis] - r + o)
    return p[tuple(at)]


def _step(kind, p, c, out):
    """out's interior = one step of the padded p."""
    r = RADIUS[kind]
    to = _inside(out, r)
    if not c:
        torch.mul(_inside(p, r), C0, out=to)
        for _, axis, o in _neighbours("7pt_const"):
            to.add_(_moved(p, r, axis, o), alpha=C1)
        return
    torch.mul(_inside(p, r), c[0], out=to)
    for m, axis, o in _neighbours(kind):
        to.addcmul_(_moved(p, r, axis, o), c[m])


def _padded(u, r):
    return torch.nn.functional.pad(u.double(), (r,) * 6)


def _exact_sweep(kind, u0, c, T):
    r = RADIUS[kind]
    p, q = _padded(u0, r), _padded(torch.zeros_like(u0), r)
    for _ in range(T):
        _step(kind, p, c, q)
        p, q = q, p
    return _inside(p, r).clone()


def _exact_adjoint(kind, u0, c, target, T):
    r = RADIUS[kind]
    states = [_padded(u0, r)]
    for _ in range(T):
        q = torch.zeros_like(states[-1])
        _step(kind, states[-1], c, q)
        states.append(q)
    uT = _inside(states.pop(), r).clone()
    lam = uT - target.double()
    gc = [torch.zeros_like(x) for x in c]
    pad = torch.zeros_like(states[0])
    for p in reversed(states):
        gc[0].addcmul_(lam, _inside(p, r))
        pad.zero_()
        _inside(pad, r).copy_(lam * c[0])
        for m, axis, o in _neighbours(kind):
            gc[m].addcmul_(lam, _moved(p, r, axis, o))
            _moved(pad, r, axis, o).add_(lam * c[m])
        lam = _inside(pad, r).clone()
    return uT, lam, torch.stack(gc)


def exact(case, seed):
    kind = case["kind"]
    if case["do"] == "batch":
        out = []
        for q, (nx, ny, nz, t) in enumerate(_batch_shapes(case)):
            g = _generator(1000003 * seed + q)
            u0 = _field(g, (nz, ny, nx), DTYPE[case["field"]])
            c = [x.double() for x in _coefs(g, kind, (nz, ny, nx), DTYPE[case["coef"]])]
            out.append(_exact_sweep(kind, u0, c, t))
        return out
    u0, c, target = _problem(case, seed)
    c = [x.double() for x in c]
    if case["do"] == "adjoint":
        return _exact_adjoint(kind, u0, c, target, case["T"])
    return _exact_sweep(kind, u0, c, case["T"])
