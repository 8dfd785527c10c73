"""What a user of the library has it do, as cases that can be timed and checked.

A case is one pass through the public entry points of `paper_2105_12764_gb300`:
a field is decomposed and recomposed (device buffers, pinned host buffers, the
class-packed, quantized, spatiotemporal and batched forms).  The sizes are those
of the repository's workloads and tests, and ragged ones between them.

`exact` evaluates the same operators densely in FP64 with torch: per axis and
level the interpolation matrix P and the correction matrix
Z = (P^T M P)^-1 P^T M, M the P1 mass matrix of the level's nodes.
"""
import itertools
import math

import numpy as np
import torch

import paper_2105_12764_gb300 as mgr

# form -> (field type of the library, precision, torch type)
FORMS = {
    "f64": (mgr.MGR_F64, mgr.MGR_PREC_NATIVE, torch.float64),
    "f32": (mgr.MGR_F32, mgr.MGR_PREC_NATIVE, torch.float32),
    "mixed": (mgr.MGR_F32, mgr.MGR_PREC_MIXED, torch.float32),
}
TAU = 1e-3  # tolerance of the quantized cases, fields have unit variance
ALIGN = 64  # elements between the starts of a batch's fields are a multiple of this


def listed():
    return [
        # the smallest call in use: one small plain field, launches and latency count
        dict(name="sines_65_f64", kind="field", shape="65x65x65", form="f64", coords="uniform", field="sines"),
        # a small ragged block on its own stretched coordinates, as a served request brings it
        dict(name="ragged_90x121x77_f32", kind="field", shape="90x121x77", form="f32", coords="stretched", field="grf"),
        # an ordinary served field in double precision
        dict(name="grf_257_f64", kind="field", shape="257x257x257", form="f64", coords="uniform", field="grf"),
        # the paper's kernel size 2^9+1: plain double precision, and single precision
        dict(name="grf_513_f64", kind="field", shape="513x513x513", form="f64", coords="uniform", field="grf"),
        dict(name="grf_513_f32", kind="field", shape="513x513x513", form="f32", coords="uniform", field="grf"),
        # a long ragged field on stretched coordinates: FP32 stencils, FP64 solves
        dict(name="bumps_1000x700x300_mixed", kind="field", shape="1000x700x300", form="mixed", coords="stretched",
             field="bumps"),
        # a plane (2D field) with long lines
        dict(name="plane_2049x3000_f32", kind="field", shape="2049x3000", form="f32", coords="uniform", field="grf"),
        # class-packed output and its progressive recomposition (all classes, and without the finest)
        dict(name="packed_385_f32", kind="packed", shape="385x385x385", form="f32", coords="uniform", field="grf"),
        # the lossy compressor's stages: int32 codes of a field, and the field of given codes
        dict(name="quantized_257_f32", kind="quantized", shape="257x257x257", form="f32", coords="uniform",
             field="grf"),
        # time steps of a volume as one (3+1)-D field
        dict(name="time_33x129_f64", kind="field", shape="33x129x129x129", form="f64", coords="uniform", field="grf"),
        # many small uneven 2D and 3D fields in one submit
        dict(name="batch_1024_f32", kind="batch", count=1024, specs=0, form="f32"),
        # a field in pinned host memory, copies inside the call
        dict(name="host_257_f64", kind="host", shape="257x257x257", form="f64", coords="uniform", field="grf"),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _sides(rng, nodes, dims):
    """Sides of a ragged block of about `nodes` nodes, aspect ratios up to about 3."""
    side = nodes ** (1.0 / dims)
    cut = [max(17, round(side * _log_uniform(rng, 0.6, 1.6))) for _ in range(dims - 1)]
    last = nodes
    for c in cut:
        last /= c
    return [int(c) for c in cut] + [int(min(max(17, round(last)), 3 * side))]


def draw(rng):
    kind = rng.choice(["field", "field", "field", "plane", "packed", "quantized", "time", "batch", "host"])
    form = rng.choice(["f64", "f32", "mixed"])
    coords = rng.choice(["uniform", "stretched"])
    if kind == "batch":
        return dict(kind="batch", count=int(_log_uniform(rng, 64, 1024)), specs=rng.randrange(1, 1 << 20), form=form)
    top = {"field": 500 ** 3, "plane": 2500 ** 2, "packed": 400 ** 3, "quantized": 300 ** 3, "time": 60e6,
           "host": 280 ** 3}[kind]
    dims = {"plane": 2, "time": 4}.get(kind, 3)
    low = {"plane": 300 ** 2, "time": 3e6, "host": 100 ** 3}.get(kind, 33 ** 3)
    if kind == "time":
        steps = rng.randrange(5, 34)
        sides = [steps] + _sides(rng, _log_uniform(rng, low, top) / steps, 3)
    else:
        sides = _sides(rng, _log_uniform(rng, low, top), dims)
    if math.prod(sides) > 513 ** 3:
        sides = [max(5, int(s * 0.8)) for s in sides]
    return dict(kind=kind if kind in ("packed", "quantized", "host") else "field", shape="x".join(map(str, sides)),
                form=form, coords=coords, field=rng.choice(["grf", "grf", "bumps"]))


# ---------------------------------------------------------------- inputs

def _shape(case):
    return tuple(int(s) for s in case["shape"].split("x"))


def _coords(shape, kind):
    """Unit spacing (None), or h_i = 1.01^i per axis."""
    if kind == "uniform":
        return None
    return [np.concatenate([[0.0], np.cumsum(1.01 ** np.arange(n - 1, dtype=np.float64))]) for n in shape]


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _grf(shape, seed):
    """Gaussian random field with power |k|^(-5/3), mean 0 and variance 1."""
    spec = torch.fft.rfftn(torch.randn(shape, generator=_gen(seed), device="cuda", dtype=torch.float64))
    k2 = 0
    for ax, n in enumerate(shape):
        k = (torch.fft.rfftfreq if ax == len(shape) - 1 else torch.fft.fftfreq)(n, device="cuda", dtype=torch.float64)
        k2 = k2 + (k * n).reshape([-1 if a == ax else 1 for a in range(len(shape))]) ** 2
    spec *= torch.where(k2 > 0, k2.clamp_min(1e-300) ** (-5.0 / 12.0), torch.zeros_like(k2))
    u = torch.fft.irfftn(spec, s=shape)
    u -= u.mean()
    u /= u.std()
    return u


def _outer(factors):
    out = factors[0]
    for f in factors[1:]:
        out = out.unsqueeze(-1) * f
    return out


def _sines(shape, seed):
    """Three sines of at most four cycles a side, and noise of 1e-3."""
    r = np.random.default_rng(seed)
    u = torch.randn(shape, generator=_gen(seed), device="cuda", dtype=torch.float64) * 1e-3
    grids = torch.meshgrid(*[torch.arange(n, device="cuda", dtype=torch.float64) / (n - 1) for n in shape],
                           indexing="ij")
    for _ in range(3):
        k, phi = r.uniform(-4 / math.sqrt(3), 4 / math.sqrt(3), len(shape)), r.uniform(0, 2 * math.pi)
        u += torch.sin(2 * math.pi * sum(float(ki) * g for ki, g in zip(k, grids)) + phi)
    return u


def _bumps(shape, seed):
    """A smooth product of cosines and 32 bumps of 2 to 20 cells."""
    r = np.random.default_rng(seed)
    x = [torch.arange(n, device="cuda", dtype=torch.float64) for n in shape]
    u = _outer([torch.cos(2 * math.pi * r.uniform(0.5, 2.0) * xi / (len(xi) - 1) + r.uniform(0, 2 * math.pi))
                for xi in x]).contiguous()
    for _ in range(32):
        width, amp = r.uniform(2.0, 20.0), r.standard_normal()
        u += amp * _outer([torch.exp(-0.5 * ((xi - r.uniform(0, len(xi) - 1)) / width) ** 2) for xi in x])
    return u


def _field(case, seed):
    """The case's field in FP64, rounded to its type."""
    u = {"grf": _grf, "sines": _sines, "bumps": _bumps}[case["field"]](_shape(case), seed)
    return u.to(FORMS[case["form"]][2])


def _batch_specs(case):
    """(shape, stretched) per field: element counts log-uniform on [17^2, 129^3], near-square 2D
    fields up to 129^2 and near-cube 3D ones above, sides in [17, 129], half on stretched coordinates."""
    r = np.random.default_rng(case["specs"])
    specs = []
    for _ in range(case["count"]):
        n = math.exp(r.uniform(math.log(17 ** 2), math.log(129 ** 3)))
        dims = 2 if n <= 129 ** 2 else 3
        sides = []
        for d in range(dims, 0, -1):
            side = n ** (1.0 / d) * (r.uniform(0.87, 1.15) if d > 1 else 1.0)
            sides.append(int(np.clip(round(side), 17, 129)))
            n /= sides[-1]
        specs.append((tuple(sides), bool(r.random() < 0.5)))
    return specs


def _batch_layout(specs):
    """Start of every field in one buffer, and the buffer's length."""
    starts, at = [], 0
    for shape, _ in specs:
        starts.append(at)
        at += -(-math.prod(shape) // ALIGN) * ALIGN
    return starts, at


def _batch_fields(case, seed):
    specs = _batch_specs(case)
    starts, total = _batch_layout(specs)
    flat = torch.zeros(total, dtype=FORMS[case["form"]][2], device="cuda")
    for i, ((shape, _), at) in enumerate(zip(specs, starts)):
        flat[at:at + math.prod(shape)] = _grf(shape, (seed * 100003 + i) & 0x7FFFFFFF).reshape(-1)
    return flat


# ---------------------------------------------------------------- the path

_context = None
_batch_plans = {}  # a batch's plans by its specification: a program with new fields of the same sizes keeps them


def _ctx():
    global _context
    if _context is None:
        _context = mgr.Context(0)
    return _context


def _plan(shape, coords, form):
    dtype, prec, _ = FORMS[form]
    return mgr.Plan(_ctx(), shape, coords, -1, dtype, prec)


def _workspace(plan):
    return torch.empty(max(plan.workspace_bytes, 256), dtype=torch.uint8, device="cuda")


def prepare(case, seed):
    if case["kind"] == "batch":
        key = (case["count"], case["specs"], case["form"])
        specs = _batch_specs(case)
        if key not in _batch_plans:
            _batch_plans[key] = [_plan(s, _coords(s, "stretched" if st else "uniform"), case["form"]) for s, st in specs]
        starts, total = _batch_layout(specs)
        u = _batch_fields(case, seed)
        coef, back = torch.zeros_like(u), torch.zeros_like(u)

        def part(t, i):
            return t[starts[i]:starts[i] + math.prod(specs[i][0])]

        plans = _batch_plans[key]
        dec = [(mgr.MGR_OP_DECOMPOSE, p, part(u, i), part(coef, i)) for i, p in enumerate(plans)]
        rec = [(mgr.MGR_OP_RECOMPOSE, p, part(coef, i), part(back, i)) for i, p in enumerate(plans)]
        torch.cuda.synchronize()  # the batch runs on the context's own stream
        return dict(kind="batch", coef=coef, back=back, dec=mgr.Context.batch_prepare(dec),
                    rec=mgr.Context.batch_prepare(rec), keep=u)
    shape = _shape(case)
    coords = _coords(shape, case["coords"])
    u = _field(case, seed)
    plan = _plan(shape, coords, case["form"])
    st = dict(kind=case["kind"], plan=plan, ws=_workspace(plan), u=u)
    if case["kind"] == "quantized":
        # codes of another field, as a reader of compressed data has them
        ops = _operators(shape, coords, plan.levels)
        other = _pack(_decompose(_field(case, seed + 500009).double(), ops), ops)
        st["given"] = torch.cat([torch.round(c / q) for c, q in zip(other, _bins(ops))]).to(torch.int32)
        st["codes"] = torch.empty(u.numel(), dtype=torch.int32, device="cuda")
    elif case["kind"] == "host":
        st["host"] = u.cpu().pin_memory()
        st["host_coef"], st["host_back"] = (torch.empty(shape, dtype=u.dtype).pin_memory() for _ in range(2))
        st["dev"] = torch.empty_like(u)
    else:
        st["coef"] = torch.empty(u.numel(), dtype=u.dtype, device="cuda") if case["kind"] == "packed" else torch.empty_like(u)
        st["coarse"] = torch.empty_like(u) if case["kind"] == "packed" else None
    st["back"] = torch.empty_like(u)
    return st


def run(st):
    if st["kind"] == "batch":
        ctx = _ctx()
        ctx.batch_submit(st["dec"])
        # (a submit runs after the one before it)
        rc, _ = ctx.batch_poll(ctx.batch_submit(st["rec"]))
        if rc != mgr.MGR_OK:
            raise RuntimeError("the batch did not finish")
        return {"coefficients": st["coef"], "field": st["back"]}
    p, ws = st["plan"], st["ws"]
    if st["kind"] == "packed":
        p.decompose_packed(st["u"], st["coef"], ws)
        p.recompose_packed(st["coef"], p.levels + 1, st["back"], ws)
        p.recompose_packed(st["coef"], p.levels, st["coarse"], ws)
        return {"classes": st["coef"], "field": st["back"], "without_finest": st["coarse"]}
    if st["kind"] == "quantized":
        p.decompose_quantized(st["u"], st["codes"], TAU, ws)
        p.recompose_dequantized(st["given"], p.levels + 1, TAU, st["back"], ws)
        return {"codes": st["codes"], "field": st["back"]}
    if st["kind"] == "host":
        p.decompose_host(st["host"], st["host_coef"], st["u"], st["dev"], ws)
        p.recompose_host(st["host_coef"], st["host_back"], st["dev"], st["back"], ws)
        torch.cuda.current_stream().synchronize()  # the results are in host memory only then
        return {"coefficients": st["host_coef"], "field": st["host_back"]}
    p.decompose(st["u"], st["coef"], ws)
    p.recompose(st["coef"], st["back"], ws)
    return {"coefficients": st["coef"], "field": st["back"]}


# ---------------------------------------------------------------- work

def _depth(shape):
    """Levels of the default hierarchy: the smallest side is halved until it has 3 nodes."""
    n, levels = min(shape), 0
    while n > 3:
        n, levels = n // 2 + 1, levels + 1
    return levels


def _flops(shape):
    """Operations of a decomposition and a recomposition (a multiply-add is two): per level the
    interpolation and difference at each node, one five-point sum per axis, one solve per axis."""
    coef = stencil = solve = 0.0
    n = list(shape)
    d = len(n)
    for _ in range(_depth(shape)):
        m = [k // 2 + 1 for k in n]
        for k in range(d):
            nodes = math.prod(m[:k]) * (n[k] - m[k]) * math.prod(n[k + 1:])
            coef += nodes * (2 if k == 0 else 3)
            stencil += 5 * math.prod(n[:k]) * math.prod(m[k:])
            solve += 2 * math.prod(m)
        # the coefficients vanish on lines whose other nodes are all coarse, but for the fine ones
        stencil -= 3 * math.prod(m)
        solve += 0.5 * math.prod(m)  # the correction's addition
        n = m
    return 2.0 * coef * 2 + 2.0 * stencil * 2 + 2.0 * solve * 2


def work(case):
    shapes = [s for s, _ in _batch_specs(case)] if case["kind"] == "batch" else [_shape(case)]
    nodes = sum(math.prod(s) for s in shapes)
    item = 8 if case["form"] == "f64" else 4
    flops = sum(_flops(s) for s in shapes)
    # decomposition: field in, coefficients out; recomposition: coefficients in, field out
    moved = {"quantized": nodes * (2 * item + 2 * 4), "packed": nodes * 5 * item + nodes * item / 2 ** len(shapes[0])}
    return {"bytes": moved.get(case["kind"], nodes * 4 * item), "flops": flops}


# ---------------------------------------------------------------- in 64 bits

def _axis_operators(x):
    """P (n x m) and Z = (P^T M P)^-1 P^T M (m x n) of one axis with nodes x; the coarse nodes."""
    n = len(x)
    keep = list(range(0, n, 2)) + ([n - 1] if n % 2 == 0 else [])
    P = np.zeros((n, len(keep)))
    for q, i in enumerate(keep):
        P[i, q] = 1.0
        if q + 1 < len(keep) and keep[q + 1] == i + 2:
            right = (x[i + 1] - x[i]) / (x[i + 2] - x[i])
            P[i + 1, q], P[i + 1, q + 1] = 1.0 - right, right
    h = np.diff(x)
    M = np.zeros((n, n))
    i = np.arange(n - 1)
    M[i, i] += h / 3
    M[i + 1, i + 1] += h / 3
    M[i, i + 1] = M[i + 1, i] = h / 6
    Z = np.linalg.solve(P.T @ M @ P, P.T @ M)
    return torch.from_numpy(P).cuda(), torch.from_numpy(Z).cuda(), torch.tensor(keep, device="cuda")


def _operators(shape, coords, levels):
    """Per level, finest first, the operators of every axis."""
    xs = [np.arange(n, dtype=np.float64) if coords is None else coords[k] for k, n in enumerate(shape)]
    ops = []
    for _ in range(levels):
        ops.append([_axis_operators(x) for x in xs])
        xs = [x[o[2].cpu().numpy()] for x, o in zip(xs, ops[-1])]
    return ops


def _apply(mats, v):
    """The tensor product of `mats` on v, one axis at a time."""
    for ax, a in enumerate(mats):
        lead = v.shape[:ax]
        tail = v.shape[ax + 1:]
        v = torch.matmul(a, v.reshape(math.prod(lead), v.shape[ax], math.prod(tail))).reshape(*lead, a.shape[0], *tail)
    return v


def _coarse(v, level):
    for ax, o in enumerate(level):
        v = v.index_select(ax, o[2])
    return v


def _decompose(v, ops):
    """[level-L coefficients on their grid, ..., level-1 ones, coarsest values]."""
    parts = []
    for level in ops:
        w = _coarse(v, level)
        c = v - _apply([o[0] for o in level], w)
        parts.append(c)
        v = w + _apply([o[1] for o in level], c)
    return parts + [v]


def _recompose(parts, ops):
    v = parts[-1]
    for c, level in zip(reversed(parts[:-1]), reversed(ops)):
        if c is None:
            v = _apply([o[0] for o in level], v)
        else:
            v = c + _apply([o[0] for o in level], v - _apply([o[1] for o in level], c))
    return v


def _nodal(parts, ops):
    """Coefficients and coarsest values at their nodes of the finest grid."""
    v = parts[-1]
    for c, level in zip(reversed(parts[:-1]), reversed(ops)):
        c = c.clone()
        c[torch.meshgrid(*[o[2] for o in level], indexing="ij")] = v
        v = c
    return v


def _fine(level):
    """True at the nodes of a level that the next coarser one leaves out."""
    grids = []
    for ax, o in enumerate(level):
        there = torch.zeros(o[0].shape[0], dtype=torch.bool, device="cuda")
        there[o[2]] = True
        grids.append(there.reshape([-1 if a == ax else 1 for a in range(len(level))]))
    out = grids[0]
    for g in grids[1:]:
        out = out & g
    return ~out


def _pack(parts, ops):
    """The classes, coarsest first."""
    return [parts[-1].reshape(-1)] + [c[_fine(level)] for c, level in zip(reversed(parts[:-1]), reversed(ops))]


def _unpack(classes, ops, shape):
    parts = []
    for c, level in zip(reversed(classes[1:]), ops):
        v = torch.zeros([o[0].shape[0] for o in level], dtype=torch.float64, device="cuda")
        v[_fine(level)] = c
        parts.append(v)
    return parts + [classes[0].reshape([o[0].shape[1] for o in ops[-1]] if ops else shape)]


def _bins(ops):
    """Bin width per class, coarsest first: an error of at most TAU in the maximum norm."""
    share = 2 * TAU / (len(ops) + 1)
    norms = [math.prod(o[1].abs().sum(1).max().item() for o in level) for level in ops]
    return [share] + [share / (1.0 + z) for z in reversed(norms)]


def exact(case, seed):
    if case["kind"] == "batch":
        specs = _batch_specs(case)
        starts, _ = _batch_layout(specs)
        u = _batch_fields(case, seed).double()
        coef = torch.zeros_like(u)
        cached = {}
        for (shape, stretched), at in zip(specs, starts):
            v = u[at:at + math.prod(shape)].reshape(shape)
            ops = _batch_operators(shape, stretched, cached)
            coef[at:at + v.numel()] = _nodal(_decompose(v, ops), ops).reshape(-1)
        return {"coefficients": coef, "field": u}
    shape = _shape(case)
    ops = _operators(shape, _coords(shape, case["coords"]), _depth(shape))
    u = _field(case, seed).double()
    if case["kind"] == "quantized":
        other = _pack(_decompose(_field(case, seed + 500009).double(), ops), ops)
        given = [torch.round(c / q) * q for c, q in zip(other, _bins(ops))]
        return {"codes": None, "field": _recompose(_unpack(given, ops, shape), ops)}
    parts = _decompose(u, ops)
    if case["kind"] == "packed":
        return {"classes": torch.cat(_pack(parts, ops)), "field": u,
                "without_finest": _recompose([None] + parts[1:], ops)}
    coef = _nodal(parts, ops)
    if case["kind"] == "host":
        return {"coefficients": coef.cpu(), "field": u.cpu()}
    return {"coefficients": coef, "field": u}


def _batch_operators(shape, stretched, cached):
    """Like _operators, with the 1D operators of each axis made once per length and level."""
    levels, axes = _depth(shape), []
    for n in shape:
        for l in itertools.count():
            if l == levels:
                break
            if (n, stretched, l) not in cached:
                x = _coords((n,), "stretched")[0] if stretched else np.arange(n, dtype=np.float64)
                for _ in range(l):
                    x = x[list(range(0, len(x), 2)) + ([len(x) - 1] if len(x) % 2 == 0 else [])]
                cached[(n, stretched, l)] = _axis_operators(x)
    for l in range(levels):
        axes.append([cached[(n, stretched, l)] for n in shape])
    return axes
