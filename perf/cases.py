"""What the derivative-evaluation library is asked to do in earnest, as measurable cases.

A case is one workload family at one size, one precision and one kind of use, each through the
public binding (`binding.exa_create_batch` and the calls of `include/exa.h`):

  step       exa_eval_all with every output: what one iteration of a second-order method with its own
             sparse assembly reads (objective, gradient, constraints, Jacobian and Hessian in COO and
             summed into CSC), replayed from the cached graph.
  callbacks  exa_obj, exa_grad, exa_cons, exa_jac_coord, exa_hess_coord one after another: the
             solver-facing callbacks of a solver that asks for them one at a time.
  csc        exa_cons, exa_jac_csc, exa_hess_csc: what a direct sparse factorisation consumes.
  products   exa_jprod, exa_jtprod, exa_hprod: matrix-free (Krylov) use.

`prepare` makes the model handle (created once, as a solver does) and device inputs and outputs;
`run` is one pass.  Models large enough for the creation-time autotuner are created with a fixed
launch configuration per family and precision, the one the tuner chose on a GB300
(`Model.tuned_options`), so that every model of a family runs the same configuration and creation
stays short; smaller ones are created with the defaults, which do not tune them either.
`exact` restates the derivatives in torch FP64: every pattern tree of the flat IR is evaluated with
second-order forward differentiation over its instances.
"""
import functools
import math

import numpy as np
import torch

import synth
from paper_2608_16265_gb300 import binding

FP64, MIXED = binding.EXA_FP64, binding.EXA_MIXED_FP32

# ------------------------------------------------------------------ the cases


def listed():
    return [
        # the smallest use: a 1000-variable model whose step is a few microseconds of work
        dict(name="rosenbrock_1k_step", family="rosenbrock", n=1000, precision="fp64", use="step"),
        # a small network in a solver that calls one callback at a time: ten launches, little work
        dict(name="acopf_500_callbacks", family="acopf", buses=500, branches=700, gens=100, precision="fp64",
             use="callbacks"),
        # a national-grid-sized network, the ordinary size of one model
        dict(name="acopf_30k_step", family="acopf", buses=30000, branches=45000, gens=5000, precision="fp64",
             use="step"),
        # the same network, mixed precision, callback by callback
        dict(name="acopf_30k_callbacks_mixed", family="acopf", buses=30000, branches=45000, gens=5000,
             precision="mixed", use="callbacks"),
        # the same network in a matrix-free method
        dict(name="acopf_30k_products", family="acopf", buses=30000, branches=45000, gens=5000, precision="fp64",
             use="products"),
        # optimal control with a free final time: one variable in every row (a 300,000-entry column)
        dict(name="goddard_100k_products", family="goddard", steps=100000, precision="fp64", use="products"),
        # PDE control, the configured grid
        dict(name="pde_1k_step", family="pde", grid=1000, precision="fp64", use="step"),
        # PDE control on a finer, odd grid in mixed precision: larger than the L2 cache
        dict(name="pde_2k_step_mixed", family="pde", grid=2001, precision="mixed", use="step"),
        # stochastic programming: 1000 buses x 256 scenarios, matrices for a direct factorisation
        dict(name="two_stage_256_csc", family="two_stage", buses=1000, branches=1500, gens=166, scenarios=256,
             precision="fp64", use="csc"),
        # a ragged batch of networks in a matrix-free method
        dict(name="batch_32_products", family="batch", members=32, smallest=200, biggest=20000, precision="fp64",
             use="products"),
        # the benchmark workload: 256 networks of 200 to 20,000 buses, FP64 and mixed
        dict(name="batch_256_step", family="batch", members=256, smallest=200, biggest=20000, precision="fp64",
             use="step"),
        dict(name="batch_256_step_mixed", family="batch", members=256, smallest=200, biggest=20000,
             precision="mixed", use="step"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["rosenbrock", "acopf", "acopf", "goddard", "pde", "two_stage", "batch"])
    c = dict(family=family)
    if family == "rosenbrock":
        c.update(n=_log(rng, 100, 300000))
    elif family == "acopf":
        b = _log(rng, 60, 60000)
        c.update(buses=b, branches=int(b * rng.uniform(1.2, 1.6)), gens=max(1, int(b / rng.uniform(4, 9))))
    elif family == "goddard":
        c.update(steps=_log(rng, 200, 200000))
    elif family == "pde":
        c.update(grid=_log(rng, 30, 2000))
    elif family == "two_stage":
        b = _log(rng, 60, 1000)
        c.update(buses=b, branches=int(b * rng.uniform(1.2, 1.6)), gens=max(1, b // 6), scenarios=_log(rng, 4, 256))
    else:
        c.update(members=_log(rng, 3, 200), smallest=rng.randint(150, 300), biggest=_log(rng, 2000, 20000))
    c.update(precision=rng.choice(["fp64", "fp64", "mixed"]),
             use=rng.choice(["step", "callbacks", "csc", "products"]))
    return c


# ------------------------------------------------------------------ models


@functools.lru_cache(maxsize=3)
def _models(key):
    """The case's workloads (host descriptions).  A network is the same for every seed; the points vary."""
    c = dict(key)
    f = c["family"]
    if f == "rosenbrock":
        return (synth.rosenbrock(c["n"]),)
    if f == "acopf":
        return (synth.acopf(c["buses"], c["branches"], c["gens"], seed=2),)
    if f == "goddard":
        return (synth.goddard(c["steps"]),)
    if f == "pde":
        return (synth.pde(c["grid"]),)
    if f == "two_stage":
        return (synth.two_stage_acopf(c["buses"], c["branches"], c["gens"], c["scenarios"], seed=4),)
    return tuple(synth.acopf_batch(c["members"], seed=7, bmin=c["smallest"], bmax=c["biggest"]))


def _workloads(case):
    return _models(tuple(sorted((k, v) for k, v in case.items() if k not in ("name", "precision", "use"))))


_POINT = dict(rosenbrock=synth.rosenbrock_point, acopf=synth.acopf_point, batch=synth.acopf_point,
              goddard=synth.goddard_point, pde=synth.pde_point, two_stage=synth.two_stage_point)


def _point(case, wls, seed):
    pts = [_POINT[case["family"]](w, seed * 1009 + i) for i, w in enumerate(wls)]
    x = np.concatenate([p[0] for p in pts])
    y = np.concatenate([p[1] for p in pts])
    rng = np.random.default_rng(seed + 77)
    # sigma: the objective scaling a solver passes
    return x, y, 1.0 + 0.25 * (seed % 3), rng.standard_normal(len(x)), rng.standard_normal(len(y))


_LAZY, _SPLIT, _SCATTER = binding.EXA_FLAG_LAZY_LOADS, binding.EXA_FLAG_SPLIT, binding.EXA_FLAG_CSC_SCATTER
_NO_HCOMP, _UPFRONT, _PFC = binding.EXA_FLAG_NO_HCOMP, binding.EXA_FLAG_UPFRONT, binding.EXA_FLAG_PF_COLUMNS

# launch configurations chosen by the tuner: (block, min_blocks, grid_factor, flags)
_TUNED = {
    ("rosenbrock", "fp64"): (64, 10, 1, _NO_HCOMP),
    ("rosenbrock", "mixed"): (64, 10, 1, _NO_HCOMP | _SCATTER | _UPFRONT | _PFC),
    ("acopf", "fp64"): (64, 0, -1, _LAZY),
    ("acopf", "mixed"): (128, 0, -1, _LAZY | _SPLIT),
    ("goddard", "fp64"): (64, 0, 1, _UPFRONT),
    ("goddard", "mixed"): (64, 0, -1, _LAZY | _NO_HCOMP),
    ("pde", "fp64"): (64, 0, 1, _SCATTER | _NO_HCOMP),
    ("pde", "mixed"): (128, 0, 1, _LAZY | _NO_HCOMP),
    ("two_stage", "fp64"): (64, 16, 4, _LAZY),
    ("two_stage", "mixed"): (128, 0, 1, 0),
    ("batch", "fp64"): (64, 14, 4, _LAZY),
    ("batch", "mixed"): (128, 8, -1, _LAZY),
}


def _options(case, wls):
    # Distinct instance counts stand for the fused groups: below 64k instances in all a model has
    # fewer tiles than the tuner asks for, and the default creation runs no tuner.
    inst = sum(sum({p.n_inst for p in w.flat.patterns}) for w in wls)
    if inst < 64000:
        return dict(flags=binding.EXA_FLAG_NO_TUNE)
    block, minb, grid, flags = _TUNED[case["family"], case["precision"]]
    return dict(block=block, min_blocks=minb, grid_factor=grid, flags=flags | binding.EXA_FLAG_NO_TUNE, chunks=1)


# ------------------------------------------------------------------ the measured path


def prepare(case, seed):
    wls = _workloads(case)
    m = binding.exa_create_batch([w.flat for w in wls], FP64 if case["precision"] == "fp64" else MIXED,
                                 **_options(case, wls))
    x, y, sigma, v, w = _point(case, wls, seed)
    dev = lambda a: torch.as_tensor(a, device="cuda")  # noqa: E731
    sizes = dict(step=dict(f=1, g=m.nvar, c=m.ncon, jac=m.nnzj, hess=m.nnzh, jac_csc=m.nnzj_csc, hess_csc=m.nnzh_csc),
                 callbacks=dict(f=1, g=m.nvar, c=m.ncon, jac=m.nnzj, hess=m.nnzh),
                 csc=dict(c=m.ncon, jac_csc=m.nnzj_csc, hess_csc=m.nnzh_csc),
                 products=dict(jv=m.ncon, jtw=m.nvar, hv=m.nvar))[case["use"]]
    out = {k: torch.empty(n, dtype=torch.float64, device="cuda") for k, n in sizes.items()}
    return dict(use=case["use"], model=m, x=dev(x), y=dev(y), sigma=sigma, v=dev(v), w=dev(w), out=out)


def run(state):
    m, x, y, s, o = state["model"], state["x"], state["y"], state["sigma"], state["out"]
    if state["use"] == "step":
        m.exa_eval_all(x, y, s, **o)
    elif state["use"] == "callbacks":
        m.exa_obj(x, o["f"])
        m.exa_grad(x, o["g"])
        m.exa_cons(x, o["c"])
        m.exa_jac_coord(x, o["jac"])
        m.exa_hess_coord(x, y, s, o["hess"])
    elif state["use"] == "csc":
        m.exa_cons(x, o["c"])
        m.exa_jac_csc(x, o["jac_csc"])
        m.exa_hess_csc(x, y, s, o["hess_csc"])
    else:
        m.exa_jprod(x, state["v"], o["jv"])
        m.exa_jtprod(x, state["w"], o["jtw"])
        m.exa_hprod(x, y, s, state["v"], o["hv"])
    return o


# ------------------------------------------------------------------ work a pass cannot do without


def work(case):
    """Inputs read once and outputs written once by each call; floating-point operations from the
    pattern trees (one per tree node for a value, two per first-order slot, three per second-order
    slot, per instance), and two per matrix entry of a product."""
    nv = nc = nj = nh = ops1 = ops2 = data = 0
    keys, narrow = 0, case["precision"] == "mixed"
    for w in _workloads(case):
        nv += w.flat.nvar
        nc += w.flat.ncon
        cols = {}
        for p in w.flat.patterns:
            sym, pairs = _slots(p)
            nodes = len(p.vop)
            if p.kind != binding.ir.K_OBJ:
                nj += p.n_inst * len(sym)
            nh += p.n_inst * len(pairs)
            ops1 += p.n_inst * (nodes + 2 * len(sym))
            ops2 += p.n_inst * (nodes + 3 * len(pairs))
            for f in p.fields:
                cols[id(f)] = f.size * (4 if f.dtype == np.int32 or narrow else 8)
        data += sum(cols.values())
        keys += _csc_count(w.flat) if case["use"] in ("step", "csc") else 0
    x, y, c = 8 * nv, 8 * nc, 8 * nc
    if case["use"] == "step":
        return dict(bytes=x + y + data + 8 + 8 * nv + c + 8 * (nj + nh) + 8 * keys, flops=ops1 + ops2)
    if case["use"] == "callbacks":
        return dict(bytes=5 * x + y + 2 * data + 8 + 8 * nv + c + 8 * (nj + nh), flops=2 * ops1 + ops2)
    if case["use"] == "csc":
        return dict(bytes=3 * x + y + 3 * data + c + 8 * keys, flops=2 * ops1 + ops2)
    return dict(bytes=7 * x + y + 3 * data + 2 * c, flops=2 * ops1 + ops2 + 4 * nj + 4 * nh)


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _csc_count(flat):
    """Distinct (row, column) entries of the Jacobian and of the Hessian's lower triangle."""
    dev, js, hs = _device(), [], []
    for p in flat.patterns:
        if not p.n_inst:
            continue
        roots, pairs = _slots(p)
        idx = [torch.broadcast_to(torch.as_tensor(_index(p, r, dev), device=dev), (p.n_inst,)) for r in roots]
        if p.kind != binding.ir.K_OBJ:
            row = _row(p, dev)
            js += [i * max(flat.ncon, 1) + row for i in idx]
        hs += [torch.minimum(idx[a], idx[b]) * flat.nvar + torch.maximum(idx[a], idx[b]) for a, b in pairs]
    return sum(torch.unique(torch.cat(k)).numel() for k in (js, hs) if k)


# ------------------------------------------------------------------ FP64 restatement

_UNARY = {  # value, first and second derivative
    binding.ir.V_NEG: lambda u, n: (-u, -torch.ones_like(u), None),
    binding.ir.V_ABS2: lambda u, n: (u * u, 2 * u, 2 * torch.ones_like(u)),
    binding.ir.V_INV: lambda u, n: (1 / u, -1 / u ** 2, 2 / u ** 3),
    binding.ir.V_EXP: lambda u, n: (torch.exp(u),) * 3,
    binding.ir.V_SIN: lambda u, n: (torch.sin(u), torch.cos(u), -torch.sin(u)),
    binding.ir.V_COS: lambda u, n: (torch.cos(u), -torch.sin(u), -torch.cos(u)),
    binding.ir.V_POWI: lambda u, n: (u ** n, n * u ** (n - 1), n * (n - 1) * u ** (n - 2)),
}
_LINEAR = (binding.ir.V_NEG, binding.ir.V_ADD, binding.ir.V_SUB)


def _index_key(p, r):
    op, a, b, v = int(p.iop[r]), int(p.ia[r]), int(p.ib[r]), int(p.ii[r])
    return (op, v) if op < binding.ir.I_ADD else (op, _index_key(p, a), _index_key(p, b))


def _slots(p):
    """First-order slots (index roots of the pattern's distinct variables, in pre-order of the tree)
    and second-order slots (pairs of them in the order the reverse pass meets them)."""
    ir, keys, roots, sym_of = binding.ir, {}, [], {}

    def visit(i):
        if p.vop[i] == ir.V_VAR:
            k = _index_key(p, p.va[i])
            if k not in keys:
                keys[k] = len(roots)
                roots.append(int(p.va[i]))
            sym_of[i] = keys[k]
        for child in _children(p, i):
            visit(child)

    root = len(p.vop) - 1
    visit(root)
    pairs, seen = [], set()

    def emit(a, b):
        if (min(a, b), max(a, b)) not in seen:
            seen.add((min(a, b), max(a, b)))
            pairs.append((a, b))

    def second(i, curved):
        """Symbols below node i in pre-order; `curved`: its second adjoint may be nonzero."""
        op, kids = p.vop[i], _children(p, i)
        if op == ir.V_VAR:
            if curved:
                emit(sym_of[i], sym_of[i])
            return [sym_of[i]]
        own = curved or not (op in _LINEAR or op == ir.V_MUL or (op == ir.V_POWI and p.vi[i] in (0, 1)))
        if len(kids) == 2:
            left = second(kids[0], curved if op == ir.V_DIV else own)
            right = second(kids[1], own)
            if left and right and (curved or op not in _LINEAR):
                for a in left:
                    for b in right:
                        emit(a, b)
            return left + right
        return second(kids[0], own) if kids else []

    second(root, False)
    return roots, pairs


def _children(p, i):
    op = p.vop[i]
    return [] if op <= binding.ir.V_PARAM else [int(p.va[i])] if op < binding.ir.V_ADD else [int(p.va[i]), int(p.vb[i])]


def _index(p, r, dev):
    """Index expression r of every instance (a tensor, or a number where it is the same for all)."""
    ir, op = binding.ir, p.iop[r]
    if op == ir.I_CONST:
        return int(p.ii[r])
    if op == ir.I_INST:
        return torch.arange(p.n_inst, device=dev)
    if op == ir.I_FIELD:
        return torch.as_tensor(p.fields[int(p.ii[r])].astype(np.int64), device=dev)
    a, b = _index(p, p.ia[r], dev), _index(p, p.ib[r], dev)
    return a + b if op == ir.I_ADD else a - b if op == ir.I_SUB else a * b


def _row(p, dev):
    if p.kind == binding.ir.K_AUG:
        return p.row_base + _index(p, p.row_root, dev)
    return p.row_base + torch.arange(p.n_inst, device=dev)


def _pattern(p, x, theta, dev):
    """Value, gradient {symbol: d} and Hessian {(a, b), a <= b: dd} of every instance, with the
    instances' variable indices per symbol."""
    ir = binding.ir
    roots, pairs = _slots(p)
    keys = {_index_key(p, r): s for s, r in enumerate(roots)}
    full = lambda i: torch.broadcast_to(torch.as_tensor(i, device=dev), (p.n_inst,))  # noqa: E731
    idx = [full(_index(p, r, dev)) for r in roots]
    ones = torch.ones(p.n_inst, dtype=torch.float64, device=dev)

    def add(d, k, v):
        d[k] = d[k] + v if k in d else v

    def ev(i):
        op, kids = p.vop[i], _children(p, i)
        if op == ir.V_CONST:
            return float(p.vf[i]) * ones, {}, {}
        if op == ir.V_DATA:
            return torch.as_tensor(p.fields[int(p.vi[i])].astype(np.float64), device=dev), {}, {}
        if op == ir.V_PARAM:
            return theta[full(_index(p, p.va[i], dev))], {}, {}
        if op == ir.V_VAR:
            s = keys[_index_key(p, p.va[i])]
            return x[idx[s]], {s: ones}, {}
        u, gu, hu = ev(kids[0])
        g, h = {}, {}
        if len(kids) == 1:
            v, d1, d2 = _UNARY[op](u, int(p.vi[i]))
            for s, t in gu.items():
                g[s] = d1 * t
            for k, t in hu.items():
                h[k] = d1 * t
            if d2 is not None:
                for a in gu:
                    for b in gu:
                        if a <= b:
                            add(h, (a, b), d2 * gu[a] * gu[b])
            return v, g, h
        w, gw, hw = ev(kids[1])
        uw = ww = None
        if op == ir.V_ADD:
            v, du, dw = u + w, ones, ones
        elif op == ir.V_SUB:
            v, du, dw = u - w, ones, -ones
        elif op == ir.V_MUL:
            v, du, dw, uw = u * w, w, u, ones
        elif op == ir.V_DIV:
            v, du, dw, uw, ww = u / w, 1 / w, -u / w ** 2, -1 / w ** 2, 2 * u / w ** 3
        else:
            raise NotImplementedError(op)
        for src, d, dst in ((gu, du, g), (gw, dw, g), (hu, du, h), (hw, dw, h)):
            for k, t in src.items():
                add(dst, k, d * t)
        if uw is not None:
            for a in gu:
                for b in gw:
                    t = uw * gu[a] * gw[b]
                    add(h, (min(a, b), max(a, b)), 2 * t if a == b else t)
        if ww is not None:
            for a in gw:
                for b in gw:
                    if a <= b:
                        add(h, (a, b), ww * gw[a] * gw[b])
        return v, g, h

    v, g, h = ev(len(p.vop) - 1)
    return v, g, h, idx, pairs, ones


def _exact_member(flat, x, y, sigma, dev):
    """f, g, c and (rows, columns, values) of the Jacobian and of the Hessian's lower triangle."""
    f = torch.zeros(1, dtype=torch.float64, device=dev)
    g, c = torch.zeros_like(x), torch.zeros(flat.ncon, dtype=torch.float64, device=dev)
    theta = torch.as_tensor(np.asarray(flat.theta, dtype=np.float64), device=dev)
    jac, hess = [], []
    for p in flat.patterns:
        if not p.n_inst:
            continue
        v, gr, he, idx, pairs, ones = _pattern(p, x, theta, dev)
        obj = p.kind == binding.ir.K_OBJ
        row = None if obj else torch.broadcast_to(torch.as_tensor(_row(p, dev), device=dev), (p.n_inst,))
        if obj:
            f += v.sum()
            for s, t in gr.items():
                g.index_add_(0, idx[s], t)
        else:
            c.index_add_(0, row, v)
            vals = [gr.get(s, 0 * ones) for s in range(len(idx))]
            if idx:
                jac.append([torch.stack(t, 1).reshape(-1) for t in ([row] * len(idx), idx, vals)])
        if pairs:
            wt = sigma if obj else y[row]
            rows = [torch.maximum(idx[a], idx[b]) for a, b in pairs]
            cols = [torch.minimum(idx[a], idx[b]) for a, b in pairs]
            vals = []
            for a, b in pairs:
                t = wt * he.get((min(a, b), max(a, b)), 0 * ones)
                vals.append(torch.where(idx[a] == idx[b], 2 * t, t) if a != b else t)
            hess.append([torch.stack(t, 1).reshape(-1) for t in (rows, cols, vals)])

    def cat(parts):
        if not parts:
            z = torch.zeros(0, dtype=torch.int64, device=dev)
            return z, z, z.double()
        return tuple(torch.cat(t) for t in zip(*parts))

    return f, g, c, cat(jac), cat(hess)


def _sum_duplicates(entries, nrow):
    r, c, v = entries
    key, at = torch.unique(c * max(nrow, 1) + r, return_inverse=True)
    return torch.zeros(key.numel(), dtype=torch.float64, device=v.device).index_add_(0, at, v)


def exact(case, seed):
    wls = _workloads(case)
    dev = _device()
    xs, ys, sigma, vs, ws = (torch.as_tensor(a, device=dev) if isinstance(a, np.ndarray) else a
                             for a in _point(case, wls, seed))
    out = {}
    ox = oc = 0

    def put(**kv):
        for k, t in kv.items():
            out.setdefault(k, []).append(t)

    for w in wls:
        n, m = w.flat.nvar, w.flat.ncon
        x, y = xs[ox:ox + n], ys[oc:oc + m]
        f, g, c, jac, hess = _exact_member(w.flat, x, y, sigma, dev)
        if case["use"] == "products":
            v, u = vs[ox:ox + n], ws[oc:oc + m]
            (jr, jc, jv), (hr, hc, hv) = jac, hess
            off = hr != hc
            hp = torch.zeros_like(x).index_add_(0, hr, hv * v[hc])
            put(jv=torch.zeros_like(c).index_add_(0, jr, jv * v[jc]), jtw=torch.zeros_like(x).index_add_(0, jc, jv * u[jr]),
                hv=hp.index_add_(0, hc[off], (hv * v[hr])[off]))
        else:
            put(f=f, g=g, c=c, jac=jac[2], hess=hess[2])
            if case["use"] != "callbacks":
                put(jac_csc=_sum_duplicates(jac, m), hess_csc=_sum_duplicates(hess, n))
        ox, oc = ox + n, oc + m
    keep = dict(step=("f", "g", "c", "jac", "hess", "jac_csc", "hess_csc"), callbacks=("f", "g", "c", "jac", "hess"),
                csc=("c", "jac_csc", "hess_csc"), products=("jv", "jtw", "hv"))[case["use"]]
    return {k: torch.stack(out[k]).sum(0) if k == "f" else torch.cat(out[k]) for k in keep}
