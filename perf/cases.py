"""Performance cases of the Bootstrap AMG library: what a user's program has it do.

The chains are random walks on weighted 2-D networks (the paper's uniform network with a
conductance per link), tandem queues near the paper's rates, and walks on planar triangulations
with a random diagonal per cell (unstructured, six links per state on average, as a Delaunay
graph).  Every input is made with plain torch on the GPU from the seed alone.

Kinds of case:
  solve     bamg.Solver(...) and .solve(tol): the whole method on one chain, from the CSR arrays
  batch     bamg.solve_batch: many small chains at once
  relax     the omega-Jacobi sweeps over the test vectors (setup, Section 3)
  shifted   the sweeps on (B - lambda_k T) x_k = 0 over the eigenvector columns (Algorithm 3)
  interp    least-squares interpolation rows of one level (Algorithm 2)
  galerkin  the coarse operators B_c = Q B P and T_c = Q T P of one level
  cr        compatible-relaxation coarsening of one level (Algorithm 1)
  vcycle    one V(2,2) cycle of an imported hierarchy (the preconditioner on its own)
  forward   the learned interpolation's network over the rows of a level
  train     one pass of its training over a data set
"""

import numpy as np
import torch

import paper_1004_1451_gb300 as bamg

DEV = "cuda"
OFFS = [(-1, -1), (0, -1), (1, -1), (-1, 0), (0, 0), (1, 0), (-1, 1), (0, 1), (1, 1)]  # (dx, dy), by index
FEATURES, HIDDEN, SLOTS = 112, 128, 16


def listed():
    return [
        # the smallest whole call: the paper's uniform network at 64 x 64, plain FP64, latency bound
        {"name": "solve grid 64 fp64", "kind": "solve", "chain": "grid", "nx": 64, "ny": 64, "r": 8, "fp64": True},
        # the flagship: a tandem queue of capacity 255 (65,536 states), mixed precision
        {"name": "solve tandem 256 mixed", "kind": "solve", "chain": "tandem", "nx": 256, "ny": 256, "r": 10,
         "fp64": False},
        # an unstructured chain of 2^18 states: compatible-relaxation coarsening, long coarse rows
        {"name": "solve planar 512 mixed", "kind": "solve", "chain": "planar", "nx": 512, "ny": 512, "r": 16,
         "fp64": False},
        # many small independent chains on one GPU
        {"name": "batch 32 grids mixed", "kind": "batch", "chains": 32, "lo": 32, "hi": 96, "r": 8, "fp64": False},
        # test-vector relaxation of a large level: the vectors and the matrix stream from HBM
        {"name": "relax grid 2048 fp32", "kind": "relax", "chain": "grid", "nx": 2048, "ny": 2048, "r": 16,
         "fp64": False, "nu": 4},
        # the eigenvector columns of the upward pass, odd sides, a middling level
        {"name": "shifted planar 701x523 fp32", "kind": "shifted", "chain": "planar", "nx": 701, "ny": 523, "r": 7,
         "fp64": False, "nu": 2},
        # the interpolation fit of an unstructured level
        {"name": "interp planar 512 fp32", "kind": "interp", "chain": "planar", "nx": 512, "ny": 512, "r": 16,
         "fp64": False},
        # a coarse operator in plain FP64
        {"name": "galerkin planar 400x384 fp64", "kind": "galerkin", "chain": "planar", "nx": 400, "ny": 384,
         "fp64": True},
        # the splitting of an unstructured level
        {"name": "cr planar 256 fp64", "kind": "cr", "chain": "planar", "nx": 256, "ny": 256},
        # one preconditioner application on a hierarchy kept from an earlier run, ragged sides
        {"name": "vcycle grid 515x509 mixed", "kind": "vcycle", "chain": "grid", "nx": 515, "ny": 509, "fp64": False},
        # the learned interpolation of a held-out queue's finest level (capacity 511)
        {"name": "forward 262144", "kind": "forward", "rows": 262144},
        # its training: one pass over 2^16 rows in batches of 4096
        {"name": "train 65536 by 4096", "kind": "train", "rows": 65536, "batch": 4096},
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["solve", "batch", "relax", "shifted", "interp", "galerkin", "cr", "vcycle", "forward", "train"])
    fp64 = rng.random() < 0.35
    if kind == "solve":
        chain = rng.choice(["grid", "tandem", "planar"])
        hi = {"grid": 256, "tandem": 256, "planar": 448}[chain]
        nx = _log(rng, 32, hi)
        ny = nx if chain == "tandem" else _log(rng, 32, hi)
        return {"kind": kind, "chain": chain, "nx": nx, "ny": ny, "r": rng.choice([6, 8, 10, 16]), "fp64": fp64}
    if kind == "batch":
        return {"kind": kind, "chains": rng.randint(4, 32), "lo": 32, "hi": rng.randint(40, 96), "r": 8, "fp64": fp64}
    if kind in ("forward", "train"):
        if kind == "forward":
            return {"kind": kind, "rows": _log(rng, 500, 262144)}
        batch = rng.choice([1024, 2048, 4096])
        return {"kind": kind, "rows": _log(rng, 2000, 65536), "batch": batch}
    c = {"kind": kind, "chain": rng.choice(["grid", "tandem", "planar"])}
    hi = {"relax": 1800, "shifted": 700, "interp": 500, "galerkin": 390, "cr": 256, "vcycle": 510}[kind]
    c["nx"], c["ny"] = _log(rng, 33, hi), _log(rng, 33, hi)
    if kind == "cr":
        return c
    c["fp64"] = fp64
    if kind == "relax":
        c["r"], c["nu"] = rng.randint(4, 16), rng.choice([2, 4])
    if kind == "shifted":
        c["r"], c["nu"] = rng.randint(3, 7), 2
    if kind == "interp":
        c["r"] = rng.choice([6, 8, 10, 16])
    return c


# ------------------------------------------------------------------ chains
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 7919 + 11)


def _fixed(case):
    """The generator of what belongs to the case and not to its inputs: the graph and its splitting
    (every input of a case has the same pattern, so the same shapes)."""
    return torch.Generator(device=DEV).manual_seed(case["nx"] * 100003 + case["ny"])


def _rand(shape, g):
    return torch.rand(shape, generator=g, device=DEV, dtype=torch.float64)


def _stencil(case, g):
    """A as (ny, nx, 9) values over OFFS (0: no entry) and the stationary weights (None: not
    in closed form) or, for a queue, its rates.  A[y, x, k]: the probability from the state at
    offset OFFS[k] to (x, y)."""
    chain, nx, ny = case["chain"], case["nx"], case["ny"]
    if chain == "tandem":
        rates = torch.tensor([11.0, 10.0, 10.0], dtype=torch.float64, device=DEV) * (0.97 + 0.06 * _rand(3, g))
        mu, mx, my = (rates / rates.sum()).unbind()
        a = torch.zeros(ny, nx, 9, dtype=torch.float64, device=DEV)
        a[:, 1:, 3] = mu  # an arrival, from (x - 1, y)
        a[1:, :-1, 2] = mx  # a transfer, from (x + 1, y - 1)
        a[:-1, :, 7] = my  # a departure, from (x, y + 1)
        a[:, -1, 4] += mu
        blocked = torch.zeros(ny, nx, dtype=torch.bool, device=DEV)
        blocked[:, 0] = True
        blocked[-1, :] = True
        a[..., 4] += mx * blocked
        a[0, :, 4] += my
        return a, torch.stack([mu, mx, my])
    w = torch.zeros(ny, nx, 9, dtype=torch.float64, device=DEV)
    e = 0.5 + _rand((ny, nx - 1), g)
    w[:, 1:, 3] = e
    w[:, :-1, 5] = e
    e = 0.5 + _rand((ny - 1, nx), g)
    w[1:, :, 1] = e
    w[:-1, :, 7] = e
    if chain == "planar":  # one of the two diagonals of every cell
        rising = _rand((ny - 1, nx - 1), _fixed(case)) < 0.5
        e = 0.5 + _rand((ny - 1, nx - 1), g)
        up = torch.where(rising, e, torch.zeros_like(e))
        dn = e - up
        w[1:, 1:, 0] = up
        w[:-1, :-1, 8] = up
        w[1:, :-1, 2] = dn
        w[:-1, 1:, 6] = dn
    deg = w.sum(2)
    a = torch.zeros_like(w)
    for k, (dx, dy) in enumerate(OFFS):  # a(to, from) = w(to, from) / deg(from)
        a[..., k] = torch.where(w[..., k] > 0, w[..., k] / _shift(deg, dx, dy, 1.0), torch.zeros_like(deg))
    return a, deg


def _shift(v, dx, dy, fill):
    """v at (x + dx, y + dy), `fill` outside."""
    ny, nx = v.shape[:2]
    out = torch.full_like(v, fill)
    out[max(0, -dy):ny - max(0, dy), max(0, -dx):nx - max(0, dx)] = \
        v[max(0, dy):ny - max(0, -dy), max(0, dx):nx - max(0, -dx)]
    return out


def _csr(values, present):
    """CSR arrays (int32, int32, values) of a stencil: entries where `present`."""
    ny, nx = present.shape[:2]
    row = torch.arange(nx * ny, device=DEV).view(ny, nx, 1)
    step = torch.tensor([dx + dy * nx for dx, dy in OFFS], device=DEV)
    ptr = torch.zeros(nx * ny + 1, dtype=torch.int64, device=DEV)
    ptr[1:] = present.sum(2).view(-1).cumsum(0)
    return ptr.int(), (row + step)[present].int(), values[present].contiguous()


def _system(a):
    """B = I - A on the stencil and the entries present (the diagonal always)."""
    b = -a
    b[..., 4] += 1.0
    present = a != 0
    present[..., 4] = True
    return b, present


def _chain(case, seed):
    a, extra = _stencil(case, _gen(seed))
    return a, extra


def _vectors(b, r, ld, g):
    """Test vectors as a level of the setup has them: U[1, 2), two plain sweeps."""
    ny, nx = b.shape[:2]
    x = 1.0 + _rand((ny, nx, r), g)
    for _ in range(2):
        y = torch.zeros_like(x)
        for k, (dx, dy) in enumerate(OFFS):
            y += b[..., k:k + 1] * _shift(x, dx, dy, 0.0)
        x = x - 0.7 * y / b[..., 4:5]
    out = torch.zeros(nx * ny, ld, dtype=torch.float64, device=DEV)
    out[:, :r] = x.view(nx * ny, r)
    return out


def _split(case, present):
    """C/F split: full coarsening, or on a triangulation a maximal independent set (Luby)."""
    ny, nx = present.shape[:2]
    if case["chain"] != "planar":
        c = torch.zeros(ny, nx, dtype=torch.bool, device=DEV)
        c[::2, ::2] = True
    else:
        pri = torch.randperm(nx * ny, generator=_fixed(case), device=DEV).view(ny, nx).double() + 1.0
        c = torch.zeros(ny, nx, dtype=torch.bool, device=DEV)
        open_ = torch.ones_like(c)
        for _ in range(64):
            best = torch.zeros_like(pri)
            for k, (dx, dy) in enumerate(OFFS):
                if k != 4:
                    best = torch.maximum(best, _shift(pri * open_, dx, dy, 0.0) * present[..., k])
            new = open_ & (pri > best)
            c |= new
            near = new.clone()
            for k, (dx, dy) in enumerate(OFFS):
                near |= _shift(new, dx, dy, False) & present[..., k]
            open_ &= ~near
        assert not bool(open_.any())
    cidx = (c.view(-1).cumsum(0) - 1).int()
    return c.view(-1), torch.where(c.view(-1), cidx, torch.full_like(cidx, -1))


def _rows_of_p(c, cidx, nx, ny, g):
    """P in ELL form with two slots: a coarse point's unit row; a fine point's up to two nearest
    coarse points of the 3 x 3 block around it, with weights about one half."""
    n = nx * ny
    ci = cidx.view(ny, nx)
    big = torch.iinfo(torch.int32).max
    cand = torch.stack([_shift(torch.where(ci >= 0, ci, torch.full_like(ci, big)), dx, dy, big)
                        for dx, dy in (OFFS[k] for k in (1, 3, 5, 7, 0, 2, 6, 8))], 2).view(n, 8)
    order = torch.argsort((cand == big).int(), dim=1, stable=True)[:, :2]
    pcol = cand.gather(1, order).sort(1).values
    pcnt = (pcol != big).sum(1).int()
    pval = 0.3 + 0.4 * _rand((n, 2), g)
    pval = torch.where(pcnt.view(n, 1) == 1, torch.ones_like(pval), pval)
    unit = torch.tensor([1.0, 0.0], dtype=torch.float64, device=DEV)
    pcol = torch.where(c.view(n, 1), torch.stack([cidx, torch.full_like(cidx, big)], 1), pcol)
    pval = torch.where(c.view(n, 1), unit, pval)
    pcnt = torch.where(c, torch.ones_like(pcnt), pcnt)
    pval = torch.where(pcol == big, torch.zeros_like(pval), pval)
    return torch.where(pcol == big, torch.full_like(pcol, -1), pcol), pval, pcnt


def _triple(b, pcol, pval, pcnt, nc, t=None):
    """Q B P (and Q T P on the same pattern) in 64 bits, Q averaging: CSR arrays."""
    ptr, col, val = b
    n = ptr.numel() - 1
    row = torch.repeat_interleave(torch.arange(n, device=DEV), (ptr[1:] - ptr[:-1]).long())
    col = col.long()
    keys, vals, tvals = [], [], []
    q = 1.0 / pcnt.double()
    for s in range(2):
        for u in range(2):
            i, j = pcol[row, s].long(), pcol[col, u].long()
            ok = (i >= 0) & (j >= 0)
            keys.append((i * nc + j)[ok])
            vals.append((q[row] * val.double() * pval[col, u].double())[ok])
            if t is not None:
                tvals.append((q[row] * t.double() * pval[col, u].double())[ok])
    key, order = torch.cat(keys).sort(stable=True)
    uniq, count = torch.unique_consecutive(key, return_counts=True)
    out = [torch.segment_reduce(torch.cat(v)[order], "sum", lengths=count) for v in (vals, tvals) if v]
    cptr = torch.zeros(nc + 1, dtype=torch.int64, device=DEV)
    cptr[1:] = torch.bincount(uniq // nc, minlength=nc).cumsum(0)
    return cptr.int(), (uniq % nc).int(), out


def _hierarchy(case, seed):
    """Levels of (B in CSR, P in ELL) by full coarsening down to at most 64 states, and B_L^+."""
    g = _gen(seed)
    a, _ = _stencil(case, g)
    b, present = _system(a)
    ptr, col, val = _csr(b, present)
    nx, ny = case["nx"], case["ny"]
    levels = []
    while nx * ny > 64:
        c = torch.zeros(ny, nx, dtype=torch.bool, device=DEV)
        c[::2, ::2] = True
        c = c.view(-1)
        cidx = torch.where(c, c.cumsum(0) - 1, torch.full_like(c, -1, dtype=torch.int64)).int()
        p = _rows_of_p(c, cidx, nx, ny, g)
        levels.append(((ptr, col, val), p))
        nx, ny = (nx + 1) // 2, (ny + 1) // 2
        ptr, col, (val,) = _triple((ptr, col, val), *p, nx * ny)
    levels.append(((ptr, col, val), None))
    n = nx * ny
    dense = np.zeros((n, n))
    row = np.repeat(np.arange(n), np.diff(ptr.cpu().numpy()))
    dense[row, col.cpu().numpy()] = val.cpu().numpy()
    u, s, vt = np.linalg.svd(dense)
    return levels, (vt[:-1].T / s[:-1]) @ u[:, :-1].T


def _network(case, seed):
    """Features (valid flags in front of each slot), targets on the valid slots, parameters."""
    g = _gen(seed)
    rows = case["rows"]
    count = torch.randint(2, SLOTS + 1, (rows, 1), generator=g, device=DEV)
    valid = torch.arange(SLOTS, device=DEV) < count
    slot = torch.empty(rows, SLOTS, 6, device=DEV).normal_(0.0, 0.5, generator=g)
    slot[..., 0] = 1.0
    feat = torch.zeros(rows, FEATURES, device=DEV)
    feat[:, :6 * SLOTS] = (slot * valid.unsqueeze(2)).view(rows, -1)
    feat[:, 6 * SLOTS] = count.view(-1) / SLOTS
    feat[:, 6 * SLOTS + 1] = 1.0
    target = torch.empty(rows, SLOTS, device=DEV).normal_(0.0, 0.4, generator=g) * valid
    parts = []
    for o, i in ((HIDDEN, FEATURES), (HIDDEN, HIDDEN), (SLOTS, HIDDEN)):
        parts += [(2 * torch.rand(o * i, generator=g, device=DEV) - 1) * (6.0 / i) ** 0.5,
                  0.02 * torch.rand(o, generator=g, device=DEV)]
    return feat, target, torch.cat(parts)


# ------------------------------------------------------------------ prepare and run
def _solver_options(case):
    o = {"precision": "fp64" if case["fp64"] else "mixed"}
    if case.get("chain") == "planar":
        return {**o, "coarsen": "cr"}, 1e-13
    return {**o, "grid": (case["nx"], case["ny"])}, 1e-12


def _batch_chains(case, seed):
    g = torch.Generator().manual_seed(case["chains"] * 1009 + case["hi"])
    sides = torch.randint(case["lo"], case["hi"] + 1, (case["chains"], 2), generator=g).tolist()
    gd = _gen(seed)
    return [(nx, ny, *_stencil({"chain": "grid", "nx": nx, "ny": ny}, gd)) for nx, ny in sides]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "solve":
        a, _ = _chain(case, seed)
        o, tol = _solver_options(case)
        return {"case": case, "A": _csr(a, a != 0), "opts": o, "tol": tol}
    if kind == "batch":
        chains = _batch_chains(case, seed)
        p = "fp64" if case["fp64"] else "mixed"
        return {"case": case, "chains": [_csr(a, a != 0) for _, _, a, _ in chains],
                "opts": [{"precision": p, "grid": (nx, ny)} for nx, ny, _, _ in chains]}
    if kind in ("forward", "train"):
        feat, target, params = _network(case, seed)
        model = bamg.Model(0)
        model.set(params.cpu().numpy())
        return {"case": case, "model": model, "feat": feat, "target": target}
    dt = torch.float64 if case.get("fp64", True) else torch.float32
    if kind == "vcycle":
        levels, pinv = _hierarchy(case, seed)
        lv = []
        for (ptr, col, val), p in levels:
            d = {"B": (ptr.cpu().numpy(), col.cpu().numpy(), val.cpu().numpy())}
            if p is not None:
                pcol, pval, pcnt = p
                pptr = torch.zeros(pcnt.numel() + 1, dtype=torch.int32, device=DEV)
                pptr[1:] = pcnt.cumsum(0)
                d["P"] = (pptr.cpu().numpy(), pcol[pcol >= 0].cpu().numpy(), pval[pcol >= 0].cpu().numpy())
            lv.append(d)
        n = lv[0]["B"][0].size - 1
        solver = bamg.import_hierarchy(lv, pinv, np.ones(n), precision="fp64" if case["fp64"] else "mixed")
        v = _rand(n, _gen(seed + 1)) - 0.5
        return {"case": case, "solver": solver, "v": v - v.mean()}
    g = _gen(seed)
    a, _ = _stencil(case, g)
    b, present = _system(a)
    ptr, col, val = _csr(b, present)
    st = {"case": case, "B": (ptr, col, val.to(dt))}
    if kind == "cr":
        return {**st, "seed": int(seed) % 1000}
    w = 2 if case["fp64"] else 4
    if kind in ("relax", "shifted"):
        ld = -(-case["r"] // w) * w
        st["X"] = _vectors(b, case["r"], ld, g).to(dt)
        if kind == "shifted":
            t = torch.where(present, 0.05 * _rand(b.shape, g), torch.zeros_like(b))
            t[..., 4] += 0.6
            st["T"] = t[present].to(dt).contiguous()
            st["lam"] = 0.02 * _rand(case["r"], g).sort().values
            st["lam"][0] = 0.0
        return st
    c, cidx = _split(case, present)
    st["nc"] = int(c.sum())
    if kind == "interp":
        ld = -(-case["r"] // w) * w
        x = _vectors(b, case["r"], ld, g)
        st["X"] = (x / torch.linalg.vector_norm(x, dim=0).clamp_min(1e-30)).to(dt)
        st["w"] = torch.cat([_rand(case["r"] - 1, g), torch.ones(1, dtype=torch.float64, device=DEV)])
        st["cf"], st["cidx"] = c.to(torch.uint8), cidx.contiguous()
        return st
    pcol, pval, pcnt = _rows_of_p(c, cidx, case["nx"], case["ny"], g)
    t = torch.where(present, 0.05 * _rand(b.shape, g), torch.zeros_like(b))
    t[..., 4] += 0.6
    st["T"] = t[present].to(dt).contiguous()
    st["P"] = (pcol.contiguous(), pval.to(dt).contiguous(), pcnt.contiguous())
    return st


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "solve":
        solver = bamg.Solver(*s["A"], r=case["r"], levels=20, **s["opts"])
        x, _ = solver.solve(s["tol"])
        solver.close()
        return x
    if kind == "batch":
        return bamg.solve_batch(s["chains"], case["r"], 20, 1e-12, opts=s["opts"])[0]
    if kind == "relax":
        return bamg.relax(s["B"], s["X"], case["r"], 0, 0.7, case["nu"])
    if kind == "shifted":
        return bamg.relax(s["B"], s["X"], case["r"], 0, 0.7, case["nu"], T_val=s["T"], lam=s["lam"])
    if kind == "interp":
        return bamg.interp_ls(s["B"], s["cf"], s["cidx"], s["X"], case["r"], s["w"], ridge=1e-4)
    if kind == "galerkin":
        return bamg.galerkin(s["B"], s["T"], s["nc"], *s["P"], 2)
    if kind == "cr":
        return bamg.coarsen_cr(s["B"], 0, s["seed"])
    if kind == "vcycle":
        return s["solver"].vcycle(s["v"])
    if kind == "forward":
        return s["model"].forward(s["feat"])
    s["model"].train(s["feat"], s["target"], 1, case["batch"], 1e-3)
    return s["model"].get()


# ------------------------------------------------------------------ work
def work(case):
    """Each input read once, each output written once; the operations of the definition."""
    kind = case["kind"]
    macs = HIDDEN * FEATURES + HIDDEN * HIDDEN + SLOTS * HIDDEN
    if kind == "forward":
        return {"bytes": 4.0 * case["rows"] * (FEATURES + SLOTS), "flops": 2.0 * macs * case["rows"]}
    if kind == "train":
        return {"bytes": 4.0 * case["rows"] * (FEATURES + SLOTS),
                "flops": 2.0 * case["rows"] * (3 * macs - HIDDEN * FEATURES)}
    if kind == "batch":
        n = case["chains"] * ((case["lo"] + case["hi"]) / 2) ** 2
        return {"bytes": n * (4 * 12 + 4 + 8), "flops": n * 4 * 2 * 100}
    n = float(case["nx"] * case["ny"])
    deg = {"grid": 4.0, "tandem": 3.0, "planar": 6.0}[case["chain"]]
    nnz = n * (deg + 1)
    v = 8.0 if case.get("fp64", True) else 4.0
    if kind == "solve":  # A in, x out; some twenty cycles, each about a hundred products a state
        return {"bytes": n * deg * 12 + 4 * n + 8 * n, "flops": n * 2 * 20 * 100}
    if kind == "relax":
        return {"bytes": nnz * (4 + v) + 4 * n + 2 * v * n * case["r"], "flops": case["nu"] * 2 * nnz * case["r"]}
    if kind == "shifted":
        return {"bytes": nnz * (4 + 2 * v) + 4 * n + 2 * v * n * case["r"], "flops": case["nu"] * 4 * nnz * case["r"]}
    if kind == "interp":
        return {"bytes": nnz * 4 + 9 * n + v * n * case["r"] + n * (2 * (4 + v) + 4),
                "flops": n * 16 * case["r"] * 2 * 6}
    if kind == "galerkin":
        return {"bytes": nnz * (4 + 2 * v) + 4 * n + n * (2 * (4 + v) + 4) + nnz / 3 * (4 + 2 * v),
                "flops": nnz * 3 * 6}
    if kind == "cr":
        return {"bytes": nnz * 12 + 9 * n, "flops": nnz * 2 * 8}
    return {"bytes": 4.0 / 3 * (nnz * (4 + v) + n * (4 * v + 12)) + 16 * n, "flops": 4.0 / 3 * 2 * nnz * 6}


# ------------------------------------------------------------------ the same in 64 bits
def _tandem_stationary(nx, ny, rates):
    """Block elimination over the second queue's length (S_j x_j = L x_{j-1})."""
    mu, mx, my = rates.tolist()
    lo = torch.diag(torch.full((nx - 1,), mx, dtype=torch.float64, device=DEV), 1)
    gs, gain = [None] * ny, None
    for j in range(ny - 1, -1, -1):
        d = torch.ones(nx, dtype=torch.float64, device=DEV)
        d[-1] -= mu
        if j == ny - 1:
            d -= mx
        else:
            d[0] -= mx
        if j == 0:
            d -= my
        s = torch.diag(d) - torch.diag(torch.full((nx - 1,), mu, dtype=torch.float64, device=DEV), -1)
        if gain is not None:
            s = s - my * gain
        if j > 0:
            gain = torch.linalg.solve(s, lo)
            gs[j] = gain
    x = torch.linalg.svd(s.cpu())[2][-1].to(DEV)
    out = [x / x.sum()]
    for j in range(1, ny):
        out.append(gs[j] @ out[-1])
    x = torch.stack(out)
    return (x / x.sum()).view(-1)


def _mv(b, x):
    ptr, col, val = b
    return torch.segment_reduce(val.double() * x[col.long()], "sum", lengths=(ptr[1:] - ptr[:-1]).long())


def _sweeps(s, case):
    ptr, col, val = s["B"]
    n = ptr.numel() - 1
    row = torch.repeat_interleave(torch.arange(n, device=DEV), (ptr[1:] - ptr[:-1]).long())
    col = col.long()
    diag = torch.zeros(n, dtype=torch.float64, device=DEV)
    at = row == col
    diag[row[at]] = val[at].double()
    x = s["X"].double().clone()
    count = (ptr[1:] - ptr[:-1]).long()
    tval = s["T"].double() if "T" in s else None
    for c in range(case["r"]):
        d = diag
        v = val.double()
        if tval is not None:
            v = v - s["lam"][c] * tval
            d = diag.clone()
            d[row[at]] -= s["lam"][c] * tval[at]
        y = x[:, c].contiguous()
        for _ in range(case["nu"]):
            y = y - 0.7 * torch.segment_reduce(v * y[col], "sum", lengths=count) / d
        x[:, c] = y
    return x


def _cycle(levels, pinv, v, l=0):
    b, p = levels[l]
    if p is None:
        return pinv @ v
    ptr, col, val = b
    n = ptr.numel() - 1
    row = torch.repeat_interleave(torch.arange(n, device=DEV), (ptr[1:] - ptr[:-1]).long())
    at = row == col.long()
    w = 0.7 / val[at]
    pcol, pval, pcnt = p
    nc = levels[l + 1][0][0].numel() - 1
    x = w * v
    x = x + w * (v - _mv(b, x))
    r = (v - _mv(b, x)) / pcnt.double()
    rc = torch.zeros(nc, dtype=torch.float64, device=DEV)
    for s in range(2):
        ok = pcol[:, s] >= 0
        rc.index_add_(0, pcol[ok, s].long(), r[ok])
    e = _cycle(levels, pinv, rc, l + 1)
    x = x + (pval * torch.where(pcol >= 0, e[pcol.clamp_min(0).long()], torch.zeros_like(pval))).sum(1)
    for _ in range(2):
        x = x + w * (v - _mv(b, x))
    return x


def _layers(params):
    out, at = [], 0
    for o, i in ((HIDDEN, FEATURES), (HIDDEN, HIDDEN), (SLOTS, HIDDEN)):
        out += [params[at:at + o * i].view(o, i), params[at + o * i:at + o * i + o]]
        at += o * i + o
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        _, extra = _chain(case, seed)
        if case["chain"] == "tandem":
            return _tandem_stationary(case["nx"], case["ny"], extra)
        return (extra / extra.sum()).view(-1)
    if kind == "batch":
        return [(deg / deg.sum()).view(-1) for _, _, _, deg in _batch_chains(case, seed)]
    if kind in ("relax", "shifted"):
        return _sweeps(prepare(case, seed), case)
    if kind == "galerkin":
        s = prepare(case, seed)
        _, _, (bv, tv) = _triple(s["B"], *s["P"], s["nc"], s["T"])
        return None, None, bv, tv
    if kind == "vcycle":
        levels, pinv = _hierarchy(case, seed)
        v = _rand(case["nx"] * case["ny"], _gen(seed + 1)) - 0.5
        return _cycle(levels, torch.from_numpy(np.ascontiguousarray(pinv)).to(DEV), v - v.mean())
    if kind == "forward":
        feat, _, params = _network(case, seed)
        w1, b1, w2, b2, w3, b3 = _layers(params.double())
        h = (feat.double() @ w1.T + b1).relu()
        return (h @ w2.T + b2).relu() @ w3.T + b3
    if kind == "train":
        feat, target, params = _network(case, seed)
        p = params.double()
        m, v = torch.zeros_like(p), torch.zeros_like(p)
        for t, r0 in enumerate(range(0, case["rows"], case["batch"]), 1):
            f, y = feat[r0:r0 + case["batch"]].double(), target[r0:r0 + case["batch"]].double()
            p.requires_grad_(True)
            w1, b1, w2, b2, w3, b3 = _layers(p)
            h = (f @ w1.T + b1).relu()
            d = ((h @ w2.T + b2).relu() @ w3.T + b3 - y) * (f[:, 0:6 * SLOTS:6] > 0)
            loss = d.square().sum() / f.shape[0]
            (g,) = torch.autograd.grad(loss, p)
            p = p.detach()
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            p = p - 1e-3 * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)
        return p.cpu().numpy()
    return None  # cr: whole numbers; interp: the greedy choice in 32 bits has near-ties
