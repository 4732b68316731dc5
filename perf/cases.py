"""Timed cases of the matrix power kernel: what users of this package have it compute.

A case is one call (or, for `setup`, one sequence of calls) of the public Python API with the
planner's own choices; only the options that a user sets by meaning are set: order, powers,
right-hand sides, value type, accumulator, and the block shape of the serving plans.  Matrices
are the repository's workloads (Laplacians, 27-point stencils, banded random graphs, the XXZ
spin chain), built on the GPU from the case and the seed.

`listed()` names the cases, `draw()` gives others of the same ranges, `prepare()` builds what a
program holds before the call, `run()` is one pass, `work()` its algorithmic bytes and flops,
`exact()` the same outputs from plain torch in binary64.
"""
import math

import numpy as np
import torch

import paper_2405_12525_gb300 as mpk
from paper_2405_12525_gb300 import serving

DTYPE = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}
VALUE_BYTES = {"f64": 8, "f32": 4, "bf16": 2}
ORDER = {"original": mpk.ORDER_ORIGINAL, "plan": mpk.ORDER_PLAN}


def listed():
    return [
        # the oracle-sized configuration, default options: an interactive call where launches count
        {"name": "small_2d", "kind": "apply", "matrix": "lap2d", "nx": 64, "ny": 64, "values": "f64",
         "order": "original", "p": 4, "nrhs": 1, "accum": "f64"},
        # a matrix that stays in L2 (the ragged grid of the level tests), default options
        {"name": "mid_3d", "kind": "apply", "matrix": "lap3d", "nx": 48, "ny": 40, "nz": 33, "values": "f64",
         "order": "original", "p": 8, "nrhs": 1, "accum": "f64"},
        # the headline benchmark: 256^3, p = 8, vectors kept in the plan's numbering
        {"name": "headline_3d", "kind": "apply", "matrix": "lap3d", "nx": 256, "ny": 256, "nz": 256, "values": "f64",
         "order": "plan", "p": 8, "nrhs": 1, "accum": "f64"},
        # the same matrix with default options: vectors in the matrix's own numbering
        {"name": "headline_original", "kind": "apply", "matrix": "lap3d", "nx": 256, "ny": 256, "nz": 256,
         "values": "f64", "order": "original", "p": 8, "nrhs": 1, "accum": "f64"},
        # the precision option of the benchmark: bfloat16 values, binary32 row sums
        {"name": "headline_acc32", "kind": "apply", "matrix": "lap3d", "nx": 256, "ny": 256, "nz": 256,
         "values": "bf16", "order": "plan", "p": 8, "nrhs": 1, "accum": "f32"},
        # a 27-point stencil of the batch configuration with a block of 8 right-hand sides
        {"name": "stencil27_rhs8", "kind": "apply", "matrix": "st27", "nx": 100, "ny": 100, "nz": 100,
         "values": "bf16", "order": "original", "p": 8, "nrhs": 8, "accum": "f64"},
        # a banded random graph of the batch configuration (odd size) with 4 right-hand sides
        {"name": "band_rhs4", "kind": "apply", "matrix": "band", "n": 300007, "values": "f32", "order": "original",
         "p": 6, "nrhs": 4, "accum": "f64"},
        # Chebyshev time propagation of the spin chain: complex state as 2 columns, degree 64
        {"name": "xxz_propagation", "kind": "cheb", "matrix": "xxz", "L": 24, "values": "f64", "order": "plan",
         "degree": 64, "p": 8, "nrhs": 2, "complex": True, "shape": 0},
        # a served Chebyshev request: the serving plans' block shape, the matrix's own numbering
        {"name": "served_filter", "kind": "cheb", "matrix": "band", "n": 100003, "values": "f32", "order": "original",
         "degree": 48, "p": 8, "nrhs": 4, "complex": False, "shape": serving.SERVING_SHAPE},
        # several uneven matrices in one launch
        {"name": "batch_stencils", "kind": "batch", "matrix": "st27", "sides": "22,29,35,41,47,53,58,64",
         "powers": "12,9,7,4,10,6,8,5", "values": "bf16", "order": "original", "nrhs": 4},
        # a matrix used once: levels, plan and one apply
        {"name": "setup_3d", "kind": "setup", "matrix": "lap3d", "nx": 131, "ny": 127, "nz": 113, "values": "f64",
         "order": "original", "p": 8, "nrhs": 1, "accum": "f64"},
        # vectors in host memory: X in, all powers out
        {"name": "host_buffers", "kind": "host", "matrix": "lap3d", "nx": 128, "ny": 128, "nz": 128, "values": "f64",
         "order": "plan", "p": 8, "nrhs": 1, "accum": "f64"},
    ]


# ----------------------------------------------------------------------------- drawn cases
def _size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(rng, n):
    """Three ragged sides with about n points."""
    s = n ** (1.0 / 3.0)
    nx = max(3, int(round(s * rng.uniform(0.6, 1.6))))
    ny = max(3, int(round(s * rng.uniform(0.6, 1.6))))
    return {"nx": nx, "ny": ny, "nz": max(3, int(round(n / (nx * ny))))}


def _powers(rng, entries, nrhs, lo=2, hi=16):
    """A number of powers that keeps the case within the headline's entries x powers."""
    return max(1, min(rng.randint(lo, hi), int(9.3e8 // max(1, entries * nrhs))))


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "apply", "apply", "cheb", "cheb", "batch", "setup", "host"])
    order = rng.choice(["original", "original", "plan"])
    if kind == "apply":
        matrix = rng.choice(["lap2d", "lap3d", "lap3d", "st27", "band"])
        if matrix == "lap2d":
            n = _size(rng, 2e3, 4e6)
            nx = max(3, int(round(n ** 0.5 * rng.uniform(0.5, 2.0))))
            c = {"matrix": matrix, "nx": nx, "ny": max(3, n // nx), "values": "f64", "nrhs": rng.choice([1, 1, 2])}
            width = 5
        elif matrix == "lap3d":
            n = _size(rng, 8e3, 1.6e7)
            c = {"matrix": matrix, **_grid(rng, n), "values": rng.choice(["f64", "f64", "f32", "bf16"]),
                 "nrhs": rng.choice([1, 1, 1, 2, 4])}
            width = 7
        elif matrix == "st27":
            n = _size(rng, 1e4, 2e6)
            c = {"matrix": matrix, **_grid(rng, n), "values": "bf16", "nrhs": rng.choice([1, 4, 8, 16])}
            width = 27
        else:
            n = _size(rng, 1e4, 1e6)
            c = {"matrix": matrix, "n": n, "values": rng.choice(["f32", "f64"]), "nrhs": rng.choice([1, 4, 8, 16])}
            width = 15
        accum = "f32" if c["values"] != "f64" and c["nrhs"] == 1 and rng.random() < 0.5 else "f64"
        return {"kind": kind, **c, "order": order, "p": _powers(rng, width * n, c["nrhs"]), "accum": accum}
    if kind == "cheb":
        if rng.random() < 0.5:
            return {"kind": kind, "matrix": "xxz", "L": rng.choice([14, 16, 18, 20, 22]), "values": "f64",
                    "order": "plan", "degree": rng.randint(16, 100), "p": 8, "nrhs": 2, "complex": True, "shape": 0}
        n, nrhs = _size(rng, 1e4, 4e5), rng.choice([1, 2, 4, 8])
        m = {"matrix": "band", "n": n} if rng.random() < 0.5 else {"matrix": "st27", **_grid(rng, n)}
        return {"kind": kind, **m, "values": "f32" if m["matrix"] == "band" else "bf16", "order": "original",
                "degree": min(rng.randint(16, 128), max(16, int(2e9 // (27 * n * nrhs)))), "p": 8, "nrhs": nrhs,
                "complex": False, "shape": serving.SERVING_SHAPE}
    if kind == "batch":
        sides = [_size(rng, 18, 70) for _ in range(rng.randint(3, 10))]
        return {"kind": kind, "matrix": "st27", "sides": ",".join(map(str, sides)),
                "powers": ",".join(str(rng.randint(4, 12)) for _ in sides), "values": "bf16", "order": order,
                "nrhs": rng.choice([1, 4])}
    if kind == "setup":
        n = _size(rng, 2e4, 4e6)
        return {"kind": kind, "matrix": "lap3d", **_grid(rng, n), "values": "f64", "order": "original",
                "p": rng.randint(4, 10), "nrhs": 1, "accum": "f64"}
    n = _size(rng, 3e4, 4e6)
    return {"kind": kind, "matrix": "lap3d", **_grid(rng, n), "values": "f64", "order": "plan",
            "p": rng.randint(2, 10), "nrhs": 1, "accum": "f64"}


# ----------------------------------------------------------------------------- matrices
def _stencil(nx, ny, nz, offsets, diagonal, dtype):
    """Constant-coefficient stencil on a lexicographic grid with open boundaries (off-diagonal
    entries -1), columns ascending in every row: (row_ptr, col, val) on the GPU."""
    offsets = sorted(offsets, key=lambda o: o[0] + nx * (o[1] + ny * o[2]))
    n = nx * ny * nz
    i = torch.arange(n, dtype=torch.int32, device="cuda")
    x, y, z = i % nx, (i // nx) % ny, i // (nx * ny)
    inside = torch.empty((n, len(offsets)), dtype=torch.bool, device="cuda")
    for q, (dx, dy, dz) in enumerate(offsets):
        inside[:, q] = ((x + dx >= 0) & (x + dx < nx) & (y + dy >= 0) & (y + dy < ny) & (z + dz >= 0) & (z + dz < nz))
    shift = torch.tensor([dx + nx * (dy + ny * dz) for dx, dy, dz in offsets], dtype=torch.int32, device="cuda")
    value = torch.tensor([diagonal if o == (0, 0, 0) else -1.0 for o in offsets], dtype=dtype, device="cuda")
    row_ptr = torch.zeros(n + 1, dtype=torch.int32, device="cuda")
    row_ptr[1:] = torch.cumsum(inside.sum(1, dtype=torch.int32), 0)
    col = (i[:, None] + shift[None, :])[inside]
    val = value[None, :].expand(n, len(offsets))[inside]
    return row_ptr, col, val


def _from_keys(n, keys, vals, dtype):
    """Entries with key row * n + column (distinct) as CSR."""
    keys, at = torch.sort(keys)
    row_ptr = torch.searchsorted(keys, torch.arange(n + 1, dtype=torch.int64, device="cuda") * n).to(torch.int32)
    return row_ptr, (keys % n).to(torch.int32), vals[at].to(dtype)


def _band(n, dtype, g):
    """Random symmetric banded graph: 7 upper entries a row within n / 100 of the diagonal
    (duplicates once), mirrored, and the diagonal; values N(0, 1)."""
    width = max(1, math.ceil(n * 0.01))
    i = torch.arange(n, dtype=torch.int64, device="cuda")
    rows = i.repeat_interleave(7)
    cols = rows + 1 + torch.randint(0, width, (7 * n,), generator=g, device="cuda")
    keys = torch.unique((rows * n + cols)[cols < n])
    v = torch.randn(keys.numel(), generator=g, dtype=torch.float64, device="cuda")
    d = torch.randn(n, generator=g, dtype=torch.float64, device="cuda")
    return _from_keys(n, torch.cat([keys, (keys % n) * n + keys // n, i * n + i]), torch.cat([v, v, d]), dtype)


def _xxz(L, dtype, g):
    """Periodic spin-1/2 XXZ chain (Jxy = 1, Jz = 0.5, fields uniform in [-1, 1)), Sz = 0 sector."""
    states = torch.arange(1 << L, dtype=torch.int32, device="cuda")
    ones = sum((states >> q) & 1 for q in range(L))
    basis = states[ones == L // 2]
    n = basis.numel()
    index = torch.zeros(1 << L, dtype=torch.int32, device="cuda")
    index[basis.long()] = torch.arange(n, dtype=torch.int32, device="cuda")
    h = 2.0 * torch.rand(L, generator=g, dtype=torch.float64, device="cuda") - 1.0
    i = torch.arange(n, dtype=torch.int64, device="cuda")
    diag = torch.zeros(n, dtype=torch.float64, device="cuda")
    keys = [i * n + i]
    for q in range(L):
        r = (q + 1) % L
        a, b = (basis >> q) & 1, (basis >> r) & 1
        sa, sb = a.double() - 0.5, b.double() - 0.5
        diag += 0.5 * sa * sb + h[q] * sa
        flip = a != b
        to = index[(basis[flip] ^ ((1 << q) | (1 << r))).long()]
        keys.append(i[flip] * n + to)
    off = torch.full((sum(k.numel() for k in keys[1:]),), 0.5, dtype=torch.float64, device="cuda")
    return _from_keys(n, torch.cat(keys), torch.cat([diag, off]), dtype)


_OFF5 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0)]
_OFF7 = _OFF5 + [(0, 0, 1), (0, 0, -1)]
_OFF27 = [(dx, dy, dz) for dz in (-1, 0, 1) for dy in (-1, 0, 1) for dx in (-1, 0, 1)]


def _matrix(case, g):
    dtype = DTYPE[case["values"]]
    if case["matrix"] == "lap2d":
        return _stencil(case["nx"], case["ny"], 1, _OFF5, 4.0, dtype)
    if case["matrix"] == "lap3d":
        return _stencil(case["nx"], case["ny"], case["nz"], _OFF7, 6.0, dtype)
    if case["matrix"] == "st27":
        return _stencil(case["nx"], case["ny"], case["nz"], _OFF27, 26.0, dtype)
    if case["matrix"] == "band":
        return _band(case["n"], dtype, g)
    return _xxz(case["L"], dtype, g)


def _vector(n, nrhs, g):
    return 2.0 * torch.rand((n, nrhs), generator=g, dtype=torch.float64, device="cuda") - 1.0


def _batch(case):
    return [{"matrix": case["matrix"], "nx": int(s), "ny": int(s), "nz": int(s), "values": case["values"],
             "p": int(p), "nrhs": case["nrhs"]} for s, p in zip(case["sides"].split(","), case["powers"].split(","))]


def _spectrum(row_ptr, col, val):
    """(scale, shift) that map the Gershgorin enclosure of the spectrum into [-1, 1]."""
    n = row_ptr.numel() - 1
    rows = torch.repeat_interleave(torch.arange(n, device="cuda"), row_ptr.diff().long())
    v = val.double()
    d = torch.zeros(n, dtype=torch.float64, device="cuda")
    on = rows == col
    d[rows[on]] = v[on]
    at = torch.cat([torch.zeros(1, dtype=torch.float64, device="cuda"), torch.cumsum(v.abs(), 0)])
    r = at[row_ptr[1:].long()] - at[row_ptr[:-1].long()] - d.abs()
    lo, hi = float((d - r).min()), float((d + r).max())
    return 1.01 * (hi - lo) / 2, (hi + lo) / 2


def _coefficients(case):
    """Degree + 1 coefficients: a time step (Bessel functions, the largest that the degree
    resolves) for complex states, else a Jackson-damped step filter."""
    d = case["degree"]
    if case["complex"]:
        z, m = 0.5 * d, 1024
        bessel = np.fft.fft(np.exp(1j * z * np.sin(2 * np.pi * np.arange(m) / m))).real[: d + 1] / m
        c = np.where(np.arange(d + 1) == 0, 1.0, 2.0) * (-1j) ** np.arange(d + 1) * bessel
        return np.ascontiguousarray(c.real), np.ascontiguousarray(c.imag)
    k, q = np.arange(d + 1), np.pi / (d + 2)
    damp = ((d - k + 2) * np.cos(q * k) + np.sin(q * k) / np.tan(q)) / (d + 2)
    step = np.where(k == 0, 0.5, 2.0 * np.sin(k * np.pi / 2) / (np.pi * np.maximum(k, 1)))
    return damp * step, None


# ----------------------------------------------------------------------------- one case
def _inputs(case, seed):
    """The matrices and vectors of a case: [(row_ptr, col, val), X] per matrix."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    out = []
    for c in (_batch(case) if case["kind"] == "batch" else [case]):
        A = _matrix(c, g)
        out.append((A, _vector(A[0].numel() - 1, c["nrhs"], g)))
    return out


def prepare(case, seed):
    state = {"case": case}
    inputs = _inputs(case, seed)
    mats = [mpk.CsrMatrix(*A, is_symmetric=True) for A, _ in inputs]
    if case["kind"] == "batch":
        state["plan"] = mpk.batch_plan(mats, [c["p"] for c in _batch(case)], nrhs=case["nrhs"],
                                       order=ORDER[case["order"]])
        state["X"] = [X for _, X in inputs]
        return state
    A, X = mats[0], inputs[0][1]
    state["X"] = X
    if case["kind"] == "setup":
        state["A"] = A
        return state
    levels = mpk.build_levels(A, root=0)
    if case["kind"] == "cheb":
        state["scale"], state["shift"] = _spectrum(*inputs[0][0])
        state["c"] = _coefficients(case)
        state["plan"] = mpk.plan(A, levels, p_max=case["p"], nrhs=case["nrhs"], order=ORDER[case["order"]],
                                 shape=case["shape"])
        return state
    state["plan"] = mpk.plan(A, levels, p_max=case["p"], nrhs=case["nrhs"], order=ORDER[case["order"]],
                             accum=mpk.MPK_F32 if case["accum"] == "f32" else mpk.MPK_F64)
    if case["kind"] == "host":
        state["X"] = X.cpu().pin_memory()
        state["Y"] = torch.empty((case["p"] + 1, A.n, case["nrhs"]), dtype=torch.float64).pin_memory()
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "apply":
        return state["plan"].apply(state["X"], case["p"])
    if case["kind"] == "cheb":
        re, im = state["c"]
        return state["plan"].cheb_filter(state["X"], case["degree"], re, im, scale=state["scale"],
                                         shift=state["shift"])
    if case["kind"] == "batch":
        return state["plan"].apply(state["X"])
    if case["kind"] == "host":
        return state["plan"].apply_host(state["X"], case["p"], Y=state["Y"])
    levels = mpk.build_levels(state["A"], root=0)
    plan = mpk.plan(state["A"], levels, p_max=case["p"], nrhs=case["nrhs"], order=ORDER[case["order"]])
    Y = plan.apply(state["X"], case["p"])
    return {"perm": levels.perm, "level_ptr": levels.level_ptr, "Y": Y}


def _count(c):
    """(rows, entries) of a case's matrix (the banded graph: expected entries)."""
    if c["matrix"] == "lap2d":
        nx, ny = c["nx"], c["ny"]
        return nx * ny, 5 * nx * ny - 2 * (nx + ny)
    if c["matrix"] == "lap3d":
        nx, ny, nz = c["nx"], c["ny"], c["nz"]
        return nx * ny * nz, 7 * nx * ny * nz - 2 * (nx * ny + ny * nz + nx * nz)
    if c["matrix"] == "st27":
        return (c["nx"] * c["ny"] * c["nz"], (3 * c["nx"] - 2) * (3 * c["ny"] - 2) * (3 * c["nz"] - 2))
    if c["matrix"] == "band":
        n, w = c["n"], max(1, math.ceil(c["n"] * 0.01))
        return n, int(n + 2 * (n - w / 2) * w * (1.0 - (1.0 - 1.0 / w) ** 7))
    n = math.comb(c["L"], c["L"] // 2)
    return n, n + 2 * c["L"] * math.comb(c["L"] - 2, c["L"] // 2 - 1)


def work(case):
    total = {"bytes": 0, "flops": 0}
    for c in (_batch(case) if case["kind"] == "batch" else [case]):
        n, nnz = _count(c)
        m = c["nrhs"]
        matrix = (VALUE_BYTES[c["values"]] + 4) * nnz + 4 * n
        if case["kind"] == "cheb":
            total["bytes"] += matrix + 16 * n * m
            total["flops"] += case["degree"] * m * (2 * nnz + (8 if case["complex"] else 6) * n)
        else:
            total["bytes"] += matrix + 8 * n * m * (c["p"] + 2)
            total["flops"] += 2 * nnz * m * c["p"]
    return total


def _plan_rows(row_ptr, col):
    """The rows in plan order: by BFS level from row 0 (a search that runs dry goes on from the
    smallest untouched row, one level further), then by row number."""
    n = row_ptr.numel() - 1
    one = torch.ones(col.numel(), dtype=torch.float32, device="cuda")
    graph = torch.sparse_csr_tensor(row_ptr, col, one, (n, n))
    level = torch.full((n,), -1, dtype=torch.int64, device="cuda")
    front = torch.zeros((n, 1), dtype=torch.float32, device="cuda")
    lev, left = 0, n
    while left:
        if not front.any():
            front[int((level < 0).int().argmax())] = 1.0
        now = front[:, 0] > 0
        level[now] = lev
        lev, left = lev + 1, left - int(now.sum())
        front = ((graph @ front > 0) & (level < 0)[:, None]).float()
    return torch.sort(level, stable=True).indices


def exact(case, seed):
    out = []
    for c, ((row_ptr, col, val), X) in zip(_batch(case) if case["kind"] == "batch" else [case], _inputs(case, seed)):
        n = X.shape[0]
        A = torch.sparse_csr_tensor(row_ptr, col, val.double(), (n, n))
        at = None
        if case["order"] == "plan":  # the call's vectors are in the plan's numbering
            at = _plan_rows(row_ptr, col)
            X = torch.empty_like(X).index_copy_(0, at, X)
        if case["kind"] != "cheb":
            Y = [X]
            for _ in range(c["p"]):
                Y.append(A @ Y[-1])
            out.append(torch.stack(Y if at is None else [y[at] for y in Y]))
            continue
        scale, shift = _spectrum(row_ptr, col, val)
        re, im = _coefficients(case)
        back, v = None, X
        for k in range(case["degree"] + 1):
            if k == 1:
                back, v = v, (A @ v - shift * v) / scale
            elif k > 1:
                back, v = v, 2.0 * (A @ v - shift * v) / scale - back
            term = re[k] * v
            if im is not None:  # columns are (real, imaginary) pairs
                w = v.reshape(n, -1, 2)
                term = term + im[k] * torch.stack([-w[..., 1], w[..., 0]], -1).reshape(n, -1)
            acc = term if k == 0 else acc + term
        out.append(acc if at is None else acc[at])
    if case["kind"] == "setup":
        return {"perm": None, "level_ptr": None, "Y": out[0]}
    return out if case["kind"] == "batch" else out[0]
