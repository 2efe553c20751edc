"""Cases of the selected-inversion library that stand for its use, timed
through the package's public entry points.

Two kinds of call are timed.  ``sweep``: the LU factors are resident and a
pass is ``selinv`` plus the extraction of the selected entries (the step of
``bench.py``).  ``solve``: new values arrive on the device and a pass is the
whole call, ``factor``, ``selinv`` and the extraction (a self-consistent
loop, or one step of a continuation).  ``poles`` is a solve of a batch of
complex shifts that ends in the pole expansion's two consumers, the weighted
sum of the selected inverses and the trace.  ``whole`` also copies out the selected
inverse on the whole pattern of L + U.  Nothing is tuned beforehand: the
plans are the library's own defaults.
"""
from __future__ import annotations

import functools

import numpy as np
import torch

import paper_1708_04539_gb300 as ps

FAMILIES = ("grid2d", "grids", "oneway", "upwind", "diffusion", "stencil27", "poles", "dg")


def _case(name, family, m, *, call="solve", precision="split", complex_values=False, count=1,
          dof=1, max_sn=256, whole=False):
    return {"name": name, "family": family, "m": m, "call": call, "precision": precision,
            "complex": complex_values, "count": count, "dof": dof, "max_sn": max_sn,
            "whole": whole}


def listed():
    return [
        # the smallest benchmark matrix (31^2, supernodes of at most 64): a sweep of a few
        # launches, bound by latency
        _case("grid31-sweep", "grid2d", 31, call="sweep", precision="fp64", max_sn=64),
        # an ordinary 2D problem in the library's default precision, odd side
        _case("grid127-solve", "grid2d", 127, precision="fp64"),
        # uneven 2D grids (20^2 .. 90^2) with complex shifts in one handle: the second half
        # of the pole batch
        _case("grids16-solve", "grids", 90, complex_values=True, count=16),
        # a pattern that is not structurally symmetric, with static pivoting
        _case("oneway90-solve", "oneway", 90, precision="fp64", max_sn=64),
        # a small 3D operator in the default precision
        _case("upwind24-solve", "upwind", 24, precision="fp64"),
        # the 40^3 benchmark matrix: the sweep alone and the whole call
        _case("upwind40-sweep", "upwind", 40, call="sweep", whole=True),
        _case("upwind40-solve", "upwind", 40),
        # symmetric values: the symmetric sweep and the lower-triangle factorisation
        _case("diffusion25-solve", "diffusion", 25, whole=True),
        # the complex 27-point operator at half the benchmark's side
        _case("stencil30-solve", "stencil27", 30, complex_values=True),
        # a pole expansion: 20 complex shifts of one 3D pattern, density and trace
        _case("poles20-solve", "poles", 16, call="poles", complex_values=True, count=20),
        # the block-sparse DG operator of the headline benchmark at sides whose states fit
        # the card several times: the whole call and the sweep alone
        _case("dg8-solve", "dg", 8, dof=64),
        _case("dg10-sweep", "dg", 10, call="sweep", dof=64),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    family = rng.choice(FAMILIES)
    call = rng.choice(("sweep", "solve"))
    precision = rng.choice(("fp64", "split"))
    if family == "grid2d":
        c = _case("", family, _log_int(rng, 15, 200), call=call, precision=precision,
                  complex_values=rng.random() < 0.3, max_sn=rng.choice((64, 256)))
    elif family == "grids":
        c = _case("", family, rng.randint(60, 110), call=call, precision=precision,
                  complex_values=rng.random() < 0.7, count=rng.randint(4, 32))
    elif family == "oneway":
        c = _case("", family, _log_int(rng, 24, 110), call=call, precision=precision,
                  complex_values=rng.random() < 0.3, max_sn=64)
    elif family == "upwind":
        c = _case("", family, _log_int(rng, 9, 28 if precision == "fp64" else 40), call=call,
                  precision=precision)
    elif family == "diffusion":
        c = _case("", family, _log_int(rng, 9, 28 if precision == "fp64" else 40), call=call,
                  precision=precision)
    elif family == "stencil27":
        c = _case("", family, _log_int(rng, 7, 20 if precision == "fp64" else 30), call=call,
                  precision=precision, complex_values=True)
    elif family == "poles":
        c = _case("", family, rng.randint(8, 16), call="poles", precision=precision,
                  complex_values=True, count=_log_int(rng, 2, 20))
    else:
        c = _case("", family, rng.randint(3, 4) if precision == "fp64" else rng.randint(3, 9),
                  call=call, precision=precision, dof=rng.randint(20, 64))
    del c["name"]
    c["whole"] = c["call"] != "poles" and rng.random() < 0.2
    return c


# ---------------------------------------------------------------------------
# patterns (CSC, int64) and orderings; the same for every seed
# ---------------------------------------------------------------------------
def _neighbours(dims, offsets):
    """(row, column) pairs of a stencil on a box grid, x fastest, without the diagonal."""
    n = int(np.prod(dims))
    idx = np.arange(n, dtype=np.int64)
    coords, rem = [], idx
    for d in dims:
        coords.append(rem % d)
        rem = rem // d
    rows, cols = [], []
    for off in offsets:
        ok, j, stride = np.ones(n, dtype=bool), np.zeros(n, dtype=np.int64), 1
        for x, o, d in zip(coords, off, dims):
            ok &= (x + o >= 0) & (x + o < d)
            j += (x + o) * stride
            stride *= d
        rows.append(j[ok])
        cols.append(idx[ok])
    return np.concatenate(rows), np.concatenate(cols)


def _csc(n, rows, cols):
    idx = np.arange(n, dtype=np.int64)
    key = np.sort(np.concatenate([cols * n + rows, idx * n + idx]))
    colptr = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(np.bincount(key // n, minlength=n), out=colptr[1:])
    return colptr, key % n


def _axes(nd):
    return [tuple(s if k == d else 0 for k in range(nd)) for d in range(nd) for s in (1, -1)]


def _nested_dissection(dims, max_sn, dof):
    """Box bisection by one-plane separators, each after its two halves (new -> old)."""
    strides = np.concatenate([[1], np.cumprod(dims[:-1])]).astype(np.int64)
    out = []

    def emit(lo, hi):
        idx = np.zeros(1, dtype=np.int64)
        for d in range(len(dims) - 1, -1, -1):
            idx = (idx[:, None] + np.arange(lo[d], hi[d]) * strides[d]).reshape(-1)
        out.append((idx[:, None] * dof + np.arange(dof)).reshape(-1))

    def split(lo, hi):
        ext = [b - a for a, b in zip(lo, hi)]
        if min(ext) <= 0:
            return
        if int(np.prod(ext)) * dof <= max_sn or max(ext) <= 2:
            emit(lo, hi)
            return
        d = ext.index(max(ext))
        mid = lo[d] + ext[d] // 2
        left, right, sep = list(hi), list(lo), (list(lo), list(hi))
        left[d], right[d] = mid, mid + 1
        sep[0][d], sep[1][d] = mid, mid + 1
        split(lo, left)
        split(right, hi)
        emit(*sep)

    split([0] * len(dims), list(dims))
    return np.concatenate(out)


@functools.lru_cache(maxsize=4)
def _pattern(family, m, dof, max_sn):
    """(n, colptr, rowind, perm) of one matrix."""
    nd = 2 if family in ("grid2d", "grids", "oneway") else 3
    dims = (m,) * nd
    if family == "stencil27":
        offs = [(a, b, c) for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1)
                if (a, b, c) != (0, 0, 0)]
    else:
        offs = _axes(nd)
    rows, cols = _neighbours(dims, offs)
    cells = m ** nd
    if family == "oneway":  # every coupling towards -x and -y, half of the others
        keep = (rows < cols) | (np.random.default_rng(m).random(rows.size) < 0.5)
        rows, cols = rows[keep], cols[keep]
    colptr, rowind = _csc(cells, rows, cols)
    if dof > 1:  # dense blocks of dof unknowns
        idx = np.arange(dof, dtype=np.int64)
        parts, count = [], []
        for e in range(cells):
            r = (rowind[colptr[e]:colptr[e + 1], None] * dof + idx).reshape(-1)
            parts.append(np.tile(r, dof))
            count.append(np.full(dof, r.size))
        rowind = np.concatenate(parts)
        colptr = np.concatenate([[0], np.cumsum(np.concatenate(count))]).astype(np.int64)
    return cells * dof, colptr, rowind, _nested_dissection(dims, max_sn, dof)


def _members(case):
    """The matrices of a case: several uneven grids for ``grids``, else one."""
    if case["family"] != "grids":
        return [_pattern(case["family"], case["m"], case["dof"], case["max_sn"])]
    top, k = case["m"], case["count"]
    return [_pattern_of_grid(20 + (top - 20) * g // max(1, k - 1), case["max_sn"])
            for g in range(k)]


@functools.lru_cache(maxsize=64)
def _pattern_of_grid(m, max_sn):
    return _pattern("grids", m, 1, max_sn)


@functools.lru_cache(maxsize=2)
def _row_permutation(m, n):
    return np.random.default_rng([m, n]).permutation(n).astype(np.int64)


# ---------------------------------------------------------------------------
# values
# ---------------------------------------------------------------------------
def _values(case, pattern, seed):
    """CSC values, [nnz] or [count, nnz] for a batch of shifts (numpy)."""
    n, colptr, rowind, _ = pattern
    rng = np.random.default_rng(seed)
    col = np.repeat(np.arange(n, dtype=np.int64), np.diff(colptr))
    diag = rowind == col
    nnz, family = rowind.size, case["family"]
    sgn = np.where(rowind > col, 1.0, -1.0)
    if family in ("grid2d", "grids"):  # convection-diffusion
        v = -1.0 + sgn * rng.uniform(0.0, 0.5, nnz)
        v[diag] = 4.1
        if case["complex"]:
            v = v + 0.1j * diag
    elif family in ("upwind", "poles"):  # upwind convection
        w = rng.uniform(-1.0, 1.0, nnz)
        v = -1.0 - np.maximum(sgn * w, 0.0)
        v[diag] = 0.0
        v[diag] = np.add.reduceat(np.abs(v), colptr[:-1]) + (3.1 if family == "poles" else 0.1)
        if family == "poles":
            theta = 2.0 * np.pi * (np.arange(case["count"]) + 0.5) / case["count"]
            z = 1.0 + 2.0 * np.exp(1j * theta)
            v = v[None, :] - z[:, None] * diag[None, :]
    elif family == "diffusion":  # A = A^T: one coefficient per edge
        lo, hi = np.minimum(rowind, col), np.maximum(rowind, col)
        order = np.lexsort((hi, lo))
        first = np.ones(nnz, dtype=bool)
        first[1:] = (lo[order][1:] != lo[order][:-1]) | (hi[order][1:] != hi[order][:-1])
        w = rng.random(int(first.sum()))
        v = np.empty(nnz)
        v[order] = -1.0 - w[np.cumsum(first) - 1]
        v[diag] = 0.0
        v[diag] = np.add.reduceat(np.abs(v), colptr[:-1]) + 0.1
    elif family == "stencil27":  # H - z S + 0.2 N
        v = rng.uniform(-1.0, 1.0, nnz) + 0.2 * rng.uniform(-1.0, 1.0, nnz)
        v[diag] = 0.0
        s = rng.uniform(1.0, 2.0, n)
        d = np.add.reduceat(np.abs(v), colptr[:-1]) + 1.0
        v = v.astype(np.complex128)
        v[diag] = d - 0.1j * s
    else:  # oneway and dg: random couplings, dominant columns
        v = -rng.random(nnz) if family == "oneway" else rng.uniform(-1.0, 1.0, nnz)
        if family == "dg":
            v *= 1.0 + 0.5 * np.where(rowind // case["dof"] == col // case["dof"], 0.0, sgn)
        if case["complex"]:
            v = v + 1j * rng.uniform(-0.5, 0.5, nnz)
        v[diag] = 0.0
        total = np.add.reduceat(np.abs(v), colptr[:-1])
        if family == "oneway":
            total = total + np.bincount(rowind, weights=np.abs(v), minlength=n)
        v[diag] = total + 1.0
    return v


def _all_values(case, seed):
    parts = [_values(case, p, [seed, k]) for k, p in enumerate(_members(case))]
    return parts[0] if len(parts) == 1 else np.concatenate(parts, axis=-1)


def _weights(case):
    theta = 2.0 * np.pi * (np.arange(case["count"]) + 0.5) / case["count"]
    return np.exp(1j * theta) / case["count"]


# ---------------------------------------------------------------------------
# the measured calls
# ---------------------------------------------------------------------------
def _handle(case, host_only=False):
    split = ps.PREC_OZAKI_FP16 if case["precision"] == "split" else ps.PREC_FP64
    kw = {"max_supernode": case["max_sn"], "precision": split, "factor_precision": split,
          "symmetric": case["family"] == "diffusion", "host_only": host_only}
    members = _members(case)
    if case["family"] == "grids":
        parts = [ps.SelInv(*p, max_supernode=case["max_sn"], host_only=True) for p in members]
        h = ps.SelInv.group(parts, **kw)
        for q in parts:
            q.close()
        return h
    n, colptr, rowind, perm = members[0]
    if case["family"] == "oneway":  # rows of A scrambled: P undoes it, Q = the ordering
        rows = _row_permutation(case["m"], n)
        col = np.repeat(np.arange(n, dtype=np.int64), np.diff(colptr))
        order = np.lexsort((rows[rowind], col))
        h = ps.SelInv.general(n, colptr, rows[rowind][order], rperm=rows[perm], cperm=perm, **kw)
        h.value_order = order
        return h
    return ps.SelInv(n, colptr, rowind, perm, **kw)


def prepare(case, seed):
    h = _handle(case)
    values = _all_values(case, seed)
    order = getattr(h, "value_order", None)
    if order is not None:
        values = values[order]
    values = torch.from_numpy(np.ascontiguousarray(values)).cuda()
    state = {"h": h, "values": values, "call": case["call"],
             "out": torch.zeros(h.nnz, dtype=values.dtype, device="cuda")}
    if case["whole"]:
        state["whole"] = torch.zeros(h.structure()["storage_size"], dtype=values.dtype,
                                     device="cuda")
    if case["call"] == "poles":  # an observable on the pattern, real, one value per entry
        obs = np.random.default_rng([seed, 1 << 20]).uniform(-1.0, 1.0, h.nnz)
        state["obs"] = torch.from_numpy(obs.astype(np.complex128)).cuda()
        state["weights"] = _weights(case)
    if case["call"] == "sweep":
        h.factor(values)
    return state


def run(state):
    h = state["h"]
    if state["call"] != "sweep":
        h.factor(state["values"])
    h.selinv()
    if state["call"] == "poles":
        density = h.weighted_sum(state["weights"], state["out"])
        trace = h.trace(state["weights"], state["obs"])
        return {"density": density, "trace": np.array([trace])}
    selected = h.get_selected(state["out"])
    if "whole" not in state:
        return selected
    return {"selected": selected,
            "whole": h.get_selected(state["whole"], layout=ps.LAYOUT_SUPERNODAL)}


@functools.lru_cache(maxsize=16)
def _counts(key):
    h = _handle(dict(key), host_only=True)
    st = h.structure()
    h.close()
    return h.nnz, st["storage_size"], st["flops_selinv_exact"], st["flops_factor"]


def work(case):
    """Flops of Algorithm 1 over the strict supernodes (and of the LU); bytes:
    a sweep reads the factors and writes the selected inverse once, a solve
    reads the values instead; what is copied out is written once."""
    nnz, storage, sweep, lu = _counts(tuple(sorted((k, v) for k, v in case.items()
                                                   if k != "name")))
    size = 16 if case["complex"] else 8
    batch = case["count"] if case["family"] == "poles" else 1
    flops = sweep + (0.0 if case["call"] == "sweep" else lu)
    flops *= batch * (4 if case["complex"] else 1) * (0.5 if case["family"] == "diffusion" else 1)
    given = storage if case["call"] == "sweep" else nnz
    copied = nnz + (storage if case["whole"] else 0)
    return {"bytes": float(size * (batch * (given + storage) + copied)), "flops": float(flops)}


def exact(case, seed):
    """Dense inverses in 64 bits, where they take seconds."""
    members = _members(case)
    batch = case["count"] if case["family"] == "poles" else 1
    cost = sum(float(p[0]) ** 3 for p in members) * batch * (4 if case["complex"] else 1)
    if cost > 6e12:
        return None
    outs, trace = [], 0.0
    for k, (n, colptr, rowind, perm) in enumerate(members):
        col = np.repeat(np.arange(n, dtype=np.int64), np.diff(colptr))
        order = np.arange(rowind.size)
        rows = rowind
        if case["family"] == "oneway":
            rows = _row_permutation(case["m"], n)[rowind]
            order = np.lexsort((rows, col))
        r = torch.from_numpy(rows[order]).cuda()
        c = torch.from_numpy(col[order]).cuda()
        values = torch.from_numpy(np.ascontiguousarray(
            _values(case, (n, colptr, rowind, perm), [seed, k])[..., order])).cuda()
        if case["family"] == "poles":
            w = _weights(case)
            obs = torch.from_numpy(
                np.random.default_rng([seed, 1 << 20]).uniform(-1.0, 1.0, r.numel())).cuda()
        out = 0.0
        for b in range(batch):
            a = torch.zeros((n, n), dtype=values.dtype, device="cuda")
            a[r, c] = values if values.dim() == 1 else values[b]
            inv = torch.linalg.inv(a)
            if case["family"] == "poles":
                out = out + complex(w[b]) * inv[r, c]
                trace = trace + complex(w[b]) * (obs * inv[c, r]).sum()
            else:  # a pattern that is not symmetric selects the transposed positions
                out = inv[c, r] if case["family"] == "oneway" else inv[r, c]
        outs.append(out)
        del a, inv
    if case["call"] == "poles":
        return {"density": outs[0], "trace": trace.reshape(1).cpu().numpy()}
    selected = outs[0] if len(outs) == 1 else torch.cat(outs)
    return {"selected": selected, "whole": None} if case["whole"] else selected
