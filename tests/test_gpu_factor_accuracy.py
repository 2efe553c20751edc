"""Accuracy of the split options' products that are not six-slice ones: panel
solves that stay on the FP64 pipe, and products of eight slices, those of badly
scaled operands included."""
from __future__ import annotations

import numpy as np
import pytest

import gen
import oracle
from helpers import selected_error

pytestmark = pytest.mark.gpu

U64 = 2.0 ** -53


@pytest.fixture(scope="module")
def torch():
    import torch as _t
    if not _t.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1708_04539_gb300 import build
    build.build()
    return _t


def csc(a, rng):
    """(colptr, rowind, values) of a dense array's non-zero pattern."""
    r, c = np.nonzero(a.T)[1], np.nonzero(a.T)[0]
    colptr = np.zeros(a.shape[0] + 1, dtype=np.int64)
    np.cumsum(np.bincount(c, minlength=a.shape[0]), out=colptr[1:])
    return colptr, r.astype(np.int64), np.ascontiguousarray(a[r, c])


@pytest.mark.parametrize("complex_values", [False, True])
@pytest.mark.parametrize("s", [20, 40])
def test_one_sided_level_solves_in_fp64(torch, s, complex_values):
    """General pattern, split factorisation: on a level with a supernode that
    has only one of R_L and R_U every panel is solved in FP64.  The first
    supernode's panels take no Schur update, so they agree with the FP64
    factorisation's to rounding: a solve against s columns errs by at most s u of
    its largest terms (diagonally dominant: of the order of the panel's largest
    entry) on each side, 8 s u in all; six slices err by 2^-43 = 1024 u a term."""
    import paper_1708_04539_gb300 as ps
    rng = np.random.default_rng(s)
    n, k = 136, 96
    a = np.zeros((n, n), dtype=complex if complex_values else float)
    a[:k, :k] = rng.uniform(-1, 1, (k, k))
    a[k:, k:] = np.triu(rng.uniform(-1, 1, (n - k, n - k)), 1)
    if complex_values:
        a = a + 1j * np.where(a != 0, rng.uniform(-1, 1, (n, n)), 0)
    np.fill_diagonal(a, np.abs(a).sum(0) + np.abs(a).sum(1) + 1)
    colptr, rowind, values = csc(a, rng)
    order = np.arange(n, dtype=np.int64)
    got = []
    for kw in ({}, {"factor_precision": ps.PREC_OZAKI_FP16, "factor_split_mflops": -1}):
        h = ps.SelInv.general(n, colptr, rowind, rperm=order, cperm=order, max_supernode=s,
                              relax_pct=0, **kw)
        st = h.structure()
        h.factor(torch.from_numpy(values).cuda())
        got.append(h.get_selected(layout=ps.LAYOUT_FACTORS))
        h.close()
    c, cu = np.diff(st["rows_ptr"]), np.diff(st["urows_ptr"])
    assert st["sn_width"][0] == s and c[0] == cu[0] == k - s
    assert ((c == 0) != (cu == 0)).any()
    w = slice(st["sn_offset"][0] + s * s, st["sn_offset"][0] + s * s + 2 * s * (k - s))
    ref, x = got[0][w], got[1][w]
    for part in (slice(0, s * (k - s)), slice(s * (k - s), None)):
        assert np.abs(x[part] - ref[part]).max() <= 8 * s * U64 * np.abs(ref[part]).max()


@pytest.mark.parametrize("kind", ["real", "complex", "symmetric"])
@pytest.mark.parametrize("s,c", [(33, 140), (64, 133), (65, 64), (256, 60)])
def test_eight_slice_outputs_keep_their_bits(torch, kind, s, c):
    """Panels over an identity block, so that the solved panels are A's own: every
    row has entries of 1 and of 2^-20.  Their digits hold 63 bits below the
    row's power of two (2 at most) and the other operand is one digit, so an entry
    is off by at most 2^-63 and its own rounding."""
    import paper_1708_04539_gb300 as ps
    n = s + c
    nb = int(1.2e8 / ((2.0 * c * c * s + 2.0 * c * s * s) * (4 if kind == "complex" else 1)
                      * (0.5 if kind == "symmetric" else 1))) + 1
    rng = np.random.default_rng(s)

    def panel():
        x = rng.uniform(0.5, 1, (c, s)) * np.where(rng.random((c, s)) < 0.2, 1.0, 2.0 ** -20)
        return x + (1j * rng.uniform(-1, 1, (c, s)) * 2.0 ** -18 if kind == "complex" else 0)
    low = panel()
    up = low if kind == "symmetric" else panel()
    a = np.zeros((n, n), dtype=low.dtype)
    a[s:, :s], a[:s, s:] = low, up.T
    a[:s, :s] = np.eye(s)
    a[s:, s:] = 4.0 * n * np.eye(c)
    colptr = np.arange(n + 1, dtype=np.int64) * n  # (the whole pattern, zeros too)
    rowind = np.tile(np.arange(n, dtype=np.int64), n)
    h = ps.SelInv(n, colptr, rowind, np.arange(n, dtype=np.int64), max_supernode=s,
                  symmetric=kind == "symmetric", factor_precision=ps.PREC_OZAKI_FP16,
                  factor_split_mflops=100000)
    st = h.structure()
    assert st["sn_width"][0] == s
    h.factor(torch.from_numpy(np.tile(a.T.reshape(-1), (nb, 1))).cuda())
    assert any(r["kind"] == "ozaki_gemm" and r["level"] == 0 for r in h.profile(1))
    h.factor(torch.from_numpy(np.tile(a.T.reshape(-1), (nb, 1))).cuda())
    for b in (0, nb - 1):
        fac = h.get_selected(batch=b, layout=ps.LAYOUT_FACTORS)
        o = st["sn_offset"][0] + s * s
        for got, ref in ((fac[o:o + c * s], low), (fac[o + c * s:o + 2 * c * s], up)):
            got = got.reshape(s, c).T
            for x, r in ((got.real, ref.real), (got.imag, ref.imag)):
                assert (np.abs(x - r) <= 2.0 ** -63 + U64 * np.abs(r)).all()
    h.close()


def scalings(kind, n, s, seed):
    """Row and column scalings by powers of two, (rows, columns)."""
    rng = np.random.default_rng(seed)
    k = np.arange(n)
    which, how = kind.split("-")
    d = []
    for x in ("rows", "cols"):
        e = {"up": 40 * k // s, "down": 40 - 40 * k // s, "random": rng.integers(0, 41, n)}[how]
        e = np.where(k < s, e - 20, 0)  # within the first supernode
        d.append(np.ldexp(1.0, e if which in (x, "both") else 0 * e))
    return d


SCALINGS = ["rows-up", "rows-down", "rows-random", "cols-up", "cols-down", "cols-random",
            "both-up", "both-down", "both-random"]


@pytest.mark.parametrize("kind", ["real", "complex"])
@pytest.mark.parametrize("scaling", SCALINGS)
def test_scaled_factors(torch, kind, scaling):
    """A level of eight-slice products whose first supernode's rows or columns are
    scaled by powers of two: the FP64 factorisation would give exactly the scaled
    factors, so they are held to the FP64 bound, 1e-12, with the scaling undone."""
    import paper_1708_04539_gb300 as ps
    from paper_1708_04539_gb300.binding import supernodal_coordinates
    s, n, nb = 96, 96 + 133, 40 if kind == "real" else 12
    ii, jj = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
    p = gen.problems._finish_small(n, ii.reshape(-1), jj.reshape(-1), 70, kind == "complex",
                                   f"dense_{n}", s)
    d1, d2 = scalings(scaling, n, s, 3)
    col = np.repeat(np.arange(n), np.diff(p.colptr))
    vals = p.values * d1[p.rowind] * d2[col]
    h = ps.SelInv.from_problem(p, factor_precision=ps.PREC_OZAKI_FP16, factor_split_mflops=100000)
    h.factor(torch.from_numpy(np.tile(vals, (nb, 1))).cuda())
    assert any(r["kind"] == "ozaki_gemm" for r in h.profile(1))
    h.factor(torch.from_numpy(np.tile(vals, (nb, 1))).cuda())
    sym = oracle.analyze(p, relax_pct=20)
    orows, ocols = sym.lu_pattern()
    grows, gcols = supernodal_coordinates(h.structure())
    gi, oi = np.argsort(grows * n + gcols), np.argsort(orows * n + ocols)
    f = oracle.lu(sym, p.colptr, p.rowind, p.values)
    ref = np.concatenate([f.diag, f.low, f.up])
    r, c = grows, gcols
    undo = np.where(r > c, d1[c] / d1[r], 1.0 / (d1[r] * d2[c]))  # L, U
    for b in (0, nb - 1):
        got = h.get_selected(batch=b, layout=ps.LAYOUT_FACTORS) * undo
        assert selected_error(got[gi], ref[oi], orows[oi], ocols[oi], n) < 1e-12
    h.close()


@pytest.mark.parametrize("kind", ["real", "complex"])
@pytest.mark.parametrize("scaling", SCALINGS)
def test_scaled_normalisation(torch, kind, scaling):
    """The same for the split sweep, whose six-slice products see nothing of a
    scaling inside one supernode: 1e-11 with the scaling undone, as unscaled."""
    import paper_1708_04539_gb300 as ps
    from paper_1708_04539_gb300.binding import supernodal_coordinates
    s, n = 96, 96 + 133
    ii, jj = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
    p = gen.problems._finish_small(n, ii.reshape(-1), jj.reshape(-1), 71, kind == "complex",
                                   f"dense_{n}", s)
    d1, d2 = scalings(scaling, n, s, 4)
    col = np.repeat(np.arange(n), np.diff(p.colptr))
    vals = p.values * d1[p.rowind] * d2[col]
    h = ps.SelInv.from_problem(p)
    nlev = int(h.structure()["nlevels"])
    h.plan_set([(lev, 3, 0) for lev in range(nlev)], ps.PREC_OZAKI_FP16)
    h.factor(torch.from_numpy(vals).cuda())
    h.selinv(precision=ps.PREC_OZAKI_FP16)
    sel = oracle.selected_inverse(p, relax_pct=20)
    orows, ocols = sel.sym.lu_pattern()
    grows, gcols = supernodal_coordinates(h.structure())
    gi, oi = np.argsort(grows * n + gcols), np.argsort(orows * n + ocols)
    got = h.get_selected(layout=ps.LAYOUT_SUPERNODAL) * (d2[grows] * d1[gcols])
    h.close()
    ref = sel.values_lu_order()
    assert selected_error(got[gi], ref[oi], orows[oi], ocols[oi], n) < 1e-11


@pytest.mark.parametrize("tiny", [2.0 ** -1060, 2.0 ** -1000, 0.0])
def test_tiny_rows(torch, tiny):
    """Rows of a panel at and below the end of the normal range, and of zeros: an
    eight-slice level gives what the FP64 one gives, to its rounding."""
    import paper_1708_04539_gb300 as ps
    s, c, nb = 64, 133, 40
    n = s + c
    rng = np.random.default_rng(8)
    a = rng.uniform(-1, 1, (n, n))
    a[s + 5, :s] *= tiny
    a[:s, s + 9] *= tiny
    np.fill_diagonal(a, 2.0 * n)
    colptr = np.arange(n + 1, dtype=np.int64) * n
    rowind = np.tile(np.arange(n, dtype=np.int64), n)
    got = []
    for kw in ({}, {"factor_precision": ps.PREC_OZAKI_FP16, "factor_split_mflops": 100000}):
        h = ps.SelInv(n, colptr, rowind, np.arange(n, dtype=np.int64), max_supernode=s, **kw)
        st = h.structure()
        h.factor(torch.from_numpy(np.tile(a.T.reshape(-1), (nb, 1))).cuda())
        got.append(h.get_selected(batch=nb - 1, layout=ps.LAYOUT_FACTORS))
        h.close()
    o = st["sn_offset"][0] + s * s
    for row, o in ((5, o), (9, o + c * s)):
        x, ref = (g[o:o + c * s].reshape(s, c)[:, row] for g in got)
        scale = max(np.abs(ref).max(), 0.0)
        assert np.abs(x - ref).max() <= max(8 * s * U64 * scale, 4 * s * 2.0 ** -1074) * (tiny != 0)
    assert np.isfinite(got[1]).all()


@pytest.mark.parametrize("s,c", [(96, 133), (128, 65)])
def test_eight_slice_schur_products(torch, s, c):
    """Schur products over an identity block against exact sums: the first row of
    the next supernode is the negated products (zeros before).  A term's digits and
    left-out pairs err by 2^-64 (standard deviation, of the rows' powers of two, 1
    here), K <= 128 of them, one exact chunk, by sqrt(K) as much; 16 standard
    deviations and one rounding.  A slice less would show 2^-56 a term."""
    from fractions import Fraction

    import paper_1708_04539_gb300 as ps
    n = s + c
    nb = int(1.2e8 / (2.0 * c * c * s + 2.0 * c * s * s)) + 1
    rng = np.random.default_rng(c)

    def panel():
        return rng.uniform(0.5, 1, (c, s)) * rng.choice([-1.0, 1.0], (c, s))
    low, up = panel(), panel()
    a = np.zeros((n, n))
    a[s:, :s], a[:s, s:] = low, up.T
    a[:s, :s] = np.eye(s)
    a[s:, s:] = 4.0 * n * np.eye(c)
    colptr = np.arange(n + 1, dtype=np.int64) * n
    rowind = np.tile(np.arange(n, dtype=np.int64), n)
    h = ps.SelInv(n, colptr, rowind, np.arange(n, dtype=np.int64), max_supernode=s,
                  factor_precision=ps.PREC_OZAKI_FP16, factor_split_mflops=100000)
    st = h.structure()
    h.factor(torch.from_numpy(np.tile(a.T.reshape(-1), (nb, 1))).cuda())
    fac = h.get_selected(batch=nb - 1, layout=ps.LAYOUT_FACTORS)
    h.close()
    w, o = int(st["sn_width"][1]), int(st["sn_offset"][1])
    assert w > 1 and st["sn_first"][1] == s
    row = fac[o:o + w * w].reshape(w, w).T[0]  # U of the second supernode, first row
    tol = 16 * np.sqrt(s) * 2.0 ** -64
    for q in range(1, w):
        ref = -sum(Fraction(float(x)) * Fraction(float(y)) for x, y in zip(low[0], up[q]))
        assert abs(Fraction(float(row[q])) - ref) <= tol + U64 * abs(float(ref)), q
