"""SpMV layouts (rs_spmv.cu) against the oracle's row-by-row product.

Matrices and vectors hold small integers, so every product and sum is exact
and the results must match bit for bit whatever their order; sizes lie at the
edges of the 32-row slices, the 512-row sorting windows and the layouts' rules.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(rs):
    return rs.Context(0)


def _vec(rs, ctx, x, shift):
    """x on the GPU; shift: at an address that is only 8-byte aligned."""
    import torch
    buf = torch.empty(x.size + 1, dtype=torch.float64, device="cuda")
    v = buf[1:] if shift else buf[:-1]
    v.copy_(torch.from_numpy(np.asarray(x, dtype=np.float64)))
    return rs.Vec(ctx, v)


def _check(rs, ctx, orc, d, rng, shift=False):
    bs = d.get("bs", 1)
    A = rs.Mat.csr(ctx, d) if bs == 1 else rs.Mat.bsr(ctx, d)
    Ao = orc.Mat.csr(d) if bs == 1 else orc.Mat.bsr(d)
    x, y0 = (rng.integers(-9, 10, size=A.n).astype(float) for _ in range(2))
    xv, y = _vec(rs, ctx, x, shift), _vec(rs, ctx, y0, shift)
    ref = orc.spmv(Ao, x)
    for a, b in ((1.0, 0.0), (-2.0, 0.0), (-1.0, 1.0), (2.0, -3.0)):
        y.t.copy_(_vec(rs, ctx, y0, False).t)
        if (a, b) == (1.0, 0.0):
            A.spmv(xv, y)
        else:
            A.amxpby(a, xv, b, y)
        assert np.array_equal(y.numpy(), a * ref + b * y0), (a, b)
    return A, Ao, x


def _offsets_matrix(n, offs, keep, bs, rng):
    """Blocks of small integers at the given offsets, a share `keep` of them
    (the diagonal always)."""
    ptr, col = [0], []
    for i in range(n):
        c = [i + o for o in sorted(offs) if 0 <= i + o < n and (o == 0 or rng.random() < keep)]
        col += c
        ptr.append(len(col))
    val = rng.integers(-5, 6, size=len(col) * bs * bs).astype(float)
    ptr, col = np.array(ptr, np.int32), np.array(col, np.int32)
    if bs == 1:
        return dict(n=n, rowptr=ptr, col=col, val=val)
    return dict(nb=n, bs=bs, browptr=ptr, bcol=col, bval=val)


@pytest.mark.parametrize("bs", [1, 2, 3])
@pytest.mark.parametrize("n,offs,keep", [
    (1, [0], 1.0), (33, [0, 1], 1.0), (257, [-1, 0, 1], 0.9), (600, [-20, -1, 0, 20], 0.8),
    (1000, [-37, -1, 0, 1, 37], 1.0), (900, [-90, -9, 0, 1, 9, 90], 0.95),
    (1287, [-117, -13, -1, 0, 1, 13, 117], 0.85), (800, [-100, -31, -3, 0, 2, 5, 77, 99], 0.9),
    (500, [-8, -7, -5, -3, 0, 1, 2, 4, 9], 1.0),       # nine offsets: no stencil layout
    (700, [-50, -5, -1, 0, 1, 5, 50], 0.4)])           # too empty for one
def test_stencil_layout(rs, ctx, orc, bs, n, offs, keep):
    rng = np.random.default_rng(n + bs)
    _check(rs, ctx, orc, _offsets_matrix(n, offs, keep, bs, rng), rng, shift=n % 2 == 1)


# block rows on both sides of 280,000, from which a thread takes a whole block
# row; sizes off the thread blocks of 32 and 256; odd offsets; 7 and 3 of them
@pytest.mark.parametrize("bs", [2, 3])
@pytest.mark.parametrize("n,offs", [(31, [-5, -1, 0, 1, 5]), (279999, [-700, -31, -1, 0, 1, 31, 700]),
                                    (280001, [-700, -31, -1, 0, 1, 31, 700]), (300015, [-1, 0, 64])])
def test_stencil_products_of_small_and_large_block_systems(rs, ctx, bs, n, offs):
    rng = np.random.default_rng(n + bs)
    i = np.arange(n)
    on = np.stack([(i + o >= 0) & (i + o < n) for o in offs], axis=1) & (rng.random((n, len(offs))) < 0.9)
    on[:, offs.index(0)] = True
    ptr = np.concatenate([[0], np.cumsum(on.sum(1))]).astype(np.int32)
    row, k = np.nonzero(on)
    col = row + np.array(offs)[k]
    val = rng.integers(-5, 6, size=(row.size, bs, bs)).astype(float)
    A = rs.Mat.bsr(ctx, dict(nb=n, bs=bs, browptr=ptr, bcol=col.astype(np.int32), bval=val.reshape(-1)))
    x, y0 = (rng.integers(-9, 10, size=n * bs).astype(float) for _ in range(2))
    ref = np.zeros((n, bs))
    np.add.at(ref, row, np.einsum("eij,ej->ei", val, x.reshape(n, bs)[col]))
    xv, y = rs.Vec(ctx, x), rs.Vec(ctx, y0)
    A.amxpby(-1.0, xv, 1.0, y)
    assert np.array_equal(y.numpy(), y0 - ref.reshape(-1))
    A.spmv(xv, y)
    assert np.array_equal(y.numpy(), ref.reshape(-1))


def test_stencil_layout_rejects_a_late_offset(rs, ctx, orc):
    """One entry off the sampled rows' offsets: the matrix keeps CSR."""
    rng = np.random.default_rng(7)
    d = _offsets_matrix(5000, [-1, 0, 1], 1.0, 1, rng)
    p = d["rowptr"][1235]            # row 1234 gets an entry at column 4000
    d["col"] = np.insert(d["col"], p, 4000).astype(np.int32)
    d["val"] = np.insert(d["val"], p, 3.0)
    d["rowptr"][1235:] += 1
    _check(rs, ctx, orc, d, rng)


@pytest.mark.parametrize("bs", [1, 3])
def test_stencil_layout_keeps_nan_and_infinity_to_the_rows_that_refer_to_them(rs, ctx, bs):
    rng = np.random.default_rng(3)
    d = _offsets_matrix(1287, [-117, -13, -1, 0, 1, 13, 117], 0.85, bs, rng)
    ptr, col = (d["rowptr"], d["col"]) if bs == 1 else (d["browptr"], d["bcol"])
    A = rs.Mat.csr(ctx, d) if bs == 1 else rs.Mat.bsr(ctx, d)
    x = rng.integers(-9, 10, size=A.n).astype(float)
    bad = np.array([5, 640, 1286])
    x[bad * bs] = [np.nan, np.inf, np.nan]
    y = rs.Vec.zeros(ctx, A.n)
    A.spmv(rs.Vec(ctx, x), y)
    rows = np.repeat(np.arange(1287), np.diff(ptr))
    hit = np.zeros(1287, bool)
    hit[rows[np.isin(col, bad)]] = True
    got = np.isfinite(y.numpy()).reshape(1287, bs).all(1)
    assert got[~hit].all()


@pytest.mark.parametrize("n", [32767, 32768, 32769, 33280, 50001])
@pytest.mark.parametrize("lo,hi", [(1, 1), (1, 9), (3, 40)])
def test_sliced_layout(rs, ctx, orc, n, lo, hi):
    """Rows of lo to hi entries in any order of lengths."""
    rng = np.random.default_rng(n + hi)
    cnt = rng.integers(lo, hi + 1, size=n)
    col = rng.integers(0, n, size=(n, hi))
    col[:, 0] = np.arange(n)
    col[np.arange(hi)[None, :] >= cnt[:, None]] = -1
    col.sort(axis=1)
    keep = col >= 0
    keep[:, 1:] &= col[:, 1:] != col[:, :-1]
    ptr = np.concatenate([[0], np.cumsum(keep.sum(1))]).astype(np.int32)
    c = col[keep].astype(np.int32)
    d = dict(n=n, rowptr=ptr, col=c, val=rng.integers(-5, 6, size=c.size).astype(float))
    _check(rs, ctx, orc, d, rng, shift=n % 2 == 1)


def test_sliced_layout_refuses_a_row_that_would_leave_a_slice_to_one_lane(rs, ctx, orc):
    rng = np.random.default_rng(11)
    n = 40000
    dense = np.arange(n, dtype=np.int32)
    col = np.concatenate([np.arange(100, dtype=np.int32), dense, np.arange(101, n, dtype=np.int32)])
    ptr = np.concatenate([np.arange(101), n + np.arange(100, n)]).astype(np.int32)
    d = dict(n=n, rowptr=ptr, col=col, val=rng.integers(-2, 3, size=col.size).astype(float))
    _check(rs, ctx, orc, d, rng)


@pytest.mark.parametrize("form", ["pf", "fp"])
@pytest.mark.parametrize("sealed", [0.0, 0.5])
def test_cpr_residual_with_and_without_the_stencil_layout(rs, ctx, orc, form, sealed):
    """sealed 0.5: the pattern is too empty for the stencil layout."""
    g = synth.Grid(13, 11, 7)
    m = synth.black_oil_bsr3(g, 4)
    if sealed:
        rng = np.random.default_rng(5)
        rows = np.repeat(np.arange(g.n), np.diff(m["browptr"]))
        pair = np.minimum(rows, m["bcol"]) * np.int64(g.n) + np.maximum(rows, m["bcol"])
        keep = (rows == m["bcol"]) | (np.random.default_rng(5).permutation(g.n * 4)[pair % (g.n * 4)] % 2 == 0)
        m["bval"] = m["bval"].reshape(-1, 9)[keep].reshape(-1)
        m["bcol"] = m["bcol"][keep]
        m["browptr"] = np.concatenate([[0], np.cumsum(np.bincount(rows[keep], minlength=g.n))]).astype(np.int32)
        assert m["bcol"].size < 0.7 * 7 * g.n
    A, Ao = rs.Mat.bsr(ctx, m), orc.Mat.bsr(m)
    M, Mo = rs.Precond(ctx, A, "cpr", form=form), orc.PC(Ao, "cpr", form=form)
    r = np.random.default_rng(6).standard_normal(A.n)
    z = rs.Vec.zeros(ctx, A.n)
    M.apply(rs.Vec(ctx, r), z)
    ref = Mo.apply(r)
    assert np.linalg.norm(z.numpy() - ref) <= 1e-12 * np.linalg.norm(ref)
