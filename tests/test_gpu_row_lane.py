"""The row-per-lane layout of the packed binary64 stream (and of the complex64
copy): slices of 32 rows, the diagonal entry in a slice's last step, groups of
8 steps.  Sizes at the edges: a partial last slice, widths around one and
several groups and at the widest slice, rows without a diagonal entry or
without any entry, duplicate diagonal entries; groups that change between real
and complex under a value refresh or a new diagonal; non-finite x.

Tolerance of a binary64 entry: any order of its 2 m products is within
(2 m + 1) 2^-53 sum |a||x| of the exact value, twice that against the oracle
(m: entries of the row; one addition more for the second chain).  Complex64:
the same with 2^-23 for 2^-52."""

import numpy as np
import pytest
import torch

import workloads as W
from tests import _cases as K

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.as_tensor(a).cuda()


def host(t):
    torch.cuda.synchronize()
    return t.cpu().numpy()


def banded(n, width, seed, real=True, diag="all"):
    """Rows of `width` entries (fewer only by the rules of `diag`) near the
    diagonal; values real off the diagonal and complex on it, or all complex."""
    rng = np.random.default_rng(seed)
    rp, cols, vals = [0], [], []
    for i in range(n):
        lo = min(max(0, i - width // 2), n - width)
        c = np.arange(lo, lo + width)
        if diag == "some" and i % 5 == 2:
            c = c[c != i]                        # no diagonal entry
        if diag == "some" and i % 37 == 11:
            c = c[:0]                            # no entry at all
        if diag == "twice" and i % 3 == 0 and c.size:
            c = np.sort(np.append(c[c != (c[0] if c[0] != i else c[-1])], i))   # the diagonal stored twice
        v = rng.standard_normal(c.size) + 0j
        cplx = np.ones(c.size, bool) if not real else c == i
        v[cplx] += 1j * rng.standard_normal(int(cplx.sum()))
        rp.append(rp[-1] + c.size)
        cols.append(c)
        vals.append(v)
    return W.CSR(n, np.array(rp, np.int32), np.concatenate(cols).astype(np.int32), np.concatenate(vals))


def bound(A, x, eps=2.0 ** -52):
    m = np.diff(A.rowptr).astype(np.float64)
    return (2.0 * m + 4.0) * eps * K.row_abs_scale(A, x) + 1e-300


@pytest.mark.parametrize("n,width,real,diag", [
    (1, 1, True, "all"), (31, 7, True, "all"), (33, 8, False, "all"), (1000, 9, True, "some"),
    (4099, 15, True, "all"), (4099, 16, False, "some"), (777, 17, True, "twice"), (500, 27, False, "all"),
    (300, 64, True, "all"), (300, 65, True, "all"), (700, 130, False, "some")])
def test_product_widths_and_rows(hz, oracle, n, width, real, diag):
    A = banded(n, width, 3 * n + width, real, diag)
    x = K.vectors(n, n + 1)[0]
    M = hz.Matrix.from_csr(A, c64=True)
    assert np.all(np.abs(host(hz.zspmv(M, dev(x))) - oracle.zspmv(A, x)) <= bound(A, x))
    x32 = x.astype(np.complex64)
    err = np.abs(host(hz.cspmv(M, dev(x32))) - oracle.cspmv(A, x32))
    assert np.all(err <= bound(A, x32.astype(np.complex128), 2.0 ** -23))
    M.close()


def test_value_refresh_and_new_diagonal(hz, oracle):
    """Real groups turn complex and back with the caller's values, the
    diagonal follows hz_mat_set_diag, with and without a complex64 copy."""
    A = banded(1500, 15, 5, real=True)
    rows = np.repeat(np.arange(A.n), np.diff(A.rowptr))
    x, th = K.vectors(A.n, 6)
    base = K.vectors(A.n, 8)[0]
    for c64 in (False, True):
        vd = dev(A.val.copy())
        M = hz.Matrix(dev(A.rowptr), dev(A.col), vd, c64=c64)
        v = A.val.copy()
        v[(rows >= 400) & (rows < 470)] *= 1j
        for cur in (v, A.val):
            vd.copy_(torch.as_tensor(cur))
            M.refresh_values()
            B = W.CSR(A.n, A.rowptr, A.col, cur)
            assert np.all(np.abs(host(hz.zspmv(M, dev(x))) - oracle.zspmv(B, x)) <= bound(B, x))
        hz.mat_set_diag(M, dev(base), -3.0 + 0.5j, dev(th))
        new = A.val.copy()
        new[A.col == rows] = base + (-3.0 + 0.5j) * th
        B = W.CSR(A.n, A.rowptr, A.col, new)
        # base + c theta: two products and two sums of unit size
        assert np.allclose(host(vd), new, rtol=0, atol=8 * 2.0 ** -53 * (np.abs(base).max() + 4 * np.abs(th).max()))
        B = W.CSR(A.n, A.rowptr, A.col, host(vd))
        assert np.all(np.abs(host(hz.zspmv(M, dev(x))) - oracle.zspmv(B, x)) <= bound(B, x))
        if c64:
            x32 = x.astype(np.complex64)
            err = np.abs(host(hz.cspmv(M, dev(x32))) - oracle.cspmv(B, x32))
            assert np.all(err <= bound(B, x32.astype(np.complex128), 2.0 ** -23))
        M.close()


@pytest.mark.parametrize("n,lens", [(5000, (33,)), (5000, (200, 33, 512, 34)), (129, (100,)), (5000, (513,))])
def test_long_rows(hz, oracle, n, lens):
    """A few rows far longer than the others (up to 512 entries in this
    layout; 513 takes the lane runs), one of them in the last slice: products,
    a new diagonal, a solve."""
    A = banded(n, 9, 31 + n, real=True)
    m = A.to_scipy().tolil()
    rng = np.random.default_rng(n)
    for k, L in enumerate(lens):
        r = n - 1 if k == 0 else 700 * k
        c = rng.choice(n, size=min(L, n), replace=False)
        c[0] = r
        m[r, :] = 0
        m[r, np.unique(c)] = rng.standard_normal(np.unique(c).size) * 0.01
    m = m.tocsr() + 40.0 * W.CSR(n, np.arange(n + 1, dtype=np.int32), np.arange(n, dtype=np.int32),
                                 np.ones(n, np.complex128)).to_scipy()
    m.sort_indices()
    A = W.CSR(n, m.indptr.astype(np.int32), m.indices.astype(np.int32), m.data.astype(np.complex128))
    x, b = K.vectors(n, 12)
    M = hz.Matrix.from_csr(A, c64=True)
    assert np.all(np.abs(host(hz.zspmv(M, dev(x))) - oracle.zspmv(A, x)) <= bound(A, x))
    x32 = x.astype(np.complex64)
    err = np.abs(host(hz.cspmv(M, dev(x32))) - oracle.cspmv(A, x32))
    assert np.all(err <= bound(A, x32.astype(np.complex128), 2.0 ** -23))
    for kw in (dict(), dict(method="tfqmr"), dict(mode="mixed")):
        y, info = hz.zsolve(M, dev(b), tol=1e-11, maxit=500, **kw)
        assert info.status == 0
        r = b - oracle.zspmv(A, host(y))
        assert np.linalg.norm(r) <= 2e-11 * np.linalg.norm(b)
    g = host(hz.outer_on_pattern(M, dev(b), dev(x)))
    rows = np.repeat(np.arange(n), np.diff(A.rowptr))
    # two products and a sum per component
    assert np.all(np.abs(g + np.conj(b[rows] * x[A.col])) <= 4 * 2.0 ** -53 * np.abs(b[rows]) * np.abs(x[A.col]))
    base, th = K.vectors(n, 13)
    hz.mat_set_diag(M, dev(base), 2.0, dev(th))
    B = W.CSR(n, A.rowptr, A.col, host(M.val))
    assert np.array_equal(host(M.val)[A.col == rows], base + 2.0 * th)
    assert np.all(np.abs(host(hz.zspmv(M, dev(x))) - oracle.zspmv(B, x)) <= bound(B, x))
    M.close()


def test_nonfinite_x(hz, oracle):
    """An infinite or NaN entry of x reaches a row as in binary64 arithmetic
    (0 * inf = NaN), in real groups, complex groups and the diagonal step."""
    A = banded(700, 15, 9, real=True)
    x = K.vectors(A.n, 10)[0]
    x[100], x[351], x[699] = complex(np.inf, 1.0), complex(2.0, np.nan), complex(0.5, -np.inf)
    M = hz.Matrix.from_csr(A)
    with np.errstate(all="ignore"):
        ref = oracle.zspmv(A, x)
    y = host(hz.zspmv(M, dev(x)))
    assert np.array_equal(np.isnan(y.real), np.isnan(ref.real))
    assert np.array_equal(np.isnan(y.imag), np.isnan(ref.imag))
    ok = np.isfinite(ref.real) & np.isfinite(ref.imag)
    assert np.allclose(y[ok], ref[ok], rtol=0, atol=1e-12)
    M.close()


def on_slices(hz, A, x):
    """Whether a product of the default kind reads the row-per-lane layout: lane
    runs form the same sums as the unpacked kind, one row per lane other ones."""
    M = hz.Matrix.from_csr(A)
    y = host(hz.zspmv(M, dev(x)))
    M.set_spmv("flat64")
    same = np.array_equal(y, host(hz.zspmv(M, dev(x))))
    M.close()
    return not same


def with_long(A, first, count, length, seed):
    """A with `count` neighbouring rows replaced by rows of `length` entries."""
    rng = np.random.default_rng(seed)
    rows = np.repeat(np.arange(A.n), np.diff(A.rowptr))
    keep = (rows < first) | (rows >= first + count)
    r, c, v = [rows[keep]], [A.col[keep]], [A.val[keep]]
    for i in range(first, first + count):
        q = rng.permutation(A.n)
        q = np.append(q[q != i][:length - 1], i)
        r.append(np.full(length, i))
        c.append(q)
        v.append(rng.standard_normal(length) + 0j)
    r, c, v = (np.concatenate(q) for q in (r, c, v))
    o = np.lexsort((c, r))
    rp = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=A.n))]).astype(np.int32)
    return W.CSR(A.n, rp, c[o].astype(np.int32), v[o])


@pytest.mark.parametrize("count,length,slices", [
    (1, 255, True), (1, 257, True), (1, 512, True), (2, 256, True), (2, 257, False), (3, 100, False),
    (32, 400, False)])
def test_long_rows_together(hz, oracle, count, length, slices):
    """Rows of up to two passes of 256 entries in a slice are summed by its
    warp; more of them, which one warp would walk through alone, take the lane
    runs."""
    A = with_long(banded(5000, 9, 3, real=False), 1024, count, length, 17)
    x = K.vectors(A.n, 18)[0]
    assert on_slices(hz, A, x) == slices
    M = hz.Matrix.from_csr(A, c64=True)
    assert np.all(np.abs(host(hz.zspmv(M, dev(x))) - oracle.zspmv(A, x)) <= bound(A, x))
    x32 = x.astype(np.complex64)
    err = np.abs(host(hz.cspmv(M, dev(x32))) - oracle.cspmv(A, x32))
    assert np.all(err <= bound(A, x32.astype(np.complex128), 2.0 ** -23))
    M.close()


@pytest.mark.parametrize("n,width,diag", [
    (1, 1, "all"), (33, 7, "all"), (1000, 7, "some"), (1000, 8, "twice"), (1000, 9, "some"), (777, 27, "some"),
    (777, 27, "twice")])
def test_outer_product_rows(hz, n, width, diag):
    """The outer product on slices of up to 256 entries and on the row blocks:
    rows without a diagonal entry or without any, a diagonal stored twice."""
    A = banded(n, width, 5 * n + width, diag=diag)
    mu, x = K.vectors(n, 21)
    M = hz.Matrix.from_csr(A)
    g = host(hz.outer_on_pattern(M, dev(mu), dev(x)))
    rows = np.repeat(np.arange(n), np.diff(A.rowptr))
    # two products and a sum per component
    assert np.all(np.abs(g + np.conj(mu[rows] * x[A.col])) <= 4 * 2.0 ** -53 * np.abs(mu[rows]) * np.abs(x[A.col]))
    M.close()


@pytest.mark.parametrize("slices_per_sm,width,slices", [
    (1.0, 39, True), (1.0, 40, False), (1.5, 40, False), (1.52, 40, True), (2.5, 52, True), (2.5, 53, False),
    (2.52, 53, True), (5.0, 41, True)])
def test_few_wide_slices(hz, oracle, slices_per_sm, width, slices):
    """A product by itself reads the row blocks where the slices are few and
    wide (complex64: above 40 steps up to 5 slices per SM); a solve on chip of
    the same handle reads the slices."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 32 * int(np.ceil(slices_per_sm * sms) if slices else slices_per_sm * sms)
    A = banded(n, width, width, real=False)
    A.val[A.col == np.repeat(np.arange(n), np.diff(A.rowptr))] += 4.0 * width   # (for the solve)
    x = K.vectors(n, 23)[0]
    assert on_slices(hz, A, x) == slices
    M = hz.Matrix.from_csr(A, c64=True)
    assert np.all(np.abs(host(hz.zspmv(M, dev(x))) - oracle.zspmv(A, x)) <= bound(A, x))
    x32 = x.astype(np.complex64)
    err = np.abs(host(hz.cspmv(M, dev(x32))) - oracle.cspmv(A, x32))
    assert np.all(err <= bound(A, x32.astype(np.complex128), 2.0 ** -23))
    for kw in (dict(), dict(mode="mixed"), dict(method="bicgstabl")):
        y, info = hz.zsolve(M, dev(x), tol=1e-11, maxit=100, **kw)
        assert info.status == 0
        assert np.linalg.norm(x - oracle.zspmv(A, host(y))) <= 2e-11 * np.linalg.norm(x)
    M.close()
