"""Solves as one persistent kernel (systems in the row-per-lane layout whose
vectors fit on chip) against the same solve on the graph of kernels, which a
handle switched to the unpacked kind takes: every method, sizes from one row to
the largest that fits and the first that does not, partial slices, CTAs that
own no, one or several slices, a matrix staged in shared memory or not.

The operator is diagonally dominant: A = d I + B with |d| >= 4 and row and
column sums of |B| at most 1, so ||A|| <= 5.2 and ||A^-1|| <= 1/3.  Two
solutions of relative residual tol differ by at most 2 tol ||A^-1|| ||b||, and
||b|| <= 5.2 ||x||: 3.5 tol ||x||."""

import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu
TOL = 1e-11


def operator(n, seed, bands=(1, 7, 40)):
    """Diagonal 4 + i and off-diagonals at the distances `bands`, of sizes
    whose sum over a row or a column is at most 1, some of them complex."""
    rng = np.random.default_rng(seed)
    off = [o for k in bands if k < n for o in (-k, k)]
    i = np.arange(n)
    cols, vals = [i], [np.full(n, 4.0 + 1.0j)]
    for o in off:
        c = i + o
        v = rng.uniform(-1, 1, n) / max(1, len(off)) + 0j
        if o == off[-1]:
            v[n // 2:] *= 1j
        cols.append(c)
        vals.append(v)
    c, v = np.stack(cols, 1), np.stack(vals, 1)
    ok = (c >= 0) & (c < n)
    order = np.argsort(np.where(ok, c, n + 1), axis=1, kind="stable")
    c, v, ok = (np.take_along_axis(q, order, 1) for q in (c, v, ok))
    rp = np.concatenate([[0], np.cumsum(ok.sum(1))]).astype(np.int32)
    return W.CSR(n, rp, c[ok].astype(np.int32), v[ok])


def vec(n, seed):
    rng = np.random.default_rng(seed)
    return torch.as_tensor(rng.standard_normal(n) + 1j * rng.standard_normal(n)).cuda()


METHODS = [dict(method="bicgstab"), dict(method="tfqmr"), dict(mode="mixed"),
           dict(method="bicgstab", precond="jacobi"), dict(method="tfqmr", precond="jacobi")]
# 12 x 512 = 6144 rows are the most of a binary64 cluster, 32 x 512 of a mixed
# one; 152 x 32 = 4864 rows give every SM one slice; 60 x 4864 is the most that
# BiCGStab in binary64 holds on chip, 47 x 4864 TFQMR
SIZES = [1, 2, 31, 33, 1000, 4864, 4865, 6144, 6145, 16384, 16385, 20011, 100003, 47 * 4864, 60 * 4864, 60 * 4864 + 1]


@pytest.mark.parametrize("n", SIZES)
def test_persistent_against_graph(hz, n):
    A = operator(n, n)
    b, x0 = vec(n, n + 1), vec(n, n + 2)
    for opt in METHODS if n <= 20011 else METHODS[:3]:
        sols = []
        for kind in ("flat64p", "flat64"):
            M = hz.Matrix.from_csr(A, c64=True)
            M.set_spmv(kind)
            hist = torch.zeros(201, dtype=torch.float64, device="cuda")
            x, info = hz.zsolve(M, b, x=x0.clone(), tol=TOL, maxit=200, hist=hist, **opt)
            assert info.status == 0 and info.relres_true <= TOL, (kind, opt, info)
            r = b - hz.zspmv(M, x)
            # b - A x again: rounding of both evaluations, (2 m + 4) 2^-52 of |A||x| + |b|
            assert abs(float(torch.linalg.vector_norm(r) / torch.linalg.vector_norm(b)) - info.relres_true) <= 2e-14
            sols.append((x, info, hist))
            M.close()
        (xa, ia, ha), (xb, ib, hb) = sols
        d = float(torch.linalg.vector_norm(xa - xb) / torch.linalg.vector_norm(xb))
        assert d <= 3.5 * TOL, (opt, d)
        assert abs(ia.iters - ib.iters) <= 2 + ib.iters // 4
        # the start's residual: sums in another order, n terms
        assert abs(float(ha[0] - hb[0])) <= 1e-12 * float(hb[0])


@pytest.mark.parametrize("opt", METHODS[:3])
def test_outcomes(hz, opt):
    n = 5000
    M = hz.Matrix.from_csr(operator(n, 3), c64=True)
    b, zero = vec(n, 4), torch.zeros(n, dtype=torch.complex128, device="cuda")
    x, info = hz.zsolve(M, zero, x=vec(n, 5), tol=TOL, maxit=50, **opt)
    assert info.status == 0 and info.iters == 0 and not bool(x.any())
    x, info = hz.zsolve(M, b, tol=TOL, maxit=0, **opt)
    assert info.status == 4 and info.iters == 0 and not bool(x.any())
    x, info = hz.zsolve(M, b, tol=1e-30, maxit=3, **opt)
    assert info.status == 4 and info.iters == 3
    bad = b.clone()
    bad[777] = complex(float("nan"), 0.0)
    x, info = hz.zsolve(M, bad, tol=TOL, maxit=50, **opt)
    assert info.status == 6
    x, info = hz.zsolve(M, b, tol=TOL, maxit=50, **opt)      # and the handle still solves
    assert info.status == 0
    y, again = hz.zsolve(M, b, tol=TOL, maxit=50, **opt)     # deterministic
    assert torch.equal(x, y) and again.iters == info.iters
    # a right-hand side whose squares are near the ends of the binary64 range
    for s in (2.0 ** -480, 2.0 ** 440):
        if opt.get("mode") != "mixed":
            z, info = hz.zsolve(M, b * s, tol=TOL, maxit=50, **opt)
            assert info.status == 0
            assert float(torch.linalg.vector_norm(z / s - x) / torch.linalg.vector_norm(x)) <= 3.5 * TOL
    M.close()


@pytest.mark.parametrize("sizes", [(4000,), (33, 20011, 1, 700), (300,) * 152, (300,) * 153, (290000, 40000)])
def test_sweep_against_single_solves(hz, sizes):
    """A sweep shares the SMs out among its systems (153 systems, and two that
    do not fit together, take the grid-wide phases); a start vector is used,
    and a zero right-hand side leaves it."""
    mats = [hz.Matrix.from_csr(operator(n, 7 + k)) for k, n in enumerate(sizes)]
    bs = [vec(n, 50 + k) for k, n in enumerate(sizes)]
    xs = [vec(n, 300 + k) for k, n in enumerate(sizes)]
    if len(sizes) == 4:
        bs[3].zero_()
        keep = xs[3].clone()
    xs, infos = hz.zsolve_batched(mats, bs, xs=xs, tol=TOL, maxit=200)
    for k, (M, b, x, info) in enumerate(zip(mats, bs, xs, infos)):
        assert info.status == 0, (k, info)
        if len(sizes) == 4 and k == 3:
            assert info.iters == 0 and torch.equal(x, keep)
        elif k < 4:
            y, _ = hz.zsolve(M, b, tol=TOL, maxit=200)
            assert float(torch.linalg.vector_norm(x - y) / torch.linalg.vector_norm(y)) <= 3.5 * TOL


@pytest.mark.parametrize("n", [3000, 20011, 200003])
def test_threads_and_streams(hz, n):
    """Solves from two host threads on streams of their own, each on its own
    handle (one cluster each; every SM each, vectors from a little to nearly
    all of their shared memory), give the answers of the same solves alone."""
    import threading

    mats = [hz.Matrix.from_csr(operator(n, 90 + k)) for k in range(2)]
    bs = [vec(n, 95 + k) for k in range(2)]
    alone = [hz.zsolve(M, b, tol=TOL, maxit=200)[0] for M, b in zip(mats, bs)]
    torch.cuda.synchronize()
    out, errors = [[], []], []

    def work(k):
        try:
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                for _ in range(20):
                    x, info = hz.zsolve(mats[k], bs[k], tol=TOL, maxit=200)
                    assert info.status == 0
                    out[k].append(x)
            s.synchronize()
        except Exception as e:   # reported below, in the main thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for k in range(2):
        assert len(out[k]) == 20 and all(torch.equal(x, alone[k]) for x in out[k])


@pytest.mark.parametrize("n", [1000, 20011])   # one cluster; every SM
@pytest.mark.parametrize("method", ["bicgstab", "tfqmr"])
def test_overflowing_ratio(hz, n, method):
    """A residual ratio that overflows while its square is finite ends the
    solve on every CTA alike, with a history (which one CTA writes) or without.

    ||b|| = 2^-530 and a start with ||r0|| = 1.5e308 ||b||; A = S + 0.01 I with
    S real and skew, so that alpha = 100 for a real r0 and the first step makes
    the residual larger (TFQMR's bound grows with sqrt(m + 1))."""
    i = np.arange(n - 1, dtype=np.int32)
    rows = np.concatenate([i, np.arange(n), i + 1])
    cols = np.concatenate([i + 1, np.arange(n), i])
    vals = np.concatenate([np.ones(n - 1), np.full(n, 0.01), -np.ones(n - 1)]) + 0j
    order = np.lexsort((cols, rows))
    rp = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=n))]).astype(np.int32)
    A = W.CSR(n, rp, cols[order].astype(np.int32), vals[order])
    x0 = np.random.default_rng(n).standard_normal(n) + 0j
    b = np.zeros(n, np.complex128)
    b[0] = 2.0 ** -530
    x0 *= 1.5e308 * 2.0 ** -530 / np.linalg.norm(A.to_scipy() @ x0)
    M = hz.Matrix.from_csr(A)
    for hist in (None, torch.zeros(51, dtype=torch.float64, device="cuda")):
        _, info = hz.zsolve(M, torch.as_tensor(b).cuda(), x=torch.as_tensor(x0).cuda(), tol=1e-10, maxit=50,
                            method=method, hist=hist)
        assert info.status == 6 and info.iters == 1, info
    assert np.isfinite(float(hist[0]))
    if method == "tfqmr":   # (BiCGStab ends in the half step, which writes none)
        assert not np.isfinite(float(hist[1]))
    M.close()


def test_threads_sweep_the_same_handles(hz):
    """Two host threads, on streams of their own, sweep over the same handles
    from their first sweep on (the workspace kept with the first handle serves
    one of them at a time): the answers are those of the sweep alone."""
    import threading

    mats = [hz.Matrix.from_csr(operator(n, 60 + n)) for n in (4865, 700, 9001)]
    bs = [vec(M.n, 70 + k) for k, M in enumerate(mats)]
    torch.cuda.synchronize()
    out, errors, gate = [[], []], [], threading.Barrier(2)

    def work(k):
        try:
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                gate.wait()
                for _ in range(20):
                    xs, infos = hz.zsolve_batched(mats, bs, tol=TOL, maxit=200)
                    assert all(i.status == 0 for i in infos)
                    out[k].append(xs)
            s.synchronize()
        except Exception as e:   # reported below, in the main thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    alone, _ = hz.zsolve_batched(mats, bs, tol=TOL, maxit=200)
    for o in out:
        assert len(o) == 20 and all(torch.equal(x, y) for xs in o for x, y in zip(xs, alone))


def unlike_the_graph(hz, mats, bs, x0s):
    """(solutions of a sweep, whether it ran on chip): the grid-wide phases give
    handles of either binary64 kind the same sums, a sweep on chip other ones."""
    out = []
    for kind in ("flat64p", "flat64"):
        for M in mats:
            M.set_spmv(kind)
        out.append(hz.zsolve_batched(mats, bs, xs=[x.clone() for x in x0s], tol=TOL, maxit=200))
    (xa, ia), (xb, _) = out
    for M in mats:
        M.set_spmv("flat64p")
    return xa, ia, not all(torch.equal(p, q) for p, q in zip(xa, xb))


@pytest.mark.parametrize("sizes,chip", [
    ((20011, 31, 4865, 700, 300), True),         # shares of 1 to 117 CTAs
    ((4865,) + (31,) * 140, True),               # small systems rounded up to one CTA each
    ((700,) * 151 + (1000,), True),              # one CTA each
    ((4865,) + (31,) * 152, False),              # more systems than SMs
    ((20011,) + (31,) * 150, False),             # two CTAs cannot hold the large one
    ((33, 20011, 1, 700), False)])               # padding keeps two of them off the layout
def test_sweep_shares(hz, sizes, chip):
    """Uneven sweeps: which of them run on chip, and every system against its
    single solve, from a start vector, a zero right-hand side among them."""
    mats = [hz.Matrix.from_csr(operator(n, 7 + k)) for k, n in enumerate(sizes)]
    bs = [vec(n, 50 + k) for k, n in enumerate(sizes)]
    x0s = [vec(n, 300 + k) for k, n in enumerate(sizes)]
    bs[3].zero_()
    xs, infos, on_chip = unlike_the_graph(hz, mats, bs, x0s)
    assert on_chip == chip
    for k, (M, b, x, info) in enumerate(zip(mats, bs, xs, infos)):
        assert info.status == 0, (k, info)
        if k == 3:
            assert info.iters == 0 and torch.equal(x, x0s[3])
        elif k < 6:
            y, one = hz.zsolve(M, b, x=x0s[k].clone(), tol=TOL, maxit=200)
            assert float(torch.linalg.vector_norm(x - y) / torch.linalg.vector_norm(y)) <= 3.5 * TOL
            assert abs(info.iters - one.iters) <= 2 + one.iters // 4
    for M in mats:
        M.close()


# sizes whose slices do not divide among a cluster's CTAs (some own none), and
# partial last slices; 1, 2 and 33 rows stay off the layout (padding)
@pytest.mark.parametrize("n,chip", [
    (1, False), (2, False), (33, False), (31, True), (32, True), (96, True), (160, True), (224, True), (290, True),
    (479, True), (513, True), (6143, True), (6177, True)])
def test_small_sizes_on_chip(hz, n, chip):
    """Which of the smallest systems are solved on chip (a solve by the graph
    gives handles of lane runs and of the unpacked kind the same sums), and
    their solutions against the graph's."""
    A = operator(n, n)
    b, x0 = vec(n, n + 1), vec(n, n + 2)
    for opt in METHODS + [dict(mode="mixed", precond="jacobi")]:
        out = []
        for kind in ("flat64p", "flat64"):
            M = hz.Matrix.from_csr(A, c64=True)
            M.set_spmv(kind)
            out.append(hz.zsolve(M, b, x=x0.clone(), tol=TOL, maxit=200, **opt))
            M.close()
        (x, i), (y, j) = out
        assert i.status == 0 and j.status == 0
        assert float(torch.linalg.vector_norm(x - y) / torch.linalg.vector_norm(y)) <= 3.5 * TOL
        if opt.get("mode") != "mixed":   # (complex64 products of both kinds read the slices)
            assert torch.equal(x, y) != chip, opt


@pytest.mark.parametrize("n", [1000, 20011])
@pytest.mark.parametrize("opt", METHODS[:2])
def test_history(hz, n, opt):
    """The whole residual history against the graph's.  One step's rounding is
    below 100 2^-53 (||A|| ||x|| + ||b||) ~ 1e-13 ||b||; the recurrences of this
    well-conditioned operator (condition below 16) may carry it on, so the two
    stay together within 1e-9 ||b||.  Entries past the end are not written."""
    A, b = operator(n, 3 * n), vec(n, 3 * n + 1)
    h = []
    for kind in ("flat64p", "flat64"):
        M = hz.Matrix.from_csr(A)
        M.set_spmv(kind)
        hist = torch.full((201,), -1.0, dtype=torch.float64, device="cuda")
        _, info = hz.zsolve(M, b, tol=TOL, maxit=200, hist=hist, **opt)
        assert info.status == 0 and info.restarts == 0
        v = hist.cpu().numpy()
        assert np.all(v[:info.iters + 1] >= 0.0) and np.all(v[info.iters + 1:] == -1.0)
        assert v[info.iters] == info.relres_rec
        h.append(v[:info.iters + 1])
        M.close()
    m = min(map(len, h))
    assert np.all(np.abs(h[0][:m] - h[1][:m]) <= 1e-9)


@pytest.mark.parametrize("n", [64, 9728])   # one cluster; every SM
@pytest.mark.parametrize("opt", METHODS[:3])
def test_breakdown(hz, n, opt):
    """Blocks [[0, 1], [-1, 0]] with b = (1, 0) in each: <r^, A r> = 0 in the
    first step.  The outcome is the graph's."""
    i = np.arange(n)
    A = W.CSR(n, np.arange(n + 1, dtype=np.int32), (i ^ 1).astype(np.int32), np.where(i % 2 == 0, 1.0, -1.0) + 0j)
    b = torch.as_tensor(np.where(i % 2 == 0, 1.0, 0.0) + 0j).cuda()
    out = []
    for kind in ("flat64p", "flat64"):
        M = hz.Matrix.from_csr(A, c64=True)
        M.set_spmv(kind)
        out.append(hz.zsolve(M, b, tol=TOL, maxit=50, **opt))
        M.close()
    (x, p), (y, q) = out
    assert (p.status, p.iters, p.outer) == (q.status, q.iters, q.outer) and p.status in (4, 5)
    assert p.relres_true == q.relres_true and torch.equal(x, y)
