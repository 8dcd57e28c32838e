"""The FP64 S block's inner iteration with rows far out (a misidentified observation, a wrong field of
view: up to 4e9 sigma), in both forms of the weight rounds, against the oracle's on the same rows.  A
rejected row has no weight, so it must leave no trace in Q, eps^2, W or the parameters, however far out.
"""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

from oracle import blocks as OB
from parity_tol import assert_stats_close

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
SIGMA = 5e-10
SIZES = [0, 1, 31, 32, 33, 64, 65, 165, 512, 513, 820, 840, 1023, 1024, 1025, 2500]
FAR = [0.0, 1e4, 1e6, 1e8, 4e9]     # in sigma


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    out = str(tmp_path_factory.mktemp("far") / "libfar.so")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared",
                    "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_1112_4139_gb300", "csrc"),
                    os.path.join(HERE, "gpu_unit", "src_solve_probe.cu"), "-o", out], check=True)
    lib = C.CDLL(out)
    P = C.c_void_p
    lib.src_solve_eval.argtypes = [C.c_int] * 6 + [C.c_int64] + [P] * 10
    return lib


def rows_of(seed=11):
    """(off, nal, rows[h, A, sigma^2]) of sources of every size with 0, 1, 3 and 10 rows far out."""
    rng = np.random.default_rng(seed)
    out, nal = [], []
    for far in FAR:
        for count in ([0] if far == 0 else [1, 3, 10]):
            for n in SIZES:
                n_al = {64: 64, 65: 0}.get(n, int(0.9 * n))        # one class alone, or both
                sig = np.where(np.arange(n) < n_al, SIGMA, 5 * SIGMA)
                if n == 840:                                       # sigma differs within the classes
                    sig = sig * rng.uniform(1.0, 1.5, n)
                A = rng.standard_normal((n, 5))
                z = rng.standard_normal(n) + np.where(rng.random(n) < 0.02, rng.uniform(-40, 40, n), 0.0)
                if n > 12 * count:
                    at = rng.choice(n, count, replace=False)
                    z[at] += far * rng.choice([-1, 1], count) * rng.uniform(0.5, 1.0, count)
                h = z * sig + A @ (SIGMA * rng.standard_normal(5))
                out.append(np.column_stack([h, A, sig ** 2]))
                nal.append(n_al)
    off = np.concatenate([[0], np.cumsum([len(v) for v in out])]).astype(np.int64)
    return off, np.array(nal, np.int32), np.ascontiguousarray(np.concatenate(out))


def oracle_of(off, rows, st):
    n_src = len(off) - 1
    R, W = np.zeros(len(rows)), np.zeros(len(rows))
    d, eps2, Q = np.zeros((n_src, 5)), np.zeros(n_src), np.zeros(n_src)
    nu, n_out = np.zeros(n_src, int), np.zeros(n_src, int)
    for i in range(n_src):
        s = slice(off[i], off[i + 1])
        if s.start < s.stop:
            r = OB.source_update_one(rows[s, 1:6], rows[s, 0], rows[s, 6], st)
            R[s], W[s], d[i], eps2[i], Q[i], nu[i], n_out[i] = r["R"], r["W"], r["d"], r["eps2"], r["Qi"], r["nu"], r["n_out"]
    return R, W, d, eps2, Q, nu, n_out


def compare(off, rows, ref, got):
    """Both sides' (R, W, d, eps2, Q, nu, n_out) within the rounding of the sums: 1e-12 (tests/parity_tol.py)."""
    size = np.diff(off)
    ok = size >= 31                          # fewer rows: weakly determined
    src = np.repeat(np.arange(len(size)), size)
    sel, sig = ok[src], np.sqrt(rows[:, 6])
    R0, W0, d0, e0, Q0, nu0, out0 = ref
    R, W, d, e, Q, nu, out = got
    assert np.array_equal(nu[ok], nu0[ok]) and np.array_equal(out[ok], out0[ok])
    assert np.isfinite(d).all() and np.isfinite(R).all()
    # R = h - A d: relative to its terms (d follows the far rows with plain weights)
    terms = np.abs(rows[:, 0]) + (np.abs(rows[:, 1:6]) * np.abs(d0)[src]).sum(1) + sig
    assert np.all(np.abs(R - R0)[sel] <= 1e-12 * terms[sel])
    z = lambda v: np.where(ok, v, 0.0)  # noqa: E731
    # a weight function below the normal range (exp(-|z| / 3) beyond |z| = 2100) has no relative accuracy:
    # there both sides only have to be below it
    low = W0 * rows[:, 6] < 2.0 ** -1021
    assert np.all((W * rows[:, 6])[low & sel] < 2.0 ** -1020)
    W0, W = np.where(low, 0.0, W0), np.where(low, 0.0, W)
    return assert_stats_close(src[sel], len(size), sig[sel], R0[sel], R[sel], W0[sel], W[sel], z(e0), z(e), z(Q0), z(Q))


@pytest.mark.parametrize("corrections", [0, 1])
@pytest.mark.parametrize("robust,n_rounds,weight_fn", [(1, 4, "agis"), (1, 4, "huber"), (1, 0, "agis"), (0, 4, "agis")])
def test_far_rows_leave_no_trace(probe, robust, n_rounds, weight_fn, corrections):
    off, nal, rows = rows_of()
    n_src, n = len(nal), len(rows)
    ref = oracle_of(off, rows, OB.Settings(robust=bool(robust), n_rounds=n_rounds, weight_fn=weight_fn))
    s = np.zeros((n_src, 5))
    e, Q, R, W = np.zeros(n_src), np.zeros(n_src), np.zeros(n), np.zeros(n)
    nu, out = np.zeros(n_src, np.int32), np.zeros(n_src, np.int32)
    assert probe.src_solve_eval(robust, n_rounds, 3, 0 if weight_fn == "agis" else 1, corrections, n_src, n,
                                *[a.ctypes.data for a in (off, nal, rows, s, e, Q, nu, out, R, W)]) == 0
    compare(off, rows, ref, (R, W, s, e, Q, nu, out))


@pytest.mark.parametrize("corrections", [0, 1])
@pytest.mark.parametrize("start", [1e2, 1e3])
def test_start_far_off(probe, start, corrections):
    """Starting parameters far off (what a rejected proposal of 1000 sigma leaves): nothing becomes non-finite, and the
    forms differ from the oracle by no more than the cancellation of the class sums, 2^-53 of sum W h^2 a row."""
    off, nal, rows = rows_of()
    rng = np.random.default_rng(5)
    size = np.diff(off)
    src = np.repeat(np.arange(len(size)), size)
    rows[:, 0] += (rows[:, 1:6] * (start * SIGMA * rng.choice([-1.0, 1.0], (len(size), 5)))[src]).sum(1)
    keep = np.isin(src, np.flatnonzero(size >= 64)) & (np.abs(rows[:, 0]) < 100 * start * SIGMA)
    nal = np.array([np.count_nonzero(keep[off[i]:off[i] + nal[i]]) for i in range(len(size))], np.int32)
    size = np.array([np.count_nonzero(keep[off[i]:off[i + 1]]) for i in range(len(size))])
    rows, off = np.ascontiguousarray(rows[keep]), np.concatenate([[0], np.cumsum(size)]).astype(np.int64)
    src = np.repeat(np.arange(len(size)), size)
    n_src, n = len(nal), len(rows)
    R0, W0, d0, e0, Q0, nu0, out0 = oracle_of(off, rows, OB.Settings())
    s = np.zeros((n_src, 5))
    e, Q, R, W = np.zeros(n_src), np.zeros(n_src), np.zeros(n), np.zeros(n)
    nu, out = np.zeros(n_src, np.int32), np.zeros(n_src, np.int32)
    assert probe.src_solve_eval(1, 4, 3, 0, corrections, n_src, n,
                                *[a.ctypes.data for a in (off, nal, rows, s, e, Q, nu, out, R, W)]) == 0
    assert all(np.isfinite(v).all() for v in (s, e, Q, R, W))
    hh = np.bincount(src, W0 * rows[:, 0] ** 2, minlength=n_src)
    # the sums of 21 products, their expansion and the three noise steps: 256 roundings
    assert np.all(np.abs(Q - Q0) <= 256 * 2.0 ** -53 * hh + 1e-12 * Q0)
    terms = np.abs(rows[:, 0]) + (np.abs(rows[:, 1:6]) * np.abs(d0)[src]).sum(1) + np.sqrt(rows[:, 6])
    assert np.all(np.abs(R - R0) <= 1e-12 * terms)


@pytest.mark.parametrize("corrections", [0, 1])
@pytest.mark.parametrize("sign", [1, -1])        # what inf - inf gives on the GPU has the sign bit set
def test_a_row_that_is_not_a_number_has_no_weight(probe, sign, corrections):
    """One such residual among those of a source of one sigma per class and of one whose sigma differs: its own weight is
    not a number either (the pivots of its source fail, so the other rows keep theirs), and the other sources are as
    without it."""
    off, nal, rows = rows_of()
    n_src, n = len(nal), len(rows)
    hit = [10, 11]                                # 820 rows of one sigma per class, 840 that differ
    assert list(np.diff(off)[hit]) == [820, 840]

    def solve(rows):
        s = np.zeros((n_src, 5))
        e, Q, R, W = np.zeros(n_src), np.zeros(n_src), np.zeros(n), np.zeros(n)
        nu, out = np.zeros(n_src, np.int32), np.zeros(n_src, np.int32)
        assert probe.src_solve_eval(1, 4, 3, 0, corrections, n_src, n,
                                    *[a.ctypes.data for a in (off, nal, rows, s, e, Q, nu, out, R, W)]) == 0
        return s, Q, R, W
    bad = rows.copy()
    bad[off[hit] + 5, 0] = np.copysign(np.nan, sign)
    a, b = solve(bad), solve(rows)
    src = np.repeat(np.arange(n_src), np.diff(off))
    own = np.isin(src, hit)
    assert np.isnan(a[3][off[hit] + 5]).all() and np.isnan(a[2][off[hit] + 5]).all()
    other = ~np.isin(np.arange(n_src), hit)
    assert np.array_equal(a[0][other], b[0][other]) and np.array_equal(a[1][other], b[1][other])
    assert np.array_equal(a[2][~own], b[2][~own]) and np.array_equal(a[3][~own], b[3][~own])
