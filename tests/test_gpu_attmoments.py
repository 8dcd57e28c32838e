"""Interval blocks of the FP64 attitude update by moments on the tensor cores, against sums in
extended precision: numbers of observations around the kernel's chunk, its shortest interval and
its longest exact accumulation, knot intervals of other lengths, magnitudes that spread, and the
intervals that must take the sums of the products (the ends, uncovered ones, values out of range).
"""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
LD = np.longdouble
NUM = np.array([[1, -3, 3, -1], [23, -15, -3, 3], [23, 15, -3, -3], [1, 3, 3, 1]])
COUNTS = (0, 1, 23, 24, 25, 31, 32, 33, 63, 64, 65, 156, 511, 512, 513, 1500)


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    out = str(tmp_path_factory.mktemp("mom") / "libmom.so")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared",
                    "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_1112_4139_gb300", "csrc"),
                    os.path.join(HERE, "gpu_unit", "att_moments_probe.cu"), "-o", out], check=True)
    lib = C.CDLL(out)
    P = C.c_void_p
    lib.att_blocks_eval.argtypes = [C.c_int64, C.c_int64, C.c_int, C.c_double, C.c_int64, P, P, P, P, P, P, P, P]
    return lib


def _run(probe, counts, dt, lam2, u_lo=0.0, u_hi=1.0, scale=None, seed=1):
    """Blocks of both kernels, of the extended sums, and the sums' magnitudes; intervals on axis 0."""
    rng = np.random.default_rng(seed)
    n_iv, knot0 = len(counts), 1_234_567_890_123
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    n = int(off[-1])
    iv = np.repeat(np.arange(n_iv), counts)
    u = rng.integers(int(u_lo * dt), max(int(u_hi * dt), int(u_lo * dt) + 1), n)
    t = (knot0 + iv * dt + u).astype(np.int64)
    W = 1e18 * np.where(rng.random(n) < 0.15, 0.04, 1.0) * rng.uniform(0.01, 1.0, n)
    R = 1e-9 * rng.standard_normal(n)
    g = rng.standard_normal((n, 4))
    if scale is not None:
        W, R, g = scale(W, R, g, iv)
    att = rng.standard_normal((n_iv + 3, 4))
    att /= np.linalg.norm(att, axis=1)[:, None]
    d, m = np.empty((n_iv, 152)), np.empty((n_iv, 152))
    arrs = [np.ascontiguousarray(a) for a in (t, R, W, g, off, att)]
    assert probe.att_blocks_eval(knot0, dt, n_iv + 3, lam2, n, *[a.ctypes.data for a in arrs], d.ctypes.data, m.ctypes.data) == 0
    x = (LD(2) * u.astype(LD) - LD(dt)) / LD(dt)
    B = np.stack([sum(int(NUM[b, k]) * x ** k for k in range(4)) / LD(48) for b in range(4)], 1)
    ref, mag = np.zeros((n_iv, 152), LD), np.zeros((n_iv, 152), LD)
    for i in range(n_iv):
        s = slice(off[i], off[i + 1])
        Bs, Ws, gs = B[s], W[s].astype(LD), g[s].astype(LD)
        q = Bs @ att[i:i + 4].astype(LD)
        rows = [Bs[:, :, None] * v[:, None, :] for v in (gs, q)]   # B_b v_c, index 4 b + c
        full = [np.einsum("oi,oj->oij", r.reshape(-1, 16), r.reshape(-1, 16)) for r in rows]
        Wx = Ws[:, None, None]
        A = (Wx * (full[0] + 4 * LD(lam2) * full[1])).sum(0)
        Am = (np.abs(Wx) * (np.abs(full[0]) + 4 * LD(lam2) * np.abs(full[1]))).sum(0)
        # right-hand side: no sign convention but that of the direct kernel
        y = (Ws[:, None] * R[s].astype(LD)[:, None] * rows[0].reshape(-1, 16))
        iu = np.triu_indices(16)
        ref[i, :136], mag[i, :136] = A[iu], Am[iu]
        ref[i, 136:], mag[i, 136:] = -y.sum(0), np.abs(y).sum(0)
    return d, m, ref, mag, off, W, R, g


def _bound(off, W, R, g, lam2):
    # every row value is rounded at 2^-56, every column value at 2^-55 of its largest one (at most 1), the digit pairs left out are
    # below 2^-58, and the products before the digits are cut at 2^-59: below 2^-53 per observation and
    # moment, times the coefficients' sum over the columns' scales (below 1.2); then 2^-52 per operation of
    # the FP64 expansion, 30 of them, on terms that sum to the moments' bound
    out = np.zeros((len(off) - 1, 152))
    for i in range(len(off) - 1):
        s = slice(off[i], off[i + 1])
        if s.start == s.stop:
            continue
        w, r, gg, n = np.abs(W[s]).max(), np.abs(W[s] * R[s]).max(), np.abs(g[s]).max(), s.stop - s.start
        out[i, :136] = n * w * (4 * gg ** 2 + 4 * lam2 * 16) * 32 * 2.0 ** -53
        out[i, 136:] = n * 2 * r * 2 * gg * 32 * 2.0 ** -53
    return out


def _within(m, ref, bound):
    # the extended sums hold the splines of regular intervals: not the two at each end
    return (np.abs(m - ref).astype(float) <= bound)[2:-2].all()


@pytest.mark.parametrize("dt_s,lam2,u_lo,u_hi", [(240.0, 1e-6, 0.0, 1.0), (1000.0, 2.0 ** -6, 0.0, 1.0), (30.0, 0.0, 0.0, 1.0),
                                                 (2.0 ** 40 / 1e9, 1e-6, 0.0, 1.0), (86400.0, 1e-6, 0.0, 1.0),
                                                 (240.0, 1e-6, 0.0, 0.4), (240.0, 1e-6, 0.6, 1.0), (240.0, 1e-6, 0.4, 0.6)])
def test_moments_match_extended_sums(probe, dt_s, lam2, u_lo, u_hi):
    counts = (40, 40) + COUNTS + (90,) * 200 + (40, 40)
    dt = int(round(dt_s * 1e9))
    d, m, ref, mag, off, W, R, g = _run(probe, counts, dt, lam2, u_lo, u_hi)
    assert _within(m, ref, _bound(off, W, R, g, lam2))
    # no less accurate than the sums of the products, over the covered intervals
    e = lambda v: np.sqrt(np.mean((np.abs(v - ref) / mag)[18:-2].astype(float) ** 2))  # noqa: E731
    assert e(m) <= e(d)
    # ends and short intervals: the products' sums, bit for bit
    same = [0, 1, 2, 3, 4, len(counts) - 2, len(counts) - 1]
    assert np.array_equal(d[same], m[same])
    assert not np.array_equal(d[5:18], m[5:18])


def test_spread_magnitudes(probe):
    def scale(W, R, g, iv):
        rng = np.random.default_rng(9)
        return W * 2.0 ** rng.uniform(-40, 0, W.size), R * 2.0 ** rng.uniform(-20, 20, W.size), g * np.array([1, 1e-3, 1, 1])
    d, m, ref, mag, off, W, R, g = _run(probe, (60,) * 100, 240 * 10**9, 1e-6, scale=scale)
    assert _within(m, ref, _bound(off, W, R, g, 1e-6))


@pytest.mark.parametrize("case", ["one end", "other end", "large lambda", "zero weights", "huge", "tiny", "nan", "inf"])
def test_other_intervals_sum_the_products(probe, case):
    lo, hi = {"one end": (0.0, 0.2), "other end": (0.8, 1.0)}.get(case, (0.0, 1.0))

    def scale(W, R, g, iv):
        if case == "zero weights":
            W = 0.0 * W
        elif case == "huge":
            g = g * 1e90
        elif case == "tiny":
            W = W * 1e-110
        elif case in ("nan", "inf"):
            R = R.copy()
            R[np.unique(iv, return_index=True)[1] + 5] = np.nan if case == "nan" else np.inf
        return W, R, g
    d, m, *_ = _run(probe, (60,) * 30, 240 * 10**9, 0.016 if case == "large lambda" else 1e-6, lo, hi, scale)
    assert np.array_equal(d, m, equal_nan=True)


def test_zero_residuals(probe):
    d, m, ref, mag, off, W, R, g = _run(probe, (60,) * 30, 240 * 10**9, 1e-6, scale=lambda W, R, g, iv: (W, 0 * R, g))
    assert (m[:, 136:] == 0).all() and _within(m, ref, _bound(off, W, R, g, 1e-6))
