"""The banded attitude solve on given normals (through the exchange calls of a source partition),
against the oracle's robust band Cholesky, at the sizes where its window, its rings and its
segments begin and end, with and without rank defects; and its integer reciprocal.
"""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

import synth
from oracle import cholesky as CH

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def _segments(n_coef, seg_len, L):
    K = n_coef - 3
    n_seg = max(1, -(-K // seg_len))
    for k in range(n_seg):
        x0, x1 = 3 + k * seg_len, 3 + (k + 1) * seg_len
        yield (max(3, x0 - L), min(n_coef - 1, x1 + L - 1), 0 if k == 0 else x0 - 1,
               n_coef - 1 if k == n_seg - 1 else x1 - 2)


# intervals (n_coef - 3), segment length, overlap, intervals without observations
CASES = [(1, 720, 12, ()), (2, 720, 12, ()), (4, 720, 12, ()), (5, 1, 0, ()), (13, 4, 2, ()), (17, 16, 12, ()),
         (31, 7, 3, ()), (64, 20, 12, range(30, 42)), (40, 720, 12, range(0, 6)), (40, 9, 5, range(33, 40)),
         (700, 2, 1, ())]


@pytest.mark.parametrize("n_iv,seg_len,L,empty", CASES)
def test_band_solve_matches_oracle(n_iv, seg_len, L, empty):
    import paper_1112_4139_gb300 as pkg
    pkg.build()
    from paper_1112_4139_gb300 import agis
    rng = np.random.default_rng(n_iv * 1000 + seg_len)
    ds = synth.simulate(synth.config("small1yr", n_src=60, span_days=n_iv / 24.0, seed=3))
    n_coef = n_iv + 3
    assert ds.n_coef == n_coef
    # one sparse and one well determined set of observations per interval: blocks J'J, rhs -J'R
    blk = np.zeros((n_iv, 152))
    iu = np.triu_indices(16)
    for i in range(n_iv):
        if i in empty:
            continue
        J = rng.normal(size=(20, 16)) * 10.0 ** rng.uniform(-1, 1)
        blk[i, :136] = (J.T @ J)[iu]
        blk[i, 136:] = J.T @ rng.normal(size=20)
    g = agis.from_dataset(ds, seg_len=seg_len, seg_overlap=L)
    g.set_exchange(agis.X_ATTITUDE, blk.reshape(-1))
    st = g.solve_exchange(agis.X_ATTITUDE)
    got = g.attitude() - ds.att0
    g.close()
    ref, rd = np.zeros((n_coef, 4)), 0
    cond = 1.0
    for lo, hi, u_lo, u_hi in _segments(n_coef, seg_len, L):
        n = 4 * (hi - lo + 4)
        Nb, b = np.zeros((n, 16)), np.zeros(n)
        for iv in range(lo - 3, hi - 2):
            r0 = 4 * (iv - (lo - 3))
            for (i, j), v in zip(zip(*iu), blk[iv, :136]):
                Nb[r0 + i, j - i] += v
            b[r0:r0 + 16] += blk[iv, 136:]
        x, _, d = CH.band_solve(Nb, b)
        rd += d
        s = np.linalg.svd(CH.band_to_dense(Nb), compute_uv=False)
        cond = max(cond, s[0] / s[s > 1e-11 * s[0]][-1])
        ref[u_lo:u_hi + 1] = x.reshape(-1, 4)[u_lo - (lo - 3):u_hi - (lo - 3) + 1]
    assert st["rank_defect"] == rd and (rd > 0) == (len(empty) > 0)
    # both are backward stable: each differs from the solution by a small multiple of cond eps of the
    # largest entry (n of up to 2812 rows of 15 products), and the attitude adds its own rounding
    tol = 100 * cond * np.finfo(float).eps * np.abs(ref).max() + 2 * np.finfo(float).eps
    assert np.abs(got - ref).max() < tol, (np.abs(got - ref).max(), tol)


@pytest.fixture(scope="module")
def rcp(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    out = str(tmp_path_factory.mktemp("rcp") / "librcp_int.so")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared",
                    "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_1112_4139_gb300", "csrc"),
                    os.path.join(HERE, "gpu_unit", "rcp_int_probe.cu"), "-o", out], check=True)
    lib = C.CDLL(out)
    lib.rcp_int_eval.argtypes = [C.c_void_p, C.c_void_p, C.c_void_p, C.c_int64]
    return lib


def test_integer_reciprocal_within_one_ulp_of_division(rcp):
    rng = np.random.default_rng(8)
    p2 = 2.0 ** np.arange(-100, 101)
    d = np.concatenate([2.0 ** rng.uniform(-100, 101, 2_000_000), rng.uniform(1.0, 2.0, 500_000),
                        1.0 + np.arange(4096) * 2.0 ** -52, 2.0 - np.arange(1, 4097) * 2.0 ** -52,
                        np.nextafter(p2, 0), p2, np.nextafter(p2, np.inf), 2.0 ** np.arange(-1022, -100, 7.0),
                        2.0 ** np.arange(101, 1023, 7.0), [5e-324, 1e-310, 1.7e308]])
    y, q = np.empty_like(d), np.empty_like(d)
    assert rcp.rcp_int_eval(d.ctypes.data, y.ctypes.data, q.ctypes.data, d.size) == 0
    u = np.abs(y - q) / np.spacing(q)
    u[np.isinf(q) & (y == q)] = 0.0
    assert u.max() <= 1.0, f"largest difference {u.max()} ulp at d = {d[np.argmax(u)]!r}"
    out = (d < 2.0 ** -100) | (d >= 2.0 ** 101)
    assert np.array_equal(y[out], q[out])
