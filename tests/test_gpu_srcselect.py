"""The quantile select of the source updates: the order statistics exactly, and one decision by all
lanes of a warp where a step of the histogram holds too many keys (ties, one value far out), since
the radix select that follows clears that histogram.
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
CAP = 96          # keys around a quantile that are ranked directly


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    out = str(tmp_path_factory.mktemp("sel") / "libsel.so")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared",
                    "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_1112_4139_gb300", "csrc"),
                    os.path.join(HERE, "gpu_unit", "select_probe.cu"), "-o", out], check=True)
    lib = C.CDLL(out)
    P = C.c_void_p
    lib.select_eval.argtypes = [C.c_int, C.c_int64, P, P, P, P]
    return lib


@pytest.mark.parametrize("shape", ["normal", "tied", "far"])
def test_select_is_exact_and_of_one_mind(probe, shape):
    rng = np.random.default_rng(3)
    sizes = [2, 3, 31, 32, 33, 96, 97, 98, 200, 500, 1023, 1024] + [int(v) for v in rng.integers(100, 1025, 2000)]
    sets = [rng.standard_normal(n) for n in sizes]
    if shape == "tied":
        sets = [np.round(2 * v) if len(v) > 3 else v for v in sets]
    elif shape == "far":
        for v in sets:
            v[rng.integers(v.size)] = rng.choice([-1, 1]) * 10.0 ** rng.uniform(3, 10)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    x = np.concatenate(sets)
    ok, q = np.full((len(sizes), 32), -1, np.int32), np.empty((len(sizes), 4))
    assert probe.select_eval(len(sizes), x.size, off.ctypes.data, x.ctypes.data, ok.ctypes.data, q.ctypes.data) == 0
    assert (ok == ok[:, :1]).all()
    done = ok[:, 0] == 1
    for i, v in enumerate(sets):
        n, s = v.size, np.sort(v)
        if done[i]:
            k = [int(np.floor(p * (n - 1))) for p in (1 / 6, 5 / 6)]
            assert np.array_equal(q[i], s[[k[0], min(k[0] + 1, n - 1), k[1], min(k[1] + 1, n - 1)]])
        else:
            assert n > CAP
    if shape == "far":
        assert not done[np.array(sizes) > 3 * CAP].any()      # one or two steps hold all but a few
    elif shape == "normal":
        assert done.all()
    else:
        assert done.any() and not done.all()
