"""Interval blocks by moments, entry by entry: small components of g, weights that spread, weights that
depend on the time within the interval or on the component, each entry's error against extended sums
relative to its place in the matrix (the root of its two diagonal entries) beside that of the products' sums.
"""
import numpy as np
import pytest
from test_gpu_attmoments import _run, probe  # noqa: F401

pytestmark = pytest.mark.gpu

DT = 240 * 10**9
N_IV = 400


def _scale(shape, u):
    rng = np.random.default_rng(41)

    def scale(W, R, g, iv):
        if shape == "component":
            g = g * np.array([1, 1e-3, 1, 30])
        elif shape == "spread":
            W = W * 2.0 ** rng.uniform(-10, 0, W.size)
        elif shape == "late":            # large weights early in the interval
            W = W * np.where(u > 0.4, 2.0 ** -10, 1.0)
        elif shape == "crossed":         # large weights where the first component is small
            big = rng.random(W.size) < 0.3
            W = np.where(big, W, W * 2.0 ** -9)
            g = g * np.where(big[:, None], np.array([1e-3, 1, 1, 1]), 1.0)
        return W, R / np.sqrt(W / 1e18), g
    return scale


@pytest.mark.parametrize("n", [24, 54, 156])
@pytest.mark.parametrize("shape", ["plain", "component", "spread", "late", "crossed"])
def test_every_entry_as_exact_as_the_products_sums(probe, shape, n):  # noqa: F811
    counts = (n,) * N_IV
    u = np.random.default_rng(1).integers(0, DT, n * N_IV) / DT      # as _run draws them
    d, m, ref, mag, off, W, R, g = _run(probe, counts, DT, 1e-6, scale=_scale(shape, u))
    iu = np.triu_indices(16)
    diag = ref[:, [k for k in range(136) if iu[0][k] == iu[1][k]]].astype(float)
    wr2 = np.add.reduceat(W * R * R, off[:-1])
    place = np.concatenate([np.sqrt(diag[:, iu[0]] * diag[:, iu[1]]), np.sqrt(diag * wr2[:, None])], 1)
    rms = lambda v: np.sqrt(np.mean(((v - ref).astype(float) / place)[2:-2] ** 2, 0))  # noqa: E731
    # the two root mean squares of 396 intervals each vary by 4%: 1.25 is over four times their ratio's
    assert (rms(m) <= 1.25 * rms(d)).all(), (rms(m) / rms(d)).max()
    if shape == "plain":
        assert not np.array_equal(m, d)
