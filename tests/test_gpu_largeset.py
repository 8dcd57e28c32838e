"""A set large enough for the forms that round otherwise (2^25 observations): its source update against the
oracle's, wrong-field rows among them, and the number of kernels by form.
"""
import dataclasses

import numpy as np
import pytest

import synth
from oracle import agis as OG
from oracle import blocks as OB
from oracle import model as OM
from parity_tol import stat_tolerances

pytestmark = pytest.mark.gpu

N_CMP = 60     # the sources compared with the oracle (the first ones)


@pytest.fixture(scope="module")
def one():
    return synth.simulate(synth.config("small1yr", n_src=40_000, seed=5, min_transits=52))


def _tiled(one, times):
    src = np.concatenate([one.src + k * one.n_src for k in range(times)]).astype(np.int32)
    return dataclasses.replace(one, src=src, **{k: np.concatenate([getattr(one, k)] * times) for k in (
        "t_ns", "ccd", "fov", "kind", "sigma", "mu", "noise", "gate", "src_true", "src_mag", "n_transits", "src0")})


def _solve(ds):
    import paper_1112_4139_gb300 as pkg
    pkg.build()
    from paper_1112_4139_gb300 import agis
    g = agis.from_dataset(ds)
    g.set_state(src=ds.src0, att=ds.att_true, cal=ds.cal_true)
    g.source_update()
    out = g.source_kernels(), g.source_stats(), g.residuals(), g.sources()
    g.close()
    return out


def differences(P, ref, R, W, eps2, Q):
    """|difference| and tolerance (tests/parity_tol.py) of W, Q and eps^2.  The weights are those of the round before
    the last residuals, so a row's own last difference, which may be small by chance, does not bound its
    weight's: every row takes the largest one of its source."""
    big = np.maximum.reduceat(np.abs(R - ref.R), P.src_offsets()[:-1])[P.src]
    tol_Q, tol_e, tol_W = stat_tolerances(P.src, P.n_src, P.sigma, ref.R, ref.R + big, ref.W, ref.eps2, ref.Qi)
    return (np.abs(W - ref.W), tol_W), (np.abs(Q - ref.Qi), tol_Q), (np.abs(eps2 - ref.eps2), tol_e)


def test_large_set_matches_oracle(one):
    times = -(-(1 << 25) // one.n_obs)
    assert (1 << 25) <= times * one.n_obs < 1.05 * (1 << 25) and one.n_obs >= 160 * one.n_src
    off = one.src_offsets()
    fov = one.fov.copy()
    for i in range(0, N_CMP, 2):          # one row and three in the other field: about 2 rad, 4e9 sigma
        fov[off[i] + np.array([5, 100, 400][:1 + 2 * (i % 4 == 0)])] ^= 1
    one = dataclasses.replace(one, fov=fov)
    sub = one.subset_sources(np.arange(N_CMP))
    P = OM.problem_from_dataset(sub)
    src1, sres, _ = OB.source_update(P, sub.src0, one.att_true, one.cal_true, OB.Settings())
    n, ss, (R, W), src = _solve(_tiled(one, times))
    assert n == 12          # corrections: a first pass, four rounds, five solves, two passes at the end
    ss = {k: v[:N_CMP] for k, v in ss.items()}
    R, W = R[:sub.n_obs], W[:sub.n_obs]
    assert np.max(np.abs(OG.source_errors(src[:N_CMP], src1))) < 0.5 * synth.UAS    # the parity bound
    assert np.array_equal(ss["nu"].astype(int), sres.nu) and np.array_equal(ss["n_out"].astype(int), sres.n_out)
    # R = h - A d inherits the rounding of d: 1e-3 uas, as in the parity tests
    assert np.all(np.abs(R - sres.R) <= 1e-9 * np.abs(sres.R) + 1e-3 * synth.UAS)
    for d, tol in differences(P, sres, R, W, ss["eps2"], ss["Q"]):
        assert np.all(d <= tol), (d - tol).max()


def test_smaller_sets_sum_every_row(one):
    # one copy less than 2^25 observations: the sums over all rows, and every copy the same bits
    times = (1 << 25) // one.n_obs
    a, b = _solve(_tiled(one, times)), _solve(one)
    assert a[0] == b[0] == 13
    for x, y in zip(a[2] + (a[3],), b[2] + (b[3],)):
        assert np.array_equal(x[:len(y)], y)
