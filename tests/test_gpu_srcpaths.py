"""The FP64 S block's weight rounds by corrections to unit-weight sums, and its order statistics,
against the oracle's source update on the same observations: long sources, sources around the
sizes of its lists and of its shared-memory keys, tied residuals (the radix select), and the
per-observation path among them.  (The direct class sums of shorter sources are those of the
parity tests.)
"""
import dataclasses

import numpy as np
import pytest

import synth
from oracle import agis as OG
from oracle import blocks as OB
from oracle import model as OM
from parity_tol import assert_stats_close

pytestmark = pytest.mark.gpu


N_CMP = 60     # the sources compared with the oracle (the first ones)


@pytest.fixture(scope="module")
def base():
    # sources with 52 transits or more in a year: above 512 observations per source; the same sources
    # 140 times, for more than 23M observations and 100 per knot interval (the lines of the dispatch)
    one = synth.simulate(synth.config("small1yr", n_src=40_000, seed=5, min_transits=52))
    tile = lambda a: np.concatenate([a] * 140)  # noqa: E731
    src = np.concatenate([one.src + k * one.n_src for k in range(140)]).astype(np.int32)
    ds = dataclasses.replace(one, src=src, **{k: tile(getattr(one, k)) for k in (
        "t_ns", "ccd", "fov", "kind", "sigma", "mu", "noise", "gate", "src_true", "src_mag", "n_transits", "src0")})
    assert ds.n_obs >= 23_500_000 and ds.n_obs >= 512 * ds.n_src and ds.n_obs >= 110 * (ds.n_coef - 3), (ds.n_obs, ds.n_src)
    return ds


def _cut(ds, keep):
    sel = lambda a: np.ascontiguousarray(a[keep])  # noqa: E731
    return dataclasses.replace(ds, t_ns=sel(ds.t_ns), src=sel(ds.src), ccd=sel(ds.ccd), fov=sel(ds.fov),
                               kind=sel(ds.kind), sigma=sel(ds.sigma), mu=sel(ds.mu), noise=sel(ds.noise), gate=sel(ds.gate))


@pytest.mark.parametrize("weight_fn", ["agis", "huber"])
@pytest.mark.parametrize("shape", ["long", "mixed", "tied", "varied", "offset"])
def test_source_update_matches_oracle(base, shape, weight_fn):
    import paper_1112_4139_gb300 as pkg
    pkg.build()
    from paper_1112_4139_gb300 import agis
    ds, off = base, base.src_offsets()
    if shape == "mixed":     # sources with none, with one, with few observations among long ones
        keep = np.ones(ds.n_obs, bool)
        for i, m in ((3, 0), (4, 1), (5, 31), (6, 32), (7, 33), (8, 64)):
            keep[off[i] + m:off[i + 1]] = False
        ds = _cut(ds, keep)
    elif shape == "tied":    # the compared sources' observations twice and more: tied order statistics, 1024 and more keys
        rep = np.concatenate([np.repeat(np.arange(o, e), 2 + k % 3) for k, (o, e) in
                              enumerate(zip(off[:N_CMP], off[1:N_CMP + 1]))])
        ds = _cut(ds, np.concatenate([rep, np.arange(off[N_CMP], ds.n_obs)]))
    elif shape == "varied":  # sigma differs within a class for every third source
        sig = ds.sigma.copy()
        sig[(ds.src % 3 == 0) & (np.arange(ds.n_obs) % 5 == 0)] *= np.float32(1.5)
        ds = dataclasses.replace(ds, sigma=sig)
    assert ds.n_obs >= 23_000_000 and ds.n_obs >= 512 * ds.n_src
    # attitude and calibration at the truth: residuals at the noise level, weights that differ
    sub = ds.subset_sources(np.arange(N_CMP))
    P = OM.problem_from_dataset(sub)
    # an offset of every residual by ten sigma: most rows are downweighted
    cal = ds.cal_true + (10.0 * float(np.median(ds.sigma)) if shape == "offset" else 0.0)
    src1, sres, _ = OB.source_update(P, sub.src0, ds.att_true, cal, OB.Settings(weight_fn=weight_fn))
    g = agis.from_dataset(ds, weight_fn=0 if weight_fn == "agis" else 1)
    g.set_state(src=ds.src0, att=ds.att_true, cal=cal)
    g.source_update()
    ss = {k: v[:N_CMP] for k, v in g.source_stats().items()}
    R, W = (v[:sub.n_obs] for v in g.residuals())
    few = np.bincount(P.src, minlength=N_CMP) < 66      # weakly determined: not compared
    e = OG.source_errors(g.sources()[:N_CMP], src1)
    g.close()
    assert np.max(np.abs(e[~few])) < 0.5 * synth.UAS       # the parity bound of the source parameters
    assert np.array_equal(ss["nu"][~few].astype(int), sres.nu[~few])
    assert np.array_equal(ss["n_out"][~few].astype(int), sres.n_out[~few])
    ok = ~few[P.src]
    # R = h - A d inherits the rounding of d: 1e-3 uas, as in the parity tests
    assert np.all(np.abs(R - sres.R)[ok] <= 1e-9 * np.abs(sres.R[ok]) + 1e-3 * synth.UAS)
    assert_stats_close(P.src[ok], N_CMP, P.sigma[ok], sres.R[ok], R[ok], sres.W[ok], W[ok],
                       np.where(few, 0, sres.eps2), np.where(few, 0, ss["eps2"]), np.where(few, 0, sres.Qi),
                       np.where(few, 0, ss["Q"]))
