"""The excess attitude noise on short buckets, FP64 form: the order statistics of runs around the
length where a lane per run gives way to a warp per run (equal to the oracle's estimate, whose products,
differences and interpolation are rounded alike), and the next source update, whose sigma differs
per observation, against the oracle's from the same state and noise.
"""
import numpy as np
import pytest

import synth
from oracle import agis as OG
from oracle import attnoise as OAN
from oracle import blocks as OB
from oracle import model as OM
from parity_tol import assert_stats_close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def data():
    ds = synth.simulate(synth.config("small1yr", n_src=400, seed=31, min_transits=8))
    return ds.subset_sources(np.arange(ds.n_src))


@pytest.mark.parametrize("bucket_s,weight_fn", [(240, "agis"), (3 * 3600, "huber"), (5 * 3600, "agis"), (12 * 3600, "agis")])
def test_short_buckets_match_oracle(data, bucket_s, weight_fn):
    import paper_1112_4139_gb300 as pkg
    pkg.build()
    from paper_1112_4139_gb300 import agis
    ds, bucket_ns = data, bucket_s * 10**9
    P = OM.problem_from_dataset(ds)
    st = OB.Settings(weight_fn=weight_fn)
    g = agis.from_dataset(ds, weight_fn=0 if weight_fn == "agis" else 1)
    g.set_state(src=ds.src0, att=ds.att_true, cal=ds.cal_true)
    g.set_attnoise(bucket_ns)
    g.source_update()
    eps2 = g.attnoise()
    R0, src1 = g.residuals()[0], g.sources()
    sig2 = P.sigma.astype(np.float64) ** 2
    comp, bucket = OAN.component(P.kind, P.fov), OAN.bucket_of(P.t_ns, P.knot0_ns, bucket_ns)
    lengths = np.bincount(comp * eps2.shape[1] + bucket, minlength=eps2.size)
    want = {240: 1, 3 * 3600: 24, 5 * 3600: 25, 12 * 3600: 32}[bucket_s]
    assert (lengths == 0).any() and (lengths >= want).any()
    est = OAN.estimate(R0, sig2, g.source_stats()["eps2"][P.src], comp, bucket, eps2.shape[1])
    assert np.array_equal(eps2, est)
    # sigma~ differs per observation
    sig2 = OAN.adjusted_variance(sig2, eps2, comp, bucket)
    src2, sres, _ = OB.source_update(P, src1, ds.att_true, ds.cal_true, st, sig2=sig2)
    g.source_update()
    ss, (R, W) = g.source_stats(), g.residuals()
    e = OG.source_errors(g.sources(), src2)
    g.close()
    assert np.max(np.abs(e)) < 0.5 * synth.UAS       # the parity bound of the source parameters
    assert np.array_equal(ss["nu"].astype(int), sres.nu) and np.array_equal(ss["n_out"].astype(int), sres.n_out)
    # R = h - A d inherits the rounding of d: 1e-3 uas, as in the parity tests
    assert np.all(np.abs(R - sres.R) <= 1e-9 * np.abs(sres.R) + 1e-3 * synth.UAS)
    assert_stats_close(P.src, P.n_src, np.sqrt(sig2), sres.R, R, sres.W, W, sres.eps2, ss["eps2"], sres.Qi, ss["Q"])
