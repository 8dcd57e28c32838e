"""The S block's direct class sums, a block per source, against the oracle's source update: numbers of
AL and AC rows around its chunks of 32 rows and its groups of 512, sources with one class alone,
robust and plain weights.
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

# rows of the two classes: chunk edges, one class alone, 16 and 17 chunks, two groups and three
SIZES = [(60, 12), (63, 1), (64, 32), (65, 33), (96, 0), (0, 160), (479, 32), (480, 31), (480, 33), (481, 1), (512, 0),
         (511, 512), (513, 40), (600, 450), (1024, 100), (1025, 0), (1300, 290)]


@pytest.mark.parametrize("robust,weight_fn", [(1, "agis"), (1, "huber"), (0, "agis")])
def test_direct_sums_match_oracle(robust, weight_fn):
    import paper_1112_4139_gb300 as pkg
    pkg.build()
    from paper_1112_4139_gb300 import agis
    ds = synth.simulate(synth.config("small1yr", n_src=60, seed=17, min_transits=10))
    off, rng = ds.src_offsets(), np.random.default_rng(4)
    keep = []
    for i in range(ds.n_src):
        rows = np.arange(off[i], off[i + 1])
        if i < len(SIZES):      # that many rows of each class, drawn over the whole year
            parts = [rng.choice(rows[ds.kind[rows] == k], m) if m else rows[:0] for k, m in enumerate(SIZES[i])]
            rows = np.concatenate(parts)
            rows = rows[np.argsort(ds.t_ns[rows], kind="stable")]
        keep.append(rows)
    keep = np.concatenate(keep)
    sel = lambda a: np.ascontiguousarray(a[keep])  # noqa: E731
    ds = dataclasses.replace(ds, **{k: sel(getattr(ds, k)) for k in ("t_ns", "src", "ccd", "fov", "kind", "sigma", "mu",
                                                                     "noise", "gate")})
    # noise of their own for the repeated rows
    ds = dataclasses.replace(ds, t_ns=ds.t_ns + np.random.default_rng(5).integers(-2000, 2000, ds.n_obs))
    P = OM.problem_from_dataset(ds)
    src1, sres, _ = OB.source_update(P, ds.src0, ds.att_true, ds.cal_true, OB.Settings(weight_fn=weight_fn, robust=bool(robust)))
    g = agis.from_dataset(ds, weight_fn=0 if weight_fn == "agis" else 1, robust=robust)
    g.set_state(src=ds.src0, att=ds.att_true, cal=ds.cal_true)
    g.source_update()
    ss, (R, W) = g.source_stats(), g.residuals()
    e = OG.source_errors(g.sources(), src1)
    g.close()
    few = np.bincount(P.src[P.kind == 0], minlength=P.n_src) < 20     # AC alone: weakly determined, not compared in parameters
    assert few.sum() < 6
    assert np.max(np.abs(e[~few])) < 0.5 * synth.UAS       # the parity bound of the source parameters
    assert np.array_equal(ss["nu"].astype(int), sres.nu) and np.array_equal(ss["n_out"].astype(int), sres.n_out)
    ok = ~few[P.src]
    # R = h - A d inherits the rounding of d: 1e-3 uas, as in the parity tests
    assert np.all(np.abs(R - sres.R)[ok] <= 1e-9 * np.abs(sres.R[ok]) + 1e-3 * synth.UAS)
    z = lambda a: np.where(few, 0, a)  # noqa: E731
    assert_stats_close(P.src[ok], P.n_src, P.sigma[ok], sres.R[ok], R[ok], sres.W[ok], W[ok], z(sres.eps2), z(ss["eps2"]),
                       z(sres.Qi), z(ss["Q"]))
