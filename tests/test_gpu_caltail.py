"""The calibration update's projection, its rank count and the source statistics against the oracle and
numpy, at the numbers of calibration intervals where their blocks change: groups of eight
intervals, 8192 parameters, more than 256 sources in a chunk.
"""
import numpy as np
import pytest

import synth
from oracle import agis as OG  # noqa: F401
from oracle import blocks as OB
from oracle import model as OM

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("span_days,n_src", [(1, 3000), (7, 2000), (8, 2000), (9, 1000), (59, 500), (60, 300), (70, 100)])
def test_projection_and_counts(span_days, n_src):
    import paper_1112_4139_gb300 as pkg
    pkg.build()
    from paper_1112_4139_gb300 import agis
    ds = synth.simulate(synth.config("small1yr", n_src=n_src, span_days=span_days, seed=3, min_transits=0))
    P = OM.problem_from_dataset(ds)
    g = agis.from_dataset(ds)
    g.set_state(src=ds.src_true, att=ds.att_true, cal=ds.cal_true)
    st = g.source_update()
    ss, (R, W) = g.source_stats(), g.residuals()
    # the totals are the sums of the sources' values: whole numbers equal, chi^2 by the rounding of the sums
    assert st["n_out"] == ss["n_out"].sum() and st["nu_sum"] == ss["nu"].sum()
    terms = W * R * R
    assert abs(st["chi2"] - terms.sum()) <= 4e-16 * ds.n_obs * np.abs(terms).sum()
    sc = g.calibration_update()
    got = g.calibration()
    g.close()
    ev = OM.evaluate(P, ds.src_true, ds.att_true, ds.cal_true)
    cal1, rdc = OB.calibration_update(P, ds.cal_true, ev, R, W)
    assert sc["rank_defect"] == rdc
    assert np.max(np.abs(got - cal1)) < 1e-3 * synth.UAS     # the parity bound of the calibration
