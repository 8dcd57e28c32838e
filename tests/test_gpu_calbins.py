"""The C block of the full geometric calibration at the numbers of AC column bins where its path
changes (reduced systems in shared memory up to 160 bins, through global memory beyond) and around
its warps' widths, against the oracle's constrained least-squares update of the same residuals."""
import dataclasses

import numpy as np
import pytest

import synth
from oracle import calgeneric as CG
from oracle import model as OM

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("col_bin,j_per_k", [(1966, 10), (983, 7), (62, 10), (61, 30), (31, 10), (16, 10), (10, 10), (9, 10)])
def test_calibration_update_matches_oracle(col_bin, j_per_k):
    import paper_1112_4139_gb300 as pkg
    pkg.build()
    from paper_1112_4139_gb300 import agis
    ds = synth.simulate(synth.config("small1yr", n_src=60_000, span_days=20, seed=13, cal_generic=True, n_gate=2,
                                     gate_g0=15.0, gate_step=10.0, cal_j_per_k=j_per_k, cal_col_bin=col_bin))
    # half of the columns of every tenth CCD without observations: unobserved bins among observed ones
    x = (ds.ccd % 10 == 3) & (ds.mu > 400) & (ds.mu < 1100)
    sel = lambda a: np.ascontiguousarray(a[~x])  # noqa: E731
    ds = dataclasses.replace(ds, **{k: sel(getattr(ds, k)) for k in ("t_ns", "src", "ccd", "fov", "kind", "sigma", "mu",
                                                                    "noise", "gate")})
    g = agis.from_dataset(ds, seg_len=720, seg_overlap=12, pivot_tol=1e-4, robust=0, frame_each_iter=0)
    # at the truth and with plain weights: the same residuals and weights on both sides
    g.set_state(src=ds.src_true, att=ds.att_true, cal=ds.cal0)
    g.source_update()
    R, W = g.residuals()
    P = OM.problem_from_dataset(ds)
    L = P.calg
    _, k = OM.observation_lines(P, ds.cal0)
    d, rd = CG.update(L, k[0], k[1], R, W)
    st = g.calibration_update()
    got = g.calibration() - ds.cal0
    g.close()
    assert st["rank_defect"] == rd
    # as in the parity tests: 1e-3 uas, on updates of several hundred uas
    assert np.abs(d).max() > 100 * synth.UAS
    assert np.abs(got - d).max() < 1e-3 * synth.UAS, np.abs(got - d).max() / synth.UAS
