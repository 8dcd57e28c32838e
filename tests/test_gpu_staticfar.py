"""The static source update from starting values far off: Q is the sum of W R^2 to the rounding of the
residuals themselves, although the residuals at the start are thousands of sigma.
"""
import dataclasses

import numpy as np
import pytest

import synth
from oracle import agis as OG
from oracle import blocks as OB
from oracle import model as OM

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("off_sigma", [1.0, 500.0, 5000.0])
@pytest.mark.parametrize("cfg", [dict(), dict(n_rounds=0), dict(robust=0), dict(weight_fn=1)])
def test_q_is_the_sum_of_the_outputs(off_sigma, cfg):
    import torch

    import paper_1112_4139_gb300 as pkg
    pkg.build()
    from paper_1112_4139_gb300 import agis
    ds = synth.simulate(synth.config("small1yr", n_src=400, seed=31, min_transits=10))
    keep = np.ones(ds.n_obs, bool)                       # a source with three observations among them: pivots fail
    keep[ds.src_offsets()[9] + 3:ds.src_offsets()[10]] = False
    ds = dataclasses.replace(ds, **{k: np.ascontiguousarray(getattr(ds, k)[keep]) for k in (
        "t_ns", "src", "ccd", "fov", "kind", "sigma", "mu", "noise", "gate")})
    rng = np.random.default_rng(2)
    src0 = ds.src_true + off_sigma * float(np.median(ds.sigma)) * rng.choice([-1.0, 1.0], (ds.n_src, 5))
    P = OM.problem_from_dataset(ds)
    ev = OM.evaluate(P, src0, ds.att_true, ds.cal_true)
    st = OB.Settings(robust=bool(cfg.get("robust", 1)), n_rounds=cfg.get("n_rounds", 4),
                     weight_fn="huber" if cfg.get("weight_fn") else "agis")
    src1, ref, _ = OB.source_update(P, src0, ds.att_true, ds.cal_true, st, ev=ev)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    s, R, W = dev(src0), dev(np.zeros(ds.n_obs)), dev(np.zeros(ds.n_obs))
    stats = dev(np.zeros((5, ds.n_src)))
    agis.source_update_static(ds.geometry, agis.default_config(**cfg), agis.obs_from_dataset(ds, device="cuda"), s,
                              dev(ds.att_true), dev(ds.cal_true), R_out=R, W_out=W, stats_out=stats)
    s, R, W = s.cpu().numpy(), R.cpu().numpy(), W.cpu().numpy()
    Q = stats.cpu().numpy()[1]
    few = np.arange(ds.n_src) == 9
    assert np.max(np.abs(OG.source_errors(s, src1))[~few]) < 0.5 * synth.UAS      # the parity bound
    sl = P.src == 9
    assert np.all(np.abs(R - ref.R)[sl] < 1e-3 * synth.UAS)      # its parameters are not unique, its residuals are
    # both sides carry residuals h - A d, rounded at 2^-53 of their terms: 16 operations each, twice in Q; and the
    # sums' own rounding
    M = np.abs(ev["R"]) + (np.abs(ev["A"]) * np.abs(ref.d[P.src])).sum(1)
    per = lambda v: np.bincount(P.src, v, minlength=ds.n_src)  # noqa: E731
    tol = 64 * 2.0 ** -53 * per(W * np.abs(R) * M) + 1e-13 * per(W * R * R)
    d = np.abs(Q - per(W * R * R))
    assert np.all(d[~few] <= tol[~few]), (d / tol)[~few].max()
