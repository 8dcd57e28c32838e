"""Timed cases of the framework: what its users have it do, through its public entry points.

A case is a dict of plain values; `kind` selects the entry point:
  iterate      Agis.iterate(1): one S[ACG] iteration in the FP64 form, state read back
  source       Agis.source_update(): the S block, either form, with or without attitude noise
  attitude     Agis.attitude_update(): the A block, either form
  calibration  Agis.calibration_update(): the C block of the full geometric calibration
  evaluate     Agis.evaluate(): residuals of all observations
  static       agis.source_update_static(): the S block on caller-owned device arrays
  train        agis.mlp_loss_grad + agis.mlp_adam: one training step of the learned proposal
Observations come from the repository's simulator (scanning law, noise, outliers and the
starting errors of its named workloads), so that residuals, weights and the distribution of
observations over sources, knot intervals and calibration parameters are those of a solution.
Sizes are those of the named workloads, the tests, the profiles and the benchmark; `draw`
spreads them over the same ranges.
"""
import dataclasses
import math

import numpy as np
import torch

import synth
from paper_1112_4139_gb300 import agis, learned

YEAR_S = synth.YEAR_S
DAYS_PER_YEAR = 365.25
OBS_PER_SOURCE_DAY = 0.451      # mean observations (AL and AC) per source and day of the scanning law
N_FEATURE_ROWS = 200_000        # rows of the training table that a batch is drawn from


def _sim(kind, **over):
    base = dict(kind=kind, n_src=10_000, span_days=DAYS_PER_YEAR, knot_dt_s=3600, precision=0, seg_len=720,
                weight_fn=0, uneven=False, min_transits=8, attnoise_s=0, n_gate=0, col_bin=0, j_per_k=0)
    base.update(over)
    return base


FIVE = 5 * DAYS_PER_YEAR


def listed():
    return [
        # the parity tests' problem: 3000 sources, one year, 1-h knots; latency and launches
        dict(_sim("iterate", n_src=3000), name="iterate_3000src_1yr"),
        # the small1yr workload: 10,000 sources, one year, 1-h knots
        dict(_sim("iterate", n_src=10_000), name="iterate_small1yr"),
        # the scale5yr workload's five years and observations per knot interval (156) at the
        # 30,000 sources of the profiles: an iteration of a large FP64 solution
        dict(_sim("iterate", n_src=30_000, span_days=FIVE, knot_dt_s=1000, min_transits=0), name="iterate_5yr"),
        # the uneven5yr workload: magnitude-dependent sigma, 40-250 transits per source
        dict(_sim("source", n_src=8_000, span_days=FIVE, knot_dt_s=3600, uneven=True, min_transits=40),
             name="source_uneven5yr"),
        # a short source update: the smoke run's 800 sources
        dict(_sim("source", n_src=800), name="source_800src_1yr"),
        # the mixed form's source update (the linearized pass, with its refresh in one of eight)
        dict(_sim("source", n_src=30_000, span_days=FIVE, knot_dt_s=1000, precision=1, min_transits=0),
             name="source_mixed_5yr"),
        # the source update with the excess attitude noise on 240-s buckets: sigma differs per observation
        dict(_sim("source", n_src=5_000, span_days=FIVE, knot_dt_s=3600, attnoise_s=240, min_transits=0),
             name="source_attnoise_5yr"),
        # the mixed form's attitude update at the density of the scale5yr workload
        dict(_sim("attitude", n_src=30_000, span_days=FIVE, knot_dt_s=1000, precision=1, min_transits=0),
             name="attitude_mixed_5yr"),
        # the paper's 240-s knots, one year of 40,000 sources: many knots, short runs of observations
        dict(_sim("attitude", n_src=40_000, knot_dt_s=240), name="attitude_240s_1yr"),
        # the full geometric calibration of the benchmark: two gates, 30-day long intervals, 16-column bins
        dict(_sim("calibration", n_src=10_000, n_gate=2, col_bin=16, j_per_k=30), name="calibration_full_1yr"),
        # a caller that owns the device memory: a few thousand sources per call
        dict(_sim("static", n_src=2_000), name="static_2000src_1yr"),
        # one step of the learned proposal's training, its default batch
        dict(kind="train", batch=8192, name="train_8192"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["iterate", "iterate", "source", "source", "source", "attitude", "attitude", "calibration",
                       "evaluate", "static", "train"])
    if kind == "train":
        return dict(kind="train", batch=_log_int(rng, 500, 8192))
    if kind == "calibration":
        return _sim("calibration", n_src=_log_int(rng, 1000, 10_000), n_gate=rng.choice([1, 2, 3]),
                    col_bin=rng.choice([16, 25, 64]), j_per_k=rng.choice([10, 17, 30]))
    if kind == "static":
        return _sim("static", n_src=_log_int(rng, 300, 4000), weight_fn=rng.choice([0, 1]))
    years = rng.choice([1, 1, 2, 5])
    # the attitude needs about 50 observations in an interval (1-h knots at the longest)
    n_src = _log_int(rng, 600 if kind in ("source", "evaluate") else 3000, 30_000)
    # the shortest knots that keep about a hundred observations in an interval (or 1 h)
    knot = next(k for k in (600, 1000, 1800, 3600) if k == 3600 or n_src * OBS_PER_SOURCE_DAY * k / 86400 > 90)
    mixed = kind in ("source", "attitude") and rng.random() < 0.5
    uneven = kind == "source" and rng.random() < 0.4
    return _sim(kind, n_src=n_src, span_days=years * DAYS_PER_YEAR, knot_dt_s=knot, precision=1 if mixed else 0,
                weight_fn=rng.choice([0, 0, 1]), uneven=uneven, min_transits=8 * years,
                seg_len=rng.choice([480, 720, 1000]))


# ---------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------
def _dataset(case, seed):
    over = {}
    if case["n_gate"]:
        over = dict(cal_generic=True, n_gate=case["n_gate"], cal_j_per_k=case["j_per_k"], cal_col_bin=case["col_bin"],
                    mag_dependent=True)
    if case["uneven"]:
        over = dict(mag_dependent=True, max_transits=50 * round(case["span_days"] / DAYS_PER_YEAR))
    # the simulator leaves out sources with too few transits: more are simulated than are kept
    n = case["n_src"]
    n_sim = n + 40 + int(0.15 * n) if case["min_transits"] else n
    ds = synth.simulate(synth.config("small1yr", n_src=n_sim, span_days=case["span_days"],
                                     knot_dt_s=case["knot_dt_s"], seed=seed, min_transits=case["min_transits"],
                                     **over))
    if ds.n_src > n:
        ds = _cut(ds, np.arange(ds.src_offsets()[n]), src_true=ds.src_true[:n], src0=ds.src0[:n])
    if case["kind"] in ("evaluate", "static"):
        # results per observation: a fixed number of them, the others rejected at random
        keep = np.sort(np.random.default_rng(seed).choice(ds.n_obs, _n_obs(case), replace=False))
        ds = _cut(ds, keep)
    return ds


def _n_obs(case):
    return int(0.85 * OBS_PER_SOURCE_DAY * case["n_src"] * case["span_days"])


def _cut(ds, keep, **over):
    names = ("t_ns", "src", "ccd", "fov", "kind", "sigma", "mu", "noise", "gate")
    return dataclasses.replace(ds, **{k: np.ascontiguousarray(getattr(ds, k)[keep]) for k in names}, **over)


def _context(case, ds):
    return agis.from_dataset(ds, seg_len=case["seg_len"], seg_overlap=12, precision=case["precision"],
                             weight_fn=case["weight_fn"], **agis.calibration_config(ds.geometry))


def _f64(*shape):
    return torch.empty(shape, dtype=torch.float64, device="cuda")


class State:
    """A context (or caller-owned arrays) and the device buffers its results are read into."""

    def __init__(self, kind, **kw):
        self.kind = kind
        self.__dict__.update(kw)


def _train_inputs(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rnd = lambda *s: torch.randn(*s, generator=gen, device="cuda")  # noqa: E731
    # features: the last four updates over their RMS, shrinking from one to the next; targets: the
    # remaining correction in the same unit
    step = rnd(N_FEATURE_ROWS, 5)
    decay = 0.4 + 0.55 * torch.rand(N_FEATURE_ROWS, 1, generator=gen, device="cuda")
    d = torch.stack([step * decay ** k + 0.05 * rnd(N_FEATURE_ROWS, 5) for k in range(4)], dim=1)
    sig = d.square().mean(dim=(1, 2), keepdim=True).sqrt()
    extra = torch.cat([0.3 * rnd(N_FEATURE_ROWS, 1), 2 * torch.rand(N_FEATURE_ROWS, 1, generator=gen, device="cuda") - 1], 1)
    X = torch.cat([(d / sig).reshape(N_FEATURE_ROWS, 20), extra], dim=1).contiguous()
    T = ((d[:, 3] * decay / (1 - decay)) / sig[:, 0]).contiguous()
    idx = torch.randint(0, N_FEATURE_ROWS, (case["batch"],), generator=gen, device="cuda", dtype=torch.int32)
    p = torch.from_numpy(learned.init_params(seed)).cuda()
    return X, T, idx, p


def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        X, T, idx, p = _train_inputs(case, seed)
        return State(kind, X=X, T=T, idx=idx, p=p, m=torch.zeros_like(p), v=torch.zeros_like(p),
                     grad=torch.empty_like(p), loss=torch.empty(1, device="cuda"), t=0)
    ds = _dataset(case, seed)
    if kind == "static":
        dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
        return State(kind, geometry=ds.geometry, cfg=agis.default_config(weight_fn=case["weight_fn"]),
                     obs=agis.obs_from_dataset(ds, device="cuda"), src=dev(ds.src0), att=dev(ds.att0), cal=dev(ds.cal0),
                     R=_f64(ds.n_obs), W=_f64(ds.n_obs), stats=_f64(5, ds.n_src),
                     n_max=int(np.diff(ds.src_offsets()).max()))
    g = _context(case, ds)
    st = State(kind, g=g, src=_f64(g.n_src, 5), att=_f64(g.n_coef, 4), cal=_f64(g.n_cal))
    if kind == "evaluate":
        st.R = _f64(g.n_obs)
    if case["attnoise_s"]:
        g.set_attnoise(case["attnoise_s"] * 10**9)
        g.source_update()      # the first estimate of the noise, which the next source update uses
    if kind in ("attitude", "calibration"):
        g.source_update()      # the residuals and weights that the block reads
    torch.cuda.synchronize()
    return st


def run(st):
    kind = st.kind
    if kind == "train":
        st.t += 1
        agis.mlp_loss_grad(st.p, st.X, st.T, st.grad, st.loss, idx=st.idx)
        agis.mlp_adam(st.p, st.grad, st.m, st.v, st.t, 1e-3)
        return dict(loss=st.loss, grad=st.grad, params=st.p)
    if kind == "static":
        agis.source_update_static(st.geometry, st.cfg, st.obs, st.src, st.att, st.cal, R_out=st.R, W_out=st.W,
                                  stats_out=st.stats, max_obs_per_source=st.n_max)
        return dict(sources=st.src, R=st.R, W=st.W, stats=st.stats)
    g = st.g
    if kind == "iterate":
        g.iterate(1)
        return dict(sources=g.sources(st.src), attitude=g.attitude(st.att), calibration=g.calibration(st.cal))
    if kind == "source":
        g.source_update()
        return dict(sources=g.sources(st.src))
    if kind == "attitude":
        g.attitude_update()
        return dict(attitude=g.attitude(st.att))
    if kind == "calibration":
        g.calibration_update()
        return dict(calibration=g.calibration(st.cal))
    return dict(R=g.evaluate(st.R))


# ---------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------
def work(case):
    kind = case["kind"]
    if kind == "train":
        n, p = case["batch"], agis.MLP_N_PARAMS
        return dict(bytes=n * (22 + 5 + 1) * 4 + 8 * 4 * p, flops=3 * 2 * n * (22 * 64 + 64 * 64 + 64 * 5))
    n_src = case["n_src"]
    n = n_src * OBS_PER_SOURCE_DAY * case["span_days"] * (1.0 if case["min_transits"] == 0 else 1.05)
    if kind in ("evaluate", "static"):
        n = _n_obs(case)
    n_coef = case["span_days"] * 86400 / case["knot_dt_s"]
    n_cal = case["span_days"] * 138
    obs = 8 + 4 + 3 + 4 + 0.1 * 8            # time, source, CCD/field/kind, sigma, mu of the AC tenth
    src, att, cal = 16 * 5 * n_src, 16 * 4 * n_coef, 16 * n_cal
    # model and partials 300, weights and source normals 40; attitude normals 2 x 116 and the band
    # factorisation 16^2 per unknown; calibration sums 4
    flops = dict(source=340 * n, attitude=232 * n + 4 * n_coef * 512, evaluate=200 * n, static=340 * n,
                 iterate=(340 + 232 + 4) * n + 4 * n_coef * 512, calibration=60 * n)[kind]
    handed = 8 + 8 + 32 + 8                  # residual, weight, attitude partial, time
    if case["precision"]:
        handed = 4 + 4 + 16 + 8
    if kind == "calibration":
        n_bin = -(-1966 // case["col_bin"])
        n_k = -(-case["span_days"] // case["j_per_k"])
        groups = 62 * case["n_gate"] * n_k
        cal = 16 * groups * (6 * case["j_per_k"] + n_bin + 6)
        flops += groups * (n_bin ** 3 * 2 / 3 + 12 * case["j_per_k"] * n_bin ** 2)
    nbytes = dict(source=n * obs + src, static=n * (obs + 16) + src, iterate=n * obs + src + att + cal,
                  evaluate=n * (obs + 8) + src / 2, attitude=n * handed + att, calibration=n * 28 + cal)[kind]
    return dict(bytes=float(nbytes), flops=float(flops))


# ---------------------------------------------------------------------------------------
# the same results in plain 64-bit torch and numpy
# ---------------------------------------------------------------------------------------
def _qmul(a, b):
    ax, ay, az, aw = a.unbind(-1)
    bx, by, bz, bw = b.unbind(-1)
    return torch.stack([ax * bw + ay * bz - az * by + aw * bx, -ax * bz + ay * bw + az * bx + aw * by,
                        ax * by - ay * bx + az * bw + aw * bz, -ax * bx - ay * by - az * bz + aw * bw], -1)


def _qconj(q):
    return q * torch.tensor([-1.0, -1.0, -1.0, 1.0], dtype=q.dtype, device=q.device)


def _rotate(q, v):
    """Components of v in the frame turned by the unit quaternion q: {v', 0} = q^-1 {v, 0} q."""
    return _qmul(_qmul(_qconj(q), torch.cat([v, torch.zeros_like(v[..., :1])], -1)), q)[..., :3]


def _triad(a, d):
    sa, ca, sd, cd = a.sin(), a.cos(), d.sin(), d.cos()
    return (torch.stack([-sa, ca, torch.zeros_like(sa)], -1), torch.stack([-sd * ca, -sd * sa, cd], -1),
            torch.stack([cd * ca, cd * sa, sd], -1))


class Problem:
    """Observations and geometry on the GPU in 64 bits, and the observation model."""

    def __init__(self, ds):
        dev = lambda a, t=torch.float64: torch.from_numpy(np.ascontiguousarray(a)).to("cuda", t)  # noqa: E731
        self.g = g = ds.geometry
        self.t, self.src = dev(ds.t_ns, torch.int64), dev(ds.src, torch.int64)
        self.ccd, self.fov, self.kind = (dev(a, torch.int64) for a in (ds.ccd, ds.fov, ds.kind))
        self.sig2, self.mu = dev(ds.sigma).square(), dev(ds.mu)
        self.eta0, self.x_fpa, self.x_centre = dev(g["eta0"]), dev(g["x_fpa"]), dev(g["x_centre"])
        self.n, self.n_src, self.n_coef, self.n_cal = ds.n_obs, ds.n_src, ds.n_coef, ds.n_cal
        self.s0, self.a0, self.c0 = dev(ds.src0), dev(ds.att0), dev(ds.cal0)
        self.ref = dev(ds.src_true[:, [0, 1, 3, 4]])
        day = ((self.t - g["cal_t0_ns"]) // g["cal_dt_ns"]).clamp(0, g["n_cal_days"] - 1)
        row = dev(g["ccd_row"], torch.int64)[self.ccd]
        self.k = torch.where(self.kind == 0, (day * 2 + self.fov) * 62 + self.ccd,
                             g["n_cal_days"] * 124 + (day * 2 + self.fov) * 7 + row)

    def spline(self, t):
        g = self.g
        l = (3 + torch.div(t - g["knot0_ns"], g["knot_dt_ns"], rounding_mode="floor")).clamp(3, self.n_coef - 1)
        at = lambda k: g["knot0_ns"] + (k - 3).clamp(0, self.n_coef - 3) * g["knot_dt_ns"]  # noqa: E731
        R = [(at(l + i + 1) - t).double() for i in range(3)]
        L = [(t - at(l - i)).double() for i in range(3)]
        b = [torch.ones_like(R[0])]
        for i in range(3):
            s, nxt = torch.zeros_like(R[0]), []
            for j in range(i + 1):
                u = b[j] / (R[j] + L[i - j])
                nxt.append(s + R[j] * u)
                s = L[i - j] * u
            b = nxt + [s]
        return l, torch.stack(b, -1)

    def observe(self, src, att, cal, partials=True):
        """Residuals, design rows -dR/ds', (dR/dq)/|s|, the spline sum, interval and B-splines."""
        out = [self._observe(src, att, cal, slice(o, o + (1 << 21)), partials) for o in range(0, self.n, 1 << 21)]
        return [torch.cat(v) for v in zip(*out)]

    def _observe(self, src, att, cal, sl, partials):
        g, t = self.g, self.t[sl]
        s5 = src[self.src[sl]]
        p, q, r = _triad(s5[:, 0], s5[:, 1])
        lon = g["orb_L0"] + 2 * math.pi * (t.double() * 1e-9 / g["year_s"])
        ce, se, w = math.cos(g["obliquity"]), math.sin(g["obliquity"]), 2 * math.pi / g["year_s"]
        b = torch.stack([lon.cos(), ce * lon.sin(), se * lon.sin()], -1)
        vc = torch.stack([-w * lon.sin(), ce * w * lon.cos(), se * w * lon.cos()], -1) * g["au_light_s"]
        rb = (r * b).sum(-1)
        tau = (((t - g["t_ep_ns"]).double() * 1e-9 + rb * g["au_light_s"]) / g["year_s"])[:, None]
        ub = r + tau * (p * s5[:, 3:4] + q * s5[:, 4:5]) - s5[:, 2:3] * b
        ub = ub / ub.norm(dim=-1, keepdim=True)
        u = ub + vc
        l, B = self.spline(t)
        s = (att[l[:, None] + torch.arange(-3, 1, device=l.device)] * B[..., None]).sum(-2)
        ns = s.norm(dim=-1, keepdim=True)
        qa = s / ns
        us = _rotate(qa, u / u.norm(dim=-1, keepdim=True))
        f = 1.0 - 2.0 * self.fov[sl].double()
        rho = (us[:, 0].square() + us[:, 1].square()).sqrt()
        zeta, phi = torch.atan2(us[:, 2], rho), torch.atan2(us[:, 1], us[:, 0])
        gh = g["gamma_c"] / 2
        cg, sg = math.cos(gh), math.sin(gh)
        eta = torch.atan2(cg * us[:, 1] - f * sg * us[:, 0], cg * us[:, 0] + f * sg * us[:, 1])
        al = self.kind[sl] == 0
        zeta0 = -(self.x_fpa[self.ccd[sl]] - (self.mu[sl] - g["mu_c"]) * g["p_ac"] - self.x_centre[self.fov[sl]]) / g["focal_length"]
        c = cal[self.k[sl]]
        R = torch.where(al, self.eta0[self.ccd[sl]] + c - eta, zeta0 + c - zeta)
        if not partials:
            return (R,)
        dpar = -(b - r * rb[:, None])
        dub = torch.stack([p, q, dpar, p * tau, q * tau], -1)
        du = (1 - (ub * vc).sum(-1))[:, None, None] * dub - ub[:, :, None] * torch.einsum("oi,oij->oj", vc, dub)[:, None, :]
        sp, cp, sz, cz = phi.sin(), phi.cos(), zeta.sin(), zeta.cos()
        m = torch.stack([-sp, cp, torch.zeros_like(sp)], -1)
        n = torch.stack([-sz * cp, -sz * sp, cz], -1)
        back = lambda v: _rotate(_qconj(qa), v)  # noqa: E731
        A = torch.einsum("oi,oij->oj", torch.where(al[:, None], back(m) / cz[:, None], back(n)), du)
        v3 = torch.where(al[:, None], n * (2 / cz)[:, None], m * -2.0)
        gq = _qmul(qa, torch.cat([v3, torch.zeros_like(v3[:, :1])], -1)) / ns
        return R, A, gq, s, l, B


def _weight(z, fn):
    a = z.abs()
    if fn == 1:
        return torch.where(a <= 2, torch.ones_like(a), 4 * (a - 1) / a.square())
    t = a - 2
    return torch.where(a <= 2, torch.ones_like(a),
                       torch.where(a < 3, 1 - 1.773735 * t ** 2 + 1.141615 * t ** 3, torch.exp(-a / 3)))


def _by_source(P, v):
    return torch.zeros((P.n_src,) + v.shape[1:], dtype=v.dtype, device=v.device).index_add_(0, P.src, v)


def _robust_scale(P, x):
    """Half the intersextile range of x per source (linear interpolation between order statistics)."""
    order = torch.argsort(x)
    order = order[torch.argsort(P.src[order], stable=True)]
    xs = x[order]
    cnt = torch.bincount(P.src, minlength=P.n_src)
    off = cnt.cumsum(0) - cnt

    def quantile(q):
        h = q * (cnt - 1).clamp(min=0).double()
        lo = h.floor().long()
        a, b = xs[(off + lo).clamp(max=P.n - 1)], xs[(off + (lo + 1).minimum((cnt - 1).clamp(min=0))).clamp(max=P.n - 1)]
        return a + (h - lo) * (b - a)
    return 0.5 * (quantile(5 / 6) - quantile(1 / 6))


def _source_update(P, src, h, A, sig2, fn, rounds=4, steps=3):
    """Inner iteration of every source: weights, excess noise, 5x5 solves."""
    vs = _robust_scale(P, h / sig2.sqrt())[P.src]
    w = torch.where(vs > 0, _weight(h / sig2.sqrt() / vs, fn), torch.ones_like(h))
    cnt = torch.bincount(P.src, minlength=P.n_src)
    s2min = torch.full((P.n_src,), math.inf, dtype=torch.float64, device=h.device).scatter_reduce_(0, P.src, sig2, "amin")

    def solve(y):
        W = w / (sig2 + y[P.src])
        N = _by_source(P, (W[:, None, None] * A[:, :, None] * A[:, None, :]).reshape(-1, 25)).reshape(-1, 5, 5)
        b = _by_source(P, (W * h)[:, None] * A)
        sc = N.diagonal(dim1=1, dim2=2).clamp(min=1e-300).rsqrt()   # unit diagonal before the solve
        d = sc * torch.linalg.solve(N * sc[:, :, None] * sc[:, None, :], sc * b)
        R = h - (A * d[P.src]).sum(-1)
        den = sig2 + y[P.src]
        return d, R, _by_source(P, w * R * R / den), _by_source(P, w * R * R / den.square())

    for rnd in range(rounds + 1):
        nu = (cnt - _by_source(P, (w < 0.2).long()) - 5).double()
        y = torch.zeros(P.n_src, dtype=torch.float64, device=h.device)
        d, R, Q, S2 = solve(y)
        live = (nu > 0) & (Q > nu)
        for _ in range(steps):
            dy = torch.where(live, (1 - Q / nu) * Q / -S2, torch.zeros_like(y))
            y = (y + dy).clamp(min=0)
            d, R, Q, S2 = solve(y)
            live = live & (dy.abs() > 1e-12 * s2min)
        W = w / (sig2 + y[P.src])
        if rnd < rounds:
            w = _weight(R / (sig2 + y[P.src]).sqrt(), fn)
    new = src.clone()
    new[:, 0] += d[:, 0] / src[:, 1].cos()
    new[:, 1:] += d[:, 1:]
    return new, R, W, y


def _segments(n_coef, seg_len, L):
    K = n_coef - 3
    n_seg = max(1, -(-K // seg_len))
    for k in range(n_seg):
        x0, x1 = 3 + k * seg_len, 3 + (k + 1) * seg_len
        yield (max(3, x0 - L), min(n_coef - 1, x1 + L - 1), 0 if k == 0 else x0 - 1,
               n_coef - 1 if k == n_seg - 1 else x1 - 2)


def _attitude_update(P, att, R, W, gq, s, l, B, seg_len, L=12, lam2=1e-6, tol=1e-12):
    """Normals of every knot interval, then the band of each overlapping segment factorised."""
    n_iv = P.n_coef - 3
    blk = torch.zeros(n_iv, 16, 16, dtype=torch.float64, device=R.device)
    rhs = torch.zeros(n_iv, 16, dtype=torch.float64, device=R.device)
    for o in range(0, P.n, 1 << 19):
        sl = slice(o, o + (1 << 19))
        G = (B[sl, :, None] * gq[sl, None, :]).reshape(-1, 16)
        D = (-2 * B[sl, :, None] * s[sl, None, :]).reshape(-1, 16)
        V = W[sl, None, None] * (G[:, :, None] * G[:, None, :] + lam2 * D[:, :, None] * D[:, None, :])
        blk.index_add_(0, l[sl] - 3, V)
        rhs.index_add_(0, l[sl] - 3, -(W[sl] * R[sl])[:, None] * G)
    blk, rhs = blk.cpu().numpy(), rhs.cpu().numpy()
    segs = list(_segments(P.n_coef, seg_len, L))
    rows = 4 * max(hi - lo + 4 for lo, hi, _, _ in segs)
    N = np.zeros((len(segs), rows + 16, 16))          # N[seg, i, j - i], j = i .. i + 15
    x = np.zeros((len(segs), rows + 16))
    for k, (lo, hi, _, _) in enumerate(segs):
        for i in range(16):
            at = 4 * np.arange(hi - lo + 1) + i
            x[k, at] += rhs[lo - 3:hi - 2, i]
            for j in range(i, 16):
                N[k, at, j - i] += blk[lo - 3:hi - 2, i, j]
    diag = N[:, :, 0].copy()
    for r in range(rows):
        ok = (N[:, r, 0] > tol * diag[:, r]) & (N[:, r, 0] > 0)
        u = np.where(ok[:, None], N[:, r] / np.where(ok, N[:, r, 0], 1.0)[:, None], 0.0)
        for a in range(1, 16):
            N[:, r + a, :16 - a] -= u[:, a:a + 1] * N[:, r, a:]
        x[:, r + 1:r + 16] -= u[:, 1:] * x[:, r:r + 1]
        x[:, r] = np.where(ok, x[:, r] / np.where(ok, N[:, r, 0], 1.0), 0.0)
        N[:, r] = u
    for r in range(rows - 1, -1, -1):
        x[:, r] -= (N[:, r, 1:] * x[:, r + 1:r + 16]).sum(-1)
    new = att.clone()
    for k, (lo, hi, u_lo, u_hi) in enumerate(segs):
        at = 4 * (u_lo - (lo - 3))
        new[u_lo:u_hi + 1] += torch.from_numpy(x[k, at:at + 4 * (u_hi - u_lo + 1)].reshape(-1, 4)).to(att)
    return new


def _calibration_update(P, cal, R, W):
    z = torch.zeros(P.n_cal, dtype=torch.float64, device=R.device)
    N, b = z.clone().index_add_(0, P.k, W), z.clone().index_add_(0, P.k, -W * R)
    d = torch.where(N > 0, b / N, z)
    n_al = 124 * P.g["n_cal_days"]
    al, ac = d[:n_al].reshape(-1, 124), d[n_al:].reshape(-1, 7)
    return cal + torch.cat([(al - al.mean(1, keepdim=True)).reshape(-1), (ac - ac.mean(1, keepdim=True)).reshape(-1)])


def _frame(P, src, att):
    """Frame rotator: (eps, omega) by least squares, then the sources and coefficients turned."""
    g = P.g
    year = lambda ns: ns.double() * 1e-9 / g["year_s"]  # noqa: E731
    p, q, r = _triad(src[:, 0], src[:, 1])
    dr = r - _triad(P.ref[:, 0], P.ref[:, 1])[2]
    z, tt = torch.zeros_like(p), (g["t_ep_ns"] - g["t_fr_ns"]) * 1e-9 / g["year_s"]
    rows = torch.cat([torch.cat(v, 1) for v in ([z, q], [z, -p], [q, tt * q], [-p, -tt * p])])
    obs = torch.cat([src[:, 3] - P.ref[:, 2], src[:, 4] - P.ref[:, 3], (p * dr).sum(-1), (q * dr).sum(-1)])
    eo = torch.linalg.solve(rows.T @ rows, rows.T @ obs)

    def turn(v):
        ang = v.norm(dim=-1, keepdim=True)
        return torch.cat([v * torch.where(ang > 0, (ang / 2).sin() / ang, 0.5 * torch.ones_like(ang)), (ang / 2).cos()], -1)

    def frame(dt):
        return _qmul(turn(dt[:, None] * eo[3:]), turn(eo[:3].expand(dt.shape[0], 3)))
    f = frame(torch.full((P.n_src,), tt, dtype=torch.float64, device=src.device))
    mu = _rotate(f, p * src[:, 3:4] + q * src[:, 4:5] - torch.linalg.cross(eo[3:].expand_as(r), r))
    rc = _rotate(f, r)
    a, d = torch.atan2(rc[:, 1], rc[:, 0]), torch.atan2(rc[:, 2], (rc[:, 0].square() + rc[:, 1].square()).sqrt())
    p, q, _ = _triad(a, d)
    new = torch.stack([torch.remainder(a, 2 * math.pi), d, src[:, 2], (p * mu).sum(-1), (q * mu).sum(-1)], 1)
    n = torch.arange(P.n_coef, device=src.device)
    at = lambda k: g["knot0_ns"] + (k - 3).clamp(0, P.n_coef - 3) * g["knot_dt_ns"]  # noqa: E731
    mid = torch.div(at(n) + at(n + 4), 2, rounding_mode="floor")
    return new, _qmul(_qconj(frame(year(mid - g["t_fr_ns"]))), att)


def _attitude_noise(P, R, eps2_src, bucket_ns):
    """max(0, 68% quantile of R^2 - sigma^2 - eps_i^2) per component and time bucket, per observation."""
    comp = torch.where(P.kind == 0, torch.zeros_like(P.fov), 1 + P.fov)
    bucket = torch.div(P.t - P.g["knot0_ns"], bucket_ns, rounding_mode="floor")
    n_b = int(bucket.max()) + 1
    key = comp * n_b + bucket
    x = R.square() - P.sig2 - eps2_src[P.src]
    order = torch.argsort(x)
    order = order[torch.argsort(key[order], stable=True)]
    xs, cnt = x[order], torch.bincount(key, minlength=3 * n_b)
    off = cnt.cumsum(0) - cnt
    hq = 0.68 * (cnt - 1).clamp(min=0).double()
    lo = hq.floor().long()
    a, b = xs[(off + lo).clamp(max=P.n - 1)], xs[(off + (lo + 1).minimum((cnt - 1).clamp(min=0))).clamp(max=P.n - 1)]
    return torch.where(cnt > 0, (a + (hq - lo) * (b - a)).clamp(min=0), torch.zeros_like(hq))[key]


def _bf16(x):
    return x.to(torch.bfloat16).double()


def _exact_train(case, seed):
    X, T, idx, p = _train_inputs(case, seed)
    sizes = [(64, 22), (64,), (64, 64), (64,), (5, 64), (5,)]
    W, at = [], 0
    for s in sizes:
        n = math.prod(s)
        v = p[at:at + n].reshape(s)
        W.append(_bf16(v) if len(s) == 2 else v.double())
        at += n
    x, t = _bf16(X[idx.long()]), T[idx.long()].double()
    h1 = _bf16((x @ W[0].T + W[1]).relu().float())
    h2 = _bf16((h1 @ W[2].T + W[3]).relu().float())
    e = h2 @ W[4].T + W[5] - t
    dy = 2 * e / e.shape[0]
    d2 = (dy @ W[4]) * (h2 > 0)
    d1 = (d2 @ W[2]) * (h1 > 0)
    grad = torch.cat([v.reshape(-1) for v in (d1.T @ x, d1.sum(0), d2.T @ h1, d2.sum(0), dy.T @ h2, dy.sum(0))])
    # the first Adam step: the moments' bias corrections cancel
    return dict(loss=e.square().sum().reshape(1) / e.shape[0], grad=grad,
                params=p.double() - 1e-3 * grad / (grad.abs() + 1e-8))


def exact(case, seed):
    if case["kind"] == "train":
        return _exact_train(case, seed)
    if case["kind"] == "calibration":
        return None       # several thousand constrained dense systems: minutes in plain numpy
    P = Problem(_dataset(case, seed))
    if case["kind"] == "evaluate":
        return dict(R=P.observe(P.s0, P.a0, P.c0, partials=False)[0])
    h, A, gq, s, l, B = P.observe(P.s0, P.a0, P.c0)
    fn = case["weight_fn"]
    src, R, W, eps2 = _source_update(P, P.s0, h, A, P.sig2, fn)
    if case["kind"] == "static":
        return dict(sources=src, R=R, W=W, stats=None)
    if case["kind"] == "source" and case["attnoise_s"]:
        noise = _attitude_noise(P, R, eps2, case["attnoise_s"] * 10**9)
        h, A = P.observe(src, P.a0, P.c0)[:2]
        return dict(sources=_source_update(P, src, h, A, P.sig2 + noise, fn)[0])
    if case["kind"] == "source":
        return dict(sources=src)
    att = _attitude_update(P, P.a0, R, W, gq, s, l, B, case["seg_len"])
    if case["kind"] == "attitude":
        return dict(attitude=att)
    cal = _calibration_update(P, P.c0, R, W)
    src, att = _frame(P, src, att)
    return dict(sources=src, attitude=att, calibration=cal)
