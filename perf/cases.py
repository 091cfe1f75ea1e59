"""What a user of the library has it do, as timed cases.

Families (a case's "family"): `step` runs the step driver (push and deposit,
field update, sort by cell) from a particle and field state; `field` advances
the fields alone; `lines` runs the batched 1D lines; `grad` takes the gradient
of the horizon flux.  `exact` restates the method in 64-bit torch from its
equations (arXiv:2503.04558), without the library.

A step pass restores the state it starts from, as a program does that restarts
from a saved state, so that every pass does the same work.  The particles of a
saved state are in the order of an earlier sort.
"""
import math

import numpy as np
import torch

from paper_2503_04558_gb300 import grpic as G

NG = 2
KINDS = {"wald": G.WALD, "split": G.SPLIT_MONOPOLE, "monopole": G.MONOPOLE}


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _step(name=None, **kw):
    c = dict(family="step", precision=32, nr=128, nth=128, n=200000, a=0.9, r_out=50.0, kind="wald", b0=1.0,
             thermal=0.0, nsteps=2, pusher=0, shape=1, tol=1e-6, rad=0)
    c.update(kw)
    return c if name is None else dict(name=name, **c)


def listed():
    return [
        # a test-sized run in the FP32 form: launches and the gaps between them count
        _step("step32_128", nsteps=8),
        # an ordinary FP32 run
        _step("step32_512", nr=512, nth=512, n=512 * 512 * 64),
        # production size: split monopole, 100 particles per cell, hot plasma
        _step("step32_2048", nr=2048, nth=2048, n=2048 * 2048 * 100, a=0.99, r_out=100.0, kind="split", thermal=0.3),
        # odd grid, every corrector, Vay's momentum update
        _step("step32_vay_odd", nr=301, nth=182, n=2000002, pusher=1, tol=0.0),
        # the FP64 path: the 20-step parity run's size
        _step("step64_128", precision=64, nsteps=4),
        # an ordinary FP64 run
        _step("step64_512", precision=64, nr=512, nth=512, n=512 * 512 * 64, a=0.99, r_out=100.0, kind="split",
              thermal=0.3),
        # FP64 with the cubic particle shape, odd sizes
        _step("step64_cubic_odd", precision=64, nr=250, nth=190, n=1500002, shape=3),
        # the 2D pair cascade: emission, conversion, injection, a growing particle number
        _step("pairs64_512", precision=64, nr=512, nth=512, n=512 * 512 * 16, a=0.99, r_out=100.0, b0=500.0, rad=1),
        # vacuum fields alone, production grid in FP32 and a parity-sized one in FP64
        dict(name="field32_2048", family="field", precision=32, nr=2048, nth=2048, a=0.99, r_out=100.0, kind="split"),
        dict(name="field64_1024", family="field", precision=64, nr=1024, nth=1024, a=0.9, r_out=50.0, kind="wald"),
        # 512 spark-gap lines of uneven particle counts
        dict(name="lines_512", family="lines", nl=512, ncells=4096, a=0.99, lo=3.0, hi=5.0, nsteps=20),
        # gradient of the horizon Poynting flux
        dict(name="grad_256", family="grad", nr=256, nth=256, n=2000000, a=0.9, r_out=50.0, nsteps=10),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _even(v):
    return int(v) // 2 * 2


def draw(rng):
    fam = rng.choice(["step32", "step32", "step32", "step64", "step64", "pairs", "field", "field", "lines", "grad"])
    a = round(rng.uniform(0.0, 0.995), 3)
    r_out = round(rng.uniform(10.0, 100.0), 1)
    if fam in ("step32", "step64"):
        p = 32 if fam == "step32" else 64
        nr = _log(rng, 64, 2048 if p == 32 else 512)
        nth = _even(_log(rng, 64, 2048 if p == 32 else 512))
        ppc = math.exp(rng.uniform(math.log(4.0), math.log(100.0 if p == 32 else 64.0)))
        kind = rng.choice(["wald", "split"])
        return _step(precision=p, nr=nr, nth=nth, n=_even(nr * nth * ppc), a=a, r_out=r_out, kind=kind,
                     thermal=0.3 if kind == "split" else 0.0, pusher=rng.choice([0, 0, 0, 1]),
                     shape=rng.choice([1, 1, 3]) if p == 64 else 1, tol=rng.choice([1e-6, 1e-6, 0.0]))
    if fam == "pairs":
        nr, nth = _log(rng, 64, 512), _even(_log(rng, 64, 512))
        return _step(precision=64, nr=nr, nth=nth, n=_even(nr * nth * rng.uniform(4.0, 16.0)), a=a, r_out=r_out,
                     b0=500.0, rad=1)
    if fam == "field":
        p = rng.choice([32, 64])
        m = 2048 if p == 32 else 1024
        return dict(family="field", precision=p, nr=_log(rng, 64, m), nth=_even(_log(rng, 64, m)), a=a, r_out=r_out,
                    kind=rng.choice(["wald", "split"]))
    if fam == "lines":
        return dict(family="lines", nl=_log(rng, 8, 512), ncells=_log(rng, 512, 4096), a=a, lo=3.0,
                    hi=round(rng.uniform(3.5, 5.0), 2), nsteps=20)
    return dict(family="grad", nr=_log(rng, 32, 256), nth=_even(_log(rng, 32, 256)), n=_even(_log(rng, 4000, 2000000)),
                a=a, r_out=r_out, nsteps=rng.randint(2, 10))


def _config(case):
    a = case["a"]
    rh = 1.0 + math.sqrt(1.0 - a * a)
    kw = {}
    if case["family"] == "step":
        p = case["precision"]
        kw = dict(precision=p, pusher=case["pusher"], shape_order=case["shape"], fp64_radius=1.5 * rh,
                  push_tol=case["tol"] if p == 32 else 0.0)
        if case["rad"]:
            kw.update(radiation=1, injection=1, gamma_thr=100.0, eps_ph=4.0, tau=2.0, sigma_thr=10.0, eps_db=1e-3,
                      seed=1)
    elif case["family"] == "field":
        kw = dict(precision=case["precision"])
    return G.Config(case["nr"], case["nth"], a, 0.9 * rh, case["r_out"], **kw)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
_MJ = {}


def _mj_quantiles(T, device):
    """Quantiles of |u| of the Maxwell-Juettner distribution at temperature T."""
    if T not in _MJ:
        u = np.linspace(0.0, 60.0 * T + 4.0, 200001)
        g = np.sqrt(1.0 + u * u)
        f = u * u * np.exp((1.0 - g) / T)
        cdf = np.concatenate([[0.0], np.cumsum(0.5 * (f[1:] + f[:-1]))])
        _MJ[T] = np.interp(np.linspace(0.0, cdf[-1] * (1 - 1e-9), 65537), cdf, u)
    return torch.from_numpy(_MJ[T]).to(device=device, dtype=torch.float32)


def _particles(case, cfg, seed, device, sort_order=True):
    """e-/e+ pairs at shared uniform positions of every cell, in cell order,
    with Gaussian (sigma 0.1) or thermal momenta: cell, o1, o2 (offsets in the
    cell, o2 from the row's lower edge), u_r, u_theta, u_phi, tag."""
    n, nr, nth = case["n"], cfg.n_r, cfg.n_theta
    m = n // 2
    gen = torch.Generator(device=device)
    gen.manual_seed(int(seed) * 7919 + 17)
    cell = (torch.arange(m, device=device, dtype=torch.int64) * (nr * nth)).div_(m, rounding_mode="floor")
    cell = cell.to(torch.int32)
    if not sort_order:
        cell = cell[torch.randperm(m, generator=gen, device=device)]
    cell = cell.repeat_interleave(2)
    o1 = torch.rand(m, generator=gen, device=device).repeat_interleave(2)
    o2 = torch.rand(m, generator=gen, device=device).repeat_interleave(2)
    if case.get("thermal"):
        q = _mj_quantiles(case["thermal"], device)
        w = torch.rand(n, generator=gen, device=device) * 65535.0
        k = w.to(torch.int32)
        w -= k
        mag = q[k] * (1.0 - w) + q[k + 1] * w
        del k, w
        z = torch.rand(n, generator=gen, device=device) * 2.0 - 1.0
        ph = torch.rand(n, generator=gen, device=device) * (2.0 * math.pi)
        s = torch.sqrt(1.0 - z * z) * mag
        u1, u2, u3 = mag.mul_(z), s * torch.cos(ph), s * torch.sin(ph)
        del z, ph, s, mag
    else:
        u1, u2, u3 = (torch.randn(n, generator=gen, device=device) * 0.1 for _ in range(3))
    j = cell.div(nr, rounding_mode="floor")
    r = cfg.r_in * torch.exp(((cell - j * nr) + o1) * cfg.dx1)
    u2.mul_(r)
    u3.mul_(r).mul_(torch.sin((j + o2) * cfg.dth))
    tag = torch.arange(n, device=device, dtype=torch.int32) & 1
    return cell, o1, o2, u1, u2, u3, tag


def _to_fp64(cfg, p):
    """(r, theta, u_r, u_theta, u_phi, tag) in 64 bits."""
    cell, o1, o2, u1, u2, u3, tag = p
    j = cell.div(cfg.n_r, rounding_mode="floor")
    r = cfg.r_in * torch.exp(((cell - j * cfg.n_r).double() + o1.double()) * cfg.dx1)
    th = (j.double() + o2.double()) * cfg.dth
    return r, th, u1.double(), u2.double(), u3.double(), tag


def _to_fp32(cfg, p):
    """The FP32 form's arrays: the last row's offset counts from the pole."""
    cell, o1, o2, u1, u2, u3, tag = p
    last = cell >= cfg.n_r * (cfg.n_theta - 1)
    return o1, torch.where(last, 1.0 - o2, o2), u1, u2, u3, tag, cell


def _lines(case, seed):
    """Line inclinations and, per line, 10^U(lo, hi) particles in pairs at
    shared uniform positions (counts and slots padded to the longest line)."""
    nl, nc = case["nl"], case["ncells"]
    rng = np.random.default_rng(nl * 10007 + nc)  # the counts are the workload's, not the draw's
    cnt = (10 ** rng.uniform(case["lo"], case["hi"], nl)).astype(np.int64) // 2 * 2
    m = int(cnt.max())
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) * 104729 + 3)
    x = (torch.rand(nl, m // 2, generator=gen, device="cuda", dtype=torch.float64) * nc).repeat_interleave(2, dim=1)
    cell = x.floor().clamp_(max=nc - 1)
    off = (x - cell).clamp_(max=1.0 - 2.0 ** -24).float().clamp_(max=1.0 - 2.0 ** -24)
    ur = torch.randn(nl, m, generator=gen, device="cuda") * 0.1
    start = torch.from_numpy(np.concatenate([[0], np.cumsum(cnt)[:-1]])).cuda()
    pid = start[:, None] + torch.arange(m, device="cuda")[None, :]
    tag = (torch.arange(m, device="cuda", dtype=torch.int32) & 1).expand(nl, m).contiguous()
    return cnt, m, dict(cell=cell.to(torch.int32), off=off, ur=ur, up=torch.zeros_like(ur), tag=tag, id=pid)


# ---------------------------------------------------------------------------
# a pass
# ---------------------------------------------------------------------------
def prepare(case, seed):
    fam = case["family"]
    if fam == "lines":
        return _prepare_lines(case, seed)
    cfg = _config(case)
    ctx = G.Context(cfg)
    F = G.Fields(cfg)
    ctx.init_fields(F, KINDS[case.get("kind", "wald")], case.get("b0", 1.0))
    s = dict(case=case, cfg=cfg, ctx=ctx, F=F)
    if fam == "field":
        # currents of a plasma: noise of a few per cent of the fields' circulation
        gen = torch.Generator(device="cuda")
        gen.manual_seed(int(seed) * 31 + 7)
        for k, J in enumerate(F.J):
            J.copy_(torch.randn(J.shape, generator=gen, device="cuda") * 1e-3)
        return s
    p = _particles(case, cfg, seed, "cuda", sort_order=fam == "step")
    if fam == "grad":
        r, th, u1, u2, u3, tag = _to_fp64(cfg, p)
        s.update(x=[r, th, u1, u2, u3], tag=tag, iH=G.horizon_index(ctx))
        return s
    arrays = _to_fp64(cfg, p) if case["precision"] == 64 else _to_fp32(cfg, p)
    del p
    s["start"] = arrays
    s["fields"] = [t.clone() for t in F.D + F.B]
    P = s["P"] = G.ParticleSet(cfg, 3 * case["n"] if case["rad"] else case["n"])
    P.load(*arrays)
    _advance(s)
    s["live"] = P.live()
    return s


def _prepare_lines(case, seed):
    rh = 1.0 + math.sqrt(1.0 - case["a"] ** 2)
    cnt, m, start = _lines(case, seed)
    cfg = G.Batch1DConfig(case["nl"], case["ncells"], case["a"], rh, 20.0, 2 * m + 1024)
    B, L = G.Batch1D(cfg), G.Lines(cfg)
    nl = case["nl"]
    theta = (torch.arange(nl, dtype=torch.float64) + 0.5) * (math.pi / 2) / nl
    L.theta.copy_(theta)
    # imposed current: horizon rotation frequency x monopole strength x sin^2
    L.I0.copy_(case["a"] / (2.0 * rh) * cfg.B0 * torch.sin(theta) ** 2)
    B.init_fields(L)
    B.set_launch(1024, 1, 1)
    s = dict(case=case, B=B, L=L, m=m, start=start, count=torch.from_numpy(cnt).to(torch.int32).cuda(),
             D=L.D.clone())
    _advance_lines(s)
    # the live slots of all lines, padded (by a slot that is never written) to a
    # length that does not depend on the draw
    n = L.count.long()
    cap = cfg.capacity
    k = torch.repeat_interleave(torch.arange(nl, device="cuda"), n)
    first = torch.cumsum(n, 0) - n
    s["slots"] = torch.full((max(int(1.5 * cnt.sum()), k.numel()),), cap - 1, device="cuda")
    s["slots"][:k.numel()] = torch.arange(k.numel(), device="cuda") - first[k] + k * cap
    return s


def _advance(s):
    P, F = s["P"], s["F"]
    n = P.n = s["case"]["n"]
    x, ints = s["start"][:5], s["start"][5:]
    now = [t[:n] for t in P.a.arrays() if t is not None]
    torch._foreach_copy_(now[:5] + F.D + F.B, list(x) + s["fields"])
    torch._foreach_copy_(now[5:], list(ints))
    P.count.fill_(n)
    s["ctx"].step(P, F, s["case"]["nsteps"])


def _advance_lines(s):
    L, m = s["L"], s["m"]
    for key, v in s["start"].items():
        L.buf[L.cur][key][:, :m].copy_(v)
    L.count.copy_(s["count"])
    L.D.copy_(s["D"])
    L.events.zero_()
    s["B"].run_graph(L, s["case"]["nsteps"], 0)


def run(s):
    fam = s["case"]["family"]
    F = s.get("F")
    if fam == "field":
        s["ctx"].field_update(F)
        return {"D": F.D, "B": F.B}
    if fam == "grad":
        L, gp, gf = G.adjoint_grad(s["ctx"], s["x"], s["tag"], F.D, F.B, s["case"]["nsteps"], s["iH"])
        return {"L": L, "grad_p": gp, "grad_f": gf}
    if fam == "lines":
        _advance_lines(s)
        L, q = s["L"], s["slots"]
        return {"count": L.count, "events": L.events, "D": L.D, "JA": L.JA,
                "particles": {k: v.view(-1)[q] for k, v in L.buf[L.cur].items()}}
    _advance(s)
    P, n = s["P"], s["live"]
    x = P.a.arrays()
    # slots past the live ones hold what was there before: cleared
    torch._foreach_zero_([t[n:] for t in x[:5]])
    out = {"D": F.D, "B": F.B, "J": F.J, "live": P.count, "x1": x[0], "x2": x[1], "u1": x[2], "u2": x[3], "u3": x[4],
           "tag": x[5]}
    if x[6] is not None:
        x[6][n:].zero_()
        out["cell"] = x[6]
    return out


def work(case):
    """Inputs and outputs once; the method's own arithmetic: per particle-step
    the metric and right-hand side four times, the momentum update, the
    interpolation and the deposit (about 600 operations); per point and stage
    of the field update about 60."""
    fam = case["family"]
    if fam == "lines":
        n = case["nl"] * (10 ** case["hi"] - 10 ** case["lo"]) / (math.log(10.0) * (case["hi"] - case["lo"]))
        return {"bytes": 56.0 * n + 8.0 * case["nl"] * case["ncells"], "flops": 300.0 * n * case["nsteps"]}
    cells = (case["nr"] + 1.0) * (case["nth"] + 1.0)
    e = 4 if case.get("precision", 64) == 32 else 8
    if fam == "field":
        return {"bytes": 15.0 * e * cells, "flops": 480.0 * cells}
    n, k = case["n"], case["nsteps"]
    if fam == "grad":
        return {"bytes": (10 * 8 + 4.0) * n + 12.0 * 8 * cells, "flops": k * (600.0 * 4 * n + 480.0 * 3 * cells)}
    per = 28.0 if e == 4 else 44.0
    f = 1000.0 if case["shape"] == 3 else 600.0
    return {"bytes": 2 * per * n + 15.0 * e * cells, "flops": k * (f * n + 480.0 * cells)}


# ---------------------------------------------------------------------------
# the method in 64-bit torch
# ---------------------------------------------------------------------------
class _Ref:
    """Kerr-Schild metric, face areas and field update of one configuration."""

    def __init__(self, cfg, device):
        self.c, self.dev = cfg, device
        self.a = cfg.a
        f = dict(device=device, dtype=torch.float64)
        i = torch.arange(cfg.ld, **f) - NG
        j = torch.arange(cfg.n_theta + 1, **f)
        ri, rh, rm, rp = (cfg.r_in * torch.exp((i + o) * cfg.dx1)[None, :] for o in (0.0, 0.5, -0.5, 1.0))
        tj, th, t1 = ((j + o)[:, None] * cfg.dth for o in (0.0, 0.5, 1.0))
        lo, hi = ((j - 0.5) * cfg.dth).clamp(min=0.0)[:, None], ((j + 0.5) * cfg.dth).clamp(max=math.pi)[:, None]
        one_r, one_t = torch.ones_like(ri), torch.ones_like(tj)
        self.top = (j == cfg.n_theta)[:, None]
        self.axis = self.top | (j == 0)[:, None]
        gx, gw = np.polynomial.legendre.leggauss(10)

        def quad(r0, r1, t0_, t1_):
            """integral of sqrt(gamma) over r (r0..r1, or at r0) and theta."""
            rs = [(r0, 1.0)] if r1 is None else [(0.5 * (r1 + r0) + 0.5 * (r1 - r0) * x, 0.5 * (r1 - r0) * w)
                                                 for x, w in zip(gx, gw)]
            ts = [(t0_, 1.0)] if t1_ is None else [(0.5 * (t1_ + t0_) + 0.5 * (t1_ - t0_) * x, 0.5 * (t1_ - t0_) * w)
                                                   for x, w in zip(gx, gw)]
            s = 0.0
            for r, wr in rs:
                for t, wt in ts:
                    s = s + self.sqrtg(r, t) * wr * wt
            return s

        def inv(A, off):
            return torch.where(off | (A <= 0), torch.zeros_like(A), 1.0 / A)

        no = torch.zeros_like(self.top)
        self.iA = [inv(quad(rh, None, lo, hi), no), inv(quad(rm, rh, th, None), self.top), inv(quad(rm, rh, lo, hi), no),
                   inv(quad(ri, None, tj, t1), self.top), inv(quad(ri, rp, tj, None), self.axis),
                   inv(quad(ri, rp, tj, t1), self.top)]
        z = lambda v: torch.where(self.top, torch.zeros_like(v), v)
        m = self.metric(rh * one_t, torch.sin(tj) * one_r, torch.cos(tj) * one_r)     # (i+1/2, j)
        self.rr_dr, self.rp_dr, self.tt_bt, self.sb_bt = (m["al"] * m["rr"], m["al"] * m["rp"], m["al"] * m["tt"],
                                                          m["sg"] * m["be"])
        m = self.metric(ri * one_t, torch.sin(tj) * one_r, torch.cos(tj) * one_r)     # (i, j)
        self.pp_dp, self.rp_dp, self.sb_dp = m["al"] * m["pp"], m["al"] * m["rp"], m["sg"] * m["be"]
        m = self.metric(ri * one_t, torch.sin(th) * one_r, torch.cos(th) * one_r)     # (i, j+1/2)
        self.tt_dt, self.sb_dt, self.rr_br, self.rp_br = (z(m["al"] * m["tt"]), z(m["sg"] * m["be"]),
                                                          z(m["al"] * m["rr"]), z(m["al"] * m["rp"]))
        m = self.metric(rh * one_t, torch.sin(th) * one_r, torch.cos(th) * one_r)     # (i+1/2, j+1/2)
        self.pp_bp, self.rp_bp, self.sb_bp = z(m["al"] * m["pp"]), z(m["al"] * m["rp"]), z(m["sg"] * m["be"])
        self.drp, self.drd = rp - ri, rh - rm
        d = cfg.damp_cells
        x0 = cfg.n_r - d
        prof = lambda o: 1.0 - cfg.damp_max * ((i + o - x0) / max(d, 1)).clamp(0.0, 1.0)[None, :] ** 3
        self.damp_i, self.damp_h = prof(0.0), prof(0.5)

    def sqrtg(self, r, th):
        rho2 = r * r + (self.a * torch.cos(th)) ** 2
        return rho2 * torch.sin(th) * torch.sqrt(1.0 + 2.0 * r / rho2)

    def metric(self, r, s, c):
        a = self.a
        s2 = s * s
        rho2 = r * r + a * a * c * c
        z = 2.0 * r / rho2
        o = 1.0 + z
        al = torch.rsqrt(o)
        return dict(al=al, be=z / o, rr=o, rp=-a * s2 * o, tt=rho2,
                    pp=s2 * (r * r + a * a + z * a * a * s2), irr=(a * a + r * r) / rho2 - z / o, irp=a / rho2,
                    itt=1.0 / rho2, ipp=1.0 / (rho2 * s2), sg=rho2 * s * torch.sqrt(o), z=z, rho2=rho2)

    # -- fields -------------------------------------------------------------
    def aux(self, X):
        R = lambda v: torch.roll(v, -1, 1)  # column i + 1
        L = lambda v: torch.roll(v, 1, 1)   # column i - 1
        hR, hL = lambda v: 0.5 * (v + R(v)), lambda v: 0.5 * (v + L(v))
        Dr, Dt, Dp, Br, Bt, Bp = X
        return dict(Hr=self.rr_br * Br + hL(self.rp_bp * Bp), Ht=self.tt_bt * Bt + hR(self.sb_dp * Dp),
                    Hp=self.pp_bp * Bp + hR(self.rp_br * Br) - hR(self.sb_dt * Dt),
                    Er=self.rr_dr * Dr + hR(self.rp_dp * Dp), Et=self.tt_dt * Dt - hL(self.sb_bp * Bp),
                    Ep=self.pp_dp * Dp + hL(self.rp_dr * Dr) + hL(self.sb_bt * Bt))

    def circ(self, X):
        A = self.aux(X)
        R = lambda v: torch.roll(v, -1, 1)
        L = lambda v: torch.roll(v, 1, 1)
        up = lambda v: torch.roll(v, -1, 0)  # row j + 1
        dn = lambda v: torch.roll(v, 1, 0)   # row j - 1
        top, axis, dth = self.top, self.axis, self.c.dth
        Z = torch.zeros((), dtype=torch.float64, device=self.dev)
        first = torch.zeros_like(top)
        first[0] = True
        hp = torch.where(top, Z, A["Hp"])
        hm = torch.where(first, Z, dn(A["Hp"]))
        C = [(hp - hm), L(A["Hp"]) - A["Hp"],
             torch.where(axis, Z, (A["Ht"] - L(A["Ht"])) * dth + (dn(A["Hr"]) - A["Hr"]) * self.drd),
             -(up(A["Ep"]) - A["Ep"]), torch.where(axis, Z, -(A["Ep"] - R(A["Ep"]))),
             -((R(A["Et"]) - A["Et"]) * dth + (A["Er"] - up(A["Er"])) * self.drp)]
        return [v * w for v, w in zip(C, self.iA)]

    def bounds(self, X, X0):
        nr, out = self.c.n_r, []
        for k, v in enumerate(X):
            half_r, half_t = k in (0, 4, 5), k in (1, 3, 5)
            if k in (2, 4):
                v = torch.where(self.axis, torch.zeros_like(v), v)
            last = (nr - 1 if half_r else nr) + NG
            v = torch.cat([v[:, NG:NG + 1].expand(-1, NG), v[:, NG:last + 1],
                           v[:, last:last + 1].expand(-1, self.c.ld - last - 1)], 1)
            out.append(torch.where(self.top, X0[k], v) if half_t else v)
        return out

    def field_update(self, X0, J):
        c = self.c
        Jd = [j * w for j, w in zip(J, self.iA)] + [0.0] * 3
        C0 = self.circ(X0)
        X = self.bounds([x + c.dt * (k - j) for x, k, j in zip(X0, C0, Jd)], X0)
        for it in range(c.n_field_iter):
            C = self.circ(X)
            Y = [x + c.dt * ((1.0 - c.beta_field) * k0 + c.beta_field * k - j) for x, k0, k, j in zip(X0, C0, C, Jd)]
            if it == c.n_field_iter - 1:
                Y = [y * (self.damp_h if k in (0, 4, 5) else self.damp_i) for k, y in enumerate(Y)]
            X = self.bounds(Y, X0)
        return X

    def flux(self, X, iH):
        A = self.aux(X)
        q, e = iH + NG, slice(0, self.c.n_theta)
        at = lambda k, i: A[k][:, i]
        Et = at("Et", q)[e]
        Hp = 0.5 * (at("Hp", q - 1) + at("Hp", q))[e]
        Ep = 0.5 * (at("Ep", q)[:-1] + at("Ep", q)[1:])
        h = at("Ht", q - 1) + at("Ht", q)
        Ht = 0.25 * (h[:-1] + h[1:])
        return ((Et * Hp - Ep * Ht) * self.c.dth).sum()

    # -- particles -----------------------------------------------------------
    def weight(self, d):
        d = d.abs()
        if self.c.shape_order == 1:
            return (1.0 - d).clamp(min=0.0)
        return torch.where(d < 1.0, 2.0 / 3.0 - d * d + 0.5 * d ** 3, (2.0 - d).clamp(min=0.0) ** 3 / 6.0)

    def mirror(self, j, half_t):
        n = self.c.n_theta
        top = n - 1 if half_t else n
        k = -1 if half_t else 0
        flip = (j < 0) | (j > top)
        return torch.where(j < 0, k - j, torch.where(j > top, 2 * n + k - j, j)), flip

    def gather(self, F, x1, x2, half_r, half_t, par):
        y1, y2 = x1 - 0.5 * half_r, x2 - 0.5 * half_t
        lo, hi = (0, 2) if self.c.shape_order == 1 else (-1, 3)
        b1, b2 = y1.detach().floor().long(), y2.detach().floor().long()
        if not half_t and self.c.shape_order == 1:
            b2 = b2.clamp(max=self.c.n_theta - 1)
        flat, v = F.reshape(-1), 0.0
        for q in range(lo, hi):
            row, flip = self.mirror(b2 + q, half_t)
            wq = self.weight(y2 - (b2 + q)) * torch.where(flip, par, 1.0)
            for p in range(lo, hi):
                v = v + wq * self.weight(y1 - (b1 + p)) * flat[row * self.c.ld + b1 + p + NG]
        return v

    def rhs(self, r, s, c, ur, ut, up, eps):
        a = self.a
        m = self.metric(r, s, c)
        rho2, z, o, al = m["rho2"], m["z"], m["rr"], m["al"]
        uu = m["irr"] * ur * ur + 2.0 * m["irp"] * ur * up + m["itt"] * ut * ut + m["ipp"] * up * up
        au0 = torch.sqrt(eps + uu)
        iu0 = al / au0
        # r and theta derivatives of rho^2, z, lapse, shift and gamma^ij
        dz = (2.0 / rho2 - z * z, -z * (-2.0 * a * a * c * s) / rho2)
        dq = (2.0 * r / rho2, -2.0 * a * a * c * s / rho2)      # d ln rho^2
        P = (a * a + r * r) * ur * ur + 2.0 * a * ur * up + ut * ut + up * up / (s * s)
        dP = (2.0 * r * ur * ur, -2.0 * c * up * up / (s ** 3))
        U = []
        for k in range(2):
            dbeta = dz[k] / (o * o)
            dG = dP[k] / rho2 - dq[k] * P / rho2 - dbeta * ur * ur
            U.append(au0 * 0.5 * dz[k] * al / o + ur * dbeta - 0.5 * iu0 * dG)
        return ((m["irr"] * ur + m["irp"] * up) * iu0 - m["be"], m["itt"] * ut * iu0,
                (m["irp"] * ur + m["ipp"] * up) * iu0, U[0], U[1])

    def kick(self, m, qm, u, D, B):
        dt = self.c.dt
        low = lambda v: (m["rr"] * v[0] + m["rp"] * v[2], m["tt"] * v[1], m["rp"] * v[0] + m["pp"] * v[2])
        up = lambda v: (m["irr"] * v[0] + m["irp"] * v[2], m["itt"] * v[1], m["irp"] * v[0] + m["ipp"] * v[2])
        dot = lambda x, y: x[0] * y[0] + x[1] * y[1] + x[2] * y[2]
        cross = lambda x, y: (x[1] * y[2] - x[2] * y[1], x[2] * y[0] - x[0] * y[2], x[0] * y[1] - x[1] * y[0])
        sg, h = m["sg"], 0.5 * qm * dt * m["al"]
        E = low(D)
        if self.c.pusher == 0:
            um = [a + h * b for a, b in zip(u, E)]
            v = up(um)
            k = h / torch.sqrt(1.0 + dot(um, v))
            t = [k * b for b in B]
            f = 2.0 / (1.0 + dot(t, low(t)))
            w = [a + sg * b for a, b in zip(um, cross(v, t))]
            x = cross(up(w), [f * b for b in t])
            return [a + sg * b + h * e for a, b, e in zip(um, x, E)]
        w = up(u)
        g = torch.sqrt(1.0 + dot(u, w))
        x = cross(w, B)
        p = [a + 2.0 * h * e + h * sg / g * b for a, e, b in zip(u, E, x)]
        t = [h * b for b in B]
        tl = low(t)
        tt, us, q = dot(t, tl), dot(p, t), up(p)
        sig = 1.0 + dot(p, q) - tt
        g1 = torch.sqrt(0.5 * (sig + torch.sqrt(sig * sig + 4.0 * (tt + us * us))))
        x = cross(q, t)
        return [(a + us * b / (g1 * g1) + sg / g1 * d) / (1.0 + tt / (g1 * g1)) for a, b, d in zip(p, tl, x)]

    def push(self, X, x, tag, alive):
        """One push and deposit: (state, alive, J)."""
        c, dev = self.c, self.dev
        r, th, u1, u2, u3 = x
        tab = lambda v: torch.tensor(v, dtype=torch.float64, device=dev)[(tag & 3).long()]
        qm, qw, mass = tab(c.q_over_m), tab(c.q_weight), tab(tuple(float(v) for v in c.massive))
        x1a, x2a = torch.log(r / c.r_in) / c.dx1, th / c.dth
        s0, c0 = torch.sin(th), torch.cos(th)
        lat = [(1, 0, 1.0), (0, 1, -1.0), (0, 0, 1.0), (0, 1, 1.0), (1, 0, -1.0), (1, 1, 1.0)]
        E = [self.gather(X[k], x1a, x2a, *lat[k]) for k in range(6)]
        k = self.kick(self.metric(r, s0, c0), qm, (u1, u2, u3), E[:3], E[3:])
        ch = (mass > 0) & (qm != 0)
        v1, v2, v3 = (torch.where(ch, a, b) for a, b in zip(k, (u1, u2, u3)))
        f0 = self.rhs(r, s0, c0, v1, v2, v3, mass)
        y = [b + c.dt * f for b, f in zip((r, th), f0[:2])] + [b + c.dt * f for b, f in zip((v1, v2), f0[3:])]
        ph = c.dt * f0[2]
        for _ in range(c.n_push_iter):
            f = self.rhs(y[0], torch.sin(y[1]), torch.cos(y[1]), y[2], y[3], v3, mass)
            y = [b + 0.5 * c.dt * (p + q) for b, p, q in
                 zip((r, th, v1, v2), f0[:2] + f0[3:], f[:2] + f[3:])]
            ph = 0.5 * c.dt * (f0[2] + f[2])
        rn, tn, w1, w2 = y
        flip = (tn < 0) | (tn > math.pi)
        tn = torch.where(tn < 0, -tn, torch.where(tn > math.pi, 2.0 * math.pi - tn, tn))
        w2 = torch.where(flip, -w2, w2)
        x1b, x2b = torch.log(rn.clamp(min=1e-3) / c.r_in) / c.dx1, tn / c.dth
        fl = lambda v: v.detach().floor()
        ok = alive & torch.isfinite(rn + tn + w1 + w2 + ph) & ((fl(x1b) - fl(x1a)).abs() <= 1) & \
            ((fl(x2b).clamp(max=c.n_theta - 1) - fl(x2a).clamp(max=c.n_theta - 1)).abs() <= 1)
        J = self.deposit(torch.where(ok, qw, 0.0), x1a, x2a, torch.where(ok, x1b, x1a), torch.where(ok, x2b, x2a),
                         torch.where(ok, ph, 0.0))
        keep = lambda a, b: torch.where(ok, a, b)
        alive = ok & (rn >= c.r_in) & (rn < c.r_out)
        return (keep(rn, r), keep(tn, th), keep(w1, u1), keep(w2, u2), keep(v3, u3)), alive, J

    def deposit(self, qw, x1a, x2a, x1b, x2b, ph):
        c = self.c
        b1 = torch.minimum(x1a.detach().floor(), x1b.detach().floor()).long() - 1
        b2 = torch.minimum(x2a.detach().floor(), x2b.detach().floor()).long() - 1
        S0r, S1r = ([self.weight(x - (b1 + k)) for k in range(5)] for x in (x1a, x1b))
        S0t, S1t = ([self.weight(x - (b2 + k)) for k in range(5)] for x in (x2a, x2b))
        n = (c.n_theta + 1) * c.ld
        J = [torch.zeros(n, dtype=torch.float64, device=self.dev) for _ in range(3)]

        def add(q, k, l, half_t, odd, v):
            row, flip = self.mirror(b2 + l, half_t)
            row = row.clamp(0, c.n_theta)
            col = b1 + k + NG
            v = torch.where((col < 0) | (col >= c.ld), 0.0, v * torch.where(flip, odd, 1.0))
            J[q] = J[q].index_add(0, row * c.ld + col.clamp(0, c.ld - 1), v)

        cr, cp = -qw / (2.0 * c.dt), qw * ph / c.dt
        p = 0.0
        for k in range(4):
            p = p + S1r[k] - S0r[k]
            for l in range(5):
                add(0, k, l, False, 1.0, cr * p * (S1t[l] + S0t[l]))
        p = 0.0
        for l in range(4):
            p = p + S1t[l] - S0t[l]
            for k in range(5):
                add(1, k, l, True, -1.0, cr * p * (S1r[k] + S0r[k]))
        for k in range(5):
            for l in range(5):
                add(2, k, l, False, 1.0, cp * (S1r[k] * (S1t[l] / 3 + S0t[l] / 6) + S0r[k] * (S1t[l] / 6 + S0t[l] / 3)))
        return [j.view(c.n_theta + 1, c.ld) for j in J]


def exact(case, seed):
    fam = case["family"]
    # emission and conversion draw random numbers of the library's own stream
    if fam == "lines" or case.get("rad") or case.get("n", 0) > 20000000:
        return None
    s = prepare(dict(case, n=min(case.get("n", 0), 64)) if fam == "step" else case, seed)
    cfg, F = s["cfg"], s["F"]
    ref = _Ref(cfg, "cuda")
    if fam == "step":
        X = [t.double() for t in s["fields"]]
        p = _particles(case, cfg, seed, "cuda")
        if case["precision"] == 32:  # the last row's offset as the FP32 form holds it
            o1, q, u1, u2, u3, tag, cell = _to_fp32(cfg, p)
            o2 = torch.where(cell >= cfg.n_r * (cfg.n_theta - 1), 1.0 - q.double(), q.double())
            p = (cell, o1, o2, u1, u2, u3, tag)
    else:
        X = [t.double().clone() for t in F.D + F.B]
    if fam == "field":
        X = ref.field_update(X, [t.double() for t in F.J])
        return {"D": X[:3], "B": X[3:]}
    if fam == "grad":
        return _exact_grad(case, s, ref, X)
    *x, tag = _to_fp64(cfg, p)
    alive = torch.ones_like(tag, dtype=torch.bool)
    x = tuple(x)
    for _ in range(case["nsteps"]):
        x, alive, J = ref.push(X, x, tag, alive)
        X = ref.field_update(X, J)
        # the order of the stable sort by cell, the dead dropped
        i = (torch.log(x[0] / cfg.r_in) / cfg.dx1).floor().long().clamp(0, cfg.n_r - 1)
        j = (x[1] / cfg.dth).floor().long().clamp(max=cfg.n_theta - 1)
        key = torch.where(alive, j * cfg.n_r + i, cfg.n_r * cfg.n_theta)
        order = torch.sort(key, stable=True).indices[:int(alive.sum())]
        x, tag, alive = tuple(v[order] for v in x), tag[order], alive[order]
    out = {"D": X[:3], "B": X[3:], "J": J}
    # the FP32 form's slots are ordered by cells that its own rounding decides
    if case["precision"] == 64:
        pad = lambda v: torch.nn.functional.pad(v, (0, case["n"] - v.numel()))
        out.update({k: pad(v) for k, v in zip(("x1", "x2", "u1", "u2", "u3"), x)})
    return out


def _exact_grad(case, s, ref, X):
    from torch.utils.checkpoint import checkpoint
    tag, n = s["tag"], case["nsteps"]
    X0 = [t.requires_grad_() for t in X]
    x0 = [t.clone().requires_grad_() for t in s["x"]]

    def step(alive, *v):
        x, ok, J = ref.push(list(v[5:]), tuple(v[:5]), tag, alive)
        Y = ref.field_update(list(v[5:]), J)
        return (ok, ref.flux(Y, s["iH"])) + tuple(x) + tuple(Y)

    alive, v, L = torch.ones_like(tag, dtype=torch.bool), tuple(x0 + X0), 0.0
    for _ in range(n):
        alive, fl, *v = checkpoint(step, alive, *v, use_reentrant=False)
        L = L + fl / n
    g = torch.autograd.grad(L, x0 + X0)
    return {"L": float(L.detach()), "grad_p": list(g[:5]), "grad_f": list(g[5:])}
