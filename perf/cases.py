"""Workloads of the GRMHD step, each a call or a few calls of the public
binding: device primitives in, N cycles, device primitives out (or, for one of
them, the flux stage alone).

Every grid, precision mode and variant here is one that the benchmark, the
tests or the serving stream of this repository run.  Inputs come from
``problems`` and the seed; a pass sets the state from the input, so that every
pass on a state does the same work.
"""
import dataclasses
import math

import numpy as np
import torch

from paper_2110_10191_gb300 import grmhd, problems as pb

# algorithmic FP64 operations (add, multiply, divide, square root: one each)
# of one reconstructed zone, of one face and of one zone update, as counted by
# the oracle on the torus; MC needs an eighth of WENO5's
WENO_FLOPS, MC_FLOPS, FACE_FLOPS, ZONE_FLOPS = 770, 96, 530, 1100


def listed():
    torus = dict(kind="torus", recon="weno5", precision="fp64", r_out=50.0, spin=0.9375)
    return [
        # the accuracy test's linear mode: far too small to fill the GPU, so
        # launches and latency count
        dict(name="mode_64x64", kind="mode", n1=64, n2=64, recon="mc", cycles=10),
        # a flat vortex at a size that no block or walk length divides
        dict(name="vortex_217x217", kind="vortex", n1=217, recon="weno5", cycles=4),
        # many uneven small 2D grids advanced together (the batched workload)
        dict(name="batch_64_grids", kind="batch", grids=64, nmin=32, nmax=256, draw=0, cycles=2),
        # a small ragged torus, all three directions odd
        dict(torus, name="torus_61x45x37", n1=61, n2=45, n3=37, cycles=2),
        # the benchmark's torus: the headline workload
        dict(torus, name="torus_128", n1=128, n2=128, n3=128, cycles=2),
        # the largest torus, FP32 fluxes with the FP64 update
        dict(torus, name="torus_288_mixed", n1=288, n2=128, n3=128, r_out=1000.0,
             precision="mixed", cycles=2),
        # float-float fluxes and update
        dict(torus, name="torus_128_ff", n1=128, n2=128, n3=128, precision="ff", cycles=2),
        # FP32 fluxes with the float-float update: the fastest mode
        dict(torus, name="torus_128_mixed_ff", n1=128, n2=128, n3=128, precision="mixed_ff",
             cycles=2),
        # an inflow as the serving stream asks for it (fixed X1 ghosts)
        dict(name="bondi_96", kind="bondi", n1=96, n2=96, n3=96, recon="mc", precision="fp64",
             cycles=2),
        # the variants: bounds in the drift frame, electron heating
        dict(torus, name="torus_96_drift", n1=96, n2=96, n3=96, drift=True, cycles=2),
        dict(torus, name="torus_96_electrons", n1=96, n2=96, n3=96, electrons="kawazura",
             cycles=2),
        # the flux stage alone, on buffers the caller owns
        dict(torus, name="fluxes_61x45x37", kind="fluxes", n1=61, n2=45, n3=37),
    ]


def _size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["mode", "vortex", "batch", "torus", "torus", "torus", "torus", "bondi", "fluxes"])
    recon = rng.choice(["mc", "weno5"])
    if kind == "mode":
        return dict(kind=kind, n1=_size(rng, 32, 512), n2=_size(rng, 32, 512), recon=recon,
                    cycles=rng.randint(2, 10))
    if kind == "vortex":
        return dict(kind=kind, n1=_size(rng, 32, 512), recon=recon, cycles=rng.randint(2, 6))
    if kind == "batch":
        lo = _size(rng, 24, 64)
        return dict(kind=kind, grids=rng.randint(8, 64), nmin=lo, nmax=_size(rng, lo, 256),
                    draw=rng.randint(1, 1000), cycles=2)
    if kind == "bondi":
        return dict(kind=kind, n1=_size(rng, 24, 128), n2=_size(rng, 24, 128),
                    n3=rng.choice([1, _size(rng, 8, 128)]), recon=recon,
                    precision=rng.choice(["fp64", "mixed"]), cycles=2)
    n1, n2, n3 = _size(rng, 24, 128), _size(rng, 24, 128), rng.choice([1, _size(rng, 8, 96), _size(rng, 8, 96)])
    if kind == "fluxes":  # at most 123 zones each way fit its scratch
        return dict(kind=kind, n1=min(n1, 120), n2=min(n2, 120), n3=min(n3, 120), recon=recon,
                    precision="fp64", r_out=50.0, spin=rng.uniform(0.0, 0.98))
    case = dict(kind=kind, n1=n1, n2=n2, n3=n3, recon=recon,
                precision=rng.choice(["fp64", "fp64", "mixed", "ff", "mixed_ff"]),
                r_out=rng.choice([50.0, 1000.0]), spin=rng.uniform(0.0, 0.98), cycles=2)
    variant = rng.choice(["", "", "drift", "electrons"])
    if variant == "drift":
        case["drift"] = True
    if variant == "electrons":
        case["electrons"] = rng.choice(["kawazura", "werner", "rowan", "sharma", "howes"])
    return case


def _recon(case):
    return pb.RECON_WENO5 if case["recon"] == "weno5" else pb.RECON_MC


def _jitter(pr, seed, size):
    """`pr` with its internal energy multiplied by 1 + size * U(-1/2, 1/2), zone by zone."""
    z = pb.splitmix_uniform(seed + 1, np.arange(pr.P[0].size, dtype=np.uint64)).reshape(pr.P[0].shape)
    pr.P[pb.UU] *= 1.0 + size * (z - 0.5)
    return pr


def _problems(case, seed):
    kind = case["kind"]
    u = pb.splitmix_uniform(seed, np.arange(4, dtype=np.uint64))
    if kind == "mode":
        return [pb.linear_mode(case["n1"], "fast", amp=10.0 ** (-4.0 + 2.0 * u[0]), n2=case["n2"],
                               recon=_recon(case), periods=0.0)]
    if kind == "vortex":
        return [pb.orszag_tang(case["n1"], scale=0.5 + u[0], recon=_recon(case))]
    if kind == "batch":
        return [_jitter(pr, seed + g, 1e-3) for g, pr in
                enumerate(pb.batch_2d(case["grids"], case["nmin"], case["nmax"], seed=case["draw"]))]
    if kind == "bondi":
        pr = _jitter(pb.bondi(case["n1"], case["n2"], n3=case["n3"], recon=_recon(case)), seed, 1e-3)
        pr.info["P_ghost"][:, 3:-3, 3:-3, 3:-3] = pr.P
    else:
        pr = pb.fm_torus(case["n1"], case["n2"], case["n3"], a=case["spin"], r_out=case["r_out"],
                         recon=_recon(case), seed=seed)
    pr.precision = dict(fp64=grmhd.PREC_FP64, mixed=grmhd.PREC_MIXED, ff=grmhd.PREC_FF,
                        mixed_ff=grmhd.PREC_MIXED_FF)[case["precision"]]
    if case.get("drift"):
        pr.floor_frame = grmhd.FLOOR_DRIFT
    if case.get("electrons"):
        pr = pb.with_electrons(pr, getattr(pb, "ELEC_" + case["electrons"].upper()))
    return [pr]


@dataclasses.dataclass
class State:
    case: dict
    problems: list
    sims: list    # one simulation per problem
    P: list       # device primitives in
    K: list       # device electron entropies in (or None)
    out: list     # device results
    batch: object = None


def prepare(case, seed):
    prs = _problems(case, seed)
    stream = torch.cuda.current_stream()
    dev = [torch.from_numpy(np.ascontiguousarray(p.info.get("P_ghost", p.P))).cuda() for p in prs]
    if case["kind"] == "fluxes":  # the caller's buffers: primitives with ghosts in, fluxes out
        sim = grmhd.Sim(prs[0], stream=stream)
        sim.set_prims(dev[0])
        P = torch.empty((8,) + tuple(n + 6 for n in prs[0].n[::-1]), dtype=torch.float64, device="cuda")
        sim.get_prims(with_ghosts=True, out=P)
        torch.cuda.synchronize()
        sim.close()
        return State(case, prs, [], [P], [None], [P.new_empty((3,) + tuple(P.shape))])
    sims = [grmhd.Sim(p, stream=stream) for p in prs]
    K = [torch.from_numpy(p.K).cuda() if p.K is not None else None for p in prs]
    out = [torch.empty((8,) + tuple(p.n[::-1]), dtype=torch.float64, device="cuda") for p in prs]
    return State(case, prs, sims, dev, K, out, grmhd.Batch(sims) if case["kind"] == "batch" else None)


def run(state):
    case = state.case
    if case["kind"] == "fluxes":
        F = state.out[0]
        ctop = grmhd.fluxes_noalloc(state.problems[0], state.P[0], F, stream=torch.cuda.current_stream())
        return [F, ctop]
    for sim, P, K in zip(state.sims, state.P, state.K):
        sim.set_prims(P)
        if K is not None:
            sim.set_electrons(K)
    if state.batch is not None:
        state.batch.step(case["cycles"])
    else:
        state.sims[0].step(case["cycles"], sync=False)
    for sim, out in zip(state.sims, state.out):
        sim.get_prims(out=out)
    if state.K[0] is not None:
        return state.out + [state.sims[0].get_electrons()]
    return state.out


def _grids(case):
    if case["kind"] == "batch":
        return [(p.n, p.recon) for p in pb.batch_2d(case["grids"], case["nmin"], case["nmax"], seed=case["draw"])]
    return [((case["n1"], case.get("n2", case["n1"]), case.get("n3", 1)), _recon(case))]


def work(case):
    """Algorithmic bytes (of the state, 336 B per zone and cycle: each stage
    reads its primitives, the corrector P^n too, and writes its result) and
    floating-point operations."""
    flops = bytes_ = 0.0
    for n, recon in _grids(case):
        zones = n[0] * n[1] * n[2]
        dirs = 3 if n[2] > 1 else 2  # 2D: the X3 faces need no reconstruction
        rec = WENO_FLOPS if recon == pb.RECON_WENO5 else MC_FLOPS
        stage = zones * (dirs * rec + 3 * FACE_FLOPS)
        if case["kind"] == "fluxes":
            return {"bytes": 8.0 * 8 * 4 * zones, "flops": float(stage)}
        extra = (dirs * 2 * rec / 8 + 200) if case.get("electrons") else ZONE_FLOPS if case.get("drift") else 0
        flops += case["cycles"] * 2 * (stage + zones * (ZONE_FLOPS + extra))
        bytes_ += case["cycles"] * 336.0 * zones * (1.25 if case.get("electrons") else 1.0)
    return {"bytes": bytes_, "flops": flops}


# ---- the same in plain torch, 64 bits -----------------------------------------------------------

def _contract(g, x):
    return [sum(g[m][n] * x[n] for n in range(4)) for m in range(4)]


def _fluid(P, geo):
    gcov, gcon, gdet, alpha = geo
    v, B = [P[2], P[3], P[4]], [P[5], P[6], P[7]]
    low = [sum(gcov[i + 1][j + 1] * v[j] for j in range(3)) for i in range(3)]
    gam = (1.0 + sum(low[i] * v[i] for i in range(3))).sqrt()
    ucon = [gam / alpha] + [v[i] - gam * alpha * gcon[0][i + 1] for i in range(3)]
    ucov = [-alpha * gam + sum(gcov[0][i + 1] * v[i] for i in range(3))] + low
    bt = sum(B[i] * low[i] for i in range(3))
    bcon = [bt] + [(B[i] + bt * ucon[i + 1]) / ucon[0] for i in range(3)]
    bcov = _contract(gcov, bcon)
    return ucon, ucov, bcon, bcov, sum(bcon[m] * bcov[m] for m in range(4))


def _flux(P, s, geo, gamma, d):
    """sqrt(-g) times the conserved densities (d = 0) or the fluxes along d."""
    ucon, ucov, bcon, bcov, bsq = s
    pg = (gamma - 1.0) * P[1]
    w, pt = P[0] + P[1] + pg + bsq, pg + 0.5 * bsq
    T = [w * ucon[d] * ucov[n] - bcon[d] * bcov[n] + (pt if n == d else 0.0) for n in range(4)]
    rows = [P[0] * ucon[d], T[0] + P[0] * ucon[d], T[1], T[2], T[3]]
    rows += [bcon[i] * ucon[d] - bcon[d] * ucon[i] for i in (1, 2, 3)]
    return torch.stack([geo[2] * r for r in rows])


def _cmax(P, s, geo, gamma, d):
    ucon, bsq, gcon = s[0], s[4], geo[1]
    ef = P[0] + gamma * P[1]
    cs2, va2 = gamma * (gamma - 1.0) * P[1] / ef, bsq / (bsq + ef)
    c2 = cs2 + va2 - cs2 * va2
    Au, Bu = ucon[d], ucon[0]
    qa = Bu * Bu - (gcon[0][0] + Bu * Bu) * c2
    hb = Au * Bu - (gcon[0][d] + Au * Bu) * c2
    qc = Au * Au - (gcon[d][d] + Au * Au) * c2
    root = (hb * hb - qa * qc).clamp(min=0.0).sqrt()
    return torch.maximum(((hb + root) / qa).abs(), ((hb - root) / qa).abs())


def _face_values(P, ax, recon):
    """(low, high) face value of every zone along axis ax (rolls wrap around)."""
    a, b, c, d, e = (P.roll(k, ax) for k in (2, 1, 0, -1, -2))
    if recon == pb.RECON_MC:
        dm, dp = c - b, d - c
        dc = 0.5 * (dm + dp)
        m = torch.minimum(torch.minimum((2 * dm).abs(), dc.abs()), (2 * dp).abs())
        h = 0.5 * torch.where(dm * dp > 0.0, torch.sign(dc) * m, torch.zeros_like(m))
        return c - h, c + h

    def high(a, b, c, d, e):
        beta = [13.0 / 12.0 * t * t + 0.25 * s * s for t, s in
                ((a - 2 * b + c, a - 4 * b + 3 * c), (b - 2 * c + d, b - d), (c - 2 * d + e, 3 * c - 4 * d + e))]
        al = [w / (1e-26 + x) ** 2 for w, x in zip((0.1, 0.6, 0.3), beta)]
        q = ((2 * a - 7 * b + 11 * c) / 6, (-b + 5 * c + 2 * d) / 6, (2 * c + 5 * d - e) / 6)
        return c + sum(w * (x - c) for w, x in zip(al, q)) / sum(al)

    return high(e, d, c, b, a), high(a, b, c, d, e)


def _face_flux(P, d, geo, gamma, recon):
    """LLF flux at every zone's low face along d (1..3) and the signal speed there."""
    ax = {1: -1, 2: -2, 3: -3}[d]
    lo, hi = _face_values(P, ax, recon)
    L, R = hi.roll(1, ax), lo
    sL, sR = _fluid(L, geo), _fluid(R, geo)
    c = torch.maximum(_cmax(L, sL, geo, gamma, d), _cmax(R, sR, geo, gamma, d))
    F = _flux(L, sL, geo, gamma, d) + _flux(R, sR, geo, gamma, d)
    return 0.5 * (F - c * (_flux(R, sR, geo, gamma, 0) - _flux(L, sL, geo, gamma, 0))), c


def _emfs(F1, F2, F3):
    jm, im, km = (lambda x: x.roll(1, -2)), (lambda x: x.roll(1, -1)), (lambda x: x.roll(1, -3))
    return (0.25 * (F2[7] + km(F2[7]) - F3[6] - jm(F3[6])), 0.25 * (F3[5] + im(F3[5]) - F1[7] - km(F1[7])),
            0.25 * (F1[6] + jm(F1[6]) - F2[5] - im(F2[5])))


def _induction(e):
    """The flux-CT induction fluxes [direction][component] of the edge EMFs."""
    jp, ip, kp = (lambda x: x.roll(-1, -2)), (lambda x: x.roll(-1, -1)), (lambda x: x.roll(-1, -3))
    z = torch.zeros_like(e[0])
    return ((z, 0.5 * (e[2] + jp(e[2])), -0.5 * (e[1] + kp(e[1]))),
            (-0.5 * (e[2] + ip(e[2])), z, 0.5 * (e[0] + kp(e[0]))),
            (0.5 * (e[1] + ip(e[1])), -0.5 * (e[0] + jp(e[0])), z))


def _flat(dev):
    one = torch.ones((), dtype=torch.float64, device=dev)
    eta = [[one * ((-1.0 if m == 0 else 1.0) if m == n else 0.0) for n in range(4)] for m in range(4)]
    return eta, eta, one, one


def _recover(U, P, gamma):
    """Primitives of the flat-space conserved vector U: Newton in W' = W - D from the guess P."""
    D, E, Q, B = U[0], U[1], U[2:5], U[5:8]
    gf = (gamma - 1.0) / gamma
    Q2, QB, B2 = (Q * Q).sum(0), (Q * B).sum(0), (B * B).sum(0)
    Wp = ((P[0] + gamma * P[1]) * (1.0 + (P[2:5] ** 2).sum(0)) - D).clamp(min=0.0)
    for it in range(14):
        W = Wp + D
        v2 = (Q2 * W * W + QB * QB * (B2 + 2 * W)) / (W * (B2 + W)) ** 2
        om = 1.0 - v2
        wmr = Wp * om - D * v2 * om.sqrt() / (1.0 + om.sqrt())
        if it == 13:
            break
        f = E + Wp - gf * wmr + 0.5 * (1.0 + v2) * B2 - 0.5 * (QB / W) ** 2
        dv = -2.0 * (Q2 * W ** 3 + QB * QB * (3 * W * W + 3 * W * B2 + B2 * B2)) / (W * (B2 + W)) ** 3
        df = 1.0 - gf * (om + dv * (0.5 * D / om.sqrt() - W)) + 0.5 * B2 * dv + QB * QB / W ** 3
        new = Wp - f / df
        Wp = torch.where(new < 0.0, 0.5 * Wp, new)
    lorentz = 1.0 / om.sqrt()
    return torch.cat([(D / lorentz)[None], (wmr / gamma)[None], lorentz / (W + B2) * (Q + QB / W * B), B])


def _flat_steps(pr, cycles, dev):
    P, geo, gamma = torch.from_numpy(pr.P).to(dev), _flat(dev), pr.gamma
    dx = [(b - a) / n for a, b, n in zip(pr.xmin, pr.xmax, pr.n)]
    dt_prev = 0.0
    for _ in range(cycles):
        U, half = _flux(P, _fluid(P, geo), geo, gamma, 0), None
        for stage in (0, 1):
            got = [_face_flux(P if stage == 0 else half, d, geo, gamma, pr.recon) for d in (1, 2, 3)]
            if stage == 0:
                dt = 1.0 / sum(float(c.max()) / (pr.cfl * h) for (_, c), h, n in zip(got, dx, pr.n) if n > 1)
                dt = min(dt, 1.3 * dt_prev) if dt_prev > 0.0 else dt
                dt_prev = dt
            F = [f for f, _ in got]
            for f, b in zip(F, _induction(_emfs(*F))):
                f[5:8] = torch.stack(b)
            div = sum((f.roll(-1, ax) - f) / h for f, ax, h in zip(F, (-1, -2, -3), dx))
            new = _recover(U - (0.5 if stage == 0 else 1.0) * dt * div, P, gamma)
            half = new
        P = half
    return P


def _kerr(pr, off1, off2, dev):
    """Metric at every (j, i), ghosts among them, offset by off1, off2 zones from the low corner."""
    n1, n2, _ = pr.n
    X1 = pr.xmin[0] + (torch.arange(-3, n1 + 3, dtype=torch.float64, device=dev) + off1) * ((pr.xmax[0] - pr.xmin[0]) / n1)
    X2 = pr.xmin[1] + (torch.arange(-3, n2 + 3, dtype=torch.float64, device=dev) + off2) * ((pr.xmax[1] - pr.xmin[1]) / n2)
    r, X2 = X1.exp()[None, :], X2[:, None]
    th = math.pi * X2 + 0.5 * (1.0 - pr.hslope) * torch.sin(2.0 * math.pi * X2)
    sth = torch.sin(th)
    sth = torch.where(sth.abs() < 1e-20, torch.where(sth >= 0, 1e-20, -1e-20).to(sth), sth)
    a, s2 = pr.a, sth * sth + 0 * r
    sig = r * r + a * a * torch.cos(th) ** 2
    tr, J2 = 2.0 * r / sig, math.pi * (1.0 + (1.0 - pr.hslope) * torch.cos(2.0 * math.pi * X2))
    g = torch.zeros(s2.shape + (4, 4), dtype=torch.float64, device=dev)
    g[..., 0, 0] = tr - 1.0
    g[..., 0, 1] = g[..., 1, 0] = tr * r
    g[..., 0, 3] = g[..., 3, 0] = -a * tr * s2
    g[..., 1, 1] = (1.0 + tr) * r * r
    g[..., 1, 3] = g[..., 3, 1] = -a * s2 * (1.0 + tr) * r
    g[..., 2, 2] = sig * J2 * J2
    g[..., 3, 3] = s2 * (sig + a * a * s2 * (1.0 + tr))
    # the inverse in closed form: the (t, 1) block at fixed (2, 3) of Kerr-Schild
    gi = torch.zeros_like(g)
    gi[..., 0, 0] = -(1.0 + tr)
    gi[..., 0, 1] = gi[..., 1, 0] = tr / r
    gi[..., 1, 1] = (r * r - 2.0 * r + a * a) / (sig * r * r)
    gi[..., 1, 3] = gi[..., 3, 1] = a / (sig * r)
    gi[..., 2, 2] = 1.0 / (sig * J2 * J2)
    gi[..., 3, 3] = 1.0 / (sig * s2)
    gdet = (sig * sth).abs() * r * J2.abs()
    pick = lambda m: [[m[..., p, q] for q in range(4)] for p in range(4)]  # noqa: E731
    return pick(g), pick(gi), gdet, (1.0 + tr).rsqrt()


def _exact_fluxes(pr, P, dev):
    n = pr.n
    out, cs = torch.zeros((3,) + tuple(P.shape), dtype=torch.float64, device=dev), []
    for d in (1, 2, 3):
        geo = _kerr(pr, 0.0 if d == 1 else 0.5, 0.0 if d == 2 else 0.5, dev)
        F, c = _face_flux(P, d, geo, pr.gamma, pr.recon)
        # axes (X3, X2, X1): faces 0 .. n along d, one extra layer across
        box = tuple(slice(3, n[q] + 4) if q == d - 1 else slice(2, n[q] + 4) for q in (2, 1, 0))
        inner = tuple(slice(3, n[q] + 4) if q == d - 1 else slice(3, n[q] + 3) for q in (2, 1, 0))
        out[(d - 1, slice(None)) + box] = F[(slice(None),) + box]
        cs.append(float(c[inner].max()))
    out[1][:, :, 3] = 0.0   # the polar faces
    out[1][:, :, n[1] + 3] = 0.0
    out[0][0, ..., 3].clamp_(max=0.0)  # no mass in through the X1 sides
    out[0][0, ..., n[0] + 3].clamp_(min=0.0)
    # flux-CT replaces the induction fluxes of the faces next to a zone
    for d, b in enumerate(_induction(_emfs(*out))):
        box = tuple(slice(3, n[q] + 4) if q == d else slice(3, n[q] + 3) for q in (2, 1, 0))
        for v in range(3):
            out[(d, 5 + v) + box] = b[v][box]
    return [out, np.array(cs)]


def exact(case, seed):
    """The flat problems and the flux stage; the curved steps (numerical
    connection, bounds, inversion failures) have none."""
    if case["kind"] in ("mode", "vortex", "batch"):
        return [_flat_steps(p, case["cycles"], "cuda") for p in _problems(case, seed)]
    if case["kind"] == "fluxes":
        s = prepare(case, seed)
        return _exact_fluxes(s.problems[0], s.P[0], "cuda")
    return None
