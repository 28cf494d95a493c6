"""The workloads whose speed is measured, with their inputs, one pass of each and its result in 64 bits.

A case is one call, or one short chain of calls, that a tracking program makes on data it holds on the GPU: the fit of
given hit lists, the refit and the smoothing of found tracks, the finding of tracks from seeds (hit binning included,
as every new set of events needs it), seed cleaning and duplicate removal around it, the learned cascade and a training
step of its network.  Events are synthetic: helices from the beam line through one of three detectors, smeared hits,
noise; drawn on the GPU from the seed alone.
"""
import math

import torch

from paper_1811_04141_gb300 import Context, HitBins
from paper_1811_04141_gb300.api import mkf_mlp_to_bf16, mkf_mlp_train_step
from paper_1811_04141_gb300.learned import cascade

DEVICE = "cuda"
K_FIELD = 0.0029979245800  # GeV / (T cm)
BZ = 3.8
PION = 0.13957
X0, ELOSS = 0.02, 0.04  # material of a layer: radiation lengths, GeV lost per radiation length
ALPHA = 1e-5  # fall-off of the parameterised field, 1/cm^2
INFLATE = 100.0
GATE_TAU = 5.0  # flags about one seed in seven
UM = 1e-4
LIST_ROWS = dict(barrel=10, endcaps=12, dense=24)  # rows of a hit list


# ---------------------------------------------------------------------------
# Detectors: the tables of the repository's configurations
# ---------------------------------------------------------------------------

def _cyl(r, half, su, sv, nphi, nz):
    return dict(kind=0, r_or_z=r, lo=-half, hi=half, sigma_u=su, sigma_v=sv, n_phi=nphi, n_zr=nz)


def _disk(z, lo, hi, su, sv, nphi, nr):
    return dict(kind=1, r_or_z=z, lo=lo, hi=hi, sigma_u=su, sigma_v=sv, n_phi=nphi, n_zr=nr)


def detector(name, material=False):
    """barrel: 10 cylinders (|eta| < 1); endcaps: those and 2 x 5 disks; dense: 17 cylinders and 2 x 14 disks."""
    if name in ("barrel", "endcaps"):
        n_phi, n_zr = (64, 8) if name == "barrel" else (256, 32)
        layers = [_cyl(4.0 + 96.0 * i / 9.0, 125.0, 20 * UM, 100 * UM, n_phi, n_zr) for i in range(10)]
        if name == "endcaps":
            layers += [_disk(s * z, 4.0, 100.0, 20 * UM, 100 * UM, n_phi, n_zr)
                       for s in (1.0, -1.0) for z in (120.0, 157.5, 195.0, 232.5, 270.0)]
    else:
        layers = [_cyl(r, 27.0, 15 * UM, 15 * UM, 256, 32) for r in (3.0, 7.0, 11.0, 16.0)]
        layers += [_cyl(25.0 + 85.0 * i / 12.0, 110.0, 30 * UM, 1000 * UM, 256, 32) for i in range(13)]
        for s in (1.0, -1.0):
            layers += [_disk(s * z, 4.5, 16.0, 15 * UM, 15 * UM, 256, 32) for z in (32.0, 40.0, 50.0)]
            layers += [_disk(s * (75.0 + 205.0 * i / 10.0), 20.0, 110.0, 30 * UM, 1000 * UM, 256, 32)
                       for i in range(11)]
    if material:
        layers = [dict(d, x0=X0, eloss=ELOSS) for d in layers]
    return layers


def _f32(x):
    return float(torch.tensor(x, dtype=torch.float32))


class Table:
    """The layers as 64-bit columns, every value as the library takes it (32 bits)."""

    def __init__(self, layers, dev):
        col = lambda k: torch.tensor([_f32(float(d.get(k, 0.0))) for d in layers], dtype=torch.float64, device=dev)
        self.cyl = torch.tensor([d["kind"] == 0 for d in layers], device=dev)
        self.rz, self.lo, self.hi = col("r_or_z"), col("lo"), col("hi")
        self.su, self.sv, self.x0, self.el = col("sigma_u"), col("sigma_v"), col("x0"), col("eloss")
        self.n = len(layers)


# ---------------------------------------------------------------------------
# Motion in 64 bits (inputs and exact())
# ---------------------------------------------------------------------------

KB = _f32(K_FIELD) * BZ


def _atanc(x):
    return torch.where(x.abs() < 1e-4, 1.0 - x * x / 3.0, torch.atan(x) / torch.where(x == 0, 1.0, x))


def _sinc(a):
    return torch.where(a.abs() < 1e-4, 1.0 - a * a / 6.0, torch.sin(a) / torch.where(a == 0, 1.0, a))


def path_to(cyl, rz, x, y, z, phi, cot, h):
    """Transverse path to the surface ahead (cylinder or disk), NaN where it is not reached within half a turn."""
    c, s = torch.cos(phi), torch.sin(phi)
    b = x * c + y * s
    nn = y * c - x * s
    D = rz * rz - x * x - y * y
    a2 = 2.0 + 2.0 * h * nn - 0.5 * h * h * D
    disc = b * b + 0.5 * a2 * D
    q = -(b + torch.copysign(torch.sqrt(disc.clamp(min=0.0)), b))
    t1, t2 = -0.5 * D / q, q / a2
    inf = torch.full_like(x, math.inf)
    s1 = torch.where(t1 > 0, 2.0 * t1 * _atanc(h * t1), inf)
    s2 = torch.where(t2 > 0, 2.0 * t2 * _atanc(h * t2), inf)
    sc = torch.minimum(s1, s2)
    sc = torch.where((disc >= 0) & torch.isfinite(sc), sc, math.nan)
    sd = (rz - z) / cot
    sd = torch.where((sd > 0) & (h.abs() * sd < math.pi), sd, math.nan)
    return torch.where(cyl, sc, sd)


def move(x, y, z, phi, cot, h, s):
    a = 0.5 * h * s
    L = s * _sinc(a)
    return x + L * torch.cos(phi + a), y + L * torch.sin(phi + a), z + s * cot, phi + 2.0 * a


def _theta0(p, x):
    beta2 = p * p / (p * p + PION * PION)
    return 0.0136 / (torch.sqrt(beta2) * p) * torch.sqrt(x) * (1.0 + 0.038 * torch.log(x / beta2))


def _rk(r, T, lam, d):
    """A Runge-Kutta step of path d in the parameterised field; r and T are lists of three tensors."""
    def turn(r, T):
        b = (KB * ALPHA * r[0] * r[2], KB * ALPHA * r[1] * r[2],
             KB * (1.0 - ALPHA * (r[2] * r[2] - 0.5 * (r[0] * r[0] + r[1] * r[1]))))
        return [lam * (T[1] * b[2] - T[2] * b[1]), lam * (T[2] * b[0] - T[0] * b[2]), lam * (T[0] * b[1] - T[1] * b[0])]
    add = lambda u, f, v: [a + f * b for a, b in zip(u, v)]
    k1 = turn(r, T)
    T2 = add(T, 0.5 * d, k1)
    k2 = turn(add(r, 0.5 * d, T), T2)
    T3 = add(T, 0.5 * d, k2)
    k3 = turn(add(r, 0.5 * d, T2), T3)
    T4 = add(T, d, k3)
    k4 = turn(add(r, d, T3), T4)
    return ([a + d / 6.0 * (p + 2 * q + 2 * u + v) for a, p, q, u, v in zip(r, T, T2, T3, T4)],
            [a + d / 6.0 * (p + 2 * q + 2 * u + v) for a, p, q, u, v in zip(T, k1, k2, k3, k4)])


# ---------------------------------------------------------------------------
# Events
# ---------------------------------------------------------------------------

def _log_spread(lo, hi, n):
    return [int(math.exp(math.log(lo) + (i + 0.5) / n * math.log(hi / lo))) for i in range(n)]


def counts(case):
    """Tracks and noise hits of each event of a case, in no particular order (noise None: 5 per signal hit)."""
    E = case["events"]
    if case.get("uneven"):
        return _log_spread(100, 20000, E), _log_spread(1000, 300000, E)
    noise = {"barrel": 0, "endcaps": None, "dense": 200000}[case["detector"]]
    return [case["tracks"]] * E, [noise if noise is None else case.get("noise", noise)] * E


def make_events(case, seed, dev):
    """Hits, seeds and hit lists of a case's events (see the module's text)."""
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))
    f8 = dict(dtype=torch.float64, device=dev)
    rand = lambda *shape: torch.rand(*shape, generator=g, **f8)
    randn = lambda *shape: torch.randn(*shape, generator=g, **f8)
    layers = detector(case["detector"], bool(case.get("material")))
    G = Table(layers, dev)
    tracks, noise = counts(case)
    if case.get("uneven"):  # which event is the crowded one, and which the noisy one, is the seed's
        cpu = torch.Generator().manual_seed(int(seed))
        tracks = [tracks[i] for i in torch.randperm(len(tracks), generator=cpu)]
        noise = [noise[i] for i in torch.randperm(len(noise), generator=cpu)]
    E = len(tracks)
    ev = torch.repeat_interleave(torch.arange(E, device=dev), torch.tensor(tracks, device=dev))
    P = ev.shape[0]
    dense, eta_max = case["detector"] == "dense", 1.0 if case["detector"] == "barrel" else 2.4
    u = rand(P)
    # pT flat in 0.5-10 GeV, or falling as pT^-3 from 0.5 to 100 GeV
    pt = (4.0 - u * (4.0 - 1e-4)) ** -0.5 if dense else 0.5 + 9.5 * u
    q = torch.where(rand(P) < 0.5, -1.0, 1.0)
    phi = math.pi * (2.0 * rand(P) - 1.0)
    cot = torch.sinh(eta_max * (2.0 * rand(P) - 1.0))
    z0 = 5.0 * (2.0 * rand(P) - 1.0)
    h = -q * KB / pt
    # crossings on the outward half turn from the beam line, in path order
    x2 = 0.5 * G.rz[None, :] * h.abs()[:, None]
    s_c = torch.where(x2 <= 1.0, 2.0 * torch.asin(x2.clamp(max=1.0)) / h.abs()[:, None], math.inf)
    s_d = (G.rz[None, :] - z0[:, None]) / cot[:, None]
    s_d = torch.where((s_d > 0) & (s_d * h.abs()[:, None] < math.pi), s_d, math.inf)
    S = torch.where(G.cyl[None, :], s_c, s_d)
    a = 0.5 * h[:, None] * torch.where(torch.isfinite(S), S, 0.0)
    zz = z0[:, None] + S * cot[:, None]
    rr = (2.0 * torch.sin(a) / h[:, None]).abs()
    at = torch.where(G.cyl[None, :], zz, rr)
    S = torch.where((at >= G.lo) & (at <= G.hi), S, math.inf)
    del s_c, s_d, a, zz, rr, at, x2
    S, order = torch.sort(S, dim=1)
    K = int(torch.isfinite(S).sum(1).max())
    S, order = S[:, :K], order[:, :K]
    hx, hy, hz, ok = (torch.zeros(P, K, dtype=t, device=dev) for t in (torch.float64,) * 3 + (torch.bool,))
    plain = not case.get("material") and not case.get("field")
    x, y, z, alive = torch.zeros_like(pt), torch.zeros_like(pt), z0.clone(), torch.ones_like(pt, dtype=torch.bool)
    w, theta = q / pt, torch.atan2(torch.ones_like(cot), cot)
    for k in range(K):
        l = order[:, k]
        c, rz = G.cyl[l], G.rz[l]
        alive = alive & torch.isfinite(S[:, k])
        if plain:
            px, py, pz, _ = move(torch.zeros_like(x), torch.zeros_like(x), z0, phi, cot, h, torch.where(alive, S[:, k], 0.0))
            pz = torch.where(c, pz, rz)
        elif case.get("field"):
            st = torch.sin(theta)
            r, T, lam = [x, y, z], [st * torch.cos(phi), st * torch.sin(phi), torch.cos(theta)], w * st
            s = path_to(c, rz, x, y, z, phi, 1.0 / torch.tan(theta), -w * KB * (1.0 - ALPHA * (z * z - 0.5 * (x * x + y * y))))
            alive = alive & torch.isfinite(s)
            d = torch.where(alive, s, 0.0) / st / 8.0
            for _ in range(8):
                r, T = _rk(r, T, lam, d)
            for _ in range(3):
                rho = torch.sqrt(r[0] * r[0] + r[1] * r[1])
                dn = torch.where(c, (rz - rho) * rho / (r[0] * T[0] + r[1] * T[1]), (rz - r[2]) / T[2])
                r, T = _rk(r, T, lam, torch.where(alive, dn, 0.0).clamp(-1.0, 1.0))
            px, py, pz = r
            alive = alive & (torch.where(c, torch.sqrt(px * px + py * py), pz) - rz).abs().lt(1e-8)
            x, y, z = px, py, pz
            phi, theta = torch.atan2(T[1], T[0]), torch.atan2(torch.sqrt(T[0] * T[0] + T[1] * T[1]), T[2])
            w = lam / torch.sin(theta)
        else:
            s = path_to(c, rz, x, y, z, phi, 1.0 / torch.tan(theta), -w * KB)
            alive = alive & torch.isfinite(s)
            x, y, z, phi = move(x, y, z, phi, 1.0 / torch.tan(theta), -w * KB, torch.where(alive, s, 0.0))
            z = torch.where(c | ~alive, z, rz)
            px, py, pz = x, y, z
            # scattering and energy loss in the layer
            p = 1.0 / (w.abs() * torch.sin(theta))
            cosa = torch.where(c, torch.sin(theta) * torch.cos(phi - torch.atan2(y, x)), torch.cos(theta)).abs().clamp(min=1e-6)
            t0, n2 = _theta0(p, X0 / cosa), randn(2, P)
            phi = phi + t0 * n2[0] / torch.sin(theta)
            theta = theta + t0 * n2[1]
            e = torch.sqrt(p * p + PION * PION) - ELOSS * (X0 / cosa) * (1.0 + PION * PION / (p * p))
            alive = alive & (e > PION + 0.02)
            p = torch.where(alive, torch.sqrt((e * e - PION * PION).clamp(min=1e-6)), p)
            w = torch.sign(w) / (p * torch.sin(theta))
        rho = torch.sqrt(px * px + py * py)
        inside = torch.where(c, (pz >= G.lo[l]) & (pz <= G.hi[l]), (rho >= G.lo[l]) & (rho <= G.hi[l]))
        n2 = randn(2, P)
        az = torch.atan2(py, px) + n2[0] * G.su[l] / rho.clamp(min=1e-3)
        rho = torch.where(c, rz, rho + n2[1] * G.sv[l])
        hx[:, k], hy[:, k] = rho * torch.cos(az), rho * torch.sin(az)
        hz[:, k] = torch.where(c, pz + n2[1] * G.sv[l], rz)
        ok[:, k] = alive & inside
    if case["detector"] != "barrel":
        ok &= rand(P, K) >= 0.02  # inefficiency
    cnt = ok.sum(1)
    first = torch.cumsum(cnt, 0) - cnt
    sig = torch.nonzero(ok.reshape(-1)).squeeze(1)
    sx, sy, sz, sl = hx.reshape(-1)[sig], hy.reshape(-1)[sig], hz.reshape(-1)[sig], order.reshape(-1)[sig]
    se = ev[sig // K]
    del hx, hy, hz, S
    # noise, uniform over each layer; and hits measured twice where sensors overlap, each with a second seed
    per = torch.zeros(E, G.n, dtype=torch.int64, device=dev)
    if noise[0] is None:
        per = 5 * torch.bincount(se * G.n + sl, minlength=E * G.n).view(E, G.n)
    else:
        nt = torch.tensor(noise, device=dev)
        per[:] = (nt // G.n)[:, None]
        per[:, 0] += nt - nt // G.n * G.n
    nl = torch.arange(G.n, device=dev).repeat(E).repeat_interleave(per.view(-1))
    ne = torch.arange(E, device=dev).repeat_interleave(per.sum(1))
    n2 = rand(2, nl.shape[0])
    c, az = G.cyl[nl], math.pi * (2.0 * n2[0] - 1.0)
    rho = torch.where(c, G.rz[nl], torch.sqrt(G.lo[nl] ** 2 + n2[1] * (G.hi[nl] ** 2 - G.lo[nl] ** 2)))
    nx, ny = rho * torch.cos(az), rho * torch.sin(az)
    nz = torch.where(c, G.lo[nl] + n2[1] * (G.hi[nl] - G.lo[nl]), G.rz[nl])
    has = torch.nonzero(cnt >= 3).squeeze(1)
    owner = torch.zeros(0, dtype=torch.int64, device=dev)
    if case.get("overlap"):
        owner = has[torch.argsort(rand(has.shape[0]))[:int(case["overlap"] * P)]].sort()[0]
        slot = torch.randint(3, owner.shape, generator=g, device=dev)
        twin_of = first[owner] + slot
        n2, tl = randn(2, twin_of.shape[0]), sl[twin_of]
        c = G.cyl[tl]
        rho = torch.sqrt(sx[twin_of] ** 2 + sy[twin_of] ** 2)
        az = torch.atan2(sy[twin_of], sx[twin_of]) + n2[0] * G.su[tl] / rho
        rho = torch.where(c, rho, rho + n2[1] * G.sv[tl])
        nx, ny = torch.cat([nx, rho * torch.cos(az)]), torch.cat([ny, rho * torch.sin(az)])
        nz = torch.cat([nz, torch.where(c, sz[twin_of] + n2[1] * G.sv[tl], G.rz[tl])])
        nl, ne = torch.cat([nl, tl]), torch.cat([ne, se[twin_of]])
    # an event's hits: its particles' in path order, then the others
    ns, nn = torch.bincount(se, minlength=E), torch.bincount(ne, minlength=E)
    offs = torch.zeros(E + 1, dtype=torch.int64, device=dev)
    offs[1:] = torch.cumsum(ns + nn, 0)
    by_ev = torch.argsort(ne, stable=True)
    sig_at = torch.arange(sig.shape[0], device=dev) + (offs[:-1] - (torch.cumsum(ns, 0) - ns))[se]
    oth_at = torch.empty_like(by_ev)
    oth_at[by_ev] = torch.arange(ne.shape[0], device=dev) + (offs[1:] - torch.cumsum(nn, 0))[ne[by_ev]]
    at = torch.cat([sig_at, oth_at])
    xyz = torch.empty(3, at.shape[0], dtype=torch.float32, device=dev)
    for i, v in enumerate((torch.cat([sx, nx]), torch.cat([sy, ny]), torch.cat([sz, nz]))):
        xyz[i, at] = v.float()
    layer = torch.empty(at.shape[0], dtype=torch.int32, device=dev)
    layer[at] = torch.cat([sl, nl]).int()
    # hit lists and seeds of the particles with three hits or more
    f, n_h, pe = first[has], cnt[has], ev[has]
    j = torch.arange(LIST_ROWS[case["detector"]], device=dev)[:, None]
    hits = torch.where(j < n_h[None, :], sig_at[(f[None, :] + j).clamp(max=sig.shape[0] - 1)], -1).int().contiguous()
    seeds = hits[:3].contiguous()
    if owner.numel():
        n2 = owner.shape[0]
        extra = torch.stack([sig_at[first[owner] + i] for i in range(3)])
        extra[slot, torch.arange(n2, device=dev)] = oth_at[ne.shape[0] - n2:]
        seeds, pe = torch.cat([seeds, extra.int()], 1), torch.cat([pe, ev[owner]])
        o = torch.argsort(pe, stable=True)
        seeds, pe = seeds[:, o].contiguous(), pe[o]
    return dict(layers=layers, table=G, xyz=xyz, layer=layer, offsets=offs.int(), hits=hits, seeds=seeds, seed_event=pe.int())


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # one event of a trigger or an interactive fit: 1000 tracks, latency counts
        dict(name="fit_event", do="fit", detector="barrel", events=1, tracks=1000),
        # a whole sample refitted at once
        dict(name="fit_tracks", do="fit", detector="barrel", events=5, tracks=200000),
        # the same through the parameterised field of a real solenoid
        dict(name="fit_field", do="fit", detector="barrel", events=5, tracks=20000, field=True),
        # found tracks refitted out and back through material, ragged lists over cylinders and disks
        dict(name="refit_material", do="refit", detector="dense", events=24, tracks=6000, noise=0, material=True),
        # the state at every hit, for alignment and resolution studies
        dict(name="smooth", do="smooth", detector="endcaps", events=50, tracks=2000),
        # one event found, ten candidates a seed: latency counts
        dict(name="find_event", do="find", detector="endcaps", events=1, tracks=2000, n_best=10),
        # the chain around finding: seeds fitted and cleaned, hits binned, tracks found, duplicates removed
        dict(name="find_chain", do="chain", detector="endcaps", events=20, tracks=2000, n_best=10, overlap=0.1),
        # best-hit finding in crowded events
        dict(name="find_best", do="find", detector="dense", events=20, tracks=6000, n_best=1),
        # ten candidates a seed through material in crowded events
        dict(name="find_material", do="find", detector="dense", events=8, tracks=6000, n_best=10, material=True),
        # the learned cascade: best hit with the network's gate, then ten candidates for the seeds it doubts
        dict(name="find_cascade", do="cascade", detector="dense", events=16, tracks=6000, n_best=10, material=True),
        # many events of uneven occupancy in one call, the widest range of event sizes
        dict(name="find_uneven", do="find", detector="dense", events=128, uneven=True, n_best=10),
        # a step of the network's training
        dict(name="train_step", do="train", batch=4096),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["fit", "fit", "field", "refit", "smooth", "find", "find", "chain", "best", "material", "cascade",
                     "uneven", "train"])
    if do == "fit":
        return dict(do="fit", detector="barrel", events=1, tracks=_log_int(rng, 700, 900000))
    if do == "field":
        return dict(do="fit", detector="barrel", events=1, tracks=_log_int(rng, 700, 90000), field=True)
    if do == "refit":
        return dict(do="refit", detector="dense", events=rng.randint(1, 20), tracks=_log_int(rng, 500, 7000), noise=0,
                    material=True)
    if do == "smooth":
        return dict(do="smooth", detector="endcaps", events=rng.randint(1, 40), tracks=_log_int(rng, 500, 2400))
    if do == "find":
        return dict(do="find", detector="endcaps", events=rng.randint(1, 20), tracks=_log_int(rng, 300, 4000),
                    n_best=rng.choice([1, 4, 10, 16]))
    if do == "chain":
        return dict(do="chain", detector="endcaps", events=rng.randint(1, 20), tracks=_log_int(rng, 300, 3000), n_best=10,
                    overlap=round(rng.uniform(0.02, 0.15), 3))
    if do == "best":
        return dict(do="find", detector="dense", events=rng.randint(1, 20), tracks=_log_int(rng, 500, 8000), n_best=1,
                    noise=_log_int(rng, 1000, 300000))
    if do == "material":
        return dict(do="find", detector="dense", events=rng.randint(1, 8), tracks=_log_int(rng, 500, 6000), n_best=10,
                    noise=_log_int(rng, 1000, 200000), material=True)
    if do == "cascade":
        return dict(do="cascade", detector="dense", events=rng.randint(1, 16), tracks=_log_int(rng, 500, 6000), n_best=10,
                    noise=_log_int(rng, 1000, 200000), material=True)
    if do == "uneven":
        return dict(do="find", detector="dense", events=rng.randint(8, 120), uneven=True, n_best=10)
    return dict(do="train", batch=_log_int(rng, 500, 60000))


def gate_weights():
    """Weights of a gate that doubts hits far from the prediction: the logit falls from 6 with chi2 / cut (feature 2),
    steeper near the cut, and a little with |u| / sigma; the other units look at every feature weakly."""
    g = torch.Generator().manual_seed(11)
    W1, b1, w2 = 0.2 * torch.randn(64, 12, generator=g), 0.1 * torch.randn(64, generator=g), 0.02 * torch.randn(64, generator=g)
    for j, (k, slope, at, out) in enumerate(((2, 1.0, 0.1, -4.0), (2, 1.0, 0.3, -8.0), (2, 1.0, 0.5, -12.0), (0, 1.0, 2.0, -0.6),
                                             (0, -1.0, 2.0, -0.6), (1, 1.0, 2.0, -0.6), (1, -1.0, 2.0, -0.6))):
        W1[j] = 0.0
        W1[j, k], b1[j], w2[j] = slope, -at, out
    return torch.cat([W1.reshape(-1), b1, w2, torch.tensor([6.0])])


def train_inputs(case, seed, dev):
    """Pairs as the finder dumps them: residuals in sigmas, chi2 as a share of the cut, counts, layer, momentum, eta."""
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))
    n = case["batch"]
    f = torch.randn(n, 12, generator=g, device=dev)
    u = torch.rand(n, 6, generator=g, device=dev)
    label = (torch.rand(n, generator=g, device=dev) < 0.6).float()
    wide = torch.where(label > 0, 1.0, 2.5)
    f[:, 0] *= wide
    f[:, 1] *= wide
    f[:, 2] = ((f[:, 0] ** 2 + f[:, 1] ** 2) / 30.0).clamp(max=1.0)
    f[:, 3] = 1.0 + 0.3 * f[:, 3]
    f[:, 4] = 0.3 + torch.floor(u[:, 0] * 14.0) * 0.1
    f[:, 5] = torch.floor(u[:, 1] * 4.0) * 0.2
    f[:, 6] = torch.floor(u[:, 2] * 45.0) / 45.0
    f[:, 7] = (u[:, 3] < 0.5).float()
    f[:, 8] = (2.0 * u[:, 4] - 1.0) * 2.0
    f[:, 9] = (2.0 * u[:, 5] - 1.0) * 0.8
    f[:, 10] = -2.0 + 0.4 * f[:, 10]
    f[:, 11] = -1.3 + 0.5 * f[:, 11]
    w = torch.randn(897, generator=g, device=dev) * 0.3
    m = torch.randn(897, generator=g, device=dev) * 1e-3
    v = (torch.randn(897, generator=g, device=dev) * 3e-3) ** 2 + 1e-7
    return f.contiguous(), label, w, m, v


def prepare(case, seed):
    dev = torch.device(DEVICE, torch.cuda.current_device())
    ctx = Context(dev.index)
    if case["do"] == "train":
        f, label, w, m, v = train_inputs(case, seed, dev)
        return dict(case=case, ctx=ctx, feat=f, label=label, w=w, m=m, v=v, w_bf16=mkf_mlp_to_bf16(ctx, w), t=100,
                    loss=torch.zeros(1, device=dev))
    s = make_events(case, seed, dev)
    ctx.geometry_load(s["layers"], BZ, field_alpha=ALPHA if case.get("field") else None)
    s.update(case=case, ctx=ctx, bins=HitBins(), n_hits=int(s["xyz"].shape[1]))
    if case["do"] == "cascade":
        s["gate"] = mkf_mlp_to_bf16(ctx, gate_weights().to(dev))
    return s


def run(state):
    case, ctx = state["case"], state["ctx"]
    do = case["do"]
    if do == "train":
        state["t"] += 1
        mkf_mlp_train_step(ctx, state["feat"], state["label"], state["w"], state["m"], state["v"], state["t"], state["w_bf16"],
                           lr=2e-3, loss=state["loss"])
        return {k: state[k] for k in ("w", "m", "v", "w_bf16", "loss")}
    xyz, layer = state["xyz"], state["layer"]
    if do == "fit":
        return ctx.fit(xyz, layer, state["hits"])
    if do == "refit":
        out = ctx.fit(xyz, layer, state["hits"])
        return {"out": out, "back": ctx.fit_backward(xyz, layer, state["hits"], out["par"], out["cov"], INFLATE)}
    if do == "smooth":
        return ctx.fit_smooth(xyz, layer, state["hits"], inflate=INFLATE)
    if do == "find":
        bins = ctx.hits_bin(xyz, layer, state["offsets"], state["bins"])
        return ctx.find(bins, state["seeds"], state["seed_event"], n_best=case["n_best"])
    if do == "cascade":
        bins = ctx.hits_bin(xyz, layer, state["offsets"], state["bins"])
        return cascade(ctx, bins, state["seeds"], state["seed_event"], state["gate"], GATE_TAU, n_best=case["n_best"])[0]
    seed = ctx.fit(xyz, layer, state["seeds"])
    clean = ctx.seeds_clean(state["seeds"], state["n_hits"], seed["par"])
    bins = ctx.hits_bin(xyz, layer, state["offsets"], state["bins"])
    out = ctx.find(bins, state["seeds"], state["seed_event"], n_best=case["n_best"])
    keep = ctx.tracks_dedup(out["hits"], state["n_hits"], out["n_hits"], out["chi2"])
    return {"seed": seed, "clean": clean, "out": out, "keep": keep}


def work(case):
    """Hits of a track and candidate-layers of a seed are the detectors' means."""
    if case["do"] == "train":
        n = case["batch"]
        return {"bytes": n * 13 * 4 + 897 * (6 * 4 + 2) + 4, "flops": n * 6 * (12 * 64 + 64)}
    tracks, noise = counts(case)
    n = sum(tracks)
    det, mat = case["detector"], bool(case.get("material"))
    per = {"barrel": 10.0, "endcaps": 9.0, "dense": 16.0}[det]
    lists = {"barrel": 10, "endcaps": 12, "dense": 21}[det]
    state = 4 * (6 + 21 + 3)
    if case["do"] in ("fit", "refit", "smooth"):
        read = n * (per * 16 + lists * 4)
        if case["do"] == "fit":
            return {"bytes": read + n * state, "flops": n * per * 850}
        if case["do"] == "refit":
            return {"bytes": read + 2 * n * state, "flops": 2 * n * per * 850}
        return {"bytes": read + n * (lists * 27 * 4 + 12), "flops": n * per * (2 * 850 + 1500)}
    hits = n * per * 6 if noise[0] is None else n * per + sum(noise)
    layers = len(detector(det))
    # candidate-layers of a seed: up to n_best candidates over the layers past the seed
    steps = {"endcaps": 6.2, "dense": 14.5}[det]
    cand = steps * (1.0 + 0.7 * (case["n_best"] - 1))
    if case["do"] == "cascade":
        cand = steps * (1.0 + 0.15 * 0.7 * (case["n_best"] - 1))
    flops = n * (2 * 850 + cand * (700 + 45 + 300))
    bytes_ = hits * 16 + n * (16 + state + 4 * (layers + 3) + 12)
    if case["do"] == "chain":
        flops += n * 3 * 850
        bytes_ += n * (12 + state + 4 + 4)
    return {"bytes": bytes_, "flops": flops * (1.1 if mat else 1.0)}


# ---------------------------------------------------------------------------
# Results in 64 bits: the filter along given hits, out, back and both (finding
# takes decisions, over far more candidates than 64-bit tensors can follow in
# the time: its results are compared with earlier ones only)
# ---------------------------------------------------------------------------

class Filter64:
    """The Kalman filter on tensors of tracks: p [6][n], C [n, 6, 6], all in 64 bits."""

    def __init__(self, G):
        self.G = G

    def at(self, l):
        G = self.G
        self.l, self.cyl, self.rz = l, G.cyl[l], G.rz[l]

    def seed(self, h1, h2, h3, l1):
        a, b, c = ([u - v for u, v in zip(*ab)] for ab in ((h2, h1), (h3, h1), (h3, h2)))
        la, lb, lc = (torch.hypot(v[0], v[1]) for v in (a, b, c))
        h = 2.0 * (a[0] * b[1] - a[1] * b[0]) / (la * lb * lc)
        asinc = lambda v: torch.where(v.abs() < 1e-4, 1.0 + v * v / 6.0, torch.asin(v.clamp(-1, 1)) / torch.where(v == 0, 1.0, v))
        xa, xb = 0.5 * h * la, 0.5 * h * lb
        cot = b[2] / (lb * asinc(xb))
        w = -h / KB
        p = [h1[0], h1[1], h1[2], w, torch.atan2(a[1], a[0]) - xa * asinc(xa), torch.atan2(torch.ones_like(cot), cot)]
        n = w.shape[0]
        C = torch.zeros(n, 6, 6, dtype=torch.float64, device=w.device)
        G = self.G
        s2 = (10.0 * torch.maximum(G.su[l1], G.sv[l1])) ** 2
        r2 = h1[0] ** 2 + h1[1] ** 2
        cyl = G.cyl[l1]
        C[:, 0, 0] = s2 * torch.where(cyl, h1[1] ** 2 / r2, 1.0)
        C[:, 1, 1] = s2 * torch.where(cyl, h1[0] ** 2 / r2, 1.0)
        C[:, 0, 1] = C[:, 1, 0] = s2 * torch.where(cyl, -h1[0] * h1[1] / r2, 0.0)
        C[:, 2, 2] = torch.where(cyl, s2, 0.0)
        C[:, 3, 3] = (0.1 * w) ** 2 + 1e-4
        C[:, 4, 4] = C[:, 5, 5] = 1e-4
        return p, C

    def propagate(self, p, C):
        """Onto the current layers; also which tracks reach them (the others stay)."""
        x, y, z, w, phi, th = p
        cot, h = 1.0 / torch.tan(th), -w * KB
        s = path_to(self.cyl, self.rz, x, y, z, phi, cot, h)
        ok = torch.isfinite(s)
        s = torch.where(ok, s, 1.0)
        a = 0.5 * h * s
        sn = _sinc(a)
        dsn = torch.where(a.abs() < 1e-3, -a / 3.0 + a ** 3 / 30.0, (a * torch.cos(a) - torch.sin(a)) / torch.where(a == 0, 1.0, a * a))
        cm, sm = torch.cos(phi + a), torch.sin(phi + a)
        dx, dy = s * sn * cm, s * sn * sm
        xe, ye = x + dx, y + dy
        cpe, spe = torch.cos(phi + 2 * a), torch.sin(phi + 2 * a)
        n = x.shape[0]
        A = torch.eye(6, dtype=torch.float64, device=x.device).expand(n, 6, 6).clone()
        A[:, 0, 3] = -KB * 0.5 * s * (s * dsn * cm - dy)
        A[:, 1, 3] = -KB * 0.5 * s * (s * dsn * sm + dx)
        A[:, 0, 4], A[:, 1, 4] = -dy, dx
        A[:, 2, 5] = -s / torch.sin(th) ** 2
        A[:, 4, 3] = -KB * s
        d = torch.stack([cpe, spe, cot, torch.zeros_like(x), h, torch.zeros_like(x)], 1)
        nv = torch.zeros(n, 6, dtype=torch.float64, device=x.device)  # surface normal
        nv[:, 0], nv[:, 1], nv[:, 2] = torch.where(self.cyl, xe, 0.0), torch.where(self.cyl, ye, 0.0), torch.where(self.cyl, 0.0, 1.0)
        g = -(nv[:, None, :] @ A)[:, 0] / (nv * d).sum(1)[:, None]
        J = A + d[:, :, None] * g[:, None, :]
        pe = [xe, ye, torch.where(self.cyl, z + s * cot, self.rz), w, phi + 2 * a, th]
        pe = [torch.where(ok, u, v) for u, v in zip(pe, p)]
        return pe, torch.where(ok[:, None, None], J @ C @ J.transpose(1, 2), C), ok

    def _cosa(self, p):
        c = torch.where(self.cyl, torch.sin(p[5]) * torch.cos(p[4] - torch.atan2(p[1], p[0])), torch.cos(p[5]))
        return c.abs().clamp(min=1e-6)

    def scatter(self, p, C):
        t = self.G.x0[self.l]
        st, ct = torch.sin(p[5]), torch.cos(p[5])
        mom = 1.0 / (p[3].abs() * st)
        v = torch.where(t > 0, _theta0(mom, t.clamp(min=1e-30) / self._cosa(p)) ** 2, 0.0)
        wc = p[3] * ct / st
        C = C.clone()
        C[:, 5, 5] += v
        C[:, 4, 4] += v / st ** 2
        C[:, 3, 3] += wc * wc * v
        C[:, 3, 5] -= wc * v
        C[:, 5, 3] -= wc * v
        return C

    def lose(self, p, C):
        t, k = self.G.x0[self.l], self.G.el[self.l]
        st, ct = torch.sin(p[5]), torch.cos(p[5])
        mom = 1.0 / (p[3].abs() * st)
        e = torch.sqrt(mom * mom + PION * PION)
        kx = k * t / self._cosa(p)
        e2 = e - kx * (e / mom) ** 2
        ok = (k > 0) & (t > 0) & (e2 > PION)
        p2 = torch.sqrt((e2 * e2 - PION * PION).clamp(min=1e-12))
        dp2 = e2 / p2 * (mom / e + 2.0 * kx * PION * PION / mom ** 3)
        gp = 1.0 / p2 - mom * dp2 / p2 ** 2
        J = torch.eye(6, dtype=torch.float64, device=mom.device).expand(mom.shape[0], 6, 6).clone()
        J[:, 3, 3] = torch.where(ok, mom / p2 - mom * gp, 1.0)
        J[:, 3, 5] = torch.where(ok, -p[3] * mom * (ct / st) * gp, 0.0)
        p = list(p)
        p[3] = torch.where(ok, p[3] * mom / p2, p[3])
        return p, J @ C @ J.transpose(1, 2)

    def update(self, p, C, hx, hy, hz):
        r = torch.hypot(p[0], p[1])
        cp, sp = p[0] / r, p[1] / r
        n = r.shape[0]
        H = torch.zeros(n, 2, 6, dtype=torch.float64, device=r.device)
        H[:, 0, 0], H[:, 0, 1] = -sp, cp
        H[:, 1, 0], H[:, 1, 1] = torch.where(self.cyl, 0.0, cp), torch.where(self.cyl, 0.0, sp)
        H[:, 1, 2] = torch.where(self.cyl, 1.0, 0.0)
        HC = H @ C
        S = HC @ H.transpose(1, 2)
        S[:, 0, 0] += self.G.su[self.l] ** 2
        S[:, 1, 1] += self.G.sv[self.l] ** 2
        det = S[:, 0, 0] * S[:, 1, 1] - S[:, 0, 1] ** 2
        I = torch.stack([S[:, 1, 1], -S[:, 0, 1], -S[:, 0, 1], S[:, 0, 0]], 1).view(n, 2, 2) / det[:, None, None]
        dphi = torch.atan2(p[0] * hy - p[1] * hx, p[0] * hx + p[1] * hy)
        res = torch.stack([torch.where(self.cyl, self.rz, r) * dphi,
                           torch.where(self.cyl, hz - p[2], torch.hypot(hx, hy) - r)], 1)
        Kt = I @ HC  # the gain's transpose
        dp = (Kt.transpose(1, 2) @ res[:, :, None])[:, :, 0]
        C = C - Kt.transpose(1, 2) @ HC
        chi2 = (res[:, None, :] @ I @ res[:, :, None])[:, 0, 0]
        return [a + dp[:, i] for i, a in enumerate(p)], 0.5 * (C + C.transpose(1, 2)), chi2


def _wrap(a):
    return torch.remainder(a + math.pi, 2.0 * math.pi) - math.pi


def _turned(p, C):
    F = torch.tensor([1.0, 1.0, 1.0, -1.0, 1.0, -1.0], dtype=torch.float64, device=C.device)
    return [p[0], p[1], p[2], -p[3], _wrap(p[4] + math.pi), math.pi - p[5]], C * F[:, None] * F[None, :]


def _pick(m, a, b):
    """a where m, else b, for a state and a covariance."""
    return [torch.where(m, u, v) for u, v in zip(a[0], b[0])], torch.where(m[:, None, None], a[1], b[1])


_LOWER = [(i, j) for i in range(6) for j in range(i + 1)]


def _packed(p, C):
    p = list(p)
    p[4] = _wrap(p[4])
    return torch.stack(p), torch.stack([C[:, i, j] for i, j in _LOWER])


def _along(s, smooth):
    """The filter along s["hits"] from the seed prior: the packed state at the end and chi2; with `smooth` also back from
    there (no material), and the packed mean of the two at each hit."""
    F = Filter64(s["table"])
    hits, xyz, layer = s["hits"].long(), s["xyz"].double(), s["layer"].long()
    rows, n = hits.shape
    at = lambda k: (hits[k] >= 0, hits[k].clamp(min=0))
    first = [at(k)[1] for k in range(3)]  # every list starts with three hits
    h = [[xyz[i][f] for i in range(3)] for f in first]
    p, C = F.seed(h[0], h[1], h[2], layer[first[0]])
    chi2 = torch.zeros(n, dtype=torch.float64, device=xyz.device)
    kept = []
    for k in range(rows):
        m, f = at(k)
        F.at(layer[f])
        np_, nC, ok = F.propagate(p, C) if k else (p, C, torch.ones_like(m))
        if k:
            nC = F.scatter(np_, nC)
            np_, nC = F.lose(np_, nC)
        m = m & ok
        up, uC, x2 = F.update(np_, nC, xyz[0][f], xyz[1][f], xyz[2][f])
        p, C = _pick(m, (up, uC), (p, C))
        chi2 = chi2 + torch.where(m, x2, 0.0)
        if smooth:
            kept.append((m, p, C))
    end = _packed(p, C)
    if not smooth:
        return end, chi2, None
    p, C = _turned(p, C)
    C = C * INFLATE
    started = torch.zeros(n, dtype=torch.bool, device=xyz.device)
    means = []
    for k in reversed(range(rows)):
        m, f = at(k)
        F.at(layer[f])
        np_, nC, ok = F.propagate(p, C)
        np_, nC = _pick(started, (np_, nC), (p, C))
        m = m & (ok | ~started)
        had, kp, kC = kept[k]
        mean = _packed(*_pick(m & started & had, _mean(F, kp, kC, *_turned(np_, nC)), (kp, kC)))
        means.append([torch.where(had, v, math.nan) for v in mean])
        p, C = _pick(m, F.update(np_, nC, xyz[0][f], xyz[1][f], xyz[2][f])[:2], (p, C))
        started = started | m
    return end, chi2, [torch.stack(v) for v in zip(*means[::-1])]


def _mean(F, pf, Cf, pb, Cb):
    """Weighted mean of two states on the current surface in its five free parameters, the sharper in q/pT as base."""
    swap = Cb[:, 3, 3] < Cf[:, 3, 3]
    (pa, Ca), (po, Co) = _pick(swap, (pb, Cb), (pf, Cf)), _pick(swap, (pf, Cf), (pb, Cb))
    n = swap.shape[0]
    r = torch.hypot(pa[0], pa[1])
    P = torch.zeros(n, 5, 6, dtype=torch.float64, device=r.device)
    P[:, 0, 0], P[:, 0, 1] = torch.where(F.cyl, -pa[1] / r, 1.0), torch.where(F.cyl, pa[0] / r, 0.0)
    P[:, 1, 2], P[:, 1, 1] = torch.where(F.cyl, 1.0, 0.0), torch.where(F.cyl, 0.0, 1.0)
    P[:, 2, 3] = P[:, 3, 4] = P[:, 4, 5] = 1.0
    Pt = P.transpose(1, 2)
    d = [a - b for a, b in zip(po, pa)]
    d[4] = _wrap(d[4])
    S = P @ (Ca + Co) @ Pt
    sc = 1.0 / torch.sqrt(torch.diagonal(S, dim1=1, dim2=2).clamp(min=1e-300))
    S = S * sc[:, :, None] * sc[:, None, :]
    S = torch.where(torch.isfinite(S), S, torch.eye(5, dtype=torch.float64, device=r.device))
    X = torch.linalg.solve_ex(S, sc[:, :, None] * (P @ Ca))[0] * sc[:, :, None]
    dp = (X.transpose(1, 2) @ (P @ torch.stack(d, 1)[:, :, None]))[:, :, 0]
    ps = [a + dp[:, i] for i, a in enumerate(pa)]
    A = torch.eye(6, dtype=torch.float64, device=r.device) - X.transpose(1, 2) @ P
    Cs = A @ Ca @ A.transpose(1, 2) + X.transpose(1, 2) @ (P @ Co @ Pt) @ X
    r = torch.hypot(ps[0], ps[1])
    nv = torch.zeros(n, 6, dtype=torch.float64, device=r.device)
    nv[:, 0], nv[:, 1] = torch.where(F.cyl, ps[0] / r, 0.0), torch.where(F.cyl, ps[1] / r, 0.0)
    nv[:, 2] = torch.where(F.cyl, 0.0, 1.0)
    f = torch.where(F.cyl, F.rz / r, 1.0)
    ps[0], ps[1], ps[2] = ps[0] * f, ps[1] * f, torch.where(F.cyl, ps[2], F.rz)
    N = torch.eye(6, dtype=torch.float64, device=r.device) - nv[:, :, None] * nv[:, None, :]
    return ps, N @ Cs @ N


def _train64(case, seed, dev):
    f, label, w, m, v = train_inputs(case, seed, dev)
    t, lr, b1, b2, eps = 101, _f32(2e-3), _f32(0.9), _f32(0.999), _f32(1e-8)
    x, y = f.double(), label.double()
    p = w.bfloat16().double().requires_grad_(True)
    z = torch.relu(x @ p[:768].view(64, 12).T + p[768:832]) @ p[832:896] + p[896]
    loss = (z.clamp(min=0) - z * y + torch.log1p(torch.exp(-z.abs()))).mean()
    loss.backward()
    g = p.grad
    m2, v2 = b1 * m.double() + (1 - b1) * g, b2 * v.double() + (1 - b2) * g * g
    w2 = w.double() - lr * (m2 / (1 - b1 ** t)) / (torch.sqrt(v2 / (1 - b2 ** t)) + eps)
    return dict(w=w2, m=m2, v=v2, w_bf16=None, loss=loss.detach().reshape(1))


def exact(case, seed):
    dev = torch.device(DEVICE, torch.cuda.current_device()) if DEVICE == "cuda" else torch.device(DEVICE)
    if case["do"] == "train":
        return _train64(case, seed, dev)
    if case["do"] not in ("fit", "refit", "smooth") or case.get("field"):
        return None  # finding: see above; the field: its integration steps are part of the result
    (par, cov), chi2, means = _along(make_events(case, seed, dev), case["do"] == "smooth")
    if means:
        par, cov = means
    out = dict(par=par, cov=cov, chi2=chi2, ndf=None, status=None)
    # back through material a few tracks in 10^5, the ones with a poor seed, take another crossing of a layer in 32 bits
    # than in 64 and end centimetres away: no value for that half
    return {"out": out, "back": None} if case["do"] == "refit" else out
