"""Performance cases of the collision library: the work its users have it do, through the
public entry points (`binding.Session` and the gd_* calls of include/gd.h).

Kinds of case
  interval  whole frozen-neighbour intervals (build, rates, sample): three calls an interval,
            or replayed as a CUDA graph; optionally a push after each.  Each pass starts from
            the same diameters (a batch of initial states handed in anew), so passes cost alike.
  lists     gd_build_neighbors with its lists and distances handed out
  fixed     gd_neighbors_fixed, the search without device allocation
  step      gd_step, the split timestep C D T D C on moving particles
  push      gd_push_staggered, plain or with radiation forces
  collide   gd_collide, a bounded collision step, in one or several spatial groups

Inputs follow the recipes of workloads.py (local patches; global disks of 5-100 au) with the
seed's own draws.
"""
import math

import numpy as np
import torch

from paper_2609_35967_gb300 import binding as gd
from paper_2609_35967_gb300 import workloads as W

AU, YR = W.AU, W.YR
PATCH_K = 32


def listed():
    return [
        # a user's first run: one small patch in the plain form, intervals replayed as a graph
        {"name": "patch4k_fp64_graph", "kind": "interval", "geometry": "patch", "n": 4096, "K": 32,
         "mixed": False, "graph": 10, "push": False, "sizes": "mono", "model": 0},
        # the same patch, one mixed interval by calls: launches and latency
        {"name": "patch4k_mixed", "kind": "interval", "geometry": "patch", "n": 4096, "K": 32,
         "mixed": True, "graph": 0, "push": False, "sizes": "mono", "model": 0},
        # a parameter study: 256 uneven patches in one context, one graph replay an interval
        {"name": "patches256_mixed_graph", "kind": "interval", "geometry": "patches", "n": 256, "K": 32,
         "mixed": True, "graph": 1, "push": False, "sizes": "mono", "model": 0},
        # a global disk of equal grains at a usual resolution
        {"name": "disk1m_mixed", "kind": "interval", "geometry": "disk", "n": 1 << 20, "K": 32,
         "mixed": True, "graph": 0, "push": False, "sizes": "mono", "model": 0},
        # the production disk: a broad size distribution, many events in few particles
        {"name": "disk4m_mixed", "kind": "interval", "geometry": "disk", "n": 1 << 22, "K": 32,
         "mixed": True, "graph": 0, "push": False, "sizes": "broad", "model": 0},
        # the plain FP64 form of a disk, with lambda*_i handed out; an odd size
        {"name": "disk1m5_fp64", "kind": "interval", "geometry": "disk", "n": 1500007, "K": 32,
         "mixed": False, "graph": 0, "push": False, "sizes": "broad", "model": 0},
        # the largest: K = 48 and a push after the interval, so every build is on moved particles
        {"name": "disk16m_k48_push", "kind": "interval", "geometry": "disk", "n": 1 << 24, "K": 48,
         "mixed": True, "graph": 0, "push": True, "sizes": "narrow", "model": 0},
        # neighbour lists as the product, a large K and an odd size
        {"name": "lists100k_k128", "kind": "lists", "geometry": "patch", "n": 100003, "K": 128, "mixed": True,
         "model": 0},
        # the split timestep of a moving disk: two collision steps, two diffusions, one push
        {"name": "step1m_mixed", "kind": "step", "n": 1 << 20, "K": 32, "mixed": True},
        # trajectories with radiation pressure, Poynting-Robertson drag and the optical depth grid
        {"name": "push2m_rad_mixed", "kind": "push", "n": 1 << 21, "mixed": True, "rad": True},
        # a bounded collision step in eight radial groups: many short rounds
        {"name": "groups8_256k_collide", "kind": "collide", "n": 1 << 18, "K": 32, "mixed": True, "groups": 8},
        # lists for a caller that cannot allocate, at an odd size
        {"name": "fixed50k_k32", "kind": "fixed", "geometry": "disk", "n": 50001, "K": 32},
    ]


def _log_int(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng):
    kind = rng.choice(("interval", "interval", "interval", "lists", "step", "push", "collide", "fixed"))
    mixed = rng.random() < 0.7
    if kind == "interval":
        geometry = rng.choice(("patch", "disk", "disk", "patches"))
        K = rng.choice((16, 32, 32, 48, 64, 100))
        n = (rng.randint(3, 200) if geometry == "patches"
             else _log_int(rng, 1500, (3 << 20) if mixed else (3 << 18)))
        push = geometry == "disk" and rng.random() < 0.3
        return {"kind": kind, "geometry": geometry, "n": n, "K": K, "mixed": mixed,
                "graph": rng.choice((0, 0, 1, 4)) if n < 300000 else 0, "push": push,
                "sizes": rng.choice(("mono", "broad", "narrow")),
                "model": rng.choice((0, 0, 0, 2)) if geometry == "disk" else 0}
    if kind == "lists":
        return {"kind": kind, "geometry": rng.choice(("patch", "disk")), "n": _log_int(rng, 1000, 1 << 20),
                "K": rng.choice((8, 32, 33, 64, 128, 200)), "mixed": mixed, "model": 0}
    if kind == "step":
        return {"kind": kind, "n": _log_int(rng, 4000, 1 << 21 if mixed else 1 << 18), "K": rng.choice((16, 32, 48)),
                "mixed": mixed}
    if kind == "push":
        return {"kind": kind, "n": _log_int(rng, 10000, 1 << 23), "mixed": mixed, "rad": rng.random() < 0.5}
    if kind == "collide":
        return {"kind": kind, "n": _log_int(rng, 4000, 1 << 19 if mixed else 1 << 16), "K": rng.choice((16, 32)),
                "mixed": mixed, "groups": rng.choice((1, 2, 5, 8, 13))}
    return {"kind": kind, "geometry": rng.choice(("patch", "disk")), "n": _log_int(rng, 1000, 65536),
            "K": rng.choice((8, 16, 32, 48, 64))}


# ------------------------------------------------------------------ inputs
SIZES = {"mono": (1.0, 0.0), "broad": (10.0, 1.0), "narrow": (1.0, 0.5)}   # median [um], sigma of ln a
ALPHA_V = {"mono": (1e-3, 100.0), "broad": (1e-3, 100.0), "narrow": (3e-3, 500.0)}


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)


def _uniform(g, n, lo, hi):
    return lo + (hi - lo) * torch.rand(n, generator=g, device="cuda", dtype=torch.float64)


def _normal(g, n):
    return torch.randn(n, generator=g, device="cuda", dtype=torch.float64)


def _numpy(ins):
    return {k: v.cpu().numpy() if isinstance(v, torch.Tensor) else v for k, v in ins.items()}


def _diameters(g, n, sizes):
    med, sig = SIZES[sizes]
    s = 2e-4 * med * torch.exp(sig * _normal(g, n)) if sig else torch.full((n,), 2e-4 * med, device="cuda",
                                                                          dtype=torch.float64)
    return torch.where(s < W.S_MIN, 2.0 * W.S_MIN - s, s)     # reflected at the smallest fragment


def _disk(n, seed, K, sizes, **extra):
    """A global disk of 5-100 au at the gas velocity (the recipe of workloads.disk_instance)."""
    alpha, vf = ALPHA_V[sizes]
    P = W.disk_instance(64, seed=int(seed) % 100000 + 1, K=K, alpha=alpha, v_frag=vf, **extra)["params"]
    g = _gen(seed)
    R = _uniform(g, n, 5 * AU, 100 * AU)
    phi = _uniform(g, n, 0.0, 2 * math.pi)
    s = _diameters(g, n, sizes)
    T, sig = 280.0 * (R / AU) ** -0.5, 1700.0 * (R / AU) ** -1.0
    om = torch.sqrt(W._G * W.MSUN / R ** 3)
    Hg = torch.sqrt(W._KB * T / (W._MU * W._MH)) / om
    St = math.pi * P["rho_s"] * s / (4.0 * sig)
    z = _normal(g, n) * Hg * torch.sqrt(alpha / (alpha + St))
    h, r = Hg / R, torch.sqrt(R * R + z * z)
    eta = -0.5 * (-2.75 * h * h - 0.5 * (1.0 - R / r))
    M = torch.full_like(R, 0.01 * 2 * math.pi * 1700.0 * AU * 95.0 * AU / n)
    return dict(params=P, x=R * torch.cos(phi), y=R * torch.sin(phi), z=z, s=s, M=M,
                vr=torch.zeros_like(R), lth=torch.zeros_like(R), lph=torch.sqrt(1.0 - 2.0 * eta) * om * R * R)


def _patch(n, seed, K, sizes="mono", **kw):
    """One local patch (the recipe of workloads.patch_instance)."""
    small = W.patch_instance(64, seed=int(seed) % 100000 + 1, K=K, **kw)
    P = small["params"]
    g = _gen(seed)
    L = P["box_x"]
    M = torch.full((n,), float(small["M"].sum()) / n, device="cuda", dtype=torch.float64)
    return dict(params=P, x=_uniform(g, n, -0.5 * L, 0.5 * L), y=_uniform(g, n, -0.5 * L, 0.5 * L),
                z=0.1 * L * _normal(g, n), s=_diameters(g, n, sizes), M=M)


RAD = dict(beta0=0.05, kappa0=3.0, rad_s0=2e-4, rad_pr=1, tau_nr=256, tau_nmu=16, tau_nphi=256,
           tau_rmin=5 * AU, tau_rmax=100 * AU, tau_mu=0.2)


def _instances(case, seed):
    kind, K = case["kind"], case.get("K", PATCH_K)
    if kind in ("step", "collide"):
        extra = {"spatial_groups": case["groups"]} if kind == "collide" else {}
        return [_disk(case["n"], seed, K, "broad", **extra)]
    if kind == "push":
        return [_disk(case["n"], seed, K, "broad", **(RAD if case["rad"] else {}))]
    if case["geometry"] == "disk":
        return [_disk(case["n"], seed, K, case.get("sizes", "mono"), model=case.get("model", 0))]
    if case["geometry"] == "patch":
        return [_patch(case["n"], seed, K, case.get("sizes", "mono"))]
    meta = np.random.default_rng(743 + case["n"])     # the batch's sizes and disks belong to the case
    out = []
    for b in range(case["n"]):
        r = meta.uniform(5.0, 50.0)
        out.append(_patch(max(K, int(2.0 ** meta.uniform(10.0, 16.0))), int(seed) * 1000 + b, K, case["sizes"],
                          r_au=r, sigma=100.0 / r, T=50.0 * (r / 10.0) ** -0.5,
                          alpha=10.0 ** meta.uniform(-4.0, -2.0), v_frag=meta.uniform(100.0, 1000.0)))
    return out


# ------------------------------------------------------------------ state and pass
def prepare(case, seed):
    insts = [_numpy(i) for i in _instances(case, seed)]
    kind = case["kind"]
    st = {"case": dict(case)}
    if kind == "fixed":
        dev = torch.device("cuda:0")
        n = case["n"]
        st["xyz"] = [torch.as_tensor(insts[0][k], device=dev) for k in ("x", "y", "z")]
        st["params"] = gd.instance_params(insts[0]["params"])
        st["nbr"] = torch.empty((n, case["K"]), dtype=torch.int32, device=dev)
        st["d"] = torch.empty(n, dtype=torch.float64, device=dev)
        return st
    vel = kind in ("step", "push") or case.get("push", False)
    K = case.get("K", PATCH_K)
    S = gd.Session(insts, K=K, precision=gd.GD_MIXED if case["mixed"] else gd.GD_FP64, velocities=vel)
    st["S"], st["s0"] = S, S.t["s"].clone()
    st["dt_coll"] = insts[0]["params"]["dt_coll"]
    if kind == "lists":
        st["nbr"] = torch.empty((S.N, S.K), dtype=torch.int32, device=S.device)
        st["d"] = torch.empty(S.N, dtype=torch.float64, device=S.device)
    if kind == "interval" and not case["mixed"] and not case["graph"]:
        st["lam"] = torch.empty(S.N, dtype=torch.float64, device=S.device)
    torch.cuda.synchronize()
    return st


def run(st):
    case, S = st["case"], st.get("S")
    kind = case["kind"]
    if kind == "fixed":
        x, y, z = st["xyz"]
        gd.gd_neighbors_fixed(x.data_ptr(), y.data_ptr(), z.data_ptr(), case["n"], case["K"], st["params"],
                              st["nbr"].data_ptr(), st["d"].data_ptr())
        return {"nbr": st["nbr"], "d": st["d"]}
    if kind == "lists":
        gd.gd_build_neighbors(S.ctx, st["nbr"].data_ptr(), st["d"].data_ptr())
        return {"nbr": st["nbr"], "d": st["d"]}
    if kind == "push":
        S.push_staggered(0.25 * YR)
        return {k: S.t[k] for k in ("x", "y", "z", "vr", "lth", "lph")}
    with torch.cuda.stream(S.stream):
        S.t["s"].copy_(st["s0"])
    if kind == "step":
        n = S.step(0.25 * YR, reuse_lists=True)
        return dict({k: S.t[k] for k in ("x", "y", "z", "vr", "lth", "lph", "s")}, intervals=n)
    if kind == "collide":
        n = S.collide(st["dt_coll"])
        return {"s": S.t["s"], "intervals": n}
    if case["graph"]:
        S.run_intervals(case["graph"], case["push"])
    else:
        S.build_neighbors()
        gd.gd_collision_rates(S.ctx, st["lam"].data_ptr() if "lam" in st else 0)
        S.sample_collisions()
        if case["push"]:
            S.push_staggered(-1.0)
    out = {"s": S.t["s"]}
    if "lam" in st:
        out["lam"] = st["lam"]
    if case["push"]:
        out.update({k: S.t[k] for k in ("x", "y", "z", "vr", "lth", "lph")})
    return out


def work(case):
    """Bytes: each array the call takes read once, each it gives written once.  Flops: 8 per
    candidate of a ball twice the neighbourhood's size and 100 per pair rate; 200 per pushed
    particle, 300 per diffused one."""
    kind, K = case["kind"], case.get("K", PATCH_K)
    n = case["n"]
    if case.get("geometry") == "patches":
        n = int(n * (2 ** 16 - 2 ** 10) / (6 * math.log(2.0)))     # mean of 2^U(10, 16)
    if kind in ("lists", "fixed"):
        return {"bytes": n * (24 + 4 * K + 8), "flops": n * 16 * K}
    if kind == "push":
        return {"bytes": n * (56 + 48 + (8 if case["rad"] else 0)), "flops": n * 200}
    pair = n * K * (16 + 100)
    if kind == "step":
        return {"bytes": n * (64 + 56), "flops": 2 * pair + n * 800}
    if kind == "collide":
        return {"bytes": n * 48, "flops": pair + n * K * 100}
    m = max(1, case["graph"])
    return {"bytes": n * (48 + (96 if case["push"] else 0)),
            "flops": m * (pair + (200 * n if case["push"] else 0))}


# ------------------------------------------------------------------ 64-bit values
def _knn64(ins, K):
    """Indices and distance^2 of the K-1 nearest others of every particle, brute force."""
    x, y, z, P = ins["x"], ins["y"], ins["z"], ins["params"]
    n, rows = len(x), max(1, (1 << 27) // len(x))
    idx = torch.empty((n, K - 1), dtype=torch.int64, device="cuda")
    far = torch.empty(n, dtype=torch.float64, device="cuda")
    for a in range(0, n, rows):
        b = min(n, a + rows)
        d2 = torch.zeros((b - a, n), dtype=torch.float64, device="cuda")
        for c, box in ((x, P["box_x"]), (y, P["box_y"]), (z, 0.0)):
            t = c[None, :] - c[a:b, None]
            if box > 0.0:
                t = torch.where(t > 0.5 * box, t - box, torch.where(t < -0.5 * box, t + box, t))
            d2 += t * t
        d2[torch.arange(b - a, device="cuda"), torch.arange(a, b, device="cuda")] = math.inf
        v, i = torch.topk(d2, K - 1, dim=1, largest=False)
        idx[a:b], far[a:b] = i, v.amax(dim=1)
    return idx, far


def _gas64(P, R, Z):
    GM = 6.674e-8 * P["M_star"]
    kB, mH, mu = 1.380649e-16, 1.6735575e-24, 2.34
    r = torch.sqrt(R * R + Z * Z)
    Om = torch.sqrt(GM / R ** 3)
    T = P["T0"] * (R / P["r0"]) ** P["q"]
    cs = torch.sqrt(kB * T / (mu * mH))
    H = cs / Om
    h = H / R
    Sig = P["sigma0"] * (R / P["r0"]) ** P["p"]
    up = Z * Z / (r * (r + R))                                      # 1 - R/r
    v = up / (h * h)
    rho = Sig / (math.sqrt(2 * math.pi) * H) * torch.exp(-v)
    eta = -0.5 * ((P["p"] + 0.5 * P["q"] - 1.5) * h * h + P["q"] * up)
    numol = 0.5 * math.sqrt(8 / math.pi) * cs * mu * mH / (rho * 2e-15)
    return dict(Om=Om, T=T, cs=cs, eta=eta, Re=P["alpha"] * cs * H / numol, H=H,
                gst=math.pi * P["rho_s"] / (4 * Sig) * torch.exp(v))


def _rates64(ins, K):
    """lambda*_i of every particle (physical kernel, 3D model)."""
    P = ins["params"]
    idx, far = _knn64(ins, K)
    idx = torch.cat([torch.arange(len(far), device="cuda")[:, None], idx], dim=1)
    d = torch.sqrt(far)
    V = 4.0 * math.pi * d ** 3 / 3.0
    if P["geometry"] == W.PATCH:
        R = P["r0"] + ins["x"]
    else:
        R = torch.sqrt(ins["x"] ** 2 + ins["y"] ** 2)
        for h in (R - P["R_in"], P["R_out"] - R):
            V = V - torch.where((h > 0) & (h < d), math.pi * (d - h) ** 2 * (2 * d + h) / 3.0, torch.zeros_like(d))
    g = {k: v[:, None] for k, v in _gas64(P, R, ins["z"]).items()}
    s, M = ins["s"], ins["M"]
    m = math.pi * P["rho_s"] * s ** 3 / 6.0
    si, mi, sj, mj = s[:, None], m[:, None], s[idx], m[idx]
    a, b = g["gst"] * si, g["gst"] * sj
    vK, half = (R[:, None] * g["Om"]), torch.full((), 0.5, dtype=torch.float64, device="cuda")
    dR = 2 * g["eta"] * vK * (a / (1 + a * a) - b / (1 + b * b))
    dZ = ins["z"][:, None] * g["Om"] * (torch.minimum(a, half) - torch.minimum(b, half))
    dP = g["eta"] * vK * (1 / (1 + a * a) - 1 / (1 + b * b))
    dB = torch.minimum(g["cs"], torch.sqrt(8 * 1.380649e-16 * g["T"] / math.pi * (1 / mi + 1 / mj)))
    s1, s2, te, Vg = torch.maximum(a, b), torch.minimum(a, b), 1 / torch.sqrt(g["Re"]), 1.5 * P["alpha"] * g["cs"] ** 2
    e = s2 / s1
    tiny = (s1 - s2) ** 2 * (s1 * s2 + te * (s1 + s2)) / ((s1 + s2) * (s1 + te) * (s2 + te))
    mid = s1 * (3.2 - (1 + e) + 2 / (1 + e) * (1 / 2.6 + e ** 3 / (1.6 + e)))
    big = 1 / (1 + s1) + 1 / (1 + s2)
    dv = torch.sqrt(dR ** 2 + dZ ** 2 + dP ** 2 + dB ** 2 + Vg * torch.where(s1 < te, tiny, torch.where(s1 < 1, mid, big)))
    psi = mj / mi
    rate = (M[idx] / mj) * math.pi * (si + sj) ** 2 * dv / 4.0 / V[:, None]
    nc = torch.where(psi <= 1e-6, torch.floor(1e-4 / psi), torch.ones_like(psi))
    erode = (1 - psi) * rate / nc + psi * rate
    return torch.where(dv < P["v_frag"], rate / nc, torch.where(psi <= 0.1, erode, rate)).sum(dim=1)


def _push64(ins, dt):
    """One staggered step (Sect. 2.3.3) with the radiation forces the parameters name."""
    P = ins["params"]
    GM, h = 6.674e-8 * P["M_star"], 0.5 * dt
    X, Y, Z, s, M = (ins[k] for k in ("x", "y", "z", "s", "M"))
    VR, LT, LP = ins["vr"], ins["lth"], ins["lph"]
    r = torch.sqrt(X * X + Y * Y + Z * Z)
    th, ph = torch.atan2(torch.sqrt(X * X + Y * Y), Z), torch.atan2(Y, X)
    ph = ph + h * LP / (r * torch.sin(th)) ** 2
    th = th + h * LT / (r * r)
    r = r + h * VR
    sn, cs = torch.sin(th), torch.cos(th)
    be, gpr = torch.zeros_like(r), torch.zeros_like(r)
    if P.get("beta0", 0.0) > 0.0:
        tau = _tau64(P, r, cs, ph, s, M)
        be = P["beta0"] * P["rad_s0"] / s * torch.exp(-tau)
        gpr = be * GM / (2.99792458e10 * r * r)
    g = _gas64(P, r * sn, r * cs)
    gam = g["Om"] / (g["gst"] * s)
    fr = -(1.0 - be) * GM / r ** 2 + LT ** 2 / r ** 3 + LP ** 2 / (r ** 3 * sn ** 2)
    ft = LP ** 2 * cs / (r ** 2 * sn ** 3)
    yg = torch.sqrt(1.0 - 2.0 * g["eta"]) * torch.sqrt(GM * r * sn)
    gr, gt = gam + 2.0 * gpr, gam + gpr
    kr, kt = -torch.expm1(-dt * gr) / gr, -torch.expm1(-dt * gt) / gt
    VR = VR + kr * (fr - gr * VR)
    LT = LT + kt * (ft - gt * LT)
    LP = LP + kt * (gam * yg - gt * LP)
    r = r + h * VR
    th = th + h * LT / (r * r)
    ph = ph + h * LP / (r * torch.sin(th)) ** 2
    sn = torch.sin(th)
    return dict(x=r * sn * torch.cos(ph), y=r * sn * torch.sin(ph), z=r * torch.cos(th), vr=VR, lth=LT, lph=LP)


def _tau64(P, r, mu, ph, s, M):
    """The optical depth at (r, mu, phi): cell deposit, radial prefix, linear interpolation."""
    nr, nm, npp = P["tau_nr"], P["tau_nmu"], P["tau_nphi"]
    dr, dm, dp = (P["tau_rmax"] - P["tau_rmin"]) / nr, 2 * P["tau_mu"] / nm, 2 * math.pi / npp
    ph = ph - 2 * math.pi * torch.floor((ph + math.pi) / (2 * math.pi))
    u, w, v = (r - P["tau_rmin"]) / dr, (mu + P["tau_mu"]) / dm, (ph + math.pi) / dp
    i, j, k = (t.floor().long() for t in (u, w, v))
    k = k.clamp(0, npp - 1)
    ok = (i >= 0) & (i < nr) & (j >= 0) & (j < nm)
    cell = ((j * npp + k) * nr + i)[ok]
    acc = torch.zeros(nm * npp * nr, dtype=torch.float64, device="cuda")
    acc.index_add_(0, cell, (P["kappa0"] * P["rad_s0"] / s * M)[ok])
    e = P["tau_rmin"] + dr * torch.arange(nr + 1, dtype=torch.float64, device="cuda")
    acc = acc.view(nm * npp, nr) / ((e[1:] ** 3 - e[:-1] ** 3) / 3.0 * dm * dp) * dr
    T = torch.cat([torch.zeros((nm * npp, 1), dtype=torch.float64, device="cuda"), acc.cumsum(dim=1)], dim=1)
    fr = (u - i).clamp(0, 1)
    i0 = i.clamp(0, nr)
    inside, beyond = u > 0, u >= nr
    wm = (w - 0.5).clamp(0, nm - 1)
    j0 = wm.floor().long().clamp(0, max(nm - 2, 0))
    fm, vp = wm - j0, v - 0.5
    k0 = vp.floor().long()
    fp = vp - k0
    tau = torch.zeros_like(r)
    for dj, wj in ((0, 1 - fm), (1, fm)):
        for dk, wk in ((0, 1 - fp), (1, fp)):
            col = (j0 + dj).clamp(0, nm - 1) * npp + (k0 + dk) % npp
            t0, t1 = T[col, i0], T[col, (i0 + 1).clamp(max=nr)]
            tau += wj * wk * torch.where(beyond, T[col, torch.full_like(i0, nr)], t0 + fr * (t1 - t0))
    return torch.where(inside, tau, torch.zeros_like(tau))


def exact(case, seed):
    """64-bit values where they follow from the inputs alone in one step: list distances,
    lambda*_i and trajectories.  Event outcomes are draws through many states: none."""
    kind = case["kind"]
    if kind in ("lists", "fixed") and case["n"] <= 120000 and case.get("model", 0) == 0:
        return {"nbr": None, "d": torch.sqrt(_knn64(_instances(case, seed)[0], case["K"])[1])}
    if kind == "push":
        return _push64(_instances(case, seed)[0], 0.25 * YR)
    if (kind == "interval" and not case["mixed"] and not case["graph"] and not case["push"]
            and case["model"] == 0 and case["geometry"] != "patches" and case["n"] <= 120000):
        return {"s": None, "lam": _rates64(_instances(case, seed)[0], case["K"])}
    return None
