"""What this library is measured on: the calls a host model or a training
script makes, over the range of grids, level counts, precisions and options
the configurations, tests and the benchmark of this repository use.

A case names one public call and its sizes:

  step     Dycore.step, the whole time step as one CUDA graph (device state)
  host     the same call on pinned host arrays (copies in and out around it)
  solve    Dycore.nh_solve, one substep, as a host model that runs its own
           substep loop calls it
  diff     Dycore.nh_diff, the horizontal diffusion alone
  learned  step_learned, the reduced step, both networks and the check
  column   column_solve_noalloc, the vertically implicit solve on the
           caller's arrays
  train    MLP.train_step, a few optimiser steps and the updated weights

States are the balanced jet with a seeded bump plus seeded small-scale noise
in vn and w, so that every term of the scheme works on nonzero values.
"""
import functools
import math

import numpy as np
import torch

import paper_2608_21150_gb300 as P
from icon_inputs import make_grid, make_vct, mountain_height, sample_perturbation_centre, terrain_following_z
from paper_2608_21150_gb300 import corrector

GRAV, RD, CPD, P00, OMEGA, RADIUS, T0 = 9.80665, 287.04, 1004.64, 1.0e5, 7.29212e-5, 6.371229e6, 250.0
CVD = CPD - RD
H = CPD * T0 / GRAV
DAMP_HEIGHT = 20000.0
FIELDS = ("vn", "w", "rho", "exner", "theta_v", "exner_pr")
REDUCED = dict(ndyn_substeps=3, exner_exfac=0.0, divdamp_fac=0.004)
HIDDEN = 512
COL_COLUMNS_LIMIT = 1047232  # column-levels of column_solve_noalloc's scratch


def listed():
    def step(name, kind, prec, bis, nlev, dt, **more):
        return dict(dict(name=name, kind=kind, prec=prec, bis=bis, nlev=nlev, dt=dt, ndyn=5, rayleigh=0.05,
                         terrain=False), **more)

    return [
        # the test configuration: a coarse grid, where launches and the column's serial chain count
        step("step_fp64_r2b2_l30", "step", "fp64", 2, 30, 1800.0, rayleigh=0.0),
        # a medium grid with Rayleigh damping
        step("step_fp64_r2b4_l65", "step", "fp64", 4, 65, 720.0),
        # the benchmark's grid in FP64 and in mixed precision
        step("step_fp64_r2b6_l90", "step", "fp64", 6, 90, 360.0),
        step("step_mixed_r2b6_l90", "step", "mixed", 6, 90, 360.0),
        # FP32 stencils with the FP64 column solve, an odd level count
        step("step_f64col_r2b4_l47", "step", "f64col", 4, 47, 720.0),
        # mixed precision over a Gaussian mountain (terrain-following heights)
        step("step_mixed_terrain_r2b5_l90", "step", "mixed", 5, 90, 360.0, terrain=True),
        # a host model's state in host memory
        step("host_fp64_r2b4_l65", "host", "fp64", 4, 65, 720.0),
        # one substep of a host model's own loop, mixed precision, few levels
        step("solve_mixed_r2b3_l31", "solve", "mixed", 3, 31, 1200.0),
        # the diffusion alone
        step("diff_fp64_r2b5_l90", "diff", "fp64", 5, 90, 360.0),
        # the learned step: 3 reduced substeps, column and edge network
        step("learned_r2b5_l90", "learned", "mixed", 5, 90, 720.0),
        # the corrector form of the column solve near the static scratch's limit
        dict(name="column_fp64_11500_l90", kind="column", prec="fp64", cols=11500, nlev=90, dt=360.0, ndyn=5,
             rayleigh=0.05, corr=True),
        # training the column network: four optimiser steps of 4096 rows
        dict(name="train_col_l90_4096", kind="train", nlev=90, edge=False, batch=4096, steps=4, lr=1e-3),
    ]


def draw(rng):
    kind = rng.choice(["step", "step", "step", "host", "solve", "diff", "learned", "column", "train"])
    nlev = rng.randint(20, 100)
    if kind == "train":
        return dict(kind=kind, nlev=nlev, edge=rng.random() < 0.5, batch=64 * int(round(2 ** rng.uniform(3, 8))),
                    steps=rng.randint(1, 6), lr=1e-3)
    if kind == "column":
        cols = int(2 ** rng.uniform(6, math.log2(COL_COLUMNS_LIMIT // (nlev + 1))))
        return dict(kind=kind, prec=rng.choice(["fp64", "mixed"]), cols=cols, nlev=nlev, dt=360.0, ndyn=5,
                    rayleigh=rng.choice([0.0, 0.05]), corr=rng.random() < 0.5)
    top = {"host": 5, "learned": 5}.get(kind, 6)
    bis = rng.choice(list(range(1, top + 1)))
    ndyn = rng.choice([3, 4, 5, 5, 6]) if kind != "learned" else 5
    prec = "mixed" if kind == "learned" else rng.choice(["fp64", "mixed", "f64col"])
    terrain = bis <= 5 and kind in ("step", "solve") and rng.random() < 0.25
    if bis == 6:  # no dearer than the largest listed case
        nlev, ndyn = min(nlev, 80), min(ndyn, 5)
    return dict(kind=kind, prec=prec, bis=bis, nlev=nlev, dt=min(1800.0, 360.0 * 2.0 ** (6 - bis)) * min(ndyn, 5) / 5,
                ndyn=ndyn, rayleigh=rng.choice([0.0, 0.05]), terrain=terrain)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _device():
    return torch.device("cuda") if torch.cuda.is_available() else torch.device("cpu")


@functools.lru_cache(maxsize=2)
def _raw_grid(bis):
    """The grid as a grid file would hold it (host arrays)."""
    return make_grid(bis)


def _heights(case):
    z = make_vct(case["nlev"])
    if not case.get("terrain"):
        return z
    return terrain_following_z(z, mountain_height(_raw_grid(case["bis"]).cell_xyz, h0=2000.0, d=1.5e6))


def _generator(seed, dev):
    g = torch.Generator(device=dev)
    g.manual_seed(1000003 + int(seed))
    return g


def _jet(phi, z):
    """Exner, theta_v and the zonal wind of the balanced jet at latitude phi and height z."""
    s = z / 11000.0
    eps = 0.12 * s * torch.exp(1.0 - s)
    deps = 0.12 / 11000.0 * (1.0 - s) * torch.exp(1.0 - s)
    ez = torch.exp(-z / H)
    c = torch.cos(phi)
    G = 8.0 / 15.0 - 4.0 * (c ** 3 / 3.0 - c ** 5 / 5.0)
    pi = ez * (1.0 - eps * G)
    theta = GRAV / (CPD * ez * ((1.0 - eps * G) / H + deps * G))
    ap = phi.abs()
    press = CPD * theta / RADIUS * ez * eps * torch.sin(ap) * torch.sin(2.0 * phi) ** 2
    f = 2.0 * OMEGA * torch.sin(ap)
    den = f + torch.sqrt(f * f + 4.0 * torch.tan(ap) / RADIUS * press)
    return pi, theta, torch.where(den > 0.0, 2.0 * press / den.clamp(min=1e-300), torch.zeros_like(den))


def _state(case, seed):
    """vn, w, rho, exner, theta_v of the case as float64 tensors."""
    dev = _device()
    g = _raw_grid(case["bis"])
    z = torch.from_numpy(_heights(case)).to(dev)
    z_mc = 0.5 * (z[..., :-1] + z[..., 1:])
    zc = z_mc[None, :] if z_mc.dim() == 1 else z_mc
    e2c = torch.from_numpy(g.e2c).to(dev).long()
    C, E = torch.from_numpy(g.cell_xyz).to(dev), torch.from_numpy(g.edge_xyz).to(dev)
    ze = zc if zc.shape[0] == 1 else 0.5 * (zc[e2c[:, 0]] + zc[e2c[:, 1]])
    exner, theta, _ = _jet(torch.asin(C[:, 2].clamp(-1, 1))[:, None], zc)
    rho = P00 * exner ** (CVD / RD) / (RD * theta)
    u = _jet(torch.asin(E[:, 2].clamp(-1, 1))[:, None], ze)[2]
    lon, lat = sample_perturbation_centre(seed)
    centre = torch.tensor([math.cos(lat) * math.cos(lon), math.cos(lat) * math.sin(lon), math.sin(lat)], device=dev,
                          dtype=torch.float64)
    r = torch.arccos((E @ centre).clamp(-1, 1))
    u = u + torch.exp(-(10.0 * r) ** 2)[:, None]
    up = torch.tensor([0.0, 0.0, 1.0], device=dev, dtype=torch.float64).expand_as(E)
    east = torch.nn.functional.normalize(torch.linalg.cross(up, E), dim=1)
    n = C[e2c[:, 1]] - C[e2c[:, 0]]
    n = torch.nn.functional.normalize(n - (n * E).sum(1, keepdim=True) * E, dim=1)
    gen = _generator(seed, dev)
    vn = u * (east * n).sum(1)[:, None]
    vn += 0.01 * torch.randn(vn.shape, generator=gen, device=dev, dtype=torch.float64)
    w = 0.005 * torch.randn((C.shape[0], z.shape[-1]), generator=gen, device=dev, dtype=torch.float64)
    w[:, 0] = 0.0
    w[:, -1] = 0.0
    return dict(vn=vn, w=w, rho=rho.contiguous(), exner=exner.contiguous(), theta_v=theta.contiguous())


def _params(case, **more):
    prec = {"fp64": P.ICON_PREC_FP64, "mixed": P.ICON_PREC_MIXED, "f64col": P.ICON_PREC_MIXED_F64COL}[case["prec"]]
    return dict(dict(dtime=case["dt"], ndyn_substeps=case["ndyn"], rayleigh_coeff=case["rayleigh"],
                     damp_height=DAMP_HEIGHT, precision=prec, synchronous=0), **more)


def _learned_weights(nlev, seed):
    rng = np.random.default_rng(77 + seed)
    return [corrector.init_params(i, HIDDEN, o, rng) for i, o in (corrector.col_dims(nlev), corrector.edge_dims(nlev))]


def _increment_scales(nlev):
    """Size of the increments the trained corrector proposes: w, exner, theta_v; vn."""
    col = np.concatenate([np.full(nlev - 1, 1e-6), np.full(nlev, 1e-8), np.full(nlev, 1e-5)])
    return col.astype(np.float32), np.full(nlev, 1e-4, dtype=np.float32)


def _feature_stats(x, nlev):
    """Per-feature mean and standard deviation with a floor of 1e-3 of each field's largest."""
    mean, std = x.double().mean(0), x.double().std(0)
    floor = 1e-3 * std.reshape(-1, nlev).amax(1).repeat_interleave(nlev)
    return mean, torch.maximum(std, floor)


def _train_data(case, seed):
    i, o = (corrector.edge_dims if case["edge"] else corrector.col_dims)(case["nlev"])
    dev = _device()
    gen = _generator(seed, dev)
    rows = case["batch"] * case["steps"]
    x = torch.randn((rows, i), generator=gen, device=dev, dtype=torch.float32)
    mix = torch.randn((i, o), generator=gen, device=dev, dtype=torch.float32) / math.sqrt(i)
    y = torch.tanh(x.double() @ mix.double()).float()
    weights = corrector.init_params(i, HIDDEN, o, np.random.default_rng(11 + seed))
    return i, o, weights, x, y


def _column_inputs(case, seed):
    """Columns of the jet at random latitudes, tendencies and flux divergences of their usual size."""
    dev = _device()
    z = make_vct(case["nlev"])
    gen = _generator(seed, dev)
    n, nlev = case["cols"], case["nlev"]

    def noise(scale, *shape):
        return scale * torch.randn(shape, generator=gen, device=dev, dtype=torch.float64)

    zt = torch.from_numpy(z).to(dev)
    phi = torch.asin(2.0 * torch.rand((n, 1), generator=gen, device=dev, dtype=torch.float64) - 1.0)
    exner, theta, _ = _jet(phi, 0.5 * (zt[:-1] + zt[1:])[None, :])
    exner = (exner * (1.0 + noise(1e-5, n, nlev))).contiguous()
    theta = (theta * (1.0 + noise(1e-4, n, nlev))).contiguous()
    rho = (P00 * exner ** (CVD / RD) / (RD * theta)).contiguous()
    w, dw0, dw1 = noise(0.02, n, nlev + 1), noise(1e-5, n, nlev + 1), noise(1e-5, n, nlev + 1)
    for a in (w, dw0, dw1):
        a[:, 0] = 0.0
        a[:, -1] = 0.0
    div_m = noise(1e-6, n, nlev) * rho
    div_t = div_m * theta * (1.0 + noise(1e-2, n, nlev))
    f = dict(w=w, rho=rho, exner=exner, theta_v=theta, ddt_w0=dw0, div_m=div_m, div_t=div_t)
    if case["corr"]:
        f.update(ddt_w1=dw1, rho_pred=rho * (1.0 + noise(1e-5, n, nlev)),
                 theta_pred=theta * (1.0 + noise(1e-5, n, nlev)))
    return z, f


# ---------------------------------------------------------------------------
# a pass
# ---------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind == "train":
        i, o, weights, s["x"], s["y"] = _train_data(case, seed)
        s["net"] = P.MLP(i, HIDDEN, o, case["batch"])
        s["net"].set_params(weights)
        return s
    if kind == "column":
        s["z"], s["in"] = _column_inputs(case, seed)
        n, nlev = case["cols"], case["nlev"]
        s["out"] = dict(w_new=torch.empty((n, nlev + 1), device="cuda", dtype=torch.float64),
                        **{k: torch.empty((n, nlev), device="cuda", dtype=torch.float64)
                           for k in ("rho_new", "exner_new", "theta_new")})
        s["params"] = P.default_params(**_params(case))
        return s
    s["grid"] = P.Grid(_raw_grid(case["bis"]), radius=RADIUS)
    z = _heights(case)
    s["dycore"] = P.Dycore(s["grid"], z, _params(case))
    st = _state(case, seed)
    if case["terrain"]:
        ref = s["dycore"].reference_columns()[1]
    else:
        ref = s["dycore"].reference_state()[1][None, :]
    st["exner_pr"] = st["exner"] - torch.from_numpy(ref).to(st["exner"].device)
    if kind == "host":
        s["state"] = {k: torch.empty(v.shape, dtype=v.dtype, pin_memory=True).copy_(v).numpy() for k, v in st.items()}
    else:
        s["state"] = st
    if kind == "learned":
        nlev, g, d = case["nlev"], s["grid"], s["dycore"]
        s["reduced"] = P.Dycore(g, z, _params(case, **REDUCED))
        cx = torch.empty((g.n_cells, 5 * nlev), dtype=torch.float32, device="cuda")
        ex = torch.empty((g.n_edges, 11 * nlev), dtype=torch.float32, device="cuda")
        d.corrector_features(st, cx, ex)
        d.synchronize()
        for key, x, w, scale in zip(("col", "edge"), (cx, ex), _learned_weights(nlev, seed), _increment_scales(nlev)):
            dims = corrector.col_dims(nlev) if key == "col" else corrector.edge_dims(nlev)
            s[key] = P.MLP(dims[0], HIDDEN, dims[1], 65536)
            s[key].set_params(w)
            mean, std = (q.float().cpu().numpy() for q in _feature_stats(x, nlev))
            s[key].set_normalization(mean, std, np.zeros(dims[1], np.float32), scale)
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind in ("step", "host"):
        s["dycore"].step(s["state"])
        return s["state"]
    if kind == "solve":
        s["dycore"].nh_solve(s["state"])
        return s["state"]
    if kind == "diff":
        s["dycore"].nh_diff(s["state"])
        return s["state"]
    if kind == "learned":
        fallback, norm = P.step_learned(s["reduced"], s["dycore"], s["col"], s["edge"], s["state"], 3.0)
        return dict(s["state"], fallback=fallback, norm=norm)
    if kind == "column":
        P.column_solve_noalloc(s["z"], s["params"], **s["in"], **s["out"])
        return s["out"]
    b = case["batch"]
    losses = [s["net"].train_step(s["x"][i * b:(i + 1) * b], s["y"][i * b:(i + 1) * b], case["lr"])
              for i in range(case["steps"])]
    return dict(losses=losses, weights=s["net"].params())


def work(case):
    """Bytes: each input read once and each output written once.  Flops: the
    arithmetic of the scheme per cell and level (edges and vertices folded in)."""
    kind, nlev = case["kind"], case["nlev"]
    if kind == "train":
        i, o = (corrector.edge_dims if case["edge"] else corrector.col_dims)(nlev)
        n = HIDDEN * (i + HIDDEN + o)
        return dict(bytes=case["steps"] * (4.0 * case["batch"] * (i + o) + 24.0 * n),
                    flops=6.0 * n * case["batch"] * case["steps"])
    if kind == "column":
        n = case["cols"] * nlev
        return dict(bytes=8.0 * n * (14 if case["corr"] else 11), flops=84.0 * n)
    cells = 80 * 4 ** case["bis"] * nlev
    nbytes = 2 * 8.0 * cells * 6.5  # vn on 1.5 edges a cell, w and four cell fields, in and out
    if kind == "diff":
        return dict(bytes=2 * 8.0 * cells * 4.5, flops=130.0 * cells)
    if kind == "solve":
        return dict(bytes=nbytes, flops=520.0 * cells)
    if kind == "learned":
        nets = sum(2.0 * r * HIDDEN * (i + HIDDEN + o) for r, (i, o) in
                   ((cells // nlev, corrector.col_dims(nlev)), (1.5 * cells // nlev, corrector.edge_dims(nlev))))
        return dict(bytes=nbytes, flops=(3 * 520.0 + 130.0) * cells + nets)
    return dict(bytes=nbytes, flops=(520.0 * case["ndyn"] + 130.0) * cells)


# ---------------------------------------------------------------------------
# the same results in plain torch, 64 bits: the scheme written with gathers
# over whole fields, no code of the library
# ---------------------------------------------------------------------------
def _dot(a, b):
    return (a * b).sum(-1)


def _arc(p, q):
    return torch.atan2(torch.linalg.norm(torch.linalg.cross(p, q), dim=-1), _dot(p, q))


def _tri(p, q, r):
    p, q, r = torch.broadcast_tensors(p, q, r)
    return 2.0 * torch.atan2(_dot(p, torch.linalg.cross(q, r)).abs(), 1.0 + _dot(p, q) + _dot(q, r) + _dot(r, p))


def _unit(x):
    return x / torch.linalg.norm(x, dim=-1, keepdim=True)


def _tangent(v, x):
    return v - (v * x).sum(-1, keepdim=True) * x


class _Plain:
    """The dynamical core's step over (flat or terrain-following) heights."""

    def __init__(self, raw, z_ifc, dt, ndyn, rayleigh, exfac=1.0 / 3.0, divdamp=0.0025):
        dev = _device()

        def load(a):
            return torch.from_numpy(a).to(dev)

        V, C, E = load(raw.vert_xyz), load(raw.cell_xyz), load(raw.edge_xyz)
        self.C, self.E, self.V = C, E, V
        self.c2e, self.e2c = load(raw.c2e).long(), load(raw.e2c).long()
        e2v, c2v = load(raw.e2v).long(), load(raw.c2v).long()
        v2e, v2c = load(raw.v2e).long(), load(raw.v2c).long()
        on_e, on_c = v2e >= 0, v2c >= 0
        self.v2e, self.v2c = v2e.clamp(min=0), v2c.clamp(min=0)
        self.dt, self.ndyn, self.exfac, self.divdamp = dt, ndyn, exfac, divdamp
        nc, ne, a = C.shape[0], E.shape[0], RADIUS
        c0, c1 = self.e2c[:, 0], self.e2c[:, 1]
        self.c0, self.c1 = c0, c1
        self.area = a * a * _tri(V[c2v[:, 0]], V[c2v[:, 1]], V[c2v[:, 2]])
        self.l, self.d = a * _arc(V[e2v[:, 0]], V[e2v[:, 1]]), a * _arc(C[c0], C[c1])
        self.abar = self.area.mean()
        self.normal = _unit(_tangent(C[c1] - C[c0], E))
        self.tang = torch.linalg.cross(E, self.normal)
        me = torch.arange(nc, device=dev)[:, None]
        first = c0[self.c2e] == me
        self.sign = torch.where(first, 1.0, -1.0).double()
        self.nbr = torch.where(first, c1[self.c2e], c0[self.c2e])
        # vm -> vp along the tangent, and the vertices opposite the edge
        ahead = _dot(V[e2v[:, 1]] - V[e2v[:, 0]], self.tang) > 0
        self.vm, self.vp = torch.where(ahead, e2v[:, 0], e2v[:, 1]), torch.where(ahead, e2v[:, 1], e2v[:, 0])
        self.vo = [torch.where((c2v[c] != e2v[:, :1]) & (c2v[c] != e2v[:, 1:]), c2v[c], -1).amax(1) for c in (c0, c1)]
        self.dn = a * _arc(V[self.vo[0]], V[self.vo[1]])
        dual = torch.where(on_e, _tri(V[:, None, :], C[c0[self.v2e]], C[c1[self.v2e]]), 0.0).sum(1) * a * a
        turn = torch.where(_dot(V[:, None, :] - E[self.v2e], self.tang[self.v2e]) > 0, 1.0, -1.0)
        self.curl_w = torch.where(on_e, turn * self.d[self.v2e] / dual[:, None], 0.0)
        self.div_w = self.sign * self.l[self.c2e] / self.area[:, None]
        self.lap_w = (self.l / self.d)[self.c2e] / self.area[:, None]
        q = self.l[self.c2e] * _arc(C[:, None, :].expand(-1, 3, -1), E[self.c2e])
        self.q = q / q.sum(1, keepdim=True)
        kite = torch.zeros(v2c.shape, dtype=torch.float64, device=dev)
        for j in range(6):
            c = self.v2c[:, j]
            mine = c2v[c] == torch.arange(V.shape[0], device=dev)[:, None]
            far = torch.where(mine, -1, c2v[c]).sort(1).values[:, 1:]  # its two other vertices
            m1, m2 = _unit(V[far[:, 0]] + V), _unit(V[far[:, 1]] + V)
            kite[:, j] = torch.where(on_c[:, j], _tri(V, m1, C[c]) + _tri(V, C[c], m2), 0.0)
        self.kite = kite / kite.sum(1, keepdim=True)
        r0, r1 = _arc(C[c0], E), _arc(C[c1], E)
        w_other = torch.stack([r0 / (r0 + r1), r1 / (r0 + r1)], 1)  # weight of the other cell, seen from c0, c1
        self.w_nbr = torch.where(first, w_other[self.c2e, 0], w_other[self.c2e, 1])
        dx = _tangent(a * (E[self.c2e] - C[:, None, :]), C[:, None, :])
        self.perot_w = self.div_w[..., None] * dx
        self.grad_w = _tangent((self.div_w * self.w_nbr)[..., None] * self.normal[self.c2e], C[:, None, :])
        mid = _unit(C[c0] + C[c1])
        arm = _tangent(a * (mid[self.v2e] - V[:, None, :]), V[:, None, :])
        self.uv_w = torch.linalg.cross(V[:, None, :].expand_as(arm), self.curl_w[..., None] * arm)
        self.f = 2.0 * OMEGA * E[:, 2:3]
        # vertical metrics and reference state, one row per column (one row over flat ground)
        z = torch.from_numpy(np.atleast_2d(z_ifc)).to(dev)
        self.terrain, self.nlev = z.shape[0] > 1, z.shape[1] - 1
        nlev = self.nlev
        zm = 0.5 * (z[:, :-1] + z[:, 1:])
        self.zm, self.dz, self.dzh = zm, z[:, :-1] - z[:, 1:], zm[:, :-1] - zm[:, 1:]
        self.wg = (z[:, 1:-1] - zm[:, 1:]) / self.dzh
        self.th_ref = T0 * torch.exp(zm / H)
        ref = [torch.exp(-zm[:, -1] / H)]
        th_ic = self.wg * self.th_ref[:, :-1] + (1.0 - self.wg) * self.th_ref[:, 1:]
        for k in range(nlev - 1, 0, -1):
            ref.append(ref[-1] - GRAV * self.dzh[:, k - 1] / (CPD * th_ic[:, k - 1]))
        self.ex_ref = torch.stack(ref[::-1], 1)
        self.dref = (self.ex_ref[:, :-1] - self.ex_ref[:, 1:]) / self.dzh
        damp = torch.sin(0.5 * math.pi * (z - DAMP_HEIGHT) / (z[:, :1] - DAMP_HEIGHT)) ** 2
        self.ray = 1.0 + dt / ndyn * rayleigh * torch.where(z > DAMP_HEIGHT, damp, 0.0)
        if self.terrain:
            ze = 0.5 * (z[c0] + z[c1])
            zem = 0.5 * (ze[:, :-1] + ze[:, 1:])
            self.dz_e = ze[:, :-1] - ze[:, 1:]
            self.wg_e = (ze[:, 1:-1] - zem[:, 1:]) / (zem[:, :-1] - zem[:, 1:])
            self.sn, self.sn_m = (z[c1] - z[c0]) / self.d[:, None], (zm[c1] - zm[c0]) / self.d[:, None]
            zv = z[self.v2c[:, 0]].clone()
            for j in range(6):
                zv += self.kite[:, j:j + 1] * (z[self.v2c[:, j]] - z[self.v2c[:, 0]])
            self.st = self.grad_t(zv)
        else:
            self.dz_e, self.wg_e = self.dz, self.wg

    def gather(self, w, idx, X):
        return sum(w[:, j:j + 1] * X[idx[:, j]] for j in range(idx.shape[1]))

    def div(self, F):
        return self.gather(self.div_w, self.c2e, F)

    def curl(self, F):
        return self.gather(self.curl_w, self.v2e, F)

    def grad_n(self, X):
        return (X[self.c1] - X[self.c0]) / self.d[:, None]

    def grad_t(self, Y):
        return (Y[self.vp] - Y[self.vm]) / self.l[:, None]

    def lap_cell(self, X):
        return sum(self.lap_w[:, j:j + 1] * (X[self.nbr[:, j]] - X) for j in range(3))

    def lap_vec(self, F):
        return self.grad_n(self.div(F)) - self.grad_t(self.curl(F))

    def vectors(self, w, idx, F):
        """Three components of sum_j w_j F_j."""
        return [self.gather(w[..., i], idx, F) for i in range(3)]

    @staticmethod
    def half(wg, X, ends):
        mid = wg * X[:, :-1] + (1.0 - wg) * X[:, 1:]
        a, b = (X[:, :1], X[:, -1:]) if ends else (torch.zeros_like(X[:, :1]),) * 2
        return torch.cat([a, mid, b], 1)

    def tangential(self, vn):
        u = self.vectors(self.perot_w, self.c2e, vn)
        return 0.5 * sum((u[i][self.c0] + u[i][self.c1]) * self.tang[:, i:i + 1] for i in range(3))

    def advection(self, vn, w):
        vt = self.tangential(vn)
        vn_i, vt_i = self.half(self.wg_e, vn, True), self.half(self.wg_e, vt, True)
        wcc = self.gather(self.q, self.c2e, vn_i * self.sn + vt_i * self.st) if self.terrain else torch.zeros_like(w)
        wc = w - wcc
        ke = self.gather(self.q, self.c2e, 0.5 * (vn * vn + vt * vt))
        wf, wcf = 0.5 * (w[:, :-1] + w[:, 1:]), 0.5 * (wc[:, :-1] + wc[:, 1:])
        zeta, wv = self.curl(vn), self.gather(self.kite, self.v2c, w)
        ddt_vn = (-self.grad_n(ke) + (0.5 * (zeta[self.vm] + zeta[self.vp]) + self.f) * vt
                  - 0.5 * (wcf[self.c0] + wcf[self.c1]) * (vn_i[:, :-1] - vn_i[:, 1:]) / self.dz_e)
        adv = self.gather(self.q, self.c2e, vn_i * self.grad_n(w) + vt_i * self.grad_t(wv))
        ddt_w = torch.zeros_like(w)
        ddt_w[:, 1:-1] = -adv[:, 1:-1] - wc[:, 1:-1] * (wf[:, :-1] - wf[:, 1:]) / self.dzh
        return ddt_vn, ddt_w, vt, wcc

    def upwind(self, X, vn, vt, dt):
        g = [sum(self.grad_w[:, j, i:i + 1] * (X[self.nbr[:, j]] - X) for j in range(3)) for i in range(3)]
        out = []
        for c in (self.c0, self.c1):
            at = RADIUS * (self.E - self.C[c])
            out.append(X[c] + sum(g[i][c] * (at[:, i:i + 1] - 0.5 * dt * (vn * self.normal[:, i:i + 1] +
                                                                            vt * self.tang[:, i:i + 1]))
                                  for i in range(3)))
        return torch.where(vn >= 0.0, out[0], out[1])

    def column(self, st, rho_m, th_m, div_m, div_t, ddt_w, dt, wcc, beta=0.65):
        """The vertically implicit solve; rho_m, th_m: full levels that the half levels come from."""
        rho, exner, theta, w, nlev = st["rho"], st["exner"], st["theta_v"], st["w"], self.nlev
        pr = exner - self.ex_ref
        zb = dt * (RD / CVD) * exner / (rho * theta * self.dz)
        ri = self.half(self.wg, rho_m, False)
        ti, tp = self.half(self.wg, th_m, False), self.half(self.wg, th_m - self.th_ref, False)
        rt = ri * ti
        wc = w - wcc
        wc[:, 0] = 0.0
        wc[:, -1] = 0.0

        def drop(F):
            return F[:, :-1] - F[:, 1:]

        rs = rho - dt * div_m - dt * (1.0 - beta) * drop(ri * wc) / self.dz
        ps = pr - zb * (self.dz * div_t + (1.0 - beta) * drop(rt * wc))
        al = beta * rt
        gam = dt * CPD * beta * ti[:, 1:-1] / self.dzh
        r = (w + dt * ddt_w - wcc)[:, 1:-1] - dt * CPD * ((1.0 - beta) * ti[:, 1:-1] * drop(pr) / self.dzh
                                                       + tp[:, 1:-1] * self.dref) - gam * drop(ps)
        a = (-gam * zb[:, :-1] * al[:, :-2]).T.contiguous()
        b = (1.0 + gam * al[:, 1:-1] * (zb[:, :-1] + zb[:, 1:])).T.contiguous()
        c = (-gam * zb[:, 1:] * al[:, 2:]).T.contiguous()
        r = r.T.contiguous()
        n = nlev - 1
        for k in range(1, n):
            m = a[k] / b[k - 1]
            b[k] -= m * c[k - 1]
            r[k] -= m * r[k - 1]
        r[n - 1] /= b[n - 1]
        for k in range(n - 2, -1, -1):
            r[k] = (r[k] - c[k] * r[k + 1]) / b[k]
        new = torch.zeros_like(w)
        new[:, 1:-1] = r.T
        new = new / self.ray
        rho_n = rs - dt * beta * drop(ri * new) / self.dz
        pr_n = ps - zb * drop(al * new)
        th_n = theta * (rho / rho_n) * (1.0 + (CVD / RD) * (pr_n - pr) / exner)
        return dict(w=new + wcc, rho=rho_n, exner=self.ex_ref + pr_n, theta_v=th_n)

    def fluxes(self, vn, rho_e, th_e):
        vf = vn + 0.07 * self.abar * self.grad_n(self.div(vn))
        F = rho_e * vf * self.dz_e
        return self.div(F) / self.dz, self.div(F * th_e) / self.dz

    def substep(self, st):
        dt = self.dt / self.ndyn
        vn, w, rho, theta = st["vn"], st["w"], st["rho"], st["theta_v"]
        dv0, dw0, vt, wcc0 = self.advection(vn, w)
        pr = st["exner"] - self.ex_ref
        pex = (1.0 + self.exfac) * pr - self.exfac * st["exner_pr"]
        rho_e, th_e = self.upwind(rho, vn, vt, dt), self.upwind(theta, vn, vt, dt)
        grad = self.grad_n(pex)
        if self.terrain:
            up, dn = torch.cat([pex[:, :1], pex[:, :-1]], 1), torch.cat([pex[:, 1:], pex[:, -1:]], 1)
            zu, zd = torch.cat([self.zm[:, :1], self.zm[:, :-1]], 1), torch.cat([self.zm[:, 1:], self.zm[:, -1:]], 1)
            slope = (up - dn) / (zu - zd)
            grad = grad - self.sn_m * 0.5 * (slope[self.c0] + slope[self.c1])
        hpg = CPD * th_e * grad
        vp = vn + dt * (dv0 - hpg)
        pred = self.column(st, rho, theta, *self.fluxes(vp, rho_e, th_e), dw0, dt, wcc0)
        dv1, dw1, _, wcc1 = self.advection(vp, pred["w"])
        vnew = (vn + dt * (0.25 * dv0 + 0.75 * dv1 - hpg)
                - self.divdamp * self.abar ** 2 * self.grad_n(self.lap_cell(self.div(vp))))
        new = self.column(st, 0.6 * rho + 0.4 * pred["rho"], 0.6 * theta + 0.4 * pred["theta_v"],
                          *self.fluxes(vnew, rho_e, th_e), 0.25 * dw0 + 0.75 * dw1, dt, wcc1)
        return dict(new, vn=vnew, exner_pr=pr)

    def diffusion(self, st):
        vn, w, theta, exner, dt = st["vn"], st["w"], st["theta_v"], st["exner"], self.dt
        uv = self.vectors(self.uv_w, self.v2e, vn)
        n, t = self.normal, self.tang
        along = [u[self.vp] - u[self.vm] for u in uv]
        across = [u[self.vo[1]] - u[self.vo[0]] for u in uv]

        def on(axis, du):
            return sum(axis[:, i:i + 1] * du[i] for i in range(3))

        l, dn = self.l[:, None], self.dn[:, None]
        tension = on(n, across) / dn - on(t, along) / l
        shear = on(n, along) / l + on(t, across) / dn
        edge_area = (self.l * self.d)[:, None]
        nu = 0.015 * edge_area * torch.sqrt(tension ** 2 + shear ** 2)
        lap = self.lap_vec(vn)
        w_new = w - (self.area ** 2)[:, None] / 288.0 * self.lap_cell(self.lap_cell(w))
        w_new[:, 0] = 0.0
        w_new[:, -1] = w[:, -1] if self.terrain else 0.0
        th = theta + dt * sum(self.lap_w[:, j:j + 1] * nu[self.c2e[:, j]] * (theta[self.nbr[:, j]] - theta)
                              for j in range(3))
        return dict(st, vn=vn + dt * nu * lap - edge_area ** 2 / 288.0 * self.lap_vec(lap), w=w_new, theta_v=th,
                    exner=exner * (1.0 + (RD / CVD) * (th - theta) / theta))

    def step(self, st):
        for _ in range(self.ndyn):
            st = self.substep(st)
        return self.diffusion(st)

    def features(self, st):
        up = torch.tensor([0.0, 0.0, 1.0], dtype=torch.float64, device=self.C.device).expand_as(self.C)
        east = _unit(torch.linalg.cross(up, self.C))
        north = torch.linalg.cross(self.C, east)
        u = self.vectors(self.perot_w, self.c2e, st["vn"])
        col = torch.cat([0.5 * (st["w"][:, :-1] + st["w"][:, 1:]), st["exner"] - self.ex_ref, st["theta_v"] - self.th_ref]
                        + [sum(u[i] * a[:, i:i + 1] for i in range(3)) for a in (east, north)], 1)
        return col, lambda r: torch.cat([col[self.c0[r]], col[self.c1[r]], st["vn"][r]], 1)


def _split(weights, i, o):
    shapes = [(HIDDEN, i), (HIDDEN,), (HIDDEN, HIDDEN), (HIDDEN,), (o, HIDDEN), (o,)]
    at, out = 0, []
    p = torch.from_numpy(weights).to(_device()).double()
    for sh in shapes:
        n = math.prod(sh)
        out.append(p[at:at + n].reshape(sh))
        at += n
    return out


def _mlp(p, x):
    g = torch.nn.functional.gelu
    return g(g(x @ p[0].T + p[1]) @ p[2].T + p[3]) @ p[4].T + p[5]


def _exact_learned(case, seed, st):
    nlev = case["nlev"]
    raw, z = _raw_grid(case["bis"]), _heights(case)
    more = dict(exfac=REDUCED["exner_exfac"], divdamp=REDUCED["divdamp_fac"])
    core = _Plain(raw, z, case["dt"], REDUCED["ndyn_substeps"], case["rayleigh"], **more)
    st["exner_pr"] = st["exner"] - core.ex_ref
    rows = torch.arange(raw.n_edges, device=core.C.device)
    col, edge = core.features(st)
    stats = [_feature_stats(col, nlev), _feature_stats(edge(rows), nlev)]
    st = core.step(st)
    col, edge = core.features(st)
    wc, we = _learned_weights(nlev, seed)
    sc, se = (torch.from_numpy(q).to(rows.device).double() for q in _increment_scales(nlev))
    pc, pe = _split(wc, *corrector.col_dims(nlev)), _split(we, *corrector.edge_dims(nlev))
    yc = _mlp(pc, (col - stats[0][0]) / stats[0][1])
    ye = torch.cat([_mlp(pe, (edge(r) - stats[1][0]) / stats[1][1]) for r in rows.split(65536)])
    inc = yc * sc
    st["w"][:, 1:-1] += inc[:, :nlev - 1]
    st["exner"] = st["exner"] + inc[:, nlev - 1:2 * nlev - 1]
    st["theta_v"] = st["theta_v"] + inc[:, 2 * nlev - 1:]
    st["vn"] = st["vn"] + ye * se
    norm = max(float(yc.square().mean().sqrt()), float(ye.square().mean().sqrt()))
    return dict(st, fallback=False, norm=norm)


def _exact_train(case, seed):
    i, o, weights, x, y = _train_data(case, seed)
    p = [q.clone().requires_grad_(True) for q in _split(weights, i, o)]
    m, v, losses = [torch.zeros_like(q) for q in p], [torch.zeros_like(q) for q in p], []
    for k in range(case["steps"]):
        rows = slice(k * case["batch"], (k + 1) * case["batch"])
        loss = (_mlp(p, x[rows].double()) - y[rows].double()).square().mean()
        losses.append(float(loss.detach()))
        grads = torch.autograd.grad(loss, p)
        with torch.no_grad():
            for q, g, a, b in zip(p, grads, m, v):
                a.mul_(0.9).add_(0.1 * g)
                b.mul_(0.999).add_(0.001 * g * g)
                q -= case["lr"] * (a / (1 - 0.9 ** (k + 1))) / ((b / (1 - 0.999 ** (k + 1))).sqrt() + 1e-8)
    return dict(losses=losses, weights=torch.cat([q.detach().reshape(-1) for q in p]))


def _exact_column(case, seed):
    z, f = _column_inputs(case, seed)
    core = _Plain(_raw_grid(0), z, case["dt"], case["ndyn"], case["rayleigh"])  # for its vertical metrics
    rho, theta, ddt_w = f["rho"], f["theta_v"], f["ddt_w0"]
    if case["corr"]:
        rho, theta = 0.6 * rho + 0.4 * f["rho_pred"], 0.6 * theta + 0.4 * f["theta_pred"]
        ddt_w = 0.25 * ddt_w + 0.75 * f["ddt_w1"]
    out = core.column(f, rho, theta, f["div_m"], f["div_t"], ddt_w, case["dt"] / case["ndyn"],
                      torch.zeros_like(f["w"]))
    return dict(w_new=out["w"], rho_new=out["rho"], exner_new=out["exner"], theta_new=out["theta_v"])


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "column":
        return _exact_column(case, seed)
    st = _state(case, seed)
    if kind == "learned":
        return _exact_learned(case, seed, st)
    core = _Plain(_raw_grid(case["bis"]), _heights(case), case["dt"], case["ndyn"], case["rayleigh"])
    st["exner_pr"] = st["exner"] - core.ex_ref
    out = {"solve": core.substep, "diff": core.diffusion}.get(kind, core.step)(st)
    return {k: out[k] for k in FIELDS}
