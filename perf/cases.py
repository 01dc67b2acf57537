"""The work that a user of this library has it do, as cases that can be timed and compared.

A model run alternates segments of dynamical-core steps with output: every pass advances
states that stay on the GPU by a number of steps through the public entry points, checks the
status, takes the air-mass integral and reads the whole prognostic state (and tracers) back
into host memory, as a forecast does at its output times. listed() spans the range from the
smallest grids, where launches and latency count, to the largest state of which three fit the
GPU, in both precisions, on flat and terrain-following levels, with tracers and options, alone,
as a batched ensemble and as a decomposed domain; draw() gives more of the same ranges.
exact() restates the method in plain torch FP64 from the grid's tables.
"""
import math

import numpy as np
import torch

from paper_2511_02021_gb300 import bind_torch_stream, capi as C, use_torch_allocator

FIELDS = ("vn", "w", "rho", "theta_v", "exner")
TOPO_RADIUS_M = 8.0e5          # the benchmark's mountain: 1500 m high, 800 km e-folding radius
NSUB = 5


def _case(bisections, nlev, precision, steps, **more):
    c = {"bisections": bisections, "nlev": nlev, "precision": precision, "steps": steps, "noise_K": 0.1,
         "topo_m": 0.0, "tracers": 0, "diff4": 0.0, "upwind": False, "members": 0, "coarse_members": 0, "parts": 0}
    c.update(more)
    return c


def listed():
    def named(name, *a, **k):
        return dict(_case(*a, **k), name=name)
    return [
        # the smallest configuration of the repository's workload table, stepped one step at a
        # time as a coupled model would: launches and the host's waits
        named("fp64 R2B2/20 one step", 2, 20, "fp64", 1, noise_K=0.01),
        # a coarse member run alone: the small grids of the ensemble workload
        named("mixed R2B4/60", 4, 60, "mixed", 4),
        # the headline workload, every operation FP64
        named("fp64 R2B6/90", 6, 90, "fp64", 2),
        # the headline grid in the production precision
        named("mixed R2B6/90", 6, 90, "mixed", 8),
        # the largest state of which three fit the GPU
        named("mixed R2B7/90", 7, 90, "mixed", 4),
        # terrain-following levels over the benchmark's mountain, both precisions
        named("fp64 R2B5/90 mountain", 5, 90, "fp64", 2, topo_m=1500.0),
        named("mixed R2B5/90 mountain", 5, 90, "mixed", 8, topo_m=1500.0),
        # moist run: water vapour and cloud water transported with the step's fluxes
        named("fp64 R2B5/60 two tracers", 5, 60, "fp64", 12, tracers=2),
        # every step option at a level count that fills no tile
        named("mixed R2B5/47 options", 5, 47, "mixed", 8, diff4=0.002, upwind=True),
        # the batched ensemble workload: 32 members on R2B4 and 32 on R2B5 in one launch per step
        named("ensemble 32 R2B4 + 32 R2B5 /60", 5, 60, "mixed", 2, members=32, coarse_members=32, noise_K=0.0),
        # the step of a horizontally decomposed run, its four parts on this GPU
        named("fp64 R2B5/60 four parts", 5, 60, "fp64", 4, parts=4),
    ]


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "ensemble", "parts"])
    if kind == "ensemble":
        # up to the listed ensemble's cells and levels
        return _case(rng.randint(3, 5), rng.randint(20, 64), "mixed", rng.randint(1, 2), noise_K=0.0,
                     members=rng.randint(2, 32), coarse_members=rng.randint(0, 32))
    if kind == "parts":
        return _case(rng.randint(3, 5), rng.randint(20, 96), "fp64", rng.randint(1, 2), parts=rng.randint(2, 6))
    precision = rng.choice(["fp64", "mixed"])
    bisections = rng.randint(2, 6 if precision == "fp64" else 7)
    nlev = rng.randint(20, 90 if bisections == 7 else 128)
    topo = rng.choice([0.0, 0.0, round(rng.uniform(200.0, 1800.0), 1)]) if bisections < 6 else 0.0
    return _case(bisections, nlev, precision, rng.randint(1, 2 if precision == "fp64" else 4), topo_m=topo,
                 tracers=rng.choice([0, 0, 1, 2]) if bisections < 6 else 0,
                 diff4=rng.choice([0.0, 0.0, 0.002]), upwind=rng.random() < 0.25)


def _dt(bisections):
    """The repository's time steps: 90 s on R2B6, halved per bisection, at most 360 s."""
    return 300.0 if bisections < 4 else 5760.0 / 2 ** bisections


class _Model:
    """Handles and output buffers of one run; freed with the object."""

    def __init__(self):
        self.grids, self.states, self.ensemble, self.domain = [], [], None, None

    def __del__(self):
        if self.ensemble is not None:
            C.icon_ensemble_free(self.ensemble)
        if self.domain is not None:
            C.icon_domain_free(self.domain)
        for s in self.states:
            C.icon_state_free(s)
        for g in self.grids:
            C.icon_grid_free(g)


_bound = []


def _pinned(*shape):
    return torch.empty(shape, dtype=torch.float64, pin_memory=True)


def _field_buffers(grid, nlev, lead=()):
    nc, ne, _ = C.icon_grid_counts(grid)
    return {f: _pinned(*lead, ne if f == "vn" else nc, nlev + 1 if f == "w" else nlev) for f in FIELDS}


def prepare(case, seed):
    if not _bound:
        use_torch_allocator(0)
        _bound.append(True)
    bind_torch_stream()
    m = _Model()
    m.case = case
    nlev = case["nlev"]
    precision = C.ICON_MIXED if case["precision"] == "mixed" else C.ICON_FP64
    # (grid level, states on it, how the state starts)
    groups = [(case["bisections"], case["members"] or 1)]
    if case["coarse_members"]:
        groups.append((case["bisections"] - 1, case["coarse_members"]))
    m.groups = []
    dts = []
    for bis, count in groups:
        grid = C.icon_grid_build(2, bis, nlev)
        m.grids.append(grid)
        states = []
        for i in range(count):
            states.append(C.icon_state_init_ex(
                grid, seed, C.ICON_CASE_MEMBER if case["members"] else C.ICON_CASE_JET, noise_K=case["noise_K"],
                precision=precision, member=i, topo_height_m=case["topo_m"],
                topo_radius_m=TOPO_RADIUS_M if case["topo_m"] else 0.0))
            m.states.append(states[-1])
            dts.append(_dt(bis))
        m.groups.append((grid, states, _field_buffers(grid, nlev, (count,) if case["members"] else ())))
    m.dts = dts
    st = m.states[0]
    if case["diff4"]:
        C.icon_state_set_option(st, C.ICON_OPT_DIFF4, case["diff4"])
    if case["upwind"]:
        C.icon_state_set_option(st, C.ICON_OPT_UPWIND_THETA, 1.0)
    if case["tracers"]:
        C.icon_state_add_tracers(st, case["tracers"])
        x = C.icon_grid_copy_table(m.grids[0], "x_c")
        rng = np.random.default_rng(seed)
        height = np.linspace(0.0, 1.0, nlev) ** 4
        for t in range(case["tracers"]):
            # a mixing ratio that falls with height and varies smoothly over the sphere
            a = rng.normal(size=3)
            C.icon_state_set_tracer(st, m.grids[0], nlev, t,
                                    0.01 * height[None, :] * (1.5 + np.sin(2.0 * (x @ a)))[:, None])
    if case["members"]:
        m.ensemble = C.icon_ensemble_create(m.states)
    if case["parts"]:
        m.domain = C.icon_domain_create(st, case["parts"], 3)
    return m


def run(m):
    case, nlev = m.case, m.case["nlev"]
    out = {}
    if m.ensemble is not None:
        C.icon_ensemble_step(m.ensemble, m.dts, NSUB, case["steps"])
        for i, (grid, states, buf) in enumerate(m.groups):
            out["mass%d" % i] = [C.icon_global_mass(s) for s in states][0]
            for f, b in buf.items():
                v = b.numpy()
                for j, s in enumerate(states):
                    C.icon_state_copy_field(s, grid, nlev, f, out=v[j])
                out["%s%d" % (f, i)] = b
        return out
    grid, (st,), buf = m.groups[0]
    if m.domain is not None:
        for _ in range(case["steps"]):
            C.icon_domain_step(m.domain, m.dts[0], NSUB)
        out["mass"] = C.icon_domain_global_mass(m.domain)
        for f in FIELDS:
            out[f] = C.icon_domain_copy_field(m.domain, grid, nlev, f)
        return out
    if case["steps"] == 1:
        C.icon_dycore_step(st, m.dts[0], NSUB)
    else:
        for _ in range(case["steps"]):
            C.icon_dycore_step_async(st, m.dts[0], NSUB)
        C.icon_state_status(st)
    out["mass"] = C.icon_global_mass(st)
    for f, b in buf.items():
        C.icon_state_copy_field(st, grid, nlev, f, out=b.numpy())
        out[f] = b
    for t in range(case["tracers"]):
        out["q%d" % t] = C.icon_state_copy_tracer(st, grid, nlev, t)
    return out


def _groups(case):
    got = [(case["bisections"], case["members"] or 1)]
    if case["coarse_members"]:
        got.append((case["bisections"] - 1, case["coarse_members"]))
    return got


def work(case):
    """A substep depends on the whole state of the one before: the prognostic state (vn on 1.5
    edges per cell; w, rho, theta_v, exner) is read and written once per substep, and the output
    once per pass. Operations: the multiplications, additions and divisions of the method's
    expressions per cell and level (predictor and corrector with damping 2 x 230, once per step
    100 in the diffusion, 110 per tracer, the terrain's metric terms 2 x 60 per substep)."""
    cells = sum(20 * 4 ** (b + 1) * n for b, n in _groups(case)) * case["nlev"]
    word = 8.0 if case["precision"] == "fp64" else 6.9       # mixed: vn in 32 bits
    steps = case["steps"]
    state = 5.5 * word
    tr = case["tracers"]
    byts = cells * (steps * (NSUB * 2 * state + 16.0 * tr) + 5.5 * 8 + 8.0 * tr)
    per_step = NSUB * (460 + (120 if case["topo_m"] else 0)) + 100 + 110 * tr + (40 if case["diff4"] else 0)
    return {"bytes": byts, "flops": float(cells * steps * per_step)}


# ---------------------------------------------------------------- the method in plain torch FP64
# Full level k = 0..N-1 top to bottom, half level h = 0..N; fields [entity, level]. Flat levels
# are terrain-following ones over no topography.
RADIUS, GRAV, RD, CPD, BETA = 6.371229e6, 9.80665, 287.04, 1004.64, 0.65
CVD = CPD - RD


class _Exact:
    def __init__(self, grid, nlev, topo_m):
        names = ("c2e", "e2c", "e2v", "v2e", "v2c", "vdeg", "e2vt", "e2q", "x_c", "n_e", "t_e", "l_e", "d_e", "A_c",
                 "A_v", "f_e", "vt_w", "kin_w", "lsq_w", "L34", "s_ce", "s_ve")
        for n in names:
            a = torch.from_numpy(C.icon_grid_copy_table(grid, n)).cuda()
            setattr(self, n, a.long() if a.dtype == torch.int32 else a)
        self.c1, self.c2 = self.e2c[:, 0], self.e2c[:, 1]
        self.v1, self.v2 = self.e2v[:, 0], self.e2v[:, 1]
        self.ide, self.ile = 1.0 / self.d_e[:, None], 1.0 / self.l_e[:, None]
        self.nc, N = self.A_c.shape[0], nlev
        self.N = N
        top, s, damp = (75000.0, 5.5, 45000.0) if N >= 60 else (30000.0, 2.0, 20000.0)
        zh = top * (np.exp(s * (N - np.arange(N + 1.0)) / N) - 1.0) / (np.exp(s) - 1.0)
        zh[0], zh[N] = top, 0.0
        self.ray = torch.from_numpy(np.where(zh > damp, 0.05 * np.sin(0.5 * np.pi * (zh - damp) / (top - damp)) ** 2,
                                             0.0)).cuda()
        b = np.sinh((top - zh) / 4000.0) / np.sinh(top / 4000.0)
        self.zh, self.b = torch.from_numpy(zh).cuda(), torch.from_numpy(b).cuda()
        self.bf = 0.5 * (self.b[:-1] + self.b[1:])
        self.topo = topo_m > 0.0
        if self.topo:
            lon, lat = math.radians(90.0), math.radians(30.0)
            xm = torch.tensor([math.cos(lat) * math.cos(lon), math.cos(lat) * math.sin(lon), math.sin(lat)],
                              dtype=torch.float64, device="cuda")
            r = RADIUS * torch.atan2(torch.linalg.cross(self.x_c, xm.expand_as(self.x_c)).norm(dim=1), self.x_c @ xm)
            hs = topo_m * torch.exp(-(r / TOPO_RADIUS_M) ** 2)
            hv = self.vertex_mean(hs[:, None])[:, 0]
            self.sn = ((hs[self.c2] - hs[self.c1]) / self.d_e)[:, None]
            self.st = ((hv[self.v2] - hv[self.v1]) / self.l_e)[:, None]
        else:
            hs = torch.zeros(1, dtype=torch.float64, device="cuda")
        self.zhc, self.zfc, self.dz, self.dzh, self.wu = self.column_levels(hs)
        he = 0.5 * (hs[self.c1] + hs[self.c2]) if self.topo else hs
        _, _, self.dze, _, self.wue = self.column_levels(he)
        self.exref = torch.exp(-GRAV * self.zfc / (CPD * 250.0))

    def column_levels(self, hs):
        hs = hs[:, None]
        zh = self.zh + hs * self.b
        zf = 0.5 * (zh[:, :-1] + zh[:, 1:])
        dz = (self.zh[:-1] - self.zh[1:]) + hs * (self.b[:-1] - self.b[1:])
        zff = 0.5 * (self.zh[:-1] + self.zh[1:])
        dzh = (zff[:-1] - zff[1:]) + hs * (self.bf[:-1] - self.bf[1:])        # half levels 1..N-1
        return zh, zf, dz, dzh, dz[:, 1:] / (dz[:, :-1] + dz[:, 1:])

    def half(self, wu, f):
        return torch.cat([f[:, :1], wu * f[:, :-1] + (1.0 - wu) * f[:, 1:], f[:, -1:]], 1)

    def vertex_mean(self, f):
        s = sum(f[self.v2c[:, j]] for j in range(5))
        return (s + torch.where((self.vdeg == 6)[:, None], f[self.v2c[:, 5]], 0.0)) / self.vdeg[:, None]

    def div(self, u):
        return sum((self.s_ce[:, s] * self.l_e[self.c2e[:, s]])[:, None] * u[self.c2e[:, s]]
                   for s in range(3)) / self.A_c[:, None]

    def grad(self, f):
        return (f[self.c2] - f[self.c1]) * self.ide

    def curl(self, u):
        return sum((self.s_ve[:, j] * self.d_e[self.v2e[:, j]])[:, None] * u[self.v2e[:, j]]
                   for j in range(6)) / self.A_v[:, None]

    def tangential(self, u):
        return sum(self.vt_w[:, j:j + 1] * u[self.e2vt[:, j]] for j in range(5))

    def kappa(self, f):
        return sum(self.kin_w[:, s:s + 1] * f[self.c2e[:, s]] for s in range(3))

    def mean(self, f):
        return 0.5 * (f[self.c1] + f[self.c2])

    def tendencies(self, vn, w):
        """A_vn, A_w (interior half levels) and the contravariant correction wcc (0 on flat ground)."""
        N = self.N
        zeta, vt = self.curl(vn), self.tangential(vn)
        K = self.kappa(0.5 * (vn * vn + vt * vt))
        vh, th = self.half(self.wue, vn), self.half(self.wue, vt)
        wcc = torch.zeros_like(w)
        if self.topo:
            X = self.kappa(vn * (self.sn * self.bf) + vt * (self.st * self.bf))
            wcc[:, 1:N] = self.half(self.wu, X)[:, 1:N]
            wcc[:, N:] = self.kappa(vn[:, -1:] * self.sn + vt[:, -1:] * self.st)
        wcon = w - wcc
        wcon[:, 0] = 0.0
        wcon[:, N] = 0.0
        we = self.mean(wcon)
        A = (-self.grad(K) + (self.mean_v(zeta) + self.f_e[:, None]) * vt
             - 0.5 * (we[:, :N] + we[:, 1:]) * (vh[:, :N] - vh[:, 1:]) / self.dze)
        wv = self.vertex_mean(w)
        h = self.kappa(vh * self.grad(w) + th * ((wv[self.v2] - wv[self.v1]) * self.ile))
        Aw = -h[:, 1:N] - wcon[:, 1:N] * (w[:, :N - 1] - w[:, 2:]) / (self.zhc[:, :N - 1] - self.zhc[:, 2:])
        return A, Aw, wcc

    def mean_v(self, f):
        return 0.5 * (f[self.v1] + f[self.v2])

    def pressure_gradient(self, s):
        ex = s["exner"]
        if not self.topo:
            return CPD * self.mean(s["theta_v"]) * self.grad(ex)
        ep = ex - self.exref
        fi = self.half(self.wu, ep)
        d = (fi[:, :-1] - fi[:, 1:]) / self.dz
        d[:, 0] = (ep[:, 0] - ep[:, 1]) / self.dzh[:, 0]
        d[:, -1] = (ep[:, -2] - ep[:, -1]) / self.dzh[:, -1]
        return CPD * self.mean(s["theta_v"]) * (self.grad(ep) - self.sn * self.bf * self.mean(d))

    def column(self, s, F, G, Aw, wcc, dtau):
        N = self.N
        rho, thv, ex, w = s["rho"], s["theta_v"], s["exner"], s["w"]
        Th = rho * thv
        ri, ti = self.half(self.wu, rho), self.half(self.wu, thv)
        M = ri * ti
        ve = (1.0 - BETA) * w - wcc
        ve[:, 0] = 0.0
        ve[:, N] = 0.0
        thick = self.dz if self.topo else 1.0
        vert = lambda f: (f[:, :N] - f[:, 1:]) / self.dz  # noqa: E731
        rx = rho - dtau * (self.div(F) / thick + vert(ri * ve))
        tx = Th - dtau * (self.div(G) / thick + vert(M * ve))
        g = (RD / CVD) * ex / Th
        px = ex + g * (tx - Th)
        gam = g * (dtau * BETA) / self.dz
        wx = w[:, 1:N] + dtau * (Aw - (1.0 - BETA) * CPD * ti[:, 1:N] * (ex[:, :-1] - ex[:, 1:]) / self.dzh - GRAV)
        a = dtau * BETA * CPD * ti[:, 1:N] / self.dzh
        lo = (-a * gam[:, :-1] * M[:, :N - 1]).t().contiguous()
        di = (1.0 + a * (gam[:, :-1] + gam[:, 1:]) * M[:, 1:N]).t().contiguous()
        up = (-a * gam[:, 1:] * M[:, 2:]).t().contiguous()
        rh = (wx - a * (px[:, :-1] - px[:, 1:])).t().contiguous()
        for i in range(N - 1):
            p = di[i] - lo[i] * up[i - 1] if i else di[i]
            rh[i] = (rh[i] - lo[i] * rh[i - 1] if i else rh[i]) / p
            up[i] = up[i] / p
        for i in range(N - 3, -1, -1):
            rh[i] -= up[i] * rh[i + 1]
        wn = torch.zeros_like(w)
        wn[:, 1:N] = rh.t()
        wn = wn / (1.0 + dtau * self.ray)
        rho_n = rx - dtau * BETA * vert(ri * wn)
        q = M * wn
        new = {"rho": rho_n, "theta_v": (tx - dtau * BETA * vert(q)) / rho_n,
               "exner": px - gam * (q[:, :N] - q[:, 1:])}
        wc = BETA * wn + (1.0 - BETA) * w - wcc
        wc[:, 0] = 0.0
        wc[:, N] = 0.0
        wn[:, N] = wcc[:, N]
        return dict(new, w=wn), ri * wc

    def step(self, s, dt, upwind, diff4):
        dtau = dt / NSUB
        abar2 = (4.0 * math.pi * RADIUS * RADIUS / self.nc) ** 2
        thick = self.dze if self.topo else 1.0

        def heat(st, vn, F):
            t = st["theta_v"]
            return F * (torch.where(vn >= 0.0, t[self.c1], t[self.c2]) if upwind else self.mean(t))
        mflx = wflx = 0.0
        for _ in range(NSUB):
            A0, Aw0, wcc = self.tendencies(s["vn"], s["w"])
            vs = s["vn"] + dtau * (A0 - self.pressure_gradient(s))
            F = self.mean(s["rho"]) * vs * thick
            star, _ = self.column(s, F, heat(s, vs, F), Aw0, wcc, dtau)
            star["vn"] = vs
            A1, Aw1, wcc = self.tendencies(vs, star["w"])
            vn = s["vn"] + dtau * (0.5 * (A0 + A1) - self.pressure_gradient(star))
            vn = vn - (0.0025 * abar2) * self.grad(self.div(self.grad(self.div(vn))))
            F = self.mean(star["rho"]) * vn * thick
            new, W = self.column(s, F, heat(star, vn, F), 0.5 * (Aw0 + Aw1), wcc, dtau)
            mflx, wflx = mflx + F / NSUB, wflx + W / NSUB
            s = dict(new, vn=vn)
        vn, thv = s["vn"], s["theta_v"]
        u = [sum(self.lsq_w.view(-1, 6, 3)[:, j, i, None] * vn[self.v2e[:, j]] for j in range(6)) for i in range(3)]
        i34 = 1.0 / self.L34[:, None]
        q = self.e2q
        DT = DS = 0.0
        for i in range(3):
            d34, d12 = u[i][q[:, 3]] - u[i][q[:, 2]], u[i][q[:, 1]] - u[i][q[:, 0]]
            n, t = self.n_e[:, i:i + 1], self.t_e[:, i:i + 1]
            DT, DS = DT + d34 * n * i34 - d12 * t * self.ile, DS + d34 * t * i34 + d12 * n * self.ile
        Kh = 0.15 ** 2 * (self.l_e * self.d_e)[:, None] * torch.sqrt(DT * DT + DS * DS)
        lap = lambda x: self.grad(self.div(x)) - (lambda z: (z[self.v2] - z[self.v1]) * self.ile)(self.curl(x))  # noqa: E731
        L1 = lap(vn)
        vnew = vn + dt * Kh * L1 - ((diff4 * abar2) * lap(L1) if diff4 else 0.0)
        fl = self.l_e[:, None] * Kh * self.grad(thv)
        dth = dt * sum(self.s_ce[:, k:k + 1] * fl[self.c2e[:, k]] for k in range(3)) / self.A_c[:, None]
        return dict(s, vn=vnew, theta_v=thv + dth, exner=s["exner"] * (1.0 + (RD / CVD) * dth / thv)), mflx, wflx

    def tracer(self, tables, q, rho0, rho1, M, W, dt):
        c2c, G, roff = tables
        N = self.N
        thick = self.dze if self.topo else 1.0
        g = [sum(G[:, s, i, None] * (q[c2c[:, s]] - q) for s in range(3)) for i in range(3)]
        up = M >= 0.0
        pick = lambda f: torch.where(up, f[self.c1], f[self.c2])  # noqa: E731
        re = self.mean(rho0) * thick
        vn, vt = M / re, self.tangential(M) / re
        qe = pick(q)
        for i in range(3):
            off = torch.where(up, roff[:, 0, i, None], roff[:, 1, i, None])
            qe = qe + pick(g[i]) * (off - 0.5 * dt * (vn * self.n_e[:, i:i + 1] + vt * self.t_e[:, i:i + 1]))
        sl = torch.zeros_like(q)
        sl[:, 1:-1] = (q[:, :-2] - q[:, 2:]) / (self.zfc[:, :-2] - self.zfc[:, 2:])
        ri = self.half(self.wu, rho0)[:, 1:N]
        Wi, zh = W[:, 1:N], self.zhc[:, 1:N]
        up = Wi >= 0.0
        qd, sd = torch.where(up, q[:, 1:], q[:, :-1]), torch.where(up, sl[:, 1:], sl[:, :-1])
        zd = torch.where(up, self.zfc[:, 1:], self.zfc[:, :-1])
        V = torch.zeros_like(W)
        V[:, 1:N] = Wi * (qd + sd * (zh - zd - 0.5 * dt * Wi / ri))
        vert = (V[:, :N] - V[:, 1:]) / self.dz
        return (rho0 * q - dt * (self.div(M * qe) / (self.dz if self.topo else 1.0) + vert)) / rho1

    def mass(self, s):
        return float((self.A_c * (s["rho"] * self.dz).sum(1)).sum())


def exact(case, seed):
    """The outputs of run() on the inputs of prepare(case, seed). None for the largest grid,
    which takes longer than about 20 seconds this way, and for the masses of the members of an
    ensemble beyond its first."""
    cells = sum(20 * 4 ** (b + 1) * n for b, n in _groups(case)) * case["nlev"] * case["steps"]
    if cells > 6.0e8:
        return None
    m = prepare(case, seed)
    nlev, out = case["nlev"], {}
    host = lambda t: t.cpu().numpy()  # noqa: E731
    for i, (grid, states, buf) in enumerate(m.groups):
        E = _Exact(grid, nlev, case["topo_m"])
        tag = str(i) if case["members"] else ""
        rows = {f: [] for f in FIELDS}
        for j, st in enumerate(states):
            s = {f: torch.from_numpy(C.icon_state_copy_field(st, grid, nlev, f)).cuda() for f in FIELDS}
            q = [torch.from_numpy(C.icon_state_copy_tracer(st, grid, nlev, t)).cuda() for t in range(case["tracers"])]
            if q:
                tabs = [torch.from_numpy(C.icon_grid_copy_table(grid, n)).cuda() for n in ("c2c", "lsq_c", "roff")]
                tabs = (tabs[0].long(), tabs[1].view(-1, 3, 3), tabs[2].view(-1, 2, 3))
            dt = _dt(_groups(case)[i][0])
            for _ in range(case["steps"]):
                rho0 = s["rho"]
                s, M, W = E.step(s, dt, case["upwind"], case["diff4"])
                q = [E.tracer(tabs, x, rho0, s["rho"], M, W, dt) for x in q]
            if j == 0:
                out["mass" + tag] = E.mass(s)
            for f in FIELDS:
                rows[f].append(host(s[f]))
            for t, x in enumerate(q):
                out["q%d" % t] = host(x)
        for f in FIELDS:
            out[f + tag] = np.stack(rows[f]) if case["members"] else rows[f][0]
    return out
