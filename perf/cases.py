"""What this library is measured on: the calls that a user's model makes.

A GRIST-like model holds one mesh handle and steps its state with
`dycore_step_hydro` / `dycore_step_nh` and `tracer_step`, reads
`vorticity` and `global_sum` at its output times, and may record the whole
coupled step as a graph.  The listed cases are those calls over the mesh
levels, level counts, tracer counts and precisions of this repository's
configurations, tests and benchmark (meshes 4 to 8: a level-9 mesh takes
minutes to generate); draw() gives more of the same ranges, odd sizes and
padded rows among them.

Inputs are built on the GPU from the seed: a balanced zonal jet with a
smooth random perturbation (and a warm bubble, a weak vertical wind) for the
dynamical core; bells, slotted cylinders and Gaussian hills in a random
deformational wind for the tracers.  exact() restates the discretisation in
plain torch in 64 bits.
"""
import math

import numpy as np
import torch

import paper_2404_08849_gb300 as G
from grist_inputs import states as S
from grist_inputs.mesh import get_mesh, lonlat, n_cells, n_edges, n_vertices

DEV = "cuda:0"
F64 = torch.float64
P_TOP = 225.0
BETA = 0.55

# tracer and level counts of the 16-member uneven ensemble (drawn once from
# {1, 4, 10, 25} x {30, 60} with the benchmark's seed)
ENSEMBLE = "1x30 25x30 10x60 10x60 4x30 25x30 4x60 4x30 1x30 4x30 4x30 4x60 25x30 25x60 25x60 1x60"


def listed():
    return [
        # the smallest use: one tracer on a test mesh, 30 levels, double
        # precision (the rotation test every transport scheme is run on)
        {"name": "rotation_l4_fp64", "kind": "tracer", "level": 4, "members": "1x30", "prec": "fp64",
         "limiter": True, "vertical": False, "pad": 0},
        # a small coupled model whose whole step is one recorded graph: launch-bound
        {"name": "coupled_l5_graph_mix", "kind": "coupled", "level": 5, "L": 30, "T": 2, "prec": "mix", "nh": True,
         "graph": True, "pad": 0},
        # the hydrostatic configuration (jet, 30 levels, dt 300 s), both precisions side by side
        {"name": "hydro_l6_mix", "kind": "dycore", "level": 6, "L": 30, "prec": "mix", "nh": False, "pad": 0},
        {"name": "hydro_l6_fp64", "kind": "dycore", "level": 6, "L": 30, "prec": "fp64", "nh": False, "pad": 0},
        # the binary32-dominant variant of the double rows at an odd level count, padded rows
        {"name": "nh_l6_mix_df_odd", "kind": "dycore", "level": 6, "L": 41, "prec": "mix_df", "nh": True, "pad": 3},
        # uneven ensemble: 16 members of different tracer and level counts in one call
        {"name": "ensemble_l6_mix", "kind": "tracer", "level": 6, "members": ENSEMBLE, "prec": "mix",
         "limiter": True, "vertical": False, "pad": 0},
        # tracers driven offline by stored mass fluxes, horizontal and vertical, both precisions
        {"name": "tracers_l7_mix", "kind": "tracer", "level": 7, "members": "4x60", "prec": "mix", "limiter": True,
         "vertical": True, "pad": 0},
        {"name": "tracers_l7_fp64", "kind": "tracer", "level": 7, "members": "4x60", "prec": "fp64", "limiter": True,
         "vertical": True, "pad": 0},
        # output-time diagnostics: vorticity on every level, dry and tracer mass
        {"name": "diagnostics_l7_mix", "kind": "diag", "level": 7, "L": 60, "prec": "mix", "pad": 0},
        # the non-hydrostatic core in double precision
        {"name": "nh_l7_fp64", "kind": "dycore", "level": 7, "L": 60, "prec": "fp64", "nh": True, "pad": 0},
        # the non-hydrostatic configuration (jet and bubble, 60 levels)
        {"name": "nh_l8_mix", "kind": "dycore", "level": 8, "L": 60, "prec": "mix", "nh": True, "pad": 0},
        # the headline workload on a level-8 mesh: core, then 4 tracers with its fluxes
        {"name": "coupled_l8_mix", "kind": "coupled", "level": 8, "L": 60, "T": 4, "prec": "mix", "nh": True,
         "graph": False, "pad": 0},
    ]


def _cell_levels(case):
    """(cell-levels of the core, tracer-cell-levels) of one pass."""
    nC = n_cells(case["level"])
    if case["kind"] == "tracer":
        return 0, nC * sum(t * l for t, l in _members(case))
    return nC * case["L"], nC * case["L"] * (case["T"] if case["kind"] == "coupled" else 0)


def draw(rng):
    while True:
        kind = rng.choice(["tracer", "tracer", "dycore", "dycore", "dycore", "coupled", "diag"])
        level = rng.choice([4, 5, 6, 6, 7, 7, 8])
        L = rng.choice([30, 60, 30, 60, rng.randint(8, 72), rng.randint(8, 72)])
        prec = rng.choice(["mix", "mix", "fp64", "mix_dbl_mass", "mix_df"])
        case = {"kind": kind, "level": level, "prec": prec, "pad": rng.choice([0, 0, rng.randint(1, 5)])}
        if kind == "tracer":
            if rng.random() < 0.4:
                mem = [(rng.choice([1, 4, 10, 25]), rng.choice([30, 60])) for _ in range(rng.randint(2, 16))]
            else:
                mem = [(int(round(25.0 ** rng.random())), L)]
            case["members"] = " ".join("%dx%d" % m for m in mem)
            case["prec"] = "fp64" if prec == "fp64" else "mix"
            case["limiter"] = rng.random() < 0.8
            case["vertical"] = rng.random() < 0.5
        elif kind == "coupled":
            case.update(L=L, T=rng.randint(1, 6), nh=rng.random() < 0.7, graph=level <= 6 and rng.random() < 0.5)
        elif kind == "dycore":
            case.update(L=L, nh=rng.random() < 0.6)
        else:
            case.update(L=L, prec="fp64" if prec == "fp64" else "mix")
        # no more than the largest listed case: double precision costs about 2.5 times as much
        core, tracer = _cell_levels(case)
        if (core * 1.0 + tracer * 0.12) * (2.6 if case["prec"] == "fp64" else 1.0) <= 39.3e6 * 1.2:
            return case


def _members(case):
    return [tuple(int(x) for x in m.split("x")) for m in case["members"].split()]


def work(case):
    """Every input read once and every output written once; flops of the
    formulas as written."""
    nC, nE, nV = n_cells(case["level"]), n_edges(case["level"]), n_vertices(case["level"])
    s = 8 if case["prec"] == "fp64" else 4
    if case["kind"] == "diag":
        L = case["L"]
        return {"bytes": L * (nE * s + nV * 8 + nC * (s + 8)) + nC * 8, "flops": L * (nV * 5 + nC * 3) + 2 * nC}
    by = fl = 0
    if case["kind"] in ("dycore", "coupled"):
        L, nh = case["L"], case["nh"]
        by += 2 * nE * L * s + 2 * nC * 8 + 2 * nC * L * 8
        fl += 3 * L * (nE * (86 + 15 + 3) + nC * (13 + 17 + 8 + 18) + nV * 13)
        if nh:
            by += 4 * nC * (L + 1) * 8 + 2 * nC * L * 8
            fl += 3 * L * nC * (43 + 70)
        else:
            fl += 3 * L * nC * 15
    if case["kind"] == "coupled":
        L, T = case["L"], case["T"]
        by += nE * L * 8 + nC * (L + 1) * 8 + nC * L * 8 + 2 * T * nC * L * s
        fl += T * L * (nE * (3 * 15 + 20) + nC * (3 * 15 + 70))
    if case["kind"] == "tracer":
        for T, L in _members(case):
            by += 2 * T * nC * L * s + nC * L * 8 + nE * L * 8 + (nC * (L + 1) * 8 if case["vertical"] else 0)
            fl += T * L * (nE * (3 * 15 + 5) + nC * (2 * 15 + 15))
            if case["limiter"]:
                fl += T * L * (nE * 5 + nC * 60)
            if case["vertical"]:
                fl += T * L * nC * 10
    return {"bytes": by, "flops": fl}


# ---------------------------------------------------------------------------
# the mesh of a level: the library's handle and, in its numbering, the tables
# the inputs are made from

class _Grid:
    def __init__(self, level):
        self.m = m = get_mesh(level)
        self.mesh = G.Mesh(m, device=0)
        self.nC, self.nE, self.nV = m["n_cells"], m["n_edges"], m["n_vertices"]
        self.radius = m["radius"]
        self.old = {"cell": self.mesh.cell_old, "edge": self.mesh.edge_old, "vertex": self.mesh.vertex_old}
        self.new = {k: torch.from_numpy(v.astype(np.int64)).to(DEV) for k, v in (
            ("cell", self.mesh.cell_new), ("edge", self.mesh.edge_new), ("vertex", self.mesh.vertex_new))}
        self._t = {}
        self.jet = S.ZonalJet(self.radius, m["omega"], t0=260.0)
        lat = lonlat(m["cell_xyz"])[1][self.old["cell"]]
        self.jet_g = [torch.from_numpy(g).to(DEV) for g in self.jet.G(lat)]
        self.jet_ps = torch.from_numpy(self.jet.surface_pressure(lat)).to(DEV)
        self.phis = torch.zeros(self.nC, dtype=F64, device=DEV)

    def t(self, name, kind, of=None):
        """Table `name` (rows of `kind` entities, entries indices of `of`
        entities where given, missing ones kept as -1) on the GPU in the
        library's numbering."""
        if name not in self._t:
            a = torch.from_numpy(np.ascontiguousarray(self.m[name][self.old[kind]])).to(DEV)
            if of:
                a = a.long()
                a = torch.where(a >= 0, self.new[of][a.clamp(min=0)], a)
            self._t[name] = a
        return self._t[name]


_GRIDS = {}
_STREAM = []


def _stream():
    """The one created stream that the recorded steps run on."""
    if not _STREAM:
        _STREAM.append(torch.cuda.Stream())
    return _STREAM[0]


def _grid(level):
    if level not in _GRIDS:
        _GRIDS[level] = _Grid(level)
    return _GRIDS[level]


# ---------------------------------------------------------------------------
# inputs from a seed

def _waves(gen, xyz, n=10, kmin=1.0, kmax=16.0):
    """Smooth random field of unit size on the sphere: n plane waves."""
    k = torch.randn((n, 3), generator=gen, dtype=F64)
    k = k / k.norm(dim=1, keepdim=True) * (kmin + (kmax - kmin) * torch.rand((n, 1), generator=gen, dtype=F64))
    ph = 2 * math.pi * torch.rand(n, generator=gen, dtype=F64)
    a = torch.randn(n, generator=gen, dtype=F64) / math.sqrt(n)
    f = torch.zeros(xyz.shape[0], dtype=F64, device=DEV)
    for i in range(n):
        f += float(a[i]) * torch.cos(xyz @ k[i].to(DEV) + float(ph[i]))
    return f


def _wind(g, gen, amp, kmax):
    """Non-divergent edge-normal wind of a random vertex stream function."""
    psi = _waves(gen, g.t("vertex_xyz", "vertex"), kmax=kmax)
    voe = g.t("vertices_on_edge", "edge", "vertex")
    u = -(psi[voe[:, 1]] - psi[voe[:, 0]]) / g.t("edge_dv", "edge")
    return u * (amp / u.abs().max())


def _col(x, n, pad, fill=0.0):
    """[.., n] with its rows padded to n + pad."""
    if not pad:
        return x.contiguous()
    y = torch.full(x.shape[:-1] + (n + pad,), fill, dtype=x.dtype, device=x.device)
    y[..., :n] = x
    return y


def _div(g, F):
    eoc, sg = g.t("edges_on_cell", "cell", "edge"), g.t("edge_sign_on_cell", "cell")
    dv, A = g.t("edge_dv", "edge"), g.t("cell_area", "cell")
    out = torch.zeros((g.nC,) + F.shape[1:], dtype=F64, device=DEV)
    for j in range(6):
        e = eoc[:, j].clamp(min=0)
        c = sg[:, j] * dv[e] / A
        out += c.view(-1, *([1] * (F.dim() - 1))) * F[e]
    return out


def _core_inputs(case, seed):
    """The dynamical core's state in 64 bits (u as the precision stores it)."""
    g, L, nh = _grid(case["level"]), case["L"], case["nh"]
    gen = torch.Generator().manual_seed(seed)
    if nh:
        B, pi_top = S.sigma_from_heights(S.stretched_heights(L), t_ref=260.0)
    else:
        B, pi_top = S.sigma_uniform(L), P_TOP
    Bt = torch.from_numpy(B).to(DEV)
    xyz = g.t("cell_xyz", "cell")
    ps = g.jet_ps * (1.0 + 2e-4 * _waves(gen, xyz, kmax=8.0))
    pint = pi_top + Bt[None, :] * (ps[:, None] - pi_top)
    pmid = 0.5 * (pint[:, 1:] + pint[:, :-1])
    jet = g.jet
    x = (torch.log(pmid) - jet.lpj) / jet.w
    Sj = torch.exp(-x * x)
    dS = -2.0 * x / jet.w * Sj
    T = jet.t0 + (dS * g.jet_g[0][:, None] + 2.0 * Sj * dS * g.jet_g[1][:, None]) / S.RD
    theta = T * (S.P0 / pmid) ** S.KAPPA
    lev = torch.linspace(0.0, math.pi, L, dtype=F64, device=DEV)
    theta += 0.3 * _waves(gen, xyz, kmax=12.0)[:, None] * torch.sin(lev)[None, :]
    if nh:   # warm bubble below about 5 km at a random place
        c = torch.randn(3, generator=gen, dtype=F64)
        r = torch.acos((xyz @ (c / c.norm()).to(DEV)).clamp(-1, 1)) * g.radius
        z = S.RD * 260.0 / S.GRAVITY * torch.log(S.P0 / pmid)
        theta += 2.0 * torch.exp(-(r / 250.0e3) ** 2)[:, None] * (z < 5.0e3)
    coe = g.t("cells_on_edge", "edge", "cell")
    pe = 0.5 * (pmid[coe[:, 0]] + pmid[coe[:, 1]])
    xe, ne = g.t("edge_xyz", "edge"), g.t("edge_normal_xyz", "edge")
    lat = torch.asin(xe[:, 2].clamp(-1, 1))
    east = torch.stack([-xe[:, 1], xe[:, 0], torch.zeros_like(lat)], 1)
    east = east / east.norm(dim=1, keepdim=True).clamp(min=1e-300)
    U = jet.umax * torch.sin(2 * lat) ** 2 * (east * ne).sum(1)
    u = U[:, None] * torch.exp(-((torch.log(pe) - jet.lpj) / jet.w) ** 2)
    u += _wind(g, gen, 1.0, 16.0)[:, None]
    out = {"u": u if case["prec"] == "fp64" else u.float(), "ps": ps, "dpi_theta": (pint[:, 1:] - pint[:, :-1]) * theta}
    out["B"], out["pi_top"] = B, pi_top
    if nh:
        dpi = pint[:, 1:] - pint[:, :-1]
        al = S.RD * theta * (pmid / S.P0) ** S.KAPPA / pmid
        phi = torch.zeros((g.nC, L + 1), dtype=F64, device=DEV)
        phi[:, :L] = torch.flip(torch.cumsum(torch.flip(al * dpi, [1]), 1), [1])
        w = torch.zeros_like(phi)
        w[:] = 0.05 * _waves(gen, xyz, kmax=12.0)[:, None] * torch.sin(math.pi * Bt)[None, :]
        w[:, 0] = w[:, L] = 0.0
        out["phi"], out["w"] = phi, w
        out["p_nh"] = S.P0 * (S.RD * out["dpi_theta"] / (S.P0 * (phi[:, :-1] - phi[:, 1:]))) ** S.GAMMA
    return out


def _tracer_shapes(g, gen, T, L):
    """Bells, slotted cylinders and Gaussian hills in turn, [T][nC][L]."""
    xyz = g.t("cell_xyz", "cell")
    lon, lat = torch.atan2(xyz[:, 1], xyz[:, 0]), torch.asin(xyz[:, 2].clamp(-1, 1))
    lev = 1.0 + 0.1 * torch.linspace(-1.0, 1.0, L, dtype=F64, device=DEV)
    q = torch.empty((T, g.nC, L), dtype=F64, device=DEV)
    for t in range(T):
        a, b, c, d, e = (float(v) for v in torch.rand(5, generator=gen, dtype=F64))
        lon0, lat0 = 2 * math.pi * a, 2.0 * b - 1.0
        centre = torch.tensor([math.cos(lat0) * math.cos(lon0), math.cos(lat0) * math.sin(lon0), math.sin(lat0)],
                              dtype=F64, device=DEV)
        r = torch.acos((xyz @ centre).clamp(-1, 1))
        if t % 3 == 0:
            r0 = 0.2 + 0.3 * c
            h = torch.where(r < r0, 0.5 * (1.0 + torch.cos(math.pi * r / r0)), torch.zeros_like(r))
        elif t % 3 == 1:
            dl = torch.remainder(lon - lon0 + math.pi, 2 * math.pi) - math.pi
            slot = (dl.abs() < 0.04 + 0.035 * d) & (lat < lat0 + 0.2 + 0.2 * e)
            h = ((r < 0.3 + 0.2 * c) & ~slot).to(F64)
        else:
            h = torch.exp(-(r / (0.1 + 0.2 * c)) ** 2)
        q[t] = 0.1 + h[:, None] * lev[None, :]
    return q


def _dt_core(case):
    return min(300.0, 300.0 * 2.0 ** (6 - case["level"])) if not case["nh"] else min(120.0, 60.0 * 2.0 ** (8 - case["level"]))


def _tracer_inputs(case, seed):
    """Members of an offline transport run: stored mass fluxes and layer
    masses of a random deformational wind, and its vertical mass flux."""
    g = _grid(case["level"])
    gen = torch.Generator().manual_seed(seed)
    qt = F64 if case["prec"] == "fp64" else torch.float32
    coe = g.t("cells_on_edge", "edge", "cell")
    out = []
    for T, L in _members(case):
        ps = 1.0e5 * (1.0 + 0.02 * _waves(gen, g.t("cell_xyz", "cell"), kmax=4.0))
        dpi = ((ps - P_TOP) / L)[:, None].expand(-1, L).contiguous()
        u = _wind(g, gen, 40.0, 4.0)
        shear = 0.7 + 0.3 * torch.cos(torch.linspace(0.0, math.pi, L, dtype=F64, device=DEV))
        F = 0.5 * (dpi[coe[:, 0]] + dpi[coe[:, 1]]) * u[:, None] * shear[None, :]
        m = {"q": _tracer_shapes(g, gen, T, L).to(qt), "dpi": dpi, "F": F, "L": L}
        if case["vertical"]:
            D = _div(g, F)
            M = torch.zeros((g.nC, L + 1), dtype=F64, device=DEV)
            B = torch.arange(1, L, dtype=F64, device=DEV) / L
            M[:, 1:L] = B[None, :] * D.sum(1, keepdim=True) - torch.cumsum(D, 1)[:, :-1]
            m["M"] = M
        out.append(m)
    return out, 0.4 * float(g.t("edge_dc", "edge").min()) / 40.0


# ---------------------------------------------------------------------------
# the calls

def prepare(case, seed):
    g, pad = _grid(case["level"]), case["pad"]
    if case["kind"] == "tracer":
        members, dt = _tracer_inputs(case, seed)
        mb = []
        for m in members:
            L = m["L"]
            d = {"q": _col(m["q"], L, pad), "dpi": _col(m["dpi"], L, pad), "mass_flux": _col(m["F"], L, pad), "n_levels": L}
            if "M" in m:
                d["vmass_flux"] = _col(m["M"], L + 1, pad)
            mb.append(d)
        return {"case": case, "mesh": g.mesh, "members": mb, "dt": dt}
    L = case["L"]
    if case["kind"] == "diag":
        c = _core_inputs(dict(case, nh=False), seed)
        q = _tracer_shapes(g, torch.Generator().manual_seed(seed + 1), 1, L)[0]
        B = torch.from_numpy(np.diff(c["B"])).to(DEV)
        return {"case": case, "mesh": g.mesh, "u": _col(c["u"], L, pad), "ps": c["ps"], "L": L,
                "q": _col(q.to(c["u"].dtype), L, pad),
                "dpi": _col((c["ps"] - P_TOP)[:, None] * B[None, :], L, pad),
                "vor": torch.zeros((g.nV, L + pad), dtype=F64, device=DEV)}
    c = _core_inputs(case, seed)
    s = {"u": _col(c["u"], L, pad), "ps": c["ps"].clone(), "dpi_theta": _col(c["dpi_theta"], L, pad)}
    if case["nh"]:
        s.update(w=_col(c["w"], L + 1, pad), phi=_col(c["phi"], L + 1, pad), p_nh=_col(c["p_nh"], L, pad), p_nh_valid=True)
    P = G.DycoreParams(L, c["B"], c["pi_top"], g.phis, ld=L + pad, ld_int=L + 1 + pad, beta=BETA)
    st = {"case": case, "mesh": g.mesh, "s": s, "P": P, "dt": _dt_core(case)}
    if case["kind"] == "coupled":
        T = case["T"]
        s["mass_flux_accum"] = torch.zeros((g.nE, L + pad), dtype=F64, device=DEV)
        s["vmass_flux_accum"] = torch.zeros((g.nC, L + 1 + pad), dtype=F64, device=DEV)
        s["dpi_start"] = torch.zeros((g.nC, L + pad), dtype=F64, device=DEV)
        q = _tracer_shapes(g, torch.Generator().manual_seed(seed + 1), T, L)
        st["q"] = _col(q if case["prec"] == "fp64" else q.float(), L, pad)
        st["members"] = [{"q": st["q"], "dpi": s["dpi_start"], "mass_flux": s["mass_flux_accum"],
                          "vmass_flux": s["vmass_flux_accum"], "n_levels": L}]
        if case["graph"]:
            # a graph program keeps a handle of its own; it has stepped before
            # the step is recorded (first calls size scratch and upload
            # tables), and the state starts over from its initial values
            st["mesh"] = G.Mesh(g.m, device=0)
            stream = _stream()
            keep = {k: v.clone() for k, v in s.items() if isinstance(v, torch.Tensor)}
            q0 = st["q"].clone()
            torch.cuda.synchronize()
            with torch.cuda.stream(stream):
                _coupled(st)
                _coupled(st)
                for k, v in keep.items():
                    s[k].copy_(v)
                st["q"].copy_(q0)
            stream.synchronize()
            st["graph"] = G.capture(lambda: _coupled(st), stream)
    return st


def _core(st):
    step = st["mesh"].dycore_step_nh if st["case"]["nh"] else st["mesh"].dycore_step_hydro
    step(st["s"], st["P"], st["dt"], prec=st["case"]["prec"])


def _coupled(st):
    s = st["s"]
    s["mass_flux_accum"].zero_()
    s["vmass_flux_accum"].zero_()
    _core(st)
    st["mesh"].tracer_step(st["members"], st["dt"], prec=st["case"]["prec"], limiter=True)


def run(st):
    case, kind = st["case"], st["case"]["kind"]
    if kind == "tracer":
        st["mesh"].tracer_step(st["members"], st["dt"], prec=case["prec"], limiter=case["limiter"])
        return [m["q"][..., :m["n_levels"]] for m in st["members"]]
    if kind == "diag":
        mesh, L = st["mesh"], st["L"]
        vor = mesh.vorticity(st["u"], L, out=st["vor"])
        dry = mesh.global_sum(G.GRIST_SUM_DRY_MASS, st["ps"], offset=P_TOP)[0]
        tr = mesh.global_sum(G.GRIST_SUM_TRACER_MASS, st["q"], st["dpi"], n_levels=L)[0]
        return {"vor": vor[:, :L], "dry": dry, "tracer": tr}
    L, s = case["L"], st["s"]
    if kind == "dycore":
        _core(st)
    elif case["graph"]:
        st["graph"].launch()
    else:
        _coupled(st)
    out = {"u": s["u"][:, :L], "ps": s["ps"], "dpi_theta": s["dpi_theta"][:, :L]}
    if case["nh"]:
        out.update(w=s["w"][:, :L + 1], phi=s["phi"][:, :L + 1], p_nh=s["p_nh"][:, :L])
    if kind == "coupled":
        out.update(q=st["q"][..., :L], mass_flux=s["mass_flux_accum"][:, :L], vmass_flux=s["vmass_flux_accum"][:, :L + 1],
                   dpi_start=s["dpi_start"][:, :L])
    return out


# ---------------------------------------------------------------------------
# the discretisation in 64 bits, plain torch

def _edge_value(g, F, q):
    """Third-order upwind edge value of the cell field q [nC][L] for the flux
    F: the cells' mean less dc^2/6 of the upwind second derivative."""
    coe, dc = g.t("cells_on_edge", "edge", "cell"), g.t("edge_dc", "edge")
    sten, coef = g.t("d2_stencil", "edge", "cell"), g.t("d2_coef", "edge")
    d = [torch.zeros_like(F), torch.zeros_like(F)]
    for side in (0, 1):
        for j in range(7):
            d[side] += coef[:, side, j, None] * q[sten[:, side, j].clamp(min=0)]
    return 0.5 * (q[coe[:, 0]] + q[coe[:, 1]]) - (dc * dc / 6.0)[:, None] * torch.where(F >= 0, d[0], d[1])


def _exact_tracer(g, q, dpi, F, dt, limiter, M=None):
    """One step of one tracer [nC][L], Courant limit 1 in the vertical."""
    D = _div(g, F)
    low = None
    x = q
    for s, h in enumerate((dt / 3.0, dt / 2.0, dt)):
        end = dpi - h * D
        FH = F * _edge_value(g, F, x)
        if s == 2 and limiter:
            coe, coc = g.t("cells_on_edge", "edge", "cell"), g.t("cells_on_cell", "cell", "cell")
            eoc, sg = g.t("edges_on_cell", "cell", "edge"), g.t("edge_sign_on_cell", "cell")
            dv, A = g.t("edge_dv", "edge"), g.t("cell_area", "cell")
            FL = F * torch.where(F >= 0, q[coe[:, 0]], q[coe[:, 1]])
            low = (dpi * q - h * _div(g, FL)) / end
            anti = FH - FL
            hi, lo = torch.maximum(q, low), torch.minimum(q, low)
            qmax, qmin = hi.clone(), lo.clone()
            pp, pm = torch.zeros_like(q), torch.zeros_like(q)
            for j in range(6):
                ok = (coc[:, j] >= 0)[:, None]
                nb = coc[:, j].clamp(min=0)
                qmax = torch.where(ok, torch.maximum(qmax, hi[nb]), qmax)
                qmin = torch.where(ok, torch.minimum(qmin, lo[nb]), qmin)
                e = eoc[:, j].clamp(min=0)
                o = (sg[:, j] * dv[e] / A)[:, None] * anti[e] * h
                pp += (-o).clamp(min=0)
                pm += o.clamp(min=0)
            tiny = 2.2250738585072014e-308
            rp = ((qmax - low) * end / (pp + tiny)).clamp(max=1.0)
            rm = ((low - qmin) * end / (pm + tiny)).clamp(max=1.0)
            c1, c2 = coe[:, 0], coe[:, 1]
            C = torch.where(anti >= 0, torch.minimum(rm[c1], rp[c2]), torch.minimum(rp[c1], rm[c2]))
            FH = FL + C * anti
        x = (dpi * q - h * _div(g, FH)) / end
    if M is None:
        return x
    L = q.shape[1]
    z = torch.zeros_like(x[:, :1])
    star = dpi - dt * D
    Mi = M[:, 1:L]
    up, dn = star[:, :-1], star[:, 1:]
    c = Mi.abs() * dt / torch.where(Mi > 0, up, dn)
    Me = torch.where(c <= 1.0, Mi, Mi / c.clamp(min=1.0))
    Fe = torch.cat([z, Me * torch.where(Mi > 0, x[:, :-1], x[:, 1:]), z], 1)
    Im = torch.cat([z, Mi - Me, z], 1)
    Mf = torch.cat([z, Mi, z], 1)
    rhs = star * x - dt * (Fe[:, 1:] - Fe[:, :-1])
    b = star - dt * (Mf[:, 1:] - Mf[:, :-1]) + dt * (Im[:, 1:].clamp(min=0) - Im[:, :-1].clamp(max=0))
    a = -dt * Im[:, :-1].clamp(min=0)
    cc = dt * Im[:, 1:].clamp(max=0)
    return _thomas(a, b, cc, rhs)


def _thomas(a, b, c, r):
    """a_k x_{k-1} + b_k x_k + c_k x_{k+1} = r_k along the second axis."""
    a, b, c, r = (v.t().contiguous() for v in (a, b, c, r))
    n = r.shape[0]
    cp, dd = torch.empty_like(r), torch.empty_like(r)
    for k in range(n):
        den = b[k] - (a[k] * cp[k - 1] if k else 0.0)
        cp[k] = c[k] / den
        dd[k] = (r[k] - (a[k] * dd[k - 1] if k else 0.0)) / den
    for k in range(n - 2, -1, -1):
        dd[k] -= cp[k] * dd[k + 1]
    return dd.t()


def _exact_core(case, c):
    """One step of the dynamical core from the inputs c; the new state and
    the last stage's fluxes."""
    g, L, nh, dt = _grid(case["level"]), case["L"], case["nh"], _dt_core(case)
    B = torch.from_numpy(c["B"]).to(DEV)
    dB, pt = B[1:] - B[:-1], c["pi_top"]
    rd, cp, grav, p0 = S.RD, S.CP, S.GRAVITY, S.P0
    kap, gam = rd / cp, cp / (cp - rd)
    coe, voe = g.t("cells_on_edge", "edge", "cell"), g.t("vertices_on_edge", "edge", "vertex")
    c1, c2 = coe[:, 0], coe[:, 1]
    eoc, coc = g.t("edges_on_cell", "cell", "edge"), g.t("cells_on_cell", "cell", "cell")
    sg, A = g.t("edge_sign_on_cell", "cell"), g.t("cell_area", "cell")
    dc, dv = g.t("edge_dc", "edge"), g.t("edge_dv", "edge")
    eov, cov = g.t("edges_on_vertex", "vertex", "edge"), g.t("cells_on_vertex", "vertex", "cell")
    sv, kite, Av = g.t("edge_sign_on_vertex", "vertex"), g.t("kite_area", "vertex"), g.t("vertex_area", "vertex")
    fv = g.t("f_vertex", "vertex")
    eoe, wt = g.t("edges_on_edge", "edge", "edge"), g.t("trisk_weight", "edge")
    z = torch.zeros((g.nC, 1), dtype=F64, device=DEV)
    n = {k: v.double() for k, v in c.items() if isinstance(v, torch.Tensor)}
    dpi_n = (n["ps"] - pt)[:, None] * dB
    s = dict(n)
    if nh:
        mid_n = 0.5 * (dpi_n[:, 1:] + dpi_n[:, :-1])
        fw = torch.cat([z, grav * ((n["p_nh"][:, 1:] - n["p_nh"][:, :-1]) / mid_n - 1.0), z], 1)
    for h in (dt / 3.0, dt / 2.0, dt):
        dpi = (s["ps"] - pt)[:, None] * dB
        dpe = 0.5 * (dpi[c1] + dpi[c2])
        F = dpe * s["u"]
        D = _div(g, F)
        pst = -D.sum(1)
        M = torch.cat([z, -B[1:L] * pst[:, None] - torch.cumsum(D, 1)[:, :-1], z], 1)
        ps = n["ps"] + h * pst
        dpo = (ps - pt)[:, None] * dB
        th = s["dpi_theta"] / dpi
        thi = torch.cat([z, 0.5 * (th[:, 1:] + th[:, :-1]), z], 1)
        Mt = M * thi
        tho = n["dpi_theta"] + h * (-_div(g, F * _edge_value(g, F, th)) - (Mt[:, 1:] - Mt[:, :-1]))
        o = {"ps": ps, "dpi_theta": tho}
        if nh:
            adv = {}
            ui = torch.cat([s["u"][:, :1], 0.5 * (s["u"][:, 1:] + s["u"][:, :-1])], 1)   # interfaces 0..L-1
            for k in ("w", "phi"):
                x = s[k]
                ha = torch.zeros_like(x[:, :L])
                for j in range(6):
                    e, nb = eoc[:, j].clamp(min=0), coc[:, j].clamp(min=0)
                    ha += (sg[:, j] * dv[e] / A)[:, None] * ui[e] * 0.5 * (x[nb, :L] - x[:, :L])
                ha[:, 1:] += M[:, 1:L] * (x[:, 2:] - x[:, :-2]) / (dpi[:, 1:] + dpi[:, :-1])
                adv[k] = ha
            ws = n["w"][:, :L] + h * (-adv["w"] + (1.0 - BETA) * fw[:, :L])
            fs = n["phi"][:, :L] + h * (-adv["phi"] + (1.0 - BETA) * grav * n["w"][:, :L])
            fs = torch.cat([fs, g.phis[:, None]], 1)
            bg = BETA * h * grav
            dfs = fs[:, :-1] - fs[:, 1:]
            dfn = n["phi"][:, :-1] - n["phi"][:, 1:]
            pss = n["p_nh"] * ((tho * dfn) / (n["dpi_theta"] * dfs)) ** gam
            C = gam * pss * bg / dfs
            a = bg / (0.5 * (dpo[:, 1:] + dpo[:, :-1]))
            up, dn = C[:, :-1], C[:, 1:]
            w = _thomas(-a * up, 1.0 + a * (up + dn), -a * dn, ws[:, 1:] - bg + a * (pss[:, 1:] - pss[:, :-1]))
            o["w"] = torch.cat([z, w, z], 1)
            o["phi"] = torch.cat([fs[:, :L] + bg * o["w"][:, :L], g.phis[:, None]], 1)
            dphi = o["phi"][:, :-1] - o["phi"][:, 1:]
            p = pss * (1.0 + bg * (o["w"][:, :-1] - o["w"][:, 1:]) / dfs) ** (-gam)
            o["p_nh"] = p
            al = dphi / dpo
            lay = 0.5 * (o["phi"][:, :-1] + o["phi"][:, 1:])
            hi = torch.cat([z + 1.0, (p[:, 1:] - p[:, :-1]) / (0.5 * (dpo[:, 1:] + dpo[:, :-1])), z + 1.0], 1)
            dpp = 0.5 * (hi[:, 1:] + hi[:, :-1])
        else:
            pi = pt + B * (ps - pt)[:, None]
            p = 0.5 * (pi[:, 1:] + pi[:, :-1])
            al = rd * tho / dpo * (p / p0) ** kap / p
            ph = torch.flip(torch.cumsum(torch.flip(al * dpo, [1]), 1), [1]) + g.phis[:, None]
            lay = ph - 0.5 * al * dpo
            dpp = torch.ones_like(p)
        zeta = torch.zeros((g.nV, L), dtype=F64, device=DEV)
        col = torch.zeros(g.nV, dtype=F64, device=DEV)
        for j in range(3):
            zeta += (sv[:, j] * dc[eov[:, j]] / Av)[:, None] * s["u"][eov[:, j]]
            col += kite[:, j] / Av * (s["ps"][cov[:, j]] - pt)
        qv = (zeta + fv[:, None]) / (col[:, None] * dB)
        qe = 0.5 * (qv[voe[:, 0]] + qv[voe[:, 1]])
        K = torch.zeros((g.nC, L), dtype=F64, device=DEV)
        for j in range(6):
            e = eoc[:, j].clamp(min=0)
            K += (sg[:, j].abs() * 0.25 * dc[e] * dv[e] / A)[:, None] * s["u"][e] ** 2
        tend = -(K[c2] - K[c1]) - 0.5 * (al[c1] + al[c2]) * (p[c2] - p[c1])
        tend = (tend - 0.5 * (dpp[c1] + dpp[c2]) * (lay[c2] - lay[c1])) / dc[:, None]
        for j in range(10):
            e = eoe[:, j].clamp(min=0)
            wj = torch.where(eoe[:, j] >= 0, wt[:, j] * dv[e] / dc, torch.zeros_like(dc))
            tend += wj[:, None] * F[e] * 0.5 * (qe + qe[e])
        ze = torch.zeros((g.nE, 1), dtype=F64, device=DEV)
        Mu = torch.cat([ze, 0.5 * (M[c1, 1:L] + M[c2, 1:L]) * (s["u"][:, 1:] - s["u"][:, :-1]), ze], 1)
        tend -= (Mu[:, 1:] + Mu[:, :-1]) / (2.0 * dpe)
        o["u"] = n["u"] + h * tend
        s = dict(n, **o)
    return s, F, M, dpi_n


def exact(case, seed):
    g = _grid(case["level"])
    if case["kind"] == "tracer":
        members, dt = _tracer_inputs(case, seed)
        return [torch.stack([_exact_tracer(g, q.double(), m["dpi"], m["F"], dt, case["limiter"], m.get("M"))
                             for q in m["q"]]) for m in members]
    L = case["L"]
    if case["kind"] == "diag":
        st = prepare(case, seed)
        eov, sv = g.t("edges_on_vertex", "vertex", "edge"), g.t("edge_sign_on_vertex", "vertex")
        dc, Av, A = g.t("edge_dc", "edge"), g.t("vertex_area", "vertex"), g.t("cell_area", "cell")
        u = st["u"][:, :L].double()
        vor = torch.zeros((g.nV, L), dtype=F64, device=DEV)
        for j in range(3):
            vor += (sv[:, j] * dc[eov[:, j]] / Av)[:, None] * u[eov[:, j]]
        return {"vor": vor, "dry": math.fsum((A * (st["ps"] - P_TOP)).tolist()),
                "tracer": float((A[:, None] * st["dpi"][:, :L] * st["q"][:, :L].double()).sum())}
    c = _core_inputs(case, seed)
    s, F, M, dpi = _exact_core(case, c)
    out = {k: s[k] for k in ("u", "ps", "dpi_theta") + (("w", "phi", "p_nh") if case["nh"] else ())}
    if case["kind"] == "coupled":
        q = _tracer_shapes(g, torch.Generator().manual_seed(seed + 1), case["T"], L)
        q = q if case["prec"] == "fp64" else q.float().double()
        out.update(q=torch.stack([_exact_tracer(g, x, dpi, F, _dt_core(case), True, M) for x in q]),
                   mass_flux=F, vmass_flux=M, dpi_start=dpi)
    return out
