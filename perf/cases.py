"""Performance cases of the hybrid force-free / PIC step.

Every case is work that a user of ``paper_2406_14512_gb300.hff`` has the GPU
do, through the public binding: whole steps of one instance or of an ensemble
(``Sim.step``, ``Ensemble.step``) with the state read afterwards on the
device, loading particles (``load_device``) and the FP64 diagnostics, maps and
spectra.  Inputs (configuration numbers, particles, fields) are made here from
the seed, on the GPU, in the shapes and distributions of the workloads of the
framework: log-spherical grids, Table 1 flux bands, co-located e-/e+ pairs
with Maxwellian or gamma^-2 momenta, radiation reaction, surface injection.

``exact`` is an independent restatement of the step in torch float64 (no code
of the framework): the arithmetic is written from the scheme's definitions,
with the particle move done in plain cylindrical coordinates.
"""
import math

import numpy as np
import torch

from paper_2406_14512_gb300 import hff

DEV = "cuda:0"
FIELDS6 = ("E_r", "E_th", "E_ph", "B_r", "B_th", "B_ph")
BANDS = ([0.85, 0.9, 2.3, 2.4], [1.0, 0.0, 0.0, 1.0])  # Table 1, units of mu / R_LC


# ------------------------------------------------------------------- cases
def _run(name, nr, nt, pairs, **kw):
    c = dict(name=name, kind="run", nr=nr, nt=nt, pairs=pairs, r_max=60.0, r_lc=6.0, geom="synth", kappa=10.0,
             momenta="maxwell", rr=False, species=2, gamma_th=0.0, precision="fp32", tile_r=16, tile_t=24,
             sort_every=12, steps=3, order="scattered", capacity=0)
    c.update(kw)
    return c


def listed():
    return [
        # The production run: 4096^2, 3e8 e+-, power-law momenta, radiation
        # reaction, injection, Table 1 bands.  The largest case.
        _run("run_4096_rr", 4096, 4096, 150_000_000, r_max=100.0, r_lc=10.0, kappa=1.0, momenta="powerlaw", rr=True),
        # A standard hybrid run: 1024^2, 5e7 Maxwellian e+- (24 per cell).
        _run("run_1024", 1024, 1024, 25_000_000),
        # The same physics as the production run late in a run: injected
        # pairs keep their order through the stable sort, so particles of one
        # cell sit next to each other.
        _run("run_2048_cell_order", 2048, 2048, 10_000_000, r_max=100.0, r_lc=10.0, kappa=1.0, momenta="powerlaw",
             rr=True, order="cell"),
        # The monopole test of the paper (PIC north, force-free south, sharp
        # cut) mid-run: field-heavy, a large capacity mostly unused.
        _run("monopole_1024", 1024, 1024, 2_000_000, r_max=50.0 / 3.0, r_lc=5.0, geom="monopole", tile_t=32,
             sort_every=8, steps=2, capacity=16_000_000),
        # Electrons, positrons and protons, crust extraction, threshold pair
        # creation, on a ragged grid.
        _run("crust_pairs_500x380", 500, 380, 1_000_000, r_max=30.0, r_lc=3.0, momenta="powerlaw", rr=True,
             species=3, gamma_th=1000.0, tile_t=32, sort_every=8, steps=2, capacity=1_500_000),
        # The FP64 reference configuration: PIC everywhere, 256 x 128, 2e5 e+-.
        _run("run_256x128_fp64", 256, 128, 100_000, r_max=30.0, r_lc=3.0, geom="dipole", precision="fp64", tile_t=32,
             sort_every=8, steps=16),
        # FP64 with radiation reaction at a size that fills the GPU.
        _run("run_512_rr_fp64", 512, 512, 2_300_000, r_max=100.0, r_lc=10.0, kappa=1.0, momenta="powerlaw", rr=True,
             precision="fp64", steps=3),
        # The smallest run: a convergence or smoke problem, launch-bound.
        _run("run_96x80", 96, 80, 6_000, tile_t=32, sort_every=8, steps=16, capacity=40_000),
        # The force-free limit without particles: the field update alone.
        _run("fields_2048", 2048, 2048, 0, r_max=50.0 / 3.0, r_lc=5.0, geom="monopole", sort_every=0, steps=4),
        # A parameter study: seven independent instances of mixed grids and
        # particle numbers, one graph launch per step.
        dict(name="ensemble_7", kind="ensemble", n_inst=7, config_seed=1234, n_lo=100_000, n_hi=5_000_000,
             rows="256,512,1024", cols="128,256,512", sort_every=16, steps=5),
        # Loading particles in arbitrary order (start of a run, exchange with
        # another code): the tile sort and the payload gather.
        dict(_run("load_1024", 1024, 1024, 12_500_000), kind="load"),
        # Monitoring a run: L(r), energies, Gauss residual, density and
        # energy maps, spectra.
        dict(_run("diagnostics_1024", 1024, 1024, 12_500_000), kind="diagnostics", nbins=200),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed kinds: odd, non-square grids over the whole
    range, any of the precisions, orders and physics options."""
    kind = rng.choice(["run", "run", "run", "run", "fields", "monopole", "ensemble", "load", "diagnostics"])
    if kind == "ensemble":
        c = dict(kind="ensemble", n_inst=rng.randint(2, 7), config_seed=rng.randint(1, 10 ** 6), n_lo=20_000,
                 n_hi=_log_int(rng, 100_000, 3_000_000), rows="100,256,333,512", cols="96,128,250,401", sort_every=16,
                 steps=5)
        return c
    nr = _log_int(rng, 40, 2048)
    nt = max(32, min(2048, _log_int(rng, 0.5 * nr, 1.5 * nr)))
    if kind == "fields":
        c = _run("", nr, nt, 0, r_max=50.0 / 3.0, r_lc=5.0, geom="monopole", sort_every=0, steps=rng.choice([1, 2, 4]),
                 precision=rng.choice(["fp32", "fp32", "fp64"]))
    else:
        fp64 = kind == "run" and nr * nt < 400_000 and rng.random() < 0.4
        pairs = int(nr * nt * math.exp(rng.uniform(math.log(0.3), math.log(8.0 if not fp64 else 3.0))))
        shape = rng.choice([dict(tile_t=32, sort_every=8, steps=2), dict(tile_t=24, sort_every=12, steps=3)])
        if kind == "monopole":
            c = _run("", nr, nt, pairs, r_max=50.0 / 3.0, r_lc=5.0, geom="monopole", **shape)
        else:
            rr = rng.random() < 0.5
            r_lc = rng.uniform(3.0, 10.0)
            c = _run("", nr, nt, pairs, r_max=10.0 * r_lc, r_lc=r_lc, kappa=1.0 if rr else 10.0, rr=rr,
                     geom=rng.choice(["synth", "synth", "dipole"]), momenta="powerlaw" if rr else "maxwell",
                     precision="fp64" if fp64 else "fp32", order=rng.choice(["scattered", "scattered", "cell"]),
                     **shape)
            if kind == "run" and rr and rng.random() < 0.25:
                # rare enough that the events of a step keep their order
                c.update(species=3, gamma_th=max(50.0, 2.0 * pairs / 2500.0), capacity=pairs + pairs // 2 + 50_000)
            if kind == "load":
                c["kind"] = "load"
            if kind == "diagnostics":
                c.update(kind="diagnostics", nbins=rng.choice([64, 200, 500]))
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs
def _config(case):
    """hff configuration dict of a case: the scale separation follows the
    workloads (omega_pe dt = 1/8 at kappa n_GJ)."""
    nr, nt, r_max, r_lc, kappa = case["nr"], case["nt"], case["r_max"], case["r_lc"], case["kappa"]
    dlog, dth = math.log(r_max) / nr, math.pi / nt
    dt = 0.5 / math.sqrt(1.0 / (math.exp(dlog) - 1.0) ** 2 + 1.0 / dth ** 2)
    omega, wpe = 1.0 / r_lc, 1.0 / (8.0 * dt)
    m_e = 4.0 * math.pi * kappa * (omega / (2.0 * math.pi)) / wpe ** 2
    crust = case["species"] == 3
    cap = case["capacity"] or case["pairs"] + case["pairs"] // 20 + (20_000 if case["pairs"] else 0)
    cfg = dict(nr=nr, nt=nt, r_min=1.0, r_max=r_max, r_lc=r_lc, b_star=1.0, geom=case["geom"], courant=0.5,
               r_abs=min(3.0 * r_lc, math.exp(dlog * (nr - 4))), absorb_strength=0.1, psi_break=[], f_break=[],
               q=[-1.0, 1.0, 1.0][:case["species"]], m=[m_e, m_e, 1836.0 * m_e][:case["species"]],
               inject_species=[0, 2 if crust else 1], inject=case["pairs"] > 0, kappa_inj=kappa,
               w_inj=kappa * omega * dlog * dth / 4.0,
               gamma_rad=0.05 * omega ** 2 / m_e if case["rr"] else 0.0, b_ref=omega ** 3, rr_scale=1.0, shell_r=2.0,
               synth_psi_open=1.25, seed=1234, capacity=cap, tile_r=case["tile_r"], tile_t=case["tile_t"],
               sort_every=case["sort_every"], precision=case["precision"], gamma_th=case["gamma_th"],
               gamma_s=0.22 * case["gamma_th"])
    if case["geom"] == "synth":
        cfg.update(psi_break=list(BANDS[0]), f_break=list(BANDS[1]))
    elif case["geom"] == "monopole":
        cut = 1.0 - 1e-4
        cfg.update(psi_break=[cut, cut], f_break=[0.0, 1.0])
    return cfg


def _members(case):
    """Cases of the instances of an ensemble case."""
    import random
    rng = random.Random(case["config_seed"])
    rows, cols = ([int(x) for x in case[k].split(",")] for k in ("rows", "cols"))
    out = []
    for _ in range(case["n_inst"]):
        r_lc = rng.uniform(3.0, 10.0)
        out.append(_run("", rng.choice(rows), rng.choice(cols), _log_int(rng, case["n_lo"], case["n_hi"]) // 2,
                        r_max=10.0 * r_lc, r_lc=r_lc, tile_t=32, sort_every=case["sort_every"], steps=case["steps"]))
    return out


def _shape(name, nr, nt):
    return {"E_r": (nr, nt + 1), "E_th": (nr + 1, nt), "E_ph": (nr + 1, nt + 1), "B_r": (nr + 1, nt),
            "B_th": (nr, nt + 1), "B_ph": (nr, nt)}[name]


def _psi_analytic(cfg, r, t):
    """Flux function of the initial field (Eqs. 32, 37 and their blend)."""
    g = cfg["geom"]
    if g == "dipole":
        return torch.sin(t) ** 2 / r
    if g == "monopole":
        return (1.0 - torch.cos(t)) * torch.ones_like(r)
    w = 0.5 * (1.0 - torch.tanh((r - cfg["r_lc"]) / (0.2 * cfg["r_lc"])))
    popen = cfg["synth_psi_open"] / cfg["r_lc"]
    return w * torch.sin(t) ** 2 / r + (1.0 - w) * popen * (1.0 - torch.abs(torch.cos(t)))


def _particles(cfg, case, g):
    """Species dicts on the GPU (working precision): pairs placed in the PIC
    region inside the absorber, a fifth in the equatorial sheet beyond R_LC,
    the species at the same places with their own momenta."""
    nr, nt, n = cfg["nr"], cfg["nt"], case["pairs"]
    real = torch.float64 if cfg["precision"] == "fp64" else torch.float32
    dlog, dth = math.log(cfg["r_max"]) / nr, math.pi / nt
    i_abs = int(math.log(cfg["r_abs"]) / dlog) - 1
    rows = torch.arange(nr, device=DEV, dtype=torch.float64)
    inside = (rows >= 1) & (rows < i_abs)
    rc = torch.exp((rows + 0.5) * dlog)
    ok = inside[:, None].expand(nr, nt)
    if cfg["psi_break"]:
        tc = (torch.arange(nt, device=DEV, dtype=torch.float64) + 0.5) * dth
        psi = _psi_analytic(cfg, rc[:, None], tc[None, :])
        unit = 1.0 / cfg["r_lc"] if case["geom"] == "synth" else 1.0
        lo = cfg["psi_break"][0] * unit if case["geom"] == "synth" else -1.0
        ok = ok & (psi > lo) & (psi < cfg["psi_break"][-1] * unit)
    cells = torch.nonzero(ok.reshape(-1))[:, 0].to(torch.int32)
    sheet = torch.zeros(nr, nt, dtype=torch.bool, device=DEV)
    sheet[:, nt // 2 - 6:nt // 2 + 6] = ((rc > cfg["r_lc"]) & inside)[:, None]
    sheet_cells = torch.nonzero((sheet & ok).reshape(-1))[:, 0].to(torch.int32)
    ns = n // 5 if case["geom"] == "synth" and len(sheet_cells) else 0

    def rand(*shape):
        return torch.rand(*shape, generator=g, device=DEV)

    ppc = max(1.0, 2.0 * n / max(1, len(cells)))

    def places():
        cell = cells[torch.randint(0, len(cells), (n,), generator=g, device=DEV)]
        if ns:
            cell[n - ns:] = sheet_cells[torch.randint(0, len(sheet_cells), (ns,), generator=g, device=DEV)]
        if case["order"] == "cell":
            cell = cell.sort()[0]
        xo, yo = rand(n), rand(n)
        i, j = torch.div(cell, nt, rounding_mode="floor"), torch.remainder(cell, nt)
        w = torch.exp((i + xo) * dlog) * torch.clamp(torch.sin((j + yo) * dth), min=0.5 * dth)
        return cell, xo, yo, w * (cfg["kappa_inj"] / cfg["r_lc"] * dlog * dth / ppc)

    out = []
    for s in range(case["species"]):
        if s == 0 or case["kind"] == "diagnostics":  # a run under way has separated its charges
            cell, xo, yo, w = places()
        if case["momenta"] == "powerlaw":  # dN/dgamma ~ gamma^-2 on [1, 1e6], isotropic
            gam = 1.0 / (1.0 - rand(n) * (1.0 - 1e-6))
            p = torch.sqrt(torch.clamp(gam * gam - 1.0, min=0.0))
            mu, ph = 2.0 * rand(n) - 1.0, 2.0 * math.pi * rand(n)
            st = p * torch.sqrt(1.0 - mu * mu)
            u = [p * mu, st * torch.cos(ph), st * torch.sin(ph)]
        else:
            u = [torch.randn(n, generator=g, device=DEV) for _ in range(3)]
        d = dict(zip(("ur", "ut", "up"), u), cell=cell, xo=xo, yo=yo, w=w)
        out.append({k: v.to(real) if k != "cell" else v for k, v in d.items()})
    return out


def _fields(cfg, g):
    """E and B_ph of a run under way: a few smooth modes and 10% noise, scaled
    like 1/r^2, tangential E zero on the walls."""
    nr, nt = cfg["nr"], cfg["nt"]
    real = torch.float64 if cfg["precision"] == "fp64" else torch.float32
    out = {}
    for name in ("E_r", "E_th", "E_ph", "B_ph"):
        shp = _shape(name, nr, nt)
        x = torch.linspace(0.0, 1.0, shp[0], device=DEV)[:, None]
        y = torch.linspace(0.0, 1.0, shp[1], device=DEV)[None, :]
        c = torch.rand(9, generator=g, device=DEV).tolist()
        a = 0.3 * torch.randn(shp, generator=g, device=DEV)
        for k in range(3):
            a += (2.0 * c[3 * k] - 1.0) * torch.sin(2 * math.pi * ((k + 1) * x + c[3 * k + 1])) * torch.sin(
                math.pi * ((k + 1) * y + c[3 * k + 2]))
        a *= (0.05 / 3.0) * torch.exp(-2.0 * math.log(cfg["r_max"]) * x)
        if name == "E_ph":
            a[0], a[-1], a[:, 0], a[:, -1] = 0, 0, 0, 0
        if name == "E_th":
            a[-1] = 0
        out[name] = a.to(real)
    return out


def _inputs(case, seed, inst=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(1_000_003 * int(seed) + 7919 * inst + 17)
    cfg = _config(case)
    f = _fields(cfg, g)
    return cfg, (_particles(cfg, case, g) if case["pairs"] else []), f


# -------------------------------------------------------------------- runs
def _give(sim, inst, parts, fields):
    for s, p in enumerate(parts):
        sim.load_device(s, p)
    for name, a in fields.items():
        hff.hff_set_field(sim.h, inst, hff.FIELDS.index(name), a.data_ptr(), a.numel() * a.element_size(), hff.DEVICE)


def prepare(case, seed):
    if case["kind"] == "ensemble":
        mem = _members(case)
        made = [_inputs(c, seed, k) for k, c in enumerate(mem)]
        ens = hff.Ensemble([m[0] for m in made], device=DEV)
        for k, (_, parts, fields) in enumerate(made):
            _give(ens[k], k, parts, fields)
        size = {n: [math.prod(_shape(n, c["nr"], c["nt"])) for c in mem] for n in FIELDS6}
        out = {n: torch.empty(sum(size[n]), device=DEV) for n in FIELDS6}
        return dict(case=case, ens=ens, n=[c["pairs"] for c in mem], flat=out,
                    out={n: list(out[n].split(size[n])) for n in FIELDS6})
    cfg, parts, fields = _inputs(case, seed)
    sim = hff.Sim(cfg, device=DEV)
    st = dict(case=case, sim=sim)
    if case["kind"] == "load":
        st["parts"] = parts
        return st
    _give(sim, 0, parts, fields)
    st["out"] = {n: torch.empty(_shape(n, cfg["nr"], cfg["nt"]), dtype=sim.tdtype, device=DEV) for n in FIELDS6}
    return st


def _read_fields(h, inst, out):
    for name, a in out.items():
        hff.hff_fields(h, inst, hff.FIELDS.index(name), a.data_ptr(), a.numel() * a.element_size(), hff.DEVICE)


def _positions(v, nt):
    """Logical coordinates (row + xo, column + yo): continuous across cells."""
    return [torch.div(v["cell"], nt, rounding_mode="floor") + v["xo"], torch.remainder(v["cell"], nt) + v["yo"]]


def _whole(arrays, n, case):
    """The arrays of one species: the first n slots of each, and the later
    slots of all of them (particles created since the load) in one array with
    room for more.  A pass that sorts compacts the removed particles: there
    the first n slots are filled up with zeros, so that shapes are the same
    for all inputs."""
    used, extra = len(arrays[0]), 20_000 + n // 50
    tail = torch.zeros(len(arrays), max(extra, used - n), dtype=arrays[0].dtype, device=arrays[0].device)
    if used > n:
        tail[:, :used - n] = torch.stack([a[n:] for a in arrays])
    if used < n and case["steps"] >= case["sort_every"]:
        return [*torch.nn.functional.pad(torch.stack(arrays), (0, n - used)), tail]
    return [a[:n] for a in arrays] + [tail]


def run(st):
    case = st["case"]
    if case["kind"] == "load":
        sim = st["sim"]
        for s, p in enumerate(st["parts"]):
            sim.load_device(s, p)
        return [sim.particle_views(s) for s in range(case["species"])]
    if case["kind"] == "diagnostics":
        sim = st["sim"]
        d, prof = sim.diagnostics()
        maps = [sim.species_maps(s) for s in range(2)]
        spec = [sim.spectrum(s, case["nbins"], 0.0, 7.0) for s in range(2)]
        num = {k: float(getattr(d, k)) for k in ("psi_open", "l_in", "l_out", "gauss_max", "gauss_rms", "rho_max",
                                                  "u_e", "u_b")}
        return dict(num, kinetic=list(d.kinetic)[:2], count=list(d.count)[:2], L=prof, maps=maps, spectra=spec)
    if case["kind"] == "ensemble":
        ens = st["ens"]
        ens.step(case["steps"])
        parts = []
        for k in range(len(ens)):
            _read_fields(ens.h, k, {n: st["out"][n][k] for n in FIELDS6})
            views = [ens[k].particle_views(s) for s in range(2)]
            parts.append([_whole([v[u] for u in ("ur", "ut", "up")], st["n"][k], case) for v in views])
        return dict(fields=st["flat"], particles=parts)
    sim = st["sim"]
    sim.step(case["steps"])
    _read_fields(sim.h, 0, st["out"])
    parts = []
    if case["pairs"]:
        for s in range(case["species"]):
            v = sim.particle_views(s)
            parts.append(_whole(_positions(v, case["nt"]) + [v["ur"], v["ut"], v["up"]], case["pairs"], case))
    return dict(fields=st["out"], particles=parts)


def work(case):
    """Bytes: per step, each live particle's seven words read and six written
    (the weight is kept), and per cell E, B read and written, B_0 and its curl
    read; a load moves the seven words once; the diagnostics read particles
    and fields and write the maps.  Flops: additions and multiplications of
    the gather, push, move and deposit per particle and of the field update
    per cell, counted in the formulas."""
    if case["kind"] == "ensemble":
        w = [work(c) for c in _members(case)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    word = 8 if case["precision"] == "fp64" else 4
    n, cells = case["pairs"] * case["species"], case["nr"] * case["nt"]
    if case["kind"] == "load":
        return dict(bytes=2.0 * n * (4 + 6 * word), flops=0.0)
    if case["kind"] == "diagnostics":
        return dict(bytes=n * (4 + 6.0 * word) + cells * (9 * word + 4 * 8.0), flops=60.0 * n + 120.0 * cells)
    k = case["steps"]
    return dict(bytes=k * (n * (8 + 11.0 * word) + cells * 18.0 * word),
                flops=k * ((460.0 if case["rr"] else 360.0) * n + 260.0 * cells))


# ------------------------------------------------------- the step in float64
class _Grid:
    def __init__(self, cfg):
        nr, nt = self.nr, self.nt = cfg["nr"], cfg["nt"]
        self.dlog, self.dth = math.log(cfg["r_max"]) / nr, math.pi / nt
        i = torch.arange(nr + 1, device=DEV, dtype=torch.float64)
        j = torch.arange(nt + 1, device=DEV, dtype=torch.float64)
        self.rn, self.rh = torch.exp(i * self.dlog), torch.exp((i[:-1] + 0.5) * self.dlog)
        one, top = torch.ones(1, device=DEV, dtype=torch.float64), self.rn[-1:]
        self.rlo, self.rhi = torch.cat([one, self.rh]), torch.cat([self.rh, top])
        self.tn, self.th = j * self.dth, (j[:-1] + 0.5) * self.dth
        self.tlo = torch.cat([0 * one, self.th])
        self.thi = torch.cat([self.th, math.pi * one])
        self.sn, self.sh = torch.sin(self.tn), torch.sin(self.th)
        self.dcp = torch.cos(self.tn[:-1]) - torch.cos(self.tn[1:])
        self.dch = torch.cos(self.tlo) - torch.cos(self.thi)
        self.vol_n = (2 * math.pi / 3) * (self.rhi ** 3 - self.rlo ** 3)[:, None] * self.dch[None]
        # Courant condition at the innermost cell (the smallest)
        dr, rt = self.rn[1:] - self.rn[:-1], self.rn[:-1] * self.dth
        self.dt = cfg["courant"] * float((1.0 / torch.sqrt(1.0 / dr ** 2 + 1.0 / rt ** 2)).min())
        self.xi_abs = math.log(cfg["r_abs"]) / self.dlog
        span = cfg["r_max"] - cfg["r_abs"]

        def sig(r):
            return cfg["absorb_strength"] * torch.clamp((r - cfg["r_abs"]) / span, min=0.0) ** 3

        self.sig_n, self.sig_h = sig(self.rn)[:, None], sig(self.rh)[:, None]


class _Exact:
    """The hybrid step in float64 on whole arrays."""
    CHUNK = 10_000_000

    def __init__(self, cfg, parts, fields):
        self.c, self.g = cfg, _Grid(cfg)
        g = self.g
        psi = _psi_analytic(cfg, g.rn[:, None], g.tn[None, :])
        br = (psi[:, 1:] - psi[:, :-1]) / (g.rn[:, None] ** 2 * g.dcp)
        bt = torch.zeros(g.nr, g.nt + 1, device=DEV, dtype=torch.float64)
        area = g.sn[None, 1:-1] * (g.rn[1:] ** 2 - g.rn[:-1] ** 2)[:, None]
        bt[:, 1:-1] = -2.0 * (psi[1:, 1:-1] - psi[:-1, 1:-1]) / area
        f = {k: v.double() for k, v in fields.items()}
        self.E = [f["E_r"], f["E_th"], f["E_ph"]]
        self.B0 = [br, bt, torch.zeros_like(f["B_ph"])]
        self.B = [br.clone(), bt.clone(), f["B_ph"]]
        self.unit = 1.0 if cfg["geom"] == "monopole" else 1.0 / cfg["r_lc"]
        self.step_no = 0
        self.tn = (cfg["nt"] + cfg["tile_t"] - 1) // cfg["tile_t"]
        self.P = [{k: (v.double() if k != "cell" else v.long()) for k, v in p.items()} for p in parts]
        for s in range(len(self.P)):
            if cfg["sort_every"]:
                self.sort(s)
        self.target = self._targets(br[0]) if cfg["inject"] else None

    # ------------------------------------------------------------- particles
    def sort(self, s):
        p, c = self.P[s], self.c
        cell = p["cell"]
        i, j = torch.div(cell, c["nt"], rounding_mode="floor"), torch.remainder(cell, c["nt"])
        key = torch.div(i, c["tile_r"], rounding_mode="floor") * self.tn
        key += torch.div(j, c["tile_t"], rounding_mode="floor")
        key[cell < 0] = 1 << 40
        live = int((cell >= 0).sum())
        o = torch.argsort(key, stable=True)[:live]
        self.P[s] = {k: v[o] for k, v in p.items()}

    def _targets(self, br0):
        c, g = self.c, self.g
        p = torch.cumsum(br0 * g.dcp, 0)
        fs = self.blend(0.5 * (p + torch.cat([p.new_zeros(1), p[:-1]])))
        ngj = br0.abs() / c["r_lc"] / (2 * math.pi)
        v = 2 * math.pi / 3 * (g.rn[1] ** 3 - g.rn[0] ** 3) * g.dcp
        return torch.where(fs < 1.0, torch.floor(c["kappa_inj"] * ngj * v / c["w_inj"] + 0.5), 0.0 * v).long()

    def blend(self, psi):
        x, y = [b * self.unit for b in self.c["psi_break"]], self.c["f_break"]
        if not x:
            return torch.zeros_like(psi)
        f = torch.full_like(psi, y[-1])
        for k in range(len(x) - 1, 0, -1):
            slope = (y[k] - y[k - 1]) / (x[k] - x[k - 1]) if x[k] > x[k - 1] else 0.0
            f = torch.where(psi < x[k], y[k - 1] + slope * (psi - x[k - 1]), f)
        return torch.where(psi < x[0], torch.full_like(psi, y[0]), f)

    @staticmethod
    def _lin(c, o, half, n):
        """First index and weight of linear interpolation on nodes (or half
        nodes, constant beyond the ends) of n points."""
        x = c + o - (0.5 if half else 0.0)
        k = torch.clamp(torch.floor(x).long(), 0, n - 2)
        return k, torch.clamp(x - k, 0.0, 1.0)

    def _push(self, s, p, J, ff, surf):
        c, g = self.c, self.g
        nr, nt, dt = g.nr, g.nt, g.dt
        cell, xo, yo = p["cell"], p["xo"], p["yo"]
        i, j = torch.div(cell, nt, rounding_mode="floor"), torch.remainder(cell, nt)
        kin, kih, kjn, kjh = (self._lin(i, xo, 0, nr + 1), self._lin(i, xo, 1, nr), self._lin(j, yo, 0, nt + 1),
                              self._lin(j, yo, 1, nt))

        def at(a, kr, kt):
            (k, w), (m, v), ld, a = kr, kt, a.shape[1], a.reshape(-1)
            b = k * ld + m
            return (1 - w) * ((1 - v) * a[b] + v * a[b + 1]) + w * ((1 - v) * a[b + ld] + v * a[b + ld + 1])

        E = torch.stack([at(self.E[0], kih, kjn), at(self.E[1], kin, kjh), at(self.E[2], kin, kjn)])
        B = torch.stack([at(self.B[0], kin, kjh), at(self.B[1], kih, kjn), at(self.B[2], kih, kjh)])
        u = torch.stack([p["ur"], p["ut"], p["up"]])

        def dot(a, b):
            return (a * b).sum(0)

        def cross(a, b):
            return torch.stack([a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]])

        qm = c["q"][s] / c["m"][s]
        h = 0.5 * qm * dt
        um = u + h * E
        t = h * B / torch.sqrt(1 + dot(um, um))
        ul = um + cross(um + cross(um, t), 2 * t / (1 + dot(t, t))) + h * E
        un = ul
        if c["gamma_rad"] > 0:  # Eqs. 16, 17 at the centred momentum, limited to half of |u|
            ratio = (c["q"][s] ** 2 / c["m"][s]) / (c["q"][0] ** 2 / c["m"][0])
            K = abs(c["q"][0]) / (c["gamma_rad"] ** 2 * c["b_ref"]) * ratio ** 2 / c["m"][s] * c["rr_scale"]
            ub = 0.5 * (u + ul)
            g2 = 1 + dot(ub, ub)
            be = ub / torch.sqrt(g2)
            F = E + cross(be, B)
            FxB = cross(F, be)
            bp2 = dot(FxB, FxB) + dot(F, F) / g2
            du = dt * K * (cross(F, B) + dot(be, E) * E - g2 * bp2 * be)
            ratio = torch.sqrt(dot(du, du) / torch.clamp(dot(ul, ul), min=1e-300))
            un = ul + du * torch.where(ratio > 0.5, 0.5 / ratio, torch.ones_like(ratio))
        r, th = torch.exp((i + xo) * g.dlog), (j + yo) * g.dth
        near = (r < c["shell_r"]) & (dot(B, B) > 1e-30)
        un = torch.where(near, B * (dot(un, B) / torch.clamp(dot(B, B), min=1e-30)), un)
        gam = torch.sqrt(1 + dot(un, un))
        v = un / gam
        # straight line from azimuth 0 in cylindrical coordinates
        sn, cs = torch.sin(th), torch.cos(th)
        vR, vz = v[0] * sn + v[1] * cs, v[0] * cs - v[1] * sn
        x, y, z = r * sn + vR * dt, v[2] * dt, r * cs + vz * dt
        R = torch.sqrt(x * x + y * y)
        rnew, tnew = torch.sqrt(R * R + z * z), torch.atan2(R, z)
        cp, sp = x / R, y / R
        uR, uz = un[0] * sn + un[1] * cs, un[0] * cs - un[1] * sn
        uR2, up2 = uR * cp + un[2] * sp, un[2] * cp - uR * sp
        s1, c1 = R / rnew, z / rnew
        X1, Y1 = xo + torch.log(rnew / r) / g.dlog, yo + (tnew - th) / g.dth
        dead = (i + X1 < 0) | (i + X1 > g.xi_abs)
        X1 = torch.maximum(X1, -i.double())
        i1 = torch.clamp(i + torch.floor(X1).long(), 0, nr - 1)
        j1 = torch.clamp(j + torch.floor(Y1).long(), 0, nt - 1)
        dead |= ff.reshape(-1)[i1 * nt + j1]
        self._deposit(c["q"][s] * p["w"], i, j, xo, yo, X1, Y1, v[2], J)
        if surf is not None:
            surf.index_add_(0, j1[(i1 == 0) & ~dead], torch.ones_like(j1[(i1 == 0) & ~dead]))
        new = dict(cell=i1 * nt + j1, xo=i + X1 - i1, yo=j + Y1 - j1, ur=uR2 * s1 + uz * c1,
                   ut=uR2 * c1 - uz * s1, up=up2)
        for k, a in new.items():
            a = torch.where(dead, torch.full_like(a, -1) if k == "cell" else p[k], a)
            p[k].copy_(a)
        if c["gamma_th"] > 0 and s < 2:
            uu = 1 + new["ur"] ** 2 + new["ut"] ** 2 + new["up"] ** 2
            e = torch.nonzero((uu > c["gamma_th"] ** 2) & ~dead)[:, 0]
            a = math.sqrt(max(c["gamma_s"] ** 2 - 1, 0)) / torch.sqrt(uu[e] - 1)
            born = {k: p[k][e].clone() for k in p}
            for k in ("ur", "ut", "up"):
                born[k] *= a
            return born
        return None

    def _deposit(self, q, i, j, x0, y0, X1, Y1, vphi, J):
        """Esirkepov: fluxes through the dual faces from the change of the
        cloud-in-cell weights on the nodes -1 .. 2 around the start cell."""
        nr, nt = self.g.nr, self.g.nt

        def weights(a0, a1):
            k = torch.arange(-1, 3, device=DEV, dtype=torch.float64)[:, None]
            return [torch.clamp(1 - (k - a).abs(), min=0.0) for a in (a0, a1)]

        (sx0, sx1), (sy0, sy1) = weights(x0, X1), weights(y0, Y1)
        fx, fy = -torch.cumsum(sx1 - sx0, 0), -torch.cumsum(sy1 - sy0, 0)
        mx, my = 0.5 * (sx0 + sx1), 0.5 * (sy0 + sy1)

        def add(a, rows, cols, val):
            m = torch.nonzero(val)[:, 0]
            a.reshape(-1).index_add_(0, rows[m] * a.shape[1] + cols[m], val[m])

        for a in range(3):  # faces between the nodes a - 1 and a of the window
            for b in range(4):
                add(J[0], i + a - 1, j + b - 1, q * fx[a] * my[b])
                add(J[1], i + b - 1, j + a - 1, q * fy[a] * mx[b])
        xm, ym = 0.5 * (x0 + X1), 0.5 * (y0 + Y1)
        k, m = torch.floor(xm), torch.floor(ym)
        wx, wy = xm - k, ym - m
        for a in (0, 1):
            for b in (0, 1):
                add(J[2], torch.clamp(i + k.long() + a, max=nr), torch.clamp(j + m.long() + b, max=nt),
                    q * vphi * (wx if a else 1 - wx) * (wy if b else 1 - wy))

    # ---------------------------------------------------------------- fields
    def _nodes(self, E, B):
        """E and B at the nodes of the interior rows (arithmetic means,
        transverse parts zero on the axis)."""
        e = torch.zeros(3, self.g.nr - 1, self.g.nt + 1, device=DEV, dtype=torch.float64)
        b = torch.zeros_like(e)
        e[0] = 0.5 * (E[0][:-1] + E[0][1:])
        e[1][:, 1:-1] = 0.5 * (E[1][1:-1, :-1] + E[1][1:-1, 1:])
        e[2][:, 1:-1] = E[2][1:-1, 1:-1]
        br = B[0][1:-1]
        b[0][:, 0], b[0][:, -1], b[0][:, 1:-1] = br[:, 0], br[:, -1], 0.5 * (br[:, :-1] + br[:, 1:])
        b[1][:, 1:-1] = 0.5 * (B[1][:-1, 1:-1] + B[1][1:, 1:-1])
        bp = B[2]
        b[2][:, 1:-1] = 0.25 * (bp[:-1, :-1] + bp[:-1, 1:] + bp[1:, :-1] + bp[1:, 1:])
        return e, b

    def _edges_r(self, a):
        """Node values of the interior rows at the radial edges (the mean of
        the edge's interior nodes)."""
        return torch.cat([a[:1], 0.5 * (a[:-1] + a[1:]), a[-1:]])

    def _faraday(self, h):
        g, (er, et, ep) = self.g, self.E
        rn, rdr = g.rn[:, None], 2.0 / (g.rn[1:] ** 2 - g.rn[:-1] ** 2)[:, None]
        self.B[0] = self.B[0] - h * (g.sn[1:] * ep[:, 1:] - g.sn[:-1] * ep[:, :-1]) / (rn * g.dcp)
        bt = self.B[1] + h * rdr * (rn[1:] * ep[1:] - rn[:-1] * ep[:-1])
        bt[:, 0], bt[:, -1] = 0, 0
        self.B[1] = bt
        dr = (g.rn[1:] - g.rn[:-1])[:, None]
        cu = (rn[1:] * et[1:] - rn[:-1] * et[:-1]) - dr / g.dth * (er[:, 1:] - er[:, :-1])
        self.B[2] = self.B[2] - h * rdr * cu

    def step(self):
        c, g = self.c, self.g
        psi = torch.zeros(g.nr + 1, g.nt + 1, device=DEV, dtype=torch.float64)
        psi[:, 1:] = torch.cumsum(self.B[0] * g.dcp, 1) * g.rn[:, None] ** 2
        ff = self.blend(0.25 * (psi[:-1, :-1] + psi[1:, :-1] + psi[:-1, 1:] + psi[1:, 1:])) >= 1.0
        # J_perp = rho E x B / B^2 at the interior nodes
        E = self.E
        ar = 2 * math.pi * g.rh[:, None] ** 2 * g.dch * E[0]
        at = math.pi * (g.rhi ** 2 - g.rlo ** 2)[1:-1, None] * g.sh * E[1][1:-1]
        flux = ar[1:] - ar[:-1]
        flux[:, :-1] += at
        flux[:, 1:] -= at
        rho = flux / (4 * math.pi * g.vol_n[1:-1])
        e, b = self._nodes(E, self.B)
        b2 = (b * b).sum(0)
        jp = torch.where(b2 > 1e-30, rho / torch.clamp(b2, min=1e-30), 0 * b2) * torch.stack(
            [e[1] * b[2] - e[2] * b[1], e[2] * b[0] - e[0] * b[2], e[0] * b[1] - e[1] * b[0]])
        # particles
        J = [torch.zeros_like(x) for x in self.E]
        surf = torch.zeros(g.nt, device=DEV, dtype=torch.long) if c["inject"] else None
        born = []
        for s, p in enumerate(self.P):
            for k in range(0, len(p["cell"]), self.CHUNK):
                q = {n: a[k:k + self.CHUNK] for n, a in p.items()}
                live = torch.nonzero(q["cell"] >= 0)[:, 0]
                part = q if len(live) == len(q["cell"]) else {n: a[live] for n, a in q.items()}
                got = self._push(s, part, J, ff, surf)
                if part is not q:
                    for n in q:
                        q[n][live] = part[n]
                if got is not None:
                    born.append(got)
        J[0] /= 2 * math.pi * g.rh[:, None] ** 2 * g.dt * g.dch
        J[1] /= math.pi * (g.rhi ** 2 - g.rlo ** 2)[:, None] * g.dt * g.sh
        J[2] /= g.vol_n
        # Faraday, Ampere with J = (1 - f) J_PIC + f J_perp, boundaries, absorber
        self._faraday(0.5 * g.dt)
        fr, ft = self.blend(0.5 * (psi[:-1] + psi[1:])), self.blend(0.5 * (psi[:, :-1] + psi[:, 1:]))
        fn = self.blend(psi)
        br, bt, bp = self.B
        dt, fp = g.dt, 4 * math.pi * g.dt
        cur = torch.zeros_like(E[0])
        cur[:, :-1] += g.sh * bp
        cur[:, 1:] -= g.sh * bp
        cur /= g.rh[:, None] * g.dch
        er = (E[0] + dt * cur - fp * ((1 - fr) * J[0] + fr * self._edges_r(jp[0]))) * (1 - g.sig_h)
        ce = 2.0 / (g.rhi ** 2 - g.rlo ** 2)[1:-1, None]
        rh = g.rh[:, None]
        et = torch.zeros_like(E[1])
        et[0] = -g.rn[0] / c["r_lc"] * g.sh * br[0]
        jt = (1 - ft[1:-1]) * J[1][1:-1] + ft[1:-1] * 0.5 * (jp[1][:, :-1] + jp[1][:, 1:])
        et[1:-1] = (E[1][1:-1] - dt * ce * (rh[1:] * bp[1:] - rh[:-1] * bp[:-1]) - fp * jt) * (1 - g.sig_n[1:-1])
        ep = torch.zeros_like(E[2])
        dr = (g.rhi - g.rlo)[1:-1, None]
        cu = ce * ((rh[1:] * bt[1:] - rh[:-1] * bt[:-1])[:, 1:-1] - dr / g.dth * (br[1:-1, 1:] - br[1:-1, :-1]))
        f1 = fn[1:-1, 1:-1]
        jn = (1 - f1) * J[2][1:-1, 1:-1] + f1 * jp[2][:, 1:-1]
        ep[1:-1, 1:-1] = (E[2][1:-1, 1:-1] + dt * cu - fp * jn) * (1 - g.sig_n[1:-1])
        # E.B = 0 and E^2 <= B^2 at the nodes, returned with the weight f
        e, b = self._nodes([er, et, ep], self.B)
        b2 = torch.clamp((b * b).sum(0), min=1e-30)
        d = e - b * ((e * b).sum(0) / b2)
        d2 = (d * d).sum(0)
        d = d * torch.where(d2 > b2, torch.sqrt(b2 / torch.clamp(d2, min=1e-300)), torch.ones_like(d2))
        d = torch.where((b * b).sum(0) > 1e-30, d, e)
        er = er + fr * (self._edges_r(d[0]) - er)
        et[1:-1] += ft[1:-1] * (0.5 * (d[1][:, :-1] + d[1][:, 1:]) - et[1:-1])
        ep[1:-1, 1:-1] += f1 * (d[2][:, 1:-1] - ep[1:-1, 1:-1])
        self.E = [er, et, ep]
        self._faraday(0.5 * g.dt)
        for k, sg in enumerate((g.sig_n, g.sig_h, g.sig_h)):
            self.B[k] = self.B[k] - sg * (self.B[k] - self.B0[k])
        if c["inject"]:
            self._inject(surf)
        if born:
            new = {k: torch.cat([x[k] for x in born]) for k in born[0]}
            for s in (0, 1):
                self.P[s] = {k: torch.cat([v, new[k]]) for k, v in self.P[s].items()}
        self.step_no += 1
        if c["sort_every"] and self.step_no % c["sort_every"] == 0:
            for s in range(len(self.P)):
                self.sort(s)

    def _inject(self, surf):
        """Top-up of the surface cells by co-located corotating pairs; offsets
        from Philox4x32-10 keyed (seed; step, column, index)."""
        c, g = self.c, self.g
        need = torch.clamp(self.target - torch.div(surf, 2, rounding_mode="floor"), min=0).cpu().numpy()
        j = np.repeat(np.arange(g.nt), need)
        k = np.concatenate([np.arange(n) for n in need]) if len(j) else j
        w32 = np.uint64(0xFFFFFFFF)
        x = [np.full(len(j), self.step_no, np.uint64), np.zeros(len(j), np.uint64), j.astype(np.uint64),
             k.astype(np.uint64)]
        k0, k1 = c["seed"] & 0xFFFFFFFF, c["seed"] >> 32
        for _ in range(10):
            a, b = x[0] * np.uint64(0xD2511F53), x[2] * np.uint64(0xCD9E8D57)
            x = [(b >> np.uint64(32)) ^ x[1] ^ np.uint64(k0), b & w32, (a >> np.uint64(32)) ^ x[3] ^ np.uint64(k1),
                 a & w32]
            k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
        ox, oy = ((x[q] >> np.uint64(8)).astype(np.float64) / 16777216.0 for q in (0, 1))
        v = np.exp(ox * g.dlog) * np.sin((j + oy) * g.dth) / c["r_lc"]
        z = np.zeros(len(j))
        new = dict(cell=j, xo=ox, yo=oy, ur=z, ut=z, up=v / np.sqrt(1 - v * v), w=z + c["w_inj"])
        new = {n: torch.from_numpy(np.ascontiguousarray(a)).to(DEV) for n, a in new.items()}
        for s in c["inject_species"]:
            self.P[s] = {n: torch.cat([a, new[n]]) for n, a in self.P[s].items()}

    # ----------------------------------------------------------- diagnostics
    def diagnostics(self, case):
        c, g, (er, et, ep), (br, bt, bp) = self.c, self.g, self.E, self.B
        rh, rn, pi = g.rh[:, None], g.rn[:, None], math.pi
        L = (0.5 * (et[:-1] + et[1:]) * bp * g.dcp).sum(1) - (0.5 * (ep[:-1] + ep[1:]) * bt * g.dch).sum(1)
        L = L * g.rh ** 2 / 2
        dr, dr2 = (g.rn[1:] - g.rn[:-1])[:, None], (g.rn[1:] ** 2 - g.rn[:-1] ** 2)[:, None]
        dl, dl2 = (g.rhi - g.rlo)[:, None], (g.rhi ** 2 - g.rlo ** 2)[:, None]
        wt = g.thi - g.tlo
        ue = (er ** 2 * 2 * pi * rh ** 2 * g.dch * dr).sum() + (et ** 2 * pi * g.sh * dl2 * rn * g.dth).sum() + (
            ep ** 2 * dl2 * wt * pi * rn * g.sn).sum()
        ub = (br ** 2 * 2 * pi * rn ** 2 * g.dcp * dl).sum() + (bt ** 2 * pi * g.sn * dr2 * rh * wt).sum() + (
            bp ** 2 * dr2 * g.dth * pi * rh * g.sh).sum()
        charge = torch.zeros_like(ep)
        kin, cnt, maps, spec = [], [], [], []
        vol = 2 * pi / 3 * (g.rn[1:] ** 3 - g.rn[:-1] ** 3)[:, None] * g.dcp
        for s, p in enumerate(self.P):
            i, j = torch.div(p["cell"], g.nt, rounding_mode="floor"), torch.remainder(p["cell"], g.nt)
            for a in (0, 1):
                for b in (0, 1):
                    w = (p["xo"] if a else 1 - p["xo"]) * (p["yo"] if b else 1 - p["yo"])
                    charge.reshape(-1).index_add_(0, (i + a) * (g.nt + 1) + j + b, c["q"][s] * p["w"] * w)
            gam = torch.sqrt(1 + p["ur"] ** 2 + p["ut"] ** 2 + p["up"] ** 2)
            ke = p["w"] * c["m"][s] * (gam * gam - 1) / (gam + 1)
            kin.append(float(ke.sum()))
            cnt.append(float(len(gam)))
            m = [torch.zeros(vol.numel(), dtype=vol.dtype, device=DEV).index_add_(0, p["cell"], x) for x in (p["w"], ke)]
            maps.append(tuple((x.reshape(vol.shape) / vol).cpu().numpy() for x in m))
            n = case["nbins"]
            h = torch.clamp(torch.floor(torch.log10(gam) * (n / 7.0)).long(), 0, n - 1)
            spec.append(torch.zeros(n, device=DEV, dtype=torch.float64).index_add_(0, h, p["w"]).cpu().numpy())
        imax = min(int(math.floor(g.xi_abs)) - 2, g.nr - 2)
        ar, at = 2 * pi * rh ** 2 * g.dch * er, pi * dl2[1:-1] * g.sh * et[1:-1]
        flux = ar[1:] - ar[:-1]
        flux[:, :-1] += at
        flux[:, 1:] -= at
        v, q = g.vol_n[2:imax + 1], charge[2:imax + 1]
        res = (flux[1:imax] / (4 * pi) - q) / v
        iout = min(int(math.floor(math.log(2.0 * c["r_lc"]) / g.dlog + 0.5)), g.nr)
        psi = float((br[iout, :g.nt // 2] * g.dcp[:g.nt // 2]).sum() * g.rn[iout] ** 2)
        lin, lout = L[(g.rh >= 1) & (g.rh <= 2)], L[(g.rh >= 2 * c["r_lc"]) & (g.rh <= 3 * c["r_lc"])]
        return dict(psi_open=psi, l_in=float(lin.mean()), l_out=float(lout.mean()), gauss_max=float(res.abs().max()),
                    gauss_rms=float(torch.sqrt((res * res).mean())), rho_max=float((q / v).abs().max()),
                    u_e=float(ue) / (8 * pi), u_b=float(ub) / (8 * pi), kinetic=kin, count=cnt, L=L.cpu().numpy(),
                    maps=maps, spectra=spec)


def exact(case, seed):
    if case["kind"] == "ensemble":
        flat, parts = {n: [] for n in FIELDS6}, []
        for k, c in enumerate(_members(case)):
            x = _Exact(*_inputs(c, seed, k))
            for _ in range(case["steps"]):
                x.step()
            for n, a in zip(FIELDS6, x.E + x.B):
                flat[n].append(a.reshape(-1))
            parts.append([_whole([p[u] for u in ("ur", "ut", "up")], c["pairs"], case) for p in x.P])
        return dict(fields={n: torch.cat(v) for n, v in flat.items()}, particles=parts)
    x = _Exact(*_inputs(case, seed))
    if case["kind"] == "load":
        return [dict(p, cell=p["cell"].int()) for p in x.P]
    if case["kind"] == "diagnostics":
        return x.diagnostics(case)
    for _ in range(case["steps"]):
        x.step()
    parts = [_whole(_positions(p, case["nt"]) + [p["ur"], p["ut"], p["up"]], case["pairs"], case) for p in x.P]
    return dict(fields=dict(zip(FIELDS6, x.E + x.B)), particles=parts)
