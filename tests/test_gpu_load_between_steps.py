"""Loads in the middle of a run: the other species have moved, lost and gained
particles since the last sort, so their tiles are no longer contiguous.  The
load then sorts them along; nothing of their unsorted state may reach the work
list (whose length is bounded for sorted particles only) or the status word."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

KEYS = ("cell", "xo", "yo", "ur", "ut", "up", "w")


def _setup(prec, n_species=2, n_pairs=1_000_000, nr=256, nt=1024):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2406_14512_gb300 import hff, workloads
    cfg = workloads._base(nr, nt, 60.0, 6.0, "synth", seed=77)
    cfg.update(psi_break=list(workloads.TABLE1_PSI), f_break=list(workloads.TABLE1_F), n_pairs=n_pairs, place="band",
               sheet_frac=0.2, momenta="maxwell", precision=prec, capacity=n_pairs + n_pairs // 25, sort_every=8,
               tile_r=16, tile_t=32)
    ps = workloads.particles(cfg, seed=5)
    if n_species == 1:
        cfg.update(q=cfg["q"][:1], m=cfg["m"][:1], inject=False, inject_species=[0, 0])
    return hff, cfg, ps[:n_species]


def _sorted(cfg, p):
    """Live particles in the stable order of their tiles."""
    ntt = -(-cfg["nt"] // cfg["tile_t"])
    key = (p["cell"] // cfg["nt"] // cfg["tile_r"]) * ntt + p["cell"] % cfg["nt"] // cfg["tile_t"]
    live = np.flatnonzero(p["cell"] >= 0)
    o = live[np.argsort(key[live], kind="stable")]
    return {k: p[k][o] for k in KEYS}


def _check(cfg, sim, want):
    assert sim.status() == 0
    for s, w in enumerate(want):
        got = sim.particles(s)
        for k in KEYS:
            assert np.array_equal(got[k], w[k]), (s, k)
    before = sim.info()
    sim.step_stages(1, 5)   # flux prefix, cell flags, push: the work list covers every particle once
    after = sim.info()
    assert after.pushed_tiled - before.pushed_tiled == sum(len(w["cell"]) for w in want)
    assert after.pushed_tail == before.pushed_tail and sim.status() == 0


def _host(sim, n):
    return [{k: v.copy() for k, v in sim.particles(s).items()} for s in range(n)]


@pytest.mark.parametrize("where", ["host", "device"])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_load_in_the_middle_of_a_cadence(prec, where):
    import torch
    hff, cfg, ps = _setup(prec)
    sim = hff.Sim(cfg)
    for s in range(2):
        sim.load(s, ps[s])
    new = {k: v[::-1].copy() for k, v in ps[0].items()}
    dt = torch.float64 if prec == "fp64" else torch.float32
    dev = {k: torch.from_numpy(v).to("cuda", dt if k != "cell" else torch.int32) for k, v in new.items()}
    for steps in (7, 5, 7):
        sim.step(steps)
        live = _host(sim, 2)
        sim.load(0, new) if where == "host" else sim.load_device(0, dev)
        want = [{k: v.astype(live[0][k].dtype) for k, v in new.items()}, live[1]]
        _check(cfg, sim, [_sorted(cfg, w) for w in want])


@pytest.mark.parametrize("n", [0, 1, 100_000, 1_000_000])
def test_load_beside_a_shuffled_species(n):
    """Species 1 put in random order through its views: as far from sorted as
    it can be."""
    import torch
    hff, cfg, ps = _setup("fp32")
    sim = hff.Sim(cfg)
    for s in range(2):
        sim.load(s, ps[s])
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    v = sim.particle_views(1)
    perm = torch.randperm(len(v["cell"]), generator=g, device="cuda")
    for k in KEYS:
        v[k].copy_(v[k][perm].clone())
    torch.cuda.synchronize()
    other = _host(sim, 2)[1]
    new = {k: a[:n].copy() for k, a in ps[0].items()}
    sim.load(0, new)
    _check(cfg, sim, [_sorted(cfg, new), _sorted(cfg, other)])


def test_load_from_views_between_steps():
    """Sources inside the instance: a species handed to the other one and a
    part of a species handed back to itself, while neither is sorted."""
    hff, cfg, ps = _setup("fp32", n_pairs=100_000, nr=128, nt=96)
    sim = hff.Sim(cfg)
    for s in range(2):
        sim.load(s, ps[s])
    sim.step(3)
    live = _host(sim, 2)
    sim.load_device(0, sim.particle_views(1))
    _check(cfg, sim, [_sorted(cfg, live[1]), _sorted(cfg, live[1])])
    sim.step(2)
    live = _host(sim, 2)
    sim.load_device(1, {k: v[1000:] for k, v in sim.particle_views(1).items()})
    _check(cfg, sim, [_sorted(cfg, live[0]), _sorted(cfg, {k: v[1000:] for k, v in live[1].items()})])
    hff, cfg, ps = _setup("fp32", n_species=1, n_pairs=100_000, nr=128, nt=96)
    sim = hff.Sim(cfg)
    sim.load(0, ps[0])
    sim.step(3)
    live = _host(sim, 1)
    sim.load_device(0, {k: v[1000:] for k, v in sim.particle_views(0).items()})
    _check(cfg, sim, [_sorted(cfg, {k: v[1000:] for k, v in live[0].items()})])


def test_load_from_views_taken_before_another_load():
    """A load between steps moves every species to the other buffer; the arrays
    of a view taken before it can still be loaded, in part, too."""
    hff, cfg, ps = _setup("fp32", n_pairs=100_000, nr=128, nt=96)
    sim = hff.Sim(cfg)
    for s in range(2):
        sim.load(s, ps[s])
    sim.step(3)
    live = _host(sim, 2)
    v = sim.particle_views(0)
    sim.load(1, ps[1])
    sim.load_device(0, {k: a[1000:] for k, a in v.items()})
    _check(cfg, sim, [_sorted(cfg, {k: a[1000:] for k, a in live[0].items()}), _sorted(cfg, ps[1])])


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("n_species", [1, 2])
@pytest.mark.parametrize("offset", [1, 4])
def test_load_from_device_arrays_at_any_address(prec, n_species, offset):
    """Device arrays that start between the addresses of their elements (one
    packed buffer: the cells, then the reals, FP64 ones at a multiple of four)."""
    import torch
    hff, cfg, ps = _setup(prec, n_species=n_species, n_pairs=100_000, nr=128, nt=96)
    sim = hff.Sim(cfg)
    for s in range(n_species):
        sim.load(s, ps[s])
    new = {k: v[::-1].astype(np.int32 if k == "cell" else sim.real) for k, v in ps[0].items()}
    raw = [np.zeros(offset, np.uint8)] + [np.ascontiguousarray(new[k]).view(np.uint8) for k in KEYS]
    buf = torch.from_numpy(np.concatenate(raw)).cuda()
    at = buf.data_ptr() + np.cumsum([len(r) for r in raw])[:-1]
    assert any(int(a) % (4 if k == 0 else new["xo"].itemsize) for k, a in enumerate(at)) or (prec, offset) == ("fp32", 4)
    hff.hff_load_particles(sim.h, 0, 0, len(new["cell"]), [int(a) for a in at], hff.DEVICE)
    want = [new] + [{k: v.astype(new[k].dtype) for k, v in p.items()} for p in ps[1:]]
    _check(cfg, sim, [_sorted(cfg, w) for w in want])
