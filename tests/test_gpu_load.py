"""Loading particles while others are there: the sorted order, the counts and
the work list that follow, whatever state the other species is in and wherever
the arrays come from, against the oracle (which sorts every species then)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

KEYS = ("cell", "xo", "yo", "ur", "ut", "up", "w")


def _setup(prec, n_species, tile, **kw):
    import __graft_entry__
    import oracle
    __graft_entry__.build()
    from paper_2406_14512_gb300 import hff, workloads
    cfg = workloads.config("small_crust" if n_species == 3 else "small_hybrid")
    cfg.update(capacity=30000, sort_every=4, precision=prec, tile_r=tile[0], tile_t=tile[1], gamma_th=0.0, **kw)
    ps = workloads.particles(cfg, n_pairs=9001, seed=19)
    return hff, cfg, (ps + [{k: v.copy() for k, v in ps[0].items()}])[:n_species], oracle


def _same(sim, ref, ns):
    for s in range(ns):
        g, o = sim.particles(s), ref.particles(s)
        for k in KEYS:
            assert np.array_equal(g[k], o[k].astype(g[k].dtype)), (s, k)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("n_species,tile", [(2, (16, 24)), (3, (4, 5))])
@pytest.mark.parametrize("n", [0, 1, 2047, 2049, 9001])
def test_load_into_settled_and_unsettled_instances(prec, n_species, tile, n):
    """A second load of species 0 (n particles in reversed order, some removed)
    after loads (the others settled) and again after steps with injection and
    removals (unsettled: they are compacted and sorted along)."""
    import torch
    hff, cfg, ps, oracle = _setup(prec, n_species, tile)
    sim, ref = hff.Sim(cfg), oracle.Oracle(cfg)
    for s in range(n_species):
        sim.load(s, ps[s])
        ref.set_particles(s, ps[s])
    ref.sort_now()
    new = {k: v[::-1][:n].copy() for k, v in ps[0].items()}
    new["cell"][::5] = -1
    for host in (True, False):
        if host:
            sim.load(0, new)
        else:
            dt = torch.float64 if prec == "fp64" else torch.float32
            sim.load_device(0, {k: torch.from_numpy(v).to("cuda", dt if k != "cell" else torch.int32) for k, v in new.items()})
        ref.set_particles(0, new)
        ref.sort_now()
        _same(sim, ref, n_species)
    sim.step(3)
    live = [{k: v for k, v in sim.particles(s).items()} for s in range(n_species)]
    sim.load(0, new)
    for s in range(n_species):
        ref.set_particles(s, new if s == 0 else live[s])
    ref.sort_now()
    _same(sim, ref, n_species)
    before = sim.info()
    sim.step_stages(1, 5)   # the work list covers every particle
    after = sim.info()
    total = sum(len(ref.particles(s)["cell"]) for s in range(n_species))
    assert after.pushed_tiled - before.pushed_tiled == total and after.pushed_tail == before.pushed_tail
    assert sim.status() == 0


def test_load_from_its_own_views():
    """The particles handed back as device arrays of the instance itself."""
    hff, cfg, ps, oracle = _setup("fp32", 2, (16, 24), inject=False)
    sim = hff.Sim(cfg)
    for s in range(2):
        sim.load(s, ps[s])
    want = [sim.particles(s) for s in range(2)]
    sim.load_device(0, sim.particle_views(0))   # onto itself
    for s in range(2):
        got = sim.particles(s)
        assert all(np.array_equal(got[k], want[s][k]) for k in KEYS)
    sim.load_device(1, sim.particle_views(0))   # one species as the other
    for s in range(2):
        got = sim.particles(s)
        assert all(np.array_equal(got[k], want[0][k]) for k in KEYS)


def test_one_species_and_invalid_cells():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2406_14512_gb300 import hff, workloads
    cfg = workloads.config("small_pic")
    cfg.update(capacity=9000, sort_every=4, precision="fp64", q=[-1.0], m=cfg["m"][:1], inject=False, inject_species=[0, 0])
    p = workloads.particles(dict(cfg, q=[-1.0, 1.0]), n_pairs=5000, seed=2)[0]
    sim = hff.Sim(cfg)
    sim.load(0, p)
    key = (p["cell"] // cfg["nt"] // cfg["tile_r"]) * (-(-cfg["nt"] // cfg["tile_t"])) + p["cell"] % cfg["nt"] // cfg["tile_t"]
    o = np.argsort(key, kind="stable")
    assert np.array_equal(sim.particles(0)["cell"], p["cell"][o]) and np.array_equal(sim.particles(0)["w"], p["w"][o])
    bad = dict(p, cell=p["cell"].copy())
    bad["cell"][7] = cfg["nr"] * cfg["nt"]
    with pytest.raises(hff.HffError) as e:
        sim.load(0, bad)
    assert e.value.code == hff.HFF_ERR_ARG and len(sim.particles(0)["cell"]) == len(o) - 1
    assert sim.status() == 0
