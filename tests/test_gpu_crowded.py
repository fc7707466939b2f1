"""Crowded cells in FP32: the accumulators of cells that take many particles of
many work items, which the tiled push sums item by item before they meet."""
import numpy as np
import pytest

from helpers import particle_mismatches, rel_l2, shared_initial_state

pytestmark = pytest.mark.gpu

ST = dict(node=1, push=4)
FIELDS6 = ("E_r", "E_th", "E_ph", "B_r", "B_th", "B_ph")


def _libs():
    import __graft_entry__
    import oracle
    __graft_entry__.build()
    from paper_2406_14512_gb300 import hff, workloads
    return hff, workloads, oracle


def test_current_of_a_tile_with_many_items():
    """295,000 particles of each species in 32 cells of one tile (36 items of
    8192 each), all of a cell alike, the species moving in opposite azimuthal
    directions: J_ph against the FP64 instance.  A sum of n equal terms in FP32
    is off by at most (n / 2) 2^-24 of itself: 7.6e-6 for the 256 particles of
    an item and a cell, 2.1e-6 for the partial sums of 72 items, and some
    2^-24 for the terms themselves: 1.1e-5.  (Added one by one, 18,400 terms may
    lose 5.5e-4.)"""
    hff, workloads, _ = _libs()
    nr, nt, n = 192, 192, 36 * 8192
    cfg = workloads._base(nr, nt, 20.0, 4.0, "dipole", seed=3)
    cfg.update(precision="fp32", inject=False, sort_every=12, tile_r=16, tile_t=24, capacity=17_000_000)
    cells = (np.arange(96, 112)[:, None] * nt + np.array([100, 103])[None, :]).ravel()
    rng = np.random.default_rng(4)
    worst = 0.0
    for x, y, u in [(0.3, 0.7, 2.0), (0.11, 0.23, 0.7), (0.62, 0.41, 5.0)]:
        one = np.full(n, 1, np.float32)
        cell = rng.permutation(np.repeat(cells, n // 32)).astype(np.int32)
        ps = [dict(cell=cell, xo=x * one, yo=y * one, ur=0 * one, ut=0 * one, up=s * np.float32(u) * one, w=np.float32(1e-3) * one)
              for s in (-1, 1)]
        ps = [{k: v.astype(np.float32) if k != "cell" else v for k, v in p.items()} for p in ps]
        sim, ref = hff.Sim(cfg), hff.Sim(dict(cfg, precision="fp64", capacity=n))
        for f in FIELDS6:
            ref.set(f, sim.get(f).astype(np.float64))
        for s in range(2):
            sim.load(s, ps[s])
            ref.load(s, ps[s])
        for q in (sim, ref):
            q.step_stages(1, ST["node"] | ST["push"])
        g, o = sim.get("J_ph").astype(np.float64), ref.get("J_ph")
        at = np.abs(o) > 1e-3 * np.abs(o).max()
        assert at.sum() >= 64
        worst = max(worst, float((np.abs(g - o)[at] / np.abs(o)[at]).max()))
        assert sim.status() == 0
        sim.close()
        ref.close()
    assert worst < 1.1e-5, worst


@pytest.mark.parametrize("tile", [(16, 24), (4, 5)])
@pytest.mark.parametrize("spread", [3, 40])
@pytest.mark.parametrize("n", [255, 256, 257, 575, 577, 2049, 20_001])
def test_crowded_cells_everywhere(n, spread, tile):
    """n particles of each species in `spread` cells at the star, on the axis, in
    the tiles' corners and inside (3 cells also sum by cell within a warp), over
    the pushes of a cadence and the one after the sort, against the oracle
    (tolerances of the FP32 parity tests, 1e-5 as on the grids of the collection
    test, whose cells are as coarse)."""
    hff, workloads, oracle = _libs()
    nr, nt = 52, 41
    cfg = workloads._base(nr, nt, 10.0, 3.0, "dipole", seed=31)
    cfg.update(precision="fp32", sort_every=4, inject=False, capacity=3 * n, tile_r=tile[0], tile_t=tile[1])
    rng = np.random.default_rng(n + spread)
    where = [(0, 0), (15, 23), (16, 24), (0, nt - 1), (17, 30), (3, 4), (4, 5), (20, 0), (30, nt - 1)]
    where = [a * nt + b for a, b in where] + list(rng.integers(0, 36 * nt, 40))
    cells = np.array(where[:spread], np.int32)
    ps = []
    for s in range(2):
        u = rng.normal(0.0, 2.0, (3, n)).astype(np.float32)
        ps.append(dict(cell=cells[rng.integers(0, spread, n)], xo=rng.random(n, dtype=np.float32),
                       yo=rng.random(n, dtype=np.float32), ur=u[0], ut=u[1], up=u[2],
                       w=(1e-3 * (0.5 + rng.random(n))).astype(np.float32)))
    sim, ref = hff.Sim(cfg), oracle.Oracle(cfg)
    shared_initial_state(sim, ref, seed=9)
    for s in range(2):
        sim.load(s, ps[s])
        ref.set_particles(s, ps[s])
    ref.sort_now()
    for k in range(2):   # the list's first push, which decides, and one that follows it
        sim.step_stages(1, ST["node"] | ST["push"])
        ref.step(1, ST["node"] | ST["push"])
        for f in ("J_r", "J_th", "J_ph"):
            assert rel_l2(sim.get(f), ref.get(f)) < 1e-5, (k, f, rel_l2(sim.get(f), ref.get(f)))
    for s in range(2):
        bad, _, e = particle_mismatches(sim.particles(s), ref.particles(s), nt)
        assert bad == 0 and e < 1e-5, (s, bad, e)
    sim.step(5)   # whole steps over a sort: the push that moves the sorted particles decides again
    ref.step(5)
    for f in FIELDS6:
        assert rel_l2(sim.get(f), ref.get(f)) < 1e-4, (f, rel_l2(sim.get(f), ref.get(f)))
    assert sim.status() == 0
    sim.close()
