"""Paths of the tiled push that a run of whole steps rarely or never takes."""
import numpy as np
import pytest

from helpers import particle_mismatches, rel_l2, shared_initial_state

pytestmark = pytest.mark.gpu

ST = dict(node=1, push=4)


def _libs():
    import __graft_entry__
    import oracle
    __graft_entry__.build()
    from paper_2406_14512_gb300 import hff, workloads
    return hff, workloads, oracle


@pytest.mark.parametrize("prec,tol,err", [("fp32", 1e-5, 1e-5), ("fp64", 1e-10, 1e-11)])
@pytest.mark.parametrize("tile", [(4, 4), (16, 24)])
def test_particles_that_drifted_out_of_their_tile(tile, prec, tol, err):
    """Twelve pushes without a sort on a cadence of one: the halo covers one
    step, so particles leave their tile's staged region and take the global
    path, among neighbours that do not (tolerances of the one-step and
    ten-step parity tests)."""
    hff, workloads, oracle = _libs()
    cfg = workloads.config("small_rr")
    cfg.update(capacity=20000, precision=prec, sort_every=1, inject=False, tile_r=tile[0], tile_t=tile[1])
    ps = workloads.particles(cfg, n_pairs=6000, seed=21)
    sim, ref = hff.Sim(cfg), oracle.Oracle(cfg)
    shared_initial_state(sim, ref, seed=7)
    for s in range(2):
        sim.load(s, ps[s])
        ref.set_particles(s, ps[s])
    ref.sort_now()
    for _ in range(12):
        sim.step_stages(1, ST["node"] | ST["push"])
        ref.step(1, ST["node"] | ST["push"])
    for f in ("J_r", "J_th", "J_ph"):
        assert rel_l2(sim.get(f), ref.get(f)) < tol, (f, rel_l2(sim.get(f), ref.get(f)))
    for s in range(2):
        g, o = sim.particles(s), ref.particles(s)
        bad, _, e = particle_mismatches(g, o, cfg["nt"])
        assert bad == 0 and e < err, (s, bad, e)
    live = sum(int((sim.particles(s)["cell"] >= 0).sum()) for s in range(2))
    assert sim.info().pushed_tiled >= 12 * live and sim.status() == 0


@pytest.mark.parametrize("prec,err", [("fp32", 1e-5), ("fp64", 1e-11)])
@pytest.mark.parametrize("n", [(0, 1), (1, 0), (31, 33), (0, 0), (7, 160_000), (160_000, 5)])
def test_tail_is_one_list_over_the_species(n, prec, err):
    """Particles outside the tiles are handed out as one list over the species,
    a warp at a time: empty species, lists that end inside a warp, and more
    particles than the launch has threads (152 x 4 x 256), one push without
    sorting (the tolerances of the one-step parity tests)."""
    hff, workloads, oracle = _libs()
    cfg = workloads.config("small_rr")
    cfg.update(capacity=170_000, precision=prec, sort_every=0, inject=False)
    ps = workloads.particles(cfg, n_pairs=max(*n, 1), seed=23)
    sim, ref = hff.Sim(cfg), oracle.Oracle(cfg)
    shared_initial_state(sim, ref, seed=7)
    for s in range(2):
        part = {k: v[:n[s]] for k, v in ps[s].items()}
        sim.load(s, part)
        ref.set_particles(s, part)
    sim.step_stages(1, ST["node"] | ST["push"])
    ref.step(1, ST["node"] | ST["push"])
    for s in range(2):
        bad, _, e = particle_mismatches(sim.particles(s), ref.particles(s), cfg["nt"])
        assert bad == 0 and e < err, (s, bad, e)
    info = sim.info()
    assert (info.pushed_tiled, info.pushed_tail) == (0, sum(n)) and sim.status() == 0


def test_fp64_momentum_whose_square_overflows():
    """|u| = 1e160: u^2 is infinite, 1/gamma zero, and the particle neither
    moves nor is removed (the reciprocal square root at the end of its range)."""
    hff, workloads, _ = _libs()
    cfg = workloads.config("small_pic")
    cfg.update(capacity=2000, precision="fp64", sort_every=4, inject=False, shell_r=0.5)
    ps = workloads.particles(cfg, n_pairs=500, seed=3)
    ps[0]["ur"] = ps[0]["ur"].astype(np.float64)
    ps[0]["ur"][::7] = 1e160
    sim = hff.Sim(cfg)
    for s in range(2):
        sim.load(s, ps[s])
    before = sim.particles(0)
    big = before["ur"] == 1e160
    sim.step_stages(1, ST["node"] | ST["push"])
    after = sim.particles(0)
    assert big.sum() > 50 and np.array_equal(after["cell"][big], before["cell"][big])
    assert np.array_equal(after["ur"][big], before["ur"][big]) and np.array_equal(after["xo"][big], before["xo"][big])
    assert sim.status() == 0
