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


@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_fp64_displacement_at_the_end_of_the_series(sign):
    """Radial moves of 2.4% to 3.4% of the radius, on both sides of where log1p
    leaves its series for the library: the new offset against the oracle.  The
    series ends below x^9 / 9 (1e-13 of the value at 0.03125); in cells of
    log(r) = 0.1 that is 3e-14, and the oracle's and the push's own rounding (a
    few 2^-53 over 0.1) as much again: 1e-13."""
    hff, workloads, oracle = _libs()
    cfg = workloads._base(32, 16, float(np.exp(3.2)), 3.0, "dipole", seed=5)
    cfg.update(precision="fp64", capacity=6000, sort_every=4, inject=False, shell_r=0.5)
    rng = np.random.default_rng(8)
    n = 4000
    sim, ref = hff.Sim(cfg), oracle.Oracle(cfg)
    dt = sim.info().dt
    for f in ("E_r", "E_th", "E_ph", "B_r", "B_th", "B_ph"):
        z = np.zeros(ref.shape(f))
        sim.set(f, z)
        ref.set(f, z)
    xi = np.log(dt / rng.uniform(0.024, 0.034, n)) / 0.1
    ps = []
    for s in range(2):
        ps.append(dict(cell=(xi.astype(np.int32) * 16 + rng.integers(3, 13, n)).astype(np.int32), xo=xi % 1.0, yo=rng.random(n),
                       ur=np.full(n, sign * 1e4), ut=np.zeros(n), up=np.zeros(n), w=np.full(n, 1e-6)))
        sim.load(s, ps[s])
        ref.set_particles(s, ps[s])
    ref.sort_now()
    sim.step_stages(1, ST["node"] | ST["push"])
    ref.step(1, ST["node"] | ST["push"])
    for s in range(2):
        bad, _, e = particle_mismatches(sim.particles(s), ref.particles(s), 16)
        assert bad == 0 and e < 1e-13, (s, bad, e)
