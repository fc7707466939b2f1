"""J_PIC out of the push's flux accumulators, against the FP64 oracle, on grids
around the widths of the collection (warps of 32 columns, blocks of 128,
segments of rows, odd and even row counts) with particles in every cell inside the absorber, from
the star and up to the axis: each location must get the parts of all the cells that meet there.

Tolerances: the tiled FP32 deposit's and the FP64 one's of the parity tests
(1e-6, 1e-10 in relative L2), a decade looser in FP32 because these grids are
coarse (8 rows), where a single particle is a visible part of J."""
import numpy as np
import pytest

from helpers import rel_l2, shared_initial_state

pytestmark = pytest.mark.gpu

ST = dict(node=1, push=4, faraday1=8, ampere=16, correct=2, faraday2=32)


@pytest.mark.parametrize("prec,tol", [("fp32", 1e-5), ("fp64", 1e-10)])
@pytest.mark.parametrize("sort_every", [0, 4])
@pytest.mark.parametrize("nr,nt", [(8, 129), (20, 31), (21, 32), (36, 126), (37, 127), (53, 128)])
def test_current_at_every_location(nr, nt, sort_every, prec, tol):
    import __graft_entry__
    import oracle
    __graft_entry__.build()
    from paper_2406_14512_gb300 import hff, workloads
    cfg = workloads._base(nr, nt, 10.0, 3.0, "dipole", seed=31)
    cfg.update(precision=prec, sort_every=sort_every, inject=False, capacity=20000)
    rng = np.random.default_rng(nr * 1000 + nt)
    inner = int(np.floor(np.log(cfg["r_abs"]) / (np.log(10.0) / nr))) * nt
    n = inner + 3000
    cell = np.concatenate([np.arange(inner), rng.integers(0, inner, 3000)]).astype(np.int32)
    ps = []
    for s in range(2):
        u = rng.normal(0.0, 2.0, (3, n)).astype(np.float32)
        ps.append(dict(cell=cell, xo=rng.random(n, dtype=np.float32), yo=rng.random(n, dtype=np.float32), ur=u[0],
                       ut=u[1], up=u[2], w=(1e-3 * (0.5 + rng.random(n))).astype(np.float32)))
    sim, ref = hff.Sim(cfg), oracle.Oracle(cfg)
    shared_initial_state(sim, ref, seed=9)
    for s in range(2):
        sim.load(s, ps[s])
        ref.set_particles(s, ps[s])
    if sort_every:
        ref.sort_now()
    for k in range(2):  # twice: the accumulators are cleared in between (J itself adds up)
        sim.step_stages(1, ST["node"] | ST["push"])
        ref.step(1, ST["node"] | ST["push"])
        for f in ("J_r", "J_th", "J_ph"):
            assert rel_l2(sim.get(f), ref.get(f)) < tol, (k, f, rel_l2(sim.get(f), ref.get(f)))
    # the collection carried by the first Faraday half step (a whole field update in the same call)
    stages = sum(ST.values())
    sim.step_stages(1, stages)
    ref.step(1, stages)
    for f in ("E_r", "E_th", "E_ph", "B_r", "B_th", "B_ph"):
        assert rel_l2(sim.get(f), ref.get(f)) < 10 * tol, (f, rel_l2(sim.get(f), ref.get(f)))
    sim.close()
