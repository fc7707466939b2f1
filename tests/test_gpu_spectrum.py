"""The spectrum's bins, taken in FP32 where that decides, against FP64 bins of
the same momenta: particles within 1e-9 (FP64 momenta) or the FP32 spacing
(FP32 momenta) of bin edges, at rest, beyond both ends, and with squares
outside the FP32 range."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("nbins,lo,hi", [(1, 0.0, 7.0), (200, 0.0, 7.0), (333, -0.5, 2.25), (4096, 0.0, 19.0)])
def test_bins_at_their_edges(prec, nbins, lo, hi):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2406_14512_gb300 import hff, workloads
    cfg = workloads.config("small_pic")
    cfg.update(capacity=70000, sort_every=4, precision=prec, inject=False)
    rng = np.random.default_rng(nbins)
    edges = lo + (hi - lo) * rng.integers(0, nbins + 1, 20000) / nbins
    lg = edges + rng.choice([-1e-6, -1e-9, 1e-9, 1e-6], edges.size)
    lg = np.concatenate([lg[lg > 1e-7], rng.uniform(0.0, hi + 1, 5000)])
    g = 10.0 ** lg
    p = np.concatenate([np.sqrt((g - 1.0) * (g + 1.0)), [0.0, 1e18, 3e19, 1e25]])
    n = len(p)
    mu, ph = rng.uniform(-1, 1, n), rng.uniform(0, 2 * np.pi, n)
    st = np.sqrt(1 - mu * mu)
    real = np.float32 if prec == "fp32" else np.float64
    u = [(p * mu).astype(real), (p * st * np.cos(ph)).astype(real), (p * st * np.sin(ph)).astype(real)]
    d = dict(cell=rng.integers(0, cfg["nr"] * cfg["nt"] // 2, n).astype(np.int32), xo=rng.random(n).astype(real),
             yo=rng.random(n).astype(real), ur=u[0], ut=u[1], up=u[2], w=(2.0 ** rng.integers(-8, 8, n)).astype(real))
    sim = hff.Sim(cfg)
    sim.load(0, d)
    got = sim.spectrum(0, nbins, lo, hi)
    x = (np.log10(np.sqrt(1.0 + sum(a.astype(np.float64) ** 2 for a in u))) - lo) * (nbins / (hi - lo))
    keep = np.abs(x - np.round(x)) > 1e-10 * (1 + np.abs(x))   # an edge to the last FP64 digits may fall either way
    want = np.bincount(np.clip(np.floor(x), 0, nbins - 1).astype(int), d["w"].astype(np.float64), nbins)
    slack = np.bincount(np.clip(np.round(x[~keep]), 0, nbins - 1).astype(int), d["w"][~keep].astype(np.float64), nbins)
    slack = slack + np.roll(slack, 1) + np.roll(slack, -1)
    assert np.all(np.abs(got - want) <= slack), np.flatnonzero(np.abs(got - want) > slack)
    assert got.sum() == d["w"].astype(np.float64).sum()   # powers of two: sums are exact


@pytest.mark.parametrize("big", [1e140, 1e160])
def test_kinetic_energy_of_extreme_momenta(big):
    """FP64 momenta whose square is near the end of the range (the sum is finite)
    or beyond it (the energy is then infinite, not undefined)."""
    import __graft_entry__
    __graft_entry__.build()
    from paper_2406_14512_gb300 import hff, workloads
    cfg = workloads.config("small_pic")
    cfg.update(capacity=2000, precision="fp64", sort_every=4, inject=False)
    p = workloads.particles(cfg, n_pairs=500, seed=3)[0]
    p["ur"] = p["ur"].astype(np.float64)
    p["ur"][::7] = big
    sim = hff.Sim(cfg)
    sim.load(0, p)
    got = sim.diagnostics()[0].kinetic[0]
    with np.errstate(over="ignore"):
        u2 = sum(p[k].astype(np.float64) ** 2 for k in ("ur", "ut", "up"))
    want = np.sum(p["w"].astype(np.float64) * cfg["m"][0] * (np.sqrt(1.0 + u2) - 1.0))
    assert got == want if np.isinf(want) else abs(got - want) <= 1e-12 * want
