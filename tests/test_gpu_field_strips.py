"""The fused field pass at the edges of its decomposition: strips of 8 warps of
28 columns (26 with the theta filter; 4 warps in FP64) and segments of 32 rows
and more, against the separate field kernels.

Two steps of the fields alone from E, dB and J_PIC filled with noise, so that
every halo column and warm-up row carries independent values: a wrong neighbour
shows at order one.  The two passes evaluate the same expressions; a location
takes some 40 roundings a step, so their rms difference stays below 40 epsilon
of the field per step: 1e-5 (FP32) and 1e-13 x 10 (FP64) leave a margin."""
import numpy as np
import pytest

from helpers import FIELDS6, rel_l2

pytestmark = pytest.mark.gpu

SIZES = [(8, 8), (9, 27), (31, 28), (32, 29), (33, 55), (64, 111), (65, 112), (70, 207), (95, 223), (96, 224),
         (97, 225), (40, 448), (130, 640)]


@pytest.mark.parametrize("prec,tol", [("fp32", 1e-5), ("fp64", 1e-12)])
@pytest.mark.parametrize("delta,filt", [(0, 0.0), (0, 1.0), (1, 0.5)])
def test_fused_pass_at_strip_and_segment_edges(prec, tol, delta, filt):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2406_14512_gb300 import hff, workloads
    for nr, nt in SIZES:
        rng = np.random.default_rng(nr * 1000 + nt)
        cfg = dict(workloads.config("small_fine"), nr=nr, nt=nt, capacity=0, precision=prec, sort_every=0, r_abs=5.0, inject=False,
                   ff_delta_only=delta, ff_filter=filt)
        sims = [hff.Sim(dict(cfg, field_pass=fp)) for fp in (1, 2)]
        for name in FIELDS6 + ("J_r", "J_th", "J_ph"):
            a = sims[0].get(name)
            scale = 0.05 * max(1e-2, float(np.sqrt(np.mean(np.square(a, dtype=np.float64)))))
            b = (a + scale * rng.standard_normal(a.shape)).astype(a.dtype)
            for sim in sims:
                sim.set(name, b)
        for sim in sims:
            sim.step(2)
            assert sim.status() == 0
        # E^2 and B^2 within rounding of each other decide differently: some 1e-6 of the nodes
        assert abs(sims[0].diagnostics()[0].clamps - sims[1].diagnostics()[0].clamps) <= 2, (nr, nt)
        for name in FIELDS6 + ("J_r", "J_th", "J_ph"):
            x, y = sims[0].get(name), sims[1].get(name)
            if name.startswith("J"):
                assert not x.any() and not y.any(), (nr, nt, name)
            else:
                assert rel_l2(y, x) < tol, (nr, nt, name, rel_l2(y, x))
        for sim in sims:
            sim.close()


@pytest.mark.parametrize("nr,nt,prec,fused", [(1448, 1448, "fp32", True), (511, 3719, "fp32", False),
                                              (511, 3720, "fp32", True), (512, 3600, "fp32", True),
                                              (2048, 2048, "fp64", False)])
def test_automatic_field_pass_takes_the_faster_one(nr, nt, prec, fused):
    """At least 500 areas of 32 rows by 120 columns, FP32 (16 x 31 = 496, 16 x 32
    and 17 x 31 at the edges)."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2406_14512_gb300 import hff, workloads
    cfg = dict(workloads.config("c1"), nr=nr, nt=nt, capacity=0, precision=prec, sort_every=0)
    sim = hff.Sim(cfg)
    assert sim.info().field_pass == (hff.FIELDS_FUSED if fused else hff.FIELDS_SPLIT)
    sim.close()
