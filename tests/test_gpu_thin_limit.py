"""Cells whose dtau ds is within a few units in the last place of tau_lim take the oracle's
side of the thin limit (the two forms differ there by tau_lim / 2 relative, 5e-8), in every
launch mode of the batched rates."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2311_01492_gb300 import synth as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
RTOL = 1e-9  # the library's bound on rates: every term has the oracle's bits


@pytest.mark.parametrize("n,nsrc,sched", [(11, 1, None), (11, 1, (128, 32, 0)), (11, 1, (128, 32, 20)),
                                          (11, 1, (128, 0, 0)), (48, 900, None)])
def test_sides_of_the_thin_limit(n, nsrc, sched):
    from paper_2311_01492_gb300 import api as A
    rng = np.random.default_rng(3)
    cm = 0.1 * S.MPC_CM
    a = rng.integers(0, 5, (n ** 3, 2))
    m = np.maximum(a.max(1), rng.integers(1, 5, n ** 3))
    ds = np.sqrt(1.0 + (a ** 2).sum(1) / m ** 2)
    nH = O.TAU_LIM / ds / (O.SIGMA0 * cm) * (1.0 + rng.integers(-3, 4, n ** 3) * 2.0 ** -52)
    xHI = np.ones(n ** 3)
    pos = np.full((1, 3), n // 2) if nsrc == 1 else np.stack(
        np.unravel_index(rng.choice(n ** 3, nsrc, replace=False), (n, n, n)), 1)
    pos = pos.astype(np.int32)
    ndot, R = np.full(nsrc, 1e52), np.full(nsrc, 5.0)
    tab = O.make_table("bb")
    ref = O.raytrace(n, cm, nH, xHI, pos, ndot, R, tab, nthreads=8)["gamma"]
    g = A.Grid(n, cm)
    g.set_tables("knots", g=tab.g, h=tab.h)
    f = dict(device="cuda", dtype=torch.float64)
    g.set_density(torch.tensor(nH, **f))
    g.set_xHI(torch.tensor(xHI, **f))
    g.set_sources(torch.tensor(pos, device="cuda"), torch.tensor(ndot, **f), torch.tensor(R, **f))
    if sched:
        g.set_schedule(*sched)
    for how in ("batched", "early_exit"):
        got = g.raytrace(schedule=how).cpu().numpy()
        nz = ref != 0
        assert np.array_equal(got == 0, ~nz)
        assert np.max(np.abs(got[nz] - ref[nz]) / ref[nz]) <= RTOL, how
    g.check()
    g.close()
