"""Optical-depth-modulated weights in each launch mode of the batched rates (quadrants per
warp, whole faces, CTAs), against the oracle: class limits, clipped windows, opaque and
nearly ionised fields, and floors on both sides of the tables' bound."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2311_01492_gb300 import synth as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
RTOL = 1e-9  # the library's bound on rates: every term has the oracle's bits


@pytest.mark.parametrize("xscale,tau_w0", [(1.0, 0.6), (1.0, 1e-3), (1.0, 1e9), (3e-4, 0.6)])
@pytest.mark.parametrize("n,counts", [
    # whole faces, two quadrants and one per warp in one trace (R = 23.4, 33.2: last radii)
    (40, ((2.0, 900), (23.4, 1200), (23.6, 500), (33.2, 300))),
    (33, ((7.5, 300), (33.0, 20))),  # clipped on one side of an even and an odd window
    (30, ((12.0, 3),)),              # few sources: CTAs
])
def test_optical_depth_modes_match_the_oracle(n, counts, xscale, tau_w0):
    from paper_2311_01492_gb300 import api as A
    rng = np.random.default_rng(17)
    nH = S.lognormal_field(n, 2e-4, seed=17)
    xHI = xscale * rng.random((n, n, n))
    R = np.concatenate([np.full(c, r) for r, c in counts])
    cells = rng.choice(n ** 3, len(R), replace=False)
    pos = np.stack(np.unravel_index(cells, (n, n, n)), 1).astype(np.int32)
    ndot = 10.0 ** rng.uniform(50, 53, len(R))
    cm = 0.78 * S.MPC_CM
    tab = O.make_table("bb")
    ref = O.raytrace(n, cm, nH, xHI, pos, ndot, R, tab, nthreads=8, interp=1,
                     tau_w0=tau_w0)["gamma"]
    g = A.Grid(n, cm)
    g.set_tables("knots", g=tab.g, h=tab.h)
    g.set_interpolation("optical_depth", tau_w0)
    f = dict(device="cuda", dtype=torch.float64)
    g.set_density(torch.tensor(nH.reshape(-1), **f))
    g.set_xHI(torch.tensor(xHI.reshape(-1), **f))
    g.set_sources(torch.tensor(pos, device="cuda"), torch.tensor(ndot, **f),
                  torch.tensor(R, **f))
    nz = ref != 0
    for sched in (None, (128, 32, 20), (128, 0, 0)):
        if sched:
            g.set_schedule(*sched)
        for how in ("batched", "early_exit"):
            got = g.raytrace(schedule=how).cpu().numpy()
            assert np.array_equal(got == 0, ~nz), (sched, how)
            assert np.max(np.abs(got[nz] - ref[nz]) / ref[nz]) <= RTOL, (sched, how)
    g.check()
    g.close()
