"""Every launch mode of the batched rates (quadrants per warp, CTAs) in one catalogue,
against the oracle: radii on both sides of the class limits, boxes that clip some of
them, opaque and nearly ionised fields, with and without the early exit."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2311_01492_gb300 import synth as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
RTOL = 1e-9  # the library's bound on rates: every term has the oracle's bits


def _workload(n, counts, xscale, seed):
    rng = np.random.default_rng(seed)
    nH = S.lognormal_field(n, 2e-4, seed=seed)
    xHI = xscale * rng.random((n, n, n))
    R = np.concatenate([np.full(c, r) for r, c in counts])
    nsrc = len(R)
    cells = rng.choice(n ** 3, nsrc, replace=False)
    pos = np.stack(np.unravel_index(cells, (n, n, n)), 1).astype(np.int32)
    ndot = 10.0 ** rng.uniform(50, 53, nsrc)
    return dict(n=n, cell_cm=0.78 * S.MPC_CM, nH=nH, xHI=xHI, pos=pos, ndot=ndot, radius=R)


@pytest.mark.parametrize("xscale", [1.0, 1e-4])
@pytest.mark.parametrize("n,counts", [
    # 4 quadrants per warp (half-width <= 16), 2 (<= 23), 1, in one trace: enough items
    # of each class for three launches (R = 23.4 and 33.2 are the classes' last radii)
    (40, ((2.0, 900), (23.4, 1700), (23.6, 700), (33.2, 600), (33.9, 30))),
    # few sources: CTAs, of 128 and of 256 threads, clipped on one side of an even box
    (33, ((7.5, 3), (12.0, 2))),
    (72, ((36.0, 2), (50.0, 1))),
])
def test_all_modes_match_the_oracle(n, counts, xscale):
    from paper_2311_01492_gb300 import api as A
    w = _workload(n, counts, xscale, 11)
    tab = O.make_table("bb")
    ref = O.raytrace(w["n"], w["cell_cm"], w["nH"], w["xHI"], w["pos"], w["ndot"], w["radius"],
                     tab, nthreads=8)["gamma"]
    g = A.Grid(n, w["cell_cm"])
    g.set_tables("knots", g=tab.g, h=tab.h)
    f = dict(device="cuda", dtype=torch.float64)
    g.set_density(torch.tensor(w["nH"].reshape(-1), **f))
    g.set_xHI(torch.tensor(w["xHI"].reshape(-1), **f))
    g.set_sources(torch.tensor(w["pos"], device="cuda"), torch.tensor(w["ndot"], **f),
                  torch.tensor(w["radius"], **f))
    for sched in (None, (128, 32, 20), (256, 10, 4), (128, 0, 0)):
        if sched:
            g.set_schedule(*sched)
        for how in ("batched", "early_exit"):
            got = g.raytrace(schedule=how).cpu().numpy()
            assert np.array_equal(got == 0, ref == 0)
            nz = ref != 0
            assert np.max(np.abs(got[nz] - ref[nz]) / ref[nz]) <= RTOL, (sched, how)
    g.check()
    g.close()
