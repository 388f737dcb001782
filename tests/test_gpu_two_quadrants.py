"""Two quadrants of a face per warp (half-widths 17 to 20, large catalogues), whose windows
differ where an even box clips the layers, against the oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2311_01492_gb300 import synth as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
RTOL = 1e-9  # the library's bound on rates


@pytest.mark.parametrize("xscale", [1.0, 1e-4])
@pytest.mark.parametrize("n,counts", [
    (34, ((30.0, 6600),)),              # clipped on one side of the window in every layer
    (35, ((30.0, 3300), (24.1, 3300))),  # an odd window; layers within it and beyond
    (64, ((24.1, 3300), (29.6, 3300))),  # no window: the class's first and last radii
])
def test_two_quadrants_per_warp_match_the_oracle(n, counts, xscale):
    from paper_2311_01492_gb300 import api as A
    rng = np.random.default_rng(21)
    nH, xHI = S.lognormal_field(n, 2e-4, seed=21), xscale * rng.random((n, n, n))
    R = np.concatenate([np.full(c, r) for r, c in counts])
    cells = rng.choice(n ** 3, len(R), replace=False)
    pos = np.stack(np.unravel_index(cells, (n, n, n)), 1).astype(np.int32)
    ndot = 10.0 ** rng.uniform(50, 53, len(R))
    cm, tab = 0.78 * S.MPC_CM, O.make_table("bb")
    ref = O.raytrace(n, cm, nH, xHI, pos, ndot, R, tab, nthreads=16)["gamma"]
    g = A.Grid(n, cm)
    g.set_tables("knots", g=tab.g, h=tab.h)
    f = dict(device="cuda", dtype=torch.float64)
    g.set_density(torch.tensor(nH.reshape(-1), **f))
    g.set_xHI(torch.tensor(xHI.reshape(-1), **f))
    g.set_sources(torch.tensor(pos, device="cuda"), torch.tensor(ndot, **f), torch.tensor(R, **f))
    nz = ref != 0
    for how in ("batched", "early_exit"):
        got = g.raytrace(schedule=how).cpu().numpy()
        st = g.stats()
        # one launch, of the mode with four warps a CTA: one quadrant per warp has at most
        # three, faces end at half-width 16, and CTAs are for small catalogues
        assert st["launches"] == 1 and st["block"] == 128, (how, st)
        assert np.array_equal(got == 0, ~nz)
        assert np.max(np.abs(got[nz] - ref[nz]) / ref[nz]) <= RTOL, how
    g.check()
    g.close()
