"""The adjoint of catalogues large enough for whole faces: faces that become opaque, that
end, and that are left to the quadrant kernels (layers wider than a face has room for),
in boxes that clip some windows and not others, against the oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2311_01492_gb300 import synth as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,counts,xscale", [
    (48, ((26.0, 60), (24.5, 2400), (9.0, 3000), (2.3, 700)), 1e-3),   # left over, and ending
    (48, ((26.0, 60), (24.5, 2400), (9.0, 3000), (2.3, 700)), 1.0),    # opaque after a few layers
    (14, ((9.5, 1400), (6.0, 900), (1.0, 50)), 1e-2),                  # windows clip layers
])
def test_adjoint_by_faces_matches_the_oracle(n, counts, xscale):
    from paper_2311_01492_gb300 import api as A
    rng = np.random.default_rng(3)
    nH = S.lognormal_field(n, 2e-4, seed=3).reshape(-1)
    nhi = nH * xscale * rng.uniform(0.1, 1.0, n ** 3)
    R = np.concatenate([np.full(c, r) for r, c in counts])
    cells = rng.choice(n ** 3, len(R), replace=False)
    pos = np.stack(np.unravel_index(cells, (n, n, n)), 1).astype(np.int32)
    ndot = 10.0 ** rng.uniform(50, 52, len(R))
    w = rng.standard_normal(n ** 3)
    cell = 0.78 * S.MPC_CM
    tab = O.make_table("bb")
    g = A.Grid(n, cell)
    g.set_tables("knots", g=tab.g, h=tab.h)
    f = dict(device="cuda", dtype=torch.float64)
    g.set_density(torch.tensor(nhi, **f))
    g.set_xHI(torch.ones(n ** 3, **f))
    g.set_sources(torch.tensor(pos, device="cuda"), torch.tensor(ndot, **f), torch.tensor(R, **f))
    dn, dq = (t.cpu().numpy() for t in g.backward(torch.tensor(w, **f)))
    g.check()
    # sources: Gamma is linear in the rates, so dL/dlog Ndot is the source's own loss
    for s in (0, 59, 65, len(R) - 900, len(R) - 1):
        gam = O.raytrace(n, cell, nhi, np.ones(n ** 3), pos[s:s + 1], ndot[s:s + 1], R[s:s + 1],
                         tab)["gamma"]
        assert abs(dq[s] - np.dot(w, gam)) <= 1e-12 * np.dot(np.abs(w), gam)
    # cells: complex steps through the whole catalogue, as in the other adjoint tests
    some = np.concatenate([np.argsort(-np.abs(dn))[:3], rng.choice(cells, 2)]).astype(np.int64)
    ref, _ = O.loss_grad_cs(n, cell, nhi, np.ones(n ** 3), pos, ndot, R, tab, w, some,
                            np.zeros(0, np.int32), nthreads=8)
    assert np.all(np.abs(dn[some] - ref) <= 1e-9 * np.abs(ref))
    # the full recompute gives the same (other kernels where layers are wide)
    g.set_adjoint_mode(False)
    dn2, dq2 = (t.cpu().numpy() for t in g.backward(torch.tensor(w, **f)))
    assert np.linalg.norm(dn2 - dn) <= 1e-12 * np.linalg.norm(dn)
    assert np.linalg.norm(dq2 - dq) <= 1e-12 * np.linalg.norm(dq)
    g.close()
