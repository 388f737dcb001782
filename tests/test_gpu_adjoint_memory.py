"""Where the list of what whole faces leave over does not fit in memory, the adjoint takes
the quadrant kernels, which need none, and gives the same gradients."""
import numpy as np
import pytest

from paper_2311_01492_gb300 import synth as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_adjoint_without_memory_for_the_leftover_list():
    from paper_2311_01492_gb300 import api as A
    n, rng = 48, np.random.default_rng(4)
    f = dict(device="cuda", dtype=torch.float64)
    g = A.Grid(n, 0.78 * S.MPC_CM)
    g.set_tables("bb")
    g.set_density(torch.tensor(S.lognormal_field(n, 2e-4, seed=4).reshape(-1), **f))
    g.set_xHI(torch.tensor(1e-3 * rng.uniform(0.1, 1.0, n ** 3), **f))
    # half-widths above and below what a face has room for
    R = np.concatenate([np.full(60, 26.0), np.full(2400, 24.5), np.full(3000, 9.0)])
    cells = rng.choice(n ** 3, len(R), replace=False)
    pos = np.stack(np.unravel_index(cells, (n, n, n)), 1).astype(np.int32)
    g.set_sources(torch.tensor(pos, device="cuda"), torch.tensor(10.0 ** rng.uniform(50, 52, len(R)), **f),
                  torch.tensor(R, **f))
    w = torch.tensor(rng.standard_normal(n ** 3), **f)
    g.set_adjoint_mode(False)
    g.backward(w)  # the quadrant kernels' stack stays with the grid
    g.set_adjoint_mode(True)
    try:
        A.set_device_memory_limit(A.device_memory_in_use())
        dn, dq = (t.cpu().numpy() for t in g.backward(w))
    finally:
        A.set_device_memory_limit(0)
    held = A.device_memory_in_use()
    dn2, dq2 = (t.cpu().numpy() for t in g.backward(w))
    assert A.device_memory_in_use() > held  # (the list is what was missing)
    g.check()
    # sums of the same terms in another order: the bound of the other adjoint tests
    assert np.linalg.norm(dn2 - dn) <= 1e-12 * np.linalg.norm(dn)
    assert np.linalg.norm(dq2 - dq) <= 1e-12 * np.linalg.norm(dq)
    g.close()
