"""An iteration whose buffers did not all fit is refused, and runs once they do."""
import numpy as np
import pytest

from paper_2311_01492_gb300 import synth as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fit", [0, 1, 2, 3])  # buffers of four that fit at first
def test_iterate_after_running_out_of_memory(fit):
    from paper_2311_01492_gb300 import api as A
    n, rng = 24, np.random.default_rng(1)
    f = dict(device="cuda", dtype=torch.float64)

    def grid():
        g = A.Grid(n, 0.1 * S.MPC_CM)
        g.set_tables("grey_exact")
        g.set_density(torch.full((n ** 3,), 1e-3, **f))
        g.set_sources(torch.tensor([[12, 12, 12]], dtype=torch.int32, device="cuda"),
                      torch.tensor([1e54], **f), torch.tensor([10.0], **f))
        return g
    x0 = torch.tensor(1e-3 * rng.random(n ** 3), **f)
    a, b = grid(), grid()
    want = x0.clone()
    gam, its = a.iterate(want, S.MYR_S)
    x = x0.clone()
    try:
        A.set_device_memory_limit(A.device_memory_in_use() + fit * 8 * n ** 3 + 64)
        with pytest.raises(A.RtError, match="RT_ERR_OOM"):
            b.iterate(x, S.MYR_S)
        assert torch.equal(x, x0)
    finally:
        A.set_device_memory_limit(0)
    gam2, its2 = b.iterate(x, S.MYR_S)
    assert its2 == its and torch.equal(x, want) and torch.equal(gam2, gam)
    a.close()
    b.close()
