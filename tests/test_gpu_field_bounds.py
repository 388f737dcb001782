"""Which field values are accepted: n_H in [+0, 1e12], x_HI in [+0, 1], wherever they lie."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,top", [("set_density", 1e12), ("set_xHI", 1.0)])
def test_edges_of_the_accepted_range(name, top):
    from paper_2311_01492_gb300 import api as A
    n = 67  # cells beyond a multiple of the unrolled stride
    g = A.Grid(n, 1e24)
    ok = [0.0, 5e-324, 1e-310, 0.5, math.nextafter(top, 0.0), top]
    refused = [-0.0, -5e-324, -1.0, math.nextafter(top, math.inf), 1e300, math.inf, -math.inf,
               math.nan]
    field = torch.full((n ** 3,), 0.25, device="cuda", dtype=torch.float64)
    for where in (0, n ** 3 // 2, n ** 3 - 1):
        for v in ok + refused:
            bad = field.clone()
            bad[where] = v
            assert np.signbit(bad[where].item()) == np.signbit(v)
            if v in ok and not np.signbit(v):
                getattr(g, name)(bad)
            else:
                with pytest.raises(Exception, match="RT_ERR_INVALID"):
                    getattr(g, name)(bad)
    g.close()
