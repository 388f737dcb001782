"""Column densities whose quotient tau / sigma0 lies next to a rounding tie: the batched
and plain schedules and the allocation-free entry point have the bits of the division."""
import ctypes as C
from math import ldexp

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _near_ties(B, count):
    out = []
    for d in range(1, 100000, 2):
        for sign in (1, -1):
            M = sign * d * pow(B, -1, 2 ** 54) % 2 ** 54
            a = (B * M - sign * d) >> 54
            if M >> 53 and a >> 52 == 1:
                out.append(a)
        if len(out) >= count:
            return out[:count]


@pytest.mark.parametrize("sigma0", [6.3e-18, 6.1e-18, 5.97e-18, 6.47e-18, 6.63e-18, 6.79e-18])
def test_columns_next_to_rounding_ties(sigma0):
    from paper_2311_01492_gb300 import api as A, _lib as L
    B = int(ldexp(sigma0, 110)) | 1  # (odd, 53 bits)
    SIGMA0 = ldexp(B, -110)
    assert B >> 52 == 1
    n, count = 8, 64
    ties = _near_ties(B, count)
    # with a cell of 1 cm, tau = sigma0 n_H: the n_H whose product rounds to 2 a
    nH = np.full(n ** 3, 1e-4)
    nH[:count] = [ldexp(a, -50) / ldexp(B, -52) for a in ties]
    assert np.array_equal(0.5 * (SIGMA0 * nH[:count]), [ldexp(a, -109) for a in ties])
    pos = np.stack(np.unravel_index(np.arange(count), (n, n, n)), 1).astype(np.int32)
    f = dict(device="cuda", dtype=torch.float64)
    g = A.Grid(n, 1.0, sigma0=SIGMA0)
    g.set_tables("grey_exact")
    d_n, d_x = torch.tensor(nH, **f), torch.ones(n ** 3, **f)
    g.set_density(d_n)
    g.set_xHI(d_x)
    g.set_sources(torch.tensor(pos, device="cuda"), torch.full((count,), 1e50, **f),
                  torch.full((count,), 1.5, **f))
    want = np.array([ldexp(a, -109) / SIGMA0 for a in ties])
    out = torch.empty(n ** 3, **f)
    for s in range(count):
        batched = g.source_coldens(s).cpu().numpy()
        assert batched[s] == want[s], s
        assert np.array_equal(batched, g.source_coldens(s, schedule="plain").cpu().numpy())
        L.check(L.lib().rt_coldens_single_noalloc(
            n, 1.0, SIGMA0, C.c_void_p(d_n.data_ptr()), C.c_void_p(d_x.data_ptr()),
            *(int(v) for v in pos[s]), 1.5, C.c_void_p(out.data_ptr()),
            C.c_void_p(torch.cuda.current_stream().cuda_stream)))
        assert np.array_equal(batched, out.cpu().numpy())
    g.close()
