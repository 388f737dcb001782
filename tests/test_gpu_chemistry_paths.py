"""The chemistry kernel's form for short decays and its general one side by side in one
warp, around the values where it changes over, against the same iteration in extended
precision.  The general form loses digits where x0 and <x> are far below the equilibrium
(x_eq + (x0 - x_eq) m with m near 1): the bound carries that factor."""
import numpy as np
import pytest

from paper_2311_01492_gb300 import synth as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _reference(nH, x0, G, dt, alpha, C_H):
    L = np.longdouble
    nH, x0, G = (np.asarray(v, dtype=L) for v in (nH, x0, G))
    xa, xn, live = x0.copy(), x0.copy(), np.ones(len(x0), bool)
    for _ in range(50):
        ne = nH * xa
        rate = G + ne * (L(C_H) + L(alpha))
        ok = rate > 0
        r = np.where(ok, rate, 1)
        xeq, y = (G + ne * L(C_H)) / r, L(dt) * r
        new = np.where(ok, xeq + (x0 - xeq) * (-np.expm1(-y) / y), x0)
        end = np.where(ok, xeq + (x0 - xeq) * np.exp(-y), x0)
        done = np.abs(new - xa) <= L(1e-10) * new
        xa, xn = np.where(live, new, xa), np.where(live, end, xn)
        live &= ~done
    return xa, xn, int(np.sum(np.abs(x0 - xa) > L(1e-3) * (1 - xa))), xeq


@pytest.mark.parametrize("C_H", [0.0, 1e-18])
@pytest.mark.parametrize("block", [1, 32])  # cells in a row with the same regime
def test_chemistry_regimes_match_extended_precision(block, C_H):
    from paper_2311_01492_gb300 import api as A
    n = 16
    rng = np.random.default_rng(5)
    dt, alpha = 5 * S.MYR_S, 2.59e-13
    # y = dt (G + n_e alpha) on both sides of 1/4 and of 1; equilibria from 0 to 1
    k = np.repeat(rng.permutation(n ** 3 // block), block)
    y = 10.0 ** (-6 + 9 * (k / k.max()))
    y[k % 7 == 0] = 0.25 * (1 + (rng.integers(-3, 4, n ** 3)[k % 7 == 0]) * 2.0 ** -50)
    share = 10.0 ** rng.uniform(-30, 0, n ** 3 // block)[k]  # of the photons in the rate
    share[k % 5 == 0] = 0.0
    share[y > 0.1] = 1.0  # (recombination alone converges too slowly there to stop alike)
    G = share * y / dt
    x0 = rng.uniform(0.0, 1.0, n ** 3)
    x0[k % 11 == 0] *= 1e-12
    x0[k % 13 == 0] = 0.0
    nH = np.maximum((1 - share) * y / dt / alpha / np.maximum(x0, 1e-3), 1e-12)
    ref_a, ref_n, ref_c, xeq = _reference(nH, x0, G, dt, alpha, C_H)
    g = A.Grid(n, S.MPC_CM)
    d = lambda v: torch.tensor(v, device="cuda", dtype=torch.float64)  # noqa: E731
    g.set_density(d(nH))
    xa, xn, cnt = g.chemistry_step(d(G), d(x0), d(x0), dt, alpha_H=alpha, C_H=C_H)
    # 1e-12 as the existing parity test (a pass more or less moves a converged cell by less
    # than 1e-10 times its contraction, at most about 1e-2 here), and eight roundings of
    # the larger terms: expm1, two divisions, y, the difference, product, sum and n_e
    for got, ref in ((xa, ref_a), (xn, ref_n)):
        got = got.cpu().numpy()
        bound = 1e-12 * np.abs(ref) + 8 * 2.0 ** -53 * np.maximum(np.abs(x0 - xeq), np.abs(ref))
        assert np.all(np.abs(got - ref) <= bound)
    assert int(cnt) == ref_c
    g.close()
