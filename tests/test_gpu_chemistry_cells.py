"""The chemistry of a cell is a function of that cell alone: the same bits wherever it lies
and whatever its neighbours are."""
import numpy as np
import pytest

from paper_2311_01492_gb300 import synth as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DT, ALPHA = 5 * S.MYR_S, 2.59e-13


def _cells(count, rng):
    """Cells of every regime in a row: y = dt / t_i from 1e-6 to 1e3, lit and dark, neutral
    and ionised, and y on both sides of 1/4."""
    y = 10.0 ** rng.uniform(-6, 3, count)
    near = rng.random(count) < 0.2
    y[near] = 0.25 * (1 + rng.integers(-3, 4, near.sum()) * 2.0 ** -50)
    share = np.where(rng.random(count) < 0.3, 0.0, 10.0 ** rng.uniform(-20, 0, count))
    x0 = rng.uniform(0.0, 1.0, count) * 10.0 ** -rng.integers(0, 4, count)
    x0[rng.random(count) < 0.05] = 0.0
    nH = np.maximum((1 - share) * y / DT / ALPHA / np.maximum(x0, 1e-3), 1e-12)
    return nH, share * y / DT, x0


def _step(sizes, nH, G, x0, C_H):
    from paper_2311_01492_gb300 import api as A
    g = A.Grid.ensemble(sizes, S.MPC_CM)
    d = lambda v: torch.tensor(v, device="cuda", dtype=torch.float64)  # noqa: E731
    g.set_density(d(nH))
    xa, xn, cnt = g.chemistry_step(d(G), d(x0), d(x0), DT, alpha_H=ALPHA, C_H=C_H)
    out = xa.cpu().numpy(), xn.cpu().numpy(), int(cnt)
    g.close()
    return out


@pytest.mark.parametrize("C_H", [0.0, 1e-18])
def test_a_cell_does_not_depend_on_its_neighbours(C_H):
    n, rng = 20, np.random.default_rng(8)
    cells = _cells(n ** 3, rng)
    xa, xn, cnt = _step([n], *cells, C_H)
    for how in range(3):  # any order: the same cells have other neighbours
        p = rng.permutation(n ** 3) if how else np.argsort(cells[1] + cells[0])
        pa, pn, pc = _step([n], *(c[p] for c in cells), C_H)
        assert np.array_equal(pa, xa[p]) and np.array_equal(pn, xn[p]) and pc == cnt
    # a box alone and behind others of an ensemble
    head = _cells(7 ** 3 + 5 ** 3, rng)
    ea, en, _ = _step([7, 5, n], *(np.concatenate(v) for v in zip(head, cells)), C_H)
    assert np.array_equal(ea[-n ** 3:], xa) and np.array_equal(en[-n ** 3:], xn)
