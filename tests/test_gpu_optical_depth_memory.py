"""The scratch that optical-depth weights are traced with: allocating it does not end a
capture under way elsewhere, it makes room where the grid needs the memory for something
else, and it stays where a caller's graph holds it."""
import numpy as np
import pytest

from paper_2311_01492_gb300 import synth as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
N, NSRC = 32, 400


def _grid(A, stream=None):
    rng = np.random.default_rng(6)
    f = dict(device="cuda", dtype=torch.float64)
    g = A.Grid(N, 0.78 * S.MPC_CM, stream=stream)
    g.set_tables("bb", bits=4)
    g.set_density(torch.tensor(S.lognormal_field(N, 2e-4, seed=6).reshape(-1), **f))
    g.set_xHI(torch.tensor(rng.random(N ** 3), **f))
    pos = np.stack(np.unravel_index(rng.choice(N ** 3, NSRC, replace=False), (N, N, N)), 1)
    src = (torch.tensor(pos.astype(np.int32), device="cuda"),
           torch.tensor(10.0 ** rng.uniform(50, 52, NSRC), **f), torch.full((NSRC,), 9.0, **f))
    torch.cuda.synchronize()
    return g, src


def _close(a, b):
    """Sums of at most NSRC non-negative terms, each with at most eight roundings."""
    a, b = a.cpu().numpy(), b.cpu().numpy()
    return np.all(np.abs(a - b) <= (NSRC + 8) * 2.0 ** -52 * b) and b.max() > 0


def test_allocating_leaves_a_capture_elsewhere_alone():
    from paper_2311_01492_gb300 import api as A
    g, src = _grid(A)
    x = torch.zeros(8, device="cuda")
    held = A.device_memory_in_use()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=torch.cuda.Stream(), capture_error_mode="global"):
        x += 1
        g.set_interpolation("optical_depth")
        x += 1
    assert A.device_memory_in_use() > held
    x.zero_()
    graph.replay()
    assert x.tolist() == [2.0] * 8
    g.close()


def test_it_makes_room_for_the_grid():
    from paper_2311_01492_gb300 import api as A
    g, src = _grid(A)
    g.set_sources(*src)
    g.set_interpolation("optical_depth")
    ref = g.raytrace()
    rng = np.random.default_rng(2)
    more = 20 * NSRC
    big = (torch.tensor(rng.integers(0, N, (more, 3)).astype(np.int32), device="cuda"),
           src[1].repeat(20), src[2].repeat(20))
    held = A.device_memory_in_use()
    try:
        A.set_device_memory_limit(held)
        g.set_sources(*big)   # larger arrays
        assert A.device_memory_in_use() < held
        g.set_sources(*src)
        assert _close(g.raytrace(), ref)
        g.set_interpolation("geometric")
        g.set_interpolation("optical_depth")  # (no room for it: the kernels without)
        assert _close(g.raytrace(), ref)
    finally:
        A.set_device_memory_limit(0)
    g.set_interpolation("optical_depth")
    assert _close(g.raytrace(), ref)
    g.check()
    g.close()


def test_it_stays_where_a_graph_holds_it():
    from paper_2311_01492_gb300 import api as A
    s = torch.cuda.Stream()
    g, src = _grid(A, stream=s)
    g.set_sources(*src)
    g.set_interpolation("optical_depth")
    out = torch.zeros(N ** 3, device="cuda", dtype=torch.float64)
    g.raytrace(out)
    torch.cuda.synchronize()
    ref = out.clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        g.raytrace(out)
    held = A.device_memory_in_use()
    try:
        A.set_device_memory_limit(held)
        with pytest.raises(A.RtError, match="RT_ERR_OOM"):
            g.set_tables("bb", bits=8)
    finally:
        A.set_device_memory_limit(0)
    assert A.device_memory_in_use() == held
    out.zero_()
    torch.cuda.synchronize()
    graph.replay()
    torch.cuda.synchronize()
    assert _close(out, ref)
    g.close()
