"""Several gradients carried back through one projection at once (objective and constraint): on two streams, from two
threads, and in captured graphs replayed beside plain calls.  Cells on both sides of 2^18 elements, above which a
call may work through a buffer of the map, with and without the octant mirror.  Every call must give the bits that
it gives alone (same FP64 sums in the same order)."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CELLS = [("sc", 64, 2, True), ("sc", 64, 1, False), ("fcc", 96, 1, False), ("bcc", 40, 1, False)]


@pytest.fixture(params=CELLS, ids=lambda c: f"{c[0]}{c[1]}")
def problem(request):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1603_06855_gb300 import build_lib
    from paper_1603_06855_gb300.solver import DesignMap
    build_lib.build()
    lattice, n, spacing, octant = request.param
    dm = DesignMap(lattice, (n, n, n), spacing=spacing, octant=octant)
    rng = np.random.default_rng(n)
    dm.project(torch.from_numpy(rng.uniform(0, 1, dm.nvars)).cuda(), 4.0)
    g = [torch.from_numpy(rng.standard_normal((n, n, n))).cuda() for _ in range(2)]
    want = [dm.backprop(t).clone() for t in g]
    torch.cuda.synchronize()
    assert not torch.equal(want[0], want[1])
    yield dm, g, want
    torch.cuda.synchronize()
    dm.close()


def test_two_streams(problem):
    dm, g, want = problem
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    out = []
    for i in range(40):
        for j in (0, 1):
            with torch.cuda.stream(streams[j]):
                out.append((j, dm.backprop(g[j])))
    torch.cuda.synchronize()
    for j, gx in out:
        assert torch.equal(gx, want[j])


def test_two_threads(problem):
    dm, g, want = problem
    out, dev = [[], []], torch.cuda.current_device()

    def work(j):
        torch.cuda.set_device(dev)
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(40):
                out[j].append(dm.backprop(g[j]))

    th = [threading.Thread(target=work, args=(j,)) for j in (0, 1)]
    [t.start() for t in th]
    [t.join() for t in th]
    torch.cuda.synchronize()
    for j in (0, 1):
        assert len(out[j]) == 40 and all(torch.equal(gx, want[j]) for gx in out[j])


def test_captured_beside_plain(problem):
    dm, g, want = problem
    side = torch.cuda.Stream()
    graphs, held = [], []
    for j in (0, 1):
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            held.append(dm.backprop(g[j]))
        graphs.append(graph)
    plain = []
    for _ in range(10):
        for j in (0, 1):
            with torch.cuda.stream(side):
                graphs[j].replay()
        plain.append(dm.backprop(g[0]))
    torch.cuda.synchronize()
    assert all(torch.equal(held[j], want[j]) for j in (0, 1))
    assert all(torch.equal(gx, want[0]) for gx in plain)
