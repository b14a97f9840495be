"""New geometries on one handle while earlier work is still running: calls that don't wait for the
stream must not lose their geometry to the next call."""
import threading

import numpy as np
import pytest

from paper_2310_05279_gb300 import workloads as wl

from ._helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    return torch


def _empty(n):
    s = (np.zeros((0, 3)), np.zeros(0, np.int32), np.eye(3) * 9.0, np.ones(3, np.int32))
    return wl.batch_of([s] * n, wl.random_tables(wl.UNEVEN_ELEMENTS, 1003))


@pytest.mark.parametrize("other_stream", [False, True])
def test_empty_structures_before_the_next_geometry(torch_cuda, other_stream):
    """Structures without atoms take no sizing pass, so the call returns while its upload waits behind
    other work: their sums stay zero whatever geometry comes next."""
    torch = torch_cuda
    from paper_2310_05279_gb300 import D3
    a, c = wl.uneven_batch(seed=21, nstruct=6, n_range=(50, 300)), wl.uneven_batch(seed=22, nstruct=6, n_range=(40, 200))
    e = _empty(6)
    d3 = D3(a.tables)
    pa, ta = to_dev(a)
    pc, tc = to_dev(c)
    pe, te = to_dev(e)
    want = {k: v.clone() for k, v in D3(c.tables).compute_batch(pc, tc, c.offsets, c.cells, c.pbc).items()}
    d3.compute_batch(pa, ta, a.offsets, a.cells, a.pbc)  # the workspace has room for all three
    torch.cuda.synchronize()
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(s1):
        torch.cuda._sleep(200_000_000)  # about 0.1 s
        empty = d3.compute_batch(pe, te, e.offsets, e.cells, e.pbc)
    with torch.cuda.stream(s2 if other_stream else s1):
        got = d3.compute_batch(pc, tc, c.offsets, c.cells, c.pbc)
    torch.cuda.synchronize()
    assert (empty["E"] == 0).all() and (empty["W"] == 0).all()
    for k in want:
        assert torch.equal(got[k], want[k]), k


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_new_geometry_refused_under_capture(torch_cuda, precision):
    """A geometry that has not been sized is refused under capture, and the plan stays as it was: the same
    geometry outside the capture, and the earlier one, give their results."""
    torch = torch_cuda
    from paper_2310_05279_gb300 import D3, D3Error
    a, c = wl.uneven_batch(seed=23, nstruct=5, n_range=(200, 400)), wl.uneven_batch(seed=24, nstruct=5, n_range=(40, 100))
    pa, ta = to_dev(a)
    pc, tc = to_dev(c)
    d3 = D3(a.tables, precision=precision)
    first = {k: v.clone() for k, v in d3.compute_batch(pa, ta, a.offsets, a.cells, a.pbc).items()}
    want = D3(c.tables, precision=precision).compute_batch(pc, tc, c.offsets, c.cells, c.pbc)
    torch.cuda.synchronize()
    for x, px, tx in ((c, pc, tc), (_empty(5), pc[:0], tc[:0])):
        out = dict(E=torch.zeros(5, dtype=torch.float64, device="cuda"), F=torch.zeros_like(px),
                   W=torch.zeros((5, 3, 3), dtype=torch.float64, device="cuda"))
        refused = False
        with torch.cuda.graph(torch.cuda.CUDAGraph()):
            out["E"].add_(1.0)  # (something to capture)
            try:
                d3.compute_batch(px, tx, x.offsets, x.cells, x.pbc, out=out)
            except D3Error:
                refused = True
        assert refused
    got = d3.compute_batch(pc, tc, c.offsets, c.cells, c.pbc)
    again = d3.compute_batch(pa, ta, a.offsets, a.cells, a.pbc)
    d3.sync_status()
    for k in want:
        assert torch.equal(got[k], want[k]), k
        assert torch.equal(again[k], first[k]), k


def test_new_geometry_on_another_stream_while_a_thread_captures(torch_cuda):
    """The workspace changes streams with a new geometry while another stream is being captured: the call
    succeeds and the capture goes on."""
    torch = torch_cuda
    from paper_2310_05279_gb300 import D3
    a, c = wl.uneven_batch(seed=26, nstruct=4, n_range=(100, 200)), wl.uneven_batch(seed=27, nstruct=4, n_range=(40, 90))
    pa, ta = to_dev(a)
    pc, tc = to_dev(c)
    want = D3(c.tables).compute_batch(pc, tc, c.offsets, c.cells, c.pbc)
    d3 = D3(a.tables)
    d3.compute_batch(pa, ta, a.offsets, a.cells, a.pbc)
    torch.cuda.synchronize()
    x, s, got = torch.zeros(8, device="cuda"), torch.cuda.Stream(), {}
    out = {k: torch.empty_like(v) for k, v in want.items()}

    def other():
        with torch.cuda.stream(s):
            try:
                d3.compute_batch(pc, tc, c.offsets, c.cells, c.pbc, out=out)
                s.synchronize()
                got["ok"] = True
            except Exception as e:  # noqa: BLE001
                got["error"] = str(e)

    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="thread_local"):
        x.add_(1.0)
        t = threading.Thread(target=other)
        t.start()
        t.join()
        x.add_(1.0)
    assert got == {"ok": True}
    graph.replay()
    torch.cuda.synchronize()
    assert (x == 2.0).all()
    for k in want:
        assert torch.equal(out[k], want[k]), k


def test_new_geometry_waits_for_a_callers_graph(torch_cuda):
    """A caller's graph that runs on a stream the handle has not seen keeps its workspace until it is done."""
    torch = torch_cuda
    from paper_2310_05279_gb300 import D3
    a, c = wl.uneven_batch(seed=28, nstruct=6, n_range=(200, 400)), wl.uneven_batch(seed=29, nstruct=6, n_range=(100, 300))
    pa, ta = to_dev(a)
    pc, tc = to_dev(c)
    d3 = D3(a.tables)
    first = {k: v.clone() for k, v in d3.compute_batch(pa, ta, a.offsets, a.cells, a.pbc).items()}
    want = D3(c.tables).compute_batch(pc, tc, c.offsets, c.cells, c.pbc)
    out = {k: torch.zeros_like(v) for k, v in first.items()}
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        d3.compute_batch(pa, ta, a.offsets, a.cells, a.pbc, out=out)
    d3.compute_batch(pa, ta, a.offsets, a.cells, a.pbc)  # the handle's last stream is the current one again
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream()):
        torch.cuda._sleep(100_000_000)
        graph.replay()
    got = d3.compute_batch(pc, tc, c.offsets, c.cells, c.pbc)
    torch.cuda.synchronize()
    for k in first:
        assert torch.equal(out[k], first[k]), k
        assert torch.equal(got[k], want[k]), k


def test_skin_after_a_captured_call_of_the_other_lists(torch_cuda):
    """With a skin, a captured build counts as not run: the next ordinary call builds its own lists."""
    torch = torch_cuda
    from paper_2310_05279_gb300 import D3
    b = wl.uneven_batch(seed=30, nstruct=4, n_range=(60, 200))
    pos, typ = to_dev(b)
    d3 = D3(b.tables, skin=0.5)
    want = {k: v.clone() for k, v in d3.compute_batch(pos, typ, b.offsets, b.cells, b.pbc).items()}
    wa = d3.compute_batch(pos, typ, b.offsets, b.cells, b.pbc, w_atom=True)  # the lists are per atom now
    out = {k: torch.empty_like(v) for k, v in want.items()}
    torch.cuda.synchronize()
    n0 = d3.build_count()
    with torch.cuda.graph(torch.cuda.CUDAGraph()):
        d3.compute_batch(pos, typ, b.offsets, b.cells, b.pbc, out=out)
    got = d3.compute_batch(pos, typ, b.offsets, b.cells, b.pbc)
    d3.sync_status()
    assert d3.build_count() == n0 + 1
    for k in want:
        assert torch.equal(got[k], want[k]), k
    assert wa["w_atom"].isfinite().all()


def test_an_odd_structure_is_forgotten(torch_cuda):
    """The list capacities of later geometries follow the last ones, not the oddest ever seen: a dense drop in
    a wide cell, then twenty ordinary structures, then a large box, which takes the memory it takes alone."""
    torch = torch_cuda
    from paper_2310_05279_gb300 import D3
    g = np.random.Generator(np.random.PCG64(33))
    box = wl.mof_like_box(seed=34, ncell=36)
    drop = g.normal(size=(400, 3))
    drop *= 5.0 * g.uniform(0.0, 1.0, (400, 1)) ** (1 / 3) / np.linalg.norm(drop, axis=1, keepdims=True)
    odd = wl.batch_of([(drop + 60.0, g.integers(0, 5, 400).astype(np.int32), np.eye(3) * 120.0, np.ones(3, np.int32))],
                      box.tables)
    small = wl.mof_like_box(seed=35, ncell=8)

    def used(d3):
        free0 = torch.cuda.mem_get_info()[0]
        pos, typ = to_dev(box)
        d3.compute_batch(pos, typ, box.offsets, box.cells, box.pbc)
        d3.sync_status()
        del pos, typ
        torch.cuda.empty_cache()
        return free0 - torch.cuda.mem_get_info()[0]

    d3 = D3(box.tables)
    pos, typ = to_dev(odd)
    d3.compute_batch(pos, typ, odd.offsets, odd.cells, odd.pbc)
    pos, typ = to_dev(small)
    for k in range(20):
        d3.compute_batch(pos * (1 + 0.001 * k), typ, small.offsets, small.cells * (1 + 0.001 * k), small.pbc)
    d3.sync_status()
    after = used(d3)
    alone = used(D3(box.tables))
    assert after <= 1.25 * alone
