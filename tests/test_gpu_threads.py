"""Two handles on two host threads, with plans that need different amounts of shared memory in the same
kernels: every call of either succeeds, with its own results."""
import threading

import numpy as np
import pytest

from paper_2310_05279_gb300 import workloads as wl

from ._helpers import to_dev

pytestmark = pytest.mark.gpu


def _sparse():
    """A few atoms in a box whose grid nearly fills a block's shared memory."""
    g = np.random.Generator(np.random.PCG64(31))
    pos = g.uniform(0.0, 90.0, (60, 3))
    return wl.batch_of([(pos, np.zeros(60, np.int32), np.eye(3) * 90.0, np.zeros(3, np.int32))], wl.carbon_table())


def _sheet(nx, ny):
    g = np.random.Generator(np.random.PCG64(32))
    return wl.batch_of([wl.bilayer(nx, ny, 3.4, wl.BOND, 20.0, 0.02, g)], wl.carbon_table())


@pytest.mark.parametrize("pair", ["split", "struct"])
def test_two_handles_two_threads(pair):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2310_05279_gb300 import D3, _lib
    # lists split over 8 and over 4 warps; grids of thousands of cells and of a few dozen
    batches = [_sheet(2, 4), _sheet(16, 16)] if pair == "split" else [_sparse(), wl.bilayer_ab_64()]
    want, errors = [], []
    for b in batches:
        pos, typ = to_dev(b)
        want.append((pos, typ, D3(b.tables).compute_batch(pos, typ, b.offsets, b.cells, b.pbc)))
    torch.cuda.synchronize()

    def run(b, pos, typ, ref):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                d3 = D3(b.tables)
                d3.set_graphs(False)
                out = d3.compute_batch(pos, typ, b.offsets, b.cells, b.pbc)
                # the C entry in a tight loop (the interpreter's own work between calls would keep them apart)
                off, cells, pbc = (np.ascontiguousarray(x, t) for x, t in ((b.offsets, np.int64), (b.cells, np.float64),
                                                                          (b.pbc, np.int32)))
                args = (d3.h, b.nstruct, off.ctypes.data_as(_lib._lp), pos.data_ptr(), typ.data_ptr(),
                        cells.ctypes.data_as(_lib._dp), pbc.ctypes.data_as(_lib._ip), out["E"].data_ptr(),
                        out["F"].data_ptr(), out["W"].data_ptr(), torch.cuda.current_stream().cuda_stream)
                for k in range(5000):
                    st = d3.lib.d3_compute_batch(*args)
                    if st != 0:
                        d3._check(st)
                d3.sync_status()
                assert all(torch.equal(out[k], ref[k]) for k in ref)
        except Exception as e:  # noqa: BLE001 (reported by the main thread)
            errors.append(f"{type(e).__name__}: {e}")

    threads = [threading.Thread(target=run, args=(b, *w)) for b, w in zip(batches, want)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
