"""Per-structure sums: one kernel up to 2048 atoms per structure, chunks of 2048 atoms and a second
kernel above, at the edges of both; E is the sum of the site energies, W that of its FP64 oracle."""
import numpy as np
import pytest

from paper_2310_05279_gb300 import workloads as wl

from ._helpers import assert_fp64_ok, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[2047, 1, 0, 255, 257], [2048], [2049, 256], [4096, 2048, 4097]])
def test_chunk_edges(oracle_mod, sizes):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2310_05279_gb300 import D3
    g = np.random.Generator(np.random.PCG64(61))
    names = ["H", "C", "O"]
    empty = (np.zeros((0, 3)), np.zeros(0, np.int32), np.eye(3) * 8.0, np.ones(3, np.int32))
    b = wl.batch_of([wl.random_structure(g, n, names) if n else empty for n in sizes], wl.random_tables(names, 6))
    d3 = D3(b.tables, precision="fp64")
    pos, typ = to_dev(b)
    out = d3.compute_batch(pos, typ, b.offsets, b.cells, b.pbc, e_atom=True)
    d3.sync_status()
    assert_fp64_ok(out, oracle_mod.compute_batch(b, dict(wl.PBE_BJ)), b.offsets)
    for s, n in enumerate(sizes):
        ea = out["e_atom"][int(b.offsets[s]):int(b.offsets[s + 1])]
        # two orders of a sum of n numbers: n epsilons of the sum of their magnitudes
        assert abs(ea.sum() - out["E"][s]).item() <= 2.3e-16 * max(n, 1) * ea.abs().sum().item()
