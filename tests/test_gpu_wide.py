"""CN and chain passes with 8 lanes per atom (few atoms) against one thread per atom: the sums are
added in list order either way, so a structure alone gives the bits it has in a large batch (which
takes one thread per atom; its per-structure sums are the same kernel)."""
import numpy as np
import pytest

from paper_2310_05279_gb300 import workloads as wl

from ._helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ntypes,max_ref", [(1, 5), (6, 4), (16, 7)])
def test_same_bits_as_one_thread_per_atom(ntypes, max_ref):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2310_05279_gb300 import D3
    g = np.random.Generator(np.random.PCG64(40 + ntypes))
    tabs = wl.random_tables([f"E{k}" for k in range(ntypes)], 41, max_ref=max_ref, nref_max=max_ref)
    small = [(np.array([[0.3, 0.2, 0.1]]), np.zeros(1, np.int32), np.diag([3.1, 3.3, 3.7]), np.ones(3, np.int32)),
             (np.array([[0.0, 0.0, 0.0], [0.0, 0.0, 30.0]]), np.zeros(2, np.int32), np.eye(3) * 60.0,
              np.zeros(3, np.int32))]  # empty lists
    for n in (7, 33, 500):
        pos, _, cell, pbc = wl.random_structure(g, n, wl.UNEVEN_ELEMENTS, dens_range=(2.0, 2.2))
        small.append((pos, g.integers(0, ntypes, n).astype(np.int32), cell, pbc))
    filler = wl.mof_like_box(seed=9, ncell=41)  # 275,684 atoms
    big = wl.batch_of(small + [(filler.pos, filler.types % ntypes, filler.cells[0], filler.pbc[0])], tabs)
    d3 = D3(tabs)
    pos, typ = to_dev(big)
    ref = d3.compute_batch(pos, typ, big.offsets, big.cells, big.pbc, e_atom=True, cn=True)
    d3.sync_status()
    for s in range(len(small)):
        one = big.subset([s])
        q, t = to_dev(one)
        d1 = D3(tabs)
        out = d1.compute_batch(q, t, one.offsets, one.cells, one.pbc, e_atom=True, cn=True)
        d1.sync_status()
        a, e = int(big.offsets[s]), int(big.offsets[s + 1])
        for k in ("F", "e_atom", "cn"):
            assert torch.equal(out[k], ref[k][a:e]), (s, k)
        for k in ("E", "W"):  # (summed in FP64 by another kernel)
            x, y = out[k][0], ref[k][s]
            assert (x - y).abs().max() <= 1e-13 * max(y.abs().max().item(), 1e-30) + 1e-18, (s, k)
