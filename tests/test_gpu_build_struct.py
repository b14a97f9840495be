"""The neighbour build by structure (one block each) against the build over the batch, which a
handle with list reuse takes (here with a skin of 1e-12 A, which leaves the lists as they are): the
same order and lists, so the same results bit for bit."""
import numpy as np
import pytest

from paper_2310_05279_gb300 import workloads as wl

from ._helpers import to_dev

pytestmark = pytest.mark.gpu
NAMES = wl.UNEVEN_ELEMENTS


def _structs(sizes, seed):
    g = np.random.Generator(np.random.PCG64(seed))
    out = []
    for n in sizes:
        if n == 0:
            out.append((np.zeros((0, 3)), np.zeros(0, np.int32), np.eye(3) * 9.0, np.ones(3, np.int32)))
            continue
        s = wl.random_structure(g, n, NAMES, dens_range=(1.5, 2.2))
        pbc = g.integers(0, 2, 3) if n % 3 == 0 else np.ones(3)
        # some atoms outside the cell, so that the wrap moves them
        pos = s[0] + (g.integers(-2, 3, (n, 3)) * pbc) @ s[2]
        out.append((pos, s[1], s[2], pbc.astype(np.int32)))
    return out


def _slab(natoms):
    """A bilayer with few images per atom: large structures stay within a block's share."""
    nx = natoms // (8 * 15)
    return [wl.bilayer(nx, 15, 3.4, wl.BOND, 20.0, 0.02, np.random.Generator(np.random.PCG64(5)))]


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("case", ["one", "edges", "many", "slab"])
def test_same_bits_as_batch_build(case, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2310_05279_gb300 import D3
    if case == "one":
        b = wl.batch_of(_structs([1], 1), wl.random_tables(NAMES, 3))
    elif case == "edges":  # around a warp, and empty structures
        b = wl.batch_of(_structs([31, 0, 32, 33, 2, 96, 0], 2), wl.random_tables(NAMES, 3))
    elif case == "many":   # more structures than SMs: half the threads per block
        b = wl.batch_of(_structs([20 + k % 40 for k in range(200)], 3), wl.random_tables(NAMES, 3))
    else:                  # around the threads of a block
        b = wl.batch_of(_slab(1080) + _slab(960) + _slab(1560), wl.carbon_table())
    pos, typ = to_dev(b)
    res, launches = [], []
    for skin in (0.0, 1e-12):
        d3 = D3(b.tables, precision=precision, skin=skin)
        d3.compute_batch(pos, typ, b.offsets, b.cells, b.pbc, e_atom=True, cn=True)  # sizes with the batch build
        d3.sync_status()
        d3.profile_reset()
        d3.set_graphs(False)
        if skin:  # a large move and back, so that the lists are built anew
            d3.compute_batch(pos + 5.0, typ, b.offsets, b.cells, b.pbc)
        out = d3.compute_batch(pos, typ, b.offsets, b.cells, b.pbc, e_atom=True, cn=True)
        d3.sync_status()
        res.append(out)
        launches.append(d3.profile_read()["launches"])
    assert launches[0] <= 9 < launches[1]  # the first took the build by structure
    for k in res[0]:
        assert torch.equal(res[0][k], res[1][k]), k
