"""Three-body pass: every unordered pair of a list is dealt to the lanes once, whatever the list's
length. Clusters in which all n atoms see one another: lists of n - 1 = 0 .. 130 entries, around the
edges of 32 lanes, odd and even (the pairs half way round), and of the staging areas (64, 128)."""
import numpy as np
import pytest

from paper_2310_05279_gb300 import workloads as wl

from ._helpers import to_dev
from .test_gpu_atm import assert_rel

pytestmark = pytest.mark.gpu
SIZES = [1, 2, 3, 4, 5, 6, 9, 10, 32, 33, 34, 63, 64, 65, 66, 67, 128, 129, 130, 131]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_list_lengths(oracle_mod, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2310_05279_gb300 import D3
    g = np.random.Generator(np.random.PCG64(23))
    m = np.arange(-4, 5)
    grid = np.stack(np.meshgrid(m, m, m, indexing="ij"), -1).reshape(-1, 3)
    grid = grid[np.argsort((grid**2).sum(1), kind="stable")] * 1.3
    names = ["H", "C", "O"]
    structs = [(grid[:n] + g.uniform(-0.1, 0.1, (n, 3)), g.integers(0, 3, n).astype(np.int32), np.eye(3) * 40.0,
                np.zeros(3, np.int32)) for n in SIZES]
    b = wl.batch_of(structs, wl.random_tables(names, 1017))
    p = dict(wl.PBE_BJ, s6=0.0, s8=0.0, rc_cn=10.0, s9=1.0, alpha9=16.0, rc3=10.0)
    d3 = D3(b.tables, p, precision=precision)
    pos, typ = to_dev(b)
    out = d3.compute_batch(pos, typ, b.offsets, b.cells, b.pbc)
    d3.sync_status()
    out = {k: v.cpu().numpy() for k, v in out.items()}
    ref = oracle_mod.compute_batch(b, p)
    # the tolerances of the three-body term alone; a pair left out or met twice is 1e-4 of it
    for s, n in enumerate(SIZES):
        one = {k: v[b.offsets[s]:b.offsets[s + 1]] if k == "F" else v[s:s + 1] for k, v in out.items() if k in "EFW"}
        r1 = {k: ref[k][b.offsets[s]:b.offsets[s + 1]] if k == "F" else ref[k][s:s + 1] for k in "EFW"}
        assert_rel(one, r1, np.array([0, n]), *((1e-11, 1e-10, 1e-11) if precision == "fp64" else (2e-6, 1e-5, 1e-5)))
