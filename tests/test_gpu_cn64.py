"""FP64 coordination numbers from integer pair vectors and the integer exponential: dimers at
distances from far below the covalent radii (f = 1) to R_cn (f near 1e-5 and less) and beyond,
in the forward's form and in that of the per-atom virial, against long double."""
import numpy as np
import pytest

from paper_2310_05279_gb300 import workloads as wl

from ._helpers import to_dev

pytestmark = pytest.mark.gpu
BOHR = 0.529177210903


@pytest.mark.parametrize("w_atom", [False, True])
@pytest.mark.parametrize("k1", [16.0, 3.0, 200.0])
def test_dimers(w_atom, k1):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2310_05279_gb300 import D3
    g = np.random.Generator(np.random.PCG64(64))
    n = 400
    tabs = wl.random_tables(["H", "C", "O"], 12)
    r = np.concatenate([10.0 ** g.uniform(-4, -0.5, 50), g.uniform(0.3, 6.2, n - 50)])
    u = g.normal(size=(n, 3))
    d = u / np.linalg.norm(u, axis=1)[:, None] * r[:, None]
    types = g.integers(0, 3, (n, 2)).astype(np.int32)
    b = wl.batch_of([(np.stack([np.zeros(3), d[k]]), types[k], np.eye(3) * 30.0, np.zeros(3, np.int32))
                     for k in range(n)], tabs)
    prm = dict(wl.PBE_BJ, k1=k1)
    d3 = D3(tabs, prm, precision="fp64")
    pos, typ = to_dev(b)
    out = d3.compute_batch(pos, typ, b.offsets, b.cells, b.pbc, cn=True, **({"w_atom": True} if w_atom else {}))
    d3.sync_status()
    got = out["cn"].cpu().numpy().reshape(n, 2)
    rb = np.sqrt((d.astype(np.longdouble) ** 2).sum(1)) / np.longdouble(BOHR)
    rc = np.longdouble(prm["k2"]) * (tabs.rcov[types[:, 0]] + tabs.rcov[types[:, 1]]).astype(np.longdouble)
    x = np.longdouble(k1) * (rc / rb - 1)
    f = np.where(rb < prm["rc_cn"] / BOHR, 1 / (1 + np.exp(np.minimum(-x, 11000))), 0)
    # roundings of the positions, r, k1 rc, x (an absolute error of x is a relative one of f,
    # times 1 - f), the exponential, the sum and the reciprocal
    tol = 2.0 ** -53 * (8 * np.abs(k1 * rc / rb) * (1 - f) + 4 * k1 + 12) * f
    assert (np.abs(got - f[:, None]) <= tol[:, None] + 1e-300).all()
