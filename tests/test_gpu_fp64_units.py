"""Units of the FP64 form's fixed-point sums (cluster lists): every atom's sums keep FP64 accuracy
relative to that atom's own terms, whatever the damping radii, the other elements of the table and
the other structures of the batch.

Tolerances, from the roundings of both sides.  A coordinate below 8 bohr is rounded by 2^-51 bohr, a
distance d of 6 bohr or more by 2^-52.6 d, and a force, which falls as d^-9 at most (and its part
through the coordination numbers as exp(k1 rc/d), k1 rc/d < 19), by 28 2^-52.6 = 4e-15; some 60
operations round by 60 2^-53 = 7e-15; twice that for the two sides: 2.2e-14.  Structures of up to 200
atoms: their forces relative to the largest in the structure, terms up to a hundred times that."""
import numpy as np
import pytest

from paper_2310_05279_gb300 import workloads as wl

from ._helpers import to_dev

pytestmark = pytest.mark.gpu
TOL_PAIR = 1e-13
TOL_SUM = 1e-12
DAMP = [{}, dict(a1=0.1, a2=0.5), dict(a1=0.1, a2=0.0), dict(a1=0.05, a2=0.2), dict(a1=0.02, a2=0.05),
        dict(a1=0.0, a2=0.003), dict(s8=-0.4, a1=0.05, a2=0.2)]


@pytest.fixture(scope="module")
def d3_class():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2310_05279_gb300 import D3
    return D3


def _open(pos, typ):
    return (pos, np.asarray(typ, np.int32), np.eye(3) * 40.0, np.zeros(3, np.int32))


def _cloud(g, n, span, sep):
    out = []
    while len(out) < n:
        x = g.uniform(-span, span, 3)
        if all(np.linalg.norm(x - y) > sep for y in out):
            out.append(x)
    return np.array(out)


@pytest.mark.parametrize("damp", DAMP)
@pytest.mark.parametrize("names", [("C",), wl.UNEVEN_ELEMENTS])
def test_pairs_against_oracle(d3_class, oracle_mod, names, damp):
    """Two atoms alone, every element pair and several distances, all in one batch."""
    g = np.random.Generator(np.random.PCG64(11))
    t = wl.carbon_table() if names == ("C",) else wl.random_tables(names, 1003)
    structs = []
    for a in range(len(names)):
        for b in range(a, len(names)):
            for d in (3.4, 5.0, 8.0, 11.0):
                u = g.normal(size=3)
                u *= 0.5 * d / np.linalg.norm(u)
                structs.append(_open(np.array([-u, u]), [a, b]))
    b = wl.batch_of(structs, t)
    prm = dict(wl.PBE_BJ, **damp)
    ref = oracle_mod.compute_batch(b, prm)
    d3 = d3_class(t, prm, precision="fp64")
    pos, typ = to_dev(b)
    for sites in (False, True):
        out = d3.compute_batch(pos, typ, b.offsets, b.cells, b.pbc, e_atom=sites)
        d3.sync_status()
        assert d3.list_stats()["list_mode"] == 1
        F, E, W = (out[k].cpu().numpy() for k in ("F", "E", "W"))
        size = np.abs(ref["F"]).max(1)
        assert (np.abs(F - ref["F"]).max(1) <= TOL_PAIR * size).all()
        assert (np.abs(E - ref["E"]) <= TOL_PAIR * np.abs(ref["E"])).all()
        wr = ref["W"].reshape(-1, 9)
        assert (np.abs(W.reshape(-1, 9) - wr).max(1) <= TOL_PAIR * np.abs(wr).max(1)).all()
        if sites:
            half = np.repeat(ref["E"] / 2, 2)
            assert (np.abs(out["e_atom"].cpu().numpy() - half) <= TOL_PAIR * np.abs(half)).all()


@pytest.mark.parametrize("rc", [{}, dict(rc_cn=1.2), dict(rc_cn=4.0), dict(rc_disp=5.0, rc_cn=6.0)])
@pytest.mark.parametrize("damp", DAMP)
def test_molecules_and_dense_clouds(d3_class, damp, rc):
    """Molecules of one element beside mixed ones, atoms as near as 0.3 A and a periodic structure, against
    the per-atom-list pass, structure by structure.  (An R_cn below 4 A keeps that pass: there the partners
    beyond R_cn, whose terms are only counted, would set the units.)"""
    g = np.random.Generator(np.random.PCG64(12))
    n_el = len(wl.UNEVEN_ELEMENTS)
    t = wl.random_tables(wl.UNEVEN_ELEMENTS, 1003)
    structs = [_open(_cloud(g, 8, 1.8, 1.0), np.full(8, k)) for k in range(n_el)]
    structs += [_open(_cloud(g, 12, 2.2, 1.0), g.integers(0, n_el, 12)) for _ in range(3)]
    structs += [_open(_cloud(g, 200, 3.0, 0.3), g.integers(0, n_el, 200))]
    structs += [wl.random_structure(g, 90, wl.UNEVEN_ELEMENTS)]
    b = wl.batch_of(structs, t)
    d3 = d3_class(t, dict(wl.PBE_BJ, **damp, **rc), precision="fp64")
    pos, typ = to_dev(b)
    full = d3.compute_batch(pos, typ, b.offsets, b.cells, b.pbc, w_atom=True, e_atom=True)
    assert d3.list_stats()["list_mode"] == 0
    full = {k: v.cpu().numpy() for k, v in full.items()}
    for sites in (False, True):
        out = d3.compute_batch(pos, typ, b.offsets, b.cells, b.pbc, e_atom=sites)
        d3.sync_status()
        assert d3.list_stats()["list_mode"] == (0 if rc.get("rc_cn") == 1.2 else 1)
        out = {k: v.cpu().numpy() for k, v in out.items()}
        for s in range(b.nstruct):
            i = slice(b.offsets[s], b.offsets[s + 1])
            for k, sl in (("F", i), ("E", s), ("W", s)) + ((("e_atom", i),) if sites else ()):
                x, y = out[k][sl], full[k][sl]
                assert np.abs(x - y).max() <= TOL_SUM * np.abs(y).max(), (k, s)


def test_positions_near_the_origin(d3_class, oracle_mod):
    """Pairs 0.2 A apart about the origin, hardly damped, so that energies go as d^-8: integer positions keep
    what FP64 holds of small coordinates.  With positions to 2^-55 bohr (d = 0.38 bohr) 8 2^-54 / 0.38 =
    1.2e-15, some 30 operations a side 6.7e-15."""
    g = np.random.Generator(np.random.PCG64(13))
    t = wl.carbon_table()
    structs = []
    for _ in range(200):
        u = g.normal(size=3)
        u *= 0.1 / np.linalg.norm(u)
        structs.append(_open(np.array([-u, u]), [0, 0]))
    b = wl.batch_of(structs, t)
    prm = dict(wl.PBE_BJ, a1=0.0, a2=0.003)
    ref = oracle_mod.compute_batch(b, prm)
    d3 = d3_class(t, prm, precision="fp64")
    pos, typ = to_dev(b)
    E = d3.compute_batch(pos, typ, b.offsets, b.cells, b.pbc)["E"].cpu().numpy()
    d3.sync_status()
    assert d3.list_stats()["list_mode"] == 1
    assert (np.abs(E - ref["E"]) <= 8e-15 * np.abs(ref["E"])).all()


@pytest.mark.parametrize("shift", [0.0, 150.0, 600.0, 3000.0])
def test_positions_far_from_the_origin(d3_class, shift):
    """Coordinates on both sides of the lines where the unit of the positions changes, up to the largest
    ones taken: the same positions through the per-atom lists."""
    g = np.random.Generator(np.random.PCG64(14))
    t = wl.random_tables(wl.UNEVEN_ELEMENTS, 1003)
    structs = [(_cloud(g, 20, 3.0, 1.0) + s * shift, g.integers(0, 6, 20).astype(np.int32), np.eye(3) * 30.0,
                np.zeros(3, np.int32)) for s in (np.ones(3), np.array([-1.0, 0.0, 0.5]))]
    structs.append(wl.random_structure(g, 60, wl.UNEVEN_ELEMENTS))
    b = wl.batch_of(structs, t)
    d3 = d3_class(t, precision="fp64")
    pos, typ = to_dev(b)
    full = d3.compute_batch(pos, typ, b.offsets, b.cells, b.pbc, w_atom=True)
    out = d3.compute_batch(pos, typ, b.offsets, b.cells, b.pbc)
    d3.sync_status()
    assert d3.list_stats()["list_mode"] == 1
    for s in range(b.nstruct):
        i = slice(b.offsets[s], b.offsets[s + 1])
        for k, sl in (("F", i), ("E", s), ("W", s)):
            x, y = out[k][sl].cpu().numpy(), full[k][sl].cpu().numpy()
            assert np.abs(x - y).max() <= TOL_SUM * np.abs(y).max(), (k, s)
