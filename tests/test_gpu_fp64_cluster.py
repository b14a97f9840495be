"""Dispersion pass of the FP64 form over cluster half lists (64-bit fixed-point sums) against the
per-atom-list pass, which a call for per-atom virials takes, and against the oracle.

Tolerances: the sums keep some 2^-57 of an atom's largest sum and the C6 interpolation 2^-61 of its
row's largest value, so the two passes differ by FP64 rounding (1e-16 a term, sums of a few hundred
terms and of their cancellations): 1e-12 of the largest energy, force and virial component."""
import dataclasses

import numpy as np
import pytest

from paper_2310_05279_gb300 import workloads as wl

from ._helpers import to_dev

pytestmark = pytest.mark.gpu
TOL = 1e-12


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    return torch


def _batch(max_ref, ntypes, spread=(2.0, 400.0)):
    """Structures of 1 (its own images only), 2, 9, 30 and 250 atoms, tiny cells and open boundaries."""
    g = np.random.Generator(np.random.PCG64(100 + max_ref))
    tabs = wl.random_tables([f"E{k}" for k in range(ntypes)], 200 + max_ref, max_ref=max_ref, nref_max=max_ref,
                            c6_range=spread)
    structs = [(np.array([[0.3, 0.2, 0.1]]), np.zeros(1, np.int32), np.diag([3.1, 3.3, 3.7]), np.ones(3, np.int32)),
               (np.zeros((0, 3)), np.zeros(0, np.int32), np.eye(3) * 7.0, np.ones(3, np.int32)),
               (np.array([[0.0, 0.0, 0.0], [0.0, 0.0, 1.9]]), np.array([0, ntypes - 1], np.int32), np.eye(3) * 40.0,
                np.zeros(3, np.int32))]
    for n in (9, 30, 250):
        pos, _, cell, pbc = wl.random_structure(g, n, wl.UNEVEN_ELEMENTS)
        structs.append((pos, g.integers(0, ntypes, n).astype(np.int32), cell, pbc))
    return wl.batch_of(structs, tabs)


def _close(a, b):
    for k in ("E", "F", "W"):
        x, y = np.asarray(a[k]), np.asarray(b[k])
        assert np.abs(x - y).max() <= TOL * max(np.abs(y).max(), 1e-3), k


@pytest.mark.parametrize("max_ref,ntypes,damp,spread", [
    (1, 1, {}, (2.0, 400.0)), (2, 3, {}, (2.0, 400.0)), (3, 16, {}, (2.0, 400.0)), (4, 2, {}, (2.0, 400.0)),
    (5, 6, {}, (2.0, 400.0)), (6, 4, {}, (2.0, 400.0)), (7, 16, {}, (2.0, 400.0)),
    (5, 3, dict(s8=-0.4), (2.0, 400.0)),          # a negative coefficient: de/dC6 of both signs
    (5, 3, dict(rc_disp=30.0, rc_cn=8.0), (2.0, 400.0)),  # wider pair vectors
    (5, 3, dict(rc_disp=5.0, rc_cn=6.0), (2.0, 400.0)),   # R_pot below R_cn
    (5, 3, dict(a1=0.2, a2=0.8), (1e-3, 1e4)),    # steep damping, references over seven decades
])
def test_cluster_pass_matches_full_lists_and_oracle(torch_cuda, oracle_mod, max_ref, ntypes, damp, spread):
    from paper_2310_05279_gb300 import D3
    b = _batch(max_ref, ntypes, spread)
    prm = dict(wl.PBE_BJ, **damp)
    d3 = D3(b.tables, prm, precision="fp64")
    pos, typ = to_dev(b)
    res = {}
    for name, kw in (("full", dict(w_atom=True, e_atom=True)), ("cluster", {}), ("sites", dict(e_atom=True, cn=True))):
        out = d3.compute_batch(pos, typ, b.offsets, b.cells, b.pbc, **kw)
        d3.sync_status()
        assert d3.list_stats()["list_mode"] == (0 if name == "full" else 1)
        res[name] = {k: v.cpu().numpy() for k, v in out.items()}
    _close(res["cluster"], res["full"])
    _close(res["sites"], res["full"])
    ea, ref = res["sites"]["e_atom"], res["full"]["e_atom"]
    assert np.abs(ea - ref).max() <= TOL * np.abs(ref).max()
    if prm["rc_disp"] <= 12.0:
        _close(res["cluster"], oracle_mod.compute_batch(b, prm))


def test_long_lists_and_reuse(torch_cuda):
    """Lists of several splits and of several thousand entries, kept by a skin while atoms move."""
    from paper_2310_05279_gb300 import D3
    b = wl.mof_like_box(seed=5, ncell=9)
    g = np.random.Generator(np.random.PCG64(3))
    d3, ref = D3(b.tables, precision="fp64", skin=1.0), D3(b.tables, precision="fp64")
    for it in range(3):
        c = dataclasses.replace(b, pos=b.pos + g.uniform(-0.2, 0.2, b.pos.shape) * (it > 0))
        pos, typ = to_dev(c)
        out = d3.compute_batch(pos, typ, c.offsets, c.cells, c.pbc)
        full = ref.compute_batch(pos, typ, c.offsets, c.cells, c.pbc, w_atom=True)
        d3.sync_status()
        _close({k: v.cpu().numpy() for k, v in out.items()}, {k: full[k].cpu().numpy() for k in ("E", "F", "W")})
    again = d3.compute_batch(pos, typ, c.offsets, c.cells, c.pbc)
    for k in out:
        assert torch_cuda.equal(again[k], out[k]), k


def test_unbounded_damping_keeps_the_full_lists(torch_cuda, oracle_mod):
    """A damping radius of zero has no bound at r = 0: the per-atom lists stay, with the oracle's results."""
    from paper_2310_05279_gb300 import D3
    b = _batch(3, 2)
    prm = dict(wl.PBE_BJ, a1=0.0, a2=0.0)
    d3 = D3(b.tables, prm, precision="fp64")
    pos, typ = to_dev(b)
    out = d3.compute_batch(pos, typ, b.offsets, b.cells, b.pbc)
    d3.sync_status()
    assert d3.list_stats()["list_mode"] == 0
    _close({k: v.cpu().numpy() for k, v in out.items()}, oracle_mod.compute_batch(b, prm))
