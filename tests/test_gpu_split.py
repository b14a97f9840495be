"""Long cluster lists split over a block (dispersion pass of the mixed form): in a batch of
few clusters, lists longer than a chunk are evaluated by several warps and summed chunk by
chunk in list order.  The results are those of one warp per list, bit for bit: a structure
alone (split lists) against the same structure in a large batch (unsplit)."""
import pytest

from paper_2310_05279_gb300 import workloads as wl

from ._helpers import to_dev

pytestmark = pytest.mark.gpu


def _carbon():
    """128 bilayers of 1440 atoms (one type: image atoms have rows of their own) and a 64-atom one
    (fewer clusters than SMs: eight warps per list)."""
    b = wl.bilayer_scan(seed=1)
    return wl.batch_of([b.structure(s) for s in range(b.nstruct)] + [wl.bilayer_ab_64().structure(0)], b.tables)


def _mixed():
    """Six types (image atoms resolve to their source), 20 to 4000 atoms, clusters of fewer than 8 atoms among them."""
    return wl.uneven_batch(seed=31, nstruct=300, n_range=(20, 4000))


@pytest.mark.parametrize("site", [False, True])
@pytest.mark.parametrize("make,pick", [(_carbon, (0, 77, 128)), (_mixed, (0, 1, 2))])
def test_split_lists_give_the_same_bits(make, pick, site):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2310_05279_gb300 import D3
    b = make()
    big = D3(b.tables)
    p, t = to_dev(b)
    all_ = big.compute_batch(p, t, b.offsets, b.cells, b.pbc, e_atom=site, cn=site)
    big.sync_status()
    assert big.list_stats()["clusters"] > 128 * 152
    sizes = b.offsets[1:] - b.offsets[:-1]
    if make is _mixed:
        pick = (int(sizes.argmin()), int(sizes.argmax()), int(abs(sizes - 200).argmin()))
    for s in pick:
        one = b.subset([s])
        d3 = D3(b.tables)
        q, u = to_dev(one)
        out = d3.compute_batch(q, u, one.offsets, one.cells, one.pbc, e_atom=site, cn=site)
        d3.sync_status()
        a, e = int(b.offsets[s]), int(b.offsets[s + 1])
        for k in out:
            ref = all_[k][s:s + 1] if k in ("E", "W") else all_[k][a:e]
            assert torch.equal(out[k], ref), (s, k)
