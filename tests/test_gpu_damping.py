"""d3_set_damping when an upload fails: asking again for the same values uploads again."""
import ctypes as C

import pytest

from paper_2310_05279_gb300 import workloads as wl

from ._helpers import to_dev

pytestmark = pytest.mark.gpu


def _cudart():
    for name in ("libcudart.so.13", "libcudart.so.12", "libcudart.so"):
        try:
            return C.CDLL(name)
        except OSError:
            pass
    pytest.skip("no shared CUDA runtime")


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_set_damping_again_after_a_failed_upload(precision):
    """A copy on the default stream is refused on the host while a stream that it would wait for is captured:
    the upload fails, and the retry with the same values must not take the tables for up to date."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2310_05279_gb300 import D3, D3Error
    rt = _cudart()
    b = wl.uneven_batch(seed=25, nstruct=4, n_range=(40, 100))
    pos, typ = to_dev(b)
    new = dict(s6=1.0, s8=1.2, a1=0.3, a2=5.1)
    want = D3(b.tables, new, precision=precision).compute_batch(pos, typ, b.offsets, b.cells, b.pbc)
    d3 = D3(b.tables, precision=precision)
    d3.compute_batch(pos, typ, b.offsets, b.cells, b.pbc)
    torch.cuda.synchronize()
    handle, graph = C.c_void_p(), C.c_void_p()
    assert rt.cudaStreamCreate(C.byref(handle)) == 0  # a stream that synchronises with the default one
    assert rt.cudaStreamBeginCapture(handle, 0) == 0
    try:
        with pytest.raises(D3Error):
            d3.set_damping(**new)
    finally:
        rt.cudaStreamEndCapture(handle, C.byref(graph))
        rt.cudaGetLastError()
        rt.cudaStreamDestroy(handle)
    d3.set_damping(**new)
    out = d3.compute_batch(pos, typ, b.offsets, b.cells, b.pbc)
    d3.sync_status()
    for k in want:
        assert torch.equal(out[k], want[k]), k
