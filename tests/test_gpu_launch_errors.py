"""A launch that the runtime refuses is reported by the library's launcher."""
import ctypes as C

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
def test_refused_removal_of_an_ensemble(precision):
    """An empty grid: refused on the host, nothing runs."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_24010_gb300 import build
    fn = C.CDLL(build.build())["_ZN3cpk18compact_ens_launchEiPKNS_4BufsEiiP11CUstream_st"]
    fn.argtypes = [C.c_int, C.c_void_p, C.c_int, C.c_int, C.c_void_p]
    assert fn(precision, None, 1, 0, None) != 0
    torch.cuda.synchronize()  # no error left behind
