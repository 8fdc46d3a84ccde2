"""A launch that CUDA refuses leaves no error behind: the call that made it
reports it, and the next call, on another stream, is not failed for it. The
refusal is made on the host: a stream whose capture has been invalidated takes
no launch."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from gpu_util import Workspace, empty, to_dev  # noqa: E402
from test_gpu_batch import GEN, ITEM, table_to_dev  # noqa: E402

RELAXED, NON_BLOCKING = 2, 1


@pytest.fixture(scope="module")
def ka(cuda_ok):
    import paper_1709_07781_gb300 as m
    return m


@pytest.fixture()
def refused(ka):
    """A stream that refuses launches once its second value is called, and a good one
    (both of the library's own CUDA runtime)."""
    rt = ka._lib.lib
    bad, good, graph = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
    for s in (bad, good):
        assert rt.cudaStreamCreateWithFlags(ctypes.byref(s), NON_BLOCKING) == 0

    def refuse():
        assert rt.cudaStreamBeginCapture(bad, RELAXED) == 0
        assert rt.cudaStreamSynchronize(bad) != 0  # not allowed in a capture: it is invalid from here on
        rt.cudaGetLastError()

    yield bad.value, refuse, good.value
    rt.cudaStreamEndCapture(bad, ctypes.byref(graph))
    rt.cudaGetLastError()
    for s in (bad, good):
        assert rt.cudaStreamSynchronize(s) == 0
        assert rt.cudaStreamDestroy(s) == 0


@pytest.mark.parametrize("what", ["wave", "tma", "scan", "batch", "generate", "map"])
def test_the_next_call_is_not_failed_for_it(ka, refused, what):
    bad, refuse, good = refused
    n = 1 << 16
    x, y, z, count = empty(n, 1), empty(n), empty(n), empty(1)
    ws, bs = Workspace(ka, n), Workspace(ka, n, None, 1)
    item, gen = np.zeros(1, ITEM), np.zeros(1, GEN)
    item["in"], item["out"], item["count"], item["n"] = x.data_ptr(), y.data_ptr(), count.data_ptr(), n
    item["pred"] = ka.KA_PRED_POPC_ODD
    gen["out"], gen["n"] = y.data_ptr(), n
    d_item, d_gen = table_to_dev(item), table_to_dev(gen)

    def call(stream):
        if what in ("wave", "tma"):
            return ka.ka_compact(x, n, None, ka.KA_PRED_POPC_ODD, 0, 0, y, count, ws.ptr, ws.nbytes,
                                 None if what == "wave" else (768, 16), stream)
        if what == "scan":
            return ka.ka_exclusive_scan(x, n, None, y, count, ws.ptr, ws.nbytes, (512, 16), stream)
        if what == "batch":
            return ka.ka_compact_batch(d_item, 1, 1, bs.ptr, bs.nbytes, stream=stream)
        if what == "generate":
            return ka.ka_generate_batch(d_gen, 1, 1, bs.ptr, bs.nbytes, stream)
        return ka.ka_map_hash(x, n, None, y, None, stream)

    assert call(good) == 0  # (set-up of a first call: function attributes, occupancy)
    torch.cuda.synchronize()
    refuse()
    assert call(bad) == ka.KA_E_CUDA
    assert ka.ka_map_hash(x, n, None, z, None, good) == 0
    assert call(good) == 0
