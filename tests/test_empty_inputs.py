"""Calls without entries: whatever the input pointer is, nothing of it is read.
The kernels read inputs in 16-byte pieces from the 16-byte boundary before
their first entry; an input without entries has no first entry."""
import pytest


@pytest.fixture(scope="module")
def ka():
    import paper_1709_07781_gb300 as m
    return m


@pytest.mark.parametrize("address", [0, 4, 0x1000, 0x1004, 0x1008, 0x100C, 0x7F0000000FFC])
def test_the_view_of_an_input(ka, address):
    assert ka.ka_debug_input_view(address, 0) == (0, 0, 0)
    for n in (1, 5, 1 << 32):
        assert ka.ka_debug_input_view(address, n) == (0, address & ~15, (address & 15) // 4)


@pytest.mark.gpu
@pytest.mark.parametrize("offset", [0, 1, 2, 3])
@pytest.mark.parametrize("tile", [None, (256, 4), (512, 8), (512, 16), (768, 16)])
def test_compaction_and_scan_of_no_entries(ka, cuda_ok, offset, tile):
    torch = pytest.importorskip("torch")
    from gpu_util import Workspace, empty, stream, to_host, word
    x = empty(64, 0)
    for live in (None, empty(1, 0)):
        ws = Workspace(ka, 4096)
        out, count = empty(64), empty(1)
        at = x.data_ptr() + 4 * offset
        assert ka.ka_compact(at, 0, live, ka.KA_PRED_LT, 1 << 31, 0, out, count, ws.ptr, ws.nbytes, tile, stream()) == 0
        torch.cuda.synchronize()
        assert word(count) == 0 and (to_host(out) == 0xDEADBEEF).all() and ws.status(ka) == 0
        count = empty(1)
        assert ka.ka_exclusive_scan(at, 0, live, out, count, ws.ptr, ws.nbytes, tile, stream()) == 0
        torch.cuda.synchronize()
        assert word(count) == 0 and (to_host(out) == 0xDEADBEEF).all() and ws.status(ka) == 0


@pytest.mark.gpu
@pytest.mark.parametrize("offset", [0, 1, 3])
def test_fused_run_of_no_entries(ka, cuda_ok, offset):
    from gpu_util import empty
    s, sys_h = ka.ka_system_create(0)
    assert s == 0
    x = empty(64, 0)
    _, a = ka.ka_spawn_stage(sys_h, ka.KA_STAGE_COMPACT, ka.KA_PRED_LT, 1 << 31, 0)
    _, b = ka.ka_spawn_stage(sys_h, ka.KA_STAGE_COMPACT, ka.KA_PRED_POPC_ODD, 0, 0)
    _, pipe = ka.ka_compose(b, a)
    _, ref = ka.ka_ref_wrap(sys_h, x.data_ptr() + 4 * offset, 0, 0)
    s, q = ka.ka_request(pipe, ka.make_msg([ref]))
    assert s == 0
    s, msg = ka.ka_receive(q)
    assert s == 0 and msg.count == 0
    assert ka.ka_system_destroy(sys_h, 1) == 0
