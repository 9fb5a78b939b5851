"""Failure detection on the GPU without a fault: a bounded wait that nothing
completes gives up, the kernel records the timeout in the device error word
and returns, fc_get_error reports FC_ERR_TIMEOUT (and clears it), and the
context keeps working; the same wait with the arrival made succeeds."""
import ctypes as C

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_17139_gb300 import build
    build.build()
    import paper_2502_17139_gb300.fastcoder as fcm
    return fcm


def test_bounded_wait_times_out_and_recovers(fc):
    assert fc.fc_get_error() == "FC_OK"
    fc.fc_selftest_wait(arrive=True)
    assert fc.fc_get_error() == "FC_OK"
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    ev0.record()
    fc.fc_selftest_wait(arrive=False, limit_cycles=2_000_000)  # ~1 ms at 2 GHz
    ev1.record()
    assert fc.fc_get_error() == "FC_ERR_TIMEOUT"
    assert ev0.elapsed_time(ev1) < 100.0  # gave up promptly
    assert fc.fc_get_error() == "FC_OK"   # read and cleared
    # the context is intact: ordinary work still runs and checks clean
    x = torch.arange(1 << 20, device="cuda", dtype=torch.float32)
    assert float(x.sum().item()) == float((1 << 20) * ((1 << 20) - 1) / 2)
    fc.fc_selftest_wait(arrive=True)
    assert fc.fc_get_error() == "FC_OK"


def test_selftest_rejects_bad_limits(fc):
    with pytest.raises(fc.FastCoderError):
        fc.fc_selftest_wait(arrive=False, limit_cycles=0)


def test_failed_launch_is_reported_once(fc):
    """A launch that the runtime refuses (its stream's capture was spoilt by a
    synchronisation) fails its own call and leaves nothing behind: the next
    call, whose kernel runs, succeeds."""
    path = next(line.split()[-1] for line in open("/proc/self/maps") if "libcudart" in line)
    rt = C.CDLL(path)  # the runtime that the library and torch share
    tok = torch.arange(4, dtype=torch.int32, device="cuda")
    table = torch.arange(4 * 64, dtype=torch.bfloat16, device="cuda").view(4, 64)
    out = torch.zeros_like(table)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        h = C.c_void_p(stream.cuda_stream)
        assert rt.cudaStreamBeginCapture(h, 2) == 0  # relaxed: other streams are not concerned
        assert rt.cudaStreamSynchronize(h) != 0
        rt.cudaGetLastError()
        with pytest.raises(fc.FastCoderError):
            fc.fc_embed(tok, table, out)
        left = rt.cudaPeekAtLastError()
        graph = C.c_void_p()
        rt.cudaStreamEndCapture(h, C.byref(graph))
        rt.cudaGetLastError()
        assert left == 0
        fc.fc_embed(tok, table, out)
    torch.cuda.synchronize()
    assert torch.equal(out, table) and fc.fc_get_error() == "FC_OK"
