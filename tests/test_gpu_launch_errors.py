"""A launch that the runtime refuses is reported by the call that made it, and by no later one."""
import ctypes

import pytest

import synth

torch = pytest.importorskip("torch")
import gpu_harness as G  # noqa: E402

pytestmark = pytest.mark.gpu


def _cudart():
    with open("/proc/self/maps") as f:
        paths = {line.split()[-1] for line in f if "libcudart.so" in line}
    return ctypes.CDLL(paths.pop())


def test_a_refused_launch_is_not_reported_again():
    N, H = 64 * 20, 2
    inp = synth.make_random_layer(N, H, 64 * H, seed=1)
    layer = G.Layer(inp, 0, [5] * H, 1).run_forward()
    r, b, rt = layer.ress, layer.buf, _cudart()
    stream = torch.cuda.Stream()
    handle = ctypes.c_void_p(stream.cuda_stream)
    assert rt.cudaStreamBeginCapture(handle, 2) == 0  # relaxed
    try:
        assert rt.cudaStreamSynchronize(handle) != 0  # not allowed: invalidates the capture
        with torch.cuda.stream(stream):
            with pytest.raises(Exception):  # the launch is refused
                r.score(layer.d, layer.Q, layer.K, layer.V, b.F, layer.c_h, b.ws)
    finally:
        graph = ctypes.c_void_p()
        rt.cudaStreamEndCapture(handle, ctypes.byref(graph))
        rt.cudaGetLastError()
    want = b.F.clone()
    b.F.zero_()
    r.prepare_wo(layer.d, layer.W, b.F)  # another stream, nothing wrong with it
    torch.cuda.synchronize()
    assert torch.equal(b.F, want)
    r.status(b.ws)
