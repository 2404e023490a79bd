"""-m gpu: launches that the runtime refuses are reported by the call that made them, and by no later one.  The refusal comes from
a stream whose capture has been broken by a synchronisation: nothing reaches the device."""
import pytest

from paper_2502_04416_b200 import binding, workloads as wl
from tests import parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,few,many", [("fp32", 64, 400), ("bf16", 1, 300), ("bf16", 16, 300), ("bf16", 300, 16)])
def test_refused_launch_is_reported_once(dtype, few, many):
    import torch
    from cuda.bindings import runtime as rt
    inp = wl.make_inputs(wl.Workload("refused", wl.LayerShape(256, 1024, 8, 2, 2, dtype), (many if many > few else few,), seed=2))
    layer = parity.gpu_layer(inp.layers[0], len(inp.x))
    x = parity.to_device(inp.x, dtype)
    want = layer.forward(x[:many].contiguous())
    xf, out, again = x[:few].contiguous(), torch.empty_like(x[:few]), torch.empty_like(want)
    xm = x[:many].contiguous()
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    s = side.cuda_stream
    assert rt.cudaStreamBeginCapture(s, rt.cudaStreamCaptureMode.cudaStreamCaptureModeRelaxed)[0] == rt.cudaError_t.cudaSuccess
    assert rt.cudaStreamSynchronize(s)[0] != rt.cudaError_t.cudaSuccess          # breaks the capture
    with pytest.raises(binding.CmoeError):
        layer.forward(xf, out, stream=side)
    rt.cudaStreamEndCapture(s)
    rt.cudaGetLastError()
    layer.forward(xm, again)
    torch.cuda.synchronize()
    assert torch.equal(again, want)
    layer.forward(xf, out, stream=side)
    torch.cuda.synchronize()
    assert torch.equal(out, layer.forward(xf))
    layer.destroy()
