"""Launches of the library overlap the kernel before them on the stream.  What a kernel reads that the one before it wrote,
and buffers that one step leaves to the next, must come out as they do with a wait for the device after every call."""
import pytest
import torch

from paper_2505_19115_b200 import binding as nb
from paper_2505_19115_b200 import synth

pytestmark = pytest.mark.gpu


def _x(shape, seed, std=1.0, dtype=torch.bfloat16):
    return synth.normal(shape, std, seed, device="cuda", dtype=dtype)


# Every tensor and scale of this chain is written by the call before the one that reads it.  Widths and heights that take the
# tile kernel (multiples of 32), the plain row and transposed kernels (multiples of 16 only) and both amax forms.
@pytest.mark.parametrize("out_dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("shape", [(512, 544, 256), (528, 528, 256), (2064, 1040, 128), (2048, 1056, 128)])
def test_operands_written_by_the_call_before(shape, out_dtype):
    M, N, K = shape
    a, b = nb.nvfp4_quantize(_x((M, K), 1), sf_layout=nb.SF_SWIZZLED), nb.nvfp4_quantize(_x((N, K), 2), sf_layout=nb.SF_SWIZZLED)
    gs = [torch.full((1,), 2.0 ** i, device="cuda") for i in range(-4, 4)]
    Y = torch.empty((M, N), dtype=out_dtype, device="cuda")
    ga, g = torch.empty(1, device="cuda"), torch.empty(1, device="cuda")
    sr = nb.Rounding(nb.SR, 3, 1)

    def chain(i, wait):
        ga.copy_(gs[i])
        nb.nvfp4_gemm(*a, ga, *b, None, out=Y)
        wait()
        nb.nvfp4_tensor_amax_scale(Y, out=g)
        wait()
        row = nb.nvfp4_quantize(Y, False, g, sr, nb.SF_SWIZZLED)
        wait()
        outs = [*row, *nb.nvfp4_quantize(Y, True, g, sr, nb.SF_SWIZZLED), *nb.nvfp4_quantize(Y, False, g, None, nb.SF_SWIZZLED)]
        wait()
        if N % 32 == 0:
            outs.append(nb.nvfp4_gemm(*row, g, *row, g))
        return outs + [Y.clone(), g.clone()]

    want = [chain(i, torch.cuda.synchronize) for i in range(8)]
    got = [chain(i, lambda: None) for i in range(8)]
    torch.cuda.synchronize()
    assert nb.nvfp4_device_error_word() == 0
    for w, o in zip(want, got):
        assert all(torch.equal(x, y) for x, y in zip(w, o))


def test_stream_handle_is_the_current_streams(monkeypatch):
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        assert nb._stream() == side.cuda_stream
        monkeypatch.setattr(nb, "_raw_stream", None)
        assert nb._stream() == side.cuda_stream
    assert nb._stream() == torch.cuda.current_stream().cuda_stream
