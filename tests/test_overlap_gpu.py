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


# Two layers that share a workspace, four steps on the same input, saved-operand and output buffers with inputs that change
# in between, against the same calls on fresh buffers with a wait after each.  256 x 512: the cluster amax; 2080 x 1056: one
# shared sweep, ragged tiles; 4096 x 1024 x 3072: the weight gradient starts in the input gradient's last wave.
def _step_buffers(M, K, N, dtype, mode):
    layers = []
    for (k, n) in ((K, N), (N, K)):
        layers.append(dict(X=torch.empty((M, k), dtype=dtype, device="cuda"), W=torch.empty((n, k), dtype=dtype, device="cuda"),
                           dY=torch.empty((M, n), dtype=dtype, device="cuda"), K=k,
                           g=[torch.empty(1, device="cuda") if mode == nb.G_GIVEN else None for _ in range(3)],
                           saved=torch.empty(nb.nvfp4_linear_saved_bytes(M, n, k), dtype=torch.uint8, device="cuda"),
                           Y=torch.empty((M, n), device="cuda"), dX=torch.empty((M, k), device="cuda"), dW=torch.empty((n, k), device="cuda")))
    ws = torch.empty(max(nb.nvfp4_linear_fused_workspace_bytes(M, *nk, w) for nk in ((N, K), (K, N))
                         for w in (nb.FUSED_FWD_SAVE, nb.FUSED_BWD_SAVED)), dtype=torch.uint8, device="cuda")
    return layers, ws


def _fill(layers, step):
    for i, l in enumerate(layers):
        for j, (name, std) in enumerate((("X", 1.0), ("W", 0.02), ("dY", 1e-3))):
            t = l[name]
            t.amax()                                            # the old contents lie in caches when the new ones are written
            t.copy_(_x(t.shape, 100 * step + 10 * i + j, std * 2.0 ** ((step + j) % 3), t.dtype))
            if l["g"][j] is not None:
                l["g"][j].copy_(t.float().abs().amax() / 2688)


def _step(layers, ws, mode, stream=None, fresh=False):
    def wait():
        if fresh:
            torch.cuda.synchronize()
    sr = [nb.Rounding(nb.SR, 11, o) for o in range(3)]
    keep = {}
    for i, l in enumerate(layers):
        gx, gw, _ = l["g"]
        kw = {} if fresh else dict(out=l["Y"], saved=l["saved"], workspace=ws)
        keep[i] = nb.nvfp4_linear_fwd_save(l["X"], l["W"], mode, gx=gx, gw=gw, rxt=sr[2], stream=stream, **kw)
        wait()
    for i, l in reversed(list(enumerate(layers))):
        kw = {} if fresh else dict(dX=l["dX"], dW=l["dW"], workspace=ws)
        Y, saved = keep[i]
        keep[i] = (Y, *nb.nvfp4_linear_bwd_saved(l["dY"], saved, l["K"], mode, gdy=l["g"][2], rdy=sr[0], rdyt=sr[1], stream=stream, **kw))
        wait()
    return [t for i in sorted(keep) for t in keep[i]]


@pytest.mark.parametrize("how", ["current stream", "given stream", "graph"])
@pytest.mark.parametrize("mode", [nb.G_AMAX, nb.G_GIVEN])
@pytest.mark.parametrize("shape,dtype", [((256, 512, 512), torch.bfloat16), ((2080, 1056, 2848), torch.bfloat16),
                                         ((4096, 1024, 3072), torch.bfloat16), ((1056, 544, 1056), torch.float32)])
def test_steps_on_the_same_buffers(shape, dtype, mode, how):
    layers, ws = _step_buffers(*shape, dtype, mode)
    want = []
    for i in range(4):
        _fill(layers, i)
        torch.cuda.synchronize()
        want.append([t.clone() for t in _step(layers, ws, mode, fresh=True)])
    side = torch.cuda.Stream()
    graph = None
    if how == "graph":
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            _step(layers, ws, mode)
    outs = [t for l in layers for t in (l["Y"], l["dX"], l["dW"])]
    got = []
    torch.cuda.synchronize()
    for i in range(4):
        if how == "given stream":
            with torch.cuda.stream(side):
                _fill(layers, i)
            _step(layers, ws, mode, stream=side)
            with torch.cuda.stream(side):
                got.append([t.clone() for t in outs])
        else:
            _fill(layers, i)
            if graph is None:
                _step(layers, ws, mode)
            else:
                graph.replay()
            got.append([t.clone() for t in outs])
    torch.cuda.synchronize()
    assert nb.nvfp4_device_error_word() == 0
    for i in range(4):
        for w, g in zip(want[i], got[i]):
            assert torch.equal(w, g), f"step {i}"
