"""GPU-vs-oracle parity of the three quantized linear-layer products (Eq. 1-6)."""
import numpy as np
import pytest
import torch

from oracle import binding as ob
from paper_2505_19115_b200 import binding as nb
from paper_2505_19115_b200 import synth

pytestmark = pytest.mark.gpu

TOL = 1e-5


def _host(x):
    return x.float().cpu().numpy()


def _oracle_operand(x, transposed, r, use_g):
    h = _host(x)
    g = ob.tensor_amax_scale(h) if use_g else 1.0
    c, s = ob.quantize(h, g=g, mode=r.mode, seed=r.seed, offset=r.offset, transposed=transposed)
    return c, s, g


def oracle_linear(which, a, b, ra, rb, use_g, sample=None):
    ta, tb = {"fwd": (False, False), "dx": (False, True), "dw": (True, True)}[which]
    ac, asf, ga = _oracle_operand(a, ta, ra, use_g)
    bc, bsf, gb = _oracle_operand(b, tb, rb, use_g)
    if sample is None:
        return ob.gemm(ac, asf, ga, bc, bsf, gb)
    return ob.gemm_sampled(ac, asf, ga, bc, bsf, gb, sample[0], sample[1])


def _assert_close(got, ref, T):
    err = np.abs(got - ref)
    assert np.all(err <= TOL * T), f"max err/T = {np.max(err / np.maximum(T, 1e-30)):.3e}"


@pytest.mark.parametrize("use_g", [True, False])
def test_single_layer_all_three_products(use_g):
    # single small layer: X 256x512 N(0,1), W 512x512 N(0,0.02^2), dY 256x512 N(0,1e-3^2)
    t = synth.TINY_LINEAR
    X, W, dY = synth.linear_inputs(t["tokens"], t["K"], t["N"], seed=1001, grad_std=1e-3)
    X, W, dY = X.cuda(), W.cuda(), dY.cuda()
    mode = nb.G_AMAX if use_g else nb.G_NONE
    rt, sr0, sr1, sr2 = nb.Rounding(nb.RTN), nb.Rounding(nb.SR, 0, 0), nb.Rounding(nb.SR, 0, 1), nb.Rounding(nb.SR, 0, 2)
    Y = nb.nvfp4_linear_fwd(X, W, gscale_mode=mode, rx=rt, rw=rt)
    dX = nb.nvfp4_linear_bwd_dx(dY, W, gscale_mode=mode, rdy=sr0, rw=rt)
    dW = nb.nvfp4_linear_bwd_dw(dY, X, gscale_mode=mode, rdy=sr1, rx=sr2)
    torch.cuda.synchronize()
    assert nb.nvfp4_device_error_word() == 0
    _assert_close(_host(Y), *oracle_linear("fwd", X, W, rt, rt, use_g))
    _assert_close(_host(dX), *oracle_linear("dx", dY, W, sr0, rt, use_g))
    _assert_close(_host(dW), *oracle_linear("dw", dY, X, sr1, sr2, use_g))
    if not use_g:
        # without a per-tensor scale the 1e-3 gradients underflow the E4M3 scale range entirely
        assert float(dX.abs().max()) == 0.0 and float(dW.abs().max()) == 0.0
    else:
        assert float(dX.abs().max()) > 0.0 and float(dW.abs().max()) > 0.0


def test_all_sr_backward_variant():
    # the single-layer config also asks for SR on W in the backward product
    t = synth.TINY_LINEAR
    X, W, dY = synth.linear_inputs(t["tokens"], t["K"], t["N"], seed=1001, grad_std=1e-3)
    W, dY = W.cuda(), dY.cuda()
    sr0, sr3 = nb.Rounding(nb.SR, 0, 0), nb.Rounding(nb.SR, 0, 3)
    dX = nb.nvfp4_linear_bwd_dx(dY, W, rdy=sr0, rw=sr3)
    _assert_close(_host(dX), *oracle_linear("dx", dY, W, sr0, sr3, True))


def test_ragged_layer_and_bf16_output():
    X, W, dY = synth.linear_inputs(160, 288, 200, seed=7, grad_std=1e-3)
    X, W, dY = X.cuda(), W.cuda(), dY.cuda()
    rt, sr = nb.Rounding(nb.RTN), nb.Rounding(nb.SR, 9, 0)
    Y = nb.nvfp4_linear_fwd(X, W, rx=rt, rw=rt)
    _assert_close(_host(Y), *oracle_linear("fwd", X, W, rt, rt, True))
    dW = nb.nvfp4_linear_bwd_dw(dY, X, rdy=sr, rx=sr)
    _assert_close(_host(dW), *oracle_linear("dw", dY, X, sr, sr, True))
    Yb = nb.nvfp4_linear_fwd(X, W, rx=rt, rw=rt, out_dtype=torch.bfloat16)
    ref, T = oracle_linear("fwd", X, W, rt, rt, True)
    assert np.all(np.abs(_host(Yb) - ref) <= TOL * T + np.abs(ref) * 2.0 ** -8)


def test_given_global_scales_and_fp32_inputs():
    X, W, _ = synth.linear_inputs(128, 256, 128, seed=8)
    X, W = X.float().cuda(), W.float().cuda()
    gx, gw = nb.nvfp4_tensor_amax_scale(X), nb.nvfp4_tensor_amax_scale(W)
    rt = nb.Rounding(nb.RTN)
    Y = nb.nvfp4_linear_fwd(X, W, gscale_mode=nb.G_GIVEN, gx=gx, gw=gw, rx=rt, rw=rt)
    _assert_close(_host(Y), *oracle_linear("fwd", X, W, rt, rt, True))


@pytest.mark.parametrize("name,K,N", [(n, k, o) for (n, k, o) in synth.LLAMA_350M["linears"] if n in ("qkv", "down")])
def test_350m_block_linears_sampled(name, K, N):
    M = synth.LLAMA_350M["tokens"]
    X, W, dY = synth.linear_inputs(M, K, N, seed=1003)
    X, W, dY = X.cuda(), W.cuda(), dY.cuda()
    rt, sr0, sr1, sr2 = nb.Rounding(nb.RTN), nb.Rounding(nb.SR, 0, 0), nb.Rounding(nb.SR, 0, 1), nb.Rounding(nb.SR, 0, 2)
    rng = np.random.default_rng(3)
    n = 2048

    def sample(R, C):
        return (np.concatenate([rng.integers(0, R, n), [0, R - 1]]), np.concatenate([rng.integers(0, C, n), [C - 1, 0]]))

    Y = nb.nvfp4_linear_fwd(X, W, rx=rt, rw=rt)
    s = sample(M, N)
    _assert_close(_host(Y)[s[0], s[1]], *oracle_linear("fwd", X, W, rt, rt, True, s))
    dX = nb.nvfp4_linear_bwd_dx(dY, W, rdy=sr0, rw=rt)
    s = sample(M, K)
    _assert_close(_host(dX)[s[0], s[1]], *oracle_linear("dx", dY, W, sr0, rt, True, s))
    dW = nb.nvfp4_linear_bwd_dw(dY, X, rdy=sr1, rx=sr2)
    s = sample(N, K)
    _assert_close(_host(dW)[s[0], s[1]], *oracle_linear("dw", dY, X, sr1, sr2, True, s))
    assert nb.nvfp4_device_error_word() == 0


# ---------------------------------------------------------------- fused layer: every tensor read once per pass
@pytest.mark.parametrize("use_g", [True, False])
@pytest.mark.parametrize("shape", [(256, 512, 512), (160, 288, 224), (512, 64, 96)])
def test_fused_layer_equals_the_separate_products(shape, use_g):
    M, K, N = shape
    X, W, dY = synth.linear_inputs(M, K, N, seed=31, grad_std=1e-3)
    X, W, dY = X.cuda(), W.cuda(), dY.cuda()
    mode = nb.G_AMAX if use_g else nb.G_NONE
    rt, sr0, sr1, sr2 = nb.Rounding(nb.RTN), nb.Rounding(nb.SR, 5, 0), nb.Rounding(nb.SR, 5, 1), nb.Rounding(nb.SR, 5, 2)
    Y = nb.nvfp4_linear_fwd(X, W, gscale_mode=mode, rx=rt, rw=rt)
    dX = nb.nvfp4_linear_bwd_dx(dY, W, gscale_mode=mode, rdy=sr0, rw=rt)
    dW = nb.nvfp4_linear_bwd_dw(dY, X, gscale_mode=mode, rdy=sr1, rx=sr2)
    Yf, saved = nb.nvfp4_linear_fwd_save(X, W, gscale_mode=mode, rx=rt, rw=rt, rxt=sr2, rwt=rt)
    dXf, dWf = nb.nvfp4_linear_bwd_saved(dY, saved, K, gscale_mode=mode, rdy=sr0, rdyt=sr1)
    dXb, dWb = nb.nvfp4_linear_bwd(dY, W, X, gscale_mode=mode, rdy=sr0, rdyt=sr1, rwt=rt, rxt=sr2)
    torch.cuda.synchronize()
    assert nb.nvfp4_device_error_word() == 0
    assert torch.equal(Y, Yf) and torch.equal(dX, dXf) and torch.equal(dW, dWf)
    assert torch.equal(dX, dXb) and torch.equal(dW, dWb)
    _assert_close(_host(Yf), *oracle_linear("fwd", X, W, rt, rt, use_g))
    _assert_close(_host(dXf), *oracle_linear("dx", dY, W, sr0, rt, use_g))
    _assert_close(_host(dWf), *oracle_linear("dw", dY, X, sr1, sr2, use_g))


def test_fused_layer_with_given_scales_and_bf16_outputs():
    M, K, N = 256, 256, 384
    X, W, dY = synth.linear_inputs(M, K, N, seed=32, grad_std=1e-3)
    X, W, dY = X.cuda(), W.cuda(), dY.cuda()
    gx, gw, gdy = (nb.nvfp4_tensor_amax_scale(t) for t in (X, W, dY))
    Y, saved = nb.nvfp4_linear_fwd_save(X, W, gscale_mode=nb.G_GIVEN, gx=gx, gw=gw, out_dtype=torch.bfloat16)
    dX, dW = nb.nvfp4_linear_bwd_saved(dY, saved, K, gscale_mode=nb.G_GIVEN, gdy=gdy, dx_dtype=torch.bfloat16)
    rt = nb.Rounding(nb.RTN)
    ref, T = oracle_linear("fwd", X, W, rt, rt, True)
    assert np.all(np.abs(_host(Y) - ref) <= TOL * T + np.abs(ref) * 2.0 ** -8)
    ref, T = oracle_linear("dx", dY, W, nb.Rounding(nb.SR, 0, 0), rt, True)
    assert np.all(np.abs(_host(dX) - ref) <= TOL * T + np.abs(ref) * 2.0 ** -8)
    _assert_close(_host(dW), *oracle_linear("dw", dY, X, nb.Rounding(nb.SR, 0, 1), nb.Rounding(nb.SR, 0, 2), True))


# One launch deals the tiles of both gradients out to the pairs of CTAs: fewer tiles than pairs, a first product that fills its
# waves exactly (9472 x 8192), one that leaves pairs over (4096 x 3072 x 1024: 48 tiles), either product being the longer one.
@pytest.mark.parametrize("shape", [(32, 32, 32), (768, 512, 1280), (18944, 512, 256), (4096, 1024, 3072), (256, 8192, 9472), (2080, 1056, 2848), (512, 2048, 8192)])
@pytest.mark.parametrize("dx_dtype,dw_dtype", [(torch.float32, torch.float32), (torch.bfloat16, torch.float32), (torch.float32, torch.bfloat16)])
def test_gradients_of_one_launch_equal_the_single_products(shape, dx_dtype, dw_dtype):
    M, K, N = shape
    X, W, dY = (t.cuda() for t in synth.linear_inputs(M, K, N, seed=33, grad_std=1e-3))
    rt, sr0, sr1, sr2 = nb.Rounding(nb.RTN), nb.Rounding(nb.SR, 6, 0), nb.Rounding(nb.SR, 6, 1), nb.Rounding(nb.SR, 6, 2)
    want = (nb.nvfp4_linear_bwd_dx(dY, W, rdy=sr0, rw=rt, out_dtype=dx_dtype), nb.nvfp4_linear_bwd_dw(dY, X, rdy=sr1, rx=sr2, out_dtype=dw_dtype))
    got = nb.nvfp4_linear_bwd(dY, W, X, rdy=sr0, rdyt=sr1, rwt=rt, rxt=sr2, dx_dtype=dx_dtype, dw_dtype=dw_dtype)
    torch.cuda.synchronize()
    assert nb.nvfp4_device_error_word() == 0
    assert torch.equal(want[0], got[0]) and torch.equal(want[1], got[1])


# Where one of the gradients is bound by its stores, they are launched apart and the other one does not wait for it: three contractions,
# either gradient being the late one.  Calls follow one another on the same buffers.
@pytest.mark.parametrize("shape", [(8224, 4736, 96), (96, 4736, 8224), (8224, 4736, 544)])
@pytest.mark.parametrize("dw_dtype", [torch.float32, torch.bfloat16])
def test_gradients_launched_apart_equal_the_single_products(shape, dw_dtype):
    M, K, N = shape
    X, W, dY = (t.cuda() for t in synth.linear_inputs(M, K, N, seed=37, grad_std=1e-3))
    grads = [dY, dY.flip(0).contiguous(), (dY * 2).contiguous()]
    rt, sr0, sr1, sr2 = nb.Rounding(nb.RTN), nb.Rounding(nb.SR, 6, 0), nb.Rounding(nb.SR, 6, 1), nb.Rounding(nb.SR, 6, 2)
    want = [(nb.nvfp4_linear_bwd_dx(g, W, rdy=sr0, rw=rt), nb.nvfp4_linear_bwd_dw(g, X, rdy=sr1, rx=sr2, out_dtype=dw_dtype)) for g in grads]
    ws = torch.empty(nb.nvfp4_linear_fused_workspace_bytes(M, N, K, nb.FUSED_BWD), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    got = [nb.nvfp4_linear_bwd(grads[i % 3], W, X, rdy=sr0, rdyt=sr1, rwt=rt, rxt=sr2, dw_dtype=dw_dtype, workspace=ws) for i in range(6)]
    torch.cuda.synchronize()
    assert nb.nvfp4_device_error_word() == 0
    for i, (dX, dW) in enumerate(got):
        assert torch.equal(want[i % 3][0], dX) and torch.equal(want[i % 3][1], dW), i


# The layer calls quantize their operands together and take the per-tensor scale from an amax sweep's maxima: below 2 MB (one
# cluster), above (sweeps, one quantizer launch for both), one operand below and one above, and operands too large for one launch.
@pytest.mark.parametrize("mode", [nb.G_AMAX, nb.G_GIVEN, nb.G_NONE])
@pytest.mark.parametrize("shape,dtype", [((64, 32, 96), torch.bfloat16), ((2080, 1056, 2848), torch.bfloat16), ((2080, 1056, 2848), torch.float32),
                                         ((8224, 160, 224), torch.bfloat16), ((16416, 4128, 32), torch.bfloat16)])
def test_layer_calls_equal_the_single_calls(shape, dtype, mode):
    M, K, N = shape
    X, W, dY = (t.cuda().to(dtype) for t in synth.linear_inputs(M, K, N, seed=34, grad_std=1e-3))
    r = [nb.Rounding(nb.RTN), nb.Rounding(nb.SR, 7, 0), nb.Rounding(nb.SR, 7, 1), nb.Rounding(nb.SR, 7, 2)]
    g = [None if mode == nb.G_NONE else nb.nvfp4_tensor_amax_scale(t) for t in (X, W, dY)]

    def product(a, b, out_dtype=torch.float32):             # each operand: tensor, transposed, scale, rounding
        qa, qb = (nb.nvfp4_quantize(t, tr, s, rr, nb.SF_SWIZZLED) for t, tr, s, rr in (a, b))
        return nb.nvfp4_gemm(*qa, a[2], *qb, b[2], out_dtype=out_dtype)
    want = (product((X, False, g[0], r[0]), (W, False, g[1], r[0])), product((dY, False, g[2], r[1]), (W, True, g[1], r[0])),
            product((dY, True, g[2], r[2]), (X, True, g[0], r[3])))
    gx, gw, gdy = g if mode == nb.G_GIVEN else (None,) * 3
    Y, saved = nb.nvfp4_linear_fwd_save(X, W, mode, gx=gx, gw=gw, rx=r[0], rw=r[0], rxt=r[3], rwt=r[0])
    single = (nb.nvfp4_linear_fwd(X, W, mode, gx=gx, gw=gw, rx=r[0], rw=r[0]), nb.nvfp4_linear_bwd_dx(dY, W, mode, gdy=gdy, gw=gw, rdy=r[1], rw=r[0]),
              nb.nvfp4_linear_bwd_dw(dY, X, mode, gdy=gdy, gx=gx, rdy=r[2], rx=r[3]))
    fused = (Y, *nb.nvfp4_linear_bwd_saved(dY, saved, K, mode, gdy=gdy, rdy=r[1], rdyt=r[2]))
    both = nb.nvfp4_linear_bwd(dY, W, X, mode, gdy=gdy, gw=gw, gx=gx, rdy=r[1], rdyt=r[2], rwt=r[0], rxt=r[3])
    torch.cuda.synchronize()
    assert nb.nvfp4_device_error_word() == 0
    for i in range(3):
        assert torch.equal(want[i], single[i]) and torch.equal(want[i], fused[i]), i
    assert torch.equal(want[1], both[0]) and torch.equal(want[2], both[1])


# The layer calls' shared quantizer has a pass of its own over the scale padding, for per-tensor scales under which the zeros beyond
# a tensor do not encode to zero scales.  Rows and columns fill neither a tile nor a scale tile; what a call leaves in its buffers
# is compared byte for byte, padding included, with the single quantizers.
@pytest.mark.parametrize("g", [0.0, 1e-40, float("nan"), 1.0])
@pytest.mark.parametrize("shape,dtype", [((96, 160, 224), torch.bfloat16), ((96, 160, 224), torch.float32), ((2080, 1056, 2848), torch.bfloat16)])
def test_layer_operands_under_any_given_scale_equal_the_single_quantizers(shape, dtype, g):
    M, K, N = shape
    X, W, dY = (t.cuda().to(dtype) for t in synth.linear_inputs(M, K, N, seed=35, grad_std=1e-3))
    g_t = torch.full((1,), g, device="cuda")
    r = [nb.Rounding(nb.RTN), nb.Rounding(nb.SR, 8, 0), nb.Rounding(nb.SR, 8, 1), nb.Rounding(nb.SR, 8, 2)]

    def buffer(nbytes):
        return torch.full((nbytes,), 0xA5, dtype=torch.uint8, device="cuda")

    def assert_holds(buf, *operands):                       # in the buffer's order, each part from a multiple of 256 bytes
        at = 0
        for x, transposed, rounding in operands:
            Rq, Kq = x.shape[::-1] if transposed else x.shape
            codes, scales = nb.nvfp4_quantize(x, transposed, g_t, rounding, nb.SF_SWIZZLED)
            for want in (codes.reshape(-1), scales[:nb.nvfp4_sf_bytes(Rq, Kq)]):
                assert torch.equal(buf[at:at + want.numel()], want), (tuple(x.shape), transposed)
                at = (at + want.numel() + 255) // 256 * 256
    saved, ws = buffer(nb.nvfp4_linear_saved_bytes(M, N, K)), buffer(nb.nvfp4_linear_fused_workspace_bytes(M, N, K, nb.FUSED_FWD_SAVE))
    nb.nvfp4_linear_fwd_save(X, W, nb.G_GIVEN, gx=g_t, gw=g_t, rx=r[0], rw=r[0], rxt=r[3], rwt=r[0], saved=saved, workspace=ws)
    assert_holds(saved, (W, True, r[0]), (X, True, r[3]))
    assert_holds(ws, (X, False, r[0]), (W, False, r[0]))
    ws = buffer(nb.nvfp4_linear_fused_workspace_bytes(M, N, K, nb.FUSED_BWD))
    nb.nvfp4_linear_bwd(dY, W, X, nb.G_GIVEN, gdy=g_t, gw=g_t, gx=g_t, rdy=r[1], rdyt=r[2], rwt=r[0], rxt=r[3], workspace=ws)
    assert_holds(ws, (dY, False, r[1]), (dY, True, r[2]), (W, True, r[0]), (X, True, r[3]))
    ws = buffer(nb.nvfp4_linear_workspace_bytes(M, N, K, nb.LINEAR_BWD_DW))
    nb.nvfp4_linear_bwd_dw(dY, X, nb.G_GIVEN, gdy=g_t, gx=g_t, rdy=r[2], rx=r[3], workspace=ws)
    assert_holds(ws, (dY, True, r[2]), (X, True, r[3]))
    assert nb.nvfp4_device_error_word() == 0


# Operands aligned to 16 bytes, but not to the 32 that the amax sweeps load at once: they take the passes for any tensor.
@pytest.mark.parametrize("moved", [(True, True, True), (True, False, False), (False, True, False)])
@pytest.mark.parametrize("shape,dtype", [((64, 32, 96), torch.bfloat16), ((2080, 1056, 2848), torch.bfloat16), ((2080, 1056, 2848), torch.float32),
                                         ((16416, 4128, 32), torch.bfloat16)])
def test_layer_calls_on_operands_aligned_to_16_bytes(shape, dtype, moved):
    M, K, N = shape
    X, W, dY = (t.cuda().to(dtype) for t in synth.linear_inputs(M, K, N, seed=36, grad_std=1e-3))

    def at_16(x):
        buf = torch.zeros(x.numel() + 16, dtype=x.dtype, device="cuda")
        view = buf[16 // x.element_size():][:x.numel()].view(x.shape)
        assert view.data_ptr() % 32 == 16
        return view.copy_(x)

    def results(X, W, dY):
        Y, saved = nb.nvfp4_linear_fwd_save(X, W)
        return (Y, *nb.nvfp4_linear_bwd_saved(dY, saved, K), *nb.nvfp4_linear_bwd(dY, W, X), nb.nvfp4_linear_fwd(X, W))
    want = results(X, W, dY)
    got = results(*(at_16(x) if m else x for x, m in zip((X, W, dY), moved)))
    torch.cuda.synchronize()
    assert nb.nvfp4_device_error_word() == 0
    for i, (a, b) in enumerate(zip(want, got)):
        assert torch.equal(a, b), i


# ---------------------------------------------------------------- non-finite inputs stay visible
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), float("-inf")])
def test_non_finite_input_propagates_through_the_per_tensor_scale(bad):
    # A NaN (or an infinity) anywhere in an operand makes its amax scale NaN (+Inf), as the oracle's does, and
    # every element of a product computed with that scale NaN; products of the other operands stay finite.
    M, K, N = 256, 512, 384
    X, W, dY = synth.linear_inputs(M, K, N, seed=77, grad_std=1e-3)
    X[131, 257] = bad
    Xd, Wd, dYd = X.cuda(), W.cuda(), dY.cuda()
    g = nb.nvfp4_tensor_amax_scale(Xd)
    want = ob.tensor_amax_scale(_host(Xd))
    got = float(g.item())
    assert (np.isnan(want) and np.isnan(got)) or (np.isinf(want) and got == want)
    for Xin in (Xd, Xd.float()):                        # bf16 and fp32 sources take different amax paths
        g32 = float(nb.nvfp4_tensor_amax_scale(Xin).item())
        assert (np.isnan(want) and np.isnan(g32)) or g32 == want
    Y = nb.nvfp4_linear_fwd(Xd, Wd)
    dW = nb.nvfp4_linear_bwd_dw(dYd, Xd)
    dX = nb.nvfp4_linear_bwd_dx(dYd, Wd)
    Yf, saved = nb.nvfp4_linear_fwd_save(Xd, Wd)
    dXf, dWf = nb.nvfp4_linear_bwd_saved(dYd, saved, K)
    torch.cuda.synchronize()
    assert nb.nvfp4_device_error_word() == 0
    for t in (Y, dW, Yf, dWf):
        assert bool(torch.isnan(t).all())
    for t in (dX, dXf):                                 # dX = Q(dY) Q(W^T)^T does not involve X
        assert bool(torch.isfinite(t).all())
    # the oracle's dequantize-then-matmul says the same
    ref, _ = oracle_linear("fwd", Xd, Wd, nb.Rounding(nb.RTN), nb.Rounding(nb.RTN), True)
    assert np.all(np.isnan(ref))


# ---------------------------------------------------------------- a chain of layers without a high-precision intermediate
@pytest.mark.parametrize("mode", [nb.RTN, nb.SR])
@pytest.mark.parametrize("shape", [(256, 512, 768, 256), (300, 288, 544, 200)])
def test_chained_layers_quantize_in_the_producer(shape, mode):
    # layer 1 writes Q(H) from its GEMM epilogue (nvfp4_linear_fwd_qout), layer 2 consumes it (nvfp4_linear_fwd_qin).
    # H itself (layer 1 through nvfp4_linear_fwd) is checked against the oracle's product; the quantized H must then
    # be the ORACLE's quantization of that H byte for byte, and the second product the oracle's product of those codes.
    M, K1, N1, N2 = shape
    X, W1, _ = synth.linear_inputs(M, K1, N1, seed=41)
    _, W2, _ = synth.linear_inputs(M, N1, N2, seed=42)
    X, W1, W2 = X.cuda(), W1.cuda(), W2.cuda()
    rt, ry = nb.Rounding(nb.RTN), nb.Rounding(mode, 77, 4)
    H = nb.nvfp4_linear_fwd(X, W1, rx=rt, rw=rt)
    ref, T = oracle_linear("fwd", X, W1, rt, rt, True)
    Hh = _host(H)
    _assert_close(Hh, ref, T)
    gh_t = nb.nvfp4_tensor_amax_scale(H)                  # the consumer's scale has to be known beforehand
    gh = ob.tensor_amax_scale(Hh)
    assert np.float32(gh) == np.float32(gh_t.item())
    hc, hs = nb.nvfp4_linear_fwd_qout(X, W1, gy=gh_t, ry=ry, rx=rt, rw=rt, sf_layout=nb.SF_SWIZZLED)
    Y = nb.nvfp4_linear_fwd_qin(hc, hs, gh_t, W2, rw=rt)
    torch.cuda.synchronize()
    assert nb.nvfp4_device_error_word() == 0
    oc, osf = ob.quantize(Hh, g=gh, mode=ry.mode, seed=ry.seed, offset=ry.offset)
    assert np.array_equal(hc.cpu().numpy(), oc)
    assert np.array_equal(hs.cpu().numpy().reshape(-1), ob.sf_swizzle(osf).reshape(-1))
    w2h = _host(W2)
    g2 = ob.tensor_amax_scale(w2h)
    wc, wsf = ob.quantize(w2h, g=g2)
    ref2, T2 = ob.gemm(oc, osf, gh, wc, wsf, g2)
    _assert_close(_host(Y), ref2, T2)
    # and the unfused pair (fp32 H, quantized by the next layer's own quantizer) gives the same bits when the
    # roundings agree (the next layer would use RtN on its input, Eq. 4)
    if mode == nb.RTN:
        Y_unfused = nb.nvfp4_linear_fwd(H, W2.float(), gscale_mode=nb.G_AMAX, rx=rt, rw=rt)   # bf16 -> fp32 is exact
        assert torch.equal(Y, Y_unfused)


# scales of a call's operands: one cluster each in one launch, one sweep shared in proportion to the sizes (a tiny operand
# beside a large one, two like ones), and one launch each above the line
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("shape", [(256, 512, 512), (32, 4096, 2080), (2080, 2848, 1056), (6144, 2048, 2048), (8192, 2048, 4096)])
def test_scales_computed_together_equal_scales_computed_alone(shape, dtype):
    M, N, K = shape
    X, W = synth.normal((M, K), 1.0, 5, device="cuda", dtype=dtype), synth.normal((N, K), 0.02, 6, device="cuda", dtype=dtype)
    dY = synth.normal((M, N), 1e-3, 7, device="cuda", dtype=dtype)
    gx, gw, gdy = (nb.nvfp4_tensor_amax_scale(t) for t in (X, W, dY))
    assert float(gx) == float(np.float32(float(X.abs().max())) / np.float32(2688))
    want = nb.nvfp4_linear_fwd(X, W, nb.G_GIVEN, gx=gx, gw=gw)
    assert torch.equal(nb.nvfp4_linear_fwd(X, W), want)
    Y, saved = nb.nvfp4_linear_fwd_save(X, W)
    assert torch.equal(Y, want)
    dX, dW = nb.nvfp4_linear_bwd_saved(dY, saved, K)
    dX2, dW2 = nb.nvfp4_linear_bwd(dY, W, X)
    dX3, dW3 = nb.nvfp4_linear_bwd(dY, W, X, nb.G_GIVEN, gdy=gdy, gw=gw, gx=gx)
    assert torch.equal(dX, dX3) and torch.equal(dW, dW3) and torch.equal(dX2, dX3) and torch.equal(dW2, dW3)
    assert nb.nvfp4_device_error_word() == 0
