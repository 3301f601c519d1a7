"""GPU-vs-oracle parity of the quantizer kernels, bit-exact on codes and scales."""
import numpy as np
import pytest
import torch

from paper_2505_19115_b200 import binding as nb
from paper_2505_19115_b200 import synth
from tests.util import assert_quantize_parity

pytestmark = pytest.mark.gpu

ROW_SHAPES = [(1, 16), (3, 48), (130, 80), (128, 512), (257, 1040), (256, 512), (129, 4112)]
# rows % 32 == 0 takes the tiled-copy kernel (ragged tiles in both directions), the others the fallback kernel
T_SHAPES = [(16, 8), (48, 24), (272, 72), (512, 200), (256, 64), (1040, 264), (4112, 136), (288, 72), (32, 8), (1056, 328)]


def _x(shape, seed, dtype=torch.bfloat16, std=1.0):
    return synth.normal(shape, std, seed, device="cpu", dtype=dtype).cuda()


@pytest.mark.parametrize("sf_layout", [nb.SF_LINEAR, nb.SF_SWIZZLED])
@pytest.mark.parametrize("mode", [nb.RTN, nb.SR])
@pytest.mark.parametrize("shape", ROW_SHAPES)
def test_row_bf16(shape, mode, sf_layout):
    assert_quantize_parity(_x(shape, 1), False, False, nb.Rounding(mode, 1234, 5), sf_layout)


@pytest.mark.parametrize("sf_layout", [nb.SF_LINEAR, nb.SF_SWIZZLED])
@pytest.mark.parametrize("mode", [nb.RTN, nb.SR])
@pytest.mark.parametrize("shape", T_SHAPES)
def test_transposed_bf16(shape, mode, sf_layout):
    assert_quantize_parity(_x(shape, 2), True, False, nb.Rounding(mode, 99, 1), sf_layout)


@pytest.mark.parametrize("transposed", [False, True])
@pytest.mark.parametrize("mode", [nb.RTN, nb.SR])
def test_fp32_input(mode, transposed):
    shape = (272, 136) if transposed else (131, 272)
    x = _x(shape, 3, dtype=torch.float32)
    assert_quantize_parity(x, transposed, False, nb.Rounding(mode, 7, 0), nb.SF_SWIZZLED)
    assert_quantize_parity(x, transposed, True, nb.Rounding(mode, 7, 0), nb.SF_LINEAR)


@pytest.mark.parametrize("transposed", [False, True])
@pytest.mark.parametrize("mode", [nb.RTN, nb.SR])
@pytest.mark.parametrize("std", [1e-4, 1e-3, 0.02, 50.0])
def test_global_scale_from_amax(std, mode, transposed):
    x = _x((256, 512), 4, std=std)
    assert_quantize_parity(x, transposed, True, nb.Rounding(mode, 0, 2), nb.SF_SWIZZLED)


def test_gradient_scale_underflow_without_global_scale():
    # N(0, 1e-4^2) with g = 1: every block scale underflows to 0 and only sign bits survive
    x = _x((128, 256), 5, std=1e-4)
    assert_quantize_parity(x, False, False, nb.Rounding(nb.RTN), nb.SF_LINEAR)
    codes, scales = nb.nvfp4_quantize(x)
    assert int(scales.max()) == 0 and int((codes & 0x77).max()) == 0


def test_special_values():
    x = torch.zeros((16, 64), dtype=torch.float32)
    x[0, :8] = torch.tensor([0.25, 0.75, 1.25, 1.75, 2.5, 3.5, 5.0, 6.0])       # tie points, scale 1
    x[1, :8] = -x[0, :8]
    x[2, 3] = -0.0
    x[3, 0] = 6.0 * 448.0 * 4                                                    # saturating scale
    x[3, 1:16] = 3000.0
    x[4, :16] = torch.linspace(-6, 6, 16)
    x[5, 16:32] = 1e-30
    x[6, 0] = 2.0 ** -9 * 6
    x[6, 1] = 2.0 ** -10 * 6
    x[7, 0] = 448.0 * 6
    x[7, 1] = 447.0
    for dt in (torch.bfloat16, torch.float32):
        xs = x.to(dt).cuda()
        for mode in (nb.RTN, nb.SR):
            assert_quantize_parity(xs, False, False, nb.Rounding(mode, 3, 3), nb.SF_LINEAR)
            assert_quantize_parity(xs, True, False, nb.Rounding(mode, 3, 3), nb.SF_LINEAR)


def test_sr_reproducible_and_offset_sensitive():
    x = _x((256, 512), 6)
    a, _ = nb.nvfp4_quantize(x, rounding=nb.Rounding(nb.SR, 1, 0))
    b, _ = nb.nvfp4_quantize(x, rounding=nb.Rounding(nb.SR, 1, 0))
    c, _ = nb.nvfp4_quantize(x, rounding=nb.Rounding(nb.SR, 1, 1))
    assert torch.equal(a, b) and not torch.equal(a, c)


def test_strided_input():
    base = _x((64, 1024), 7)
    view = base[:, 256:768]
    assert_quantize_parity(view, False, False, nb.Rounding(nb.SR, 5, 5), nb.SF_SWIZZLED)
    assert_quantize_parity(view, True, False, nb.Rounding(nb.SR, 5, 5), nb.SF_SWIZZLED)


@pytest.mark.parametrize("n_elem", [2 ** 20, 2 ** 24])
@pytest.mark.parametrize("transposed", [False, True])
@pytest.mark.parametrize("mode", [nb.RTN, nb.SR])
def test_heavy_tailed_sweep(n_elem, transposed, mode):
    x = synth.heavy_tailed(synth.square_shape(n_elem), seed=1001, device="cpu").cuda()
    assert_quantize_parity(x, transposed, True, nb.Rounding(mode, 1, 0), nb.SF_SWIZZLED)


# ---------------------------------------------------------------- both orientations from one read
DUAL_SHAPES = [(256, 64), (512, 192), (288, 96), (32, 32), (1056, 352), (48, 80), (272, 48)]   # the last two: fallback path


@pytest.mark.parametrize("sf_layout", [nb.SF_LINEAR, nb.SF_SWIZZLED])
@pytest.mark.parametrize("modes", [(nb.RTN, nb.SR), (nb.SR, nb.SR), (nb.RTN, nb.RTN), (nb.SR, nb.RTN)])
@pytest.mark.parametrize("shape", DUAL_SHAPES)
def test_dual_matches_the_oracle_in_both_orientations(shape, modes, sf_layout):
    from oracle import binding as ob
    from tests.util import oracle_quantize
    x = _x(shape, 11)
    g_t = nb.nvfp4_tensor_amax_scale(x)
    g = float(g_t.item())
    rr, rt = nb.Rounding(modes[0], 21, 4), nb.Rounding(modes[1], 21, 5)
    cr, sr, ct, st = nb.nvfp4_quantize_dual(x, g_t, rr, rt, sf_layout)
    torch.cuda.synchronize()
    assert nb.nvfp4_device_error_word() == 0
    for got_c, got_s, transposed, r in ((cr, sr, False, rr), (ct, st, True, rt)):
        oc, osf = oracle_quantize(x, transposed, g, r)
        if sf_layout == nb.SF_SWIZZLED:
            osf = ob.sf_swizzle(osf)
        assert np.array_equal(got_c.cpu().numpy(), oc)
        assert np.array_equal(got_s.cpu().numpy().reshape(-1), osf.reshape(-1))


def test_dual_heavy_tailed_2p24():
    from oracle import binding as ob
    from tests.util import oracle_quantize
    x = synth.heavy_tailed(synth.square_shape(2 ** 24), seed=1001, device="cpu").cuda()
    g_t = nb.nvfp4_tensor_amax_scale(x)
    rr, rt = nb.Rounding(nb.SR, 1, 0), nb.Rounding(nb.SR, 1, 1)
    cr, sr, ct, st = nb.nvfp4_quantize_dual(x, g_t, rr, rt, nb.SF_SWIZZLED)
    for got_c, got_s, transposed, r in ((cr, sr, False, rr), (ct, st, True, rt)):
        oc, osf = oracle_quantize(x, transposed, float(g_t.item()), r)
        assert np.array_equal(got_c.cpu().numpy(), oc)
        assert np.array_equal(got_s.cpu().numpy().reshape(-1), ob.sf_swizzle(osf).reshape(-1))


# one tile and less, ragged in both directions, and more tiles than two per resident block (the two slots of the ring
# are reused; 592 blocks for bf16, 296 for fp32): the last block of the walk gets fewer tiles than the first
@pytest.mark.parametrize("shape", [(32, 32), (128, 64), (160, 96), (2080, 1056), (1056, 8224), (8224, 1760)])
@pytest.mark.parametrize("modes", [(nb.RTN, nb.SR), (nb.SR, nb.SR)])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_dual_tiles_of_a_persistent_block(shape, modes, dtype):
    from oracle import binding as ob
    from tests.util import oracle_quantize
    x = _x(shape, 13, dtype=dtype)
    g_t = nb.nvfp4_tensor_amax_scale(x)
    rr, rt = nb.Rounding(modes[0], 3, 1), nb.Rounding(modes[1], 3, 2)
    cr, sr, ct, st = nb.nvfp4_quantize_dual(x, g_t, rr, rt, nb.SF_SWIZZLED)
    torch.cuda.synchronize()
    assert nb.nvfp4_device_error_word() == 0
    for got_c, got_s, transposed, r in ((cr, sr, False, rr), (ct, st, True, rt)):
        oc, osf = oracle_quantize(x, transposed, float(g_t.item()), r)
        assert np.array_equal(got_c.cpu().numpy(), oc)
        assert np.array_equal(got_s.cpu().numpy().reshape(-1), ob.sf_swizzle(osf).reshape(-1))


@pytest.mark.parametrize("sf_layout", [nb.SF_LINEAR, nb.SF_SWIZZLED])
@pytest.mark.parametrize("mode", [nb.RTN, nb.SR])
@pytest.mark.parametrize("shape", [(32, 8), (288, 72), (1056, 328)])
def test_transposed_fp32_tiles(shape, mode, sf_layout):
    assert_quantize_parity(_x(shape, 14, dtype=torch.float32), True, True, nb.Rounding(mode, 8, 1), sf_layout)


# the row output of the tile kernel: edges of a tile in both directions, and a tensor on either side of 48 Mi elements
# (bf16 rounded to nearest changes kernels there; the strided case reads rows that do not follow one another)
@pytest.mark.parametrize("sf_layout", [nb.SF_LINEAR, nb.SF_SWIZZLED])
@pytest.mark.parametrize("mode", [nb.RTN, nb.SR])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("shape", [(1, 32), (127, 96), (129, 64), (257, 1056), (3001, 608)])
def test_row_tiles(shape, dtype, mode, sf_layout):
    assert_quantize_parity(_x(shape, 15, dtype=dtype), False, True, nb.Rounding(mode, 4, 9), sf_layout)
    base = _x((shape[0], shape[1] + 40), 16, dtype=dtype)
    assert_quantize_parity(base[:, 16:16 + shape[1]], False, True, nb.Rounding(mode, 4, 9), sf_layout)


def test_row_kernels_agree_across_the_size_line():
    x = _x((12289, 4096), 17)                                    # 48 Mi + 4096 elements: the plain row kernel
    g = nb.nvfp4_tensor_amax_scale(x)
    codes, scales = nb.nvfp4_quantize(x, global_scale=g)
    part_c, part_s = nb.nvfp4_quantize(x[:12000], global_scale=g)  # the tile kernel
    assert torch.equal(codes[:12000], part_c) and torch.equal(scales[:12000], part_s)


# the per-tensor scale of small dense tensors: one block's share of a load and less (the other blocks of the cluster have
# nothing to read), a remainder, and both sides of the 2 MB line; the largest value in the first, a middle and the last place
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("shape", [(1, 16), (1, 48), (1, 8192), (3, 5456), (1024, 1024), (1025, 1024)])
def test_small_scales_on_repeated_calls(shape, dtype):
    x = _x(shape, 18, dtype=dtype)
    flat, outs = x.view(-1), torch.zeros(96, dtype=torch.float32, device="cuda")
    n = flat.numel()
    for i in range(96):                       # no wait in between: each call overlaps the one before it
        flat[(0, n // 2, n - 1)[i % 3]] = 64.0 + i
        nb.nvfp4_tensor_amax_scale(x, out=outs[i:i + 1])
    assert np.array_equal(outs.cpu().numpy(), (np.arange(96, dtype=np.float32) + 64) / np.float32(2688))


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_small_scales_of_a_call_together(dtype):
    # operands of 1 KB to 16 KB, a cluster each in one launch
    M, K, N = 8, 64, 64
    X, W = _x((M, K), 19, dtype=dtype), _x((N, K), 20, dtype=dtype, std=0.02)
    for i in range(32):
        X[i % M, (7 * i) % K] = 8.0 + i
        W[(5 * i) % N, i % K] = 1.0 + i
        want = nb.nvfp4_linear_fwd(X, W, nb.G_GIVEN, gx=nb.nvfp4_tensor_amax_scale(X), gw=nb.nvfp4_tensor_amax_scale(W))
        assert torch.equal(nb.nvfp4_linear_fwd(X, W), want)


# Padding of swizzled scale tiles is zero whatever the per-tensor scale: NaN (a diverged tensor), 0 and a subnormal one make
# the scale of a block of zeros encode as NaN.  Rows and columns that leave padding in both directions, through the tile
# kernel (multiples of 32), the plain kernels (multiples of 16 only) and the product's quantizing epilogue.
@pytest.mark.parametrize("g", [float("nan"), 0.0, 1e-40])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("shape", [(96, 96), (160, 352), (48, 80), (272, 1040)])
def test_padding_scales_are_zero_under_any_global_scale(shape, dtype, g):
    from oracle import binding as ob
    rows, cols = shape
    x, g_t = _x(shape, 21, dtype=dtype), torch.full((1,), g, device="cuda")

    def padding(Rq, Kq):
        return ob.sf_swizzle(np.ones((Rq, Kq // 16), np.uint8)) == 0
    for mode in (nb.RTN, nb.SR):
        r = nb.Rounding(mode, 1, 2)
        sr = nb.nvfp4_quantize(x, False, g_t, r, nb.SF_SWIZZLED)[1]
        st = nb.nvfp4_quantize(x, True, g_t, r, nb.SF_SWIZZLED)[1]
        _, dr, _, dt = nb.nvfp4_quantize_dual(x, g_t, r, r, nb.SF_SWIZZLED)
        for sf, (Rq, Kq) in ((sr, (rows, cols)), (dr, (rows, cols)), (st, (cols, rows)), (dt, (cols, rows))):
            assert not sf.cpu().numpy()[:nb.nvfp4_sf_bytes(Rq, Kq)][padding(Rq, Kq)].any()
    a = nb.nvfp4_quantize(_x((rows, 64), 22), sf_layout=nb.SF_SWIZZLED)
    b = nb.nvfp4_quantize(_x(((cols + 31) // 32 * 32, 64), 23), sf_layout=nb.SF_SWIZZLED)
    sf = nb.nvfp4_gemm_quantized(*a, None, *b, None, g_t, sf_layout=nb.SF_SWIZZLED)[1].cpu().numpy()
    N = b[0].shape[0]
    assert not sf[:nb.nvfp4_sf_bytes(rows, N)][padding(rows, N)].any()


# ---------------------------------------------------------------- the 256-row form of the tile kernel
# Large bf16 tensors take it: from 2^26 elements with both outputs, from 2^25 transposed and rounded to nearest.  Rows and
# columns that fill neither a tile nor a scale tile, both layouts.
@pytest.fixture(scope="module")
def tall_dual():
    from tests.util import to_host_f32
    x = _x((8224, 8224), 24)
    g_t = nb.nvfp4_tensor_amax_scale(x)
    return x, g_t, {tr: to_host_f32(x.T.contiguous() if tr else x) for tr in (False, True)}, {}


def _sf_wanted(osf, sf_layout):
    from oracle import binding as ob
    return (ob.sf_swizzle(osf) if sf_layout == nb.SF_SWIZZLED else osf).reshape(-1)


@pytest.mark.parametrize("sf_layout", [nb.SF_LINEAR, nb.SF_SWIZZLED])
@pytest.mark.parametrize("modes", [(nb.RTN, nb.SR), (nb.SR, nb.SR), (nb.RTN, nb.RTN), (nb.SR, nb.RTN)])
def test_dual_tall_tiles_ragged(tall_dual, modes, sf_layout):
    from oracle import binding as ob
    x, g_t, host, known = tall_dual
    for tr, mode in ((False, modes[0]), (True, modes[1])):
        if (tr, mode) not in known:
            known[tr, mode] = ob.quantize(host[tr], g=float(g_t.item()), mode=mode, seed=6, offset=int(tr))
    cr, sr, ct, st = nb.nvfp4_quantize_dual(x, g_t, nb.Rounding(modes[0], 6, 0), nb.Rounding(modes[1], 6, 1), sf_layout)
    torch.cuda.synchronize()
    assert nb.nvfp4_device_error_word() == 0
    for got_c, got_s, key in ((cr, sr, (False, modes[0])), (ct, st, (True, modes[1]))):
        oc, osf = known[key]
        assert np.array_equal(got_c.cpu().numpy(), oc)
        assert np.array_equal(got_s.cpu().numpy().reshape(-1), _sf_wanted(osf, sf_layout))


@pytest.mark.parametrize("sf_layout", [nb.SF_LINEAR, nb.SF_SWIZZLED])
def test_transposed_tall_tiles_ragged(sf_layout):
    assert_quantize_parity(_x((8224, 4104), 25), True, True, nb.Rounding(nb.RTN), sf_layout)


def test_padding_scales_of_tall_tiles_are_zero_under_a_nan_scale():
    from oracle import binding as ob
    x, nan = _x((8224, 8224), 26), torch.full((1,), float("nan"), device="cuda")
    _, sr, _, st = nb.nvfp4_quantize_dual(x, nan, nb.Rounding(nb.SR, 1, 1), nb.Rounding(nb.SR, 1, 2), nb.SF_SWIZZLED)
    sf = nb.nvfp4_quantize(x, True, nan, None, nb.SF_SWIZZLED)[1]
    padding = ob.sf_swizzle(np.ones((8224, 514), np.uint8)) == 0
    for s in (sr, st, sf):
        assert not s.cpu().numpy()[padding].any()
