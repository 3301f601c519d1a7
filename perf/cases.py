"""Performance cases of the library: the work a training or evaluation program has it do, through the public binding.

A case is a dict of plain values; its "op" names the sequence of calls.  Every op reads torch tensors in device
memory and keeps what a program would keep between steps: workspaces, saved-operand buffers, output buffers, rounding
descriptors, quantized weights where they are fixed, per-tensor scales where they are carried over.

  step      one training step of one linear layer: nvfp4_linear_fwd_save + nvfp4_linear_bwd_saved
  wgrad     the weight gradient alone (update pass): nvfp4_linear_bwd_dw
  chain     two layers, the intermediate quantized in the producer: nvfp4_linear_fwd_qout -> nvfp4_linear_fwd_qin
  kept      evaluation with weights quantized once: per-tensor scale and quantization of the activations, nvfp4_gemm
  quantize  the quantizers alone: per-tensor scale, then row and transposed layouts with both roundings
  qaf       the fine-tuning phase: forward in NVFP4, backward and update in bf16
  mx        the MXFP4 format: both operands quantized and multiplied (forward, or the transposed update product)
"""
import math

import torch

from paper_2505_19115_b200 import binding as nb
from paper_2505_19115_b200 import synth

_TORCH = {"bf16": torch.bfloat16, "fp32": torch.float32}
_BYTES = {"bf16": 2, "fp32": 4}


def listed():
    return [
        # the single small layer: launches and host time are what it costs
        dict(name="step_small_256", op="step", M=256, K=512, N=512, x="bf16", y="fp32", scales="amax", grad=1e-3),
        # 350M-class block, fused QKV projection: short contractions forward and backward, few weight-gradient tiles
        dict(name="step_350m_qkv", op="step", M=16384, K=1024, N=3072, x="bf16", y="fp32", scales="amax", grad=1e-4),
        # 7B-class block, SwiGLU gate (the up projection has the same shape): the bulk of a training step
        dict(name="step_7b_gate", op="step", M=16384, K=4096, N=11008, x="bf16", y="fp32", scales="amax", grad=1e-4),
        # 7B-class block, down projection with bf16 activations and the per-tensor scales of the previous step
        dict(name="step_7b_down_bf16", op="step", M=16384, K=11008, N=4096, x="bf16", y="bf16", scales="given", grad=1e-4),
        # a short, odd micro-batch: no size a multiple of a tile
        dict(name="step_odd_2080", op="step", M=2080, K=1056, N=2848, x="bf16", y="bf16", scales="amax", grad=1e-4),
        # fp32 activations, weights and gradients (350M-class down projection)
        dict(name="step_350m_down_fp32", op="step", M=16384, K=2816, N=1024, x="fp32", y="fp32", scales="amax", grad=1e-4),
        # up projection feeding the down projection, token count of a partly filled batch
        dict(name="chain_7b_3001", op="chain", M=3001, K=4096, N=11008, N2=4096, y="bf16"),
        # evaluation on a handful of tokens with weights quantized once
        dict(name="kept_7b_16_tokens", op="kept", M=16, K=4096, N=11008, y="bf16"),
        # long token axis: the largest weight gradient
        dict(name="wgrad_7b_65536", op="wgrad", M=65536, K=4096, N=11008, x="bf16"),
        # heavy-tailed tensor through every quantizer variant
        dict(name="quantize_2p26", op="quantize", rows=8192, cols=8192, x="bf16", swizzled=True),
        # fine-tuning phase, attention output projection
        dict(name="qaf_7b_o", op="qaf", M=16384, K=4096, N=4096, y="fp32"),
        # MXFP4 forward of the 350M-class gate projection
        dict(name="mx_350m_gate", op="mx", M=16384, K=1024, N=2816, which="fwd", y="bf16"),
    ]


def _log(rng, lo, hi, step):
    """A multiple of `step` in [lo, hi], spread evenly over the logarithm."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, min(hi, int(round(v / step)) * step))


def draw(rng):
    op = rng.choice(["step", "step", "step", "wgrad", "chain", "kept", "quantize", "qaf", "mx"])
    if op == "step":
        x = rng.choice(["bf16", "bf16", "bf16", "fp32"])
        return dict(op=op, M=_log(rng, 256, 16384, 32), K=_log(rng, 512, 11008, 32), N=_log(rng, 512, 11008, 32), x=x,
                    y=rng.choice(["bf16", "fp32"]), scales=rng.choice(["amax", "amax", "given"]), grad=rng.choice([1e-3, 1e-4]))
    if op == "wgrad":
        return dict(op=op, M=_log(rng, 4096, 65536, 32), K=_log(rng, 512, 4096, 8), N=_log(rng, 512, 11008, 8),
                    x=rng.choice(["bf16", "bf16", "fp32"]) if rng.random() < 0.5 else "bf16")
    if op == "chain":
        return dict(op=op, M=_log(rng, 256, 16384, 1), K=_log(rng, 512, 4096, 32), N=_log(rng, 1024, 11008, 32),
                    N2=_log(rng, 512, 4096, 8), y=rng.choice(["bf16", "fp32"]))
    if op == "kept":
        return dict(op=op, M=_log(rng, 1, 512, 1), K=_log(rng, 512, 11008, 32), N=_log(rng, 512, 12288, 8),
                    y=rng.choice(["bf16", "fp32"]))
    if op == "quantize":
        return dict(op=op, rows=_log(rng, 1024, 16384, 16), cols=_log(rng, 1024, 16384, 16),
                    x=rng.choice(["bf16", "bf16", "fp32"]), swizzled=rng.choice([True, True, False]))
    if op == "qaf":
        return dict(op=op, M=_log(rng, 256, 16384, 32), K=_log(rng, 512, 4096, 32), N=_log(rng, 512, 11008, 32),
                    y=rng.choice(["bf16", "fp32"]))
    return dict(op=op, M=_log(rng, 256, 16384, 32), K=_log(rng, 512, 4096, 32), N=_log(rng, 512, 11008, 32),
                which=rng.choice(["fwd", "dw"]), y=rng.choice(["bf16", "fp32"]))


def _normal(shape, std, seed, dtype="bf16"):
    return synth.normal(shape, std, seed, device="cuda", dtype=_TORCH[dtype])


def _empty(shape, dtype):
    return torch.empty(shape, dtype=_TORCH[dtype], device="cuda")


def _u8(n):
    return torch.empty(max(int(n), 256), dtype=torch.uint8, device="cuda")


def prepare(case, seed):
    op, s = case["op"], dict(case)
    sd = int(seed) * 8
    rtn = s["rtn"] = nb.Rounding(nb.RTN)
    s["sr"] = [nb.Rounding(nb.SR, int(seed), o) for o in range(3)]     # a stream of its own for every rounding site
    if op == "quantize":
        R, C = case["rows"], case["cols"]
        layout = s["layout"] = nb.SF_SWIZZLED if case["swizzled"] else nb.SF_LINEAR
        s["x"] = synth.heavy_tailed((R, C), sd, device="cuda", dtype=_TORCH[case["x"]])
        s["g"] = _empty(1, "fp32")
        s["bufs"] = [(transposed, rounding, _u8(R * C // 2), _u8(nb.nvfp4_sf_bytes(*((C, R) if transposed else (R, C)), layout)))
                     for transposed in (False, True) for rounding in (rtn, s["sr"][0])]
        return s
    M, K, N = case["M"], case["K"], case["N"]
    if op in ("step", "wgrad", "qaf"):
        x = case.get("x", "bf16")
        s["X"] = _normal((M, K), 1.0, sd, x)
        s["dY"] = _normal((M, N), case.get("grad", 1e-4), sd + 2, x)
    if op in ("step", "qaf"):
        s["W"] = _normal((N, K), 0.02, sd + 1, case.get("x", "bf16"))
    if op == "step":
        s["saved"] = _u8(nb.nvfp4_linear_saved_bytes(M, N, K))
        s["ws"] = _u8(max(nb.nvfp4_linear_fused_workspace_bytes(M, N, K, w) for w in (nb.FUSED_FWD_SAVE, nb.FUSED_BWD_SAVED)))
        s["Y"], s["dX"], s["dW"] = _empty((M, N), case["y"]), _empty((M, K), case["y"]), _empty((N, K), "fp32")
        s["mode"] = nb.G_AMAX
        s["gx"] = s["gw"] = s["gdy"] = None
        if case["scales"] == "given":
            s["mode"] = nb.G_GIVEN
            s["gx"], s["gw"], s["gdy"] = (nb.nvfp4_tensor_amax_scale(s[k]) for k in ("X", "W", "dY"))
    elif op == "wgrad":
        s["ws"] = _u8(nb.nvfp4_linear_workspace_bytes(M, N, K, nb.LINEAR_BWD_DW))
        s["dW"] = _empty((N, K), "fp32")
    elif op == "qaf":
        s["ws"] = _u8(nb.nvfp4_linear_workspace_bytes(M, N, K, nb.LINEAR_FWD))
        s["Y"] = _empty((M, N), case["y"])
    elif op == "chain":
        N2 = case["N2"]
        s["X"] = _normal((M, K), 1.0, sd)
        s["W1"], s["W2"] = _normal((N, K), 0.02, sd + 1), _normal((N2, N), 0.02, sd + 2)
        s["ws"] = _u8(max(nb.nvfp4_linear_workspace_bytes(M, N, K, nb.LINEAR_FWD),
                          nb.nvfp4_linear_workspace_bytes(M, N2, N, nb.LINEAR_FWD)))
        s["gx"], s["g1"], s["g2"] = (nb.nvfp4_tensor_amax_scale(s[k]) for k in ("X", "W1", "W2"))
        # the intermediate's scale, as carried over from a previous step
        s["gh"] = nb.nvfp4_tensor_amax_scale(nb.nvfp4_linear_fwd(s["X"], s["W1"], nb.G_GIVEN, gx=s["gx"], gw=s["g1"],
                                                                 out_dtype=torch.bfloat16, workspace=s["ws"]))
        s["codes"], s["sf"] = torch.empty((M, N // 2), dtype=torch.uint8, device="cuda"), _u8(nb.nvfp4_sf_bytes(M, N))
        s["Y"] = _empty((M, N2), case["y"])
    elif op == "kept":
        W = _normal((N, K), 0.02, sd + 1)
        s["gw"] = nb.nvfp4_tensor_amax_scale(W)
        s["w"] = nb.nvfp4_quantize(W, global_scale=s["gw"], sf_layout=nb.SF_SWIZZLED)
        s["X"] = _normal((M, K), 1.0, sd)
        s["gx"] = _empty(1, "fp32")
        s["x"] = torch.empty((M, K // 2), dtype=torch.uint8, device="cuda"), _u8(nb.nvfp4_sf_bytes(M, K))
        s["Y"] = _empty((M, N), case["y"])
    elif op == "mx":
        if case["which"] == "fwd":
            s["A"], s["B"], s["transposed"], s["r"] = _normal((M, K), 1.0, sd), _normal((N, K), 0.02, sd + 1), False, (rtn, rtn)
        else:
            s["A"], s["B"], s["transposed"], s["r"] = _normal((M, N), 1e-4, sd), _normal((M, K), 1.0, sd + 1), True, s["sr"][1:]
        s["D"] = _empty((M, N) if case["which"] == "fwd" else (N, K), case["y"])
    return s


def run(s):
    op = s["op"]
    if op == "step":
        rtn, sr = s["rtn"], s["sr"]
        nb.nvfp4_linear_fwd_save(s["X"], s["W"], s["mode"], gx=s["gx"], gw=s["gw"], rx=rtn, rw=rtn, rxt=sr[2], rwt=rtn,
                                 out=s["Y"], saved=s["saved"], workspace=s["ws"])
        nb.nvfp4_linear_bwd_saved(s["dY"], s["saved"], s["K"], s["mode"], gdy=s["gdy"], rdy=sr[0], rdyt=sr[1], dX=s["dX"],
                                  dW=s["dW"], workspace=s["ws"])
        return s["Y"], s["dX"], s["dW"]
    if op == "wgrad":
        return nb.nvfp4_linear_bwd_dw(s["dY"], s["X"], nb.G_AMAX, rdy=s["sr"][1], rx=s["sr"][2], out=s["dW"], workspace=s["ws"])
    if op == "chain":
        nb.nvfp4_linear_fwd_qout(s["X"], s["W1"], gy=s["gh"], ry=s["rtn"], gscale_mode=nb.G_GIVEN, gx=s["gx"], gw=s["g1"],
                                 rx=s["rtn"], rw=s["rtn"], codes=s["codes"], scales=s["sf"], workspace=s["ws"])
        return nb.nvfp4_linear_fwd_qin(s["codes"], s["sf"], s["gh"], s["W2"], nb.G_GIVEN, gw=s["g2"], rw=s["rtn"], out=s["Y"],
                                       workspace=s["ws"])
    if op == "kept":
        codes, sf = s["x"]
        nb.nvfp4_tensor_amax_scale(s["X"], out=s["gx"])
        nb.nvfp4_quantize(s["X"], False, s["gx"], s["rtn"], nb.SF_SWIZZLED, codes=codes, scales=sf)
        return nb.nvfp4_gemm(codes, sf, s["gx"], s["w"][0], s["w"][1], s["gw"], out=s["Y"])
    if op == "quantize":
        nb.nvfp4_tensor_amax_scale(s["x"], out=s["g"])
        for transposed, rounding, codes, sf in s["bufs"]:
            nb.nvfp4_quantize(s["x"], transposed, s["g"], rounding, s["layout"], codes=codes, scales=sf)
        # the bytes a call writes: a buffer of this program is at least 256 bytes long
        R, C = s["rows"], s["cols"]
        return [(codes[:R * C // 2], sf[:nb.nvfp4_sf_bytes(*((C, R) if tr else (R, C)), s["layout"])]) for tr, _, codes, sf in s["bufs"]]
    if op == "qaf":
        Y = nb.nvfp4_linear_fwd(s["X"], s["W"], nb.G_AMAX, rx=s["rtn"], rw=s["rtn"], out=s["Y"], workspace=s["ws"])
        dX, dW = nb.nvfp4_linear_bwd_bf16(s["dY"], s["W"], s["X"], dx_dtype=s["Y"].dtype)
        return Y, dX, dW
    ga, gb = nb.nvfp4_tensor_amax_scale(s["A"]), nb.nvfp4_tensor_amax_scale(s["B"])
    ac, asf = nb.nvfp4_quantize_mx(s["A"], s["transposed"], ga, s["r"][0], nb.SF_SWIZZLED)
    bc, bsf = nb.nvfp4_quantize_mx(s["B"], s["transposed"], gb, s["r"][1], nb.SF_SWIZZLED)
    return nb.nvfp4_gemm_mx(ac, asf, ga, bc, bsf, gb, out=s["D"])


def work(case):
    """Bytes of every input read once and every output written once, and the multiply-adds of the products."""
    op = case["op"]
    if op == "quantize":
        n = case["rows"] * case["cols"]
        return {"bytes": n * (_BYTES[case["x"]] + 4 * (0.5 + 1 / 16)), "flops": 0}
    M, K, N = case["M"], case["K"], case["N"]
    b, y = _BYTES[case.get("x", "bf16")], _BYTES[case.get("y", "fp32")]
    if op == "step":
        return {"bytes": b * (M * K + N * K + M * N) + y * (M * N + M * K) + 4 * N * K, "flops": 6.0 * M * N * K}
    if op == "wgrad":
        return {"bytes": b * (M * N + M * K) + 4 * N * K, "flops": 2.0 * M * N * K}
    if op == "chain":
        N2 = case["N2"]
        return {"bytes": 2 * (M * K + N * K + N2 * N) + y * M * N2, "flops": 2.0 * M * N * (K + N2)}
    if op == "kept":
        return {"bytes": 2 * M * K + N * K * (0.5 + 1 / 16) + y * M * N, "flops": 2.0 * M * N * K}
    if op == "qaf":
        return {"bytes": 2 * (M * K + N * K + M * N) + y * (M * N + M * K) + 4 * N * K, "flops": 6.0 * M * N * K}
    if case["which"] == "fwd":
        return {"bytes": 2 * (M * K + N * K) + y * M * N, "flops": 2.0 * M * N * K}
    return {"bytes": 2 * (M * K + M * N) + y * N * K, "flops": 2.0 * M * N * K}


def tolerance(case):
    """About four times the error measured against the same codes (or bf16 values) multiplied in float64: one bf16 rounding
    of the result is 1.7e-3 (largest 3.9e-3 of the value); fp32 sums of NVFP4 products differ by 4e-8 (largest 2e-7) at
    contractions of 512 to 65536, a few times that when added in another order; fp32 sums of bf16 products by 2e-5
    (largest 6e-5) at a contraction of 16384.  Codes and scales are whole values."""
    if case["op"] == "quantize":
        return "exact"
    if case.get("y", "fp32") == "bf16":
        return {"rel": 6e-3, "max": 2e-2}
    return {"rel": 8e-5, "max": 3e-4} if case["op"] == "qaf" else {"rel": 1e-6, "max": 1e-5}


# ---- the same results in 64 bits, from plain torch -----------------------------------------------------------------
_GRID = (0.0, 0.5, 1.0, 1.5, 2.0, 3.0, 4.0, 6.0)


def _scale64(x):
    amax = x.abs().max().float()
    return torch.where(amax == 0, torch.ones_like(amax), amax / torch.full_like(amax, 2688.0))   # by a tensor: a number's reciprocal would be rounded


def _philox(seed, offset, blk):
    """Philox4x32-10 of the counters (blk, offset) under the key `seed`: four tensors of 32-bit words."""
    low = 0xFFFFFFFF
    key = [seed & low, (seed >> 32) & low]
    c = [blk & low, blk >> 32, torch.full_like(blk, offset & low), torch.full_like(blk, offset >> 32)]
    for _ in range(10):
        p, q = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57            # wraps mod 2^64: the shifted word is masked below
        c = [((q >> 32) & low) ^ c[1] ^ key[0], q & low, ((p >> 32) & low) ^ c[3] ^ key[1], p & low]
        key = [(key[0] + 0x9E3779B9) & low, (key[1] + 0xBB67AE85) & low]
    return c


def _quantized64(x, g, rounding, block=16):
    """x, in float64, after the quantization of its rows in blocks: E4M3 scales of 16 (or E8M0 scales of 32), E2M1 values."""
    out = torch.empty(x.shape, dtype=torch.float64, device=x.device)
    rows, cols = x.shape
    bit = torch.arange(16, device=x.device)
    chunk = max(1, (1 << 26) // cols)
    for r in range(0, rows, chunk):
        v = x[r:r + chunk].contiguous().float().reshape(-1, block)
        a = v.abs().amax(1) * ((torch.ones((), device=x.device) / 6.0) / g)
        if block == 16:
            sf = a.clamp(max=448.0).to(torch.float8_e4m3fn).float()
        else:
            m, e = torch.frexp(a)
            sf = torch.where(a > 0, torch.ldexp(torch.ones_like(a), e - (m == 0.5).to(e.dtype)), torch.zeros_like(a))
        inv = torch.where(sf > 0, 1.0 / (sf * g), torch.zeros_like(sf))
        y = (v * inv[:, None]).abs().clamp(max=6.0).double()
        step = torch.where(y < 2, 0.5, torch.where(y < 4, 1.0, 2.0))
        t = y / step
        if rounding.mode == nb.SR:
            blk = torch.arange(r * cols // 16, (r * cols + v.numel()) // 16, device=x.device)
            draws = []
            for w in _philox(rounding.seed, rounding.offset, blk):
                for half in (((w >> 8) & 0xFF00) | (w & 0xFF), ((w >> 16) & 0xFF00) | ((w >> 8) & 0xFF)):
                    draws += [half, (((half[:, None] >> bit) & 1) << (15 - bit)).sum(1)]
            u = torch.stack(draws, 1).reshape(y.shape)
            t = t.floor() + (((t - t.floor()) * 65536).floor() + u >= 65536)
        else:
            t = t.round()                                      # half to even: the even code, its mantissa bit being 0
        out[r:r + chunk] = (torch.copysign(t * step, v.double()) * sf.double()[:, None]).reshape(-1, cols)
    return out * g.double()


def exact(case, seed):
    """What run() returns, in float64: operands quantized as the number formats and the random streams define it (or taken
    as they are where the product is a bf16 one), then multiplied in float64."""
    op, sd = case["op"], int(seed) * 8
    if op == "quantize":
        return None                                            # codes and scales are whole values
    M, K, N, x = case["M"], case["K"], case["N"], case.get("x", "bf16")
    rtn, sr = nb.Rounding(nb.RTN), [nb.Rounding(nb.SR, int(seed), o) for o in range(3)]
    if op in ("step", "qaf", "wgrad"):
        X, dY = _normal((M, K), 1.0, sd, x), _normal((M, N), case.get("grad", 1e-4), sd + 2, x)
        gx, gdy = _scale64(X), _scale64(dY)
        if op != "qaf":
            dW = _quantized64(dY.T, gdy, sr[1]) @ _quantized64(X.T, gx, sr[2]).T
        if op == "wgrad":
            return dW
        W = _normal((N, K), 0.02, sd + 1, x)
        gw = _scale64(W)
        Y = _quantized64(X, gx, rtn) @ _quantized64(W, gw, rtn).T
        if op == "qaf":
            return Y, dY.double() @ W.double(), dY.double().T @ X.double()
        return Y, _quantized64(dY, gdy, sr[0]) @ _quantized64(W.T, gw, rtn).T, dW
    if op == "mx":
        if case["which"] == "fwd":
            A, B, ra, rb = _normal((M, K), 1.0, sd), _normal((N, K), 0.02, sd + 1), rtn, rtn
        else:
            A, B, ra, rb = _normal((M, N), 1e-4, sd).T, _normal((M, K), 1.0, sd + 1).T, sr[1], sr[2]
        return _quantized64(A, _scale64(A), ra, 32) @ _quantized64(B, _scale64(B), rb, 32).T
    X, W = _normal((M, K), 1.0, sd), _normal((N, K), 0.02, sd + 1)
    Y = _quantized64(X, _scale64(X), rtn) @ _quantized64(W, _scale64(W), rtn).T
    if op == "kept":
        return Y
    W2 = _normal((case["N2"], N), 0.02, sd + 2)
    gh = _scale64(Y.bfloat16())
    return _quantized64(Y.float(), gh, rtn) @ _quantized64(W2, _scale64(W2), rtn).T
