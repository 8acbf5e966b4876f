"""Timed cases of the quantized-linear path, through the package's public entry points.

Four kinds of work, the ones a program built on this package has it do:

  linear    one quantized linear, ``lrq_qlinear`` (rotate, quantize, contract, scale): what a model's forward calls
  block     the four linears of a DiT block (qkv, proj, fc1, fc2) or the two of an MLP through ``lrq_qlinear_stack``
  quantize  the activation side alone, ``lrq_rotate_quantize_act``
  convert   the offline side of one layer: metric of Eq. 11 on calibration tokens (``lrq_ars_select``), weight rotation
            (``lrq_rotate_weights``), twin-log quantization with its clipping search (``lrq_tlq_quantize_weights``)

Shapes are those of the package's workloads (``lrq_workloads``): a single small linear, PixArt-, MMDiT- and FLUX-shaped
layers and a video-DiT block.  Weights are long-tailed (Student-t), activations N(0, 1) with mild outliers and, for the
layers that need the outlier-aware rotation, salient channels.  A program keeps its layers, its workspace and (for a
stack) its output buffers; a single linear returns a new tensor, as a module's forward does.
"""
import math

import torch

import paper_2508_03485_b200 as P

_OUT = {"f32": P.F32, "f16": P.F16, "bf16": P.BF16}
_TORCH_OUT = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
_ROT = {"hadamard": P.ROT_HADAMARD, "dense": P.ROT_DENSE, "dual": P.ROT_DUAL}
_GRID = [round(1.0 + 0.02 * i, 2) for i in range(31)]      # clipping factors of the search
_DUAL_BLOCK = 128


# ------------------------------------------------------------------------------------------------- cases
def _linear(name, M, K, N, w_bits, a_bits, rot, block, out, group=0, packed3=False, bias=True, smooth=False):
    return {"name": name, "kind": "linear", "M": M, "K": K, "N": N, "w_bits": w_bits, "a_bits": a_bits, "rot": rot,
            "block": block, "out": out, "group": group, "packed3": packed3, "bias": bias, "smooth": smooth}


def listed():
    return [
        # the smallest configuration: one call of a few microseconds, 3-bit codes in their true packing
        _linear("linear_m256_w3a4_packed", 256, 1024, 1024, 3, 4, "hadamard", 1024, "f32", packed3=True, bias=False),
        # the text side of a joint-attention model: 333 tokens, grouped tables
        _linear("text_m333_w3a4_g128", 333, 1536, 1536, 3, 4, "hadamard", 512, "f16", group=128),
        # image generation at 4096 tokens, hidden 1152: one block's linears, smoothing and biases on
        {"name": "pixart_block_m4096_w4a8", "kind": "block", "M": 4096, "hidden": 1152, "mlp": 4608, "attention": True,
         "w_bits": 4, "a_bits": 8, "group": 0, "block": 128, "mlp_block": 128, "out": "bf16", "smooth": True},
        # joint attention, 4096 image + 333 text tokens: down projection behind a large Hadamard block, grouped tables
        _linear("mmdit_fc2_m4429_w3a4_g128", 4429, 6144, 1536, 3, 4, "hadamard", 2048, "f16", group=128),
        # the same model's up projection on a layer with salient channels: dense outlier-aware rotation
        _linear("mmdit_fc1_dense_m4429_w3a4", 4429, 1536, 6144, 3, 4, "dense", 0, "f16", group=128),
        # 4096 image + 512 text tokens, hidden 3072: both linears of the MLP (Hadamard blocks of 1024 and 4096)
        {"name": "flux_mlp_m4608_w4a4", "kind": "block", "M": 4608, "hidden": 3072, "mlp": 12288, "attention": False,
         "w_bits": 4, "a_bits": 4, "group": 0, "block": 1024, "mlp_block": 4096, "out": "bf16", "smooth": False},
        # its qkv on a salient layer, the rotation as one dense matrix ...
        _linear("flux_qkv_dense_m4608_w4a4", 4608, 3072, 9216, 4, 4, "dense", 0, "bf16"),
        # ... and kept in the factors of the dual transformation
        _linear("flux_qkv_dual_m4608_w4a4", 4608, 3072, 9216, 4, 4, "dual", _DUAL_BLOCK, "bf16"),
        # the largest: one block of a video DiT, 2 x 16 frames x 1024 tokens, fp32 outputs
        {"name": "video_block_m32768_w4a8", "kind": "block", "M": 32768, "hidden": 1152, "mlp": 4608, "attention": True,
         "w_bits": 4, "a_bits": 8, "group": 0, "block": 128, "mlp_block": 128, "out": "f32", "smooth": False},
        # the activation side alone, for codes that several consumers share
        {"name": "quantize_m32768_k4608_a8", "kind": "quantize", "M": 32768, "K": 4608, "a_bits": 8, "rot": "hadamard",
         "block": 128, "smooth": False},
        # offline conversion of one layer: Hadamard, 4 bits per channel
        {"name": "convert_4608x1152_w4", "kind": "convert", "M": 4096, "K": 1152, "N": 4608, "w_bits": 4, "group": 0,
         "rot": "hadamard", "block": 128},
        # and of a salient one: dense rotation, 3 bits, groups of 128
        {"name": "convert_dense_4608x1536_w3_g128", "kind": "convert", "M": 4429, "K": 1536, "N": 4608, "w_bits": 3,
         "group": 128, "rot": "dense", "block": 0},
    ]


def _log_int(rng, lo, hi, step=1):
    """A multiple of `step` between lo and hi, evenly spread over the logarithm."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, min(hi, int(round(v / step)) * step))


def _pow2_divisor(K, most):
    b = K & -K
    return min(b, most)


def _block_of(rng, K):
    """The block of a Hadamard layer: 128 where the workload says so, else the largest power of two dividing K."""
    big = _pow2_divisor(K, 4096)
    return 128 if big > 128 and rng.random() < 0.4 else big


def draw(rng):
    kind = rng.choice(["linear"] * 6 + ["block"] * 2 + ["quantize", "convert"])
    w_bits, a_bits = rng.choice([(4, 8), (4, 4), (3, 4), (3, 8), (4, 8), (4, 4)])
    if kind == "linear":
        rot = rng.choice(["hadamard", "hadamard", "hadamard", "dense", "dual"])
        M = _log_int(rng, 16, 32768)
        K = _log_int(rng, 512, 4096 if rot != "hadamard" else 12288, 128 if rot == "dual" else 64)
        N = _log_int(rng, 512, 12288, 8)
        while M * K * (N + (K if rot == "dense" else 0)) > 2.5e11:
            M = max(16, M // 2)
        packed3 = w_bits == 3 and M <= 512 and rng.random() < 0.5
        group = 0 if packed3 or K % 128 or rng.random() < 0.5 else 128
        block = _block_of(rng, K) if rot == "hadamard" else _DUAL_BLOCK if rot == "dual" else 0
        c = _linear("", M, K, N, w_bits, a_bits, rot, block, rng.choice(["f32", "f16", "bf16", "bf16"]), group, packed3,
                    rng.random() < 0.7, rot == "hadamard" and rng.random() < 0.3)
        del c["name"]
        return c
    if kind == "block":
        hidden = _log_int(rng, 768, 3072, 128)
        M = _log_int(rng, 256, 32768)
        while M * hidden * hidden * 12 > 5e11:
            M = max(256, M * 3 // 4)
        group = 128 if rng.random() < 0.3 else 0
        return {"kind": "block", "M": M, "hidden": hidden, "mlp": 4 * hidden, "attention": rng.random() < 0.7,
                "w_bits": w_bits, "a_bits": a_bits, "group": group, "block": _block_of(rng, hidden),
                "mlp_block": _block_of(rng, 4 * hidden), "out": rng.choice(["f32", "f16", "bf16"]),
                "smooth": rng.random() < 0.3}
    if kind == "quantize":
        K = _log_int(rng, 512, 12288, 64)
        M = _log_int(rng, 64, 32768)
        while M * K > 32768 * 4608:
            M //= 2
        return {"kind": "quantize", "M": M, "K": K, "a_bits": a_bits, "rot": "hadamard", "block": _block_of(rng, K),
                "smooth": rng.random() < 0.3}
    rot = rng.choice(["hadamard", "dense"])
    K = _log_int(rng, 512, 2048 if rot == "dense" else 6144, 64)
    N = _log_int(rng, 512, 9216, 8)
    while N * K > 16e6:
        N //= 2
    group = 128 if K % 128 == 0 and rng.random() < 0.5 else 0
    return {"kind": "convert", "M": _log_int(rng, 256, 8192), "K": K, "N": N, "w_bits": w_bits, "group": group, "rot": rot,
            "block": _block_of(rng, K) if rot == "hadamard" else 0}


# ------------------------------------------------------------------------------------------------- inputs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _weights(g, N, K):
    """Student-t with 4 degrees of freedom, standard deviation 0.02, float32 [N, K]."""
    z = torch.randn((N, K), generator=g, device="cuda")
    chi2 = torch.zeros((N, K), device="cuda")
    for _ in range(4):
        chi2 += torch.randn((N, K), generator=g, device="cuda").square_()
    return z.mul_((chi2 / 4.0).rsqrt_()).mul_(0.02 / math.sqrt(2.0))


def _activations(g, M, K, salient):
    """bf16 [M, K]: N(0, 1), 0.5 % of the entries x5; `salient` fixed channels x100."""
    out = torch.empty((M, K), dtype=torch.bfloat16, device="cuda")
    channels = torch.randperm(K, generator=g, device="cuda")[:salient]
    for m0 in range(0, M, 8192):
        n = min(M, m0 + 8192) - m0
        x = torch.randn((n, K), generator=g, device="cuda")
        x = torch.where(torch.rand((n, K), generator=g, device="cuda") < 0.005, x * 5.0, x)
        if salient:
            x[:, channels] *= 100.0
        out[m0:m0 + n] = x
    return out


def _orthogonal(g, K):
    q, r = torch.linalg.qr(torch.randn((K, K), generator=g, device="cuda"))
    return (q * torch.sign(torch.diagonal(r))[None, :]).bfloat16().contiguous()


def _block_rotations(g, K):
    q, r = torch.linalg.qr(torch.randn((K // _DUAL_BLOCK, _DUAL_BLOCK, _DUAL_BLOCK), generator=g, device="cuda"))
    return (q * torch.sign(torch.diagonal(r, dim1=1, dim2=2))[:, None, :]).bfloat16().contiguous()


def _smoothing(g, K):
    return torch.rand((K,), generator=g, device="cuda") * 1.5 + 0.25


def _layer(g, K, N, w_bits, a_bits, group, rot, block, packed3, bias, smooth):
    """One layer's handle: weights drawn in the rotated basis, quantized once; the handle keeps what it points to."""
    tlq = P.lrq_tlq_quantize_weights(_weights(g, N, K), w_bits, group, 7, _GRID, _GRID,
                                     code_layout=P.CODES_PACKED3 if packed3 else P.CODES_NIBBLE)
    R = _orthogonal(g, K) if rot == "dense" else None
    dual = None
    if rot == "dual":
        dual = P.DualRotation(_DUAL_BLOCK, _block_rotations(g, K),
                              torch.randperm(K, generator=g, device="cuda").to(torch.int32), _block_rotations(g, K))
    return P.QLayer(tlq, N, K, _ROT[rot], a_bits, block, R, dual=dual,
                    bias=torch.randn((N,), generator=g, device="cuda") if bias else None,
                    prescale=_smoothing(g, K) if smooth else None)


def _block_shapes(c):
    h, f = c["hidden"], c["mlp"]
    shapes = [(h, 3 * h, c["block"]), (h, h, c["block"])] if c["attention"] else []
    return shapes + [(h, f, c["block"]), (f, h, c["mlp_block"])]


def prepare(case, seed):
    c, g = case, _generator(seed)
    if c["kind"] == "linear":
        layer = _layer(g, c["K"], c["N"], c["w_bits"], c["a_bits"], c["group"], c["rot"], c["block"], c["packed3"], c["bias"],
                       c["smooth"])
        X = _activations(g, c["M"], c["K"], 0 if c["rot"] == "hadamard" else 16)
        return {"run": "linear", "layer": layer, "X": X, "out": _OUT[c["out"]],
                "workspace": torch.empty(layer.workspace_bytes(c["M"]), dtype=torch.uint8, device="cuda")}
    if c["kind"] == "block":
        layers, Xs, Ys, by_k = [], [], [], {}
        for K, N, block in _block_shapes(c):
            layers.append(_layer(g, K, N, c["w_bits"], c["a_bits"], c["group"], "hadamard", block, False, True, c["smooth"]))
            if K not in by_k:
                by_k[K] = _activations(g, c["M"], K, 0)
            Xs.append(by_k[K])
            Ys.append(torch.empty((c["M"], N), dtype=_TORCH_OUT[c["out"]], device="cuda"))
        plan = P.StackPlan(layers, Xs, Ys, _OUT[c["out"]])
        return {"run": "block", "plan": plan, "Ys": Ys, "workspace": torch.empty(plan.need, dtype=torch.uint8, device="cuda")}
    if c["kind"] == "quantize":
        return {"run": "quantize", "X": _activations(g, c["M"], c["K"], 0), "a_bits": c["a_bits"], "block": c["block"],
                "prescale": _smoothing(g, c["K"]) if c["smooth"] else None}
    salient = 16 if c["rot"] == "dense" else 0
    return {"run": "convert", "X": _activations(g, c["M"], c["K"], salient), "W": _weights(g, c["N"], c["K"]),
            "R": _orthogonal(g, c["K"]) if c["rot"] == "dense" else None, "rot": _ROT[c["rot"]], "block": c["block"],
            "w_bits": c["w_bits"], "group": c["group"]}


# ------------------------------------------------------------------------------------------------- the pass
def run(state):
    s = state
    if s["run"] == "linear":
        return P.lrq_qlinear(s["layer"], s["X"], s["out"], workspace=s["workspace"])
    if s["run"] == "block":
        P.lrq_qlinear_stack(s["plan"], s["workspace"])
        return s["Ys"]
    if s["run"] == "quantize":
        return P.lrq_rotate_quantize_act(s["X"], P.ROT_HADAMARD, s["a_bits"], s["block"], prescale=s["prescale"])
    J, kind = P.lrq_ars_select(s["X"], 1.0)
    W = P.lrq_rotate_weights(s["W"], s["rot"], s["block"], s["R"])
    t = P.lrq_tlq_quantize_weights(W, s["w_bits"], s["group"], 7, _GRID, _GRID)
    return {"J": J, "kind": kind, "W_rot": W, "codes": t.codes, "levels": t.levels, "wsum": t.wsum}


# ------------------------------------------------------------------------------------------------- its work
def _rotation_work(M, K, rot, block):
    """(bytes of the rotation's own operands, operations) of rotating M rows of K."""
    if rot == "dense":
        return 2 * K * K, 2.0 * M * K * K
    if rot == "dual":
        return 4 * K * _DUAL_BLOCK + 4 * K, 4.0 * M * K * _DUAL_BLOCK
    return 0, float(M) * K * math.log2(block)


def _linear_work(M, K, N, w_bits, group, rot, block, out_bytes):
    rb, rf = _rotation_work(M, K, rot, block)
    tables = N * (K // group if group else 1) * (1 << w_bits) * 4
    return 2 * M * K + N * K * w_bits // 8 + tables + 4 * N + out_bytes * M * N + rb, 2.0 * M * N * K + rf


def work(case):
    c = case
    if c["kind"] == "linear":
        b, f = _linear_work(c["M"], c["K"], c["N"], c["w_bits"], c["group"], c["rot"], c["block"], 4 if c["out"] == "f32" else 2)
    elif c["kind"] == "block":
        parts = [_linear_work(c["M"], K, N, c["w_bits"], c["group"], "hadamard", block, 4 if c["out"] == "f32" else 2)
                 for K, N, block in _block_shapes(c)]
        b, f = sum(p[0] for p in parts), sum(p[1] for p in parts)
    elif c["kind"] == "quantize":
        b = c["M"] * c["K"] * (2 + c["a_bits"] / 8) + 8 * c["M"]
        f = c["M"] * c["K"] * (math.log2(c["block"]) + 4.0)
    else:
        rb, rf = _rotation_work(c["N"], c["K"], c["rot"], c["block"])
        groups = c["K"] // c["group"] if c["group"] else 1
        b = 2 * c["M"] * c["K"] + 8 * c["N"] * c["K"] + c["N"] * c["K"] // 2 + c["N"] * groups * (4 << c["w_bits"]) + rb
        # one de-quantization and squared error per weight and factor is what the search means
        f = 2.0 * c["M"] * c["K"] + rf + 4.0 * len(_GRID) * c["N"] * c["K"]
    return {"bytes": float(b), "flops": float(f)}


def tolerance(case):
    # Measured against the same path in fp64 (about four times what was seen).  What shows is Eq. 1's rounding: an
    # element whose y/s lies on a rounding boundary may take the neighbouring code (at most 1e-4 of them), worth
    # s |w| in one token's outputs.  With 8-bit codes that came to 1.9e-4 relative and 2e-2 of the root mean square
    # at most, with 4-bit codes to 7.6e-4 and 0.32; the fp32 sums themselves are three orders below.
    if case["kind"] == "convert":
        # fp64 rounded once to fp32 (an ulp where the rounding is close); codes and tables are the same bits
        return {"rel": 1e-6, "max": 1e-5, "differ": 1e-6}
    if case["a_bits"] == 8:
        return {"rel": 8e-4, "max": 0.1, "differ": 1e-4}
    return {"rel": 3e-3, "max": 0.9, "differ": 1e-4}
