"""Long batches of rotate + quantize: blocks of 128 channels on the tensor cores."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import oracle
import parity as PU

pytestmark = pytest.mark.gpu

B = 128


@pytest.fixture(scope="module")
def P():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2508_03485_b200 as P
    P.load_library()
    return P


def _codes(q, a_bits):
    return q.int() if a_bits == 8 else torch.stack([q & 15, q >> 4], -1).reshape(q.shape[0], -1).int()


def _kernels(calls):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, os.path.join(root, "tests", "quantizer_kernels.py")], input=json.dumps(calls), capture_output=True,
                       text=True, timeout=300, env={**os.environ, "PYTHONPATH": root})
    assert r.returncode == 0, r.stderr
    return json.loads(r.stdout.splitlines()[-1])


def _layer(P, K, a_bits, mode=0):
    g = torch.Generator(device="cuda").manual_seed(K)
    tlq = P.lrq_tlq_quantize_weights(0.02 * torch.randn((32, K), generator=g, device="cuda"), 4, 0, 7, [1.0, 1.2], [1.0, 1.2])
    return P.QLayer(tlq, 32, K, P.ROT_HADAMARD, a_bits, B, mode=mode), tlq


def test_which_calls_take_it(P):
    calls, want = [], []

    def case(expected, M, K, what="codes", a_bits=8, block=B, **kw):
        calls.append({"M": M, "K": K, "what": what, "a_bits": a_bits, "block": block, **kw})
        want.append(expected)

    # both sides of each line; the operand also wants a block quantizer of at most five sub-groups an SM (ten of one or two warps at 512,
    # 2048 and 4096 channels, six of three at 3072 and 6144)
    for K, few in ((512, False), (768, True), (1152, True), (2048, False), (3072, False), (4096, False), (4608, True), (6144, False), (8320, True),
                   (16384, True)):
        codes, operand = -(-PU.TC_CODES // K), -(-PU.TC_OPERAND // K)
        for a_bits in (8, 4):
            case(False, codes - 1, K, a_bits=a_bits)
            case(K >= 768, codes, K, a_bits=a_bits)
            case(False, operand - 1, K, "operand", a_bits)
            case(K >= 768 and few, operand, K, "operand", a_bits)
    # multipliers, other blocks, codes that do not start on 32 bytes
    M = -(-PU.TC_OPERAND // 6144)
    case(True, M, 6144)
    case(False, M, 6144, smooth=True)
    for block in (64, 512, 2048):
        case(False, M, 6144, block=block)
    case(False, M, 6144, offset=16)
    case(True, M, 6144, offset=32)
    case(False, -(-PU.TC_OPERAND // 12288), 12288, "operand", block=4096)
    for c, n, w in zip(calls, _kernels(calls), want):
        assert ("rotq_tc_kernel" in n) == w, (c, n)


def test_codes_that_start_on_16_bytes(P):
    K, M = 1152, PU.TC_CODES // 1152 + 1
    X = torch.randn((M, K + 8), device="cuda").bfloat16()[:, :K]
    q, s, z = P.lrq_rotate_quantize_act(X, P.ROT_HADAMARD, 8, B)
    out = (torch.empty(M * K + 16, dtype=torch.uint8, device="cuda")[16:], torch.empty_like(s), torch.empty_like(z))
    P.lrq_rotate_quantize_act(X, P.ROT_HADAMARD, 8, B, out=out)
    assert (out[0].view(M, K) != q).sum() <= 1e-6 * M * K and (out[2] != z).sum() <= 1
    assert P.lrq_device_status() == 0


# tokens that fill their steps unevenly: 1, 2, 3, 9 and 21 a step, blocks of a token from 6 to 128, rows of a part warp, pitches
@pytest.mark.parametrize("K,a_bits,pad,symmetric", [(768, 8, 0, False), (1152, 8, 8, False), (1664, 4, 0, True), (4608, 8, 0, True),
                                                    (8320, 4, 24, False), (16384, 8, 0, False)])
def test_against_oracle_and_general_path(P, K, a_bits, pad, symmetric):
    M = PU.TC_OPERAND // K + 2
    g = torch.Generator(device="cuda").manual_seed(K + B)
    whole = torch.randn((M, K + pad), generator=g, device="cuda")
    whole = torch.where(torch.rand(whole.shape, generator=g, device="cuda") < 0.005, whole * 5, whole).bfloat16()
    X = whole[:, :K]
    # tokens with something else in them: zeros, one value (a range of zero behind the first channel of a block), large and tiny
    # magnitudes, one side of zero, an infinity, two of them, a NaN, nothing but NaN
    X[1] = 0; X[2] = 3; X[3] *= 1e30; X[4] *= 1e-30; X[5] = X[5].abs() * 0.1 + 4
    X[6, K - 3] = float("inf"); X[7, 0] = float("inf"); X[7, 1] = -float("inf"); X[8, K // 2] = float("nan"); X[9] = float("nan")
    mode = P.ACT_SYM if symmetric else P.ACT_ASYM
    q, s, z = P.lrq_rotate_quantize_act(X, P.ROT_HADAMARD, a_bits, B, mode=mode)
    # the general path: the same tokens a few at a time.  Special tokens give the same bits, ordinary ones the same but for sums of inputs
    # many octaves apart (an ulp of the step, a code on a rounding boundary)
    few = [P.lrq_rotate_quantize_act(X[i:i + 64], P.ROT_HADAMARD, a_bits, B, mode=mode) for i in (0, M - 64)]
    for (q1, s1, z1), rows in zip(few, (slice(0, 64), slice(M - 64, M))):
        d = _codes(q[rows], a_bits) - _codes(q1, a_bits)
        assert ((s[rows] == s1) | ((s[rows] - s1).abs() <= 1.2e-7 * s1)).all() and (z[rows] == z1).all()
        assert (d.abs() <= 1).all() and (d != 0).sum() <= 1
        if rows.start == 0:
            special = [1, 2, 6, 7, 9]
            assert torch.equal(s[special], s1[special]) and (d[special] == 0).all()
    # a NaN is kept out of the token's range: as if its block were zeros, and coded 0
    k0 = K // 2 // 128 * 128
    clean = X[:64].clone()
    clean[8, k0:k0 + 128] = 0
    q1, s1, z1 = P.lrq_rotate_quantize_act(clean, P.ROT_HADAMARD, a_bits, B, mode=mode)
    c, c1 = _codes(q[8:9], a_bits)[0], _codes(q1[8:9], a_bits)[0]
    assert (s[8] - s1[8]).abs() <= 1.2e-7 * s1[8] and z[8] == z1[8] and (c[k0:k0 + 128] == 0).all()
    assert (c != c1)[:k0].sum() + (c != c1)[k0 + 128:].sum() <= 1
    # the oracle, on tokens from both ends of the batch
    rows = np.r_[10:26, M - 16:M]
    Yr = oracle.rotate_hadamard_fwht(X[torch.as_tensor(rows, device="cuda")].double().cpu().numpy(), B)
    oq, os_, oz = oracle.quantize_act(Yr, a_bits, mode)
    PU.check_act(_codes(q, a_bits)[rows].cpu().numpy(), s[rows].cpu().numpy(), z[rows].cpu().numpy(), oq, os_, oz, Yr, "hadamard", B, f"{M}x{K} B={B}")
    # the contraction's operand holds the same codes, whichever kernel writes it: the linear against the sums of these codes in
    # fp64.  Its K / 16 chained additions round toward zero, each by at most an ulp of a partial sum, taken as four times the outputs' root mean square at most
    layer, tlq = _layer(P, K, a_bits, mode)
    some = slice(M - 500, M)
    T = tlq.levels.reshape(32, 16).gather(1, _codes(tlq.codes, 4).long()).double()
    ref = s[some].double()[:, None] * ((_codes(q[some], a_bits) + z[some][:, None]).double() @ T.t())
    Y = P.lrq_qlinear(layer, X, P.F32)[some].double()
    assert (Y - ref).abs().max() <= K / 16 * 2.0 ** -23 * 4 * ref.pow(2).mean().sqrt()
    assert P.lrq_device_status() == 0
