"""A token's codes, step and zero-point do not depend on the batch it is in, nor on the tokens beside it."""
import pytest
import torch

import parity as PU

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2508_03485_b200 as P
    P.load_library()
    return P


def _tokens(M, K, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.randn((M, K), generator=g, device="cuda")
    return torch.where(torch.rand(X.shape, generator=g, device="cuda") < 0.005, X * 5, X).bfloat16()


@pytest.mark.parametrize("K,B,a_bits,symmetric", [(2048, 2048, 4, False), (6144, 2048, 8, True), (10240, 2048, 8, False), (4096, 4096, 8, False),
                                                  (12288, 4096, 4, False)])
def test_large_blocks_in_long_and_short_batches(P, K, B, a_bits, symmetric):
    M = 12_100_000 // K + 2
    X = _tokens(M, K, K + B)
    # inputs over 16 octaves, whose sums are rounded at every stage
    X[:16] = (torch.sign(X[:16].float()) * torch.exp2(-16 * torch.rand((16, K), device="cuda"))).bfloat16()
    # sums that overflow, in the block's first blocks of 128 channels to +inf, -inf, +inf, +inf: NaN for every other channel two
    # stages on, among finite values
    X[20, :512] = 0
    for i, v in enumerate((3e38, -3e38, 3e38, 3e38)):
        X[20, 128 * i:128 * i + 2] = v
    X[21, 5] = float("inf"); X[22, 7] = float("nan"); X[23] = float("nan"); X[24] = 0
    mode = P.ACT_SYM if symmetric else P.ACT_ASYM
    long = P.lrq_rotate_quantize_act(X, P.ROT_HADAMARD, a_bits, B, mode=mode)
    for i in (0, M // 2, M - 64):
        for a, b in zip(long, P.lrq_rotate_quantize_act(X[i:i + 64], P.ROT_HADAMARD, a_bits, B, mode=mode)):
            assert torch.equal(a[i:i + 64], b)
    # the contraction's operand: no NaN of an overflow in it
    g = torch.Generator(device="cuda").manual_seed(7)
    tlq = P.lrq_tlq_quantize_weights(0.02 * torch.randn((32, K), generator=g, device="cuda"), 4, 0, 7, [1.0, 1.2], [1.0, 1.2])
    layer = P.QLayer(tlq, 32, K, P.ROT_HADAMARD, a_bits, B, mode=mode)
    Y = P.lrq_qlinear(layer, X, P.F32)
    assert torch.isfinite(Y[20]).all() and torch.equal(Y[20], P.lrq_qlinear(layer, X[:64], P.F32)[20])
    assert P.lrq_device_status() == 0


@pytest.mark.parametrize("symmetric", [False, True])
@pytest.mark.parametrize("K,B", [(128, 8), (384, 16), (2048, 64), (1152, 128), (4608, 128), (12288, 128)])
def test_nan_of_a_small_block_has_no_part_in_the_range(P, K, B, symmetric):
    # A NaN makes its block NaN.  The block takes code 0, the others are coded as if it were zeros; whether the NaN's threads share
    # their warp with the whole token, with the element that sets its range, or with neither.
    X = _tokens(70, K, K)
    X[:, K - 1] = 30
    X[:, 0] = -30
    at = {3: 1, 4: K // 2, 5: K - B - 1, 37: K // 2 + 1}
    clean = X.clone()
    for m, k in at.items():
        X[m, k] = float("nan")
        clean[m, k // B * B:k // B * B + B] = 0
    X[40] = float("nan")                               # nothing else: unit step
    mode = P.ACT_SYM if symmetric else P.ACT_ASYM
    for a_bits in (8, 4):
        (q, s, z), (q1, s1, z1) = (P.lrq_rotate_quantize_act(t, P.ROT_HADAMARD, a_bits, B, mode=mode) for t in (X, clean))
        if a_bits == 4:
            q, q1 = (torch.stack([t & 15, t >> 4], -1).reshape(70, -1) for t in (q, q1))
        others = [m for m in range(70) if m != 40]
        assert torch.equal(s[others], s1[others]) and torch.equal(z[others], z1[others]) and s[40] == 1
        for m, k in at.items():
            q1[m, k // B * B:k // B * B + B] = 0
        assert torch.equal(q[others], q1[others])
    assert P.lrq_device_status() == 0


@pytest.mark.parametrize("K,a_bits,symmetric", [(768, 8, False), (1152, 4, False), (1664, 8, True), (4608, 8, False), (8320, 4, False)])
def test_blocks_of_128_in_long_and_short_batches(P, K, a_bits, symmetric):
    # Inputs on a grid, so that every sum of the transform is exact whatever its order: all that is left are the token's parameters and
    # the rounding of its codes, which are one arithmetic in every kernel.
    M = PU.TC_OPERAND // K + 70
    X = (_tokens(M, K, K).float() * 16).round().clamp(-1000, 1000).div(16).bfloat16()
    plain = X.clone()
    # tokens that need the clamp or have no numbers, beside ordinary ones in the same warp
    X[3] = 0; X[9, 5] = float("inf"); X[20, 7] = float("nan"); X[33] = 3; X[40] = float("nan"); X[M - 9, 1] = -float("inf")
    X[50] *= 2.0 ** 100; X[51] *= 2.0 ** -100
    special = [3, 9, 20, 33, 40, 50, 51, M - 9]
    mode = P.ACT_SYM if symmetric else P.ACT_ASYM
    long, alone = (P.lrq_rotate_quantize_act(t, P.ROT_HADAMARD, a_bits, 128, mode=mode) for t in (X, plain))
    for i in (0, M // 2, M - 64):
        for a, b in zip(long, P.lrq_rotate_quantize_act(X[i:i + 64], P.ROT_HADAMARD, a_bits, 128, mode=mode)):
            assert torch.equal(a[i:i + 64], b)
    ordinary = torch.ones(M, dtype=torch.bool, device="cuda")
    ordinary[special] = False
    for a, b in zip(long, alone):
        assert torch.equal(a[ordinary], b[ordinary])
    # the contraction's operand, by the outputs
    g = torch.Generator(device="cuda").manual_seed(7)
    tlq = P.lrq_tlq_quantize_weights(0.02 * torch.randn((32, K), generator=g, device="cuda"), 4, 0, 7, [1.0, 1.2], [1.0, 1.2])
    layer = P.QLayer(tlq, 32, K, P.ROT_HADAMARD, a_bits, 128, mode=mode)
    Y = P.lrq_qlinear(layer, X, P.F32)
    for i in (0, M // 2, M - 64):
        assert torch.equal(Y[i:i + 64].nan_to_num(1.5), P.lrq_qlinear(layer, X[i:i + 64], P.F32).nan_to_num(1.5))
    assert torch.equal(Y[ordinary], P.lrq_qlinear(layer, plain, P.F32)[ordinary])
    assert P.lrq_device_status() == 0


@pytest.mark.parametrize("kind", ["octaves", "salient", "gelu"])
def test_sums_of_a_long_batch_are_as_close_as_those_of_short_ones(P, kind):
    # A token's step in symmetric mode is its largest |y|, so its error is that of the transform's sums and a last rounding.  Inputs of
    # many octaves, whose sums need more bits than fp32 has.
    K, B = 1152, 128
    M = PU.TC_CODES // K + 2
    g = torch.Generator(device="cuda").manual_seed(11)
    X = torch.randn((M, K), generator=g, device="cuda")
    if kind == "octaves":
        X = torch.sign(X) * torch.exp2(-16 * torch.rand((M, K), generator=g, device="cuda"))
    elif kind == "salient":
        X[:, ::72] *= 100
    else:
        X = torch.nn.functional.gelu(1.5 * X, approximate="tanh")
    X = X.bfloat16()
    H = torch.ones((1, 1), dtype=torch.float64, device="cuda")
    while H.shape[0] < B:
        H = torch.cat([torch.cat([H, H], 1), torch.cat([H, -H], 1)])
    exact = (X.double().view(M, K // B, B) @ H).abs().amax((1, 2)) / B ** 0.5 / 127
    long = P.lrq_rotate_quantize_act(X, P.ROT_HADAMARD, 8, B, mode=P.ACT_SYM)
    short = [torch.cat(t) for t in zip(*(P.lrq_rotate_quantize_act(X[i:i + 2048], P.ROT_HADAMARD, 8, B, mode=P.ACT_SYM) for i in range(0, M, 2048)))]
    rms = [((s.double() - exact) / exact).pow(2).mean().sqrt() for s in (long[1], short[1])]
    # the two differ in the rounding of a few sums of sixteen only; chained products on the tensor cores had 1.08 to 2.7 times the error
    assert rms[0] <= 1.02 * rms[1]
    # and a code differs where such a sum lies on a rounding boundary
    assert (long[0] != short[0]).sum() <= 1e-6 * M * K


@pytest.mark.parametrize("a_bits", [8, 4])
def test_overflow_within_a_block_of_128(P, a_bits):
    # Sums that overflow in sixteens of a block to +inf, -inf, +inf, +inf: NaN for every other channel, finite values beside them.
    # They have no part in the range and take code 0, in the operand its lowest value.
    K = 1152
    M = PU.TC_OPERAND // K + 2
    X = _tokens(M, K, 3)
    for m in (20, M - 5):
        X[m, 128:256] = 0
        for i, v in enumerate((3e38, -3e38, 3e38, 3e38)):
            X[m, 128 + 16 * i:130 + 16 * i] = v
    long = P.lrq_rotate_quantize_act(X, P.ROT_HADAMARD, a_bits, 128)
    for i in (0, M - 64):
        m = 20 if i == 0 else 59
        short = P.lrq_rotate_quantize_act(X[i:i + 64], P.ROT_HADAMARD, a_bits, 128)
        for a, b in zip(long, short):
            assert torch.equal(a[i:i + 64][m], b[m])
    g = torch.Generator(device="cuda").manual_seed(7)
    tlq = P.lrq_tlq_quantize_weights(0.02 * torch.randn((32, K), generator=g, device="cuda"), 4, 0, 7, [1.0, 1.2], [1.0, 1.2])
    layer = P.QLayer(tlq, 32, K, P.ROT_HADAMARD, a_bits, 128)
    Y = P.lrq_qlinear(layer, X, P.F32)
    assert torch.isfinite(Y).all() and torch.equal(Y[20], P.lrq_qlinear(layer, X[:64], P.F32)[20])
    assert P.lrq_device_status() == 0
