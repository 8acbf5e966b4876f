"""Long batches of rotate + quantize: the Hadamard transform on the tensor cores (blocks of 128, 2048 and 4096 channels)."""
import numpy as np
import pytest
import torch

import oracle
import parity as PU

pytestmark = pytest.mark.gpu

# Calls of at least this many elements take the tensor-core kernel, a token at a time the CUDA-core kernels.
LONG = {128: 9_000_000, 2048: 12_000_000, 4096: 12_000_000}


@pytest.fixture(scope="module")
def P():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2508_03485_b200 as P
    P.load_library()
    return P


def _codes(q, a_bits):
    return q.int() if a_bits == 8 else torch.stack([q & 15, q >> 4], -1).reshape(q.shape[0], -1).int()


# tokens that fill their steps unevenly: 1, 2, 3, 9, 14 and 32 a step, blocks of a token from 4 to 128, rows of a part warp, pitches
@pytest.mark.parametrize("K,B,a_bits,pad,symmetric", [(512, 128, 8, 0, False), (1152, 128, 8, 8, False), (1664, 128, 4, 0, True), (4608, 128, 8, 0, True),
                                                      (8320, 128, 4, 24, False), (16384, 128, 8, 0, False), (2048, 2048, 4, 0, False),
                                                      (6144, 2048, 8, 8, True), (10240, 2048, 4, 0, False), (4096, 4096, 8, 0, False),
                                                      (12288, 4096, 4, 0, False), (16384, 4096, 8, 16, False)])
def test_against_oracle_and_general_path(P, K, B, a_bits, pad, symmetric):
    M = LONG[B] // K + 2
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
    # the general path: the same tokens a few at a time.  Special tokens give the same bits, ordinary ones the same but for codes on a
    # rounding boundary and extremes an ulp apart
    few = [P.lrq_rotate_quantize_act(X[i:i + 64], P.ROT_HADAMARD, a_bits, B, mode=mode) for i in (0, M - 64)]
    for (q1, s1, z1), rows in zip(few, (slice(0, 64), slice(M - 64, M))):
        d = _codes(q[rows], a_bits) - _codes(q1, a_bits)
        ordinary = torch.ones(64, dtype=torch.bool, device="cuda")
        if rows.start == 0:
            ordinary[[6, 7, 9] if B == 128 else [6, 7, 8, 9]] = False
        assert ((s[rows] - s1).abs() <= 5e-7 * s1)[ordinary].all() and (z[rows] == z1)[ordinary].all()
        assert (d[ordinary].abs() <= 1).all() and (d != 0).sum() <= max(4, 2e-4 * d.numel())
        if rows.start == 0:
            same = [6, 7, 9] if B == 128 else [6, 7, 8, 9]
            assert torch.equal(s[same], s1[same]) and torch.equal(z[same], z1[same]) and (d[same] == 0).all()
    if B == 128:
        # a NaN is kept out of the token's range: as if its block were zeros, and coded 0
        k0 = K // 2 // 128 * 128
        clean = X[:64].clone()
        clean[8, k0:k0 + 128] = 0
        q1, s1, z1 = P.lrq_rotate_quantize_act(clean, P.ROT_HADAMARD, a_bits, B, mode=mode)
        c, c1 = _codes(q[8:9], a_bits)[0], _codes(q1[8:9], a_bits)[0]
        assert (s[8] - s1[8]).abs() <= 5e-7 * s1[8] and z[8] == z1[8] and (c[k0:k0 + 128] == 0).all()
        assert ((c != c1)[:k0].sum() + (c != c1)[k0 + 128:].sum()) <= max(1, 2e-4 * K)
    # the oracle, on tokens from both ends of the batch
    rows = np.r_[10:26, M - 16:M]
    Yr = oracle.rotate_hadamard_fwht(X[torch.as_tensor(rows, device="cuda")].double().cpu().numpy(), B)
    oq, os_, oz = oracle.quantize_act(Yr, a_bits, mode)
    PU.check_act(_codes(q, a_bits)[rows].cpu().numpy(), s[rows].cpu().numpy(), z[rows].cpu().numpy(), oq, os_, oz, Yr, "hadamard", B, f"{M}x{K} B={B}")
    # the contraction's operand holds the same codes: the linear against the sums of these codes in fp64.  Its K / 16 chained additions
    # round toward zero, each by at most an ulp of a partial sum, taken as four times the outputs' root mean square at most
    W = 0.02 * torch.randn((32, K), generator=g, device="cuda")
    tlq = P.lrq_tlq_quantize_weights(W, 4, 0, 7, [1.0, 1.2], [1.0, 1.2])
    layer = P.QLayer(tlq, 32, K, P.ROT_HADAMARD, a_bits, B, mode=mode)
    some = slice(M - 500, M)
    T = tlq.levels.reshape(32, 16).gather(1, _codes(tlq.codes, 4).long()).double()
    ref = s[some].double()[:, None] * ((_codes(q[some], a_bits) + z[some][:, None]).double() @ T.t())
    Y = P.lrq_qlinear(layer, X, P.F32)[some].double()
    assert (Y - ref).abs().max() <= K / 16 * 2.0 ** -23 * 4 * ref.pow(2).mean().sqrt()
    assert P.lrq_device_status() == 0
