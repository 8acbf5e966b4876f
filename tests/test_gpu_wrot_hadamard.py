"""Hadamard rotation of weights by warps: blocks of 16 to 256 channels, chunks of 512 elements that rows and the matrix do not fill, more
chunks than the grid has warps."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,B,colmul,pad", [(1, 16, 16, False, 0), (3, 64, 64, True, 0), (5, 48, 16, False, 4), (17, 96, 32, True, 0), (31, 144, 16, True, 4),
                                              (7, 768, 256, False, 0), (2, 256, 256, True, 4), (33, 1152, 128, True, 8), (301, 1600, 64, False, 0),
                                              (9, 4608, 128, True, 0), (4609, 1168, 16, True, 0), (3, 512, 512, False, 0), (11, 1152, 128, False, 1)])
def test_against_oracle(N, K, B, colmul, pad):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2508_03485_b200 as P
    g = torch.Generator(device="cuda").manual_seed(N * K + B)
    whole = torch.randn((N, K + pad), generator=g, device="cuda")
    W = whole[:, :K]
    c = torch.rand(K, generator=g, device="cuda") + 0.5 if colmul else None
    rows = list(range(N)) if N <= 1000 else list(range(40)) + list(range(N - 40, N))
    ref = oracle.rotate_weights(W[rows].double().cpu().numpy(), None if c is None else c.double().cpu().numpy(), "hadamard", B)
    # fp64 sums rounded once: an ulp where the fp64 value is on a rounding boundary, else the same
    for out in (None, whole[:, :K]):                         # the second in the place of W
        got = P.lrq_rotate_weights(W, P.ROT_HADAMARD, B, None, colmul=c, out=out)[rows].double().cpu().numpy()
        assert (np.abs(got - ref) <= 2.0 ** -23 * np.abs(ref) + 1e-14).all()
        assert (got != ref.astype(np.float32)).mean() <= 1e-3
    if pad:
        again = torch.randn((N, K + pad), generator=torch.Generator(device="cuda").manual_seed(N * K + B), device="cuda")
        assert torch.equal(whole[:, K:], again[:, K:])       # nothing beside the rows is written
