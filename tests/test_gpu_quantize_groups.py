"""Bit parity of the warp-per-groups quantizer at the ends of its blocks of 1024 columns: matrices
smaller than one block, that end inside a block or a warp's quarter, groups of 4 to 32 lanes, tie rows,
one-sided and constant groups."""
import numpy as np
import pytest
import torch

import oracle
from paper_2305_14152_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits", [3, 4])
@pytest.mark.parametrize("g", [32, 64, 128, 256])
@pytest.mark.parametrize("N,K", [(1, 256), (3, 256), (5, 768), (13, 1280), (67, 2304), (1031, 512)])
def test_groups_bit_exact(bits, g, N, K):
    rng = np.random.default_rng(N * K + g + bits)
    W = (rng.standard_normal((N, K)) * 0.02).astype(np.float32)
    W[rng.random((N, K)) < 1e-2] *= np.float32(20.0)
    W[:, :g] = rng.integers(-4, 5, size=(N, g)).astype(np.float32) * np.float32(0.5)     # ties
    if N > 2:
        W[1] = np.abs(W[1]) + np.float32(1.0)                                            # one-sided
        W[2, -g:] = np.float32(0.25)                                                     # constant
    codes, zeros, scales = oracle.quantize_rtn(W, bits, g)
    qw = binding.quantize_rtn(torch.from_numpy(W).cuda(), bits, g)
    torch.cuda.synchronize()
    assert np.array_equal(qw.qweight.cpu().numpy().view(np.uint32), oracle.pack(codes, bits))
    assert np.array_equal(qw.zeros.cpu().numpy(), zeros)
    assert np.array_equal(qw.scales.cpu().numpy(), scales)
