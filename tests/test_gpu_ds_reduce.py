"""The reductions behind the scale and zero-point gradients of groups wider than 128 columns: pieces of 128 columns lie in the
workspace, and their sums are those of binary32 additions in index order, bit for bit, whether a thread reads an
output's pieces itself (up to 24) or a block reads those of 32 outputs through shared memory; at the edges of either, of
a tile of 32 pieces and of a block of 32 outputs, with one group per row and with several."""
import numpy as np
import pytest
import torch

import oracle
from paper_2305_14152_b200 import binding, synth
from gpu_util import assert_close, bf16_to_dev, dev_to_f64, oracle_layer, to_qweight

pytestmark = pytest.mark.gpu


def _in_order(pieces):
    """[outputs, pieces] fp32 -> [outputs], added one after the other."""
    acc = np.zeros(pieces.shape[0], np.float32)
    for q in range(pieces.shape[1]):
        acc = (acc + pieces[:, q]).astype(np.float32)
    return acc


# (rows, pieces of a group, groups of a row)
@pytest.mark.parametrize("N,pieces,groups", [(40, 2, 1), (264, 24, 1), (8, 25, 1), (32, 25, 1), (264, 31, 1), (40, 32, 1), (72, 33, 1),
                                             (264, 64, 1), (40, 75, 1), (24, 25, 3), (40, 4, 5), (16, 172, 1)])
def test_pieces_are_added_in_order(N, pieces, groups):
    K, T, bits = 128 * pieces * groups, 72, 4
    g = 0 if groups == 1 else 128 * pieces
    d = synth.custom(N + pieces, N, K, T, bits, g, outliers=True, sigma_dy=1e-2)
    codes, zeros, scales, packed = oracle_layer(d, bits, g)
    qw = to_qweight(packed, zeros, scales, bits, g, K)
    X, dY = bf16_to_dev(d["X"]), bf16_to_dev(d["dY"])
    guard = torch.full((N * groups + 64,), 7.0, device="cuda")
    dS = guard[32:32 + N * groups].view(N, groups)
    ws = binding.alloc_workspace(binding.OP_BWD, T, qw)
    binding.qlinear_bwd(qw, X, dY, dS=dS, workspace=ws, need_dx=False)
    binding.check_status()
    assert torch.all(guard[:32] == 7.0) and torch.all(guard[-32:] == 7.0), "wrote outside its output"
    partial = ws.view(torch.float32)[:N * K // 128].view(N * groups, pieces).cpu().numpy()
    assert np.array_equal(dS.cpu().numpy().ravel(), _in_order(partial))
    assert_close(dev_to_f64(dS), oracle.bwd_ds(d["X"], d["dY"], packed, zeros, bits, g), "dS")

    # scale and zero-point gradient, and the same with real-valued zero-points
    ws2 = binding.alloc_workspace(binding.OP_BWD_DSDZ, T, qw)
    dS2, dZ2 = binding.qlinear_bwd_dsdz(qw, X, dY, workspace=ws2)
    both = ws2.view(torch.float32)[:2 * N * K // 128].view(2, N * groups, pieces).cpu().numpy()
    s = scales.ravel()
    assert np.array_equal(dS2.cpu().numpy().ravel(), _in_order(both[0]))
    assert np.array_equal(dZ2.cpu().numpy().ravel(), -s * _in_order(both[1]))
    zf = qw.zeros.float()                                     # whole zero-points: no correction is left
    _, dS3, dZ3 = binding.qlinear_bwd_zf(qw, zf, X, dY, need_dx=False, workspace=ws2)
    binding.check_status()
    assert torch.equal(dS3, dS2) and torch.equal(dZ3, dZ2)


@pytest.mark.parametrize("N,pieces", [(40, 24), (40, 25), (264, 75)])
def test_the_optimizer_step_behind_the_sum(N, pieces):
    """qlinear_bwd_ds_adamw gives the bits of the two calls."""
    K, T = 128 * pieces, 40
    d = synth.custom(N * pieces, N, K, T, 3, 0, outliers=True, sigma_dy=1e-2)
    codes, zeros, scales, packed = oracle_layer(d, 3, 0)
    X, dY = bf16_to_dev(d["X"]), bf16_to_dev(d["dY"])
    one, two = (to_qweight(packed, zeros, scales, 3, 0, K) for _ in range(2))
    states = [(torch.zeros_like(w.scales), torch.zeros_like(w.scales)) for w in (one, two)]
    dS1 = binding.qlinear_bwd_ds_adamw(one, X, dY, *states[0], 1e-3)
    _, dS2 = binding.qlinear_bwd(two, X, dY, need_dx=False)
    binding.scale_adamw(two.scales, dS2, *states[1], 1e-3)
    binding.check_status()
    for a, b in zip((dS1, one.scales, *states[0]), (dS2, two.scales, *states[1])):
        assert torch.equal(a, b)
