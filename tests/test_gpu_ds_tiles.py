"""GPU parity of dS and its AdamW step when a CTA pair works through several tiles with few tokens:
code slots, accumulators and optimizer state of one tile follow closely on those of the last."""
import numpy as np
import pytest
import torch

import oracle
from paper_2305_14152_b200 import binding, synth
from gpu_util import adamw_scale_tol, assert_close, bf16_to_dev, dev_to_f64, oracle_layer, to_qweight

pytestmark = pytest.mark.gpu


# 160 or more tiles of 256 x 256 over 74 pairs; K % 128 == 64 (no TMA for 3-bit codes, and groups
# whose pieces cannot be read as vectors); optimizer state at an odd address
@pytest.mark.parametrize("K,bits,g,off", [(2560, 3, 64, 0), (2560, 4, 32, 1), (2560, 4, 128, 0), (2560, 4, 0, 0),
                                          (2496, 3, 64, 0), (2496, 4, 192, 0)])
def test_several_tiles_per_pair(K, bits, g, off):
    N, T = 4096, 72
    lr = float(np.float32(1e-3))
    d = synth.custom(K + g, N, K, T, bits, g, outliers=True, sigma_dy=1e-2)
    codes, zeros, scales, packed = oracle_layer(d, bits, g)
    ref = oracle.bwd_ds(d["X"], d["dY"], packed, zeros, bits, g)
    X, dY = bf16_to_dev(d["X"]), bf16_to_dev(d["dY"])
    n = scales.size
    for _ in range(3):
        qw = to_qweight(packed, zeros, scales, bits, g, K)
        m = torch.zeros(n + off, device="cuda")[off:].view(scales.shape)
        v = torch.zeros(n + off, device="cuda")[off:].view(scales.shape)
        dS = binding.qlinear_bwd_ds_adamw(qw, X, dY, m, v, lr, step=1)
        plain = binding.qlinear_bwd(qw, X, dY, need_dx=False)[1]
        binding.check_status()
        assert_close(dev_to_f64(dS), ref, "dS")
        assert torch.equal(dS, plain)
        got = dS.cpu().numpy()
        zero = np.zeros_like(scales)
        s_ref, _, _ = oracle.adamw(scales, got, zero, zero, lr, float(np.float32(0.9)), float(np.float32(0.999)),
                                   float(np.float32(1e-8)), 0.0, 1)
        tol = adamw_scale_tol(scales, got, zero, zero, lr, 0.9, 0.999, 1e-8, 0.0, 1)
        assert np.all(np.abs(qw.scales.cpu().numpy().ravel().astype(np.float64) - s_ref) <= tol)
