"""GPU parity of the forward for few and for some hundred tokens: the cluster-split kernel, whose weights lie in
tensor memory, with one and with two accumulators beside them and with token tiles of 16 to 256; either kernel with a
last tile of a few tokens and a channel tile of eight; the scale gradient from the forward's sums."""
import numpy as np
import pytest
import torch

import oracle
from paper_2305_14152_b200 import binding, synth
from gpu_util import assert_close, bf16_to_dev, dev_to_f64, oracle_layer, to_qweight

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [31, 129, 257, 545, 800, 1025])
@pytest.mark.parametrize("bits,g", [(3, 64), (4, 0)])
def test_token_tiles(bits, g, T):
    N, K = 2312, 640
    d = synth.custom(T + g, N, K, T, bits, g, outliers=True)
    codes, zeros, scales, packed = oracle_layer(d, bits, g)
    qw = to_qweight(packed, zeros, scales, bits, g, K)
    flat = torch.full((T * N + 512,), 7.0, dtype=torch.bfloat16, device="cuda")
    Y = flat[256:256 + T * N].view(T, N)
    binding.qlinear_fwd(qw, bf16_to_dev(d["X"]), Y)
    binding.check_status()
    assert torch.all(flat[:256] == 7.0) and torch.all(flat[-256:] == 7.0), "wrote outside its output"
    assert_close(dev_to_f64(Y), oracle.fwd(d["X"], packed, zeros, scales, bits, g), "Y")


@pytest.mark.parametrize("N,K,T", [(1288, 2048, 545), (2056, 1152, 330), (1032, 4096, 1030)])
def test_scale_gradient_of_token_tiles(N, K, T):
    d = synth.custom(N + T, N, K, T, 4, 0, outliers=True, sigma_dy=1e-2)
    codes, zeros, scales, packed = oracle_layer(d, 4, 0)
    qw = to_qweight(packed, zeros, scales, 4, 0, K)
    new = lambda r, c: torch.empty((r, c), dtype=torch.bfloat16, device="cuda")
    L = binding.LayerLinear(w=qw, X=bf16_to_dev(d["X"]), dY=bf16_to_dev(d["dY"]), Y=new(T, N), dX=new(T, K),
                            dS=torch.empty_like(qw.scales), workspace=binding.alloc_workspace(binding.OP_BWD, T, qw))
    binding.layer_train_step([L], apply_adamw=False)
    binding.check_status()
    toks, rows = np.arange(0, T, 37), np.arange(0, N, 11)
    assert_close(dev_to_f64(L.Y)[toks], oracle.fwd(d["X"], packed, zeros, scales, 4, 0, tokens=toks), "Y")
    assert_close(dev_to_f64(L.dX)[toks], oracle.bwd_dx(d["dY"], packed, zeros, scales, K, 4, 0, tokens=toks), "dX")
    assert_close(dev_to_f64(L.dS)[rows], oracle.bwd_ds(d["X"], d["dY"], packed, zeros, 4, 0, rows=rows), "dS")


@pytest.mark.parametrize("T", [769, 1001])
@pytest.mark.parametrize("N,K,g", [(9728, 1024, 0), (1024, 9728, 64)])
def test_short_last_round_of_ragged_tokens(N, K, g, T):
    """76 tiles of 512 x 256 on 74 CTA pairs (forward of the first shape, dX of the second): the last two are halved,
    and the last row of tiles has from one token on in its second half."""
    d = synth.custom(N + T, N, K, T, 4, g, outliers=True, sigma_dy=1e-2)
    codes, zeros, scales, packed = oracle_layer(d, 4, g)
    qw = to_qweight(packed, zeros, scales, 4, g, K)
    new = lambda c: torch.full((T + 2, c), 7.0, dtype=torch.bfloat16, device="cuda")
    Y, dX = new(N), new(K)
    L = binding.LayerLinear(w=qw, X=bf16_to_dev(d["X"]), dY=bf16_to_dev(d["dY"]), Y=Y[1:T + 1], dX=dX[1:T + 1],
                            dS=torch.empty_like(qw.scales), workspace=binding.alloc_workspace(binding.OP_BWD, T, qw))
    binding.layer_train_step([L], apply_adamw=False)
    binding.check_status()
    for out in (Y, dX):
        assert torch.all(out[0] == 7.0) and torch.all(out[-1] == 7.0), "wrote outside its output"
    toks, rows = np.array([0, 255, 256, 511, 512, 767, 768, T - 1]), np.arange(0, N, 997)
    assert_close(dev_to_f64(L.Y)[toks], oracle.fwd(d["X"], packed, zeros, scales, 4, g, tokens=toks), "Y")
    assert_close(dev_to_f64(L.dX)[toks], oracle.bwd_dx(d["dY"], packed, zeros, scales, K, 4, g, tokens=toks), "dX")
    assert_close(dev_to_f64(L.dS)[rows], oracle.bwd_ds(d["X"], d["dY"], packed, zeros, 4, g, rows=rows), "dS")
