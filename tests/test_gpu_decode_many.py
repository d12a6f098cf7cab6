"""GPU parity of the canonical decode around eight tokens, where calls change over to the cluster-split
forward: grouped and per-channel scales, more rows than columns and the other way round."""
import pytest
import torch

import oracle
from paper_2305_14152_b200 import binding, synth
from gpu_util import assert_close, bf16_to_dev, dev_to_f64, oracle_layer, to_qweight

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,bits,g", [(136, 4096, 4, 32), (264, 5120, 3, 64), (4104, 4096, 4, 128), (520, 4224, 3, 0),
                                        (5128, 4224, 4, 0), (8, 128, 4, 32)])
@pytest.mark.parametrize("M", [8, 9, 16])
def test_around_eight_tokens(N, K, bits, g, M):
    d = synth.custom(N + K, N, K, 16, bits, g, outliers=True)
    codes, zeros, scales, packed = oracle_layer(d, bits, g)
    qw = to_qweight(packed, zeros, scales, bits, g, K)
    X = bf16_to_dev(d["X"][:M])
    guard = torch.full((M * N + 512,), 7.0, dtype=torch.bfloat16, device="cuda")
    Y = guard[256:256 + M * N].view(M, N)
    binding.qlinear_decode(qw, X, Y)
    again = binding.qlinear_decode(qw, X)
    binding.check_status()
    assert torch.all(guard[:256] == 7.0) and torch.all(guard[-256:] == 7.0), "wrote outside its output"
    assert torch.equal(Y, again)
    assert_close(dev_to_f64(Y), oracle.fwd(d["X"][:M], packed, zeros, scales, bits, g), "Y")
