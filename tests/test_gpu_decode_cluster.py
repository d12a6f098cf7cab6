"""GPU parity of the prepared decode where the activations are spread over a cluster of CTAs: two,
four and eight CTAs per range of rows, ranges that end inside a pair of row groups, a last step that
is not full, one and two token tiles, scales per channel, per group and per task."""
import numpy as np
import pytest
import torch

import oracle
from paper_2305_14152_b200 import binding, synth
from gpu_util import assert_close, bf16_to_dev, dev_to_f64, oracle_layer, to_qweight

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,bits,g", [(2056, 8192, 3, 0), (8, 6272, 4, 0), (4104, 4224, 4, 128), (2056, 11008, 3, 64),
                                        (1000, 12288, 4, 256), (264, 22016, 3, 0)])
def test_tokens_spread_over_a_cluster(N, K, bits, g):
    d = synth.custom(N + K, N, K, 16, bits, g, outliers=True)
    codes, zeros, scales, packed = oracle_layer(d, bits, g)
    qw = to_qweight(packed, zeros, scales, bits, g, K)
    prep = binding.decode_prepare(qw)
    rng = np.random.default_rng(K)
    table = (scales[None] * rng.uniform(0.5, 2.0, size=(3,) + scales.shape)).astype(np.float32)
    # a table at an address that allows no vector reads
    flat = torch.zeros(table.size + 1, device="cuda")
    tab = flat[1:].view(table.shape)
    tab.copy_(torch.from_numpy(table))
    torch.cuda.synchronize()
    ref = oracle.fwd(d["X"], packed, zeros, scales, bits, g)
    for M in (1, 5, 8, 9, 13, 16):
        Xb = d["X"][:M]
        X = bf16_to_dev(Xb)
        guard = torch.full((M * N + 512,), 7.0, dtype=torch.bfloat16, device="cuda")
        Y = guard[256:256 + M * N].view(M, N)
        binding.qlinear_decode_prepared(qw, prep, X, Y)
        ids = rng.integers(0, 3, size=M).astype(np.int32)
        Yt = binding.qlinear_decode_prepared(qw, prep, X, scale_table=tab, task_ids=torch.from_numpy(ids).cuda())
        again = binding.qlinear_decode_prepared(qw, prep, X)
        binding.check_status()
        assert torch.all(guard[:256] == 7.0) and torch.all(guard[-256:] == 7.0), "wrote outside its output"
        assert torch.equal(Y, again)
        assert_close(dev_to_f64(Y), ref[:M], f"M={M}")
        assert_close(dev_to_f64(Yt), oracle.fwd_multitask(Xb, packed, zeros, table, ids, bits, g), f"tasks, M={M}")
