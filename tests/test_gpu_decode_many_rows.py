"""Prepared decode of nine to sixteen tokens on layers with as many rows as an output head: one launch
for all tokens does not fit there and the call is served by two."""
import numpy as np
import pytest
import torch

import oracle
from paper_2305_14152_b200 import binding, synth
from gpu_util import assert_close, bf16_to_dev, dev_to_f64, kernels_of, to_qweight

pytestmark = pytest.mark.gpu

BITS, TASKS = 4, 3


# all at once does not fit for 16 tokens, for 16, for 12 and 16
@pytest.mark.parametrize("N,K,g,two", [(102400, 1536, 64, (16,)), (151936, 512, 0, (16,)), (151936, 2560, 0, (12, 16))])
def test_rows_of_an_output_head(N, K, g, two):
    rng = np.random.default_rng(N + g)
    G = K // g if g else 1
    packed = rng.integers(0, 1 << 32, size=(N, K * BITS // 32), dtype=np.uint32)     # every word is eight codes
    zeros = rng.integers(0, 1 << BITS, size=(N, G), dtype=np.uint8)
    table = rng.uniform(0.01, 0.02, size=(TASKS, N, G)).astype(np.float32)
    qw = to_qweight(packed, zeros, table[0], BITS, g, K)
    prep = binding.decode_prepare(qw)
    torch.cuda.synchronize()
    tab = torch.from_numpy(table).cuda()
    Xb = synth.f32_to_bf16_bits(rng.standard_normal((16, K)).astype(np.float32))
    ref = oracle.fwd(Xb, packed, zeros, table[0], BITS, g)
    ids = rng.integers(0, TASKS, size=16).astype(np.int32)
    ref_tasks = oracle.fwd_multitask(Xb, packed, zeros, table, ids, BITS, g)
    for M in (9, 12, 16):
        X = bf16_to_dev(Xb[:M])
        Y = binding.qlinear_decode_prepared(qw, prep, X)
        Yt = binding.qlinear_decode_prepared(qw, prep, X, scale_table=tab, task_ids=torch.from_numpy(ids[:M]).cuda())
        binding.check_status()
        if M in two:
            assert len(kernels_of(lambda: binding.qlinear_decode_prepared(qw, prep, X))) == 2
        assert_close(dev_to_f64(Y), ref[:M], f"M={M}")
        assert_close(dev_to_f64(Yt), ref_tasks[:M], f"tasks, M={M}")
