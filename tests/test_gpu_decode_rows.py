"""GPU parity of the canonical decode around its dispatch (of these shapes those with groups of 128 and 256 of a row and
the long rows of one scale go by rows through the kernel of the prepared decode, the others to the streaming kernel and, with
more than eight tokens, to the cluster kernels; test_gpu_decode_routes.py asserts which) and of the prepared decode's fp16 and
integer operands: a row group alone, half pairs, rows that end inside a step; tokens of any magnitude in one batch."""
import numpy as np
import pytest
import torch

import oracle
from paper_2305_14152_b200 import binding, synth
from gpu_util import assert_close, bf16_to_dev, dev_to_f64, oracle_layer, to_qweight

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,bits,g", [(8, 128, 3, 0), (8, 128, 4, 128), (200, 1408, 3, 128), (200, 1408, 4, 0),
                                        (1032, 1280, 3, 256), (2056, 8192, 4, 512), (264, 22016, 3, 0), (4104, 4224, 4, 128)])
def test_canonical_rows(N, K, bits, g):
    d = synth.custom(N + K, N, K, 16, bits, g, outliers=True)
    codes, zeros, scales, packed = oracle_layer(d, bits, g)
    qw = to_qweight(packed, zeros, scales, bits, g, K)
    ref = oracle.fwd(d["X"], packed, zeros, scales, bits, g)
    for M in (1, 2, 3, 8, 9, 16):
        guard = torch.full((M * N + 512,), 7.0, dtype=torch.bfloat16, device="cuda")
        Y = guard[256:256 + M * N].view(M, N)
        X = bf16_to_dev(d["X"][:M])
        binding.qlinear_decode(qw, X, Y)
        again = binding.qlinear_decode(qw, X)
        binding.check_status()
        assert torch.all(guard[:256] == 7.0) and torch.all(guard[-256:] == 7.0), "wrote outside its output"
        assert torch.equal(Y, again)
        assert_close(dev_to_f64(Y), ref[:M], f"M={M}")


@pytest.mark.parametrize("N,K,bits", [(4744, 128, 4), (4744, 256, 3), (4752, 384, 4), (5008, 512, 3), (6120, 128, 3), (6120, 640, 4), (264, 256, 4),
                                      (4744, 4096, 3)])
def test_canonical_rows_of_several_tasks(N, K, bits):
    """One scale per row, also where the row is as long as a group of 128 or 256 columns; by rows from 4744 rows on."""
    rng = np.random.default_rng(N + K)
    d = synth.custom(N + K, N, K, 16, bits, 0, outliers=True)
    codes, zeros, scales, packed = oracle_layer(d, bits, 0)
    qw = to_qweight(packed, zeros, scales, bits, 0, K)
    table = rng.uniform(0.01, 0.02, size=(3, N, 1)).astype(np.float32)
    ids = rng.integers(0, 3, size=8).astype(np.int32)
    ids[:2] = (2, 1)
    ref = oracle.fwd_multitask(d["X"][:8], packed, zeros, table, ids, bits, 0)
    tab = torch.from_numpy(table[:, :, 0].copy()).cuda()
    for M in (1, 2, 3, 8):
        Y = binding.qlinear_decode_multitask(qw, tab, torch.from_numpy(ids[:M]).cuda(), bf16_to_dev(d["X"][:M]))
        binding.check_status()
        assert_close(dev_to_f64(Y), ref[:M], f"M={M}")


@pytest.mark.parametrize("bits,g", [(3, 0), (4, 0), (3, 64), (4, 128), (3, 256)])
def test_tokens_of_any_magnitude(bits, g):
    """A token (in a call of one or two: a step of it) is brought to the range of its operands by a power of two of
    its own, so its result is as exact at 2^-90 as at 2^90 and with one element 2^12 times the others; a token of
    zeros gives zeros, one with an infinity or a NaN nothing finite, and neither touches its neighbours."""
    N, K, M = 264, 1536, 8
    d = synth.custom(5 + bits + g, N, K, M, bits, g, outliers=True)
    codes, zeros, scales, packed = oracle_layer(d, bits, g)
    qw = to_qweight(packed, zeros, scales, bits, g, K)
    prep = binding.decode_prepare(qw)
    X = synth.bf16_bits_to_f32(d["X"]).astype(np.float32)
    X[1] *= 2.0 ** -90
    X[2] *= 2.0 ** 90
    X[3, 700] = 4096.0
    X[4] = 0.0
    X[5, 3] = np.inf
    X[6, 1500] = np.nan
    Xb = synth.f32_to_bf16_bits(X)
    torch.cuda.synchronize()
    Xd, out = bf16_to_dev(Xb), []
    for at_once in (8, 2, 1):
        parts = [Xd[m:m + at_once].contiguous() for m in range(0, M, at_once)]
        out.append(torch.cat([binding.qlinear_decode_prepared(qw, prep, x) for x in parts]))
        if g != 64:
            out.append(torch.cat([binding.qlinear_decode(qw, x) for x in parts]))
    binding.check_status()
    ref = oracle.fwd(Xb[[0, 1, 2, 3, 7]], packed, zeros, scales, bits, g)
    for Y in out:
        got = dev_to_f64(Y)
        for i, m in enumerate((0, 1, 2, 3, 7)):
            assert_close(got[m] / np.abs(ref[i]).max(), ref[i] / np.abs(ref[i]).max(), f"token {m}")
        assert np.all(got[4] == 0.0)
        assert not np.any(np.isfinite(got[5])) and not np.any(np.isfinite(got[6]))


@pytest.mark.parametrize("K,bits,g", [(128, 3, 64), (640, 4, 64), (768, 3, 64), (1024, 4, 64), (384, 3, 128), (768, 4, 128),
                                      (1024, 3, 128)])
def test_scales_and_zero_points_off_a_vector(K, bits, g):
    """Rows whose groups are aligned vectors are read as such; a scale or zero-point array that starts one element
    off takes the other kernel, with the same bits."""
    N, M = 72, 16
    d = synth.custom(N + K + bits, N, K, M, bits, g, outliers=True)
    codes, zeros, scales, packed = oracle_layer(d, bits, g)
    qw = to_qweight(packed, zeros, scales, bits, g, K)
    prep = binding.decode_prepare(qw)
    G = K // g
    s_off = torch.zeros(N * G + 1, dtype=torch.float32, device="cuda")[1:].view(N, G).copy_(qw.scales)
    z_off = torch.zeros(N * G + 1, dtype=torch.uint8, device="cuda")[1:].view(N, G).copy_(qw.zeros)
    table = torch.stack([qw.scales, 2 * qw.scales])
    t_off = torch.zeros(2 * N * G + 1, dtype=torch.float32, device="cuda")[1:].view(2, N, G).copy_(table)
    ids = (torch.arange(M, device="cuda", dtype=torch.int32) % 2).contiguous()
    X = bf16_to_dev(d["X"])
    ref = oracle.fwd(d["X"], packed, zeros, scales, bits, g)
    for m in (1, 2, 7, 16):
        Y = binding.qlinear_decode_prepared(qw, prep, X[:m])
        Yt = binding.qlinear_decode_prepared(qw, prep, X[:m], scale_table=table, task_ids=ids[:m])
        assert_close(dev_to_f64(Y), ref[:m], f"M={m}")
        for s, z in ((s_off, qw.zeros), (qw.scales, z_off)):
            off = binding.QWeight(bits, N, K, g, qw.qweight, z, s)
            assert torch.equal(binding.qlinear_decode_prepared(off, prep, X[:m]), Y)
            assert torch.equal(binding.qlinear_decode_prepared(off, prep, X[:m], scale_table=t_off, task_ids=ids[:m]), Yt)
    binding.check_status()
