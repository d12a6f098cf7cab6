"""GPU parity of the cluster-split forward and dX (few tokens) at the edges of its token tiles, row
tiles, contraction stages and cluster splits, against the fp64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2305_14152_b200 import binding, synth
from gpu_util import assert_close, bf16_to_dev, dev_to_f64, oracle_layer, to_qweight

pytestmark = pytest.mark.gpu

# N, K: a single ragged row tile and one stage; three row tiles over eight CTAs; a contraction that
# ends in half a stage (4-bit, K % 128 == 64); one tile per cluster in all of them.
# dX of the first three has too little to split from 129 tokens on and runs in the pair kernel
SHAPES = [(8, 64, 4, 0), (264, 1088, 4, 32), (136, 2048, 3, 64), (1000, 640, 3, 0), (3080, 1152, 4, 128)]


@pytest.mark.parametrize("N,K,bits,g", SHAPES)
@pytest.mark.parametrize("T", [1, 16, 17, 129, 256, 257])
def test_token_and_row_edges(N, K, bits, g, T):
    d = synth.custom(N + T, N, K, T, bits, g)
    codes, zeros, scales, packed = oracle_layer(d, bits, g)
    qw = to_qweight(packed, zeros, scales, bits, g, K)
    X, dY = bf16_to_dev(d["X"]), bf16_to_dev(d["dY"])
    guard = torch.full((T * N + 512,), 7.0, dtype=torch.bfloat16, device="cuda")
    Y = guard[256:256 + T * N].view(T, N)
    binding.qlinear_fwd(qw, X, Y)
    guard_x = torch.full((T * K + 512,), 7.0, dtype=torch.bfloat16, device="cuda")
    dX = guard_x[256:256 + T * K].view(T, K)
    binding.qlinear_bwd(qw, None, dY, dX=dX, need_ds=False)
    zf = qw.zeros.float() + 0.3
    Yz = binding.qlinear_fwd_zf(qw, zf, X)
    dXz, _, _ = binding.qlinear_bwd_zf(qw, zf, None, dY, need_grads=False)
    again = binding.qlinear_fwd(qw, X)
    binding.check_status()
    for gb in (guard, guard_x):
        assert torch.all(gb[:256] == 7.0) and torch.all(gb[-256:] == 7.0), "a kernel wrote outside its output"
    assert torch.equal(Y, again)
    z64 = dev_to_f64(zf).astype("float32")
    assert_close(dev_to_f64(Y), oracle.fwd(d["X"], packed, zeros, scales, bits, g), "Y")
    assert_close(dev_to_f64(dX), oracle.bwd_dx(d["dY"], packed, zeros, scales, K, bits, g), "dX")
    assert_close(dev_to_f64(Yz), oracle.fwd_zf(d["X"], packed, z64, scales, bits, g), "Y, real zero-point")
    assert_close(dev_to_f64(dXz), oracle.bwd_dx_zf(d["dY"], packed, z64, scales, K, bits, g), "dX, real zero-point")


# Three tiles over four CTAs of a cluster on 148 SMs, so that a CTA works on the end of one tile and the
# beginning of the next; the last cluster has two.  The forward splits the first shape so, dX the second.
@pytest.mark.parametrize("N,K", [(11008, 4096), (4096, 11008)])
@pytest.mark.parametrize("bits,g", [(4, 128), (3, 64), (4, 0)])
def test_several_tiles_per_cluster(N, K, bits, g):
    T = 77
    rng = np.random.default_rng(N + bits + g)
    G = K // g if g else 1
    packed = rng.integers(0, 1 << 32, size=(N, K * bits // 32), dtype=np.uint32)
    zeros = rng.integers(0, 1 << bits, size=(N, G), dtype=np.uint8)
    scales = rng.uniform(0.01, 0.02, size=(N, G)).astype(np.float32)
    zf = (zeros + rng.uniform(-0.5, 0.5, size=zeros.shape)).astype(np.float32)
    Xb = synth.f32_to_bf16_bits(rng.standard_normal((T, K)).astype(np.float32))
    dYb = synth.f32_to_bf16_bits(rng.standard_normal((T, N)).astype(np.float32))
    qw, zd = to_qweight(packed, zeros, scales, bits, g, K), torch.from_numpy(zf).cuda()
    X, dY = bf16_to_dev(Xb), bf16_to_dev(dYb)
    Y, Yz = binding.qlinear_fwd(qw, X), binding.qlinear_fwd_zf(qw, zd, X)
    dX = binding.qlinear_bwd(qw, None, dY, need_ds=False)[0]
    dXz = binding.qlinear_bwd_zf(qw, zd, None, dY, need_grads=False)[0]
    binding.check_status()
    toks = np.array([0, 1, 31, 32, 64, T - 1])
    assert_close(dev_to_f64(Y)[toks], oracle.fwd(Xb, packed, zeros, scales, bits, g, tokens=toks), "Y")
    assert_close(dev_to_f64(Yz)[toks], oracle.fwd_zf(Xb, packed, zf, scales, bits, g, tokens=toks), "Y, real zero-point")
    assert_close(dev_to_f64(dX)[toks], oracle.bwd_dx(dYb, packed, zeros, scales, K, bits, g, tokens=toks), "dX")
    assert_close(dev_to_f64(dXz)[toks], oracle.bwd_dx_zf(dYb, packed, zf, scales, K, bits, g, tokens=toks),
                 "dX, real zero-point")
