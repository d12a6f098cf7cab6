"""GPU parity of the CTA-pair forward and dX at the edges of their 512-token x 256-output tiles, on shapes
that the cluster-split kernel does not take: a channel (column) tile of 8 or 64, a token tile of 10
tokens, one of 266 (a whole first token block, 10 tokens in the second), a contraction that ends in half a
128-column piece, groups narrower than a stage, wider, and such that a stage begins inside one; integer and
real-valued zero-points."""
import numpy as np
import pytest
import torch

import oracle
from paper_2305_14152_b200 import binding, synth
from gpu_util import assert_close, bf16_to_dev, dev_to_f64, oracle_layer, to_qweight

pytestmark = pytest.mark.gpu

SCALES = [(4, 32), (3, 64), (3, 192), (4, 0), (3, 0)]


def _kernels_of(call):
    """Names of the kernels a call launches."""
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
        call()
        torch.cuda.synchronize()
    return [e.name for e in prof.events() if "kernel" in e.name]


def _layer(seed, N, K, T, bits, g):
    d = synth.custom(seed, N, K, T, bits, g, outliers=True, sigma_dy=1e-2)
    codes, zeros, scales, packed = oracle_layer(d, bits, g)
    zf = (zeros + np.random.default_rng(seed).uniform(-1.3, 1.3, size=zeros.shape)).astype(np.float32)
    toks = np.unique(np.concatenate([[0, 127, 128, 255, 256, 511, 512], np.arange(2040, 2056), np.arange(T - 12, T)]))
    return d, zeros, scales, packed, zf, to_qweight(packed, zeros, scales, bits, g, K), toks


def _guarded(rows, cols):
    flat = torch.full((rows * cols + 512,), 7.0, dtype=torch.bfloat16, device="cuda")
    return flat, flat[256:256 + rows * cols].view(rows, cols)


@pytest.mark.parametrize("T", [2058, 2314])
@pytest.mark.parametrize("bits,g", SCALES)
def test_forward_edges(bits, g, T):
    N, K = 2056, 1088 if g == 32 else 1152
    d, zeros, scales, packed, zf, qw, toks = _layer(61 + g + T, N, K, T, bits, g)
    X, zd = bf16_to_dev(d["X"]), torch.from_numpy(zf).cuda()
    flat, Y = _guarded(T, N)
    names = _kernels_of(lambda: binding.qlinear_fwd(qw, X, Y))
    assert len(names) == 1 and "qfwd_pair_kernel" in names[0], names
    Yz = binding.qlinear_fwd_zf(qw, zd, X)
    binding.check_status()
    assert torch.all(flat[:256] == 7.0) and torch.all(flat[-256:] == 7.0), "wrote outside its output"
    assert_close(dev_to_f64(Y)[toks], oracle.fwd(d["X"], packed, zeros, scales, bits, g, tokens=toks), "Y")
    assert_close(dev_to_f64(Yz)[toks], oracle.fwd_zf(d["X"], packed, zf, scales, bits, g, tokens=toks), "Y, real zero-point")


@pytest.mark.parametrize("T", [2058, 2314])
@pytest.mark.parametrize("bits,g", SCALES)
def test_dx_edges(bits, g, T):
    N, K = 1160, 2112 if g == 32 else 2304 if g == 192 else 2176
    d, zeros, scales, packed, zf, qw, toks = _layer(67 + g + T, N, K, T, bits, g)
    dY, zd = bf16_to_dev(d["dY"]), torch.from_numpy(zf).cuda()
    flat, dX = _guarded(T, K)
    names = _kernels_of(lambda: binding.qlinear_bwd(qw, None, dY, dX=dX, need_ds=False))
    assert len(names) == 1 and "qdx_pair_kernel" in names[0], names
    dXz = binding.qlinear_bwd_zf(qw, zd, None, dY, need_grads=False)[0]
    binding.check_status()
    assert torch.all(flat[:256] == 7.0) and torch.all(flat[-256:] == 7.0), "wrote outside its output"
    assert_close(dev_to_f64(dX)[toks], oracle.bwd_dx(d["dY"], packed, zeros, scales, K, bits, g, tokens=toks), "dX")
    assert_close(dev_to_f64(dXz)[toks], oracle.bwd_dx_zf(d["dY"], packed, zf, scales, K, bits, g, tokens=toks),
                 "dX, real zero-point")


def test_calls_go_to_the_faster_kernel():
    """One measured call on either side of each rule, in us: forward 10.3 in the pair kernel / 15.1 in the
    cluster-split one, 133 / 99; dX 25.7 / 39.8, 215 / 93; canonical decode of nine tokens 14.6 in its own
    kernel / 16.5 in the cluster-split one, 90 / 60."""
    def layer(N, K, bits, g):
        w = torch.randn((N, K), device="cuda")
        return binding.quantize_rtn(w, bits, g)

    def act(T, cols):
        return torch.randn((T, cols), device="cuda").to(torch.bfloat16)

    for N, K, T, bits, g, name in [(2360, 256, 1134, 3, 128, "qfwd_pair_kernel"), (4096, 11008, 1001, 3, 128, "qsplit_kernel")]:
        w, X = layer(N, K, bits, g), act(T, K)
        assert name in _kernels_of(lambda: binding.qlinear_fwd(w, X))[0]
    for N, K, T, bits, g, name in [(1656, 3328, 977, 4, 128, "qdx_pair_kernel"), (22016, 8192, 256, 3, 64, "qsplit_kernel")]:
        w, dY = layer(N, K, bits, g), act(T, N)
        assert name in _kernels_of(lambda: binding.qlinear_bwd(w, None, dY, need_ds=False))[0]
    for N, K, bits, name in [(4096, 8192, 3, "decode_kernel"), (8192, 22016, 3, "qsplit_kernel")]:
        w, X = layer(N, K, bits, 0), act(9, K)
        assert name in _kernels_of(lambda: binding.qlinear_decode(w, X))[0]
    binding.check_status()
