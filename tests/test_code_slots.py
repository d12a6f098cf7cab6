"""Shared-memory slots that a copy engine fills with packed codes and threads read: the hand-back for
the next copy.  Threads read through the generic proxy, copies write through the async proxy, and an
mbarrier orders threads but not proxies: a proxy fence has to stand between the reads and the arrive
(or the copy itself).  A refill that lands first is rare and leaves no trace but a wrong sum, so the
order is checked in the sources, and on the GPU by many repetitions with the codes in L2."""
import glob
import os
import re

import numpy as np
import pytest
import torch

import oracle
from paper_2305_14152_b200 import binding, synth
from gpu_util import assert_close, bf16_to_dev, dev_to_f64, oracle_layer, to_qweight

CSRC = os.path.join(os.path.dirname(os.path.abspath(binding.__file__)), "csrc")

# a hand-back, or (prepared decode) the refill of the slot just read
HANDBACK = re.compile(r"mbar_arrive\(.*(pk_empty|empty_pk)\[")
REFILL = re.compile(r"if \(lane == 0\) issue_next\(\);")


def test_a_proxy_fence_stands_before_every_hand_back():
    found = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        lines = open(path).read().splitlines()
        for i, line in enumerate(lines):
            if not (HANDBACK.search(line) or REFILL.search(line)):
                continue
            found += 1
            before = "\n".join(lines[max(0, i - 6):i])
            assert re.search(r"fence_proxy_async_smem\(\);.*\n(.*\n)*?\s*__syncwarp\(\);", before), f"{path}:{i + 1}: {line.strip()}"
    assert found >= 5      # forward, dX, dS, few tokens, prepared decode


@pytest.mark.gpu
@pytest.mark.parametrize("bits,g", [(3, 64), (4, 0)])
def test_contractions_repeat_exactly(bits, g):
    # 64 stages per tile, one tile for most CTA pairs, codes (6 or 8 MiB) in L2
    N = K = 4096
    T = 2048
    d = synth.custom(41 + bits, N, K, T, bits, g, outliers=True, sigma_dy=1e-2)
    codes, zeros, scales, packed = oracle_layer(d, bits, g)
    qw = to_qweight(packed, zeros, scales, bits, g, K)
    zf = qw.zeros.float() + 0.25
    X, dY = bf16_to_dev(d["X"]), bf16_to_dev(d["dY"])

    def once():
        dXz = binding.qlinear_bwd_zf(qw, zf, None, dY, need_grads=False)[0]
        return (binding.qlinear_fwd(qw, X), *binding.qlinear_bwd(qw, X, dY), binding.qlinear_fwd_zf(qw, zf, X), dXz)

    first = once()
    for _ in range(20):
        for a, b in zip(first, once()):
            assert torch.equal(a, b)
    binding.check_status()
    toks, rows = np.arange(0, T, 311), np.arange(0, N, 331)
    assert_close(dev_to_f64(first[0])[toks], oracle.fwd(d["X"], packed, zeros, scales, bits, g, tokens=toks), "Y")
    assert_close(dev_to_f64(first[1])[toks], oracle.bwd_dx(d["dY"], packed, zeros, scales, K, bits, g, tokens=toks), "dX")
    assert_close(dev_to_f64(first[2])[rows], oracle.bwd_ds(d["X"], d["dY"], packed, zeros, bits, g, rows=rows), "dS")


@pytest.mark.gpu
@pytest.mark.parametrize("bits,g", [(3, 64), (4, 0), (3, 0), (4, 128), (4, 32)])
def test_decodes_repeat_exactly(bits, g):
    N = K = 4096
    d = synth.custom(43 + bits + g, N, K, 16, bits, g, outliers=True)
    codes, zeros, scales, packed = oracle_layer(d, bits, g)
    qw = to_qweight(packed, zeros, scales, bits, g, K)
    prep = binding.decode_prepare(qw) if g != 32 else None
    torch.cuda.synchronize()
    ref = oracle.fwd(d["X"], packed, zeros, scales, bits, g)
    for M in (1, 4, 8, 16):
        X = bf16_to_dev(d["X"][:M])

        def once():
            out = [binding.qlinear_decode(qw, X), binding.qlinear_fwd(qw, X)]
            return out if prep is None else out + [binding.qlinear_decode_prepared(qw, prep, X)]

        first = once()
        for _ in range(50):
            for a, b in zip(first, once()):
                assert torch.equal(a, b)
        binding.check_status()
        for Y in first:
            assert_close(dev_to_f64(Y), ref[:M], f"M={M}")
