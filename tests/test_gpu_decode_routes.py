"""The canonical decode by rows, through the kernel of the prepared decode: every form that is dispatched there, on
shapes that are (the kernel's name is asserted, so that a change of the rule cannot empty these tests), and no
form compiled that is not."""
import os
import re
import subprocess

import numpy as np
import pytest
import torch

import oracle
from paper_2305_14152_b200 import binding, build, synth
from gpu_util import assert_close, bf16_to_dev, dev_to_f64, kernels_of, oracle_layer, to_qweight


def test_canonical_instances_have_one_token_tile():
    build.build()
    symbols = subprocess.run(["nm", "-C", binding.LIB_PATH], capture_output=True, text=True, check=True).stdout
    found = {tuple(m.split(", ")) for m in re.findall(r"decode_prep_kernel<([^>]*)>", symbols)}
    assert {a[4] for a in found} == {"true", "false"}                    # CANON
    for bits, tiles, gsh, tasks, canon, i8, vec in found:
        assert canon == "false" or (tiles == "1" and tasks == "false"), "more than eight tokens go elsewhere"
        assert i8 == "false" or tiles == "1"


def _rows_kernel(name):
    """decode_prep_kernel<bits, 1, gsh, tasks, CANON = true, i8, vec>, mangled."""
    return re.search(r"decode_prep_kernelILi[34]ELi1ELi\dELb0ELb1E", name) is not None


# one row group; half pairs; rows that end inside a step; few rows and long ones; more than 32 rows per CTA
SHAPES = [(8, 256, 3, 128), (8, 512, 4, 256), (8, 5632, 3, 0), (8, 5632, 4, 0), (264, 5760, 4, 0), (264, 22016, 3, 0),
          (200, 1408, 3, 128), (1032, 1280, 3, 256), (4104, 4224, 4, 128), (5128, 1024, 3, 0), (5128, 1152, 4, 0)]


@pytest.mark.gpu
@pytest.mark.parametrize("N,K,bits,g", SHAPES)
def test_canonical_rows(N, K, bits, g):
    d = synth.custom(N + K, N, K, 8, bits, g, outliers=True)
    codes, zeros, scales, packed = oracle_layer(d, bits, g)
    qw = to_qweight(packed, zeros, scales, bits, g, K)
    ref = oracle.fwd(d["X"], packed, zeros, scales, bits, g)
    for M in (1, 2, 3, 5, 8):
        guard = torch.full((M * N + 512,), 7.0, dtype=torch.bfloat16, device="cuda")
        Y = guard[256:256 + M * N].view(M, N)
        X = bf16_to_dev(d["X"][:M])
        names = kernels_of(lambda: binding.qlinear_decode(qw, X, Y))
        assert len(names) == 1 and _rows_kernel(names[0]), names
        again = binding.qlinear_decode(qw, X)
        binding.check_status()
        assert torch.all(guard[:256] == 7.0) and torch.all(guard[-256:] == 7.0), "wrote outside its output"
        assert torch.equal(Y, again)
        assert_close(dev_to_f64(Y), ref[:M], f"M={M}")


@pytest.mark.gpu
@pytest.mark.parametrize("bits", [3, 4])
@pytest.mark.parametrize("N,K,most", [(264, 5632, 5), (5128, 1024, 8)])
def test_canonical_rows_with_the_scales_of_a_task(N, K, most, bits):
    d = synth.custom(N + bits, N, K, 8, bits, 0, outliers=True)
    codes, zeros, scales, packed = oracle_layer(d, bits, 0)
    rng = np.random.default_rng(N)
    table = (scales[:, 0][None, :] * rng.uniform(0.5, 2.0, size=(3, N))).astype(np.float32)
    qw, tab = to_qweight(packed, zeros, scales, bits, 0, K), torch.from_numpy(table).cuda()
    for M in [m for m in (1, 2, 5, 8) if m <= most]:              # (the call refuses more activations than that)
        ids = rng.integers(0, 3, size=M).astype(np.int32)
        ids[-1] = 2
        beyond = np.where(ids == 2, 7, ids).astype(np.int32)              # clamped to the last row
        X = bf16_to_dev(d["X"][:M])

        def call(ids):
            return binding.qlinear_decode_multitask(qw, tab, torch.from_numpy(ids).cuda(), X)

        dev = torch.from_numpy(ids).cuda()
        names = kernels_of(lambda: binding.qlinear_decode_multitask(qw, tab, dev, X))
        assert len(names) == 1 and _rows_kernel(names[0]), names
        Y = call(ids)
        binding.check_status()
        assert_close(dev_to_f64(Y), oracle.fwd_multitask(d["X"][:M], packed, zeros, table, ids, bits), f"M={M}")
        assert torch.equal(call(beyond), Y)


@pytest.mark.gpu
@pytest.mark.parametrize("bits,g", [(3, 0), (4, 0), (3, 128), (4, 256)])
def test_tokens_of_any_magnitude_by_rows(bits, g):
    """As test_gpu_decode_rows.py has it for the prepared decode, where the canonical one goes by rows too: magnitudes
    from 2^-90 to 2^90, one element 2^20 times the others (of three-bit codes' activations, for which the operands keep the
    fewest bits, those 2^18 and more below the largest of a step or 2^25 below that of a token lose some), zeros, an
    infinity and a NaN beside other tokens."""
    N, K, M = 264, 5632, 8
    d = synth.custom(15 + bits + g, N, K, M, bits, g, outliers=True)
    codes, zeros, scales, packed = oracle_layer(d, bits, g)
    qw = to_qweight(packed, zeros, scales, bits, g, K)
    prep = binding.decode_prepare(qw)
    X = synth.bf16_bits_to_f32(d["X"]).astype(np.float32)
    X[1] *= 2.0 ** -90
    X[2] *= 2.0 ** 90
    X[3, 700] = 2.0 ** 20
    X[4] = 0.0
    X[5, 3] = np.inf
    X[6, 5500] = np.nan
    Xb = synth.f32_to_bf16_bits(X)
    Xd = bf16_to_dev(Xb)
    ref = oracle.fwd(Xb[[0, 1, 2, 3, 7]], packed, zeros, scales, bits, g)
    for at_once in (8, 2, 1):
        parts = [Xd[m:m + at_once].contiguous() for m in range(0, M, at_once)]
        for name in kernels_of(lambda: [binding.qlinear_decode(qw, x) for x in parts]):
            assert _rows_kernel(name), name
        for call in (lambda x: binding.qlinear_decode(qw, x), lambda x: binding.qlinear_decode_prepared(qw, prep, x)):
            got = dev_to_f64(torch.cat([call(x) for x in parts]))
            for i, m in enumerate((0, 1, 2, 3, 7)):
                assert_close(got[m] / np.abs(ref[i]).max(), ref[i] / np.abs(ref[i]).max(), f"token {m}")
            assert np.all(got[4] == 0.0)
            assert not np.any(np.isfinite(got[5])) and not np.any(np.isfinite(got[6]))
    binding.check_status()
