"""Bounded waits of whole warps.  Every wait gives up after a while, lane by lane; a lane that left on its own
would be missed by the warp-wide instructions behind the wait (shuffles, tensor-memory loads, __syncwarp),
which have no bound.  So mbar_wait / mbar_wait_cluster are for a single lane, and a warp that goes on together waits
through warp_wait / warp_wait_cluster, whose lanes agree on the outcome, or notes the outcome and goes on all the same.  A time-out that only some lanes see cannot be
provoked from outside, so the sources are checked."""
import glob
import os
import re

import pytest
import torch

from paper_2305_14152_b200 import binding
from gpu_util import kernels_of

CSRC = os.path.join(os.path.dirname(os.path.abspath(binding.__file__)), "csrc")


def _waits(text):
    """(line, function, whether only lane 0 gets there, whether its outcome is noted and nothing more) of every wait."""
    text = re.sub(r"//[^\n]*", lambda m: " " * len(m.group()), text)
    heads, start = [], 0                                  # what stands before each open brace
    for m in re.finditer(r"[{};]|\b(?:mbar_wait|mbar_wait_cluster|warp_wait|warp_wait_cluster)\(", text):
        token = m.group()
        if token == "{":
            heads.append(text[start:m.start()])
        elif token == "}":
            heads.pop()
        elif token != ";":
            around = "".join(heads) + text[start:m.start()]
            statement = text[start:text.index(";", m.start()) + 1].strip()
            noted = re.fullmatch(r"(if \(!mbar_wait\(.*\)\) i_ch = p\.nchunks|\(void\)ptx::mbar_wait\(.*\));", statement, re.S) is not None
            yield text.count("\n", 0, m.start()) + 1, token[:-1], "lane == 0" in around, noted
            continue
        start = m.end()


def test_warps_leave_a_wait_together():
    alone, together = 0, 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        for line, name, single, noted in _waits(open(path).read()):
            assert name.startswith("mbar_wait") == (single or noted), f"{os.path.basename(path)}:{line}: {name}"
            alone += single
            together += not single
    assert alone >= 15 and together >= 18
    helper = open(os.path.join(CSRC, "sm100_ptx.cuh")).read()
    for name in ("mbar_wait", "mbar_wait_cluster"):
        assert f"__all_sync(0xffffffffu, {name}(bar, parity, abort_flag))" in helper


@pytest.mark.gpu
def test_a_starved_layer_step_times_out_and_the_next_is_correct():
    """One scale per channel: the epilogue of the pair forward hands scales round and folds dY over its lanes."""
    N, K, T = 4096, 4096, 4096
    gen = torch.Generator(device="cuda").manual_seed(9)
    new = lambda *shape: torch.randn(shape, generator=gen, device="cuda")
    w = binding.quantize_rtn(new(N, K), 4, 0)
    L = binding.LayerLinear(w=w, X=new(T, K).bfloat16(), dY=new(T, N).bfloat16(), Y=torch.empty((T, N), dtype=torch.bfloat16, device="cuda"),
                            dX=torch.empty((T, K), dtype=torch.bfloat16, device="cuda"), dS=torch.empty_like(w.scales),
                            workspace=binding.alloc_workspace(binding.OP_BWD, T, w))

    def step():
        binding.layer_train_step([L], apply_adamw=False)
        binding.check_status()
        return L.Y.clone(), L.dX.clone(), L.dS.clone()

    names = kernels_of(lambda: binding.layer_train_step([L], apply_adamw=False))
    assert any("qfwd_pair_kernel" in name for name in names), names
    first = step()
    binding.selftest_configure(wait_limit_us=1000, starve_forward=True)
    try:
        with pytest.raises(binding.PeqaError) as err:
            step()
        assert err.value.status == -8                     # PEQA_ERR_DEVICE_TIMEOUT
    finally:
        binding.selftest_configure()
    for a, b in zip(first, step()):
        assert torch.equal(a, b)
