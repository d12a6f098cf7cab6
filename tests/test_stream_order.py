"""Kernels that are launched programmatically begin before the kernel in front of them in the stream has ended, and see
its results behind griddepcontrol.wait.  A read through the non-coherent path (__ldg, ld.global.nc, or a const __restrict__
parameter that the compiler takes for one) promises data that nobody writes while the kernel lives, which does not hold
for anything an earlier kernel may have written.  No value shows that reliably, so the sources are checked; on the
GPU chains of calls that read what the call before has written give what the same calls give one at a time."""
import glob
import os
import re

import pytest
import torch

from paper_2305_14152_b200 import binding

CSRC = os.path.join(os.path.dirname(os.path.abspath(binding.__file__)), "csrc")
NON_COHERENT = re.compile(r"\b__ldg\(|ld\.global\.nc|\bconst\b[^,()]*\*\s*(const\s+)?__restrict__")


def test_programmatic_kernels_read_coherently():
    waiting = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        kernels = re.split(r"(?=\b__global__\b)", text)
        helpers, kernels = kernels[0], kernels[1:]
        programmatic = [k for k in kernels if "griddepcontrol.wait" in k]
        waiting += len(programmatic)
        for k in programmatic:
            found = NON_COHERENT.search(k)
            assert found is None, f"{os.path.basename(path)}: {k.split('(')[0].split()[-1]}: {found.group()}"
        if programmatic and len(programmatic) == len(kernels):     # then the device functions before are theirs
            assert NON_COHERENT.search(helpers) is None, os.path.basename(path)
    assert waiting >= 9                  # forward, dX, dS, the fallback, few tokens, decode, three reductions, AdamW


def test_kernels_side_by_side_hand_over_what_came_before():
    """A kernel that begins without the wait (`beside`) acquires what the one that let it in has released.  Hardware
    that happens to order both shows no difference, so the sources are checked."""
    helpers = open(os.path.join(CSRC, "sm100_ptx.cuh")).read()
    body = lambda name: re.search(r"void %s\(bool \w+\) \{(.*?)\n\}" % name, helpers, re.S).group(1)
    begins, lets_in = body("begin_beside"), body("let_next_in")
    assert 0 < begins.index("if (beside)") < begins.index("fence.acq_rel.gpu") < begins.index("fence.proxy.async.global")
    assert 0 < lets_in.index("if (followed)") < lets_in.index("fence.acq_rel.gpu") < lets_in.index("griddepcontrol.launch_dependents")
    beside = first = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for k in re.split(r"(?=\b__global__\b)", text)[1:]:
            k = k[:k.index("\n}\n")]                               # the kernel, without what follows it
            wait = 'asm volatile("griddepcontrol.wait;" ::: "memory");\n  let_next_in(p.side == kFollowed);'
            if "kBeside" in k:
                beside += 1
                assert k.index("begin_beside(beside);") < k.index("__syncthreads()") < k.index("if (!beside) " + wait)
                assert len(re.findall(r"const bool beside = (TRANS && )?p\.side == kBeside;\s+begin_beside\(beside\);", k)) == k.count("kBeside") == 1
                assert "launch_dependents" not in k
            elif "kFollowed" in k:
                first += 1
                assert "\n  " + wait in k and "launch_dependents" not in k
    assert beside == 3 and first == 1          # dX, dS and the kernel of few tokens; the forward


def _weight(N, K, bits, g, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    w = binding.quantize_rtn(torch.randn((N, K), generator=gen, device="cuda"), bits, g)
    w.scales.mul_(1.0 / (K ** 0.5))                                # outputs of the size of the inputs
    return w


@pytest.mark.gpu
@pytest.mark.parametrize("bits,g", [(4, 0), (3, 64), (4, 128)])
@pytest.mark.parametrize("M", [1, 2, 3, 8])
def test_a_call_reads_what_the_call_before_has_written(bits, g, M):
    """Each call's Y is the next one's X, and all buffers are written again in every pass."""
    K, depth, passes = 1024, 8, 30
    ws = [_weight(K, K, bits, g, i) for i in range(depth)]
    preps = [binding.decode_prepare(w) for w in ws]
    gen = torch.Generator(device="cuda").manual_seed(M)
    starts = torch.randn((passes, M, K), generator=gen, device="cuda").to(torch.bfloat16)
    bufs = [torch.zeros((M, K), dtype=torch.bfloat16, device="cuda") for _ in range(2 * depth + 1)]
    torch.cuda.synchronize()

    def chain(start, between):
        bufs[0].copy_(start)
        for i, (w, p) in enumerate(zip(ws, preps)):
            binding.qlinear_decode_prepared(w, p, bufs[i], bufs[i + 1])
            between()
        for i, w in enumerate(ws):
            binding.qlinear_decode(w, bufs[depth + i], bufs[depth + i + 1])
            between()
        return bufs[-1].clone()

    together = [chain(s, lambda: None) for s in starts]
    apart = [chain(s, torch.cuda.synchronize) for s in starts]
    binding.check_status()
    for a, b in zip(together, apart):
        assert torch.isfinite(a).all() and torch.equal(a, b)


@pytest.mark.gpu
@pytest.mark.parametrize("T", [40, 1024])
def test_steps_read_the_scales_of_the_step_before(T):
    """Forward, gradients and AdamW in one stream: every forward sees the scales the step before has left."""
    N, K = 1024, 1024
    gen = torch.Generator(device="cuda").manual_seed(T)
    X, dY = (torch.randn((T, c), generator=gen, device="cuda").to(torch.bfloat16) for c in (K, N))

    def run(between):
        w = _weight(N, K, 4, 0, 3)
        m, v = torch.zeros_like(w.scales), torch.zeros_like(w.scales)
        ws, out = binding.alloc_workspace(binding.OP_BWD, T, w), []
        for step in range(1, 21):
            out.append(binding.qlinear_fwd(w, X))
            between()
            dX, dS = binding.qlinear_bwd(w, X, dY, workspace=ws)
            between()
            binding.scale_adamw(w.scales, dS, m, v, 1e-2, step=step)
            between()
            out += [dX, dS]
        return out + [w.scales, m, v]

    together, apart = run(lambda: None), run(torch.cuda.synchronize)
    binding.check_status()
    for a, b in zip(together, apart):
        assert torch.equal(a, b)
