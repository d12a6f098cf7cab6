"""The ring of the streaming decode: four producer warps fill its slots, each step is read by one of sixteen warps, and
a wait on a barrier tells a turn from the one before it by parity alone.  The protocol runs here as a model (phases,
parities, copies that land late, warps in any order): with as many pairs of barriers as the kernel takes no
warp reads a step that has not landed, no copy meets a step that has not been read, and nobody is stuck; with a pair
per slot, which a wait cannot tell apart as soon as a block has more steps than the ring slots, all three happen."""
import os
import random
import re

import numpy as np
import pytest
import torch

import oracle
from paper_2305_14152_b200 import binding, synth
from gpu_util import assert_close, bf16_to_dev, dev_to_f64, kernels_of

SOURCE = os.path.join(os.path.dirname(os.path.abspath(binding.__file__)), "csrc", "decode_stream.cu")
PRODUCERS, READERS = 4, 16


def stream_bars(steps, nchunks, slots):
    return min(steps, nchunks + max(slots, 4))


def run_ring(nchunks, blocks, slots, bars, rng):
    """What goes wrong in one run: None, or the first violation."""
    steps = nchunks * blocks
    full, empty = [0] * bars, [0] * bars                    # completed phases
    passed = lambda phases, turn: (phases & 1) != (turn & 1)
    holds, landed, read = [None] * slots, set(), set()
    flying = []
    producers = [q for q in range(PRODUCERS)]               # next step of each
    block = 0
    todo = {w: list(range(w, nchunks, READERS)) for w in range(READERS)}
    slow = rng.choice(list(range(READERS)) + [None])         # a warp that hardly ever gets its turn
    late = rng.choice([0.02, 0.3, 1.0])                      # how readily copies land
    idle = 0
    while block < blocks:
        moved = False
        actors = [("p", q) for q in range(PRODUCERS)] + [("r", w) for w in range(READERS)] + [("c", 0)]
        rng.shuffle(actors)
        for kind, i in actors:
            if kind == "p":
                s = producers[i]
                if s >= steps:
                    continue
                if s >= slots:
                    t = s - slots
                    if not passed(empty[t % bars], t // bars):
                        continue
                    if t not in read:
                        return f"step {s} copied over step {t}"
                holds[s % slots] = s
                flying.append(s)
                producers[i] += PRODUCERS
                moved = True
            elif kind == "c":
                for s in [s for s in flying if rng.random() < late]:
                    flying.remove(s)
                    landed.add(s)
                    full[s % bars] += 1
                moved = moved or bool(flying)
            elif todo[i]:
                if i == slow and rng.random() < 0.95:
                    moved = True
                    continue
                s = block * nchunks + todo[i][0]
                if not passed(full[s % bars], s // bars):
                    continue
                if s not in landed or holds[s % slots] != s:
                    return f"step {s} read before it landed"
                read.add(s)
                empty[s % bars] += 1
                todo[i].pop(0)
                moved = True
        if not any(todo.values()):                          # the named barrier at the end of a block
            block += 1
            todo = {w: list(range(w, nchunks, READERS)) for w in range(READERS)}
            moved = True
        idle = 0 if moved else idle + 1
        if idle > 50:
            return "stuck"
    return None


# (steps of a block, blocks, slots): a block of more steps than slots, of as many, of fewer, a single block
RINGS = [(16, 5, 15), (43, 5, 13), (41, 1, 17), (9, 4, 9), (7, 5, 8), (10, 1, 10), (64, 2, 8), (3, 6, 11), (22, 3, 32)]


@pytest.mark.parametrize("nchunks,blocks,slots", RINGS)
def test_the_kernel_s_barriers_tell_all_turns_apart(nchunks, blocks, slots):
    bars = stream_bars(nchunks * blocks, nchunks, slots)
    for seed in range(60):
        assert run_ring(nchunks, blocks, slots, bars, random.Random(seed)) is None


def test_a_pair_per_slot_does_not():
    assert any(run_ring(43, 5, 13, 13, random.Random(seed)) for seed in range(60))


def test_the_kernel_takes_that_many():
    text = open(SOURCE).read()
    assert "const int n = nchunks + (slots > 4 ? slots : 4);" in text and "return n < steps ? n : steps;" in text
    used = re.findall(r"\b(?:full|empty)\[([^\]]*)\]\)", text)
    assert len(used) == 6 and set(used) == {"q", "(s - p.slots) % p.bars", "s < p.bars ? s : s % p.bars", "bar"}, used


@pytest.mark.gpu
@pytest.mark.parametrize("N,K,bits,g,M", [(22016, 8192, 4, 512, 2), (4104, 8192, 4, 512, 4), (5128, 22016, 4, 512, 1),
                                          (2056, 22016, 3, 11008, 1), (5128, 7680, 3, 384, 4), (1032, 16384, 4, 1024, 2)])
def test_rows_of_more_steps_than_slots(N, K, bits, g, M):
    w = binding.quantize_rtn(torch.randn((N, K), device="cuda", generator=torch.Generator(device="cuda").manual_seed(N)), bits, g)
    X = synth.f32_to_bf16_bits(np.random.default_rng(K).standard_normal((M, K)).astype(np.float32))
    Xd = bf16_to_dev(X)
    names = kernels_of(lambda: binding.qlinear_decode(w, Xd))
    assert names and all("decode_stream_kernel" in name for name in names), names
    Y = binding.qlinear_decode(w, Xd)
    for _ in range(20):
        assert torch.equal(binding.qlinear_decode(w, Xd), Y)
    binding.check_status()
    packed, zeros, scales = (t.cpu().numpy() for t in (w.qweight, w.zeros, w.scales))
    rows = np.arange(0, N, 7)
    ref = oracle.fwd(X, np.ascontiguousarray(packed[rows]).view(np.uint32), np.ascontiguousarray(zeros[rows]),
                     np.ascontiguousarray(scales[rows]), bits, g)
    assert_close(dev_to_f64(Y)[:, rows], ref, "Y")
