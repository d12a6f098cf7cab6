"""Performance cases of the quantized-linear path, as a training or serving program calls it.

A case names one kind of work (``kind``) and its sizes.  ``layers`` is the list of linears of one
pass, written "NxK,NxK,..." (out_features x in_features); consecutive linears with a "+" between
them ("NxK+NxK") are fed the same activations, as q, k, v or gate and up are.  ``group`` 0 is one
scale per output channel.

  train      forward, dX, dS and the AdamW step on the scales of every linear, one call
  train_zp   one linear, scales and real-valued zero-points trained together
  prefill    forward of every linear (a prompt, an evaluation batch)
  decode     token generation for M sequences from the prepared weights
  multitask  the same, every sequence with the scales of its own task
  canonical  token generation straight from the packed weights (no second copy kept)
  quantize   round-to-nearest quantization and packing of fp32 weights
"""
import math

import torch

from paper_2305_14152_b200 import binding

LAYER_7B = "4096x4096+4096x4096+4096x4096,4096x4096,11008x4096+11008x4096,4096x11008"
MLP_7B = "11008x4096+11008x4096,4096x11008"
LAYER_65B = "8192x8192+8192x8192+8192x8192,8192x8192,22016x8192+22016x8192,8192x22016"

LR = 1e-5          # AdamW on the scales
TASKS = 4          # rows of a multi-task scale table


def _case(name, kind, layers, tokens, bits, group):
    return {"name": name, "kind": kind, "layers": layers, "tokens": tokens, "bits": bits, "group": group}


def listed():
    return [
        # the smallest call: one 256 x 256 layer, 64 tokens; launches and host work are all there is
        _case("train_toy", "train", "256x256", 64, 4, 0),
        # LLaMA-7B attention projection, groups of 128: one linear tuned on one 2048-token sequence
        _case("train_7b_attn", "train", "4096x4096", 2048, 3, 128),
        # LLaMA-7B MLP, one scale per channel (the paper's main setting), two 2048-token sequences
        _case("train_7b_mlp", "train", MLP_7B, 4096, 4, 0),
        # a whole LLaMA-65B decoder layer, groups of 64: the largest training step
        _case("train_65b_layer", "train", LAYER_65B, 4096, 3, 64),
        # zero-points trained beside the scales, a ragged batch of short instruction samples
        _case("train_zp_ragged", "train_zp", "4096x11008", 1001, 3, 128),
        # a short prompt through a LLaMA-7B layer
        _case("prefill_7b_short", "prefill", LAYER_7B, 77, 4, 128),
        # one sequence generated on a LLaMA-7B layer: the latency of a chat server
        _case("decode_7b_m1", "decode", LAYER_7B, 1, 4, 0),
        # one sequence on a LLaMA-65B layer with grouped scales: streams 3-bit weights
        _case("decode_65b_m1_g64", "decode", LAYER_65B, 1, 3, 64),
        # a full serving batch on a LLaMA-65B layer
        _case("decode_65b_m16", "decode", LAYER_65B, 16, 3, 0),
        # several users, each with the scales of their own task
        _case("multitask_7b_m7", "multitask", LAYER_7B, 7, 3, 128),
        # generation where no second copy of the weights is kept
        _case("canonical_7b_m3", "canonical", LAYER_7B, 3, 4, 128),
        # quantizing the MLP of a LLaMA-65B layer once, before tuning
        _case("quantize_65b_mlp", "quantize", "22016x8192,8192x22016", 1, 3, 64),
    ]


def _log_int(rng, lo, hi, step=1):
    """A multiple of `step` in [lo, hi], spread over the logarithm."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(max(int(round(v / step)), -(-lo // step)), hi // step) * step


def draw(rng):
    kind = rng.choice(["train", "train", "train", "train_zp", "prefill", "prefill", "decode", "decode", "decode",
                       "multitask", "canonical", "quantize"])
    bits = rng.choice([3, 4])
    group = rng.choice([0, 0, 64, 128])
    named = {LAYER_7B: 0.25, MLP_7B: 0.15, LAYER_65B: 0.2}
    layers, at = None, rng.random()
    for text, share in named.items():
        at -= share
        if at < 0:
            layers = text
            break
    if layers is None or kind in ("train_zp", "quantize"):
        # one linear of any size: rows in steps of 8, columns in steps of 128 (64 where a
        # contraction over many tokens allows it and no group is wider)
        few = kind in ("decode", "multitask", "canonical") or group == 128
        layers = "%dx%d" % (_log_int(rng, 256, 22016, 8), _log_int(rng, 256, 22016, 128 if few else 64))
    if kind in ("train", "train_zp"):
        tokens = _log_int(rng, 33, 4096)
    elif kind == "prefill":
        tokens = _log_int(rng, 17, 4096)
    elif kind == "quantize":
        tokens = 1
    else:
        tokens = rng.choice([1, 1, 2, 3, 4, 5, 6, 7, 8, 9, 11, 13, 16])
    return {"kind": kind, "layers": layers, "tokens": tokens, "bits": bits, "group": group}


def _linears(case):
    """[(N, K, index of the activations it reads)] of one pass."""
    out = []
    for shared, part in enumerate(case["layers"].split(",")):
        for shape in part.split("+"):
            n, k = shape.split("x")
            out.append((int(n), int(k), shared))
    return out


def _weight(gen, N, K):
    """fp32 weights with the heavy tail of trained transformers: 1 in 1000 entries is 20 times larger."""
    W = torch.randn((N, K), generator=gen, device="cuda") * 0.02
    tail = torch.rand((N, K), generator=gen, device="cuda") < 1e-3
    return torch.where(tail, W * 20.0, W)


def _bf16(gen, rows, cols, sigma=1.0):
    return (torch.randn((rows, cols), generator=gen, device="cuda") * sigma).to(torch.bfloat16)


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kind, T, bits, group = case["kind"], case["tokens"], case["bits"], case["group"]
    linears, state, acts = _linears(case), [], {}
    for N, K, shared in linears:
        W = _weight(gen, N, K)
        if kind == "quantize":
            out = binding.quantize_rtn(W, bits, group)
            state.append((W, out))
            continue
        if shared not in acts:
            acts[shared] = _bf16(gen, T, K)
        X = acts[shared]
        w = binding.quantize_rtn(W, bits, group)
        del W
        if kind == "train":
            state.append(binding.LayerLinear(
                w=w, X=X, dY=_bf16(gen, T, N, 1e-2),
                Y=torch.empty((T, N), dtype=torch.bfloat16, device="cuda"),
                dX=torch.empty((T, K), dtype=torch.bfloat16, device="cuda"),
                dS=torch.empty_like(w.scales), m=torch.zeros_like(w.scales), v=torch.zeros_like(w.scales),
                workspace=binding.alloc_workspace(binding.OP_BWD, T, w)))
        elif kind == "train_zp":
            # zero-points some way into training: off the integer grid
            zf = w.zeros.float() + 0.1 * torch.randn(w.zeros.shape, generator=gen, device="cuda")
            moments = [torch.zeros_like(w.scales) for _ in range(4)]
            state.append((w, zf, X, _bf16(gen, T, N, 1e-2), moments,
                          binding.alloc_workspace(binding.OP_BWD_DSDZ, T, w)))
        elif kind == "prefill":
            state.append((w, X))
        elif kind == "canonical":
            state.append((w, X, binding.alloc_workspace(binding.OP_DECODE, T, w)))
        else:
            prepared = binding.decode_prepare(w)
            table = ids = None
            if kind == "multitask":
                spread = 1.0 + 0.05 * torch.randn((TASKS,) + tuple(w.scales.shape), generator=gen, device="cuda")
                table = (w.scales * spread).contiguous()
                ids = torch.randint(0, TASKS, (T,), generator=gen, device="cuda", dtype=torch.int32)
            state.append((w, prepared, X, table, ids))
    return {"kind": kind, "items": state}


def run(state):
    kind, items = state["kind"], state["items"]
    if kind == "train":
        binding.layer_train_step(items, lr=LR, weight_decay=0.0, step=1)
        return [(L.Y, L.dX, L.dS, L.w.scales, L.m, L.v) for L in items]
    if kind == "train_zp":
        out = []
        for w, zf, X, dY, (ms, vs, mz, vz), workspace in items:
            Y = binding.qlinear_fwd_zf(w, zf, X)
            dX, dS, dZ = binding.qlinear_bwd_zf(w, zf, X, dY, workspace=workspace)
            binding.scale_adamw(w.scales, dS, ms, vs, LR)
            binding.zero_adamw(zf, dZ, mz, vz, LR)
            out.append((Y, dX, dS, dZ, w.scales, zf))
        return out
    if kind == "prefill":
        return [binding.qlinear_fwd(w, X) for w, X in items]
    if kind == "canonical":
        return [binding.qlinear_decode(w, X, workspace=workspace) for w, X, workspace in items]
    if kind == "quantize":
        for W, out in items:
            binding.quantize_rtn(W, out.bits, out.group_size, out=out)
        return [(out.qweight, out.zeros, out.scales) for _, out in items]
    return [binding.qlinear_decode_prepared(w, prepared, X, scale_table=table, task_ids=ids)
            for w, prepared, X, table, ids in items]


def _rtn64(W, bits, group):
    """Codes, zero-points and scales by Eq. 1: integer decisions, so taken in binary32, returned as
    binary64 tensors [N, G, g], [N, G, 1], [N, G, 1]."""
    N, K = W.shape
    g = K if group in (0, K) else group
    Wg = W.view(N, K // g, g)
    lo, hi = Wg.amin(2, keepdim=True), Wg.amax(2, keepdim=True)
    top = float(2 ** bits - 1)
    s = (hi - lo) / top
    s = torch.where(hi == lo, torch.ones_like(s), s)
    z = torch.clamp(torch.round(-lo / s), 0.0, top)
    q = torch.clamp(torch.round(Wg / s) + z, 0.0, top)
    return q.double(), z.double(), s.double()


def _adamw64(p, grad):
    """First AdamW step from zero moments, no decay: new value, m, v."""
    m, v = (1.0 - 0.9) * grad, (1.0 - 0.999) * grad * grad
    return p - LR * (m / (1.0 - 0.9)) / (torch.sqrt(v / (1.0 - 0.999)) + 1e-8), m, v


def exact(case, seed):
    """What run() returns after prepare(case, seed), in binary64; the draws follow prepare()'s order."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kind, T, bits, group = case["kind"], case["tokens"], case["bits"], case["group"]
    out, acts = [], {}
    for N, K, shared in _linears(case):
        W = _weight(gen, N, K)
        if kind == "quantize":
            q, z, s = _rtn64(W, bits, group)
            out.append((None, None, s.view(N, -1)))       # packed codes have no value in binary64
            continue
        if shared not in acts:
            acts[shared] = _bf16(gen, T, K)
        X = acts[shared].double()
        q, z, s = _rtn64(W, bits, group)
        del W
        if kind in ("train", "train_zp"):
            if kind == "train_zp":
                z = (z.float() + 0.1 * torch.randn((N, z.shape[1]), generator=gen, device="cuda").view(z.shape)).double()
            dY = _bf16(gen, T, N, 1e-2).double()
            q -= z
            W64 = (q * s).view(N, K)
            Y, dX = X @ W64.T, dY @ W64
            del W64
            dW = (dY.T @ X).view(q.shape)
            dS = (q * dW).sum(2)
            s2, m, v = _adamw64(s.view(N, -1), dS)
            if kind == "train":
                out.append((Y, dX, dS, s2, m, v))
            else:
                dZ = -s.view(N, -1) * dW.sum(2)
                out.append((Y, dX, dS, dZ, s2, _adamw64(z.view(N, -1), dZ)[0]))
            continue
        q -= z
        if kind != "multitask":
            out.append(X @ (q * s).view(N, K).T)
            continue
        s32 = s.float().view(N, -1)
        table = s32 * (1.0 + 0.05 * torch.randn((TASKS,) + tuple(s32.shape), generator=gen, device="cuda"))
        ids = torch.randint(0, TASKS, (T,), generator=gen, device="cuda", dtype=torch.int32)
        Y = torch.empty((T, N), dtype=torch.float64, device="cuda")
        for task in ids.unique().tolist():
            Y[ids == task] = X[ids == task] @ (q * table[task].double().view(s.shape)).view(N, K).T
        out.append(Y)
    return out


def work(case):
    kind, T, bits, group = case["kind"], case["tokens"], case["bits"], case["group"]
    byts = flops = 0
    seen = set()
    for N, K, shared in _linears(case):
        G = 1 if group in (0, K) else K // group
        Q, zs = N * K * bits // 8, 5 * N * G
        if kind == "quantize":
            byts += 4 * N * K + Q + zs
            flops += 4 * N * K
            continue
        x = 0 if shared in seen else 2 * T * K
        seen.add(shared)
        if kind in ("train", "train_zp"):
            # in: X, dY, Q, z, s, m, v; out: Y, dX, dS, s, m, v (twice the optimizer with zero-points)
            trained = 1 if kind == "train" else 2
            byts += x + 2 * T * N + Q + zs + 2 * T * N + 2 * T * K + trained * 24 * N * G
            # one scale per channel: its gradient is a dot product with the forward's sums
            # (sum_t dY * Y / s), not a third contraction, when one call has both in hand
            flops += (4 if kind == "train" and G == 1 else 6) * T * N * K
        else:
            tasks = min(TASKS, T) if kind == "multitask" else 1
            byts += x + Q + N * G * (1 + 4 * tasks) + 2 * T * N
            flops += 2 * T * N * K
    return {"bytes": byts, "flops": flops}


def tolerance(case):
    if case["kind"] == "quantize":
        return "exact"        # codes, zero-points and scales are IEEE binary32 decisions
    # Measured against binary64 on the same inputs: bf16 results are off by 1.7e-3 (rounding of the
    # result alone) to 2.8e-3 (scales folded into bf16 operands), the largest element by 2.6e-2;
    # gradients of the scales by 4e-6.  Two correct implementations differ by up to twice that.
    return {"rel": 6e-3, "max": 6e-2}
