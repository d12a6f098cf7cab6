"""Contractions of one call run side by side where none writes what another reads or writes.  Whatever SMs and tiles they
get, the results are the bits of the same contractions one after the other; calls whose buffers meet stay in order."""
import ctypes

import pytest
import torch

from paper_2305_14152_b200 import binding

pytestmark = pytest.mark.gpu


def _inputs(N, K, bits, g, T, seed=5):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    new = lambda *s: torch.randn(s, generator=gen, device="cuda")
    w = binding.quantize_rtn(new(N, K) * 0.02, bits, g)
    return w, new(T, K).bfloat16(), (new(T, N) * 1e-2).bfloat16()


def _linear(w, X, dY, T):
    z = lambda: torch.zeros_like(w.scales)
    return binding.LayerLinear(w=w, X=X, dY=dY, Y=torch.zeros((T, w.N), dtype=torch.bfloat16, device="cuda"),
                               dX=torch.zeros((T, w.K), dtype=torch.bfloat16, device="cuda"), dS=z(), m=z(), v=z(),
                               workspace=binding.alloc_workspace(binding.OP_BWD, T, w))


def _one_by_one(L, lr, step):
    """The step's contractions, each alone on the GPU."""
    out = []
    for f in (lambda: binding.qlinear_fwd(L.w, L.X, L.Y), lambda: binding.qlinear_bwd(L.w, None, L.dY, dX=L.dX, need_ds=False),
              lambda: binding.qlinear_bwd_ds_adamw(L.w, L.X, L.dY, L.m, L.v, lr, step=step, dS=L.dS, workspace=L.workspace)):
        f()
        torch.cuda.synchronize()
    return [t.clone() for t in (L.Y, L.dX, L.dS, L.w.scales, L.m, L.v)]


# fewer tiles of dS than CTA pairs; more, dealt (AdamW in the kernel, up to 320 tokens) and taken over (81 and more), ragged;
# both kernels for few tokens; codes that need no TMA row pitch
@pytest.mark.parametrize("N,K,bits,g,T", [(256, 256, 4, 0, 64), (1024, 512, 3, 64, 200), (2304, 2304, 4, 128, 384), (2312, 2432, 3, 64, 401),
                                          (2560, 2304, 4, 0, 33), (4096, 2048, 3, 128, 1500), (2304, 2368, 3, 64, 512), (2304, 2304, 4, 64, 320),
                                          (2312, 2432, 3, 64, 321), (2304, 2304, 4, 256, 65), (2560, 2304, 3, 256, 1)])
def test_a_step_side_by_side_is_the_step_one_by_one(N, K, bits, g, T):
    w, X, dY = _inputs(N, K, bits, g, T)
    a = _linear(w, X, dY, T)
    b = _linear(binding.QWeight(bits, N, K, g, w.qweight, w.zeros, w.scales.clone()), X, dY, T)
    for step in range(1, 7):                           # AdamW moves the scales the next step's contractions read
        binding.layer_train_step([a], lr=1e-2, step=step)
        got = [t.clone() for t in (a.Y, a.dX, a.dS, a.w.scales, a.m, a.v)]
        for x, y in zip(got, _one_by_one(b, 1e-2, step)):
            assert torch.equal(x, y)
    binding.check_status()


@pytest.mark.parametrize("N,K,bits,g,T", [(2304, 2304, 4, 128, 384), (1024, 512, 3, 64, 200), (4096, 2048, 3, 0, 700)])
def test_both_gradients_with_real_zero_points(N, K, bits, g, T):
    w, X, dY = _inputs(N, K, bits, g, T)
    zf = w.zeros.float() + 0.1
    alone = [binding.qlinear_bwd_zf(w, zf, None, dY, need_grads=False)[0]]
    torch.cuda.synchronize()
    alone += binding.qlinear_bwd_zf(w, zf, X, dY, need_dx=False)[1:]
    torch.cuda.synchronize()
    for _ in range(5):
        for x, y in zip(binding.qlinear_bwd_zf(w, zf, X, dY), alone):
            assert torch.equal(x, y)


# both kernels for dX; AdamW in the kernel of dS (groups up to 128), in its reduction and, from 2^28 products on, in the pass
# that adds the forward's sums (one scale per channel); dS by tiles that are taken over
@pytest.mark.parametrize("N,bits,g,T", [(256, 4, 0, 64), (512, 4, 32, 40), (1024, 4, 64, 1500), (1024, 3, 256, 333), (2304, 4, 128, 400), (2304, 4, 256, 100), (2048, 4, 0, 77),
                                        (2048, 3, 0, 1500)])
def test_steps_follow_one_another(N, bits, g, T):
    """Each linear's Y and dX are the next one's X and dY, and AdamW moves the scales that the next step reads: nothing lies between
    the calls that would make up for a read that comes early or finds an old value."""
    depth, steps = 3, 6
    gen = torch.Generator(device="cuda").manual_seed(N + T)
    new = lambda *s: torch.randn(s, generator=gen, device="cuda")
    ws = [binding.quantize_rtn(new(N, N) / N ** 0.5, bits, g) for _ in range(depth)]
    X, dY = new(T, N).bfloat16(), new(T, N).bfloat16()
    first = [w.scales.clone() for w in ws]
    m, v = ([torch.zeros_like(w.scales) for w in ws] for _ in range(2))
    work = [binding.alloc_workspace(binding.OP_BWD, T, w) for w in ws]
    act = lambda: torch.zeros((T, N), dtype=torch.bfloat16, device="cuda")

    def outputs():
        lists = []
        for _ in range(steps):
            x, dy, linears = X, dY, []
            for i, w in enumerate(ws):
                linears.append(binding.LayerLinear(w=w, X=x, dY=dy, Y=act(), dX=act(), dS=torch.zeros_like(w.scales), m=m[i], v=v[i], workspace=work[i]))
                x, dy = linears[-1].Y, linears[-1].dX
            lists.append(linears)
        return lists

    def reset():
        for i, w in enumerate(ws):
            w.scales.copy_(first[i])
            m[i].zero_()
            v[i].zero_()
        torch.cuda.synchronize()

    def all_steps(lists):
        for step, linears in enumerate(lists, 1):
            binding.layer_train_step(linears, lr=1e-3, step=step)

    def results(lists):
        torch.cuda.synchronize()
        binding.check_status()
        return [t.clone() for linears in lists for L in linears for t in (L.Y, L.dX, L.dS)] + [t.clone() for t in [w.scales for w in ws] + m + v]

    apart = outputs()
    reset()
    for step, linears in enumerate(apart, 1):
        for L in linears:
            alone = binding.qlinear_fwd(L.w, L.X), binding.qlinear_bwd(L.w, None, L.dY, need_ds=False)[0]
            torch.cuda.synchronize()
            binding.layer_train_step([L], lr=1e-3, step=step)
            torch.cuda.synchronize()
            assert torch.equal(L.Y, alone[0]) and torch.equal(L.dX, alone[1])
    expected = results(apart)
    assert all(torch.isfinite(t).all() for t in expected) and not torch.equal(first[0], ws[0].scales)

    together = outputs()
    reset()
    all_steps(together)
    for a, b in zip(results(together), expected):
        assert torch.equal(a, b)

    captured, graph = outputs(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        all_steps(captured)
    for _ in range(3):
        reset()
        graph.replay()
        for a, b in zip(results(captured), expected):
            assert torch.equal(a, b)


@pytest.mark.parametrize("shared", ["dX is X", "Y is dY", "workspace is dX", "dS is dX", "m is dX"])
def test_buffers_that_meet_keep_the_order(shared):
    """What the contractions one after the other leave: a later one's results, or sums under way, where an earlier one's lay."""
    N = K = 1024
    T = 256
    g = 128 if shared in ("dS is dX", "m is dX") else 256          # 128: dS and AdamW in the contraction itself
    w, X, dY = _inputs(N, K, 4, g, T)

    def linear():
        L = _linear(binding.QWeight(4, N, K, g, w.qweight, w.zeros, w.scales.clone()), X.clone(), dY.clone(), T)
        as_scales = lambda t: t.view(torch.float32).view(-1)[:w.scales.numel()].view(w.scales.shape)
        if shared == "dX is X":
            L.dX = L.X
        elif shared == "Y is dY":
            L.Y = L.dY
        elif shared == "workspace is dX":
            L.workspace = L.dX.view(torch.uint8).view(-1)
        elif shared == "dS is dX":
            L.dS = as_scales(L.dX)
        else:
            L.m = as_scales(L.dX)
        return L

    a, b = linear(), linear()
    binding.layer_train_step([a], lr=1e-2, step=1)
    _one_by_one(b, 1e-2, 1)
    for x, y in ((a.Y, b.Y), (a.dX, b.dX), (a.dS, b.dS), (a.w.scales, b.w.scales), (a.m, b.m), (a.v, b.v)):
        assert torch.equal(x.contiguous().view(torch.uint8), y.contiguous().view(torch.uint8))     # (bits: pieces of sums read as bf16 may be NaN)
    binding.check_status()


def test_gradients_of_zero_points_that_meet_dX_keep_the_order():
    N, K, T = 1024, 1024, 256
    w, X, dY = _inputs(N, K, 3, 128, T)
    zf = w.zeros.float() + 0.1
    dX, dS, dZ = binding.qlinear_bwd_zf(w, zf, X, dY, need_grads=False)[0], *binding.qlinear_bwd_zf(w, zf, X, dY, need_dx=False)[1:]
    torch.cuda.synchronize()
    out, got_s = torch.zeros_like(dX), torch.zeros_like(dS)
    got_z = out.view(torch.float32).view(-1)[:dZ.numel()].view(dZ.shape)
    q = w.c_struct()
    assert binding.lib().peqa_qlinear_bwd_zf(ctypes.byref(q), zf.data_ptr(), X.data_ptr(), dY.data_ptr(), T, out.data_ptr(), got_s.data_ptr(),
                                             got_z.data_ptr(), 0, 0, torch.cuda.current_stream().cuda_stream) == 0
    assert torch.equal(got_s, dS) and torch.equal(got_z, dZ)
    assert torch.equal(out.view(-1)[2 * dZ.numel():], dX.view(-1)[2 * dZ.numel():])
