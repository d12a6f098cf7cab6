"""GPU parity of the layer step where a linear with one scale per channel takes dS from the forward's
fp32 sums: through the cluster-split forward and through the CTA-pair forward, with ragged token
blocks, row tiles and channel tiles, with and without the optimizer step."""
import numpy as np
import pytest
import torch

import oracle
from paper_2305_14152_b200 import binding, synth
from gpu_util import adamw_scale_tol, assert_close, bf16_to_dev, dev_to_f64, oracle_layer, to_qweight

pytestmark = pytest.mark.gpu

LR = float(np.float32(1e-3))


# few tokens: one and several token tiles, two passes per tile, rows beyond a tile; many tokens: token
# blocks that end inside a half tile, a channel tile of 8 columns, tiles of one token block only
@pytest.mark.parametrize("N,K,bits,T", [(4104, 4096, 4, 17), (1000, 8192, 3, 200), (2056, 1152, 4, 300), (520, 4096, 3, 129),
                                        (8456, 2048, 4, 1030), (9736, 1280, 3, 1279), (10248, 1536, 4, 700)])
def test_channel_ds_from_the_forward(N, K, bits, T):
    d = synth.custom(N + T, N, K, T, bits, 0, outliers=True, sigma_dy=1e-2)
    codes, zeros, scales, packed = oracle_layer(d, bits, 0)
    rows = np.unique(np.concatenate([np.arange(40), np.arange(N - 40, N), np.arange(0, N, 97)]))
    toks = np.unique(np.concatenate([np.arange(3), [T // 2, T - 2, T - 1]]))
    ref = oracle.bwd_ds(d["X"], d["dY"], packed, zeros, bits, 0, rows=rows)
    X, dY = bf16_to_dev(d["X"]), bf16_to_dev(d["dY"])
    out = []
    for apply in (True, False, True):
        qw = to_qweight(packed, zeros, scales, bits, 0, K)
        L = binding.LayerLinear(w=qw, X=X, dY=dY, Y=torch.empty((T, N), dtype=torch.bfloat16, device="cuda"),
                                dX=torch.empty((T, K), dtype=torch.bfloat16, device="cuda"),
                                dS=torch.full((N, 1), 9.0, device="cuda"), m=torch.zeros((N, 1), device="cuda"),
                                v=torch.zeros((N, 1), device="cuda"),
                                workspace=binding.alloc_workspace(binding.OP_BWD, T, qw))
        L.workspace.fill_(255)
        binding.layer_train_step([L], LR, step=1, apply_adamw=apply)
        binding.check_status()
        out.append(L)
        ds = L.dS.cpu().numpy()
        assert_close(ds[rows].astype(np.float64), ref, "dS")
        # both are binary32 sums of the same products: far closer than the bound for bf16 results
        assert np.linalg.norm(ds[rows] - ref) <= 2e-6 * np.linalg.norm(ref)
        assert_close(dev_to_f64(L.Y)[toks], oracle.fwd(d["X"], packed, zeros, scales, bits, 0, tokens=toks), "Y")
        assert_close(dev_to_f64(L.dX)[toks], oracle.bwd_dx(d["dY"], packed, zeros, scales, K, bits, 0, tokens=toks), "dX")
        if apply:
            zero = np.zeros_like(scales)
            s_ref, _, _ = oracle.adamw(scales, ds, zero, zero, LR, float(np.float32(0.9)), float(np.float32(0.999)),
                                       float(np.float32(1e-8)), 0.0, 1)
            tol = adamw_scale_tol(scales, ds, zero, zero, LR, 0.9, 0.999, 1e-8, 0.0, 1)
            assert np.all(np.abs(qw.scales.cpu().numpy().ravel().astype(np.float64) - s_ref) <= tol)
        else:
            assert np.array_equal(qw.scales.cpu().numpy(), scales)
    for L in out[1:]:
        assert torch.equal(L.dS, out[0].dS) and torch.equal(L.Y, out[0].Y) and torch.equal(L.dX, out[0].dX)
    single = binding.qlinear_bwd(to_qweight(packed, zeros, scales, bits, 0, K), X, dY, need_dx=False)[1]
    assert torch.allclose(single, out[0].dS, rtol=1e-3, atol=1e-4 * float(single.abs().mean()))


def _linear(N, K, T, bits):
    d = synth.custom(N + T, N, K, T, bits, 0, outliers=True, sigma_dy=1e-2)
    codes, zeros, scales, packed = oracle_layer(d, bits, 0)
    qw = to_qweight(packed, zeros, scales, bits, 0, K)
    L = binding.LayerLinear(w=qw, X=bf16_to_dev(d["X"]), dY=bf16_to_dev(d["dY"]),
                            Y=torch.empty((T, N), dtype=torch.bfloat16, device="cuda"),
                            dX=torch.empty((T, K), dtype=torch.bfloat16, device="cuda"),
                            dS=torch.full((N, 1), 9.0, device="cuda"), m=torch.zeros((N, 1), device="cuda"),
                            v=torch.zeros((N, 1), device="cuda"))
    return d, packed, zeros, L


# through the cluster-split forward and through the CTA-pair forward
@pytest.mark.parametrize("N,T", [(2048, 96), (4096, 2048)])
def test_y_and_dx_may_share_a_buffer(N, T):
    """The forward is enqueued before dX: a caller that wants no Y may give both the same scratch."""
    K = N
    _, _, _, L = _linear(N, K, T, 4)
    L.workspace = binding.alloc_workspace(binding.OP_BWD, T, L.w)
    binding.layer_train_step([L], LR, step=1, apply_adamw=False)
    dX, dS = L.dX, L.dS.clone()
    L.Y = L.dX = torch.empty_like(dX)
    binding.layer_train_step([L], LR, step=1, apply_adamw=True)
    binding.check_status()
    assert torch.equal(L.dX, dX) and torch.equal(L.dS, dS)


@pytest.mark.parametrize("N,K,T", [(1024, 1024, 4096), (4104, 512, 1030), (2048, 2048, 2048)])
def test_surplus_workspace_changes_no_bit(N, K, T):
    # more tokens than columns in the first two: partial sums of the forward would only fit the larger one
    d, packed, zeros, L = _linear(N, K, T, 4)
    exact = binding.alloc_workspace(binding.OP_BWD, T, L.w)
    out = []
    for workspace in (exact, torch.empty(16 * exact.numel(), dtype=torch.uint8, device="cuda")):
        L.workspace = workspace
        binding.layer_train_step([L], LR, step=1, apply_adamw=False)
        binding.check_status()
        out.append(L.dS.clone())
    assert torch.equal(out[0], out[1])
    rows = np.arange(0, N, 131)
    assert_close(out[0].cpu().numpy()[rows].astype(np.float64),
                 oracle.bwd_ds(d["X"], d["dY"], packed, zeros, 4, 0, rows=rows), "dS")


def test_a_workspace_that_is_not_needed_is_not_touched():
    # one group of 128 columns is one piece: no scratch is asked for, so any pointer may be given
    N, K, T = 2048, 128, 1024
    d, packed, zeros, L = _linear(N, K, T, 4)
    assert binding.workspace_bytes(binding.OP_BWD, T, L.w) == 0
    scratch = torch.full((16 * N * 4 + 256,), 77, dtype=torch.uint8, device="cuda")
    L.workspace = scratch[4:]
    binding.layer_train_step([L], LR, step=1, apply_adamw=False)
    binding.check_status()
    assert torch.all(scratch == 77)
    assert_close(L.dS.cpu().numpy().astype(np.float64), oracle.bwd_ds(d["X"], d["dY"], packed, zeros, 4, 0), "dS")
