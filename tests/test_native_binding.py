"""The extension module that marshals the frequent calls: its name carries the interpreter and torch it was built for,
the C library is built without it where its prerequisites are missing, and it refuses what the calls have always
refused before anything is enqueued."""
import os
import sysconfig

import numpy as np
import pytest
import torch

from paper_2305_14152_b200 import binding, build


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def _weight(device="cpu", N=64, K=128):
    return binding.QWeight(4, N, K, 0, torch.zeros((N, K // 8), dtype=torch.int32, device=device),
                           torch.zeros((N, 1), dtype=torch.uint8, device=device), torch.ones((N, 1), device=device))


def test_the_file_is_for_this_interpreter_and_this_torch(monkeypatch):
    path = build.native_path()
    assert os.path.exists(path)
    assert sysconfig.get_config_var("SOABI") in path and torch.__version__ in path
    monkeypatch.setattr(torch, "__version__", "0.0.0")
    monkeypatch.setattr(binding, "_native", None)
    assert build.native_path() != path
    with pytest.raises(RuntimeError, match="is missing"):        # an older file is not taken in its place
        binding.qlinear_fwd(_weight(), torch.zeros((2, 128), dtype=torch.bfloat16))


@pytest.mark.parametrize("what", ["compiler", "headers"])
def test_the_c_library_is_built_without_it(what, monkeypatch, capsys):
    if what == "compiler":
        monkeypatch.setenv("CXX", "/nonexistent/c++")
    else:
        monkeypatch.setattr(sysconfig, "get_paths", lambda: {"include": "/nonexistent"})
    monkeypatch.setattr(build, "native_path", lambda: "/nonexistent/_native.so")
    assert os.path.exists(build.build())
    assert "is missing" in capsys.readouterr().err


def test_refusals_need_no_gpu():
    w, f32 = _weight(), torch.zeros(64)
    X = torch.zeros((2, 128), dtype=torch.bfloat16)
    for call in (binding.qlinear_fwd, binding.qlinear_decode, lambda w, X: binding.qlinear_fwd_zf(w, w.scales, X),
                 lambda w, X: binding.qlinear_decode_prepared(w, w.qweight, X)):
        with pytest.raises(ValueError, match="contiguous CUDA tensor"):
            call(w, X)
    with pytest.raises(AttributeError):
        binding.qlinear_fwd(w, np.zeros((2, 128), np.float32))
    for call in (binding.scale_adamw, binding.zero_adamw):
        with pytest.raises(ValueError, match="contiguous CUDA tensor"):
            call(f32, f32, f32, f32, 1e-3)
    with pytest.raises(IndexError):
        binding.layer_train_step([])
    L = binding.LayerLinear(w=w, X=X, dY=X, Y=X, dX=X, dS=f32)
    with pytest.raises(ValueError, match="X: expected"):
        binding.layer_train_step([L])
    for refused in ((L for _ in range(1)), {0: L}, 3):           # a list or tuple, nothing that is used up by a look
        with pytest.raises(TypeError):
            binding.layer_train_step(refused)


@pytest.mark.gpu
def test_refusals_on_the_gpu():
    w = _weight("cuda")
    X = torch.zeros((4, 128), dtype=torch.bfloat16, device="cuda")
    for bad in (X.float(), X[:, ::2], X.t()):
        with pytest.raises(ValueError, match="X: expected a contiguous CUDA tensor of torch.bfloat16"):
            binding.qlinear_fwd(w, bad)
    new = lambda T, c: torch.zeros((T, c), dtype=torch.bfloat16, device="cuda")
    ls = [binding.LayerLinear(w=w, X=new(T, 128), dY=new(T, 64), Y=new(T, 64), dX=new(T, 128), dS=torch.zeros_like(w.scales),
                              workspace=binding.alloc_workspace(binding.OP_BWD, T, w)) for T in (8, 16)]
    with pytest.raises(ValueError, match="same number of tokens"):
        binding.layer_train_step(ls, apply_adamw=False)
    with pytest.raises(binding.PeqaError) as err:
        binding.qlinear_decode(w, new(17, 128))
    assert err.value.status == -3                                # PEQA_ERR_BAD_SHAPE
    with pytest.raises(TypeError):
        binding.scale_adamw(w.scales, w.scales, w.scales, w.scales, 1e-3, step=1.0)
    assert binding.qlinear_fwd(w, X).shape == (4, 64)
    binding.check_status()


@pytest.mark.gpu
def test_outputs_are_of_the_activations_class():
    class Tagged(torch.Tensor):
        pass

    w, X = _weight("cuda"), torch.ones((3, 128), dtype=torch.bfloat16, device="cuda")
    plain = binding.qlinear_fwd(w, X)
    tagged = binding.qlinear_fwd(w, X.as_subclass(Tagged))
    assert type(plain) is torch.Tensor and type(tagged) is Tagged
    assert type(binding.qlinear_fwd(w, torch.nn.Parameter(X))) is torch.Tensor
    assert torch.equal(plain, tagged.as_subclass(torch.Tensor))
