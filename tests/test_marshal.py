"""The native marshalling of the plain calls (csrc/marshal.c): what it does not take goes to the Python code, which refuses or runs it."""
import os
import sysconfig

import pytest
import torch

import paper_2608_13426_b200 as rmm
from paper_2608_13426_b200 import binding, synth
from paper_2608_13426_b200 import build as rmm_build


class Sub(torch.Tensor):
    pass


@pytest.fixture(scope="module")
def native():
    rmm_build.build()
    return binding._native()


def test_what_is_not_plain_is_left_to_python(native):
    A, B = torch.zeros(4, 8), torch.zeros(8, 8)                   # not on a GPU
    for a, b, rho, k, scale in [(A, B, 0.5, 0, 1.0), (None, B, 0.5, 0, 1.0), (A, 3, 0.5, 0, 1.0), (A.as_subclass(Sub), B, 0.5, 0, 1.0),
                                (A, B, "half", 0, 1.0), (A, B, 0.5, 1.5, 1.0), (A, B, 0.5, 1 << 70, 1.0)]:
        assert native.product(a, b, rho, k, scale) is None
    Q = torch.zeros(1, 2, 4, 8, dtype=torch.bfloat16)
    assert native.attn(Q, Q, Q, True, 0.5, 1.0) is None and native.attn(Q, Q, None, 1, 0.5, 1.0) is None
    assert native.product() is None and native.attn(1) is None
    with pytest.raises(binding.RmmError) as e:
        rmm.rmm(A, B, 0.5)
    assert e.value.code == binding.RMM_ERR_INVALID_ARG
    with pytest.raises(binding.RmmError) as e:
        rmm.rmm_reduced_attn(Q, Q, Q, True, 0.5)
    assert e.value.code == binding.RMM_ERR_UNSUPPORTED


def test_another_interpreter_builds_its_own(native, tmp_path, monkeypatch):
    suffix = sysconfig.get_config_var("EXT_SUFFIX")
    assert binding.MARSHAL_PATH == rmm_build.MARSHAL and binding.MARSHAL_PATH.endswith("rmm_marshal" + suffix) and suffix != ".so"
    other = tmp_path / "rmm_marshal.cpython-399.so"
    monkeypatch.setattr(rmm_build, "MARSHAL", str(other))
    before = os.path.getmtime(rmm_build.LIB)
    rmm_build.build()                                             # the module alone: the library serves every interpreter
    assert other.exists() and os.path.getmtime(rmm_build.LIB) == before


@pytest.fixture
def missing(native, monkeypatch):
    monkeypatch.setattr(binding, "_marshal", None)
    monkeypatch.setattr(binding, "MARSHAL_PATH", "/nowhere/rmm_marshal.so")


def test_without_the_module_calls_reach_python(missing):
    assert binding._native() is None
    with pytest.raises(binding.RmmError) as e:
        rmm.rmm(torch.zeros(4, 8), torch.zeros(8, 8), 0.5)
    assert e.value.code == binding.RMM_ERR_INVALID_ARG
    Q = torch.zeros(1, 2, 4, 8, dtype=torch.bfloat16)
    with pytest.raises(binding.RmmError) as e:
        rmm.rmm_reduced_attn(Q, Q, Q, True, 0.5)
    assert e.value.code == binding.RMM_ERR_UNSUPPORTED


@pytest.mark.gpu
def test_without_the_module_results_are_the_same(missing):
    A, B = synth.mlp_product(40, 512, 72, device="cuda")
    Q, K, V = synth.attention_qkv(1, 4, 2, 70, 70, 64, seed=1, device="cuda")
    for got, want in zip(rmm.rmm(A, B, 0.5), rmm.rmm_product(A, B, 0.5, want_retained=True)):
        assert torch.equal(got, want)
    assert torch.equal(rmm.rmm_reduced_attn(Q, K, V, True, 0.5), rmm.rmm_reduced_attn(Q, K, V, True, 0.5, want_idx=True)[0])


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("batch, M, K, N, cut", [(0, 33, 512, 72, 0), (0, 1, 1000, 264, 0), (3, 20, 264, 40, 0), (0, 50, 300, 61, 7), (1, 40, 96, 130, 0)])
def test_products_as_by_python(native, dtype, batch, M, K, N, cut):
    A, B = synth.mlp_product((batch or 1) * M, K + cut, N, seed=M, dtype=dtype, device="cuda")
    A = A[:, cut:].reshape(batch, M, K) if batch else A[:, cut:]
    B = B[cut:].expand(batch, K, N) if batch else B[cut:]
    for b in (B, torch.nn.Parameter(B)):
        Y, idx = native.product(A, b, 0.37, 0, 2.0)
        want = rmm.rmm_product(A, b, 0.37, scale=2.0, want_retained=True)      # goes through Python
        assert Y.dtype == dtype and Y.shape == want[0].shape and idx.dtype == torch.int32 and not Y.requires_grad
        assert torch.equal(Y, want[0]) and torch.equal(idx, want[1])
        Y, idx = rmm.rmm_product(A, b, k=3)
        assert idx.shape[-1] == 3 and torch.equal(Y, rmm.rmm_product(A, b, k=3, want_retained=True)[0])
    assert rmm.rmm_status_read() == 0


@pytest.mark.gpu
def test_refusals_as_by_python(native):
    A, B = synth.mlp_product(16, 64, 32, device="cuda")
    for a, b, kw in [(A, B.float(), {"rho": 0.5}), (A, B[:-1], {"rho": 0.5}), (A, B, {"rho": 1.5}), (A, B, {"k": 65}), (A, B, {"k": -1, "rho": 0.5}),
                     (A[0], B, {"rho": 0.5}), (A.half(), B, {"rho": 0.5})]:
        got = []
        for more in ({}, {"ws": torch.zeros(1 << 24, dtype=torch.uint8, device="cuda")}):   # the second through Python
            with pytest.raises(binding.RmmError) as e:
                rmm.rmm_product(a, b, **kw, **more)
            got.append((e.value.code, str(e.value)))
        assert got[0] == got[1]


@pytest.mark.gpu
@pytest.mark.parametrize("B, Hq, Hkv, Lq, Lk, Dh, causal, rho_d, rho_t", [
    (2, 4, 2, 1, 500, 64, True, 0.5, 1.0), (1, 2, 1, 130, 130, 128, False, 0.25, 1.0), (1, 4, 4, 60, 200, 64, True, 1, 0.5)])
def test_attention_as_by_python(native, B, Hq, Hkv, Lq, Lk, Dh, causal, rho_d, rho_t):
    Q, K, V = synth.attention_qkv(B, Hq, Hkv, Lq, Lk, Dh, seed=1, device="cuda")
    for q in (Q, Q.transpose(1, 2).contiguous().transpose(1, 2)):
        O = native.attn(q, K, V, causal, rho_d, rho_t)
        assert torch.equal(O, rmm.rmm_reduced_attn(q, K, V, causal, rho_d, rho_t, want_idx=True)[0]) and O.is_contiguous()
    with pytest.raises(binding.RmmError):
        rmm.rmm_reduced_attn(Q, K, V, causal, 1.5)


@pytest.mark.gpu
def test_the_workspace_grows_and_streams_are_followed(native):
    A, B = synth.mlp_product(300, 2048, 1024, device="cuda")
    want = rmm.rmm_product(A, B, 0.5, want_retained=True)
    binding._ws_cache.clear()
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        small = rmm.rmm(A[:8, :256], B[:256, :64], 0.5)
        Y, idx = rmm.rmm(A, B, 0.5)
    s.synchronize()
    assert torch.equal(Y, want[0]) and torch.equal(idx, want[1]) and torch.isfinite(small[0]).all()


@pytest.mark.gpu
def test_names_bound_anew_in_the_middle_of_a_call(native, monkeypatch):
    """A mode's Python code runs inside the tensors' methods; what the module's names held before may be gone after it."""
    A, B = synth.mlp_product(40, 512, 72, device="cuda")
    want = rmm.rmm(A, B, 0.5)
    original = binding.workspace

    class Mode(torch.overrides.TorchFunctionMode):
        def __torch_function__(self, func, types, args=(), kwargs=None):
            binding._ws_cache = {}
            binding.workspace = original
            return func(*args, **(kwargs or {}))

    monkeypatch.setattr(binding, "_ws_cache", {})
    monkeypatch.setattr(binding, "workspace", lambda n, device: original(n, device))
    with Mode():
        got = rmm.rmm(A, B, 0.5)
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
