"""The native form of the tensor entry points: argument errors raise before anything touches a GPU, and what a caller passes
for the output and the stream is honoured."""
import numpy as np
import pytest
import torch

import oracle
from helpers import assert_close_to_oracle, bits_to_cuda_bf16, small_fused_inputs


@pytest.fixture(scope="module")
def binding():
    from paper_2407_13885_b200 import build
    build.build_library()
    from paper_2407_13885_b200 import binding
    return binding


def test_host_tensors_are_refused(binding):
    x = torch.zeros(1, 1, 8, 64, dtype=torch.bfloat16)
    for call in (lambda: binding.attnw_fused(x, x, 0.125), lambda: binding.attn_fused(x, x, x, 0.125),
                 lambda: binding.project_qk(x[0], x[0], x[0]), lambda: binding.softmax_rows(x[0, 0].float()),
                 lambda: binding.attnw_fused(None, x, 0.125)):
        with pytest.raises(TypeError, match="must be a CUDA tensor"):
            call()


@pytest.mark.gpu
def test_bad_arguments_on_the_gpu(binding):
    q = torch.zeros(1, 2, 64, 64, dtype=torch.bfloat16, device="cuda")
    for exc, call in ((TypeError, lambda: binding.attnw_fused(q.float(), q, 0.125)),
                      (ValueError, lambda: binding.attnw_fused(q, q[:, :1], 0.125)),
                      (ValueError, lambda: binding.attnw_fused(q.transpose(1, 2), q.transpose(1, 2), 0.125)),
                      (ValueError, lambda: binding.attnw_fused(q, q, 0.125, out_dtype=torch.float16)),
                      (ValueError, lambda: binding.attnw_fused(q, q, 0.125, P=q[:, :1].contiguous())),
                      (ValueError, lambda: binding.attn_fused(q, q, q, 0.125, O=q[:, :1].contiguous())),
                      (ValueError, lambda: binding.project_qk(q[0], q[0], q[0, :1].contiguous())),
                      (ValueError, lambda: binding.softmax_rows(q.float())),
                      (TypeError, lambda: binding.attnw_fused(q, q, None))):
        with pytest.raises(exc):
            call()
    with pytest.raises(binding.AttnwError) as e:
        binding.attnw_fused(q, q, -1.0)
    assert e.value.code == 2


@pytest.mark.gpu
def test_no_type_is_the_default_type(binding):
    q, k = small_fused_inputs(1, 1, 64, 64, stream=7)
    P = binding.attnw_fused(bits_to_cuda_bf16(q), bits_to_cuda_bf16(k), 0.125, out_dtype=None)
    assert P.dtype == torch.float32
    assert_close_to_oracle(P, oracle.attnw(q, k, 0.125))
    assert binding.softmax_rows(P[0, 0].contiguous(), out_dtype=None).dtype == torch.float32


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_given_output_and_stream(binding, dtype):
    q, k = small_fused_inputs(1, 2, 200, 64, stream=5)
    Q, K = bits_to_cuda_bf16(q), bits_to_cuda_bf16(k)
    P = torch.empty(1, 2, 200, 200, dtype=dtype, device="cuda")
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    for stream in (s, s.cuda_stream):
        P.fill_(float("nan"))
        torch.cuda.synchronize()
        assert binding.attnw_fused(Q, K, np.float32(0.125), P=P, stream=stream) is P
        s.synchronize()
        assert_close_to_oracle(P, oracle.attnw(q, k, 0.125), f"{dtype}")


def test_tensors_without_storage_are_refused(binding):
    # torch.func.vmap hands over wrappers that have no address: the calls raise, also where there is no GPU (fake tensors)
    from torch._subclasses.fake_tensor import FakeTensorMode
    with FakeTensorMode():
        q = torch.empty(2, 1, 1, 64, 64, dtype=torch.bfloat16, device="cuda")
        for call, x in ((lambda x: binding.attnw_fused(x, x, 0.125), q), (lambda x: binding.attn_fused(x, x, x, 0.125), q),
                        (lambda x: binding.project_qk(x, x, x), q[0]), (binding.softmax_rows, q[0, 0].float())):
            with pytest.raises(RuntimeError, match="storage"):
                torch.func.vmap(call)(x)


@pytest.mark.gpu
def test_vmap_is_refused(binding):
    q = torch.zeros(2, 1, 1, 64, 64, dtype=torch.bfloat16, device="cuda")
    p = torch.zeros(1, 1, 64, 64, dtype=torch.bfloat16, device="cuda")
    for call, x in ((lambda x: binding.attnw_fused(x, x, 0.125), q), (lambda x: binding.attnw_fused(p, p, 0.125, P=x), q),
                    (lambda x: binding.attn_fused(x, x, x, 0.125), q), (lambda x: binding.attn_fused(p, p, p, 0.125, O=x), q),
                    (lambda x: binding.project_qk(x, x, x), q[0]), (binding.softmax_rows, q[0, 0].float())):
        with pytest.raises(RuntimeError, match="storage"):
            torch.func.vmap(call)(x)


def test_tensors_of_several_devices_are_refused(binding):
    # (fake tensors: the check comes before anything asks for an address, and needs neither one GPU nor two)
    from torch._subclasses.fake_tensor import FakeTensorMode
    with FakeTensorMode():
        q, far = (torch.empty(1, 1, 64, 64, dtype=torch.bfloat16, device=f"cuda:{n}") for n in range(2))
        s, far_s = q[0, 0].float(), far[0, 0].float()
        for call in (lambda: binding.attnw_fused(q, far, 0.125), lambda: binding.attnw_fused(q, q, 0.125, P=far),
                     lambda: binding.attn_fused(q, far, q, 0.125), lambda: binding.attn_fused(q, q, far, 0.125),
                     lambda: binding.attn_fused(q, q, q, 0.125, O=far), lambda: binding.project_qk(q[0], far[0], q[0]),
                     lambda: binding.project_qk(q[0], q[0], far[0]), lambda: binding.project_qk(q[0], q[0], q[0], Q=far),
                     lambda: binding.project_qk(q[0], q[0], q[0], Q=q, K=far), lambda: binding.softmax_rows(s, P=far_s),
                     lambda: binding.softmax_rows(s, P=far[0, 0]), lambda: binding.attnw_fused_noalloc(q, far, 0.125),
                     lambda: binding.attnw_fused_noalloc(q, q, 0.125, P=far)):
            with pytest.raises(ValueError, match="must be on cuda:0"):
                call()


def test_extension_is_built_again_for_another_torch_or_python(binding, monkeypatch):
    import sysconfig

    from paper_2407_13885_b200 import build
    assert not build.ext_is_stale() and binding._native.__doc__ == build.built_for()
    with monkeypatch.context() as m:
        m.setattr(torch, "__version__", torch.__version__ + ".1")
        assert build.ext_is_stale()
    soabi = sysconfig.get_config_var("SOABI")
    with monkeypatch.context() as m:
        m.setattr(sysconfig, "get_config_var", lambda name: soabi + "x" if name == "SOABI" else None)
        assert build.ext_is_stale()
    assert not build.ext_is_stale()
