"""The native entry of binding.gemm takes plain calls only: whatever it does not take as it is goes through the general
checks, with their errors.  (CPU: nothing is launched.  GPU: the same result on both routes.)"""
import numpy as np
import pytest
import torch

import paper_2609_36800_b200 as bd
from paper_2609_36800_b200 import binding, synth


@pytest.fixture(scope="module", autouse=True)
def lib():
    from paper_2609_36800_b200 import build
    build.build()
    return bd.load_library()


def test_the_module_is_built_and_leaves_cpu_tensors_to_the_general_checks():
    assert binding._fast is not None
    X, W = torch.zeros(1, 2, 128, dtype=torch.bfloat16), torch.zeros(4, 128, dtype=torch.bfloat16)
    bits, alpha = torch.zeros(1, 4, 4, dtype=torch.int32), torch.zeros(1)
    out, ws = torch.zeros(1, 2, 4, dtype=torch.bfloat16), torch.zeros(1024, dtype=torch.uint8)
    assert binding._fast(X, W, bits, alpha, None, out, ws, 0, 0) is None
    with pytest.raises(TypeError, match="contiguous CUDA tensor"):
        bd.gemm(X, W, bits, alpha, out=out, workspace=ws)
    with pytest.raises(ValueError, match="inconsistent shapes"):
        bd.gemm(X, W[:, :64], bits, alpha, out=out, workspace=ws)
    with pytest.raises(TypeError, match="bfloat16 or float16"):
        bd.gemm(X.float(), W, bits, alpha, out=out, workspace=ws)
    with pytest.raises(ValueError, match="unknown activation"):
        bd.gemm(X, W, bits, alpha, out=out, workspace=ws, act="relu")


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,bias,act", [(torch.bfloat16, False, "none"), (torch.float16, True, "silu"), (torch.bfloat16, True, "silu_gate")])
def test_both_routes_give_the_same_result_and_the_same_refusals(dtype, bias, act, monkeypatch):
    B, m, N, K = 3, 2, 256, 256
    g = torch.Generator(device="cuda").manual_seed(1)
    X = torch.randn(B, m, K, device="cuda", generator=g).to(dtype)
    W = (torch.randn(N, K, device="cuda", generator=g) * 0.02).to(dtype)
    bits = torch.randint(-2**31, 2**31, (B, N, K // 32), device="cuda", dtype=torch.int32, generator=g)
    alpha = torch.rand(B, device="cuda", generator=g) * 0.01
    b = torch.randn(N, device="cuda", generator=g).to(dtype) if bias else None
    ws = bd.make_workspace(B, m, N, K)
    shape = (B, m, N // 2 if act == "silu_gate" else N)

    def run(**kw):
        out = torch.full(shape, float("nan"), dtype=dtype, device="cuda")
        assert bd.gemm(X, W, bits, alpha, out=out, workspace=ws, bias=b, act=act, **kw) is out
        return out

    fast = run()
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        on_side = run()
    torch.cuda.current_stream().wait_stream(side)
    for refused, err in ((dict(X=X[:, :, ::2]), ValueError), (dict(X=X.transpose(0, 1)), (ValueError, TypeError)),
                         (dict(alpha=alpha.double()), TypeError), (dict(workspace=ws[:64]), bd.BitDeltaError)):
        a = dict(X=X, W_base=W, bits=bits, alpha=alpha, out=fast.clone(), workspace=ws, bias=b, act=act)
        a.update(refused)
        with pytest.raises(err):
            bd.gemm(**a)
    monkeypatch.setattr(binding, "_fast", None)
    slow = run()
    torch.cuda.synchronize()
    assert torch.equal(fast.view(torch.int16), slow.view(torch.int16)) and torch.equal(on_side.view(torch.int16), slow.view(torch.int16))


def _child(code):
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    return subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True)


@pytest.mark.parametrize("other", ["torch.__version__ = '2.0.0'", "import sysconfig; sysconfig._CONFIG_VARS['EXT_SUFFIX'] = '.cpython-39-x86_64-linux-gnu.so'"])
def test_a_module_built_against_another_torch_or_python_is_not_loaded(other):
    r = _child(f"import torch, sysconfig; sysconfig.get_config_vars(); {other}; import paper_2609_36800_b200 as bd; bd.load_library(); "
               "assert bd.binding._fast is None")
    assert r.returncode == 0, r.stderr


@pytest.mark.parametrize("error", ["ImportError('no torch')", "FileNotFoundError('g++')", "subprocess.CalledProcessError(1, 'g++')"])
def test_the_library_is_built_without_the_module(error):
    # (nothing is compiled or linked: the steps are replaced by records of them)
    r = _child(f"""
import subprocess
from paper_2609_36800_b200 import build
ran = []
def fail(*a): raise {error}
build.build_fastcall, build._compile = fail, lambda src, *a: src
build.subprocess.run = lambda cmd, **kw: ran.append(cmd)
assert build.build(force=True) == build.LIB
assert any(build.LIB in cmd for cmd in ran), ran
""")
    assert r.returncode == 0, r.stderr
