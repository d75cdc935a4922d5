"""Host-side checks of the C ABI that need no GPU: the library builds for sm_100a, loads, exports
every function include/bfq.h declares, the binding lists the same set, and the entry points that
can answer without a device (status strings, argument validation that precedes any CUDA call) do."""
import ctypes
import os
import re

import pytest

from paper_2509_09679_b200 import binding, build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def declared_functions():
    text = open(os.path.join(ROOT, "include", "bfq.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(bfq_[a-z0-9_]+)\s*\(", text)))


@pytest.fixture(scope="module")
def lib():
    build.build()
    return binding.lib()


def test_header_functions_are_exported_and_bound(lib):
    names = declared_functions()
    for required in ("bfq_forward_quant", "bfq_inverse", "bfq_backward", "bfq_fold_weights"):
        assert required in names
    for name in names:
        assert hasattr(lib, name), f"{name} declared in bfq.h but not exported by libbfq.so"
    assert sorted(binding.SIGNATURES) == names


def test_status_strings(lib):
    codes = sorted(binding.STATUS_NAMES)
    assert codes == list(range(min(codes), 1))
    seen = {lib.bfq_status_string(c).decode() for c in codes}
    assert len(seen) == len(codes) and "unknown status" not in seen
    assert lib.bfq_status_string(-99).decode() == "unknown status"


def test_validation_that_precedes_any_cuda_call(lib):
    h = ctypes.c_void_p()
    assert lib.bfq_plan_create(None, 256, 0, 0) == -1                      # BFQ_ERR_NULL
    assert lib.bfq_plan_create(ctypes.byref(h), 100, 0, 0) == -2           # not a power of two
    assert lib.bfq_plan_create(ctypes.byref(h), 8, 0, 0) == -2             # below BFQ_MIN_N
    assert lib.bfq_plan_create(ctypes.byref(h), 16384, 0, 0) == -2         # above BFQ_MAX_N
    assert lib.bfq_plan_create(ctypes.byref(h), 256, -1, 0) == -5          # negative max_rows
    assert h.value is None
    assert lib.bfq_plan_destroy(None) == -1
    assert lib.bfq_last_cuda_error(None) == 0
    assert lib.bfq_backward_partials(None) == 0
    assert lib.bfq_forward_quant(None, None, 0, 0, 0, 4, None, None, None) == -1
    assert lib.bfq_forward_quant_host(None, None, 0, 0, 0, 4, None, None, None, 0, None) == -1
    assert lib.bfq_forward_quant_host_workspace(None, 0, 4, 128) == 0
    # the no-allocation backward checks its sizes before it touches the device
    assert lib.bfq_backward_noalloc(2048, None, None, 0, None, 0, 0, 2048, None, 0, None, None) == -10
    assert lib.bfq_backward_noalloc(100, None, None, 0, None, 0, 0, 100, None, 0, None, None) == -2
    assert lib.bfq_backward_noalloc(256, None, None, 0, None, 0, 0, 256, None, 0, None, None) == -1


def _planless(n=256):
    """A Plan object without a device handle: every check below must raise before the library is reached."""
    import torch

    p = object.__new__(binding.Plan)
    p.n, p.L, p.device, p._h = n, n.bit_length() - 1, torch.device("cuda", 0), ctypes.c_void_p()
    return p


def test_binding_rejects_bad_tensors_before_any_launch(monkeypatch):
    import torch

    def no_library():
        raise AssertionError("a bad tensor reached the C ABI")

    monkeypatch.setattr(binding, "lib", no_library)
    p = _planless(256)
    x = torch.zeros((4, 256))
    with pytest.raises(ValueError, match="is on cpu"):
        p.forward_quant(x, 4)                                   # host tensor
    with pytest.raises(ValueError, match="is on cpu"):
        p.backward(x, x)
    with pytest.raises(ValueError):
        p.forward(torch.zeros((4, 128)))                        # wrong row length
    with pytest.raises(ValueError):
        p.forward(torch.zeros((4, 512))[:, ::2])                # inner stride 2
    with pytest.raises(ValueError):
        p.set_angles(torch.zeros((8, 64)))                      # theta of a smaller n
    with pytest.raises(ValueError):
        p.set_angles(torch.zeros((8, 128), dtype=torch.float64))
    # caller-supplied outputs: exact dtype and shape, checked before the device
    with pytest.raises(ValueError, match="codes"):
        p._outputs(4, 256, 4, torch.zeros((4, 64), dtype=torch.uint8), torch.zeros((4,), dtype=torch.float16))
    with pytest.raises(ValueError, match="scales: expected"):
        binding._exact(torch.zeros((3,), dtype=torch.float16), torch.float16, (4,), p.device, "scales")
    with pytest.raises(ValueError, match="codes: tensor is on cpu"):
        p._outputs(4, 256, 4, torch.zeros((4, 128), dtype=torch.uint8), torch.zeros((4,), dtype=torch.float16))
    with pytest.raises(ValueError, match="codes"):
        p._outputs(4, 256, 4, torch.zeros((4, 128), dtype=torch.int8), torch.zeros((4,), dtype=torch.float16))
    # the plan-less entry point sizes theta and dtheta from x
    with pytest.raises(ValueError):
        binding.backward_noalloc(torch.zeros((8, 128)), x, x, None, torch.zeros((8, 128)))
    with pytest.raises(ValueError):
        binding._rows(torch.zeros((4, 300)).as_strided((4, 256), (100, 1)), 256)   # overlapping rows
    with pytest.raises(ValueError, match="expected 4 rows"):
        binding._rows(torch.zeros((5, 256)), 256, None, 4, "out")


def test_the_plain_forms_leave_everything_else_to_the_binding():
    """fast_calls answers None to what is not plain rows on a plan's device: no plan, host tensors, other types and counts."""
    import torch
    binding.lib()
    fast = binding._fast
    assert fast.__file__ == build.FAST  # the compiled module, not what answers None to everything
    x = torch.zeros((2, 8))
    for call in (fast.forward, fast.inverse):
        assert call(0, 8, 0, x) is None and call(64, 8, 0, x) is None and call(64, 8, 0, [1.0]) is None and call(64, 8, 0) is None
        assert call("plan", 8, 0, x) is None and call(64, 8.0, 0, x) is None
    assert fast.forward_quant(64, 8, 0, x, 4) is None and fast.forward_quant(64, 8, 0, x, "4") is None


def test_the_library_is_built_where_the_extension_cannot_be(monkeypatch, capsys):
    """The C++ part of the binding is optional: without a compiler or headers for it the CUDA library is built all the same."""
    from paper_2509_09679_b200 import build
    done = []
    monkeypatch.setattr(build, "build_library", lambda *a: done.append("library"))
    for error in (FileNotFoundError("g++"), build.subprocess.CalledProcessError(1, "g++"), ModuleNotFoundError("torch")):
        def fails(force, error=error):
            raise error
        monkeypatch.setattr(build, "build_fast_calls", fails)
        assert build.build() == build.LIB and done.pop() == "library" and "was not built" in capsys.readouterr().err


def test_the_extension_is_used_with_the_torch_it_was_built_against_only(monkeypatch, tmp_path):
    """Another torch: the module that is there is not called, and the next build compiles it again."""
    import sys
    import torch
    from paper_2509_09679_b200 import build
    assert binding._native_calls() is sys.modules["paper_2509_09679_b200.fast_calls"]
    commands = []
    monkeypatch.setattr(build, "FAST", str(tmp_path / "fast_calls.so"))
    monkeypatch.setattr(build, "FAST_TORCH", str(tmp_path / "fast_calls.torch"))

    def compiler(command, check):
        commands.append(command)
        (tmp_path / "fast_calls.so").touch()
    monkeypatch.setattr(build.subprocess, "run", compiler)
    for _ in range(2):
        build.build_fast_calls()
    assert len(commands) == 1
    monkeypatch.setattr(torch, "__version__", "0.1")
    assert binding._native_calls() is binding._Interpreted and binding._Interpreted.forward(64, 8, 0, None) is None
    for _ in range(2):
        build.build_fast_calls()
    assert len(commands) == 2 and '-DBFQ_TORCH="0.1"' in commands[1]


def test_the_extension_says_what_it_does_not_find():
    with pytest.raises(OSError):
        binding._native_calls().attach("/nonexistent/libbfq.so")


def test_importing_the_package_loads_no_compiled_code():
    import subprocess
    import sys
    code = "import sys, paper_2509_09679_b200 as p; assert not any(m.endswith('fast_calls') for m in sys.modules) and p.binding._lib is None"
    subprocess.run([sys.executable, "-c", code], check=True, cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
