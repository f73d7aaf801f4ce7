"""CPU-side checks of the boundary: the library builds, loads, and exports what the header declares."""
import ctypes
import os
import re
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    from paper_2509_15235_b200 import build
    return ctypes.CDLL(build.build())


def _declared():
    text = open(os.path.join(ROOT, "include", "vispec.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(vispec_[a-z_0-9]+)\s*\(", text)))


def test_every_declared_symbol_is_exported(lib):
    names = _declared()
    assert "vispec_tree_verify_attn" in names and "vispec_kv_compact" in names and len(names) >= 12
    for n in names:
        assert hasattr(lib, n), f"{n} declared in vispec.h but not exported"


def test_binding_lists_the_same_entry_points():
    from paper_2509_15235_b200 import binding
    assert sorted(binding.EXPORTS) == _declared()


def test_strerror_and_null_argument_handling_need_no_gpu(lib):
    lib.vispec_strerror.restype = ctypes.c_char_p
    assert lib.vispec_strerror(0) == b"ok"
    assert b"tree" in lib.vispec_strerror(-8)
    assert lib.vispec_ctx_create(None, None, 0) == -1          # VISPEC_E_NULL
    assert lib.vispec_ctx_destroy(None) == 0
    assert lib.vispec_workspace_bytes(None, None) == -1


def test_shape_validation_precedes_any_cuda_call(lib):
    from paper_2509_15235_b200.binding import VispecShape
    h = ctypes.c_void_p()
    for bad in (VispecShape(1, 129, 4, 4, 64, 512, 1), VispecShape(1, 8, 6, 4, 64, 512, 1),
                VispecShape(1, 8, 4, 4, 96, 512, 1), VispecShape(0, 8, 4, 4, 64, 512, 1),
                VispecShape(1, 8, 4, 4, 64, 4, 1)):
        assert lib.vispec_ctx_create(ctypes.byref(h), ctypes.byref(bad), 0) == -3   # VISPEC_E_SHAPE


@pytest.mark.parametrize("call", ["tree_mask_build(0, t, t, None)", "accept(0, t, t, t, t, t, t)",
                                  "tree_rerank(0, t, t, t, 1, t, t, None)"])
def test_a_tensor_without_storage_raises_in_python(lib, call):
    """A fake CUDA tensor has no data pointer: torch throws inside the native module, which must come out as an exception
    and not end the process (hence the child)."""
    code = f"""
import torch
from torch._subclasses.fake_tensor import FakeTensorMode
from paper_2509_15235_b200 import binding
binding.load()
with FakeTensorMode():
    t = torch.empty(1, 4, device="cuda", dtype=torch.int32)
assert t.is_cuda
try:
    binding._native.{call}
except RuntimeError as e:
    print("raised", type(e).__name__)
"""
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, cwd=ROOT, timeout=300)
    assert r.returncode == 0 and "raised RuntimeError" in r.stdout, (r.returncode, r.stderr[-500:])


def test_product_package_does_not_import_the_oracle():
    pkg = os.path.join(ROOT, "paper_2509_15235_b200")
    for dirpath, _, files in os.walk(pkg):
        for f in files:
            if f.endswith((".py", ".cu", ".h", ".cuh")):
                src = open(os.path.join(dirpath, f)).read()
                assert "import oracle" not in src and "from oracle" not in src and "vispec_oracle" not in src
    for f in os.listdir(os.path.join(ROOT, "oracle")):
        if f.endswith((".py", ".c")):
            src = open(os.path.join(ROOT, "oracle", f)).read()
            assert "paper_2509_15235_b200" not in src and "vispec.h" not in src


@pytest.mark.parametrize("source", ["attn_tc5.cu", "attn_tc5_wide.cu"])
def test_no_attention_kernel_spills_registers(source, tmp_path):
    """The kernels are compiled for one CTA per SM with every register in use: one value too many and the step loop goes through
    local memory.  What the assembler reports, kernel by kernel."""
    from paper_2509_15235_b200 import build
    cmd = [os.environ.get("NVCC", "nvcc"), *build.NVCC_FLAGS, "-I", os.path.join(build.ROOT, "include"), "-I", build.CSRC, "-c",
           os.path.join(build.CSRC, source), "-o", str(tmp_path / "out.o")]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    said = re.findall(r"Compiling entry function '(\w+)'.*?(\d+) bytes spill stores, (\d+) bytes spill loads", res.stdout + res.stderr, flags=re.S)
    attn = [s for s in said if "attn_tc5" in s[0]]
    assert len(attn) >= 6
    assert [s for s in attn if s[1:] != ("0", "0")] == []
