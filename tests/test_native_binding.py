"""The native entry points (csrc/binding.cpp): arguments by position and by keyword, the errors raised before anything reaches
the library, and what a binding that is missing or of another torch says (no GPU needed)."""
import inspect
import os
import shutil
import subprocess
import sys

import pytest
import torch

from paper_1905_10759_b200 import build, hbmm


def test_signatures():
    want = {
        "quantize": "(x, out, stream=None)", "gemm": "(A, W, C, workspace=None, stream=None)",
        "gemm_ex": "(A, W, C, path, workspace=None, stream=None)",
        "conv_im2col": "(x, geom, beta_a, a_scale_dtype, W, C_out, workspace, stream=None, flags=0)",
        "conv_im2col_fused": "(x, geom, beta_a, a_scale_dtype, W, ep, workspace, stream=None, flags=0)",
        "binarize_dense": "(x, beta, out_dtype=0, out=None, stream=None)",
        "binarize_backward": "(x, gy, beta, gx=None, stream=None)",
    }
    assert {n: str(inspect.signature(getattr(hbmm, n))) for n in want} == want


@pytest.mark.parametrize("call,error,text", [
    (lambda x, op: hbmm.quantize(x, op), ValueError, "device tensor expected"),
    (lambda x, op: hbmm.quantize(out=op, x=x), ValueError, "device tensor expected"),
    (lambda x, op: hbmm.quantize(x.t(), op), ValueError, "row-major"),
    (lambda x, op: hbmm.quantize(x[0], op), ValueError, "row-major"),
    (lambda x, op: hbmm.gemm(op, op, x), ValueError, "device tensor expected"),
    (lambda x, op: hbmm.gemm_ex(op, op, x, hbmm.PATH_AUTO, workspace=x), ValueError, "device tensor expected"),
    (lambda x, op: hbmm.binarize_dense(x.double(), 4), ValueError, "fp32 matrix"),
    (lambda x, op: hbmm.binarize_dense(x, 4, hbmm.BF16, x), ValueError, "requested type"),
    (lambda x, op: hbmm.binarize_backward(x, x[:1], 4), ValueError, "one shape"),
    (lambda x, op: hbmm.binarize_backward(x.t(), x.t(), 4), ValueError, "contiguous"),
    (lambda x, op: hbmm.conv_im2col(x.t(), hbmm.make_geom(1, 1, 2, 32, 1, 1), 32, hbmm.F32, op, x, x), ValueError, "contiguous"),
    (lambda x, op: hbmm.quantize(x), TypeError, "out"),
    (lambda x, op: hbmm.quantize(x, op, None, None), TypeError, "positional"),
    (lambda x, op: hbmm.quantize(x, op, x=x), TypeError, "multiple values"),
    (lambda x, op: hbmm.gemm(op, op, x, ws=None), TypeError, "unexpected"),
    (lambda x, op: hbmm.quantize([1.0], op), TypeError, "Tensor"),
    (lambda x, op: hbmm.conv_im2col(x, hbmm.make_geom(1, 1, 2, 32, 1, 1), 32, hbmm.F32, op, x, x, flags=None), ValueError, "device tensor"),
])
def test_errors_before_the_library(call, error, text):
    x = torch.ones((2, 32))
    with pytest.raises(error, match=text):
        call(x, hbmm.alloc_operand(2, 32, 32, device="cpu"))


GEOM, EP, OPERAND = hbmm.make_geom(1, 1, 2, 32, 1, 1), hbmm.hbmm_epilogue(), hbmm.hbmm_operand()


@pytest.mark.parametrize("desc", [GEOM, EP, bytes(256), bytearray(256), None])
def test_operands_of_another_type(desc):
    x, bad = torch.ones((2, 32)), hbmm.Operand(desc)
    good = hbmm.alloc_operand(2, 32, 32, device="cpu")
    for call in (lambda: hbmm.quantize(x, bad), lambda: hbmm.gemm(bad, good, x), lambda: hbmm.gemm(good, bad, x),
                 lambda: hbmm.gemm_ex(good, bad, x, hbmm.PATH_AUTO), lambda: hbmm.conv_im2col(x, GEOM, 32, hbmm.F32, bad, x, x),
                 lambda: hbmm.conv_im2col_fused(x, GEOM, 32, hbmm.F32, bad, EP, x)):
        with pytest.raises(TypeError, match="hbmm_operand expected"):
            call()


@pytest.mark.parametrize("other", [OPERAND, bytes(256), (1, 1, 2, 32, 1, 1, 1, 1, 0, 0)])
def test_geometries_and_epilogues_of_another_type(other):
    x, op = torch.ones((2, 32)), hbmm.alloc_operand(2, 32, 32, device="cpu")
    for geom in (other, EP):
        with pytest.raises(TypeError, match="hbmm_conv_geom expected"):
            hbmm.conv_im2col(x, geom, 32, hbmm.F32, op, x, x)
        with pytest.raises(TypeError, match="hbmm_conv_geom expected"):
            hbmm.conv_im2col_fused(x, geom, 32, hbmm.F32, op, EP, x)
    for ep in (other, GEOM):
        with pytest.raises(TypeError, match="hbmm_epilogue expected"):
            hbmm.conv_im2col_fused(x, GEOM, 32, hbmm.F32, op, ep, x)


def import_copy(where, change):
    """Imports a copy of the package whose _binding.so has been changed; the error it ends with."""
    pkg = where / "paper_1905_10759_b200"
    pkg.mkdir()
    for f in ("__init__.py", "hbmm.py", "build.py", "libhbmm.so", "_binding.so"):
        src = os.path.join(build.HERE, f)
        (os.symlink if f == "libhbmm.so" else shutil.copy)(src, pkg / f)
    change(pkg / "_binding.so")
    run = subprocess.run([sys.executable, "-c", "import paper_1905_10759_b200.hbmm"], cwd=where, capture_output=True, text=True)
    assert run.returncode != 0
    return run.stderr.strip().splitlines()[-1]


def test_missing_or_foreign_binding(tmp_path):
    hint = "python -m paper_1905_10759_b200.build"
    for name, change, text in (("a", os.remove, "missing or does not load"), ("b", lambda p: p.write_bytes(b"no library"), "missing or does not load"),
                               ("c", lambda p: p.write_bytes(p.read_bytes().replace(build.built_for().encode(), build.built_for().encode()[::-1])), "is built for")):
        where = tmp_path / name
        where.mkdir()
        error = import_copy(where, change)
        assert error.startswith("ImportError: _binding.so") and text in error and hint in error


def test_binding_of_another_torch_is_stale(monkeypatch):
    assert not build.binding_is_stale()
    monkeypatch.setattr(torch, "__version__", "0.0")
    assert build.binding_is_stale() and not build.lib_is_stale()
