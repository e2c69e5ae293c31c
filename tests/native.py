"""Small native programs that reach the library's internals: compiled by the tests that need them."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_1301_3794_gb300")


def _builder():
    import importlib.util
    spec = importlib.util.spec_from_file_location("_dmeig_build", os.path.join(PKG, "_build.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod


def run_without_device(source, tmp_path):
    """Compile the CUDA program `source` against the library, run it with no device visible and return its
    standard output; it fails the test unless it exits 0."""
    b = _builder()
    b.build()
    src, exe = tmp_path / "check.cu", tmp_path / "check"
    src.write_text(source)
    cmd = [b.nvcc(), *b.ARCH, "-std=c++17", "-O0", "-I", b.INCLUDE, "-I", b.CSRC, "--expt-relaxed-constexpr", str(src), b.LIB,
           "-Xlinker", "-rpath," + PKG, "-o", str(exe)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, env={**os.environ, "CUDA_VISIBLE_DEVICES": ""}, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout


def host_library(source, tmp_path):
    """Compile the C++ source (no CUDA headers) against the library and load it."""
    import ctypes
    b = _builder()
    src, so = tmp_path / "host.cpp", tmp_path / "host.so"
    src.write_text(source)
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", str(src), b.LIB, "-Wl,-rpath," + PKG, "-o", str(so)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    return ctypes.CDLL(str(so))
