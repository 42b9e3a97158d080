"""The build: what it refuses, and the optional extension module beside the library."""
import os
import subprocess
import sysconfig

import pytest

import paper_2402_18096_gb300 as pkg
from paper_2402_18096_gb300 import build as libbuild

SOURCE = """
#define N 96
__global__ void __launch_bounds__(1024, 2) many_live_values(float* x) {  // 32 registers a thread
  float v[N];
#pragma unroll
  for (int i = 0; i < N; ++i) v[i] = x[i * 1024 + threadIdx.x];
  __syncthreads();
#pragma unroll
  for (int i = 0; i < %d; ++i) x[i * 1024 + threadIdx.x] = v[i] * v[(i * 7 + 5) %% N];
}
"""


def _compile(tmp_path, text, flags):
    src = tmp_path / "k.cu"
    src.write_text(text)
    cmd = [libbuild._nvcc(), *libbuild.ARCH, *flags, "-c", str(src), "-o", str(tmp_path / "k.o")]
    return subprocess.run(cmd, capture_output=True, text=True)


@pytest.mark.parametrize("debug", [False, True])
def test_spill_by_a_tensor_memory_load_is_an_error(tmp_path, debug):
    """The flags of the translation unit with tcgen05.ld refuse a kernel that spills, and nothing else."""
    flags = libbuild.source_flags("mikv_prefill.cu", debug)
    assert _compile(tmp_path, SOURCE % 2, flags).returncode == 0
    r = _compile(tmp_path, SOURCE % 96, flags)
    assert r.returncode != 0 and "spilled" in r.stdout + r.stderr
    assert _compile(tmp_path, SOURCE % 96, libbuild.source_flags("mikv_quant.cu", debug)).returncode == 0


def test_users_of_tensor_memory_loads_are_covered():
    for name in libbuild.SOURCES:
        with open(os.path.join(libbuild.CSRC, name)) as f:
            if "tmem_ld32" in f.read():
                assert name in libbuild.SOURCE_FLAGS


needs_tools = pytest.mark.skipif(libbuild._pycall_tools() is None, reason="no C compiler or no Python headers")


@pytest.fixture
def out_dir(tmp_path, monkeypatch):
    """An output folder whose library is current and which holds no extension module."""
    monkeypatch.setattr(libbuild, "OUT_DIR", str(tmp_path))
    monkeypatch.setattr(libbuild, "LIB", str(tmp_path / "libmikv.so"))
    (tmp_path / "libmikv.so").write_bytes(b"")
    return tmp_path


@needs_tools
def test_module_is_built_when_missing_or_stale(out_dir):
    """The module carries this interpreter's ABI in its name, and the library being current does not hide its absence or
    its age. The library is not built again for it."""
    module = libbuild.pycall_path()
    assert module.endswith(sysconfig.get_config_var("EXT_SUFFIX")) and os.path.dirname(module) == str(out_dir)
    assert not libbuild.up_to_date()
    libbuild.build()
    assert os.path.getsize(module) > 0 and libbuild.up_to_date()
    os.utime(module, (1, 1))
    assert not libbuild.up_to_date()
    libbuild.build()
    assert libbuild.up_to_date() and (out_dir / "libmikv.so").read_bytes() == b""


@needs_tools
def test_module_that_does_not_compile_is_left_out(out_dir, monkeypatch):
    """A failing compiler costs the module, not the library, and leaves no older module behind."""
    module = libbuild.pycall_path()
    with open(module, "wb"):
        os.utime(module, (1, 1))
    bad = out_dir / "cc"
    bad.write_text("#!/bin/sh\necho no such header; exit 1\n")
    bad.chmod(0o755)
    monkeypatch.setattr(libbuild, "_pycall_tools", lambda: (str(bad), "/nowhere"))
    with pytest.warns(UserWarning, match="ctypes"):
        assert libbuild.build() == str(out_dir / "libmikv.so")
    assert not os.path.exists(module)


def test_module_that_does_not_load_is_left_out(tmp_path):
    lib = pkg.load()
    bad = tmp_path / "mikv_pycall.so"
    bad.write_bytes(b"not a shared object")
    with pytest.warns(UserWarning, match="ctypes"):
        assert pkg._load_pycall(str(bad), lib) is None
    assert pkg._load_pycall(str(tmp_path / "none.so"), lib) is None


@needs_tools
def test_module_is_loaded_where_it_can_be_built():
    pkg.load()
    assert pkg._pycall is not None
