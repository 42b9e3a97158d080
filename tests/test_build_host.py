"""The build: what it refuses."""
import subprocess

import pytest

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
    import os
    for name in libbuild.SOURCES:
        with open(os.path.join(libbuild.CSRC, name)) as f:
            if "tmem_ld32" in f.read():
                assert name in libbuild.SOURCE_FLAGS
