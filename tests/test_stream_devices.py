"""The streaming hopping kernel on several devices of one process, without a
GPU: the launcher of csrc/dhop_impl.cuh linked against a stand-in for the CUDA
runtime calls it makes, with two devices that each need their own opt-in to
large shared memory and count their own SMs."""
import os
import shutil
import subprocess

import pytest

from paper_2103_05034_gb300 import build

RUNTIME = r"""
#include <cstring>
#include <cuda.h>
#include <cuda_runtime_api.h>

int dev = 0, opted[4] = {0, 0, 0, 0}, refused[4] = {0, 0, 0, 0}, launched = 0, bad = 0, last_grid = 0;
int sms[4] = {152, 76, 152, 152};

static CUresult fake_encode(CUtensorMap* m, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                            const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                            CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
  std::memset(m, 0, sizeof(*m));
  return CUDA_SUCCESS;
}
static cudaError_t launch(size_t smem, int grid) {
  if ((size_t)opted[dev] < smem) {
    bad++;
    return cudaErrorInvalidValue;
  }
  launched++;
  last_grid = grid;
  return cudaSuccess;
}

extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = dev; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int d) { *v = sms[d]; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int bytes) {
  if (refused[dev]) return cudaErrorInvalidValue;
  opted[dev] = bytes;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult*) {
  *f = (void*)fake_encode;
  return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void*, void**) {
  return launch(c->dynamicSmemBytes, c->gridDim.x);
}
cudaError_t cudaLaunchKernel(const void*, dim3 g, dim3, void**, size_t smem, cudaStream_t) { return launch(smem, g.x); }
}
"""

PROGRAM = r"""
#include <cstdio>
#include <cstring>
#include "dhop_impl.cuh"

extern int dev, refused[4], launched, bad, last_grid, sms[4];

int main() {
  dwfk::HopParams hp;
  std::memset(&hp, 0, sizeof(hp));
  hp.L0 = hp.L1 = hp.L2 = 16;
  hp.L3 = 32;
  hp.Lxh = 8;
  hp.Vh = 16 * 16 * 16 * 32 / 2;
  hp.d = 3.2;
  hp.rhs_stride = (long long)hp.Vh * 12 * 16;
  const int order[6] = {0, 1, 0, 1, 2, 3};
  refused[3] = 1;
  for (int k = 0; k < 6; k++) {
    dev = order[k];
    int nb = 0;
    const bool ran = dwfk::launch_hop_stream<DWF_F32, 16, 4>(hp, 1, nullptr, &nb);
    // a device that refuses the shared memory leaves the launch to the scalar kernel
    if (ran != (dev != 3) || (ran && last_grid > sms[dev])) {
      std::printf("call %d on device %d: %d\n", k, dev, ran);
      bad++;
    }
  }
  if (launched != 5) bad++;
  std::printf("bad %d\n", bad);
  return bad != 0;
}
"""


def test_every_device_is_opted_in(tmp_path):
    try:
        nvcc = build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    (tmp_path / "program.cu").write_text(PROGRAM)
    (tmp_path / "runtime.cpp").write_text(RUNTIME)
    exe = tmp_path / "devices"
    subprocess.run([nvcc, *build.ARCH, "-std=c++17", "-O1", "--expt-relaxed-constexpr", "-cudart", "shared", "-I", build.CSRC,
                    str(tmp_path / "program.cu"), str(tmp_path / "runtime.cpp"), "-o", str(exe)], check=True,
                   capture_output=True)
    env = dict(os.environ)
    env["LD_LIBRARY_PATH"] = os.path.join(os.path.dirname(os.path.dirname(nvcc)), "lib64") + ":" + env.get("LD_LIBRARY_PATH", "")
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60, env=env)
    assert r.returncode == 0 and r.stdout.strip() == "bad 0", r.stdout + r.stderr
