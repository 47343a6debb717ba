"""Which kernel a hopping launch runs, without a GPU: the launcher of
csrc/dhop_impl.cuh linked against a stand-in for the CUDA runtime that records
the kernel and the grid instead of launching."""
import os
import shutil
import subprocess

import pytest

from paper_2103_05034_gb300 import build

RUNTIME = r"""
#include <cstring>
#include <cuda.h>
#include <cuda_runtime_api.h>

const void* kernel = nullptr;
int grid = 0, streams = 0;

static CUresult fake_encode(CUtensorMap* m, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                            const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                            CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
  std::memset(m, 0, sizeof(*m));
  return CUDA_SUCCESS;
}

extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) { *n = 4; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  *n = 4;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult*) {
  *f = (void*)fake_encode;
  return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  kernel = f;
  grid = c->gridDim.x;
  streams++;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3, void**, size_t, cudaStream_t) {
  kernel = (const void*)k;
  grid = g.x;
  return cudaSuccess;
}
}
"""

# the launch's route; Route::kernel compares with that of another launch
COMMON = r"""
#include <cstdio>
#include <cstring>
#include "dhop_impl.cuh"

extern const void* kernel;
extern int grid, streams;

struct Route {
  const void* kernel;
  int grid;
  bool streamed;
  bool operator==(const Route& o) const { return kernel == o.kernel && grid == o.grid && streamed == o.streamed; }
};

template <int P, int LS>
Route route(int x, int y, int z, int t, int nrhs, int variant, int scalar, bool cheb = false) {
  dwfk::HopParams hp;
  std::memset(&hp, 0, sizeof(hp));
  hp.L0 = x;
  hp.L1 = y;
  hp.L2 = hp.zc = z;
  hp.L3 = t;
  hp.Lxh = x / 2;
  hp.Vh = x * y * z * t / 2;
  hp.d = 3.2;
  hp.rhs_stride = (long long)hp.Vh * 12 * LS;
  hp.cheb_mode = cheb;
  kernel = nullptr;
  grid = streams = 0;
  bool s = false;
  const int rc = dwfk::launch_hop_at<P, LS>(hp, nrhs, variant, scalar, nullptr, nullptr, &s);
  if (rc || !kernel || s != (streams == 1)) std::printf("launch failed\n");
  return {kernel, grid, s};
}
static int bad = 0;
#define CHECK(c)                              \
  if (!(c)) {                                 \
    std::printf("line %d: %s\n", __LINE__, #c); \
    bad++;                                    \
  }
"""

SCALAR = COMMON + r"""
int main() {
  // 16^3x32 streams; its Chebyshev launches take the scalar variant
  const auto r = [](int variant, int scalar, bool cheb) { return route<DWF_F32, 16>(16, 16, 16, 32, 1, variant, scalar, cheb); };
  CHECK(r(0, 0, false).streamed && r(0, 16, false).streamed);
  CHECK(!r(0, 0, true).streamed);
  for (int v = 1; v < DWF_HOP_VARIANTS; v++) {
    CHECK(!r(v, 0, false).streamed);
    CHECK(r(0, v, true) == r(v, 0, true));
    CHECK(r(v, 5, true) == r(v, 0, true));  // a choice other than 0 is everybody's
  }
  CHECK(r(0, 16, true).grid == 16 * 16 * 16 * 32 / 2 / 32);  // CTAs of eight sites on four rows
  CHECK(!(r(0, 16, true) == r(0, 3, true)));
  // a lattice that does not stream takes it for every launch
  CHECK(!(route<DWF_F32, 16>(16, 4, 4, 4, 1, 0, 0).streamed));
  CHECK((route<DWF_F32, 16>(16, 4, 4, 4, 1, 0, 26) == route<DWF_F32, 16>(16, 4, 4, 4, 1, 26, 0)));
  std::printf("bad %d\n", bad);
  return bad != 0;
}
"""


CAPS = COMMON + r"""
// the scalar kernel of a variant id on a launch of this size
template <int P, int LS, int V>
const void* scalar() {
  dwfk::HopParams hp;
  std::memset(&hp, 0, sizeof(hp));
  dwfk::launch_hop_v<P, LS, V>(hp, dim3(1), nullptr);
  return kernel;
}
// register cap that the untuned choice runs at x CTAs an SM (0: none)
template <int P, int LS>
int cap(double x, bool fused = false) {
  constexpr int SB = dwfk::HopShape<LS>::SB;
  dwfk::HopParams hp;
  std::memset(&hp, 0, sizeof(hp));
  hp.Vh = (int)(x * 152 + 0.5) * SB;
  hp.Lxh = hp.L0 = hp.L1 = 2;
  hp.cg_mode = fused;
  hp.inv_mode = !fused;  // (the streaming kernel leaves both to the scalar one: no single sweep)
  if (dwfk::launch_hop_at<P, LS>(hp, 1, 0, 0, nullptr, nullptr, nullptr)) return -1;
  const void* k = kernel;
  return k == scalar<P, LS, 26>() ? 0 : k == scalar<P, LS, 1>() ? 96 : k == scalar<P, LS, 2>() ? 80 : k == scalar<P, LS, 3>() ? 64 : -1;
}

int main() {
  const double x[] = {0.1, 3, 3.2, 6, 6.2, 8, 8.4, 9, 9.2, 11, 12, 12.4, 16.2, 24, 31, 33, 200};
  const int f32_4[] = {0, 0, 80, 80, 64, 64, 0, 0, 96, 96, 96, 96, 96, 96, 96, 96, 96};
  const int f16_4[] = {0, 0, 80, 80, 64, 64, 96, 96, 96, 96, 96, 96, 96, 96, 96, 96, 96};
  const int f32_8[] = {0, 0, 80, 80, 64, 64, 96, 96, 80, 80, 80, 64, 80, 80, 64, 64, 64};
  const int f16_8[] = {0, 0, 80, 80, 64, 64, 80, 80, 80, 80, 80, 64, 64, 64, 64, 64, 64};
  CHECK((cap<DWF_F32, 8>(27) == 80 && cap<DWF_F32, 8>(27, true) == 64));  // rounds 0.84 and 0.90 full
  CHECK((cap<DWF_F32, 8>(16.8) == 80 && cap<DWF_F32, 8>(16.8, true) == 80));
  CHECK((cap<DWF_F32, 8>(5, true) == 80 && cap<DWF_F32, 8>(7, true) == 64 && cap<DWF_F32, 8>(2, true) == 0));
  for (int i = 0; i < 17; i++) {
    const int got[4] = {cap<DWF_F32, 4>(x[i]), cap<DWF_F16S, 4>(x[i]), cap<DWF_F32, 8>(x[i]), cap<DWF_F16S, 8>(x[i])};
    const int want[4] = {f32_4[i], f16_4[i], f32_8[i], f16_8[i]};
    for (int k = 0; k < 4; k++)
      if (got[k] != want[k]) {
        std::printf("x %g case %d: %d, not %d\n", x[i], k, got[k], want[k]);
        bad++;
      }
  }
  std::printf("bad %d\n", bad);
  return bad != 0;
}
"""


F64 = COMMON + r"""
// sites per CTA of an FP64 launch of `ctas` CTAs of the default size
template <int LS>
int sites(int ctas, int inv, int g5) {
  dwfk::HopParams hp;
  std::memset(&hp, 0, sizeof(hp));
  hp.Vh = ctas * dwfk::HopShape<LS>::SB;
  hp.Lxh = hp.L0 = hp.L1 = 2;
  hp.d = 3.2;
  hp.inv_mode = inv;
  hp.g5r5 = g5;
  int parts = 0;
  if (dwfk::launch_hop_at<DWF_F64, LS>(hp, 1, 0, 0, nullptr, &parts, nullptr) || parts != grid) return -1;
  return hp.Vh / grid;
}

int main() {
  for (int inv = 0; inv < 2; inv++)
    for (int g5 = 0; g5 < 2; g5++) {
      CHECK((sites<24>(76, inv, g5) == 4));                   // half a CTA an SM
      CHECK((sites<24>(77, inv, g5) == (inv ? 4 : 8)));
      CHECK((sites<24>(456, inv, g5) == (inv ? 4 : 8)));      // three an SM
      CHECK((sites<24>(457, inv, g5) == 4));
      CHECK((sites<24>(2431, inv, g5) == 4 && sites<24>(2432, inv, g5) == 8));
      CHECK((sites<16>(100, inv, g5) == 2 && sites<8>(300, inv, g5) == 4));
    }
  std::printf("bad %d\n", bad);
  return bad != 0;
}
"""


PARTIALS = COMMON + r"""
template <int P, int LS>
void all(int prec) {
  const int L[][4] = {{2, 2, 2, 2}, {4, 4, 4, 4}, {6, 4, 10, 6}, {8, 8, 8, 16}, {12, 12, 12, 24}, {8, 16, 16, 32}, {16, 16, 16, 32}, {24, 24, 24, 48}};
  for (const auto& l : L)
    for (int nrhs = 1; nrhs <= 64; nrhs += nrhs < 6 ? 1 : 29) {
      dwfk::HopParams hp;
      std::memset(&hp, 0, sizeof(hp));
      hp.L0 = l[0], hp.L1 = l[1], hp.L2 = hp.zc = l[2], hp.L3 = l[3];
      hp.Lxh = l[0] / 2;
      hp.Vh = l[0] * l[1] * l[2] * l[3] / 2;
      hp.d = 3.2;
      hp.rhs_stride = (long long)hp.Vh * 12 * LS;
      for (int inv = 0; inv < 2; inv++) {
        hp.inv_mode = inv;
        hp.one_sweep = 1;
        int parts = 0;
        dwfk::launch_hop_at<P, LS>(hp, nrhs, 0, 0, nullptr, &parts, nullptr);
        CHECK(parts > 0 && (size_t)parts <= dwfk::hop_partials(prec, hp.Vh, LS, nrhs, 152));
      }
      // what a context reserves when it is made holds every small launch: no allocation on the way
      if (nrhs <= 4 && hp.Vh * nrhs <= 65536) CHECK(dwfk::hop_partials(prec, hp.Vh, LS, nrhs, 152) <= 65536);
    }
}
int main() {
  all<DWF_F64, 8>(DWF_F64);
  all<DWF_F64, 24>(DWF_F64);
  all<DWF_F64, 4>(DWF_F64);
  all<DWF_F32, 8>(DWF_F32);
  all<DWF_F16S, 8>(DWF_F16S);
  all<DWF_F32, 16>(DWF_F32);
  std::printf("bad %d\n", bad);
  return bad != 0;
}
"""


LINES = COMMON + r"""
int main() {
  // fills 0.68 and 0.72 (a tile's rows of six sites), 0.80, 0.84
  CHECK((route<DWF_F32, 8>(18, 24, 22, 28, 1, 0, 0).streamed && !route<DWF_F16S, 8>(18, 24, 22, 28, 1, 0, 0).streamed));
  CHECK((route<DWF_F32, 8>(18, 22, 24, 38, 3, 0, 0).streamed && !route<DWF_F16S, 8>(18, 22, 24, 38, 3, 0, 0).streamed));
  CHECK((route<DWF_F32, 8>(12, 18, 12, 36, 1, 0, 0).streamed && route<DWF_F16S, 8>(12, 18, 12, 36, 1, 0, 0).streamed));
  CHECK((route<DWF_F32, 8>(12, 18, 18, 36, 1, 0, 0).streamed && route<DWF_F16S, 8>(12, 18, 18, 36, 1, 0, 0).streamed));
  std::printf("bad %d\n", bad);
  return bad != 0;
}
"""


def _run(tmp_path, program):
    try:
        nvcc = build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    (tmp_path / "program.cu").write_text(program)
    (tmp_path / "runtime.cpp").write_text(RUNTIME)
    exe = tmp_path / "routes"
    # the host side is what runs: device code only as far as PTX
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=compute_103a", "-std=c++17", "-O1", "--expt-relaxed-constexpr",
                    "-cudart", "shared", "-I", build.CSRC, str(tmp_path / "program.cu"), str(tmp_path / "runtime.cpp"),
                    "-o", str(exe)], check=True, capture_output=True)
    env = dict(os.environ)
    env["LD_LIBRARY_PATH"] = os.path.join(os.path.dirname(os.path.dirname(nvcc)), "lib64") + ":" + env.get("LD_LIBRARY_PATH", "")
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60, env=env)
    assert r.returncode == 0 and r.stdout.strip() == "bad 0", r.stdout + r.stderr


def test_launches_that_do_not_stream_take_the_scalar_choice(tmp_path):
    _run(tmp_path, SCALAR)


def test_untuned_register_cap_by_number_of_ctas(tmp_path):
    """Nothing runs under a cap that one round of CTAs does not need, and the cap
    just above a full round is not the one whose last round is empty."""
    _run(tmp_path, CAPS)


def test_small_fp64_ctas(tmp_path):
    _run(tmp_path, F64)


def test_partial_sums_fit_what_is_reserved(tmp_path):
    """The bound that a launch reserves by holds for every route, and a reduction
    over a few fields of a small lattice needs no more than a context has."""
    _run(tmp_path, PARTIALS)


def test_streaming_line_of_fp16_storage(tmp_path):
    _run(tmp_path, LINES)
