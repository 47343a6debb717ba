// C ABI: context, operators and the red-black CG solver (arXiv:2103.05034,
// Sec. 2 and Sec. 5.1).  Every step of the path runs in this library's
// kernels; the host only sequences launches and reads back scalars.
#include <math.h>
#include <string.h>

#include <chrono>
#include <new>

#include "dhop_impl.cuh"
#include "dwf_internal.cuh"

// ------------------------------------------------------------------ errors
int dwf_fail(dwf_ctx* c, int code, const std::string& msg) {
  if (c) c->err = msg;
  return code;
}

int dwf_cuda_check(dwf_ctx* c, cudaError_t e, const char* where) {
  std::string m = std::string("CUDA error ") + cudaGetErrorName(e) + " (" + cudaGetErrorString(e) +
                  ") in " + where;
  return dwf_fail(c, DWF_ECUDA, m);
}

extern "C" const char* dwf_last_error(const dwf_ctx* c) { return c ? c->err.c_str() : "null context"; }

size_t dwf_complex_bytes(int prec) {
  switch (prec) {
    case DWF_F64:
      return 16;
    case DWF_F32:
      return 8;
    case DWF_F16S:
      return 4;
    default:
      return 0;
  }
}

bool dwf_is_device_ptr(const void* p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

void* dwf_workspace(dwf_ctx* c, int slot, size_t bytes) {
  if (slot < 0 || slot >= DWF_NWS) return nullptr;
  if (c->ws_bytes[slot] >= bytes && c->ws[slot]) return c->ws[slot];
  if (c->ws[slot]) cudaFree(c->ws[slot]);
  c->ws[slot] = nullptr;
  c->ws_bytes[slot] = 0;
  void* p = nullptr;
  if (cudaMalloc(&p, bytes) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  c->ws[slot] = p;
  c->ws_bytes[slot] = bytes;
  return p;
}

int dwf_reserve_partials(dwf_ctx* c, size_t n) {
  if (c->partials_n >= n) return DWF_OK;
  if (c->partials) cudaFree(c->partials);
  c->partials = nullptr;
  c->partials_n = 0;
  if (cudaMalloc(&c->partials, n * sizeof(double)) != cudaSuccess) {
    cudaGetLastError();
    return dwf_fail(c, DWF_ENOMEM, "cannot allocate reduction partials");
  }
  c->partials_n = n;
  return DWF_OK;
}

// ------------------------------------------------------------------ links
// Canonical complex128 [T][Z][Y][X][mu][3][3] -> per output parity p
// [Vh][8][3][3]: slot 2mu = U_mu(x), slot 2mu+1 = U_mu(x-mu)^dag.
__global__ void k_build_links(const double2* __restrict__ U, double2* l64, float2* l32, int L0, int L1,
                              int L2, int L3, int parity) {
  const int Lxh = L0 / 2;
  const long long Vh = (long long)L0 * L1 * L2 * L3 / 2;
  const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (gid >= Vh * 8) return;
  const int h = (int)(gid / 8), slot = (int)(gid % 8);
  const int mu = slot / 2, bwd = slot & 1;
  int rem = h / Lxh;
  const int xh = h - rem * Lxh;
  const int y = rem % L1;
  rem /= L1;
  const int z = rem % L2;
  const int t = rem / L2;
  int c[4] = {2 * xh + ((y + z + t + parity) & 1), y, z, t};
  const int Ld[4] = {L0, L1, L2, L3};
  if (bwd) c[mu] = (c[mu] == 0) ? Ld[mu] - 1 : c[mu] - 1;
  const long long lex = c[0] + (long long)L0 * (c[1] + (long long)L1 * (c[2] + (long long)L2 * c[3]));
  const double2* src = U + (lex * 4 + mu) * 9;
  double2* d64 = l64 + gid * 9;
  float2* d32 = l32 + gid * 9;
  for (int a = 0; a < 3; a++)
    for (int b = 0; b < 3; b++) {
      double2 v = bwd ? make_double2(src[b * 3 + a].x, -src[b * 3 + a].y) : src[a * 3 + b];
      d64[a * 3 + b] = v;
      d32[a * 3 + b] = make_float2((float)v.x, (float)v.y);
    }
}

extern "C" int dwf_ctx_create(dwf_ctx** out, const int L[4], int Ls, double M5, const void* gauge,
                              void* stream) {
  if (!out || !L || !gauge) return DWF_EINVAL;
  *out = nullptr;
  for (int m = 0; m < 4; m++)
    if (L[m] < 2 || (L[m] & 1)) return DWF_EINVAL;
  if (Ls != 4 && Ls != 8 && Ls != 16 && Ls != 24) return DWF_EINVAL;
  const long long V4 = (long long)L[0] * L[1] * L[2] * L[3];
  if (V4 / 2 * 12LL * Ls >= (1LL << 40) || V4 / 2 >= (1LL << 31) / 12) return DWF_EINVAL;
  dwf_ctx* c = new (std::nothrow) dwf_ctx();
  if (!c) return DWF_ENOMEM;
  for (int m = 0; m < 4; m++) c->g.L[m] = L[m];
  c->g.Lxh = L[0] / 2;
  c->g.Vh = V4 / 2;
  c->g.Ls = Ls;
  c->M5 = M5;
  cudaGetDevice(&c->device);
  cudaDeviceGetAttribute(&c->sms, cudaDevAttrMultiProcessorCount, c->device);
  cudaStream_t st = (cudaStream_t)stream;
  const size_t glinks = (size_t)V4 * 4 * 9;
  const void* Ud = gauge;
  void* tmp = nullptr;
  int rc = DWF_OK;
  if (!dwf_is_device_ptr(gauge)) {
    if (cudaMalloc(&tmp, glinks * sizeof(double2)) != cudaSuccess) {
      cudaGetLastError();
      delete c;
      return DWF_ENOMEM;
    }
    cudaMemcpyAsync(tmp, gauge, glinks * sizeof(double2), cudaMemcpyHostToDevice, st);
    Ud = tmp;
  }
  for (int p = 0; p < 2 && rc == DWF_OK; p++) {
    if (cudaMalloc(&c->links64[p], (size_t)c->g.Vh * 72 * sizeof(double2)) != cudaSuccess ||
        cudaMalloc(&c->links32[p], (size_t)c->g.Vh * 72 * sizeof(float2)) != cudaSuccess) {
      cudaGetLastError();
      rc = DWF_ENOMEM;
      break;
    }
    const long long n = c->g.Vh * 8;
    k_build_links<<<(unsigned)((n + 255) / 256), 256, 0, st>>>((const double2*)Ud, c->links64[p],
                                                                c->links32[p], L[0], L[1], L[2], L[3], p);
  }
  if (rc == DWF_OK) {
    if (cudaMalloc(&c->dscal, S_NSCAL * sizeof(double)) != cudaSuccess ||
        cudaMallocHost(&c->hscal, (S_NSCAL + 1) * sizeof(double)) != cudaSuccess) {
      cudaGetLastError();
      rc = DWF_ENOMEM;
    }
  }
  if (rc == DWF_OK) rc = dwf_reserve_partials(c, 1 << 16);
  if (rc == DWF_OK) {
    c->wait_flag = (int*)(c->hscal + S_NSCAL);
    *c->wait_flag = 0;
  }
  cudaError_t e = cudaStreamSynchronize(st);
  if (tmp) cudaFree(tmp);
  if (rc == DWF_OK && e != cudaSuccess) rc = DWF_ECUDA;
  if (rc != DWF_OK) {
    dwf_ctx_destroy(c);
    return rc;
  }
  *out = c;
  return DWF_OK;
}

// A context on the same lattice and links with another fifth-dimension
// extent (used to apply the 4D hopping term to a batch of ls 4D fields stored
// as the s-slices of one field).
int dwf_ctx_clone_ls(const dwf_ctx* src, int ls, dwf_ctx** out, cudaStream_t st) {
  *out = nullptr;
  if (ls != 4 && ls != 8 && ls != 16 && ls != 24) return DWF_EINVAL;
  dwf_ctx* c = new (std::nothrow) dwf_ctx();
  if (!c) return DWF_ENOMEM;
  c->g = src->g;
  c->g.Ls = ls;
  c->M5 = src->M5;
  c->device = src->device;
  c->sms = src->sms;
  int rc = DWF_OK;
  const size_t lb = (size_t)c->g.Vh * 72;
  for (int p = 0; p < 2 && rc == DWF_OK; p++) {
    if (cudaMalloc(&c->links64[p], lb * sizeof(double2)) != cudaSuccess ||
        cudaMalloc(&c->links32[p], lb * sizeof(float2)) != cudaSuccess) {
      cudaGetLastError();
      rc = DWF_ENOMEM;
      break;
    }
    if (cudaMemcpyAsync(c->links64[p], src->links64[p], lb * sizeof(double2), cudaMemcpyDeviceToDevice, st) !=
            cudaSuccess ||
        cudaMemcpyAsync(c->links32[p], src->links32[p], lb * sizeof(float2), cudaMemcpyDeviceToDevice, st) !=
            cudaSuccess)
      rc = DWF_ECUDA;
  }
  if (rc == DWF_OK && (cudaMalloc(&c->dscal, S_NSCAL * sizeof(double)) != cudaSuccess ||
                       cudaMallocHost(&c->hscal, S_NSCAL * sizeof(double)) != cudaSuccess)) {
    cudaGetLastError();
    rc = DWF_ENOMEM;
  }
  if (rc == DWF_OK) rc = dwf_reserve_partials(c, 1 << 16);
  c->wait_flag = src->wait_flag;  // (a clone lives within one call on its source)
  if (rc == DWF_OK && cudaStreamSynchronize(st) != cudaSuccess) rc = DWF_ECUDA;
  if (rc != DWF_OK) {
    dwf_ctx_destroy(c);
    return rc;
  }
  *out = c;
  return DWF_OK;
}

extern "C" int dwf_ctx_destroy(dwf_ctx* c) {
  if (!c) return DWF_OK;
  for (int p = 0; p < 2; p++) {
    if (c->links64[p]) cudaFree(c->links64[p]);
    if (c->links32[p]) cudaFree(c->links32[p]);
  }
  for (int i = 0; i < DWF_NWS; i++)
    if (c->ws[i]) cudaFree(c->ws[i]);
  if (c->partials) cudaFree(c->partials);
  if (c->dscal) cudaFree(c->dscal);
  if (c->hscal) cudaFreeHost(c->hscal);
  delete c;
  return DWF_OK;
}

extern "C" int64_t dwf_half_sites(const dwf_ctx* c) { return c ? c->g.Vh : 0; }
extern "C" int64_t dwf_half_bytes(const dwf_ctx* c, int prec) {
  return c ? c->g.Vh * 12 * c->g.Ls * (int64_t)dwf_complex_bytes(prec) : 0;
}

static int64_t half_elems(const dwf_ctx* c) { return c->g.Vh * 12 * c->g.Ls; }

// ------------------------------------------------------------------ launchers
static void fill_fifth(const dwf_ctx* c, dwfk::HopParams& hp, const double* mf, int nrhs) {
  const double d = 5.0 - c->M5;
  hp.d = d;
  hp.one_sweep = fabs(d) >= 1.0;
  for (int r = 0; r < nrhs && r < DWF_MAX_RHS; r++) {
    const double m = mf ? mf[r] : 0.0;
    const double md = m * pow(d, -(double)c->g.Ls);
    hp.m[r] = m;
    hp.kappa[r] = 1.0 / (1.0 + md);
    if (!(fabs(md) <= 1.0)) hp.one_sweep = 0;
    hp.dls1[r] = pow(d, 1.0 - (double)c->g.Ls);
  }
}

int dwf_wait_status(dwf_ctx* c) {
  volatile int* f = c->wait_flag;
  if (!*f) return DWF_OK;
  *f = 0;
  return dwf_fail(c, DWF_ETIMEOUT, "a bounded wait of a hopping launch gave up: its output is incomplete");
}

extern "C" int dwf_status(dwf_ctx* c, void* stream) {
  if (!c) return DWF_EINVAL;
  DWF_CUDA(c, cudaStreamSynchronize((cudaStream_t)stream));
  return dwf_wait_status(c);
}

extern "C" int dwf_selftest_raise_timeout(dwf_ctx* c, void* stream) {
  if (!c) return DWF_EINVAL;
  DWF_CUDA(c, cudaLaunchHostFunc((cudaStream_t)stream, [](void* f) { *(volatile int*)f = 1; }, c->wait_flag));
  return DWF_OK;
}

int launch_hop(dwf_ctx* c, const HopLaunch& h, int prec, cudaStream_t st, int* nblocks) {
  if (h.nrhs < 1 || h.nrhs > DWF_MAX_RHS) return dwf_fail(c, DWF_EINVAL, "nrhs out of range");
  dwfk::HopParams hp;
  memset(&hp, 0, sizeof(hp));
  hp.out = h.out;
  hp.in = h.in;
  hp.aux = h.aux;
  const int po = h.out_parity;
  hp.links = (prec == DWF_F64) ? (const void*)c->links64[po] : (const void*)c->links32[po];
  hp.L0 = c->g.L[0];
  hp.L1 = c->g.L[1];
  hp.L2 = c->g.L[2];
  hp.L3 = c->g.L[3];
  hp.Lxh = c->g.Lxh;
  hp.Vh = (int)c->g.Vh;
  hp.sms = c->sms;
  {
    // z-chunk: the largest even divisor of Lz whose input slab (zc planes of
    // one time slice, over the t-1, t, t+1 slices plus the output) stays
    // within the L2 budget (48 MB unless the autotuner chose another); the
    // whole Lz (lexicographic order) when it fits.
    const double budget = c->hop_l2_budget[prec] > 0 ? c->hop_l2_budget[prec] : 48e6;
    const double plane = (double)c->g.L[1] * c->g.Lxh * c->g.Ls * h.nrhs * 12.0 * dwf_complex_bytes(prec);
    int zc = c->g.L[2];
    if (4.0 * plane * zc > budget) {
      zc = 2;
      for (int q = 2; q <= c->g.L[2]; q += 2)
        if (c->g.L[2] % q == 0 && 4.0 * plane * q <= budget) zc = q;
    }
    hp.zc = zc;
  }
  hp.out_parity = po;
  hp.sg = h.dagger ? -1.f : 1.f;
  hp.alpha = h.alpha;
  hp.aux_mode = h.aux_mode;
  hp.inv_mode = h.inv_mode;
  hp.g5r5 = h.g5r5;
  hp.reduce = h.reduce;
  hp.rhs_stride = h.rhs_stride ? h.rhs_stride : half_elems(c);
  fill_fifth(c, hp, h.mf, h.nrhs);
  if (h.reduce) {
    const size_t nb = dwfk::hop_partials(prec, c->g.Vh, c->g.Ls, h.nrhs, dwfk::hop_sms(hp));
    int rc = dwf_reserve_partials(c, nb);
    if (rc) return rc;
  }
  hp.partials = c->partials;
  hp.wait_err = c->wait_flag;
  if (int rc = dwf_wait_status(c)) return rc;
  if (h.cheb_tp) {
    hp.cheb_mode = 1;
    hp.cheb_x = h.cheb_x;
    hp.cheb_tp = h.cheb_tp;
    hp.cheb_acc = h.cheb_acc;
    hp.cheb_ta = h.cheb_ta;
    hp.cheb_tb = h.cheb_tb;
    hp.cheb_cacc = h.cheb_cacc;
  }
  if (h.cg_x) {
    hp.cg_mode = 1;
    hp.cg_x = h.cg_x;
    hp.cg_r = h.cg_r;
    hp.cg_p = h.cg_p;
    hp.cg_alpha = h.cg_alpha;
    hp.cg_astride = h.cg_alpha_stride;
    hp.cg_x32 = h.cg_x32;
  }
  int rc;
  bool streamed = false;
  switch (prec) {
    case DWF_F64:
      rc = c->f64_arith == DWF_ARITH_FLOAT_FLOAT ? dwf_launch_hop_df(hp, c->g.Ls, h.nrhs, c->hop_variant[0], st, nblocks)
                                                 : dwf_launch_hop_f64(hp, c->g.Ls, h.nrhs, c->hop_variant[0], st, nblocks);
      break;
    case DWF_F32:
      rc = dwf_launch_hop_f32(hp, c->g.Ls, h.nrhs, c->hop_variant[1], c->hop_scalar[1], st, nblocks, &streamed);
      break;
    case DWF_F16S:
      rc = dwf_launch_hop_f16(hp, c->g.Ls, h.nrhs, c->hop_variant[2], c->hop_scalar[2], st, nblocks, &streamed);
      break;
    default:
      return dwf_fail(c, DWF_EINVAL, "bad precision");
  }
  if (rc) return dwf_fail(c, rc, "unsupported Ls");
  c->launches++;
  c->streamed += streamed;
  const double w = (double)dwf_complex_bytes(prec), wl = prec == DWF_F64 ? 16.0 : 8.0;
  c->hop_bytes += (double)c->g.Vh * ((double)c->g.Ls * h.nrhs * (24.0 + (h.aux_mode ? 12.0 : 0.0)) * w +
                                     72.0 * wl);
  return DWF_OK;
}

// ------------------------------------------------------------------ autotuner
// A variant whose CTAs cover several y-rows needs the x segment to divide
// Lx/2 and the row count to divide Ly.
static bool hop_variant_fits(const dwf_ctx* c, int prec, int v) {
  if (prec == DWF_F64 || c->g.Ls < 16) return true;  // always the plain kernel
  const int ry = dwfk::hop_variant_rows(v);
  const int sb = c->g.Ls >= 16 ? 8 : 128 / c->g.Ls;
  return ry == 1 || (c->g.Lxh % sb == 0 && c->g.L[1] % ry == 0);
}

extern "C" int dwf_set_f64_arithmetic(dwf_ctx* c, int mode) {
  if (!c || (mode != DWF_ARITH_FP64 && mode != DWF_ARITH_FLOAT_FLOAT)) return DWF_EINVAL;
  c->f64_arith = mode;
  return DWF_OK;
}

extern "C" int dwf_get_f64_arithmetic(const dwf_ctx* c) { return c ? c->f64_arith : DWF_EINVAL; }

extern "C" int dwf_set_hop_variant(dwf_ctx* c, int prec, int variant) {
  if (!c || prec < DWF_F64 || prec > DWF_F16S || variant < 0 || variant >= DWF_HOP_VARIANTS) return DWF_EINVAL;
  if (!hop_variant_fits(c, prec, variant)) return dwf_fail(c, DWF_EINVAL, "hop variant does not tile the lattice");
  c->hop_variant[prec] = variant;
  c->hop_scalar[prec] = 0;
  return DWF_OK;
}

extern "C" int dwf_get_hop_variant(const dwf_ctx* c, int prec) {
  if (!c || prec < DWF_F64 || prec > DWF_F16S) return DWF_EINVAL;
  return c->hop_variant[prec];
}

extern "C" int dwf_set_hop_scalar_variant(dwf_ctx* c, int prec, int variant) {
  if (!c || prec < DWF_F64 || prec > DWF_F16S || variant < 0 || variant >= DWF_HOP_VARIANTS) return DWF_EINVAL;
  if (!hop_variant_fits(c, prec, variant)) return dwf_fail(c, DWF_EINVAL, "hop variant does not tile the lattice");
  c->hop_scalar[prec] = variant;
  return DWF_OK;
}

extern "C" int dwf_get_hop_scalar_variant(const dwf_ctx* c, int prec) {
  if (!c || prec < DWF_F64 || prec > DWF_F16S) return DWF_EINVAL;
  return c->hop_scalar[prec];
}

// Times `reps` plain D_hop launches of the context's present choice after one
// to warm up; *streamed: the streaming kernel took them.
static int time_hop(dwf_ctx* c, void* out, const void* in, int prec, int reps, cudaEvent_t e0, cudaEvent_t e1, float* ms,
                    bool* streamed, cudaStream_t st) {
  HopLaunch h;
  memset(&h, 0, sizeof(h));
  h.out = out;
  h.in = in;
  h.nrhs = 1;
  h.alpha = 1.0;
  const int64_t s0 = c->streamed;
  int rc = launch_hop(c, h, prec, st, nullptr);
  if (rc) return rc;
  *streamed = c->streamed != s0;
  DWF_CUDA(c, cudaEventRecord(e0, st));
  for (int r = 0; r < reps; r++) {
    rc = launch_hop(c, h, prec, st, nullptr);
    if (rc) return rc;
  }
  DWF_CUDA(c, cudaEventRecord(e1, st));
  DWF_CUDA(c, cudaEventSynchronize(e1));
  DWF_CUDA(c, cudaEventElapsedTime(ms, e0, e1));
  *ms /= reps;
  return DWF_OK;
}

// The choice by time.  Launches that the streaming kernel does not take (those
// that end in a CG or Chebyshev step above all) are left to the fastest variant
// that does not stream, and the L2 budget is that of the launches that walk the
// lattice by it (the streaming kernel does not).
static int tune_hop(dwf_ctx* c, void* out, const void* in, int prec, int reps, cudaEvent_t e0, cudaEvent_t e1, float* best_ms,
                    cudaStream_t st) {
  // FP64: one kernel, or four register caps of the float-float kernel
  const int nv = c->g.Ls < 16 ? 1 : prec == DWF_F64 ? (c->f64_arith == DWF_ARITH_FLOAT_FLOAT ? 4 : 1) : DWF_HOP_VARIANTS;
  int best = 0, best_scalar = 0;
  float t_best = 1e30f, t_scalar = 1e30f;
  bool best_streams = false;
  c->hop_scalar[prec] = 0;
  for (int v = 0; v < nv; v++) {
    if (!hop_variant_fits(c, prec, v)) continue;
    c->hop_variant[prec] = v;
    float ms = 0;
    bool streamed = false;
    int rc = time_hop(c, out, in, prec, reps, e0, e1, &ms, &streamed, st);
    if (rc) return rc;
    if (ms < t_best) {
      t_best = ms;
      best = v;
      best_streams = streamed;
    }
    if (!streamed && ms < t_scalar) {
      t_scalar = ms;
      best_scalar = v;
    }
  }
  // then the L2 budget of the z-chunked traversal for the chosen variant
  c->hop_variant[prec] = best_scalar;
  const double budgets[5] = {48e6, 16e6, 32e6, 80e6, 120e6};
  double best_budget = 48e6;
  for (int bi = 1; bi < 5 && nv > 1; bi++) {
    c->hop_l2_budget[prec] = budgets[bi];
    float ms = 0;
    bool streamed = false;
    int rc = time_hop(c, out, in, prec, reps, e0, e1, &ms, &streamed, st);
    if (rc) return rc;
    if (ms < 0.98f * t_scalar) {  // a clear gain over the default
      t_scalar = ms;
      best_budget = budgets[bi];
    }
  }
  c->hop_l2_budget[prec] = best_budget;
  if (t_scalar < t_best) best_streams = false;
  c->hop_variant[prec] = best_streams ? best : best_scalar;
  c->hop_scalar[prec] = best_streams ? best_scalar : 0;
  *best_ms = best_streams ? t_best : t_scalar;
  return DWF_OK;
}

extern "C" int dwf_autotune(dwf_ctx* c, int prec, int reps, double* best_ms, void* stream) {
  if (!c || prec < DWF_F64 || prec > DWF_F16S || reps < 1) return DWF_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  const size_t bytes = (size_t)dwf_half_bytes(c, prec);
  void* a = dwf_workspace(c, 30, bytes);
  void* b = dwf_workspace(c, 31, bytes);
  if (!a || !b) return dwf_fail(c, DWF_ENOMEM, "autotune workspace");
  DWF_CUDA(c, cudaMemsetAsync(a, 0, bytes, st));
  cudaEvent_t e0, e1;
  DWF_CUDA(c, cudaEventCreate(&e0));
  DWF_CUDA(c, cudaEventCreate(&e1));
  const int64_t launches0 = c->launches, streamed0 = c->streamed;
  const double bytes0 = c->hop_bytes, budget0 = c->hop_l2_budget[prec];
  const int variant0 = c->hop_variant[prec], scalar0 = c->hop_scalar[prec];
  float best_t = 0;
  const int rc = tune_hop(c, b, a, prec, reps, e0, e1, &best_t, st);
  if (rc) {  // the choice stays what it was
    c->hop_variant[prec] = variant0;
    c->hop_scalar[prec] = scalar0;
    c->hop_l2_budget[prec] = budget0;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  c->launches = launches0;  // tuning launches are not counted
  c->hop_bytes = bytes0;
  c->streamed = streamed0;
  // the two tuning fields are released (at 48^3 x 96 x 24 they are 24 GB)
  DWF_CUDA(c, cudaStreamSynchronize(st));
  for (int slot = 30; slot <= 31; slot++) {
    if (c->ws[slot]) cudaFree(c->ws[slot]);
    c->ws[slot] = nullptr;
    c->ws_bytes[slot] = 0;
  }
  if (rc) return rc;
  if (best_ms) *best_ms = best_t;
  DWF_CUDA(c, cudaGetLastError());
  return dwf_wait_status(c);
}

extern "C" int dwf_counters(const dwf_ctx* c, int64_t* launches, double* hop_bytes) {
  if (!c) return DWF_EINVAL;
  if (launches) *launches = c->launches;
  if (hop_bytes) *hop_bytes = c->hop_bytes;
  return DWF_OK;
}

extern "C" int dwf_streamed_launches(const dwf_ctx* c, int64_t* launches) {
  if (!c || !launches) return DWF_EINVAL;
  *launches = c->streamed;
  return DWF_OK;
}

extern "C" int dwf_reset_counters(dwf_ctx* c) {
  if (!c) return DWF_EINVAL;
  c->launches = 0;
  c->hop_bytes = 0;
  c->streamed = 0;
  return DWF_OK;
}

int launch_mooee(dwf_ctx* c, void* out, const void* in, const double* mf, int dagger, int inverse,
                 int prec, int nrhs, int64_t rhs_stride, cudaStream_t st) {
  if (nrhs < 1 || nrhs > DWF_MAX_RHS) return dwf_fail(c, DWF_EINVAL, "nrhs out of range");
  dwfk::HopParams hp;
  memset(&hp, 0, sizeof(hp));
  hp.Vh = (int)c->g.Vh;
  fill_fifth(c, hp, mf, nrhs);
  const long long rs = rhs_stride ? rhs_stride : half_elems(c);
  int rc;
  switch (prec) {
    case DWF_F64:
      rc = dwf_launch_mooee_f64(out, in, hp, dagger, inverse, c->g.Ls, nrhs, rs, st);
      break;
    case DWF_F32:
      rc = dwf_launch_mooee_f32(out, in, hp, dagger, inverse, c->g.Ls, nrhs, rs, st);
      break;
    case DWF_F16S:
      rc = dwf_launch_mooee_f16(out, in, hp, dagger, inverse, c->g.Ls, nrhs, rs, st);
      break;
    default:
      return dwf_fail(c, DWF_EINVAL, "bad precision");
  }
  if (rc) return dwf_fail(c, rc, "unsupported Ls");
  c->launches++;
  return DWF_OK;
}

// ------------------------------------------------------------------ argument checks
static int check_fields(dwf_ctx* c, int prec, int nrhs, std::initializer_list<const void*> ptrs) {
  if (!c) return DWF_EINVAL;
  if (prec < DWF_F64 || prec > DWF_F16S) return dwf_fail(c, DWF_EINVAL, "bad precision");
  if (nrhs < 1 || nrhs > DWF_MAX_RHS) return dwf_fail(c, DWF_EINVAL, "nrhs out of range");
  for (const void* p : ptrs) {
    if (!p) return dwf_fail(c, DWF_EINVAL, "null field pointer");
    if (((uintptr_t)p) & 15) return dwf_fail(c, DWF_EINVAL, "field pointer not 16-byte aligned");
  }
  return DWF_OK;
}

static HopLaunch hop_base(void* out, const void* in, int po, int dag, int nrhs, double alpha) {
  HopLaunch h;
  memset(&h, 0, sizeof(h));
  h.out = out;
  h.in = in;
  h.out_parity = po;
  h.dagger = dag;
  h.nrhs = nrhs;
  h.alpha = alpha;
  return h;
}

// ------------------------------------------------------------------ operators
extern "C" int dwf_dhop(dwf_ctx* c, void* out, const void* in, int out_parity, int dagger, int prec,
                        int nrhs, void* stream) {
  int rc = check_fields(c, prec, nrhs, {out, in});
  if (rc) return rc;
  if (out_parity != 0 && out_parity != 1) return dwf_fail(c, DWF_EINVAL, "bad parity");
  HopLaunch h = hop_base(out, in, out_parity, dagger ? 1 : 0, nrhs, 1.0);
  rc = launch_hop(c, h, prec, (cudaStream_t)stream, nullptr);
  if (rc) return rc;
  DWF_CUDA(c, cudaGetLastError());
  return DWF_OK;
}

static int mooee_common(dwf_ctx* c, void* out, const void* in, double mf, int dagger, int inverse,
                        int prec, int nrhs, void* stream) {
  int rc = check_fields(c, prec, nrhs, {out, in});
  if (rc) return rc;
  std::vector<double> m(nrhs, mf);
  rc = launch_mooee(c, out, in, m.data(), dagger ? 1 : 0, inverse, prec, nrhs, 0, (cudaStream_t)stream);
  if (rc) return rc;
  DWF_CUDA(c, cudaGetLastError());
  return DWF_OK;
}

extern "C" int dwf_mooee(dwf_ctx* c, void* out, const void* in, double mf, int dagger, int prec,
                         int nrhs, void* stream) {
  return mooee_common(c, out, in, mf, dagger, 0, prec, nrhs, stream);
}

extern "C" int dwf_mooee_inv(dwf_ctx* c, void* out, const void* in, double mf, int dagger, int prec,
                             int nrhs, void* stream) {
  return mooee_common(c, out, in, mf, dagger, 1, prec, nrhs, stream);
}

// M_pc (dagger=0) or M_pc^dag (dagger=1) on nrhs even fields, odd temporary tmp.
// M_pc    = M_ee + 1/2 D_eo M_oo^-1 (-1/2 D_oe)
// M_pc^dag = M_ee^dag + 1/2 D^dag_eo M_oo^-dag (-1/2 D^dag_oe)
int mpc_apply(dwf_ctx* c, void* out, const void* in, void* tmp, const double* mf, int dagger,
                     int prec, int nrhs, int reduce, cudaStream_t st, int* nparts) {
  HopLaunch h1 = hop_base(tmp, in, 1, dagger, nrhs, -0.5);
  h1.inv_mode = dagger ? 2 : 1;
  h1.mf = mf;
  int rc = launch_hop(c, h1, prec, st, nullptr);
  if (rc) return rc;
  HopLaunch h2 = hop_base(out, tmp, 0, dagger, nrhs, 0.5);
  h2.aux = in;
  h2.aux_mode = dagger ? 3 : 2;
  h2.mf = mf;
  h2.reduce = reduce;
  return launch_hop(c, h2, prec, st, nparts);
}

// The second Schur form of Table 5, M2 = 1 - M_ee^-1 M_eo M_oo^-1 M_oe =
// M_ee^-1 M_pc: the second hopping launch of M_pc ends with M_ee^-1 in its
// epilogue, M_ee^-1 (M_ee in + 1/2 D_eo tmp).  reduce: |out|^2 partials.
static int mpc2_apply(dwf_ctx* c, void* out, const void* in, void* tmp, const double* mf, int prec, int nrhs,
                      int reduce, cudaStream_t st, int* nparts) {
  HopLaunch h1 = hop_base(tmp, in, 1, 0, nrhs, -0.5);
  h1.inv_mode = 1;
  h1.mf = mf;
  int rc = launch_hop(c, h1, prec, st, nullptr);
  if (rc) return rc;
  HopLaunch h2 = hop_base(out, tmp, 0, 0, nrhs, 0.5);
  h2.aux = in;
  h2.aux_mode = 2;
  h2.inv_mode = 1;
  h2.mf = mf;
  h2.reduce = reduce;
  return launch_hop(c, h2, prec, st, nparts);
}

// M_ee^-dag M_ee^-1 v in place (one field of precision prec): the factor that
// turns M_pc^dag into M2^dag M_ee^-1 (M2^dag = M_pc^dag M_ee^-dag).
static int mee_inv_pair(dwf_ctx* c, void* v, const double* mf, int prec, cudaStream_t st) {
  int rc = launch_mooee(c, v, v, mf, 0, 1, prec, 1, 0, st);
  if (rc) return rc;
  return launch_mooee(c, v, v, mf, 1, 1, prec, 1, 0, st);
}

enum { WS_TMP_O = 0, WS_TMP_E = 1 };

extern "C" int dwf_mpc(dwf_ctx* c, void* out, const void* in, double mf, int dagger, int prec, int nrhs,
                       void* stream) {
  int rc = check_fields(c, prec, nrhs, {out, in});
  if (rc) return rc;
  if (out == in) return dwf_fail(c, DWF_EINVAL, "out must not alias in");
  const size_t bytes = (size_t)dwf_half_bytes(c, prec) * nrhs;
  void* tmp = dwf_workspace(c, WS_TMP_O, bytes);
  if (!tmp) return dwf_fail(c, DWF_ENOMEM, "workspace");
  std::vector<double> m(nrhs, mf);
  rc = mpc_apply(c, out, in, tmp, m.data(), dagger ? 1 : 0, prec, nrhs, 0, (cudaStream_t)stream, nullptr);
  if (rc) return rc;
  DWF_CUDA(c, cudaGetLastError());
  return DWF_OK;
}

extern "C" int dwf_mpcdag_mpc(dwf_ctx* c, void* out, const void* in, double mf, int prec, int nrhs,
                              void* stream) {
  int rc = check_fields(c, prec, nrhs, {out, in});
  if (rc) return rc;
  if (out == in) return dwf_fail(c, DWF_EINVAL, "out must not alias in");
  const size_t bytes = (size_t)dwf_half_bytes(c, prec) * nrhs;
  void* tmp = dwf_workspace(c, WS_TMP_O, bytes);
  void* y = dwf_workspace(c, WS_TMP_E, bytes);
  if (!tmp || !y) return dwf_fail(c, DWF_ENOMEM, "workspace");
  std::vector<double> m(nrhs, mf);
  cudaStream_t st = (cudaStream_t)stream;
  rc = mpc_apply(c, y, in, tmp, m.data(), 0, prec, nrhs, 0, st, nullptr);
  if (rc) return rc;
  rc = mpc_apply(c, out, y, tmp, m.data(), 1, prec, nrhs, 0, st, nullptr);
  if (rc) return rc;
  DWF_CUDA(c, cudaGetLastError());
  return DWF_OK;
}

// Full-lattice D_DW (or D_DW^dag, or H_DW = Gamma_5 D_DW when g5 = 1) of nrhs full fields.
int ddw_apply(dwf_ctx* c, void* out, const void* in, const double* mf, int dagger, int g5, int prec,
              int nrhs, cudaStream_t st, const ChebFuse* cf) {
  const int64_t he = half_elems(c);
  const size_t cb = dwf_complex_bytes(prec);
  for (int po = 0; po < 2; po++) {
    HopLaunch h = hop_base(cf ? nullptr : (char*)out + po * he * cb, (const char*)in + (1 - po) * he * cb, po,
                           dagger, nrhs, -0.5);
    h.rhs_stride = 2 * he;
    h.aux = (const char*)in + po * he * cb;
    h.aux_mode = dagger ? 3 : 2;
    h.mf = mf;
    h.g5r5 = g5;
    if (cf) {
      h.cheb_x = (const char*)cf->x + po * he * cb;
      h.cheb_tp = (char*)cf->tp + po * he * cb;
      h.cheb_acc = cf->acc ? (char*)cf->acc + po * he * cb : nullptr;
      h.cheb_ta = cf->ta;
      h.cheb_tb = cf->tb;
      h.cheb_cacc = cf->cacc;
    }
    int rc = launch_hop(c, h, prec, st, nullptr);
    if (rc) return rc;
  }
  return DWF_OK;
}

extern "C" int dwf_ddw(dwf_ctx* c, void* out, const void* in, double mf, int dagger, int prec, int nrhs,
                       void* stream) {
  int rc = check_fields(c, prec, nrhs, {out, in});
  if (rc) return rc;
  if (out == in) return dwf_fail(c, DWF_EINVAL, "out must not alias in");
  std::vector<double> m(nrhs, mf);
  rc = ddw_apply(c, out, in, m.data(), dagger ? 1 : 0, 0, prec, nrhs, (cudaStream_t)stream);
  if (rc) return rc;
  DWF_CUDA(c, cudaGetLastError());
  return DWF_OK;
}

extern "C" int dwf_hdw(dwf_ctx* c, void* out, const void* in, double mf, int prec, int nrhs,
                       void* stream) {
  int rc = check_fields(c, prec, nrhs, {out, in});
  if (rc) return rc;
  if (out == in) return dwf_fail(c, DWF_EINVAL, "out must not alias in");
  std::vector<double> m(nrhs, mf);
  rc = ddw_apply(c, out, in, m.data(), 0, 1, prec, nrhs, (cudaStream_t)stream);
  if (rc) return rc;
  DWF_CUDA(c, cudaGetLastError());
  return DWF_OK;
}

// ------------------------------------------------------------------ reductions (host results)
int read_scalars(dwf_ctx* c, int first, int n, cudaStream_t st) {
  DWF_CUDA(c, cudaMemcpyAsync(c->hscal + first, c->dscal + first, n * sizeof(double),
                              cudaMemcpyDeviceToHost, st));
  DWF_CUDA(c, cudaStreamSynchronize(st));
  return dwf_wait_status(c);
}

int norm2_dev(dwf_ctx* c, const void* a, int64_t n, int prec, int dst, cudaStream_t st) {
  int np = 0;
  int rc = blas_norm2_partials(c, a, n, prec, st, &np);
  if (rc) return rc;
  return blas_finalize(c, np, 1, dst, st);
}

extern "C" int dwf_norm2(dwf_ctx* c, double* result, const void* a, int64_t n, int prec, void* stream) {
  int rc = check_fields(c, prec, 1, {a});
  if (rc) return rc;
  if (!result || n < 0) return dwf_fail(c, DWF_EINVAL, "bad argument");
  cudaStream_t st = (cudaStream_t)stream;
  rc = norm2_dev(c, a, n, prec, S_TMP0, st);
  if (rc) return rc;
  rc = read_scalars(c, S_TMP0, 1, st);
  if (rc) return rc;
  *result = c->hscal[S_TMP0];
  return DWF_OK;
}

extern "C" int dwf_cdot(dwf_ctx* c, double* result2, const void* a, const void* b, int64_t n, int prec,
                        void* stream) {
  int rc = check_fields(c, prec, 1, {a, b});
  if (rc) return rc;
  if (!result2 || n < 0) return dwf_fail(c, DWF_EINVAL, "bad argument");
  cudaStream_t st = (cudaStream_t)stream;
  int np = 0;
  rc = blas_cdot_partials(c, a, b, n, prec, st, &np);
  if (rc) return rc;
  rc = blas_finalize(c, np, 2, S_TMP0, st);
  if (rc) return rc;
  rc = read_scalars(c, S_TMP0, 2, st);
  if (rc) return rc;
  result2[0] = c->hscal[S_TMP0];
  result2[1] = c->hscal[S_TMP0 + 1];
  return DWF_OK;
}

// ------------------------------------------------------------------ red-black CGNR
namespace {

struct Timer {
  std::chrono::steady_clock::time_point t0 = std::chrono::steady_clock::now();
  double sec() const {
    return std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
  }
};

}  // namespace

// Inner CG operator: Ap = M_pc^dag M_pc p, with |M_pc p|^2 = <p, A p> reduced
// into dscal[S_PAP] and alpha = rr / pAp computed on the device.
static int cg_apply(dwf_ctx* c, void* Ap, const void* p, void* y, void* todd, const double* mf, int prec,
                    cudaStream_t st) {
  int np = 0;
  int rc = mpc_apply(c, y, p, todd, mf, 0, prec, 1, 1, st, &np);
  if (rc) return rc;
  rc = blas_finalize_mode(c, np, 1, S_PAP, 1, st);
  if (rc) return rc;
  return mpc_apply(c, Ap, y, todd, mf, 1, prec, 1, 0, st, nullptr);
}

// One fused CG step: y = M_pc p (|y|^2 = <p, A p> -> alpha), then
// A p = M_pc^dag y whose last hopping launch updates x += alpha p,
// r -= alpha A p and reduces |r|^2 (A p is never stored); *nparts partials.
// Schur form 2 (form = 2): y = M2 p, then w = M_ee^-dag y in wtmp and A p =
// M_pc^dag w, so that A = M2^dag M2.
static int cg_step_fused(dwf_ctx* c, void* x, void* r, const void* p, void* y, void* todd, const double* mf,
                         int prec, cudaStream_t st, int* nparts, int form = 1, void* wtmp = nullptr) {
  int np = 0;
  int rc = form == 2 ? mpc2_apply(c, y, p, todd, mf, prec, 1, 1, st, &np)
                     : mpc_apply(c, y, p, todd, mf, 0, prec, 1, 1, st, &np);
  if (rc) return rc;
  rc = blas_finalize_mode(c, np, 1, S_PAP, 1, st);
  if (rc) return rc;
  if (form == 2) {
    rc = launch_mooee(c, wtmp, y, mf, 1, 1, prec, 1, 0, st);
    if (rc) return rc;
    y = wtmp;
  }
  HopLaunch h1 = hop_base(todd, y, 1, 1, 1, -0.5);
  h1.inv_mode = 2;
  h1.mf = mf;
  rc = launch_hop(c, h1, prec, st, nullptr);
  if (rc) return rc;
  HopLaunch h2 = hop_base(nullptr, todd, 0, 1, 1, 0.5);
  h2.aux = y;
  h2.aux_mode = 3;
  h2.mf = mf;
  h2.reduce = 1;
  h2.cg_x = x;
  h2.cg_r = r;
  h2.cg_p = p;
  h2.cg_alpha = c->dscal + S_ALPHA;
  h2.cg_x32 = prec == DWF_F16S;  // the FP16-storage CG accumulates x in FP32
  return launch_hop(c, h2, prec, st, nparts);
}

// A block of CG iterations captured once as a CUDA graph and replayed (on a
// private stream, ordered after and before the solver's stream by events);
// the library's launch and byte counters advance by the block's own counts
// at every replay.  If the capture cannot be made, the solve keeps plain
// launches (state -1).
struct CGGraph {
  cudaStream_t gs = nullptr;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  cudaGraphExec_t exec = nullptr;
  int64_t launches = 0, streamed = 0;
  double bytes = 0;
  int state = 0;  // 0: not built, 1: ready, -1: plain launches
  template <class F>
  void build(dwf_ctx* c, int n, F&& body) {
    state = -1;
    if (cudaStreamCreateWithFlags(&gs, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&e0, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&e1, cudaEventDisableTiming) != cudaSuccess) {
      cudaGetLastError();
      return;
    }
    const int64_t l0 = c->launches, s0 = c->streamed;
    const double b0 = c->hop_bytes;
    const std::string err_before = c->err;
    cudaGraph_t g = nullptr;
    if (cudaStreamBeginCapture(gs, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
      cudaGetLastError();
      return;
    }
    int rc = DWF_OK;
    for (int k = 0; k < n && rc == DWF_OK; k++) rc = body(gs);
    const cudaError_t ec = cudaStreamEndCapture(gs, &g);
    launches = c->launches - l0;
    streamed = c->streamed - s0;
    bytes = c->hop_bytes - b0;
    c->launches = l0;
    c->streamed = s0;
    c->hop_bytes = b0;
    if (rc || ec != cudaSuccess || !g || cudaGraphInstantiate(&exec, g, 0) != cudaSuccess) {
      if (g) cudaGraphDestroy(g);
      exec = nullptr;
      c->err = err_before;
      cudaGetLastError();
      return;
    }
    cudaGraphDestroy(g);
    state = 1;
  }
  int run(dwf_ctx* c, cudaStream_t st) {
    DWF_CUDA(c, cudaEventRecord(e0, st));
    DWF_CUDA(c, cudaStreamWaitEvent(gs, e0, 0));
    DWF_CUDA(c, cudaGraphLaunch(exec, gs));
    DWF_CUDA(c, cudaEventRecord(e1, gs));
    DWF_CUDA(c, cudaStreamWaitEvent(st, e1, 0));
    c->launches += launches;
    c->streamed += streamed;
    c->hop_bytes += bytes;
    return DWF_OK;
  }
  ~CGGraph() {
    if (gs) cudaStreamSynchronize(gs);
    if (exec) cudaGraphExecDestroy(exec);
    if (gs) cudaStreamDestroy(gs);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
  }
};

// CG on M_pc^dag M_pc x_e = rhs with FP64 reliable updates.  With bp set (the
// red-black solve) the stopping residual is the Schur residual |b'_e - M_pc x|
// / bnorm, which equals the full true residual after reconstruction; without
// it (normal-equation solve) it is |rhs - M^dag M x| / bnorm.  x_e holds the
// FP64 solution; the caller owns every buffer.
struct CGBufs {
  void *rhs, *bp, *rhi, *yhi, *ohi, *xlo, *rlo, *p, *Ap, *ylo, *olo;
};

static int cg_core(dwf_ctx* c, double2* x_e, const CGBufs& B, double bnorm, double tol, int maxiter, int plo,
                   const double* mfa, dwf_solve_stats& S, double& matmuls, cudaStream_t st, int form = 1) {
  const int64_t he = half_elems(c);
  const size_t b64 = he * 16, blo = he * dwf_complex_bytes(plo);
  int rc;
  DWF_CUDA(c, cudaMemsetAsync(x_e, 0, b64, st));
  void* xin = plo == DWF_F64 ? (void*)x_e : B.xlo;  // inner accumulator
  const double delta = 0.1;
  double true_res = 0, rr_hi = 0, rho = 1, rr_max = 0, rr_lo = 0;
  bool have_x = false;
  bool restart_p = false;  // next reliable update restarts the directions, p = r
  // FP16 storage keeps the inner system scaled: r_lo = r / sigma with sigma
  // = |r| / sqrt(n) at every reliable update, so that the stored components
  // are of order one (unscaled they would fall below FP16's range as the
  // residual shrinks); the inner correction is scaled back, x += sigma x_lo.
  // FP32 and FP64 inner precisions keep sigma = 1.
  const bool scaled = plo == DWF_F16S;
  double sigma = 1.0;
  // the inner x accumulates the scaled correction A^-1 r / sigma, whose
  // entries can exceed FP16's range (the low modes of M_pc^dag M_pc); it is
  // kept in FP32 when the other inner vectors are FP16
  const int px = scaled ? DWF_F32 : plo;
  void *rhi = B.rhi, *yhi = B.yhi, *ohi = B.ohi, *xlo = B.xlo, *rlo = B.rlo, *p = B.p, *Ap = B.Ap;

  auto reliable = [&]() -> int {
    int r;
    const double sigma_prev = sigma;
    const bool had_x = have_x;
    if (have_x && plo != DWF_F64) {
      r = blas_axpby(c, sigma, xlo, px, 1.0, x_e, DWF_F64, he, st);
      if (r) return r;
    }
    if (plo != DWF_F64) DWF_CUDA(c, cudaMemsetAsync(xlo, 0, he * dwf_complex_bytes(px), st));
    if (have_x) {
      // While the residual is far above FP32 rounding (true residual > 1e-4),
      // M_pc x is formed by the FP32 operator on x rounded to FP32 (error about
      // 1e-7 of |b|, three decades below the residual it corrects); below that
      // in FP64.  FP32 inner policy of the red-black solve only; the stopping
      // decision (true residual <= tol) is always taken on an FP64 residual.
      if (plo == DWF_F32 && B.bp && true_res > 1e-4) {
        r = blas_copy(c, B.ylo, DWF_F32, x_e, DWF_F64, he, st);
        if (r) return r;
        r = mpc_apply(c, B.Ap, B.ylo, B.olo, mfa, 0, DWF_F32, 1, 0, st, nullptr);
        if (r) return r;
        r = blas_copy(c, yhi, DWF_F64, B.Ap, DWF_F32, he, st);
      } else {
        r = mpc_apply(c, yhi, x_e, ohi, mfa, 0, DWF_F64, 1, 0, st, nullptr);
      }
      if (r) return r;
      if (B.bp) {
        // y = b'_e - M_pc x in FP64 (the true residual); r = M_pc^dag y only
        // steers the inner CG, so it is applied in the inner precision.
        r = blas_axpby(c, 1.0, B.bp, DWF_F64, -1.0, yhi, DWF_F64, he, st);
        if (r) return r;
        r = norm2_dev(c, yhi, he, DWF_F64, S_TMP2, st);
        if (r) return r;
        if (plo == DWF_F64) {
          if (form == 2) {  // r = M2^dag M_ee^-1 y = M_pc^dag M_ee^-dag M_ee^-1 y
            r = mee_inv_pair(c, yhi, mfa, DWF_F64, st);
            if (r) return r;
          }
          r = mpc_apply(c, rhi, yhi, ohi, mfa, 1, DWF_F64, 1, 0, st, nullptr);
        } else if (scaled) {  // M_pc^dag on y / sigma_y, scaled back into rhi
          r = read_scalars(c, S_TMP2, 1, st);
          if (r) return r;
          const double sy = sqrt(c->hscal[S_TMP2] / (double)he);
          if (!(sy > 0) || !isfinite(sy)) return dwf_fail(c, DWF_ENAN, "NaN in CG residual");
          r = blas_axpby(c, 1.0 / sy, yhi, DWF_F64, 0.0, B.ylo, plo, he, st);
          if (r) return r;
          r = mpc_apply(c, rlo, B.ylo, B.olo, mfa, 1, plo, 1, 0, st, nullptr);
          if (r) return r;
          r = blas_axpby(c, sy, rlo, plo, 0.0, rhi, DWF_F64, he, st);
        } else {
          r = blas_copy(c, B.ylo, plo, yhi, DWF_F64, he, st);
          if (r) return r;
          if (form == 2) {
            r = mee_inv_pair(c, B.ylo, mfa, plo, st);
            if (r) return r;
          }
          r = mpc_apply(c, rlo, B.ylo, B.olo, mfa, 1, plo, 1, 0, st, nullptr);
          if (r) return r;
          r = blas_copy(c, rhi, DWF_F64, rlo, plo, he, st);
        }
      } else {  // r = rhs - M^dag M x
        r = mpc_apply(c, rhi, yhi, ohi, mfa, 1, DWF_F64, 1, 0, st, nullptr);
        if (r) return r;
        r = blas_axpby(c, 1.0, B.rhs, DWF_F64, -1.0, rhi, DWF_F64, he, st);
        if (r) return r;
        r = norm2_dev(c, rhi, he, DWF_F64, S_TMP2, st);
      }
      if (r) return r;
      matmuls += 4;
    } else {
      r = blas_copy(c, rhi, DWF_F64, B.rhs, DWF_F64, he, st);
      if (r) return r;
      r = norm2_dev(c, B.bp ? B.bp : B.rhs, he, DWF_F64, S_TMP2, st);
      if (r) return r;
    }
    r = norm2_dev(c, rhi, he, DWF_F64, S_TMP3, st);
    if (r) return r;
    if (scaled) {
      r = read_scalars(c, S_TMP3, 1, st);
      if (r) return r;
      sigma = sqrt(c->hscal[S_TMP3] / (double)he);
      if (!isfinite(sigma)) return dwf_fail(c, DWF_ENAN, "NaN in CG residual");
      if (!(sigma > 0)) sigma = 1.0;  // exact solution: the inner solve is not entered
      r = blas_axpby(c, 1.0 / sigma, rhi, DWF_F64, 0.0, rlo, plo, he, st);
      if (r) return r;
      // FP16 vectors: the CG restarts from the new residual (p = r); the
      // direction carried over in FP16 loses conjugacy and can grow without
      // bound over many updates
      if (had_x) r = blas_copy(c, p, plo, rlo, plo, he, st);
      (void)sigma_prev;
    } else {
      r = blas_copy(c, rlo, plo, rhi, DWF_F64, he, st);
    }
    if (r) return r;
    r = norm2_dev(c, rlo, he, plo, S_RR, st);
    if (r) return r;
    // The next step length alpha = |r|^2 / <p, A p> assumes <r, p> = |r|^2,
    // which holds for the recursive residual but not for the recomputed one.
    // With p kept across the update (FP32 and FP64 inner vectors) it is
    // restored by p += (1 - <r, p> / |r|^2) r; without it the inner CG can
    // stall or diverge once the two residuals differ by more than rounding.
    const bool fix_p = had_x && !scaled && !restart_p;
    if (fix_p) {
      int np = 0;
      r = blas_cdot_partials(c, rlo, p, he, plo, st, &np);
      if (r) return r;
      r = blas_finalize(c, np, 2, S_TMP0, st);
      if (r) return r;
    }
    r = read_scalars(c, S_RR, S_TMP3 + 1 - S_RR, st);
    if (r) return r;
    if (fix_p && c->hscal[S_RR] > 0) {
      const double rr = c->hscal[S_RR];
      r = blas_caxpy(c, 1.0 - c->hscal[S_TMP0] / rr, -c->hscal[S_TMP1] / rr, rlo, plo, p, plo, he, st);
      if (r) return r;
    } else if (had_x && !scaled && restart_p) {
      r = blas_copy(c, p, plo, rlo, plo, he, st);
      if (r) return r;
    }
    restart_p = false;
    true_res = sqrt(c->hscal[S_TMP2]) / bnorm;
    rr_hi = c->hscal[S_TMP3];
    rho = rr_hi > 0 ? sqrt(c->hscal[S_TMP2] / rr_hi) : 1.0;
    rr_max = rr_hi;
    rr_lo = rr_hi;
    have_x = true;
    S.reliable_updates++;
    if (!isfinite(true_res) || !isfinite(rr_hi)) return dwf_fail(c, DWF_ENAN, "NaN in CG residual");
    return DWF_OK;
  };

  rc = reliable();
  if (rc) return rc;
  S.reliable_updates = 0;
  rc = blas_copy(c, p, plo, rlo, plo, he, st);
  if (rc) return rc;
  int it = 0, last_reliable_it = 0;
  const int check_every = 8;
  bool converged = true_res <= tol;
  // One CG iteration is a fixed launch sequence on fixed buffers whose step
  // lengths live in device scalars, so the check_every iterations between two
  // host checks are captured once as a CUDA graph (after the first block has
  // run with plain launches and sized every workspace) and replayed.
  CGGraph graph;
  auto one_iteration = [&](cudaStream_t s2) -> int {
    int np = 0;
    int r = cg_step_fused(c, xin, rlo, p, B.ylo, B.olo, mfa, plo, s2, &np, form, B.Ap);
    if (r) return r;
    r = blas_finalize_mode(c, np, 1, S_RRNEW, 2, s2);
    if (r) return r;
    return blas_cg_p(c, p, rlo, he, plo, S_BETA, s2);
  };
  while (!converged && it < maxiter) {
    if (it % check_every == 0 && it + check_every <= maxiter && it >= check_every && graph.state == 0)
      graph.build(c, check_every, one_iteration);
    if (it % check_every == 0 && it + check_every <= maxiter && graph.state == 1) {
      rc = graph.run(c, st);
      if (rc) return rc;
      matmuls += 4 * check_every;
      it += check_every;
      S.graph_replays++;
    } else {
      rc = one_iteration(st);
      if (rc) return rc;
      matmuls += 4;
      it++;
    }
    if (it % check_every == 0 || it == maxiter) {
      rc = read_scalars(c, S_RR, 1, st);
      if (rc) return rc;
      rr_lo = sigma * sigma * c->hscal[S_RR];  // in the units of rr_hi
      if (!isfinite(rr_lo)) return dwf_fail(c, DWF_ENAN, "NaN in CG residual");
      if (rr_lo > rr_max) rr_max = rr_lo;
      const double predicted = rho * sqrt(rr_lo) / bnorm;
      // a recursive residual grown a hundredfold above its value at the last
      // reliable update means the directions have lost conjugacy: update and
      // restart them
      const bool diverging = rr_lo > 1e4 * rr_hi;
      if (diverging) restart_p = true;
      // FP16 inner vectors also take a reliable update (a restart) every 64
      // iterations, in case their recursive residual stalls above delta
      if (rr_lo < delta * delta * rr_max || predicted <= tol || it == maxiter || diverging ||
          (scaled && it - last_reliable_it >= 64)) {
        last_reliable_it = it;
        rc = reliable();
        if (rc) return rc;
        converged = true_res <= tol;
        // the recurrence continues from the new residual: rr = |r_new|^2
      }
    }
  }
  S.iterations = it;
  S.true_residual = true_res;
  return DWF_OK;
}

// |b_e - (D x)_e|^2 into dscal[dst] and |b_o - (D x)_o|^2 into dscal[dst+1]
// for full FP64 fields x, b (FP64 D_DW at mass mfa[0]); te, to: half temporaries.
static int true_residual_halves(dwf_ctx* c, const void* x, const void* b, void* te, void* to, const double* mfa,
                                int dst, cudaStream_t st) {
  const int64_t he = half_elems(c);
  for (int po = 0; po < 2; po++) {
    void* t = po ? to : te;
    HopLaunch h = hop_base(t, (const double2*)x + (1 - po) * he, po, 0, 1, -0.5);
    h.aux = (const double2*)x + po * he;
    h.aux_mode = 2;
    h.mf = mfa;
    int rc = launch_hop(c, h, DWF_F64, st, nullptr);
    if (rc) return rc;
    rc = blas_axpby(c, 1.0, (const double2*)b + po * he, DWF_F64, -1.0, t, DWF_F64, he, st);
    if (rc) return rc;
    rc = norm2_dev(c, t, he, DWF_F64, dst + po, st);
    if (rc) return rc;
  }
  return DWF_OK;
}

// Red-black CGNR on Schur form `form` (1: M_pc, 2: M2 = M_ee^-1 M_pc).
static int rbcg_solve_form(dwf_ctx* c, void* x, const void* b, double mf, double tol, int maxiter, int policy,
                           dwf_solve_stats* stats, void* stream, int form) {
  Timer timer;
  if (!c || !x || !b) return DWF_EINVAL;
  if (!(tol > 0) || maxiter < 1) return dwf_fail(c, DWF_EINVAL, "bad tol or maxiter");
  if (policy < DWF_SOLVE_F64 || policy > DWF_SOLVE_MIXED_F16 || (form == 2 && policy == DWF_SOLVE_MIXED_F16))
    return dwf_fail(c, DWF_EINVAL, "bad policy");
  cudaStream_t st = (cudaStream_t)stream;
  const int plo = policy == DWF_SOLVE_F64 ? DWF_F64 : policy == DWF_SOLVE_MIXED_F16 ? DWF_F16S : DWF_F32;
  const int64_t he = half_elems(c);
  const size_t b64 = he * 16, blo = he * dwf_complex_bytes(plo);
  dwf_solve_stats S;
  memset(&S, 0, sizeof(S));

  const bool host_b = !dwf_is_device_ptr(b);
  const bool host_x = !dwf_is_device_ptr(x);
  const double2* db = (const double2*)b;
  double2* dx = (double2*)x;
  if (host_b) {
    void* w = dwf_workspace(c, WS_B, 2 * b64);
    if (!w) return dwf_fail(c, DWF_ENOMEM, "workspace");
    DWF_CUDA(c, cudaMemcpyAsync(w, b, 2 * b64, cudaMemcpyHostToDevice, st));
    db = (const double2*)w;
  }
  if (host_x) {
    void* w = dwf_workspace(c, WS_X, 2 * b64);
    if (!w) return dwf_fail(c, DWF_ENOMEM, "workspace");
    dx = (double2*)w;
  }
  if (((uintptr_t)db & 15) || ((uintptr_t)dx & 15)) return dwf_fail(c, DWF_EINVAL, "alignment");
  // Buffers that are never live at the same time share memory, so that the
  // solve fits one GPU at 48^3 x 96 x 24 (one FP64 half field: 24.5 GB):
  //  * rhs is read once, by the first reliable update, which copies it into rhi;
  //  * FP64 inner vectors: rlo is rhi's copy made at every reliable update, and
  //    the step temporaries ylo, olo are free while the reliable update uses
  //    yhi, ohi;
  //  * FP32 inner vectors: rhi is only the FP64 copy of rlo, formed after the
  //    reliable update is done with yhi; the FP32 M_pc x of an early update
  //    goes to rlo, which the update then recomputes;
  //  * Ap is needed only by the second Schur form (M_ee^-dag M2 p).
  // FP16-storage vectors keep separate buffers (rhi holds the unscaled residual).
  const bool f64 = plo == DWF_F64, f32 = plo == DWF_F32;
  void* bp = dwf_workspace(c, WS_BP, b64);
  void* yhi = dwf_workspace(c, WS_YHI, b64);
  void* ohi = dwf_workspace(c, WS_OHI, b64);
  void* rhi = f32 ? yhi : dwf_workspace(c, WS_RHI, b64);
  void* rhs = rhi;
  void* xlo = f64 ? nullptr : dwf_workspace(c, WS_XLO, plo == DWF_F16S ? he * 8 : blo);
  void* rlo = f64 ? rhi : dwf_workspace(c, WS_RLO, blo);
  void* p = dwf_workspace(c, WS_P, blo);
  void* ylo = f64 ? yhi : dwf_workspace(c, WS_YLO, blo);
  void* olo = f64 ? ohi : dwf_workspace(c, WS_OLO, blo);
  void* Ap = (form == 2 || plo == DWF_F16S) ? dwf_workspace(c, WS_AP, blo) : rlo;
  if (!bp || !rhs || !rhi || !yhi || !ohi || (!f64 && !xlo) || !rlo || !p || !Ap || !ylo || !olo)
    return dwf_fail(c, DWF_ENOMEM, "solver workspace");
  const double2* b_e = db;
  const double2* b_o = db + he;
  double2* x_e = dx;
  double2* x_o = dx + he;
  int rc;
  const double mfa[1] = {mf};
  double matmuls = 0;  // in half-lattice hopping terms; /4*2 at the end

  // |b|^2
  rc = norm2_dev(c, db, 2 * he, DWF_F64, S_TMP1, st);
  if (rc) return rc;
  rc = read_scalars(c, S_TMP1, 1, st);
  if (rc) return rc;
  const double bnorm = sqrt(c->hscal[S_TMP1]);
  if (!(bnorm > 0)) {
    DWF_CUDA(c, cudaMemsetAsync(dx, 0, 2 * b64, st));
    if (host_x) DWF_CUDA(c, cudaMemcpyAsync(x, dx, 2 * b64, cudaMemcpyDeviceToHost, st));
    DWF_CUDA(c, cudaStreamSynchronize(st));
    if (stats) *stats = S;
    return bnorm == 0 ? DWF_OK : dwf_fail(c, DWF_ENAN, "source is not finite");
  }

  // b'_e = b_e + 1/2 D_eo M_oo^-1 b_o
  rc = launch_mooee(c, ohi, b_o, mfa, 0, 1, DWF_F64, 1, 0, st);
  if (rc) return rc;
  {
    HopLaunch h = hop_base(bp, ohi, 0, 0, 1, 0.5);
    h.aux = b_e;
    h.aux_mode = 1;
    rc = launch_hop(c, h, DWF_F64, st, nullptr);
    if (rc) return rc;
  }
  // rhs = M_pc^dag b'_e (form 1) or M2^dag M_ee^-1 b'_e = M_pc^dag M_ee^-dag
  // M_ee^-1 b'_e (form 2; yhi is free here and is not rhs in that form)
  if (form == 2) {
    // with FP32 inner vectors rhs is yhi: the temporary is then x_e, which
    // the CG clears before its first use
    void* t = rhs == yhi ? (void*)x_e : yhi;
    DWF_CUDA(c, cudaMemcpyAsync(t, bp, b64, cudaMemcpyDeviceToDevice, st));
    rc = mee_inv_pair(c, t, mfa, DWF_F64, st);
    if (rc) return rc;
    rc = mpc_apply(c, rhs, t, ohi, mfa, 1, DWF_F64, 1, 0, st, nullptr);
  } else {
    rc = mpc_apply(c, rhs, bp, ohi, mfa, 1, DWF_F64, 1, 0, st, nullptr);
  }
  if (rc) return rc;
  matmuls += 3;

  CGBufs B = {rhs, bp, rhi, yhi, ohi, xlo, rlo, p, Ap, ylo, olo};
  rc = cg_core(c, x_e, B, bnorm, tol, maxiter, plo, mfa, S, matmuls, st, form);
  if (rc) return rc;


  // x_o = M_oo^-1 (b_o + 1/2 D_oe x_e)
  {
    HopLaunch h = hop_base(x_o, x_e, 1, 0, 1, 0.5);
    h.aux = b_o;
    h.aux_mode = 1;
    h.inv_mode = 1;
    h.mf = mfa;
    rc = launch_hop(c, h, DWF_F64, st, nullptr);
    if (rc) return rc;
  }
  matmuls += 1;
  // true residual ||b - D x|| / ||b|| in FP64, one parity at a time in the
  // half-field temporaries: (D x)_p = M_pp x_p - 1/2 D_hop x_{1-p}
  rc = true_residual_halves(c, dx, db, yhi, ohi, mfa, S_TMP2, st);
  if (rc) return rc;
  matmuls += 2;
  if (host_x) DWF_CUDA(c, cudaMemcpyAsync(x, dx, 2 * b64, cudaMemcpyDeviceToHost, st));
  rc = read_scalars(c, S_TMP2, 2, st);
  if (rc) return rc;
  S.true_residual = sqrt(c->hscal[S_TMP2] + c->hscal[S_TMP2 + 1]) / bnorm;
  S.fine_matmuls = matmuls / 2.0;
  S.seconds = timer.sec();
  S.status = S.true_residual <= tol ? DWF_OK : DWF_ENOCONV;
  DWF_CUDA(c, cudaGetLastError());
  if (stats) *stats = S;
  if (S.status == DWF_ENOCONV) return dwf_fail(c, DWF_ENOCONV, "maxiter reached before tol");
  return DWF_OK;
}

extern "C" int rbcg_solve(dwf_ctx* c, void* x, const void* b, double mf, double tol, int maxiter, int policy,
                          dwf_solve_stats* stats, void* stream) {
  return rbcg_solve_form(c, x, b, mf, tol, maxiter, policy, stats, stream, 1);
}

extern "C" int rbcg2_solve(dwf_ctx* c, void* x, const void* b, double mf, double tol, int maxiter, int policy,
                           dwf_solve_stats* stats, void* stream) {
  return rbcg_solve_form(c, x, b, mf, tol, maxiter, policy, stats, stream, 2);
}

extern "C" int rbcg_normal_solve(dwf_ctx* c, void* x, const void* phi, double mf, double tol, int maxiter,
                                 int policy, dwf_solve_stats* stats, void* stream) {
  Timer timer;
  if (!c || !x || !phi) return DWF_EINVAL;
  if (!(tol > 0) || maxiter < 1) return dwf_fail(c, DWF_EINVAL, "bad tol or maxiter");
  if (policy != DWF_SOLVE_F64 && policy != DWF_SOLVE_MIXED_F32) return dwf_fail(c, DWF_EINVAL, "bad policy");
  if (!dwf_is_device_ptr(x) || !dwf_is_device_ptr(phi)) return dwf_fail(c, DWF_EINVAL, "device buffers required");
  if (((uintptr_t)x & 15) || ((uintptr_t)phi & 15)) return dwf_fail(c, DWF_EINVAL, "alignment");
  cudaStream_t st = (cudaStream_t)stream;
  const int plo = policy == DWF_SOLVE_F64 ? DWF_F64 : DWF_F32;
  const int64_t he = half_elems(c);
  const size_t b64 = he * 16, blo = he * dwf_complex_bytes(plo);
  dwf_solve_stats S;
  memset(&S, 0, sizeof(S));
  CGBufs B;
  B.rhs = (void*)phi;
  B.bp = nullptr;
  B.rhi = dwf_workspace(c, WS_RHI, b64);
  B.yhi = dwf_workspace(c, WS_YHI, b64);
  B.ohi = dwf_workspace(c, WS_OHI, b64);
  B.xlo = plo == DWF_F64 ? nullptr : dwf_workspace(c, WS_XLO, blo);
  B.rlo = dwf_workspace(c, WS_RLO, blo);
  B.p = dwf_workspace(c, WS_P, blo);
  B.Ap = dwf_workspace(c, WS_AP, blo);
  B.ylo = dwf_workspace(c, WS_YLO, blo);
  B.olo = dwf_workspace(c, WS_OLO, blo);
  if (!B.rhi || !B.yhi || !B.ohi || (plo != DWF_F64 && !B.xlo) || !B.rlo || !B.p || !B.Ap || !B.ylo || !B.olo)
    return dwf_fail(c, DWF_ENOMEM, "solver workspace");
  int rc = norm2_dev(c, phi, he, DWF_F64, S_TMP1, st);
  if (rc) return rc;
  rc = read_scalars(c, S_TMP1, 1, st);
  if (rc) return rc;
  const double bnorm = sqrt(c->hscal[S_TMP1]);
  if (!(bnorm > 0)) {
    DWF_CUDA(c, cudaMemsetAsync(x, 0, b64, st));
    DWF_CUDA(c, cudaStreamSynchronize(st));
    if (stats) *stats = S;
    return bnorm == 0 ? DWF_OK : dwf_fail(c, DWF_ENAN, "source is not finite");
  }
  const double mfa[1] = {mf};
  double matmuls = 0;
  rc = cg_core(c, (double2*)x, B, bnorm, tol, maxiter, plo, mfa, S, matmuls, st);
  if (rc) return rc;
  DWF_CUDA(c, cudaStreamSynchronize(st));
  S.fine_matmuls = matmuls / 2.0;
  S.seconds = timer.sec();
  S.status = S.true_residual <= tol ? DWF_OK : DWF_ENOCONV;
  if (stats) *stats = S;
  if (S.status == DWF_ENOCONV) return dwf_fail(c, DWF_ENOCONV, "maxiter reached before tol");
  return DWF_OK;
}

// ------------------------------------------------------------------ power method
extern "C" int dwf_power_max(dwf_ctx* c, double* lmax, const void* v0, double mf, int iters, int prec,
                             void* stream) {
  int rc = check_fields(c, DWF_F64, 1, {v0});
  if (rc) return rc;
  if (!lmax || iters < 1) return dwf_fail(c, DWF_EINVAL, "bad argument");
  if (prec != DWF_F64 && prec != DWF_F32) return dwf_fail(c, DWF_EINVAL, "bad precision");
  cudaStream_t st = (cudaStream_t)stream;
  const int64_t n = 2 * half_elems(c);
  const size_t bytes = n * dwf_complex_bytes(prec);
  void* v = dwf_workspace(c, WS_FULL, bytes);
  void* w = dwf_workspace(c, WS_B, bytes);
  void* t = dwf_workspace(c, WS_X, bytes);
  if (!v || !w || !t) return dwf_fail(c, DWF_ENOMEM, "workspace");
  const double mfa[1] = {mf};
  rc = norm2_dev(c, v0, n, DWF_F64, S_TMP0, st);
  if (rc) return rc;
  rc = read_scalars(c, S_TMP0, 1, st);
  if (rc) return rc;
  double nv = sqrt(c->hscal[S_TMP0]);
  if (!(nv > 0)) return dwf_fail(c, DWF_EINVAL, "zero start vector");
  rc = blas_axpby(c, 1.0 / nv, v0, DWF_F64, 0.0, v, prec, n, st);
  if (rc) return rc;
  double lam = 0;
  for (int k = 0; k < iters; k++) {  // v <- A v / |A v|, lambda = <v, A v>
    rc = ddw_apply(c, t, v, mfa, 0, 0, prec, 1, st);
    if (rc) return rc;
    rc = ddw_apply(c, w, t, mfa, 1, 0, prec, 1, st);
    if (rc) return rc;
    int np = 0;
    rc = blas_cdot_partials(c, v, w, n, prec, st, &np);
    if (rc) return rc;
    rc = blas_finalize(c, np, 2, S_TMP0, st);
    if (rc) return rc;
    rc = norm2_dev(c, w, n, prec, S_TMP2, st);
    if (rc) return rc;
    rc = read_scalars(c, S_TMP0, 3, st);
    if (rc) return rc;
    lam = c->hscal[S_TMP0];
    const double nw = sqrt(c->hscal[S_TMP2]);
    if (!isfinite(nw) || !(nw > 0)) return dwf_fail(c, DWF_ENAN, "power method breakdown");
    rc = blas_axpby(c, 1.0 / nw, w, prec, 0.0, v, prec, n, st);
    if (rc) return rc;
  }
  DWF_CUDA(c, cudaStreamSynchronize(st));
  *lmax = lam;
  return DWF_OK;
}
