// Hopping term streamed along t through shared memory (arXiv:2103.05034,
// Sec. 2, Eq. 2), with the epilogues of hop_kernel (same HopParams) but the
// CG and Chebyshev steps.
//
// One persistent CTA per SM walks units: a 2 x 2 (y, z) tile of x-segments of
// up to SX checkerboard sites, all Ls slices, over a run of t.  Every input
// site of the tile is copied to shared memory once (tensor-map copies issued by
// one thread: a step is ten of them; the same rows as 24 to 36 plain bulk
// copies cost 60 ns each and bound the kernel) and read there as the t-1, in-slice and t+1 neighbour of
// three consecutive steps; only the halo rows are extra.  Per output site
// that is 3.25 (Ls 16, SX 4) or 3.5 (Ls 24, SX 2) site reads from L2 against
// 7 or more for a kernel whose CTAs read every neighbour row from global
// memory, and no read holds a register while it is in flight.
//
// Rings in shared memory: three slots of centre rows (slice t of the tile's
// four rows plus the one x-neighbour site outside the segment) and two slots
// of halo rows (the eight rows around the tile in y and z).  Two consumer
// groups take alternate steps, so that one group's epilogue (global loads,
// the fifth-dimension scan, stores) overlaps the other's arithmetic.  A step
// uses its halo rows first, so that theirs of the group's next step arrive
// during its second half, and the t+1 slice last: the slot that t-1 frees
// receives t+2, which has more than a step to arrive.
//
// A thread holds one s-slice of one site.  A site's slices sit on LPS lanes of
// a warp (Ls = 24: 8 lanes of each of three warps).
#pragma once

#include <cuda.h>

#include <type_traits>

#include "ring_roles.cuh"

namespace dwfk {

template <int P, int LS, int SXV>
struct StreamCfg {
  static constexpr int SX = SXV;                                  // sites per row of the tile
  static constexpr int SITES = 4 * SX;
  static constexpr int LPS = LS == 24 ? 8 : LS;                   // lanes per site and warp
  static constexpr int WPS = LS / LPS;                            // warps that share a site
  static constexpr int SPW = 32 / LPS;                            // sites per warp
  static constexpr int NTG = SITES * LS;                          // threads per consumer group
  static constexpr int NWG = NTG / 32;
  static constexpr int NG = 2;                                    // consumer groups
  // One producer warp; where it would be a seventeenth (a scheduler with five
  // warps caps a thread at 96 registers) the producer is a warpgroup that
  // hands registers to the consumers' four warpgroups (setmaxnreg: 512 x 112
  // + 128 x 32 of the 640 x 96 the block is launched with).
  static constexpr bool REGSPLIT = NG * NWG == 16;
  static constexpr int NT = NG * NTG + (REGSPLIT ? 128 : 32);
  static constexpr int CB = P == DWF_F32 ? 8 : 4;                 // stored bytes of a complex number
  // Records in shared memory: 12 rows of Ls numbers, the rows lengthened by 16
  // bytes (out-of-range elements of the copied box) where a site's lanes do
  // not fill a 128-byte access phase, which puts neighbouring sites half a
  // phase apart.
  static constexpr int RB = LS * CB + (LPS * CB == 128 ? 0 : 16);
  static constexpr int SS = 12 * RB;                              // bytes of a record
  static constexpr int SSA = (SS + 127) / 128 * 128;
  static constexpr int COFF = SITES * SS;                         // the four extra sites follow the centre rows
  static constexpr int CSLOT = COFF + 4 * SSA;
  static constexpr int HSLOT = 8 * SX * SS;
  static constexpr int LSTR = 72 * 8 + (SPW > 2 ? 16 : 0);        // links of a site
  static constexpr int LSLOT = SITES * LSTR;
  static constexpr int XBUF = WPS > 1 ? SITES * 12 * WPS * 8 : 0; // fifth-dimension totals of the warps (two buffers)
  static constexpr int OFF_H = 3 * CSLOT;
  static constexpr int OFF_L = OFF_H + 2 * HSLOT;
  static constexpr int OFF_X = OFF_L + 3 * LSLOT;
  static constexpr int OFF_B = OFF_X + 2 * NG * XBUF;                 // mbarriers
  static constexpr int BYTES = OFF_B + 20 * 8;
  static_assert(COFF % 128 == 0 && HSLOT % 512 == 0 && LSLOT % 128 == 0, "alignment of the copies");
  static_assert(NTG % 32 == 0 && SITES % SPW == 0, "tile shape");
  static_assert(BYTES <= 227 * 1024, "shared memory");
};

// Decomposition of the lattice, the powers d^-k and the flag that a wait
// which gave up raises (host-mapped).  A unit is a tile over all of t,
// numbered x-segment first, then y, z, rhs.  CTA i takes units i, i + grid, ...
// while all CTAs have one.  Of the units that remain, fewer than CTAs, each
// gets a CTA for its first `head` steps, and the CTAs without one share the
// rest of their steps out.  So neighbouring tiles are at the same t at the
// same time and their halo rows meet in L2: sharing the steps out evenly
// without regard to t read 244 MB of a 16^3x32x16 launch from DRAM, this
// 145 MB (138 MB is the least).
struct StreamGrid {
  int nseg, ny, nz;
  int units, rounds, head;
  float dp[25];
  int* err;
};

// Tensor maps of the copies (dhop_impl.cuh builds them): the input field as
// [rhs][t z][y][x site, spin, colour][s] with the boxes of the centre rows, of
// one site and of two halo rows in y and in z; the links as [t z][y][x][72].
struct StreamMaps {
  CUtensorMap centre, site, hy, hz, links;
};

__device__ __forceinline__ uint32_t st_smem(int off) {
  return (uint32_t)__cvta_generic_to_shared(hop_dyn_smem) + off;
}
__device__ __forceinline__ void st_bar_init(uint32_t bar, uint32_t n) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(n));
}
__device__ __forceinline__ void st_bar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void st_bar_expect(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool st_bar_wait(uint32_t bar, uint32_t parity) {  // bounded
  for (unsigned i = 0; i < (1u << 22); i++) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}
__device__ __forceinline__ void st_copy5(uint32_t dst, const CUtensorMap& m, int c1, int c2, int c3, int c4, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], "
      "[%7];" ::"r"(dst),
      "l"(&m), "r"(0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void st_copy4(uint32_t dst, const CUtensorMap& m, int c1, int c2, int c3, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
      "[%6];" ::"r"(dst),
      "l"(&m), "r"(0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void st_group_sync(int g, int n) {
  asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "r"(n) : "memory");
}

// A CTA's next piece of work: nt steps from t0 of one unit.
struct StreamWork {
  int k;             // pieces of whole units (or heads) taken
  long long at, end; // a sharing CTA's range of the steps after the heads
  int rhs, xs, len, y0, z0, t0, nt;
  __device__ __forceinline__ StreamWork(const HopParams& p, const StreamGrid& g) : k(0), at(0), end(0) {
    const int left = g.units - g.rounds * (int)gridDim.x;
    const int n = (int)gridDim.x - left, i = (int)blockIdx.x - left;
    if (i >= 0 && left > 0) {
      const long long rest = (long long)left * (p.L3 - g.head);
      at = rest * i / n;
      end = rest * (i + 1) / n;
    }
  }
  __device__ __forceinline__ bool next(const HopParams& p, const StreamGrid& g) {
    int u;
    if (k <= g.rounds && k * (int)gridDim.x + (int)blockIdx.x < g.units) {
      nt = k < g.rounds ? p.L3 : g.head;
      u = k++ * gridDim.x + blockIdx.x;
      t0 = 0;
    } else {
      if (at >= end) return false;
      const int tail = p.L3 - g.head;
      const int r = (int)(at / tail), s = (int)(at - (long long)r * tail);
      nt = (int)(end - at < tail - s ? end - at : tail - s);
      t0 = g.head + s;
      at += nt;
      u = g.rounds * gridDim.x + r;
    }
    const int seg = u % g.nseg;
    u /= g.nseg;
    y0 = 2 * (u % g.ny);
    u /= g.ny;
    z0 = 2 * (u % g.nz);
    rhs = u / g.nz;
    xs = seg * p.Lxh / g.nseg;
    len = (seg + 1) * p.Lxh / g.nseg - xs;
    return true;
  }
};

// Half spinor h of (1 - sg gamma_mu) psi, packed (re, im): spins 0 and 1.
template <int MU>
__device__ __forceinline__ void stream_project(f2p (&h)[6], const f2p (&ps)[12], float sg, f2p NSG, f2p SG) {
#pragma unroll
  for (int c = 0; c < 3; c++) {
    float x, y, a, b;
    if (MU == 0) {  // h0 = p0 + s i p3, h1 = p1 + s i p2
      upk2(ps[c], x, y);
      upk2(ps[9 + c], a, b);
      h[c] = pk2(fmaf(-sg, b, x), fmaf(sg, a, y));
      upk2(ps[3 + c], x, y);
      upk2(ps[6 + c], a, b);
      h[3 + c] = pk2(fmaf(-sg, b, x), fmaf(sg, a, y));
    } else if (MU == 1) {  // h0 = p0 + s p3, h1 = p1 - s p2
      h[c] = fma2(SG, ps[9 + c], ps[c]);
      h[3 + c] = fma2(NSG, ps[6 + c], ps[3 + c]);
    } else if (MU == 2) {  // h0 = p0 + s i p2, h1 = p1 - s i p3
      upk2(ps[c], x, y);
      upk2(ps[6 + c], a, b);
      h[c] = pk2(fmaf(-sg, b, x), fmaf(sg, a, y));
      upk2(ps[3 + c], x, y);
      upk2(ps[9 + c], a, b);
      h[3 + c] = pk2(fmaf(sg, b, x), fmaf(-sg, a, y));
    } else {  // h0 = p0 - s p2, h1 = p1 - s p3
      h[c] = fma2(NSG, ps[6 + c], ps[c]);
      h[3 + c] = fma2(NSG, ps[9 + c], ps[3 + c]);
    }
  }
}

// acc += the full spinor of (1 - sg gamma_mu) U psi from the half spinor h, in
// packed FP32 on (re, im) pairs: A = sum u (h.re, h.re) and B = sum u (h.im,
// h.im) need no swapped operand, and U h = (A.re - B.im, A.im + B.re).  `d`:
// link slot.
template <int MU>
__device__ __forceinline__ void stream_apply(f2p (&acc)[12], const f2p (&h)[6], const unsigned char* Us, int d, float sg,
                                             f2p NSG, f2p SG) {
  f2p u[9];
  const unsigned char* ub = Us + d * 72;
#pragma unroll
  for (int k = 0; k < 9; k++) u[k] = *(const f2p*)(ub + 8 * k);
  f2p hr[6], hi[6];
#pragma unroll
  for (int c = 0; c < 6; c++) {
    float x, y;
    upk2(h[c], x, y);
    hr[c] = pk2(x, x);
    hi[c] = pk2(y, y);
  }
#pragma unroll
  for (int a = 0; a < 3; a++) {
    f2p A0 = mul2(u[a * 3], hr[0]), B0 = mul2(u[a * 3], hi[0]);
    f2p A1 = mul2(u[a * 3], hr[3]), B1 = mul2(u[a * 3], hi[3]);
#pragma unroll
    for (int b = 1; b < 3; b++) {
      A0 = fma2(u[a * 3 + b], hr[b], A0);
      B0 = fma2(u[a * 3 + b], hi[b], B0);
      A1 = fma2(u[a * 3 + b], hr[3 + b], A1);
      B1 = fma2(u[a * 3 + b], hi[3 + b], B1);
    }
    float ar, ai, br, bi;
    upk2(A0, ar, ai);
    upk2(B0, br, bi);
    const float g0r = ar - bi, g0i = ai + br;
    upk2(A1, ar, ai);
    upk2(B1, br, bi);
    const float g1r = ar - bi, g1i = ai + br;
    const f2p g0 = pk2(g0r, g0i), g1 = pk2(g1r, g1i);
    acc[a] = add2(acc[a], g0);
    acc[3 + a] = add2(acc[3 + a], g1);
    float x, y;
    if (MU == 0) {  // lower: -s i g1, -s i g0
      upk2(acc[6 + a], x, y);
      acc[6 + a] = pk2(fmaf(sg, g1i, x), fmaf(-sg, g1r, y));
      upk2(acc[9 + a], x, y);
      acc[9 + a] = pk2(fmaf(sg, g0i, x), fmaf(-sg, g0r, y));
    } else if (MU == 1) {  // -s g1, s g0
      acc[6 + a] = fma2(NSG, g1, acc[6 + a]);
      acc[9 + a] = fma2(SG, g0, acc[9 + a]);
    } else if (MU == 2) {  // -s i g0, s i g1
      upk2(acc[6 + a], x, y);
      acc[6 + a] = pk2(fmaf(sg, g0i, x), fmaf(-sg, g0r, y));
      upk2(acc[9 + a], x, y);
      acc[9 + a] = pk2(fmaf(-sg, g1i, x), fmaf(sg, g1r, y));
    } else {  // -s g0, -s g1
      acc[6 + a] = fma2(NSG, g0, acc[6 + a]);
      acc[9 + a] = fma2(NSG, g1, acc[9 + a]);
    }
  }
}

// Inverse of the fifth-dimension matrix on this thread's slice of every row,
// in registers: with the sweep direction's position q, F_q = v_q + F_{q-1}/d
// (a scan over the site's lanes) and x_q = (F_q - m kappa d^-(q+1) F_last)/d.
// Spins 0,1 of M^-1 and spins 2,3 of M^-dag sweep upward in s, the others
// downward.  Two neighbouring lanes first swap halves, so that the even one
// holds spins 0,1 of both slices and the odd one spins 2,3: that halves the
// shuffles of the scan.  The warps that share a site (Ls = 24) exchange their
// totals through shared memory.
template <class C>
__device__ __forceinline__ void stream_minv(cpx<float> (&v)[12], const HopParams& p, const StreamGrid& g, int rhs, int lq,
                                            int wq, int site, int grp, int buf) {
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int K = C::LPS / 2;                 // slice pairs of the warp's part
  const float dinv = g.dp[1];
  const int lane = threadIdx.x & 31;
  const bool odd = lq & 1;
  const bool up = odd == (p.inv_mode == 2);     // this lane's rows
  const int dir = up ? -2 : 2;                  // lane of the preceding pair: lane + dir
  const int kq = up ? lq >> 1 : K - 1 - (lq >> 1);
  const int part = up ? wq : C::WPS - 1 - wq;   // place of the warp and of the pair in the sweep
  cpx<float> f0[6], f1[6];                      // the pair in the order of the sweep
#pragma unroll
  for (int c = 0; c < 6; c++) {
    const cpx<float> keep = odd ? v[6 + c] : v[c], give = odd ? v[c] : v[6 + c];
    const cpx<float> got = cmake<float>(__shfl_xor_sync(FULL, give.re, 1), __shfl_xor_sync(FULL, give.im, 1));
    const bool mine = odd != up;                // the own slice comes first
    f0[c] = mine ? keep : got;
    const cpx<float> w = mine ? got : keep;
    f1[c] = cmake<float>(fmaf(dinv, f0[c].re, w.re), fmaf(dinv, f0[c].im, w.im));
  }
#pragma unroll
  for (int o = 1; o < K; o *= 2) {
    const float r = g.dp[2 * o];
#pragma unroll
    for (int c = 0; c < 6; c++) {
      const float x = __shfl_sync(FULL, f1[c].re, lane + dir * o), y = __shfl_sync(FULL, f1[c].im, lane + dir * o);
      if (kq >= o) f1[c] = cmake<float>(fmaf(r, x, f1[c].re), fmaf(r, y, f1[c].im));
    }
  }
  const int q0 = (part * K + kq) * 2;           // sweep position of the pair's first slice
  const float mk = (float)(p.m[rhs] * p.kappa[rhs]), c0 = mk * g.dp[q0 + 1], c1 = mk * g.dp[q0 + 2];
  float2* x = nullptr;
  if constexpr (C::WPS > 1) {
    x = (float2*)(hop_dyn_smem + C::OFF_X + (2 * grp + buf) * C::XBUF) + (site * 12 + (odd ? 6 : 0)) * C::WPS;
    if (kq == K - 1) {
#pragma unroll
      for (int c = 0; c < 6; c++) x[c * C::WPS + part] = make_float2(f1[c].re, f1[c].im);
    }
    st_group_sync(grp, C::NTG);  // (the step after next writes this buffer, past the next step's barrier)
  }
  const int lend = lane + (up ? 2 * (K - 1 - kq) : -2 * (K - 1 - kq));
#pragma unroll
  for (int c = 0; c < 6; c++) {
    cpx<float> e = cmake<float>(__shfl_sync(FULL, f1[c].re, lane + dir), __shfl_sync(FULL, f1[c].im, lane + dir));
    if (kq == 0) e = cmake<float>(0.f, 0.f);    // the sweep's value before the pair
    cpx<float> last;
    if constexpr (C::WPS > 1) {
      cpx<float> in = cmake<float>(0.f, 0.f);
      last = in;
#pragma unroll
      for (int k = 0; k < C::WPS; k++) {
        if (k == part) in = last;
        const float2 t = x[c * C::WPS + k];
        last = cmake<float>(fmaf(g.dp[C::LPS], last.re, t.x), fmaf(g.dp[C::LPS], last.im, t.y));
      }
      const float rc = g.dp[2 * kq];            // decay of the carry up to the pair
      in = cmake<float>(rc * in.re, rc * in.im);
      e = cmake<float>(e.re + in.re, e.im + in.im);
      f1[c] = cmake<float>(fmaf(g.dp[2], in.re, f1[c].re), fmaf(g.dp[2], in.im, f1[c].im));
    } else {
      last = cmake<float>(__shfl_sync(FULL, f1[c].re, lend), __shfl_sync(FULL, f1[c].im, lend));
    }
    f0[c] = cmake<float>(fmaf(dinv, e.re, f0[c].re), fmaf(dinv, e.im, f0[c].im));
    f0[c] = cmake<float>(dinv * fmaf(-c0, last.re, f0[c].re), dinv * fmaf(-c0, last.im, f0[c].im));
    f1[c] = cmake<float>(dinv * fmaf(-c1, last.re, f1[c].re), dinv * fmaf(-c1, last.im, f1[c].im));
    const bool mine = odd != up;
    const cpx<float> keep = mine ? f0[c] : f1[c], give = mine ? f1[c] : f0[c];
    const cpx<float> got = cmake<float>(__shfl_xor_sync(FULL, give.re, 1), __shfl_xor_sync(FULL, give.im, 1));
    v[c] = odd ? got : keep;
    v[6 + c] = odd ? keep : got;
  }
}

template <int P, int LS, int SXV>
__global__ void __launch_bounds__(StreamCfg<P, LS, SXV>::NT, 1) hop_stream(const __grid_constant__ HopParams p,
                                                                    const __grid_constant__ StreamGrid g,
                                                                    const __grid_constant__ StreamMaps m) {
  typedef StreamCfg<P, LS, SXV> C;
  typedef typename Prec<P>::S S;
  constexpr int SX = C::SX;
  const uint32_t bars = st_smem(C::OFF_B);
  const auto fullC = [&](int k) { return bars + 8 * k; };
  const auto emptyC = [&](int k) { return bars + 24 + 8 * k; };
  const auto fullL = [&](int k) { return bars + 48 + 8 * k; };
  const auto emptyL = [&](int k) { return bars + 72 + 8 * k; };
  // halo slots: y rows (part 0) and z rows (part 1) on barriers of their own
  const auto fullH = [&](int k, int part) { return bars + 96 + 16 * part + 8 * k; };
  const auto emptyH = [&](int k, int part) { return bars + 128 + 16 * part + 8 * k; };
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) {
    for (int k = 0; k < 3; k++) {
      st_bar_init(fullC(k), 1);
      st_bar_init(emptyC(k), 3 * C::NWG);
      st_bar_init(fullL(k), 1);
      st_bar_init(emptyL(k), C::NWG);
    }
    for (int k = 0; k < 2; k++) {
      for (int h = 0; h < 2; h++) {
        st_bar_init(fullH(k, h), 1);
        st_bar_init(emptyH(k, h), C::NWG);
      }
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  const int L1 = p.L1, L2 = p.L2, L3 = p.L3, Lxh = p.Lxh;

  if (warp >= C::NG * C::NWG) {
    // ------------------------------------------------------------ producer
    if constexpr (C::REGSPLIT) asm volatile("setmaxnreg.dec.sync.aligned.u32 32;");
    if (warp > C::NG * C::NWG) return;
    if (lane != 0) return;
    StreamWork w(p, g);
    const auto bar = [&](int ring, int slot, bool full) {
      return ring == RING_C   ? (full ? fullC(slot) : emptyC(slot))
             : ring == RING_L ? (full ? fullL(slot) : emptyL(slot))
                              : (full ? fullH(slot, ring - RING_Y) : emptyH(slot, ring - RING_Y));
    };
    const auto centre = [&](int i, int slot) {  // slice t0 - 1 + i
      int t = w.t0 - 1 + i;
      t = t < 0 ? t + L3 : t >= L3 ? t - L3 : t;
      // the x-neighbours outside the segment are read in the slice's own step only
      const bool ext = i > 0 && i <= w.nt && g.nseg > 1;
      const uint32_t dst = st_smem(slot * C::CSLOT);
      st_bar_expect(fullC(slot), C::COFF + (ext ? 4 * C::SS : 0));
      st_copy5(dst, m.centre, 12 * w.xs, w.y0, t * L2 + w.z0, w.rhs, fullC(slot));
      if (ext) {
        const int left = w.xs == 0 ? Lxh - 1 : w.xs - 1, right = w.xs + w.len == Lxh ? 0 : w.xs + w.len;
        const int b = (w.y0 + w.z0 + t + p.out_parity) & 1;  // of rows 0 and 3; rows 1 and 2 differ
#pragma unroll
        for (int r = 0; r < 4; r++) {
          const bool up = (b != 0) != (r == 1 || r == 2);
          st_copy5(dst + C::COFF + r * C::SSA, m.site, 12 * (up ? right : left), w.y0 + (r & 1), t * L2 + w.z0 + (r >> 1),
                   w.rhs, fullC(slot));
        }
      }
    };
    const auto halo = [&](int i, int part, int slot) {
      const int tz = (w.t0 + i) * L2;
      const uint32_t dst = st_smem(C::OFF_H + slot * C::HSLOT), bh = fullH(slot, part);
      constexpr int TWO = 2 * SX * C::SS;  // two rows
      st_bar_expect(bh, 2 * TWO);
      if (part == 0) {
        st_copy5(dst, m.hy, 12 * w.xs, w.y0 == 0 ? L1 - 1 : w.y0 - 1, tz + w.z0, w.rhs, bh);
        st_copy5(dst + TWO, m.hy, 12 * w.xs, w.y0 + 2 == L1 ? 0 : w.y0 + 2, tz + w.z0, w.rhs, bh);
      } else {
        st_copy5(dst + 2 * TWO, m.hz, 12 * w.xs, w.y0, tz + (w.z0 == 0 ? L2 - 1 : w.z0 - 1), w.rhs, bh);
        st_copy5(dst + 3 * TWO, m.hz, 12 * w.xs, w.y0, tz + (w.z0 + 2 == L2 ? 0 : w.z0 + 2), w.rhs, bh);
      }
    };
    const auto links = [&](int i, int slot) {
      st_bar_expect(fullL(slot), C::LSLOT);
      st_copy4(st_smem(C::OFF_L + slot * C::LSLOT), m.links, w.xs, w.y0, (w.t0 + i) * L2 + w.z0, fullL(slot));
    };
    const auto wait_empty = [&](int ring, int slot, uint32_t par) { return st_bar_wait(bar(ring, slot, false), par); };
    const auto wait_full = [&](int ring, int slot, uint32_t par) { return st_bar_wait(bar(ring, slot, true), par); };
    const auto raise = [&]() { *(volatile int*)g.err = 1; };
    // (order of the copies and their waits: ring_roles.cuh)
    StreamProducer prod;
    while (prod.ok && w.next(p, g)) prod.run(w.nt, wait_empty, centre, links, halo);
    prod.finish(wait_full, raise);
    return;
  }

  // -------------------------------------------------------------- consumers
  if constexpr (C::REGSPLIT) asm volatile("setmaxnreg.inc.sync.aligned.u32 112;");
  const int grp = warp / C::NWG, wg = warp - grp * C::NWG;
  const int wq = C::WPS > 1 ? wg % C::WPS : 0;              // the warp's part of the s range
  const int st = (wg / C::WPS) * C::SPW + lane / C::LPS;    // site in the tile
  const int lq = lane % C::LPS;
  const int s5 = wq * C::LPS + lq;
  const int row = st / SX, j = st - row * SX;
  const int ry = row & 1, rz = row >> 1;
  const int so = s5 * C::CB;
  const int offC = st * C::SS + so;
  const float sg = p.sg;
  const f2p SG = pk2(sg, sg), NSG = pk2(-sg, -sg);
  bool ok = true;
  unsigned kcb = 0, ns = 0;  // slices and steps of the units before this one
  PartialSum<float> sum;
  int sum_rhs = 0;
  const int pwarp = blockIdx.x * (C::NG * C::NWG) + warp, nparts = gridDim.x * (C::NG * C::NWG);
  const auto flush = [&]() {
    double acc = sum.value();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if (lane == 0) p.partials[(size_t)sum_rhs * nparts + pwarp] = acc;
    sum = PartialSum<float>();
  };

  // after a wait that gave up nothing is released: the producer gives up in turn
  const auto release = [&](uint32_t bar) {
    __syncwarp();
    if (lane == 0 && ok) st_bar_arrive(bar);
  };
  StreamWork w(p, g);
  while (w.next(p, g)) {
    if (p.reduce && w.rhs != sum_rhs) {
      for (; sum_rhs < w.rhs; sum_rhs++) flush();
    }
    const int y = w.y0 + ry, z = w.z0 + rz;
    const bool inside = j < w.len;
    // Step s uses slices s, s+1, s+2 of the run's nt + 2.  Steps -2, -1, nt and
    // nt+1 only pass the slices they would have used on: so each slice is seen
    // and released by three steps in turn, that is by both groups, and neither
    // can miss a phase of a barrier.
    for (int s = -2 + (int)((ns ^ grp) & 1); s < w.nt + 2; s += C::NG) {
      const unsigned kc = kcb + s, kh = ns + s;
      if (s < 0 || s >= w.nt) {
        for (int i = s < 0 ? 0 : s; i <= s + 2 && i < w.nt + 2; i++) {
          const unsigned k = kcb + i;
          ok = ok && st_bar_wait(fullC(k % 3), (k / 3) & 1);
          release(emptyC(k % 3));
        }
        continue;
      }
      const int t = w.t0 + s;
      const int b = (y + z + t + p.out_parity) & 1;
      const int site = ((t * L2 + z) * L1 + y) * Lxh + w.xs + j;
      f2p acc[12], ps[12];
#pragma unroll
      for (int c = 0; c < 12; c++) acc[c] = 0ull;
      const int c0 = (kc % 3) * C::CSLOT, c1 = ((kc + 1) % 3) * C::CSLOT, c2 = ((kc + 2) % 3) * C::CSLOT;
      const int offX = g.nseg == 1 ? (row * SX + (b ? 0 : w.len - 1)) * C::SS + so : C::COFF + row * C::SSA + so;
      const int hb = C::OFF_H + (kh & 1) * C::HSLOT + j * C::SS + so;
      const unsigned char* U = hop_dyn_smem + C::OFF_L + (kh % 3) * C::LSLOT + st * C::LSTR;
      const auto dir = [&](auto dc) {  // direction d: even slots the neighbours at +mu, odd at -mu
        constexpr int d = decltype(dc)::value;
        f2p h[6];
        stream_project<d / 2>(h, ps, d & 1 ? -sg : sg, d & 1 ? SG : NSG, d & 1 ? NSG : SG);
        stream_apply<d / 2>(acc, h, U, d, d & 1 ? -sg : sg, d & 1 ? SG : NSG, d & 1 ? NSG : SG);
      };
      const auto ld = [&](int off) { load_spinor_x2<P, C::RB / C::CB>(ps, (const S*)(hop_dyn_smem + off)); };
      ok = ok && st_bar_wait(fullC((kc + 1) % 3), ((kc + 1) / 3) & 1);
      // (the links' slot was the other group's last: that step is over, since the
      // slice waited for above has taken the slot of one that it read)
      ok = ok && st_bar_wait(fullL(kh % 3), (kh / 3) & 1);
      ok = ok && st_bar_wait(fullH(kh & 1, 0), (kh / 2) & 1);
      ld(ry == 0 ? c1 + offC + SX * C::SS : hb + (2 + rz) * SX * C::SS);
      dir(std::integral_constant<int, 2>());  // y+1
      ld(ry == 1 ? c1 + offC - SX * C::SS : hb + rz * SX * C::SS);
      dir(std::integral_constant<int, 3>());  // y-1
      release(emptyH(kh & 1, 0));
      ok = ok && st_bar_wait(fullH(kh & 1, 1), (kh / 2) & 1);
      ld(rz == 0 ? c1 + offC + 2 * SX * C::SS : hb + (6 + ry) * SX * C::SS);
      dir(std::integral_constant<int, 4>());  // z+1
      ld(rz == 1 ? c1 + offC - 2 * SX * C::SS : hb + (4 + ry) * SX * C::SS);
      dir(std::integral_constant<int, 5>());  // z-1
      release(emptyH(kh & 1, 1));
      ok = ok && st_bar_wait(fullC(kc % 3), (kc / 3) & 1);
      ld(c0 + offC);
      dir(std::integral_constant<int, 7>());  // t-1
      release(emptyC(kc % 3));
      // one x-neighbour has the site's own index, the other may be outside the segment
      ld(c1 + (b == 0 ? offC : j < w.len - 1 ? offC + C::SS : offX));
      dir(std::integral_constant<int, 0>());  // x+1
      ld(c1 + (b == 1 ? offC : j > 0 ? offC - C::SS : offX));
      dir(std::integral_constant<int, 1>());  // x-1
      release(emptyC((kc + 1) % 3));
      // operands of the aux epilogue, in flight during the last direction
      const size_t base = (size_t)w.rhs * p.rhs_stride + (size_t)site * 12 * LS;
      const bool dagM = p.aux_mode == 3;
      const int sm = s5 > 0 ? s5 - 1 : LS - 1, sp = s5 < LS - 1 ? s5 + 1 : 0;
      cpx<float> ax[12], ae[12];
      if (p.aux_mode) {
        const S* aux = (const S*)p.aux + base;
#pragma unroll
        for (int c = 0; c < 12; c++) ax[c] = inside ? ld_c(aux + c * LS + s5) : cmake<float>(0.f, 0.f);
      }
      ok = ok && st_bar_wait(fullC((kc + 2) % 3), ((kc + 2) / 3) & 1);
      ld(c2 + offC);
      dir(std::integral_constant<int, 6>());  // t+1
      release(emptyC((kc + 2) % 3));
      release(emptyL(kh % 3));

      cpx<float> v[12];
      const float al = (float)p.alpha;
#pragma unroll
      for (int c = 0; c < 12; c++) {
        upk2(acc[c], v[c].re, v[c].im);
        v[c].re *= al;
        v[c].im *= al;
      }
      if (p.aux_mode == 1) {
#pragma unroll
        for (int c = 0; c < 12; c++) cacc(v[c], ax[c]);
      } else if (p.aux_mode) {
        // M psi_s = d psi_s - psi_{s-+1} (+ m psi at the wall), as in hop_kernel
        const float d = (float)p.d, m = (float)p.m[w.rhs];
        const float cm = s5 > 0 ? -1.f : m, cp = s5 < LS - 1 ? -1.f : m;
        if (C::WPS == 1) {  // the neighbouring slices are on the neighbouring lanes
          const int lm = lane - s5 + sm, lp = lane - s5 + sp;
#pragma unroll
          for (int c = 0; c < 12; c++) {
            const int src = (c < 6) != dagM ? lm : lp;
            ae[c].re = __shfl_sync(0xffffffffu, ax[c].re, src);
            ae[c].im = __shfl_sync(0xffffffffu, ax[c].im, src);
          }
        } else {  // (just read by other warps' lanes: L1 or L2)
          const S* aux = (const S*)p.aux + base;
#pragma unroll
          for (int c = 0; c < 12; c++)
            ae[c] = inside ? ld_c(aux + c * LS + ((c < 6) != dagM ? sm : sp)) : cmake<float>(0.f, 0.f);
        }
#pragma unroll
        for (int c = 0; c < 12; c++) {
          const float co = (c < 6) != dagM ? cm : cp;
          v[c].re += fmaf(d, ax[c].re, co * ae[c].re);
          v[c].im += fmaf(d, ax[c].im, co * ae[c].im);
        }
      }
      if (p.inv_mode) stream_minv<C>(v, p, g, w.rhs, lq, wq, st, grp, (kh >> 1) & 1);
      if (inside && ok) {
        hop_put<P, LS>(v, p, base, s5);
        if (p.reduce) {
#pragma unroll
          for (int c = 0; c < 12; c++) sum.add(fmaf(v[c].re, v[c].re, v[c].im * v[c].im));
        }
      }
    }
    kcb += w.nt + 2;
    ns += w.nt;
  }
  if (p.reduce) {
    const int nrhs = g.units / (g.nseg * g.ny * g.nz);
    for (; sum_rhs < nrhs; sum_rhs++) flush();
  }
  if (!ok && lane == 0) *(volatile int*)g.err = 1;
}

}  // namespace dwfk
