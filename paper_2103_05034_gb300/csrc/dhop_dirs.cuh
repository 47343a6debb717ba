// FP64 hopping term with the eight neighbours of a site on eight groups of
// threads (arXiv:2103.05034, Sec. 2, Eq. 2), for small lattices; the epilogues
// of hop_kernel (same HopParams).
//
// GB300 issues one FP64 warp instruction about every 70 cycles on a quarter of
// an SM, so a thread that sums all eight directions (some 930 FP64
// instructions a site and slice) takes 35 us however few CTAs there are.  Here
// a thread projects and multiplies one neighbour (84 instructions) and leaves
// the six colour-spin components of U h in shared memory; the lower spins are
// those components times +-1 or +-i, so nothing more is stored.  The CTA's
// threads then add the eight terms of each output (14 additions).  The two signs of a direction share a warp,
// different directions never do.
#pragma once

namespace dwfk {

template <int LS>
struct DirsCfg {
  static constexpr int SITES = LS == 24 ? 2 : LS == 16 ? 1 : 16 / LS;  // 2 LS SITES: whole warps
  static constexpr int NT = 8 * LS * SITES;
  static constexpr int ROWS = 12 * SITES;
};

// Epilogue store of one component c at slice s of the field at `base`.
template <int LS>
__device__ __forceinline__ cpx<double> dirs_store(cpx<double> v, const HopParams& p, int rhs, size_t base, int c, int s) {
  if (p.cg_mode) {
    const size_t off = base + c * LS + s;
    const double alpha = p.cg_alpha[(size_t)rhs * p.cg_astride];
    double2* xs = (double2*)p.cg_x + off;
    double2* rs = (double2*)p.cg_r + off;
    const cpx<double> pv = ld_c((const double2*)p.cg_p + off);
    cpx<double> xv = ld_c(xs), rv = ld_c(rs);
    xv.re = fma(alpha, pv.re, xv.re);
    xv.im = fma(alpha, pv.im, xv.im);
    rv.re = fma(-alpha, v.re, rv.re);
    rv.im = fma(-alpha, v.im, rv.im);
    st_c(xs, xv);
    st_c(rs, rv);
    return rv;
  }
  const cpx<double> keep = v;
  const size_t off = base + c * LS + (p.g5r5 ? LS - 1 - s : s);
  if (p.g5r5 && c >= 6) v = cmake<double>(-v.re, -v.im);
  if (p.cheb_mode) {
    double2* ct = (double2*)p.cheb_tp + off;
    const cpx<double> xv = ld_c((const double2*)p.cheb_x + off), tv = ld_c(ct);
    v.re = fma(p.cheb_ta, v.re, fma(p.cheb_tb, xv.re, -tv.re));
    v.im = fma(p.cheb_ta, v.im, fma(p.cheb_tb, xv.im, -tv.im));
    st_c(ct, v);
    if (p.cheb_acc) {
      double2* ca = (double2*)p.cheb_acc + off;
      cpx<double> av = ld_c(ca);
      av.re = fma(p.cheb_cacc, v.re, av.re);
      av.im = fma(p.cheb_cacc, v.im, av.im);
      st_c(ca, av);
    }
  } else {
    st_c((double2*)p.out + off, v);
  }
  return keep;
}

template <int LS>
__global__ void __launch_bounds__(DirsCfg<LS>::NT) hop_dirs_f64(const HopParams p) {
  typedef DirsCfg<LS> C;
  __shared__ double2 g[8][6][C::SITES * LS];     // U h of every direction
  __shared__ cpx<double> stage[C::ROWS * (LS + 1)];
  __shared__ double red[C::NT / 32];
  const int tid = threadIdx.x;
  const int rhs = blockIdx.y;
  const int site0 = blockIdx.x * C::SITES;

  {
    const int mu = tid / (2 * LS * C::SITES), r = tid - mu * (2 * LS * C::SITES);
    const int sign = r / (LS * C::SITES), i = r - sign * (LS * C::SITES);  // 0: neighbour at +mu, 1: at -mu
    const int sl = i / LS, s = i - sl * LS;
    const int site = site0 + sl;
    if (site < p.Vh) {
      int rem = site / p.Lxh;
      const int xh = site - rem * p.Lxh;
      int y = rem % p.L1;
      rem /= p.L1;
      int z = rem % p.L2, t = rem / p.L2;
      int x = 2 * xh + ((y + z + t + p.out_parity) & 1);
      const int step = sign ? -1 : 1;
      const auto wrap = [](int a, int n) { return a < 0 ? a + n : a >= n ? a - n : a; };
      if (mu == 0) x = wrap(x + step, p.L0);
      if (mu == 1) y = wrap(y + step, p.L1);
      if (mu == 2) z = wrap(z + step, p.L2);
      if (mu == 3) t = wrap(t + step, p.L3);
      const int nb = ((t * p.L2 + z) * p.L1 + y) * p.Lxh + (x >> 1);
      const double2* in = (const double2*)p.in + (size_t)rhs * p.rhs_stride + (size_t)nb * 12 * LS + s;
      cpx<double> ps[12];
      load_spinor<DWF_F64, LS>(ps, in, 0);
      const double2* gl = (const double2*)p.links + (size_t)site * 72 + (2 * mu + sign) * 9;
      cpx<double> U[9];
#pragma unroll
      for (int k = 0; k < 9; k++) U[k] = ld_c(gl + k);
      const double sg = sign ? -(double)p.sg : (double)p.sg;
      // h0 = p0 - sg A p(2,3), h1 likewise (the rules of hop_dir)
      cpx<double> h[6];
#pragma unroll
      for (int c = 0; c < 3; c++) {
        const cpx<double> p0 = ps[c], p1 = ps[3 + c], p2 = ps[6 + c], p3 = ps[9 + c];
        if (mu == 0) {
          h[c] = cmake<double>(fma(-sg, p3.im, p0.re), fma(sg, p3.re, p0.im));
          h[3 + c] = cmake<double>(fma(-sg, p2.im, p1.re), fma(sg, p2.re, p1.im));
        } else if (mu == 1) {
          h[c] = cmake<double>(fma(sg, p3.re, p0.re), fma(sg, p3.im, p0.im));
          h[3 + c] = cmake<double>(fma(-sg, p2.re, p1.re), fma(-sg, p2.im, p1.im));
        } else if (mu == 2) {
          h[c] = cmake<double>(fma(-sg, p2.im, p0.re), fma(sg, p2.re, p0.im));
          h[3 + c] = cmake<double>(fma(sg, p3.im, p1.re), fma(-sg, p3.re, p1.im));
        } else {
          h[c] = cmake<double>(fma(-sg, p2.re, p0.re), fma(-sg, p2.im, p0.im));
          h[3 + c] = cmake<double>(fma(-sg, p3.re, p1.re), fma(-sg, p3.im, p1.im));
        }
      }
#pragma unroll
      for (int k = 0; k < 6; k++) {
        const int a = k % 3, h0 = k - a;
        double re = U[a * 3].re * h[h0].re, im = U[a * 3].re * h[h0].im;
        re = fma(-U[a * 3].im, h[h0].im, re);
        im = fma(U[a * 3].im, h[h0].re, im);
#pragma unroll
        for (int b = 1; b < 3; b++) {
          const cpx<double> u = U[a * 3 + b];
          re = fma(u.re, h[h0 + b].re, re);
          re = fma(-u.im, h[h0 + b].im, re);
          im = fma(u.re, h[h0 + b].im, im);
          im = fma(u.im, h[h0 + b].re, im);
        }
        g[2 * mu + sign][k][i] = make_double2(re, im);
      }
    }
  }
  __syncthreads();

  // outputs (row = site, spin, colour; slice s): one or two of them a thread
  constexpr int N = C::ROWS * LS, PER = (N + C::NT - 1) / C::NT;
  const double* m = p.m;
  cpx<double> v[PER];
#pragma unroll
  for (int k = 0; k < PER; k++) {
    const int e = k * C::NT + tid, rw = e / LS, s = e - rw * LS;
    const int sl = rw / 12, c = rw - sl * 12, spin = c / 3, a = c - spin * 3;
    if (e >= N || site0 + sl >= p.Vh) continue;
    const int i = sl * LS + s;
    double re = 0, im = 0;
#pragma unroll
    for (int d = 0; d < 8; d++) {
      const int mu = d / 2;
      const bool pos = ((d & 1) != 0) != (p.sg < 0);  // the sign -s of the lower spins, s = +-sg
      if (spin < 2) {
        const double2 t = g[d][spin * 3 + a][i];
        re += t.x;
        im += t.y;
      } else {
        // spin 2: -s {i g1, g1, i g0, g0}, spin 3: -s {i g0, -g0, -i g1, g1}
        const int from = (mu < 2) == (spin == 2) ? 1 : 0;
        const double2 t = g[d][from * 3 + a][i];
        const bool flip = (spin == 3 && (mu == 1 || mu == 2)) == pos;
        const double x = mu == 0 || mu == 2 ? -t.y : t.x, y = mu == 0 || mu == 2 ? t.x : t.y;
        re += flip ? -x : x;
        im += flip ? -y : y;
      }
    }
    re *= p.alpha;
    im *= p.alpha;
    if (p.aux_mode) {
      const double2* aux = (const double2*)p.aux + (size_t)rhs * p.rhs_stride + ((size_t)(site0 + sl) * 12 + c) * LS;
      const cpx<double> q = ld_c(aux + s);
      if (p.aux_mode == 1) {
        re += q.re;
        im += q.im;
      } else {
        // M psi_s = d psi_s - psi_{s-+1} (+ m psi at the wall), as in hop_kernel
        const bool lower = (c < 6) != (p.aux_mode == 3);
        const bool wall = lower ? s == 0 : s == LS - 1;
        const int sn = lower ? (wall ? LS - 1 : s - 1) : (wall ? 0 : s + 1);
        const cpx<double> n = ld_c(aux + sn);
        const double co = wall ? m[rhs] : -1.0;
        re += fma(p.d, q.re, co * n.re);
        im += fma(p.d, q.im, co * n.im);
      }
    }
    v[k] = cmake<double>(re, im);
    if (p.inv_mode) stage[rw * (LS + 1) + s] = v[k];
  }
  if (p.inv_mode) {
    __syncthreads();
    if (tid < C::ROWS && site0 + tid / 12 < p.Vh)
      minv_row_inplace<double, LS>(stage + tid * (LS + 1), (tid % 12 < 6) != (p.inv_mode == 2), p.d, m[rhs], p.kappa[rhs],
                                   p.dls1[rhs], p.one_sweep);
    __syncthreads();
  }
  double sum = 0;
#pragma unroll
  for (int k = 0; k < PER; k++) {
    const int e = k * C::NT + tid, rw = e / LS, s = e - rw * LS;
    const int sl = rw / 12, c = rw - sl * 12;
    if (e >= N || site0 + sl >= p.Vh) continue;
    if (p.inv_mode) v[k] = stage[rw * (LS + 1) + s];
    const cpx<double> o =
        dirs_store<LS>(v[k], p, rhs, (size_t)rhs * p.rhs_stride + (size_t)(site0 + sl) * 12 * LS, c, s);
    sum += fma(o.re, o.re, o.im * o.im);
  }
  if (p.reduce) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, o);
    if ((tid & 31) == 0) red[tid >> 5] = sum;
    __syncthreads();
    if (tid == 0) {
      double tot = 0.0;
      for (int i = 0; i < C::NT / 32; i++) tot += red[i];
      p.partials[blockIdx.y * gridDim.x + blockIdx.x] = tot;
    }
  }
}

}  // namespace dwfk
