// Adjoint of one 2D semi-implicit Fourier-spectral step.  The step maps the
// real state u to u'_phi = F^-1[ D1_phi F u_phi + D2_phi F f_phi(u) ] with
//   c:     D1 = 1/(1 + M dt kc K2^2),  D2 = -M dt K2 / (1 + M dt kc K2^2)
//   eta_i: D1 = 1/(1 + L dt ke K2),    D2 = -L dt / (1 + L dt ke K2)
// (Eqs. C-H_discrete_fft .. A-C_discrete_fft_eta), f_phi = df_chem/dphi.
// D1, D2 are real and even in k, so G = F^-1 D F is real symmetric, and
//   lambda_phi = G1_phi lam'_phi + sum_psi H_phi,psi(u) G2_psi lam'_psi
// with H the pointwise Hessian of f_chem.  Parameter sensitivities of
// <lam', u'> for theta = (M, L, kappa_c, kappa_eta) follow from Parseval:
//   d/dtheta = (1/N) sum_k conj(Lam'(k)) (dD1/dtheta U(k) + dD2/dtheta Fu(k)).
// Three passes (adjoint workspace: 3 nf packed half-spectrum slots):
//   adj row forward  x transforms of lam'_phi, u_phi, f_phi(u)
//   adj column       y transforms, G1/G2 multipliers, sensitivities, inverse y
//   adj row inverse  inverse x transforms and the pointwise Hessian product
#pragma once

#include "fs_kernels.cuh"

namespace fs {

// Pointwise Hessian of f_chem in (c, eta_1..eta_p):
//   H_cc = 2 rho2, H_c,k = -2 rho2 (cb - ca) h'(eta_k),
//   H_k,k = rho2 (cb - ca)(cb + ca - 2c) h''(eta_k)
//           + w [2 - 12 eta_k + 12 eta_k^2 + 4 alpha sum_{j != k} eta_j^2],
//   H_k,l = 8 w alpha eta_k eta_l (k != l),  h''(e) = 60 e (1 - e)(1 - 2e).
// out = H mu on the two grid points of a pair (lane-wise), P = p known at
// compile time.
template <int P, typename T>
__device__ __forceinline__ void hessian_apply(const Pointwise<T>& pw, const cplx<T> (&u)[P + 1],
                                              const cplx<T> (&mu)[P + 1], cplx<T> (&out)[P + 1]) {
  using C = cplx<T>;
  auto k = [](T v) { return vsplat<C>(v); };
  const T wa8 = T(2) * pw.w * pw.four_alpha;  // 8 w alpha
  C S2 = k(T(0)), em = k(T(0));               // sum eta_j^2, sum eta_j mu_j
#pragma unroll
  for (int i = 1; i <= P; ++i) {
    S2 = vfma(u[i], u[i], S2);
    em = vfma(u[i], mu[i], em);
  }
  const C chem = vfma(u[0], k(T(-120) * pw.rho2dcab), k(T(60) * pw.rho2dcab * pw.cab));  // 60 rho2 dcab (cab - 2c)
  out[0] = vmul(mu[0], k(pw.two_rho2));
#pragma unroll
  for (int i = 1; i <= P; ++i) {
    const C e = u[i], ne = mk<C>(-e.x, -e.y);
    const C q = vfma(e, ne, e);                                             // e (1 - e)
    const C hck = vmul(k(T(-30) * pw.two_rho2 * pw.dcab), vmul(q, q));      // H_c,i
    const C dw = vfma(q, k(T(-12)), k(T(2)));                               // 2 - 12 e + 12 e^2
    // + 4 alpha (S2 - e^2), the sum over the other etas (P = 1: there is none)
    const C well = P == 1 ? dw : vfma(vfma(e, ne, S2), k(pw.four_alpha), dw);
    const C hkk = vfma(vmul(chem, q), vfma(e, k(T(-2)), k(T(1))), vmul(well, k(pw.w)));
    out[0] = vfma(hck, mu[i], out[0]);
    const C cross = P == 1 ? k(T(0)) : vmul(vmul(e, k(wa8)), vfma(ne, mu[i], em));  // sum over j != i
    out[i] = vfma(hck, mu[0], vfma(hkk, mu[i], cross));
  }
}

// The steps' row and column tiles with the adjoint's pass tables
// (adj_line_fft; KArgs::tw_row and tw_col of an adjoint launch hold them).
template <typename T, int NX>
struct AdjRowCfg : RowCfg<T, NX> {
  using B = RowCfg<T, NX>;
  static constexpr int TWS = adj_table_size<T>(B::L, B::E);
  static constexpr int TW_BYTES = ((TWS * (int)sizeof(cplx<T>)) + 127) & ~127;
  static constexpr size_t smem(int nf) {
    return B::BAR_BYTES + TW_BYTES + (size_t)3 * nf * B::R * B::PL * sizeof(cplx<T>);
  }
};

// B w of the row pass's post-processing; FP32 in the arithmetic the
// sensitivities are to keep (cmul rounds the other product of the imaginary part).
template <typename C>
__device__ __forceinline__ C adj_cmul(C b, C w) {
  if constexpr (sizeof(C) == 8)
    return mk<C>(fmaf(b.x, w.x, -__fmul_rn(b.y, w.y)), fmaf(b.x, w.y, __fmul_rn(b.y, w.x)));
  else return cmul(b, w);
}

// ---------------------------------------------------------------------------
// Adjoint row forward: CTA of 3 nf warps, one per transform, and R rows.
// Inputs real: lam' (a.real), u (a.aux).  Outputs 2 x^ of lam'_phi, u_phi,
// f_phi(u) into adjoint slots [0, nf), [nf, 2nf), [2nf, 3nf).  f(u) in FP32 is
// formed term by term (Pointwise::fc, feta): the sensitivities keep its
// rounding too.
// ---------------------------------------------------------------------------
template <typename T, int NX, int P>
__global__ void __launch_bounds__(96 * (P + 1)) fs_adj_row_fwd_kernel(KArgs a) {
  using C = cplx<T>;
  using Cfg = AdjRowCfg<T, NX>;
  constexpr int L = Cfg::L, E = Cfg::E, TPL = Cfg::TPL, R = Cfg::R, PL = Cfg::PL;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem_raw);
  C* twr = reinterpret_cast<C*>(smem_raw + Cfg::BAR_BYTES);
  C* slots = reinterpret_cast<C*>(smem_raw + Cfg::BAR_BYTES + Cfg::TW_BYTES);
  constexpr int nf = P + 1;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane / TPL, t = lane % TPL;
  const int Reff = a.lines < R ? (int)a.lines : R;
  const bool active = g < Reff;
  const long long row0 = (long long)blockIdx.x * Reff, row = row0 + g;
  const C* __restrict__ twh = reinterpret_cast<const C*>(a.tw_half);
  const long long half_stride = a.npts / 2;
  auto slot = [slots](int f, int r) { return slots + (f * R + r) * PL; };
  auto wsync = []() { __syncwarp(); };
  copy_to_smem(twr, reinterpret_cast<const C*>(a.tw_row), Cfg::TWS);
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
  }
  griddep_wait();  // everything read or written below may belong to the previous grid
  griddep_launch_dependents();
  __syncthreads();
  if (threadIdx.x == 0) {
    const uint32_t bytes = (uint32_t)(L * sizeof(C));
    mbar_arrive_expect_tx(bar, bytes * Reff * 2 * nf);
    for (int f = 0; f < nf; ++f)
      for (int r = 0; r < Reff; ++r) {
        bulk_g2s(slot(f, r), reinterpret_cast<const C*>(a.real) + f * half_stride + (row0 + r) * L, bytes, bar);
        bulk_g2s(slot(nf + f, r), reinterpret_cast<const C*>(a.aux) + f * half_stride + (row0 + r) * L, bytes,
                 bar);
      }
  }
  if (!mbar_wait_bounded(bar, 0, first_wait_polls(a))) {
    if (threadIdx.x == 0) atomicOr(a.flag, FS_FLAG_TIMEOUT);
    mbar_wait_bounded(bar, 0, kWaitPolls);
    return;
  }
  // f(u) into slots [2nf, 3nf)
  {
    const Pointwise<T> pw(a);
    const T A = T(-60) * pw.rho2dcab, B = T(30) * pw.rho2dcab * pw.cab, W = T(2) * pw.w, F = pw.w * pw.four_alpha;
    for (int idx = threadIdx.x; idx < Reff * L; idx += blockDim.x) {
      const int r = idx / L, i0 = idx % L;
      const C c = slot(nf, r)[i0];
      C e[nf], h = vsplat<C>(T(0)), S2 = vsplat<C>(T(0));
#pragma unroll
      for (int i = 1; i < nf; ++i) {
        e[i] = slot(nf + i, r)[i0];
        h = pw.add_h2(e[i], h);
        S2 = sizeof(T) == 4 ? cadd(S2, vmul(e[i], e[i])) : vfma(e[i], e[i], S2);
      }
      if constexpr (sizeof(T) == 4) {
        slot(2 * nf, r)[i0] = mk<C>(pw.fc(c.x, h.x), pw.fc(c.y, h.y));
#pragma unroll
        for (int i = 1; i < nf; ++i)
          slot(2 * nf + i, r)[i0] = mk<C>(pw.feta(c.x, e[i].x, S2.x), pw.feta(c.y, e[i].y, S2.y));
      } else {
        slot(2 * nf, r)[i0] = pw.fc2(c, h);
        const C chem = vfma(c, vsplat<C>(A), vsplat<C>(B));  // 30 rho2 dcab (cab - 2c)
#pragma unroll
        for (int i = 1; i < nf; ++i) {
          const C ne = mk<C>(-e[i].x, -e[i].y), q = vfma(e[i], ne, e[i]);
          const C in = vfma(chem, q, vfma(e[i], vsplat<C>(T(-2) * W), vsplat<C>(W)));
          slot(2 * nf + i, r)[i0] = P == 1 ? vmul(q, in)  // no other eta
                                           : vfma(q, in, vmul(vmul(e[i], vsplat<C>(F)), vfma(e[i], ne, S2)));
        }
      }
    }
  }
  __syncthreads();
  C* spec = reinterpret_cast<C*>(a.spec);
  {
    const int o = w;
    C* s = slot(o, g);
    auto st = [s](int i, C v) { s[Cfg::P16 ? pad16(i) : pad32(i)] = v; };
    auto ld = [s](int i) { return s[Cfg::P16 ? pad16(i) : pad32(i)]; };
    C v[E];
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = s[t + TPL * m];
    adj_line_fft<L, E, -1>(v, t, twr, st, ld, wsync);
    wsync();
#pragma unroll
    for (int m = 0; m < E; ++m) s[t + TPL * m] = v[m];
    wsync();
    C* dst = spec + o * a.slot_stride + row * L;
    if (active) {
#pragma unroll
      for (int m = 0; m < E; ++m) {
        const int k = t + TPL * m;
        const C zk = s[k];
        C out;
        if (k == 0) {
          out = mk<C>(T(2) * (zk.x + zk.y), T(2) * (zk.x - zk.y));
        } else {
          const C zm = cconj(s[L - k]);
          const C A = cadd(zk, zm), B = csub(zk, zm);
          out = cadd(A, mul_i<-1>(adj_cmul(B, __ldg(&twh[k]))));
        }
        dst[k] = out;
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Adjoint column pass: one CTA per (kx tile, field phi).  Loads the tiles of
// lam'_phi, u_phi, f_phi; forward y; sensitivities into acc[0..3]; writes
// D1 lam'^ (slot phi) and D2 lam'^ (slot nf + phi), inverse y, scaled 1/(2N).
// ---------------------------------------------------------------------------
// A field kind has two parameters: the rate (M or L) and its gradient
// coefficient; their sums accumulate per thread in FP64, or in FP32 as exact
// products added into an unevaluated pair (two-sum, about 48 bits): GB300 issues
// one FP64 instruction where it issues 32 to 64 FP32 ones, and with FP64 sums
// (six conversions and four products per mode) the 512^2, p = 2 column pass takes
// 51 us against 27.  A pair is as good as FP64 only while its products neither
// overflow nor come so close to the end of the range that their rounding errors
// vanish (an error is at least 2^-149, so 2^-69 of the largest product at 2^-80);
// a thread whose largest product is outside (2^-80, 2^120) -- a strongly scaled
// cotangent -- adds its modes again in FP64.
template <typename T>
struct AdjSum;
template <>
struct AdjSum<double> {
  double s = 0.0;
  template <typename V> __device__ __forceinline__ void add(V a, V b) { s = fma((double)a, (double)b, s); }
  __device__ __forceinline__ double value() const { return s; }
  __device__ __forceinline__ bool in_range() const { return true; }
};
template <>
struct AdjSum<float> {
  float hi = 0.f, lo = 0.f, most = 0.f;
  __device__ __forceinline__ void add(float a, float b) {
    const float p = __fmul_rn(a, b), e = fmaf(a, b, -p);  // a b = p + e
    const float t = __fadd_rn(hi, p), v = __fadd_rn(t, -hi);
    lo = __fadd_rn(lo, __fadd_rn(__fadd_rn(__fadd_rn(hi, -__fadd_rn(t, -v)), __fadd_rn(p, -v)), e));
    hi = t;
    most = fmaxf(most, fabsf(p));
  }
  __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
  // (an underflow to zero throughout is out of range too, unless lam' is zero: FP64 adds the same zeros)
  __device__ __forceinline__ bool in_range() const { return most > 8.2718061e-25f && most < 1.3292279e36f; }
};

template <typename T>
struct AdjCoef {
  T Mdt, Ldt, kc, ke, dt;
  __device__ explicit AdjCoef(const KArgs& a) {
    const Coef<T>& co = coef<T>(a);
    Mdt = co.Mdt;
    Ldt = co.Ldt;
    kc = co.kc;
    ke = co.ke;
    dt = co.dt;
  }
  // 1 / y rounded, y >= 1: one Newton step from the hardware's approximation
  // (1 ulp) is the rounded reciprocal for every FP32 mantissa (all 2^23 tried),
  // as long as it is a normal number; the factors 1/16 keep the step in range up
  // to the largest y.  No branches: 32 rounded divisions in a thread's modes
  // took 9 us of 36 of the 512^2, p = 2 column pass.
  __device__ __forceinline__ static float recip(float y) {
    const float s = y * 0.0625f;
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(s));
    r = fmaf(r, fmaf(-s, r, 1.f), r) * 0.0625f;
    return y <= 3.402823466e38f ? r : (y != y ? y : 0.f);
  }
  // One mode at K2 of field kind f (0: c): va = D1 lam', vb = D2 lam' (times
  // scale), and Re conj(lam') (dD1 u + dD2 f) of its two parameters into r, g.
  template <typename C, class Sum>
  __device__ __forceinline__ void mode(int f, T k2, T scale, C l, C u, C fu, C& va, C& vb, Sum& r, Sum& g) const {
    T d1, d2, r1, r2, g1, g2;  // D1, D2, their d/d rate, their d/d kappa
    if constexpr (sizeof(T) == 4) {  // rounded quotients: the sensitivities keep their digits
      if (f == 0) {
        const T den = T(1) + Mdt * kc * k2 * k2, i2 = recip(den * den);
        d1 = recip(den);
        d2 = -Mdt * k2 * d1;
        r1 = -dt * kc * k2 * k2 * i2;
        r2 = -dt * k2 * i2;
        g1 = -Mdt * k2 * k2 * i2;
        g2 = Mdt * Mdt * k2 * k2 * k2 * i2;
      } else {
        const T den = T(1) + Ldt * ke * k2, i2 = recip(den * den);
        d1 = recip(den);
        d2 = -Ldt * d1;
        r1 = -dt * ke * k2 * i2;
        r2 = -dt * i2;
        g1 = -Ldt * k2 * i2;
        g2 = Ldt * Ldt * k2 * i2;
      }
    } else {
      const T kk = f == 0 ? k2 * k2 : k2, rate = f == 0 ? Mdt : Ldt, kap = f == 0 ? kc : ke, m2 = f == 0 ? k2 : T(1);
      d1 = KUpdate<T>::quot(T(1), T(1) + rate * kap * kk);
      const T i2 = d1 * d1;
      d2 = -rate * m2 * d1;
      r1 = -dt * kap * kk * i2;
      r2 = -dt * m2 * i2;
      g1 = -rate * kk * i2;
      g2 = rate * rate * kk * m2 * i2;
    }
    va = cscale(l, d1 * scale);
    vb = cscale(l, d2 * scale);
    const C tr = vfma(u, vsplat<C>(r1), vmul(fu, vsplat<C>(r2))), tg = vfma(u, vsplat<C>(g1), vmul(fu, vsplat<C>(g2)));
    r.add(l.x, tr.x);
    r.add(l.y, tr.y);
    g.add(l.x, tg.x);
    g.add(l.y, tg.y);
  }
  // The E modes of a thread, one(m, va, vb, r, g) each: into FP32 pairs, and
  // again into FP64 where the pairs left their range.
  template <int E, typename C, class One>
  __device__ __forceinline__ static void modes(One one, C (&va)[E], C (&vb)[E], double& r, double& g) {
    AdjSum<T> sr, sg;
#pragma unroll
    for (int m = 0; m < E; ++m) one(m, va[m], vb[m], sr, sg);
    r = sr.value();
    g = sg.value();
    if (!sr.in_range() || !sg.in_range()) {
      AdjSum<double> dr, dg;
#pragma unroll 1
      for (int m = 0; m < E; ++m) {
        C a, b;
        one(m, a, b, dr, dg);
      }
      r = dr.value();
      g = dg.value();
    }
  }
  // The sums of a warp, each thread's times its weight w, into acc (c: M and
  // kappa_c; eta: L and kappa_eta).
  __device__ __forceinline__ static void reduce(int f, double r, double g, double w, double* acc) {
    double v[2] = {w * r, w * g};
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      v[q] = warp_sum(v[q]);
      if ((threadIdx.x & 31) == 0 && v[q] != 0.0) atomicAdd(&acc[2 * q + (f == 0 ? 0 : 1)], v[q]);
    }
  }
};

// Columns per CTA of the adjoint column pass: about 64 threads (tiles of 16
// bytes or more per row), so that the pass reaches every SM on small grids:
// three transforms forward and two back per tile and field, 512^2, p = 2,
// FP32: 105 us with 96 CTAs of 256 threads, 27 us now.
template <typename T, int NY>
struct AdjColCfg {
  using CC = ColCfg<T, NY>;
  static constexpr int T0 = col_tk(NY, CC::F64, 64);
  static constexpr int TK = (!CC::F64 && T0 < 2) ? 2 : T0;
  // a whole number of warps (the shuffles of the sums)
  static constexpr int THREADS = TK * CC::TPL;
  static constexpr int TWS = adj_table_size<T>(NY, CC::E);
  static constexpr int TW_BYTES = ((TWS * (int)sizeof(cplx<T>)) + 127) & ~127;
  static constexpr int HEAD = CC::BAR_BYTES + TW_BYTES + CC::K2_BYTES;
  static constexpr size_t smem(int tk) { return HEAD + (size_t)3 * CC::TROWS * tk * sizeof(cplx<T>); }
};

// TKC: columns per CTA known at compile time (0: a short x axis has fewer).
template <typename T, int NY, int TKC>
__global__ void __launch_bounds__(AdjColCfg<T, NY>::THREADS < 32 ? 32 : AdjColCfg<T, NY>::THREADS)
    fs_adj_col_kernel(KArgs a, const __grid_constant__ CUtensorMap tmap) {
  using C = cplx<T>;
  using Cfg = ColCfg<T, NY>;
  using Adj = AdjColCfg<T, NY>;
  constexpr int E = Cfg::E, TPL = Cfg::TPL, BH = Cfg::BH, TROWS = Cfg::TROWS, LOGE = Cfg::LOGE;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem_raw);
  C* twc = reinterpret_cast<C*>(smem_raw + Cfg::BAR_BYTES);
  T* k2yt = reinterpret_cast<T*>(smem_raw + Cfg::BAR_BYTES + Adj::TW_BYTES);
  C* tiles = reinterpret_cast<C*>(smem_raw + Adj::HEAD);  // [3][TROWS][tk]
  const int Lh = a.nx / 2, nf = a.nf;
  const int tk = TKC ? TKC : (AdjColCfg<T, NY>::TK < Lh ? AdjColCfg<T, NY>::TK : Lh);
  const int j = threadIdx.x % tk, t0 = threadIdx.x / tk, t = t0 & (TPL - 1);
  // a CTA is rounded up to whole warps: the threads beyond the tile repeat
  // its values without storing them
  const bool live = t0 < TPL;
  const int kx0 = blockIdx.x * tk, kx = kx0 + j, phi = blockIdx.y;
  const int fk = phi == 0 ? 0 : 1;
  const int cx = kx0 * (int)(sizeof(C) / 8);
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    griddep_wait();  // the tiles are the row pass's output
    mbar_arrive_expect_tx(bar, (uint32_t)(3 * NY * tk * sizeof(C)));
    for (int i = 0; i < 3; ++i)
      for (int y0 = 0; y0 < NY; y0 += BH) tma_load_3d(tiles + (i * TROWS + y0) * tk, &tmap, cx, y0, i * nf + phi, bar);
  }
  copy_to_smem(twc, reinterpret_cast<const C*>(a.tw_col), Adj::TWS);
  for (int i = threadIdx.x; i < NY; i += blockDim.x) k2yt[i] = reinterpret_cast<const T*>(a.k2y)[i];
  griddep_wait();
  griddep_launch_dependents();
  __syncthreads();
  if (!mbar_wait_bounded(bar, 0, first_wait_polls(a))) {
    if (threadIdx.x == 0) atomicOr(a.flag, FS_FLAG_TIMEOUT);
    mbar_wait_bounded(bar, 0, kWaitPolls);
    return;
  }
  auto sync = []() { __syncthreads(); };
  // forward y of the three tiles, results back in natural layout
#pragma unroll 1
  for (int i = 0; i < 3; ++i) {
    C* tl = tiles + i * TROWS * tk + j;
    auto st = [tl, tk, live](int q, C x) { if (live) tl[(q + (q >> LOGE)) * tk] = x; };
    auto ld = [tl, tk](int q) { return tl[(q + (q >> LOGE)) * tk]; };
    C v[E];
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = tl[(t + TPL * m) * tk];
    adj_line_fft<NY, E, -1>(v, t, twc, st, ld, sync);
    sync();
#pragma unroll
    for (int m = 0; m < E; ++m)
      if (live) tl[(t + TPL * m) * tk] = v[m];
  }
  sync();
  const AdjCoef<T> ac(a);
  const T* k2xt = reinterpret_cast<const T*>(a.k2x);
  const T kx2 = k2xt[kx], kxn2 = k2xt[Lh], scale = coef<T>(a).scale;
  const C* TL = tiles + 0 * TROWS * tk;  // Lam'
  const C* TU = tiles + 1 * TROWS * tk;  // U
  const C* TF = tiles + 2 * TROWS * tk;  // Fu
  double sr, sg;
  C va[E], vb[E];
  const bool col0 = (kx0 == 0 && j == 0);
  auto one = [&](int m, C& a1, C& a2, auto& s1, auto& s2) {
    const int ky = t + TPL * m;
    const T ky2 = k2yt[ky];
    const C l = TL[ky * tk + j], u = TU[ky * tk + j], f = TF[ky * tk + j];
    if (col0) {
      // split the packed column into its kx = 0 (P) and kx = nx/2 (Q) parts
      const int kq = (NY - ky) & (NY - 1);
      const C lq = cconj(TL[kq * tk]), uq = cconj(TU[kq * tk]), fq = cconj(TF[kq * tk]);
      const C lP = cscale(cadd(l, lq), T(0.5)), lQ = cscale(mul_i<-1>(csub(l, lq)), T(0.5));
      const C uP = cscale(cadd(u, uq), T(0.5)), uQ = cscale(mul_i<-1>(csub(u, uq)), T(0.5));
      const C fP = cscale(cadd(f, fq), T(0.5)), fQ = cscale(mul_i<-1>(csub(f, fq)), T(0.5));
      C aP, bP, aQ, bQ;
      ac.mode(fk, kx2 + ky2, scale, lP, uP, fP, aP, bP, s1, s2);
      ac.mode(fk, kxn2 + ky2, scale, lQ, uQ, fQ, aQ, bQ, s1, s2);
      a1 = cadd(aP, mul_i<1>(aQ));
      a2 = cadd(bP, mul_i<1>(bQ));
    } else {
      ac.mode(fk, kx2 + ky2, scale, l, u, f, a1, a2, s1, s2);
    }
  };
  AdjCoef<T>::template modes<E>(one, va, vb, sr, sg);
  // the conjugate half of the columns kx > 0 is not stored: weight 2
  AdjCoef<T>::reduce(fk, sr, sg, live ? (col0 ? 1.0 : 2.0) : 0.0, a.acc);
  sync();
  // inverse y of D1 lam'^ (exchange in tile 0, to slot phi) and D2 lam'^
  // (tile 1, to slot nf + phi), out through the tiles
  auto inverse = [&](C(&v)[E], C* tile) {
    C* tl = tile + j;
    auto st = [tl, tk, live](int q, C x) { if (live) tl[(q + (q >> LOGE)) * tk] = x; };
    auto ld = [tl, tk](int q) { return tl[(q + (q >> LOGE)) * tk]; };
    adj_line_fft<NY, E, 1>(v, t, twc, st, ld, sync);
    sync();
#pragma unroll
    for (int m = 0; m < E; ++m)
      if (live) tl[(t + TPL * m) * tk] = v[m];
  };
  inverse(va, tiles);
  inverse(vb, tiles + TROWS * tk);
  fence_proxy_async_smem();
  sync();
  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i)
      for (int y0 = 0; y0 < NY; y0 += BH) tma_store_3d(&tmap, cx, y0, i * nf + phi, tiles + (i * TROWS + y0) * tk);
    bulk_commit();
    bulk_wait_read();
  }
}

// ---------------------------------------------------------------------------
// Adjoint row inverse: inverse x transforms of G1 lam' (slots [0, nf)) and
// G2 lam' (slots [nf, 2nf)); lambda_phi = G1 lam'_phi + sum H_phi,psi G2 lam'_psi
// with H at u (a.aux, real); result to a.real (lambda_out).  2 nf warps, one
// per transform.
// ---------------------------------------------------------------------------
template <typename T, int NX, int P>
__global__ void __launch_bounds__(64 * (P + 1)) fs_adj_row_inv_kernel(KArgs a) {
  using C = cplx<T>;
  using Cfg = AdjRowCfg<T, NX>;
  constexpr int L = Cfg::L, E = Cfg::E, TPL = Cfg::TPL, R = Cfg::R, PL = Cfg::PL;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem_raw);
  C* twr = reinterpret_cast<C*>(smem_raw + Cfg::BAR_BYTES);
  C* slots = reinterpret_cast<C*>(smem_raw + Cfg::BAR_BYTES + Cfg::TW_BYTES);
  constexpr int nf = P + 1;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane / TPL, t = lane % TPL;
  const int Reff = a.lines < R ? (int)a.lines : R;
  const long long row0 = (long long)blockIdx.x * Reff;
  const C* __restrict__ twh = reinterpret_cast<const C*>(a.tw_half);
  const long long half_stride = a.npts / 2;
  auto slot = [slots](int f, int r) { return slots + (f * R + r) * PL; };
  auto wsync = []() { __syncwarp(); };
  copy_to_smem(twr, reinterpret_cast<const C*>(a.tw_row), Cfg::TWS);
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
  }
  griddep_wait();  // everything read or written below may belong to the previous grid
  griddep_launch_dependents();
  __syncthreads();
  if (threadIdx.x == 0) {
    const uint32_t bytes = (uint32_t)(L * sizeof(C));
    mbar_arrive_expect_tx(bar, bytes * Reff * 3 * nf);
    for (int f = 0; f < 2 * nf; ++f)
      for (int r = 0; r < Reff; ++r)
        bulk_g2s(slot(f, r), reinterpret_cast<const C*>(a.spec) + f * a.slot_stride + (row0 + r) * L, bytes, bar);
    for (int f = 0; f < nf; ++f)
      for (int r = 0; r < Reff; ++r)
        bulk_g2s(slot(2 * nf + f, r), reinterpret_cast<const C*>(a.aux) + f * half_stride + (row0 + r) * L, bytes,
                 bar);
  }
  if (!mbar_wait_bounded(bar, 0, first_wait_polls(a))) {
    if (threadIdx.x == 0) atomicOr(a.flag, FS_FLAG_TIMEOUT);
    mbar_wait_bounded(bar, 0, kWaitPolls);
    return;
  }
  {
    const int o = w;
    C* s = slot(o, g);
    auto st = [s](int i, C v) { s[Cfg::P16 ? pad16(i) : pad32(i)] = v; };
    auto ld = [s](int i) { return s[Cfg::P16 ? pad16(i) : pad32(i)]; };
    C v[E];
#pragma unroll
    for (int m = 0; m < E; ++m) {
      const int k = t + TPL * m;
      const C pk = s[k];
      if (k == 0) {
        v[m] = mk<C>(pk.x + pk.y, pk.x - pk.y);
      } else {
        const C pm = cconj(s[L - k]);
        const C A = cadd(pk, pm), B = csub(pk, pm);
        v[m] = cadd(A, mul_i<1>(mul_tw<1>(B, __ldg(&twh[k]))));
      }
    }
    adj_line_fft<L, E, 1>(v, t, twr, st, ld, wsync);
    wsync();
#pragma unroll
    for (int m = 0; m < E; ++m) s[t + TPL * m] = v[m];
  }
  __syncthreads();
  const Pointwise<T> pw(a);
  C* out = reinterpret_cast<C*>(a.real);
  for (int idx = threadIdx.x; idx < Reff * L; idx += blockDim.x) {
    const int r = idx / L, i0 = idx % L;
    C u[nf], mu[nf], res[nf];
#pragma unroll
    for (int f = 0; f < nf; ++f) {
      u[f] = slot(2 * nf + f, r)[i0];
      mu[f] = slot(nf + f, r)[i0];
    }
    hessian_apply<P, T>(pw, u, mu, res);
#pragma unroll
    for (int f = 0; f < nf; ++f) out[f * half_stride + (row0 + r) * L + i0] = cadd(slot(f, r)[i0], res[f]);
  }
}

}  // namespace fs
