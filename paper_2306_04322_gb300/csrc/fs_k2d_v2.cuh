// Warp-per-line forms of the row and column passes.  FP32: every line
// transform is held by one warp, E = L / 32 values per thread (radix 32 x 32
// at L = 1024: one exchange), so the FFT exchanges synchronise the warp only;
// CTA-wide barriers remain only where fields meet (the pointwise stage of the
// row pass) and named 64-thread barriers where the column pass hands df/dc^
// to the c update.  FP64: G warps per line with 2 to 8 values per thread
// (see row2_g64).
//
// Row pass, pair form.  Grid rows a and b of one field are transformed as
// the single complex line z = a + i b of length nx:
//   inverse: Z[k] = X_a[k] + i X_b[k] over all nx bins, built from the two
//            packed half spectra with X[nx - k] = conj X[k]; the inverse DFT
//            of Z gives a + i b at once;
//   forward: Z = DFT(g_a + i g_b), then 2 X_a[k] = Z[k] + conj Z[nx - k]
//            and 2 X_b[k] = -i (Z[k] - conj Z[nx - k]) (k <= nx/2), which is
//            the factor-2 scaling the column pass expects.
// The two rows' values sit in the two lanes of a float2 in real space, so the
// pointwise derivative stage (Section 2.1 definitions) runs lane-wise on the
// pair.  Modes as the row pass of fs_kernels.cuh: 0 step from spectra, 1 step
// from real fields, 2 inverse only (mode 3, the free-energy diagnostic, keeps
// the half-length kernel).
//
// Column pass, warp per column.  A CTA holds one, two or four adjacent kx
// columns (16- or 32-byte TMA rows) of one field group -- {df/dc, c} or one or
// two eta -- one warp (FP64 and 2048 points: several) per (slot, column).  All warps transform forward; the df/dc warps publish their
// result for the c warps of the same column, and the c and eta warps apply
// the k-space update (Eqs. A-C_discrete_fft_c, A-C_discrete_fft_eta) and
// transform back.
#pragma once

#include "fs_k2d_impl.cuh"

namespace fs {

// Padded exchange layout of a line: FP32 one spare slot every 32 elements;
// FP64 (16-byte elements, 8 lanes per shared-memory wavefront) every 8, so
// that the writes of E consecutive elements per thread fall on different
// banks (every 16 at 2048 points, where six padded areas must fit an SM).
template <typename T, int L>
__device__ __forceinline__ int line_pad(int i) {
  if constexpr (sizeof(T) == 4) return pad32(i);
  else return i + (i >> (L >= 2048 ? 4 : 3));
}
template <typename T>
constexpr int line_pad_len(int L) {
  return sizeof(T) == 4 ? (padded_len(L) + 1) & ~1 : L + (L >> (L >= 2048 ? 4 : 3)) + 1;
}

// G warps per line (FP32: 1, or 2 to double the warps in flight when lines
// are few); a line's TPL = 32 G threads hold E = NX / TPL values each.
template <typename T, int NX, int G = 1>
struct Row2Cfg {
  static constexpr bool F64 = sizeof(T) == 8;
  static constexpr int TPL = 32 * G;                          // threads per line
  static constexpr int E = NX / TPL;                          // values per thread
  static constexpr int H = NX / 2;                            // packed bins per row
  static constexpr int PL = line_pad_len<T>(NX);           // complex per field area (16-byte multiple)
  static constexpr int TWS = pass_table_size(NX, E);
  static constexpr int TW_BYTES = ((TWS * (int)sizeof(cplx<T>)) + 127) & ~127;
  static constexpr int BAR_BYTES = 128;
  static constexpr int MAX_THREADS = TPL * 5;                 // one line per field, nf <= 5
};

// One area per field; df/dc takes c's place after the pointwise stage, but for
// mode 1, whose forward phase still needs c (the area it saves is a CTA or two
// more per SM: a 64-member ensemble, with the tighter register budgets of its
// kernels, 403 us per step against 431).
template <typename T, int NX, int G = 1>
constexpr size_t row2_smem_bytes(int nf, int mode) {
  using Cfg = Row2Cfg<T, NX, G>;
  return Cfg::BAR_BYTES + Cfg::TW_BYTES + (size_t)(nf + (mode == 1 ? 1 : 0)) * Cfg::PL * sizeof(cplx<T>);
}

// Synchronisation of the threads of one line: the warp itself, or the G
// warps of a line through named barrier BASE + line (32 G threads).  With an
// id in a register a kernel reserves all 16 barriers, which limits an SM to
// four CTAs; CONST takes compile-time ids from a warp-uniform switch instead
// (the small FP64 CTAs; the FP32 columns of 2048, two CTAs per SM, lost 5 % to
// the longer code).
template <int G, int BASE, bool CONST>
struct LineSync {
  int line;
  __device__ __forceinline__ void operator()() const {
    if constexpr (G == 1) {
      __syncwarp();
    } else if constexpr (!CONST) {
      bar_sync(BASE + line, 32 * G);
    } else {
      switch (line) {
        case 0: bar_sync(BASE, 32 * G); break;
        case 1: bar_sync(BASE + 1, 32 * G); break;
        case 2: bar_sync(BASE + 2, 32 * G); break;
        case 3: bar_sync(BASE + 3, 32 * G); break;
        default: bar_sync(BASE + 4, 32 * G); break;
      }
    }
  }
};

// Pointwise stage of the pair-form row pass (Section 2.1 derivatives, lane-
// wise on the two rows of a pair) with p = P known at compile time: U (FP32:
// four) independent points per iteration -- all loads, then the arithmetic, then
// the stores (points past the rows repeat point n).  areas: [nf][PR][PL]
// (PR row pairs), c, eta_i (replaced by g_i); df/dc to the area at fcd (may be
// c's own).  df/dc is non-finite
// whenever c or any eta_i is (see the row pass of fs_kernels.cuh), so testing
// it covers all inputs.
template <typename T, int P, int NX, int PL, int PR = 1>
__device__ __forceinline__ void row2_pointwise_fixed(const Pointwise<T>& pw, cplx<T>* areas, cplx<T>* fcd, bool& bad) {
  using C = cplx<T>;
  constexpr int PE = P > 0 ? P : 1, U = sizeof(T) == 4 ? 4 : 1;  // FP64: bound by its pipe, not by latency
  constexpr int FS = PR * PL;
  for (int n = threadIdx.x; n < PR * NX; n += U * blockDim.x) {
    int k[U];
    C c[U], e[U][PE], fc[U], g[U][PE];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      k[u] = n + u * (int)blockDim.x < PR * NX ? n + u * (int)blockDim.x : n;
      if (PR > 1) k[u] = (k[u] / NX) * PL + k[u] % NX;
      c[u] = areas[k[u]];
#pragma unroll
      for (int i = 0; i < P; ++i) e[u][i] = areas[(1 + i) * FS + k[u]];
    }
    FiniteCheck<T> chk;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      C h = vsplat<C>(T(0)), S2 = vsplat<C>(T(0));
#pragma unroll
      for (int i = 0; i < P; ++i) {
        h = pw.add_h2(e[u][i], h);
        S2 = vfma(e[u][i], e[u][i], S2);
      }
      fc[u] = pw.fc2(c[u], h);
      chk.add(fc[u]);
#pragma unroll
      for (int i = 0; i < P; ++i) g[u][i] = pw.template g2<P == 1>(c[u], e[u][i], S2);
    }
    bad |= chk.bad();
#pragma unroll
    for (int u = 0; u < U; ++u) {
      fcd[k[u]] = fc[u];
#pragma unroll
      for (int i = 0; i < P; ++i) areas[(1 + i) * FS + k[u]] = g[u][i];
    }
  }
}

// One row pair (rows 2 pair and 2 pair + 1) of the simulation `a`, one warp
// per field (blockDim = 32 nf).  Field areas [nf][PL], one more in mode 1
// (row2_smem_bytes): staging of the bulk copies, then the warp's exchange buffer (pad32
// layout), then the pair values in natural order for the pointwise stage.
// `bar` is an initialised mbarrier whose next phase has parity `parity` (the
// fused step takes several items with one).  Returns false if a bounded wait
// gave up.  PC >= 0: the caller guarantees nf = PC + 1, and the
// pointwise stage is compiled for that p alone (the 96-thread kernel, whose
// nf is 3: a kernel holding the code for every p measured slower there).
// EARLY: see griddep_launch_dependents.
template <typename T, int NX, int G = 1, int PC = -1, bool EARLY = false>
__device__ __forceinline__ bool row2_body(const KArgs& a, long long pair, unsigned char* smem_raw, uint64_t* bar,
                                          uint32_t parity) {
  using C = cplx<T>;
  using Cfg = Row2Cfg<T, NX, G>;
  constexpr int E = Cfg::E, H = Cfg::H, PL = Cfg::PL, TPL = Cfg::TPL;
  C* tw = reinterpret_cast<C*>(smem_raw + Cfg::BAR_BYTES);
  C* areas = reinterpret_cast<C*>(smem_raw + Cfg::BAR_BYTES + Cfg::TW_BYTES);
  const int nf = a.nf;
  C* fcd = a.mode == 1 ? areas + nf * PL : areas;  // area of df/dc
  const int line = (threadIdx.x >> 5) / G, t = threadIdx.x % TPL;  // line of this thread, thread within it
  const int nw = blockDim.x / TPL;  // lines per CTA = nf
  const long long row0 = 2LL * pair;  // row a; row b = row0 + 1
  const LineSync<G, 1, Cfg::F64> lsync{line};
  const bool from_real = (a.mode == 1);

  if (threadIdx.x == 0) {
    // the fused step reuses the areas: order the previous item's generic
    // accesses (ended by the caller's CTA barrier) before the bulk writes
    fence_proxy_async_smem();
    // both rows of a field are contiguous: NX complex (packed) or 2 NX reals
    const uint32_t bytes = (uint32_t)(NX * sizeof(C));
    const uint32_t tbytes = (uint32_t)(Cfg::TWS * sizeof(C));
    mbar_arrive_expect_tx(bar, tbytes + bytes * nf);
    // the constant pass table first, overlapping the previous grid's tail
    bulk_g2s(tw, G == 1 || Cfg::F64 ? a.tw_row2 : a.tw_row2w, tbytes, bar);
    griddep_wait();  // the spectra are the previous pass's output
    const C* spec = reinterpret_cast<const C*>(a.spec);
    const T* real = reinterpret_cast<const T*>(a.real);
    for (int f = 0; f < nf; ++f) {
      // 3D carry: c's x spectrum sits in slot nf
      const int sl = (f == 0 && a.carry3) ? nf : f;
      const void* src = from_real ? (const void*)(real + f * a.npts + row0 * NX)
                                  : (const void*)(spec + sl * a.slot_stride + row0 * H);
      if (from_real ? real_ok(a, src, bytes) : spec_ok(a, src, bytes)) bulk_g2s(areas + f * PL, src, bytes, bar);
    }
  }
  // all threads: the bounded wait starts when the copies do, however long the
  // previous pass takes, and no lane of warp 0 polls before lane 0 has issued
  griddep_wait();
  __syncwarp();
  if (EARLY) griddep_launch_dependents();
  if (!mbar_wait_bounded(bar, parity, first_wait_polls(a))) {
    if (threadIdx.x == 0) atomicOr(a.flag, FS_FLAG_TIMEOUT);
    mbar_wait_bounded(bar, parity, kWaitPolls);  // let the copies land before exiting
    return false;
  }

  C* spec = reinterpret_cast<C*>(a.spec);
  T* real = reinterpret_cast<T*>(a.real);
  bool bad = false;
  // Both transform phases share one FFT call site (the inverse is computed as
  // conj(FFT(conj(.)))): ph 0 inverse of the nf fields (modes 0, 2; mode 1
  // only interleaves the real rows), ph 1 forward of g_1..g_p and df/dc (and
  // of c in mode 1).
  for (int ph = 0; ph < 2; ++ph) {
    const bool inv = (ph == 0);
    const int f0 = inv ? 0 : (from_real ? 0 : 1);
    const int items = nf + 1 - f0 - (inv ? 1 : 0);  // inverse: fields 0..nf-1; forward: f0..nf
    for (int i = line; i < items; i += nw) {
      const int f = f0 + i;
      C* s = f == nf ? fcd : areas + f * PL;
      auto st = [s](int q, C x) { s[line_pad<T, NX>(q)] = x; };
      auto ld = [s](int q) { return s[line_pad<T, NX>(q)]; };
      C v[E];
      if (inv) {
        if (from_real) {
          // rows a and b (NX reals each) -> pairs (a[n], b[n]) in natural order
          const T* r = reinterpret_cast<const T*>(s);
          T xa[E], xb[E];
#pragma unroll
          for (int m = 0; m < E; ++m) {
            xa[m] = r[t + TPL * m];
            xb[m] = r[NX + t + TPL * m];
          }
          lsync();
#pragma unroll
          for (int m = 0; m < E; ++m) s[t + TPL * m] = mk<C>(xa[m], xb[m]);
          continue;
        }
        // conj(Z), Z[k] = X_a[k] + i X_b[k]; staging: row a bins [0, H), row b [H, 2H);
        // bin 0 of a packed row holds (X[0], X[H]), both real
#pragma unroll
        for (int m = 0; m < E; ++m) {
          const int k = t + TPL * m;
          C z;
          if (k < H) {
            const C xa = s[k], xb = s[H + k];
            z = (k == 0) ? mk<C>(xa.x, xb.x) : cadd(xa, mul_i<1>(xb));
          } else if (k == H) {
            z = mk<C>(s[0].y, s[H].y);
          } else {
            const C xa = s[NX - k], xb = s[H + NX - k];
            z = cadd(cconj(xa), mul_i<1>(cconj(xb)));
          }
          v[m] = cconj(z);
        }
        lsync();  // the staging area becomes the exchange buffer
      } else {
#pragma unroll
        for (int m = 0; m < E; ++m) v[m] = s[t + TPL * m];  // z = g_a + i g_b, natural order
      }
      line_fft<NX, E, -1>(v, t, tw, st, ld, lsync);
      if (!EARLY && !inv) griddep_launch_dependents();
      if (inv) {
        // a + i b = conj(v)
        if (a.mode == 2) {
          T* ra = real + f * a.npts + row0 * NX;
#pragma unroll
          for (int m = 0; m < E; ++m) {
            const int n = t + TPL * m;
            if (real_ok(a, &ra[n], sizeof(T))) ra[n] = v[m].x;
            if (real_ok(a, &ra[NX + n], sizeof(T))) ra[NX + n] = -v[m].y;
          }
        } else {
          lsync();
#pragma unroll
          for (int m = 0; m < E; ++m) s[t + TPL * m] = cconj(v[m]);
        }
      } else {
        // separate the two rows' spectra; Z[nx - k] through shared memory
        lsync();
#pragma unroll
        for (int m = 0; m < E; ++m) s[t + TPL * m] = v[m];
        lsync();
        const bool c_carried = (f == 0);  // mode 1: c stored as x spectrum / nx
        const T cs = c_carried ? T(0.5) / T(NX) : T(1);
        C* Pa = spec + f * a.slot_stride + row0 * H;
        C* Pb = Pa + H;
#pragma unroll
        for (int m = 0; m < E / 2; ++m) {
          const int k = t + TPL * m;
          const C zk = v[m];
          C pa, pb;
          if (k == 0) {
            const C zh = s[H];
            pa = mk<C>(T(2) * zk.x, T(2) * zh.x);
            pb = mk<C>(T(2) * zk.y, T(2) * zh.y);
          } else {
            const C zm = s[NX - k];
            pa = cadd(zk, cconj(zm));
            pb = cadd(mul_i<-1>(zk), mul_i<1>(cconj(zm)));
          }
          if (c_carried) {
            pa = cscale(pa, cs);
            pb = cscale(pb, cs);
          }
          if (spec_ok(a, &Pa[k], sizeof(C))) Pa[k] = pa;
          if (spec_ok(a, &Pb[k], sizeof(C))) Pb[k] = pb;
        }
      }
    }
    if (!inv) break;
    if (a.mode == 2) return true;
    __syncthreads();

    // pointwise stage: pairs (row a, row b) of every field, lane-wise
    const Pointwise<T> pw(a);
    if constexpr (PC >= 0) {
      row2_pointwise_fixed<T, PC, NX, PL>(pw, areas, fcd, bad);
    } else {
      switch (nf) {  // p known at compile time for every supported field count
        case 1: row2_pointwise_fixed<T, 0, NX, PL>(pw, areas, fcd, bad); break;
        case 2: row2_pointwise_fixed<T, 1, NX, PL>(pw, areas, fcd, bad); break;
        case 3: row2_pointwise_fixed<T, 2, NX, PL>(pw, areas, fcd, bad); break;
        case 4: row2_pointwise_fixed<T, 3, NX, PL>(pw, areas, fcd, bad); break;
        case 5: row2_pointwise_fixed<T, 4, NX, PL>(pw, areas, fcd, bad); break;
        default: break;
      }
    }
    __syncthreads();
  }
  if (bad) atomicOr(a.flag, FS_FLAG_NONFINITE);
  return true;
}

// Several row pairs per CTA (FP32, rows of 64 to 512 points of 3D grids and of
// 2D grids with many rows; steady steps and the inverse only: modes 0 and 2).
// Such a pass has rows enough for every SM, so what counts is instructions, not
// the reach of a few rows over the chip: 16 values per thread and 4 to 32
// threads per line (two register passes, one exchange), so that one warp per
// field carries PR = 32 / TPL pairs
// and the table fetch and the set-up are shared by them.  Against the
// half-length kernel (one real row per line of nx / 2, with its real <->
// half-length step), 256^3, p = 2: 97 us per pass against 118.  Small CTAs, so
// that an SM always has some in each of load, transform and store: with two
// warps per field a step takes 284 us (p = 4: 481) against 281 (464), with
// four 302 (471); 64x256x256, p = 4: 124 against 116; 512-point rows, p = 1,
// whose CTAs then hold a single pair: 96.5 against 97.
template <int NX>
struct Row3Cfg {
  static constexpr int E = 16, TPL = NX / E, PR = 32 / TPL, H = NX / 2;
  // pitch of a line's area: pad16 layout, a multiple of 16 bytes, and = TPL
  // (mod 16) where a warp holds several lines, so that a half-warp's lines
  // start on different banks
  static constexpr int PL0 = (padded16_len(NX) + 1) & ~1;
  static constexpr int PL = TPL < 16 ? PL0 + ((TPL - PL0 % 16) + 16) % 16 : PL0;
  static constexpr int TWS = pass_table_size(NX, E);
  static constexpr int TW_BYTES = ((TWS * 8) + 127) & ~127;
  static constexpr size_t smem(int nf) { return 128 + TW_BYTES + (size_t)nf * PR * PL * 8; }
};

// NW: the most fields (warps) the instantiation takes.
template <int NX, int NW>
__global__ void __launch_bounds__(32 * NW, NW == 3 ? 10 : 6) fs_row3_kernel(KArgs a) {
  using C = float2;
  using Cfg = Row3Cfg<NX>;
  constexpr int E = Cfg::E, TPL = Cfg::TPL, PR = Cfg::PR, PL = Cfg::PL, H = Cfg::H;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem_raw);
  C* tw = reinterpret_cast<C*>(smem_raw + 128);
  C* areas = reinterpret_cast<C*>(smem_raw + 128 + Cfg::TW_BYTES);  // [nf][PR][PL], df/dc over c
  const int nf = a.nf;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, t = lane % TPL;
  const int q = lane / TPL;                              // the line's pair; the warp's field is w
  const long long row0 = 2LL * PR * blockIdx.x;          // first row of the CTA
  C* spec = reinterpret_cast<C*>(a.spec);
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
    mbar_arrive_expect_tx(bar, (uint32_t)(Cfg::TWS * sizeof(C) + nf * PR * NX * sizeof(C)));
    bulk_g2s(tw, a.tw_row3, (uint32_t)(Cfg::TWS * sizeof(C)), bar);
  }
  griddep_wait();  // the spectra are the previous pass's output
  if (a.nz > 1) griddep_launch_dependents();  // 2D: after the last transform, as row2_body
  if (w == 0) {
    __syncwarp();
    for (int i = lane; i < nf * PR; i += 32) {
      const int f = i / PR, sl = (f == 0 && a.carry3) ? nf : f;  // 3D carry: c's x spectrum sits in slot nf
      const C* src = spec + sl * a.slot_stride + (row0 + 2 * (i % PR)) * H;
      if (spec_ok(a, src, NX * sizeof(C))) bulk_g2s(areas + i * PL, src, NX * sizeof(C), bar);
    }
  }
  __syncthreads();
  if (!mbar_wait_bounded(bar, 0, first_wait_polls(a))) {
    if (threadIdx.x == 0) atomicOr(a.flag, FS_FLAG_TIMEOUT);
    mbar_wait_bounded(bar, 0, kWaitPolls);  // let the copies land before exiting
    return;
  }
  bool bad = false;
  auto wsync = []() { __syncwarp(); };
  for (int ph = 0; ph < 2; ++ph) {
    const int f = w + ph;  // inverse: fields 0..nf-1; forward: g_1..g_p and df/dc
    C* s = areas + ((f == nf ? 0 : f) * PR + q) * PL;
    auto st = [s](int i, C x) { s[pad16(i)] = x; };
    auto ld = [s](int i) { return s[pad16(i)]; };
    C v[E];
    if (ph == 0) {
      // conj(Z), Z[k] = X_a[k] + i X_b[k] (as row2_body)
#pragma unroll
      for (int m = 0; m < E; ++m) {
        const int k = t + TPL * m;
        if (m < E / 2) {
          const C xa = s[k], xb = s[H + k];
          v[m] = cadd(cconj(xa), mul_i<-1>(cconj(xb)));
          if (m == 0 && t == 0) v[m] = mk<C>(xa.x, -xb.x);
        } else {
          const int kr = (m == E / 2 && t == 0) ? 0 : NX - k;
          const C xa = s[kr], xb = s[H + kr];
          v[m] = cadd(xa, mul_i<-1>(xb));
          if (m == E / 2 && t == 0) v[m] = mk<C>(xa.y, -xb.y);
        }
      }
      __syncwarp();  // the staging area becomes the exchange buffer
    } else {
#pragma unroll
      for (int m = 0; m < E; ++m) v[m] = s[t + TPL * m];
    }
    line_fft<NX, E, -1>(v, t, tw, st, ld, wsync);
    if (ph == 1 && a.nz == 1) griddep_launch_dependents();
    if (ph == 0) {
      if (a.mode == 2) {
        float* ra = reinterpret_cast<float*>(a.real) + f * a.npts + (row0 + 2 * q) * NX;
#pragma unroll
        for (int m = 0; m < E; ++m) {
          const int n = t + TPL * m;
          if (real_ok(a, &ra[n], 4)) ra[n] = v[m].x;
          if (real_ok(a, &ra[NX + n], 4)) ra[NX + n] = -v[m].y;
        }
        return;
      }
      __syncwarp();
#pragma unroll
      for (int m = 0; m < E; ++m) s[t + TPL * m] = cconj(v[m]);
      __syncthreads();
      const Pointwise<float> pw(a);
      switch (nf) {
        case 1: row2_pointwise_fixed<float, 0, NX, PL, PR>(pw, areas, areas, bad); break;
        case 2: row2_pointwise_fixed<float, 1, NX, PL, PR>(pw, areas, areas, bad); break;
        case 3: row2_pointwise_fixed<float, 2, NX, PL, PR>(pw, areas, areas, bad); break;
        case 4: row2_pointwise_fixed<float, 3, NX, PL, PR>(pw, areas, areas, bad); break;
        default: row2_pointwise_fixed<float, 4, NX, PL, PR>(pw, areas, areas, bad); break;
      }
      __syncthreads();
    } else {
      // separate the two rows' spectra; Z[nx - k] through shared memory
      __syncwarp();
#pragma unroll
      for (int m = 0; m < E; ++m) s[t + TPL * m] = v[m];
      __syncwarp();
      C* Pa = spec + f * a.slot_stride + (row0 + 2 * q) * H;
      C* Pb = Pa + H;
#pragma unroll
      for (int m = 0; m < E / 2; ++m) {
        const int k = t + TPL * m;
        const C zk = v[m], zm = s[(m == 0 && t == 0) ? H : NX - k];
        C pa = cadd(zk, cconj(zm)), pb = cadd(mul_i<-1>(zk), mul_i<1>(cconj(zm)));
        if (m == 0 && t == 0) {
          pa = mk<C>(2.f * zk.x, 2.f * zm.x);
          pb = mk<C>(2.f * zk.y, 2.f * zm.y);
        }
        if (spec_ok(a, &Pa[k], sizeof(C))) Pa[k] = pa;
        if (spec_ok(a, &Pb[k], sizeof(C))) Pb[k] = pb;
      }
    }
  }
  if (bad) atomicOr(a.flag, FS_FLAG_NONFINITE);
}

template <int NX, int NW>
cudaError_t row3_launch_nw(const KArgs& a, cudaStream_t s) {
  using Cfg = Row3Cfg<NX>;
  static unsigned done = 0;
  cudaError_t e = allow_big_smem(fs_row3_kernel<NX, NW>, &done);
  if (e != cudaSuccess) return e;
  return launch_pdl(fs_row3_kernel<NX, NW>, dim3((unsigned)(a.lines / (2 * Cfg::PR))), dim3((unsigned)(32 * a.nf)),
                    Cfg::smem(a.nf), s, a);
}

// NW: the most warps per line group the instantiation takes (nf <= NW).
// With one warp per line and nf = 3 the register budget is that of four
// 96-thread CTAs per SM (170 per thread; a pass of 1024 rows stays one
// wave), which leaves the compiler room to schedule the values of each
// thread; otherwise three 160-thread CTAs (136).  Measured (L2 flushed
// before each step, p = 2): 512^2 step 17.1 us against 19.1 us, 1024^2
// unchanged; with nf = 2 the 1024^2 step lost 4 %, so only nf = 3 takes it.
// FP64: as many CTAs as leave the registers of E values per thread.
template <typename T, int G, int NW>
constexpr int row2_min_blocks() {
  if (sizeof(T) == 8) return 32 * G * NW > 400 ? 1 : (32 * G * NW > 250 ? 2 : 4);
  return (G == 1 && NW <= 3) ? 4 : (G == 1 ? 3 : 2);
}
template <typename T, int NX, int G, int NW>
__global__ void __launch_bounds__(32 * G * NW, row2_min_blocks<T, G, NW>())
    fs_row2_kernel(KArgs a) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem_raw);
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  row2_body<T, NX, G, (sizeof(T) == 4 && G == 1 && NW == 3) ? 2 : -1>(a, blockIdx.x, smem_raw, bar, 0);
}

// A column CTA: NR regions (slots) of TK adjacent kx columns, one line of
// 32 G threads per (region, column).  Wide tiles matter: TMA takes 1.5 cycles
// of an SM for a tile row of 16 or of 32 bytes alike (measured: copies in 16-,
// 32- and 64-byte rows run at 3.3, 6.0 and 8.2 TB/s), and 16-byte rows alone
// made 9 us of a 1024^2 pass (p = 2, FP32).  Four FP32 columns (32-byte rows)
// come in with the 32-byte swizzle, which puts rows four apart on different
// banks when a warp reads its column.
template <typename T, int NY, int G, int TK_, int NR_>
struct Col2Cfg {
  static constexpr bool F64 = sizeof(T) == 8;
  static constexpr int CS = 2 * (int)sizeof(T);               // bytes of a complex value
  static constexpr int TPL = 32 * G;                          // threads per line
  static constexpr int E = NY / TPL;
  static constexpr int TK = TK_, NR = NR_;
  static constexpr int NE = F64 ? 1 : NR;                     // eta_i per field group
  static constexpr int THREADS = TPL * TK * NR;
  static constexpr bool SWZ = TK * CS == 32;                  // 32-byte rows: swizzled (box of encode_col_map)
  static constexpr int BH = NY < 256 ? NY : 256;              // TMA box height (rows)
  static constexpr int PL = line_pad_len<T>(NY);              // complex per compact column area
  // slot region: the [NY][TK] tile as loaded, then TK compact areas, then the
  // [NY][TK] tile again for the TMA store; every region starts on 256 bytes
  // (TMA, the swizzle's period)
  static constexpr int SLOT = (((NY * TK > TK * PL) ? NY * TK : TK * PL) + 31) & ~31;
  static constexpr int TWS = pass_table_size(NY, E);
  static constexpr int TW_BYTES = ((TWS * CS) + 127) & ~127;
  static constexpr int K2_BYTES = ((NY * (int)sizeof(T)) + 127) & ~127;
  static constexpr int HEAD = (128 + TW_BYTES + K2_BYTES + 255) & ~255;
  static constexpr size_t SMEM = HEAD + (size_t)NR * SLOT * CS;
  // The 32-byte swizzle goes by the address bits 4 and 7, undone from the row
  // in the tile (col2_body): every region on 256 bytes of a base on 256 bytes.
  static_assert(!SWZ || (HEAD % 256 == 0 && SLOT * CS % 256 == 0 && BH * TK * CS % 256 == 0), "swizzled regions");
  // CTAs per SM the registers are budgeted for: FP32 128 per thread at 32
  // values, FP64 at least 64
  static constexpr int MIN_BLOCKS =
      F64 ? (G <= 2 ? 8 / G : (G == 4 ? 3 : 1)) : (E >= 32 ? 512 / THREADS : (G == 1 ? 512 : 768) / THREADS);
};

// The packed kx = 0 / Nyquist column of the first CTA: y holds this warp's
// forward transform Z = A + i B (A the kx = 0 column, B the kx = nx/2 one,
// both Hermitian in ky), fz the same packing of df/dc^ (c only).  A and B are
// separated through Z(ky) and conj Z(ny - ky), updated with their own K2
// (Eqs. A-C_discrete_fft_c / _eta) and repacked, in place.  The update maps
// each pair {ky, ny - ky} onto itself (A(ny - ky) = conj A(ky), the same for
// B, and the update is real-linear with the same K2 at ky and ny - ky), so a
// thread owns both entries of its pairs and no other thread touches them.  A
// few warps of the grid run this, so it stays out of line and rolled.
template <typename T, int NY, int TPL>
__device__ __noinline__ void col2_packed_update(cplx<T>* __restrict__ y, const cplx<T>* __restrict__ fz, int t,
                                                bool isC, KUpdate<T> up, T kx2, T kxn2,
                                                const T* __restrict__ k2yt, const double* csum,
                                                double inv_npts) {
  using C = cplx<T>;
#pragma unroll 1
  for (int m = 0; m <= NY / (2 * TPL); ++m) {
    const int ky = t + TPL * m;  // pairs ky = 0 .. ny/2
    if (ky > NY / 2) break;
    const int kq = (NY - ky) & (NY - 1);
    const T ky2 = k2yt[ky];
    const C z = y[ky], pz = cconj(y[kq]);
    const C A = cscale(cadd(z, pz), T(0.5)), B = cscale(mul_i<-1>(csub(z, pz)), T(0.5));
    C An, Bn;
    if (isC) {
      const C zf = fz[ky], pf = cconj(fz[kq]);
      const C Af = cscale(cadd(zf, pf), T(0.5)), Bf = cscale(mul_i<-1>(csub(zf, pf)), T(0.5));
      An = up.c(A, Af, kx2 + ky2);
      Bn = up.c(B, Bf, kxn2 + ky2);
      if (ky == 0 && csum) An = mk<C>((T)(*csum * inv_npts), T(0));
    } else {
      An = up.eta(A, kx2 + ky2);
      Bn = up.eta(B, kxn2 + ky2);
    }
    y[ky] = cadd(An, mul_i<1>(Bn));
    if (kq != ky) y[kq] = cadd(cconj(An), mul_i<1>(cconj(Bn)));
  }
}

// Field groups: group 0 holds df/dc and c, group g >= 1 the NE eta_i from
// eta_{NE (g - 1) + 1}; line (region r, column j).  FP64 CTA: one column of
// {df/dc, c} or of one eta_i, the smallest unit there is: the pass is bound by
// the FP64 pipe, so its time is the busiest SM's share of the transforms
// (256^2, p = 4: 9.3 transforms per SM on average; 16 on the busiest with
// pairs of columns and eta_i, 11 with these).  The tiles come in by TMA, every
// line copies its column to registers, then its region becomes TK compact
// per-column areas (exchange buffers, line_pad layout).  After the update and
// the inverse transform the results go back to the interleaved tile layout
// and out by TMA, so the global writes are whole tile rows instead of one
// 8-byte value per lane and row.
// Column block `cblk` (TK columns), field group `group` of the simulation `a`
// (blockDim = THREADS); `bar` as for row2_body.  Returns false if a bounded
// wait gave up.  EARLY: see griddep_launch_dependents.
template <typename T, int NY, int G, int TK, int NR, bool EARLY = false>
__device__ __forceinline__ bool col2_body(const KArgs& a, const CUtensorMap* tmap, int cblk, int group,
                                          unsigned char* smem_raw, uint64_t* bar, uint32_t parity) {
  using C = cplx<T>;
  using Cfg = Col2Cfg<T, NY, G, TK, NR>;
  constexpr int E = Cfg::E, BH = Cfg::BH, PL = Cfg::PL, SLOT = Cfg::SLOT, TPL = Cfg::TPL;
  C* tw = reinterpret_cast<C*>(smem_raw + 128);
  T* k2yt = reinterpret_cast<T*>(smem_raw + 128 + Cfg::TW_BYTES);
  C* regions = reinterpret_cast<C*>(smem_raw + Cfg::HEAD);
  const int nf = a.nf, p = nf - 1;
  const int line = (threadIdx.x >> 5) / G, t = threadIdx.x % TPL;  // line (region, column), thread in it
  constexpr int NE = Cfg::NE;
  const int j = line % TK, r = line / TK;
  const int nreg = group == 0 ? 2 : (p - NE * (group - 1) >= NE ? NE : 1);
  // slot of region q of this group: group 0: df/dc (nf), c (0); else eta_{NE (g - 1) + 1 + q}
  auto slot_of = [nf, group](int q) { return group == 0 ? (q == 0 ? nf : 0) : NE * (group - 1) + 1 + q; };
  const bool isF = (group == 0 && r == 0), isC = (group == 0 && r == 1);
  const int kx0 = cblk * TK, kx = kx0 + j;
  const int H = a.nx / 2;

  if (r >= nreg) return true;  // the second region of a last group with one eta
  if (threadIdx.x == 0) {
    // the fused step reuses the regions: order the previous item's
    // generic accesses (ended by the caller's CTA barrier) before the TMA writes
    fence_proxy_async_smem();
    const uint32_t tbytes = (uint32_t)(Cfg::TWS * sizeof(C)), kbytes = (uint32_t)(NY * sizeof(T));
    mbar_arrive_expect_tx(bar, tbytes + kbytes + (uint32_t)(nreg * NY * TK * sizeof(C)));
    // the constant tables first, overlapping the previous grid's tail
    bulk_g2s(tw, G == 1 || Cfg::F64 ? a.tw_col2 : a.tw_col2w, tbytes, bar);
    bulk_g2s(k2yt, a.k2y, kbytes, bar);
    griddep_wait();  // the tiles are the previous pass's output
    for (int q = 0; q < nreg; ++q)
      // innermost coordinate kx0 in 8-byte units is even: 16-byte aligned
      for (int y0 = 0; y0 < NY; y0 += BH)
        tma_load_3d(regions + q * SLOT + y0 * TK, tmap, kx0 * (Cfg::CS / 8), y0, slot_of(q), bar);
  }
  const T* __restrict__ k2xt = reinterpret_cast<const T*>(a.k2x);
  const T kx2 = k2xt[kx];
  // all threads: the bounded wait starts when the copies do, however long the
  // previous pass takes, and no lane of warp 0 polls before lane 0 has issued
  griddep_wait();
  __syncwarp();
  if (EARLY) griddep_launch_dependents();
  if (!mbar_wait_bounded(bar, parity, first_wait_polls(a))) {
    if (threadIdx.x == 0) atomicOr(a.flag, FS_FLAG_TIMEOUT);
    mbar_wait_bounded(bar, parity, kWaitPolls);
    return false;
  }

  // this thread's first tile element; the others are TPL rows (a multiple of
  // the swizzle's period) apart
  C* reg = regions + r * SLOT;
  C* mine = reg + t * TK + (Cfg::SWZ ? j ^ (((t >> 2) & 1) << 1) : j);
  C v[E];
#pragma unroll
  for (int m = 0; m < E; ++m) v[m] = mine[TPL * m * TK];
  // named barriers: 1, 2 per region (its TK column lines), from 3 per column
  // (df/dc^ handed to the c line), from 3 + TK per line (its G warps)
  auto region_sync = [r]() { if (r == 0) bar_sync(1, 32 * TK * G); else bar_sync(2, 32 * TK * G); };
  const LineSync<G, 3 + TK, Cfg::F64> lsync{line};
  // both columns of this region have left the tile: it becomes two compact areas
  region_sync();
  C* xa = reg + j * PL;
  auto st = [xa](int q, C x) { xa[line_pad<T, NY>(q)] = x; };
  auto ld = [xa](int q) { return xa[line_pad<T, NY>(q)]; };
  const KUpdate<T> up(a);
  const bool special = (a.kx_base + kx0 == 0 && j == 0);  // the packed kx = 0 / Nyquist column
  const C* fz = regions + j * PL;             // df/dc^ of this column (region 0 of group 0)

  // One FFT call site: it 0 forward (all warps), it 1 inverse (c, eta) as
  // conj(FFT(conj(.))).
  for (int it = 0; it < 2; ++it) {
    line_fft<NY, E, -1>(v, t, tw, st, ld, lsync);
    if (it == 1) break;
    if (isF) {
      // df/dc^: natural layout for the c warp of this column
      lsync();
#pragma unroll
      for (int m = 0; m < E; ++m) xa[t + TPL * m] = v[m];
      if (j == 0) bar_arrive(3, 64 * G); else if (j == 1) bar_arrive(4, 64 * G); else if (j == 2) bar_arrive(5, 64 * G); else bar_arrive(6, 64 * G);
      return true;
    }
    if (isC) {
      if (j == 0) bar_sync(3, 64 * G); else if (j == 1) bar_sync(4, 64 * G); else if (j == 2) bar_sync(5, 64 * G); else bar_sync(6, 64 * G);
    }
    if (special) {
      lsync();
#pragma unroll
      for (int m = 0; m < E; ++m) xa[t + TPL * m] = v[m];
      lsync();
      col2_packed_update<T, NY, TPL>(xa, fz, t, isC, up, kx2, k2xt[H], k2yt, a.csum, a.inv_npts);
      lsync();
#pragma unroll
      for (int m = 0; m < E; ++m) v[m] = cconj(xa[t + TPL * m]);
    } else if constexpr (Cfg::F64) {
      // bound by the FP64 pipe: c and eta each with their own operations only
      if (isC) {
#pragma unroll
        for (int m = 0; m < E; ++m) {
          const int ky = t + TPL * m;
          v[m] = cconj(up.c(v[m], fz[ky], kx2 + k2yt[ky]));
        }
      } else {
#pragma unroll
        for (int m = 0; m < E; ++m) v[m] = cconj(up.eta(v[m], kx2 + k2yt[t + TPL * m]));
      }
    } else {
      // c^' = (c^ - M dt K2 f^) / (1 + M dt kappa_c K2^2), eta^' = g^ / (1 + L dt kappa_eta K2)
      // (scales folded as in KUpdate); one code path for both, the quotient by
      // the fast reciprocal (the denominators are >= 1)
      const float num = isC ? up.scale_c : up.scale;
      const float qk = isC ? up.Mdtkc : up.Ldtke;
      const float bk = isC ? up.Mdt_c : 0.f;
#pragma unroll
      for (int m = 0; m < E; ++m) {
        const int ky = t + TPL * m;
        const float k2 = kx2 + k2yt[ky];
        const float d = __fdividef(num, fmaf(qk, isC ? k2 * k2 : k2, 1.f));
        const C zf = isC ? fz[ky] : make_float2(0.f, 0.f);
        v[m] = cconj(cscale(vfma(zf, vsplat<C>(-bk * k2), v[m]), d));
      }
    }
  }
  // results (conj of the last transform) back to the interleaved tile layout
  // of this region, then out by TMA: c -> slot 0, eta_i -> slot i
  if (!EARLY) griddep_launch_dependents();
  region_sync();  // both columns are done with their compact areas
#pragma unroll
  for (int m = 0; m < E; ++m) mine[TPL * m * TK] = cconj(v[m]);
  fence_proxy_async_smem();
  region_sync();
  if (j == 0 && t == 0) {  // one thread of the region's column-0 line
    for (int y0 = 0; y0 < NY; y0 += BH) tma_store_3d(tmap, kx0 * (Cfg::CS / 8), y0, slot_of(r), reg + y0 * TK);
    bulk_commit();
    // the tile is read before the region is reused or the CTA exits; its
    // writes are performed before the grid completes (waiting for them here
    // kept the CTA's registers and shared memory a microsecond longer)
    bulk_wait_read();
  }
  return true;
}

// Uniform CTAs: grid (column blocks, field groups).
template <typename T, int NY, int G, int TK, int NR>
__global__ void __launch_bounds__(Col2Cfg<T, NY, G, TK, NR>::THREADS, Col2Cfg<T, NY, G, TK, NR>::MIN_BLOCKS)
    fs_col2_kernel(KArgs a, const __grid_constant__ CUtensorMap tmap) {
  extern __shared__ __align__(256) unsigned char col_smem[];  // Col2Cfg: regions on 256 bytes
  uint64_t* bar = reinterpret_cast<uint64_t*>(col_smem);
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  col2_body<T, NY, G, TK, NR>(a, &tmap, blockIdx.x, blockIdx.y, col_smem, bar, 0);
}

// Mixed CTAs of four lines each (FP32): {df/dc, c} of two columns first, then
// each eta_i of four columns.
template <int NY, int G>
__global__ void __launch_bounds__(128 * G, Col2Cfg<float, NY, G, 2, 2>::MIN_BLOCKS)
    fs_col2m_kernel(KArgs a, const __grid_constant__ CUtensorMap tmap2, const __grid_constant__ CUtensorMap tmap4) {
  extern __shared__ __align__(256) unsigned char col_smem[];  // Col2Cfg: regions on 256 bytes
  uint64_t* bar = reinterpret_cast<uint64_t*>(col_smem);
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  const int n2 = a.nx / 4, n4 = a.nx / 8, b = (int)blockIdx.x - n2;
  if (b < 0) col2_body<float, NY, G, 2, 2>(a, &tmap2, blockIdx.x, 0, col_smem, bar, 0);
  else col2_body<float, NY, G, 4, 1>(a, &tmap4, b % n4, 1 + b / n4, col_smem, bar, 0);
}

// Launchers: cudaErrorNotSupported when this form does not cover the
// request (the caller falls back to the half-length / tile kernels).
template <typename T, int NX, int G, int NW>
cudaError_t row2_launch_nw(const KArgs& a, cudaStream_t s) {
  static unsigned done = 0;
  cudaError_t e = allow_big_smem(fs_row2_kernel<T, NX, G, NW>, &done);
  if (e != cudaSuccess) return e;
  const int lines = a.nf < NW ? a.nf : NW;  // lines in flight; more fields take a second round
  return launch_pdl(fs_row2_kernel<T, NX, G, NW>, dim3((unsigned)(a.lines / 2)), dim3((unsigned)(32 * G * lines)),
                    row2_smem_bytes<T, NX, G>(a.nf, a.mode), s, a);
}

template <typename T, int NY, int G, int TK, int NR>
cudaError_t col2_launch_n(const KArgs& a, const CUtensorMap& tm, cudaStream_t s) {
  static unsigned done = 0;
  cudaError_t e = allow_big_smem(fs_col2_kernel<T, NY, G, TK, NR>, &done);
  if (e != cudaSuccess) return e;
  using Cfg = Col2Cfg<T, NY, G, TK, NR>;
  const unsigned groups = (unsigned)(1 + (a.nf - 1 + Cfg::NE - 1) / Cfg::NE);  // {df/dc, c}; NE eta_i each
  return launch_pdl(fs_col2_kernel<T, NY, G, TK, NR>, dim3((unsigned)(a.nx / 2 / TK), groups),
                    dim3((unsigned)Cfg::THREADS), Cfg::SMEM, s, a, tm);
}

template <int NY, int G>
cudaError_t col2m_launch_n(const KArgs& a, const CUtensorMap& tm2, const CUtensorMap& tm4, cudaStream_t s) {
  static unsigned done = 0;
  cudaError_t e = allow_big_smem(fs_col2m_kernel<NY, G>, &done);
  if (e != cudaSuccess) return e;
  using C2 = Col2Cfg<float, NY, G, 2, 2>;
  using C4 = Col2Cfg<float, NY, G, 4, 1>;
  const size_t smem = C2::SMEM > C4::SMEM ? C2::SMEM : C4::SMEM;
  return launch_pdl(fs_col2m_kernel<NY, G>, dim3((unsigned)(a.nx / 4 + (a.nf - 1) * (a.nx / 8))), dim3(128u * G), smem,
                    s, a, tm2, tm4);
}

}  // namespace fs
