// Explicit finite-difference comparison scheme of Boccardo et al. (arXiv
// 2306.04322, Section 2.2): forward Euler in time, second-order centred
// 5-point (2D) / 7-point (3D) Laplacian on a periodic grid, three stages per
// step
//   (i)   mu    = df/dc - kappa_c lap(c)
//   (ii)  c'    = c + dt M lap(mu)
//   (iii) eta'_i = eta_i - dt L (df/deta_i - kappa_eta lap(eta_i))
// In 2D fused into one kernel: a CTA loads a tile with a two-point halo
// (periodic wrap instead of the paper's ghost layers), forms mu on the tile
// plus a one-point halo in shared memory, then updates its interior.  In 3D
// two kernels: mu and the eta_i, then c.
//
// Both use the constants of fill_pointwise and fill_fd (multiplied out): about
// 21 operations per eta and point in 2D where the stages term by term take 30,
// which is the time of the FP64 kernels (512 x 256, p = 4: 35.3 us per step
// against 48.8); every thread takes adjacent points along x, so
// that loads, index arithmetic and the FP32 arithmetic (packed two-lane
// instructions) serve two points or more (3D 128^3, p = 4, FP32: 24.8 us per
// step against 70; one thread per point and 64-bit neighbour indices had made
// it 530 instructions per point).
#include "fs_k2d_impl.cuh"

namespace fs {

namespace {

// The inputs are written by the kernel before, which may still run when one
// of these starts (programmatic dependent launch): they are read through
// plain pointers (no __restrict__ const, no __ldg), so that no load becomes a
// non-coherent one or moves above griddep_wait().

// Neighbour sums along x of the pair (v.x, v.y) at x, x + 1 with left
// neighbour l (at x - 1) and right neighbour r (at x + 2).
template <typename C, typename T>
__device__ __forceinline__ C xsum(T l, C v, T r) {
  return mk<C>(l + v.y, v.x + r);
}

// -dt L df/deta_i of a pair (S2 = sum_j eta_j^2; see Pointwise::g2), NF fields.
template <int NF, typename C, typename T>
__device__ __forceinline__ C eta_rate(const Coef<T>& k, C chem, C e, C S2) {
  const C ne = mk<C>(-e.x, -e.y);
  const C q = vfma(e, ne, e);
  const C in = vfma(chem, q, vfma(e, vsplat<C>(T(-2) * k.g_dw), vsplat<C>(k.g_dw)));
  if (NF == 2) return vmul(q, in);  // one eta: the sum over the others is empty
  return vfma(q, in, vmul(vmul(e, vsplat<C>(k.g_pair)), vfma(e, ne, S2)));
}

// 2D tile: TX x TY points, one pair of x neighbours per thread.  FP32 64 x 8;
// FP64, bound by its pipe and so by the busiest SM's share of the points,
// 32 x 8.
template <typename T>
struct FdTile {
  static constexpr int TX = sizeof(T) == 4 ? 64 : 32, TY = 8;
  static constexpr int THREADS = TX / 2 * TY;
  static constexpr int W = TX + 4, H = TY + 4;   // loaded tile (halo 2)
  static constexpr int MH = TY + 2;              // rows of mu (halo 1); columns as the tile (its first and
                                                 // last are not used)
  // one unused pair before the tile: the mu stage reads (not uses) x - 1 of its first column
  static constexpr size_t bytes(int nf) { return sizeof(T) * (2 + (size_t)nf * W * H + (size_t)W * MH + 2); }
};

template <typename T, int NF>
__global__ void __launch_bounds__(FdTile<T>::THREADS) fs_fd_kernel(KArgs a, const T* in, T* __restrict__ out) {
  using C = cplx<T>;
  using Cfg = FdTile<T>;
  constexpr int TX = Cfg::TX, TY = Cfg::TY, W = Cfg::W, H = Cfg::H, MH = Cfg::MH, HW = W / 2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* tile = reinterpret_cast<T*>(smem_raw) + 2;  // [NF][H][W]
  T* mu = tile + NF * H * W;                     // [MH][W]
  const int nx = a.nx, ny = a.ny;
  const long long N = a.npts;
  const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
  const int tid = threadIdx.x;
  griddep_wait();  // `in` is the previous step's output, `out` its input
  for (int i = tid; i < HW * H; i += Cfg::THREADS) {
    const int lp = i % HW, ly = i / HW;
    const int gx = (x0 + 2 * lp - 2) & (nx - 1), gy = (y0 + ly - 2) & (ny - 1);  // periodic (powers of two)
    const T* src = in + (gy * nx + gx);
    C v[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) v[f] = *reinterpret_cast<const C*>(src + f * N);
#pragma unroll
    for (int f = 0; f < NF; ++f) *reinterpret_cast<C*>(&tile[(f * H + ly) * W + 2 * lp]) = v[f];
  }
  griddep_launch_dependents();
  __syncthreads();
  const Coef<T>& k = coef<T>(a);
  const Pointwise<T> pw(a);
  auto at = [tile](int f, int ly, int lx) { return &tile[(f * H + ly) * W + lx]; };
  auto pairp = [](const T* p) { return *reinterpret_cast<const C*>(p); };
  const C m2 = vsplat<C>(T(-2));
  // (i) mu on the tile plus a one-point halo
  for (int i = tid; i < HW * MH; i += Cfg::THREADS) {
    const int lx = 2 * (i % HW), my = i / HW;
    const T* c = at(0, my + 1, lx);
    const C v = pairp(c);
    C h = vsplat<C>(T(0));
#pragma unroll
    for (int f = 1; f < NF; ++f) h = pw.add_h2(pairp(at(f, my + 1, lx)), h);
    C m = vfma(vfma(v, m2, xsum(c[-1], v, c[2])), vsplat<C>(k.mu_d[0]), pw.fc2(v, h));
    m = vfma(vfma(v, m2, cadd(pairp(c - W), pairp(c + W))), vsplat<C>(k.mu_d[1]), m);
    *reinterpret_cast<C*>(&mu[my * W + lx]) = m;
  }
  __syncthreads();
  // (ii), (iii) interior update
  const int px = tid % (TX / 2), ty = tid / (TX / 2);
  const int gx = x0 + 2 * px, gy = y0 + ty;
  if (gx >= nx || gy >= ny) return;
  const int lx = 2 * px + 2, ly = ty + 2;
  const long long o = (long long)gy * nx + gx;
  const long long out_bytes = (long long)NF * N * (long long)sizeof(T);
  auto store = [&](int f, C v) {
    if (in_bounds(a, &out[f * N + o], sizeof(C), out, out_bytes)) *reinterpret_cast<C*>(&out[f * N + o]) = v;
  };
  const T* m = &mu[(ty + 1) * W + lx];
  const C mv = pairp(m), c = pairp(at(0, ly, lx));
  C d = vmul(vfma(mv, m2, xsum(m[-1], mv, m[2])), vsplat<C>(k.dc_d[0]));
  d = vfma(vfma(mv, m2, cadd(pairp(m - W), pairp(m + W))), vsplat<C>(k.dc_d[1]), d);
  const C cn = cadd(c, d);
  FiniteCheck<T> chk;
  chk.add(cn);
  store(0, cn);
  C S2 = vsplat<C>(T(0));
  const C chem = vfma(c, vsplat<C>(k.g_c), vsplat<C>(k.g_0));
#pragma unroll
  for (int f = 1; f < NF; ++f) {
    const C e = pairp(at(f, ly, lx));
    S2 = vfma(e, e, S2);
  }
#pragma unroll
  for (int f = 1; f < NF; ++f) {
    const T* ep = at(f, ly, lx);
    const C e = pairp(ep);
    C r = eta_rate<NF>(k, chem, e, S2);
    r = vfma(vfma(e, m2, xsum(ep[-1], e, ep[2])), vsplat<C>(k.de_d[0]), r);
    r = vfma(vfma(e, m2, cadd(pairp(ep - W), pairp(ep + W))), vsplat<C>(k.de_d[1]), r);
    const C en = cadd(e, r);
    chk.add(en);
    store(f, en);
  }
  if (chk.bad()) atomicOr(a.flag, FS_FLAG_NONFINITE);
}

// 3D: the same three stages with the 7-point Laplacian, as two kernels, one
// 16-byte vector of points along x per thread (neighbours through the
// caches).  Kernel 1 forms mu (stage i) into a scratch field and writes the
// updated eta_i (stage iii); kernel 2 applies stage ii to c.  Axes are powers
// of two of at least 8 points, so the periodic neighbours are masks and a
// vector never wraps.
template <typename T>
struct Vec3 {
  using C = cplx<T>;
  static constexpr int V = 16 / sizeof(T), NC = V / 2;  // points and pairs per vector
  int c, ym, yp, zm, zp, xm, xp;                        // element offsets of the vector and its neighbours
  __device__ __forceinline__ Vec3(const KArgs& a, int i) {
    const int nx = a.nx, ny = a.ny, nz = a.nz, lx = __ffs(nx) - 1, lxy = lx + __ffs(ny) - 1;
    c = i * V;
    const int x = c & (nx - 1), y = (c >> lx) & (ny - 1), z = c >> lxy;
    const int row = c - x, col = x + (y << lx);
    xm = row + ((x - 1) & (nx - 1));
    xp = row + ((x + V) & (nx - 1));
    ym = c + ((((y - 1) & (ny - 1)) - y) << lx);
    yp = c + ((((y + 1) & (ny - 1)) - y) << lx);
    zm = col + (((z - 1) & (nz - 1)) << lxy);
    zp = col + (((z + 1) & (nz - 1)) << lxy);
  }
  __device__ __forceinline__ static void load(const T* p, C (&v)[NC]) {
    const int4 w = *reinterpret_cast<const int4*>(p);
    memcpy(v, &w, 16);
  }
  __device__ __forceinline__ static void store(T* p, const C (&v)[NC]) {
    int4 w;
    memcpy(&w, v, 16);
    *reinterpret_cast<int4*>(p) = w;
  }
  // acc + sum_d w_d (sum of the two neighbours along d less twice the value) of
  // field f, whose values at the vector are v
  __device__ __forceinline__ void neighbours(const T* f, const C (&v)[NC], const T (&w)[3],
                                             C (&acc)[NC]) const {
    C a0[NC], a1[NC], b0[NC], b1[NC];
    load(f + ym, a0);
    load(f + yp, a1);
    load(f + zm, b0);
    load(f + zp, b1);
    const T l = f[xm], r = f[xp];
#pragma unroll
    for (int q = 0; q < NC; ++q) {
      C s[3] = {xsum(q == 0 ? l : v[q - 1].y, v[q], q == NC - 1 ? r : v[q + 1].x), cadd(a0[q], a1[q]),
                cadd(b0[q], b1[q])};
#pragma unroll
      for (int d = 0; d < 3; ++d) acc[q] = vfma(vfma(v[q], vsplat<C>(T(-2)), s[d]), vsplat<C>(w[d]), acc[q]);
    }
  }
};

template <typename T, int NF>
__global__ void __launch_bounds__(256) fs_fd3_mu_eta_kernel(KArgs a, const T* in, T* __restrict__ out,
                                                            T* __restrict__ mu) {
  using V3 = Vec3<T>;
  using C = cplx<T>;
  constexpr int NC = V3::NC;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  griddep_wait();  // `in` is the previous step's output
  griddep_launch_dependents();
  if (i >= a.npts / V3::V) return;
  const V3 g(a, i);
  const long long N = a.npts;
  const Pointwise<T> pw(a);
  const Coef<T>& k = coef<T>(a);
  C c[NC], e[NF][NC], S2[NC], m[NC], chem[NC];
#pragma unroll
  for (int f = 0; f < NF; ++f) V3::load(in + f * N + g.c, e[f]);
#pragma unroll
  for (int q = 0; q < NC; ++q) {
    c[q] = e[0][q];
    C h = vsplat<C>(T(0));
    S2[q] = vsplat<C>(T(0));
#pragma unroll
    for (int f = 1; f < NF; ++f) {
      h = pw.add_h2(e[f][q], h);
      S2[q] = vfma(e[f][q], e[f][q], S2[q]);
    }
    m[q] = pw.fc2(c[q], h);
    chem[q] = vfma(c[q], vsplat<C>(k.g_c), vsplat<C>(k.g_0));
  }
  g.neighbours(in, c, k.mu_d, m);
  V3::store(mu + g.c, m);
  FiniteCheck<T> chk;
#pragma unroll
  for (int f = 1; f < NF; ++f) {
    C r[NC];
#pragma unroll
    for (int q = 0; q < NC; ++q) r[q] = eta_rate<NF>(k, chem[q], e[f][q], S2[q]);
    g.neighbours(in + f * N, e[f], k.de_d, r);
#pragma unroll
    for (int q = 0; q < NC; ++q) {
      r[q] = cadd(e[f][q], r[q]);
      chk.add(r[q]);
    }
    V3::store(out + f * N + g.c, r);
  }
  if (chk.bad()) atomicOr(a.flag, FS_FLAG_NONFINITE);
}

template <typename T>
__global__ void __launch_bounds__(256) fs_fd3_c_kernel(KArgs a, const T* in, T* __restrict__ out,
                                                       const T* mu) {
  using V3 = Vec3<T>;
  using C = cplx<T>;
  constexpr int NC = V3::NC;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  griddep_wait();  // mu is the previous kernel's output
  griddep_launch_dependents();
  if (i >= a.npts / V3::V) return;
  const V3 g(a, i);
  const Coef<T>& k = coef<T>(a);
  C c[NC], m[NC], d[NC];
  V3::load(in + g.c, c);
  V3::load(mu + g.c, m);
#pragma unroll
  for (int q = 0; q < NC; ++q) d[q] = vsplat<C>(T(0));
  g.neighbours(mu, m, k.dc_d, d);
  FiniteCheck<T> chk;
#pragma unroll
  for (int q = 0; q < NC; ++q) {
    d[q] = cadd(c[q], d[q]);
    chk.add(d[q]);
  }
  V3::store(out + g.c, d);
  if (chk.bad()) atomicOr(a.flag, FS_FLAG_NONFINITE);
}

template <typename T, int NF>
cudaError_t fd_launch_nf(const KArgs& a, const T* in, T* out, T* scratch, cudaStream_t s) {
  if (a.nz > 1) {
    const unsigned blocks = (unsigned)((a.npts / Vec3<T>::V + 255) / 256);
    cudaError_t e = launch_pdl(fs_fd3_mu_eta_kernel<T, NF>, dim3(blocks), dim3(256), 0, s, a, in, out, scratch);
    if (e != cudaSuccess) return e;
    return launch_pdl(fs_fd3_c_kernel<T>, dim3(blocks), dim3(256), 0, s, a, in, out, (const T*)scratch);
  }
  using Cfg = FdTile<T>;
  const dim3 grid((unsigned)((a.nx + Cfg::TX - 1) / Cfg::TX), (unsigned)((a.ny + Cfg::TY - 1) / Cfg::TY));
  return launch_pdl(fs_fd_kernel<T, NF>, grid, dim3((unsigned)Cfg::THREADS), Cfg::bytes(NF), s, a, in, out);
}

template <typename T>
cudaError_t fd_launch_t(const KArgs& a, const void* in, void* out, void* scratch, cudaStream_t s) {
  const T* i = reinterpret_cast<const T*>(in);
  T *o = reinterpret_cast<T*>(out), *m = reinterpret_cast<T*>(scratch);
  switch (a.nf) {
    case 1: return fd_launch_nf<T, 1>(a, i, o, m, s);
    case 2: return fd_launch_nf<T, 2>(a, i, o, m, s);
    case 3: return fd_launch_nf<T, 3>(a, i, o, m, s);
    case 4: return fd_launch_nf<T, 4>(a, i, o, m, s);
    case 5: return fd_launch_nf<T, 5>(a, i, o, m, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

int fd_launches_per_step(const KArgs& a) { return a.nz > 1 ? 2 : 1; }

cudaError_t fd_launch(bool f64, const KArgs& a, const void* in, void* out, void* scratch, cudaStream_t s) {
  return f64 ? fd_launch_t<double>(a, in, out, scratch, s) : fd_launch_t<float>(a, in, out, scratch, s);
}

}  // namespace fs
