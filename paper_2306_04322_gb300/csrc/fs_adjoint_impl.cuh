// Launch sequence of the adjoint of one 2D step (three kernels).
#pragma once

#include "fs_adjoint.cuh"
#include "fs_adjoint3.cuh"
#include "fs_k2d_impl.cuh"

namespace fs {

template <typename T, int NX, int P>
cudaError_t adj_row_p(const KArgs& a, bool inverse, cudaStream_t s) {
  using RC = AdjRowCfg<T, NX>;
  const long long reff = a.lines < RC::R ? a.lines : RC::R;
  const size_t smem = RC::smem(a.nf);
  static unsigned d1 = 0, d2 = 0;
  cudaError_t e;
  const dim3 grid((unsigned)(a.lines / reff));
  if (!inverse) {
    e = allow_big_smem(fs_adj_row_fwd_kernel<T, NX, P>, &d1);
    if (e != cudaSuccess) return e;
    return launch_pdl(fs_adj_row_fwd_kernel<T, NX, P>, grid, dim3(96 * (P + 1)), smem, s, a);
  }
  e = allow_big_smem(fs_adj_row_inv_kernel<T, NX, P>, &d2);
  if (e != cudaSuccess) return e;
  return launch_pdl(fs_adj_row_inv_kernel<T, NX, P>, grid, dim3(64 * (P + 1)), smem, s, a);
}

template <typename T, int NX>
cudaError_t adj_row_n(const KArgs& a, bool inverse, cudaStream_t s) {
  switch (a.nf) {
    case 1: return adj_row_p<T, NX, 0>(a, inverse, s);
    case 2: return adj_row_p<T, NX, 1>(a, inverse, s);
    case 3: return adj_row_p<T, NX, 2>(a, inverse, s);
    case 4: return adj_row_p<T, NX, 3>(a, inverse, s);
    case 5: return adj_row_p<T, NX, 4>(a, inverse, s);
    default: return cudaErrorInvalidValue;
  }
}

template <typename T, int NY, int TKC>
cudaError_t adj_col_tk(const KArgs& a, const CUtensorMap& tm, int tk, cudaStream_t s) {
  static unsigned d = 0;
  cudaError_t e = allow_big_smem(fs_adj_col_kernel<T, NY, TKC>, &d);
  if (e != cudaSuccess) return e;
  const unsigned threads = ((unsigned)(tk * ColCfg<T, NY>::TPL) + 31) / 32 * 32;
  return launch_pdl(fs_adj_col_kernel<T, NY, TKC>, dim3((unsigned)(a.nx / 2 / tk), (unsigned)a.nf), dim3(threads),
                    AdjColCfg<T, NY>::smem(tk), s, a, tm);
}

template <typename T, int NY>
int adj_tk(int nx) {
  return AdjColCfg<T, NY>::TK < nx / 2 ? AdjColCfg<T, NY>::TK : nx / 2;
}

template <typename T, int NY>
cudaError_t adj_col_n(const KArgs& a, const CUtensorMap& tm, cudaStream_t s) {
  const int tk = adj_tk<T, NY>(a.nx);
  if (tk == AdjColCfg<T, NY>::TK) return adj_col_tk<T, NY, AdjColCfg<T, NY>::TK>(a, tm, tk, s);
  return adj_col_tk<T, NY, 0>(a, tm, tk, s);
}

#define FS_ADJ_SIZES(X) X(8) X(16) X(32) X(64) X(128) X(256) X(512) X(1024)

template <typename T>
int adj_tile_width_t(int nx, int ny) {
  switch (ny) {
#define FS_CASE(n) \
  case n: return adj_tk<T, n>(nx);
    FS_ADJ_SIZES(FS_CASE)
#undef FS_CASE
    default: return 0;
  }
}

template <typename T>
cudaError_t adjoint_launch_t(const KArgs& a0, const CUtensorMap& tm, void* lam_out, cudaStream_t s) {
  cudaError_t e = cudaErrorInvalidValue;
  switch (a0.nx) {
#define FS_CASE(n) \
  case n: e = adj_row_n<T, n>(a0, false, s); break;
    FS_ADJ_SIZES(FS_CASE)
#undef FS_CASE
    default: break;
  }
  if (e != cudaSuccess) return e;
  e = cudaErrorInvalidValue;
  switch (a0.ny) {
#define FS_CASE(n) \
  case n: e = adj_col_n<T, n>(a0, tm, s); break;
    FS_ADJ_SIZES(FS_CASE)
#undef FS_CASE
    default: break;
  }
  if (e != cudaSuccess) return e;
  KArgs a1 = a0;
  a1.real = lam_out;
  e = cudaErrorInvalidValue;
  switch (a0.nx) {
#define FS_CASE(n) \
  case n: e = adj_row_n<T, n>(a1, true, s); break;
    FS_ADJ_SIZES(FS_CASE)
#undef FS_CASE
    default: break;
  }
  return e;
}

template <typename T, int NZ>
cudaError_t adj_z_n(const KArgs& a, const CUtensorMap& tm, cudaStream_t s) {
  using Cfg = AdjLineCfg<T, NZ>;
  const int tk = line_tk<T, NZ>(a.nx);
  const size_t smem = Cfg::HEAD + (size_t)3 * Cfg::TROWS * tk * sizeof(cplx<T>);
  static unsigned d = 0;
  cudaError_t e = allow_big_smem(fs_adj_z_kernel<T, NZ>, &d);
  if (e != cudaSuccess) return e;
  dim3 grid((unsigned)(a.nx / 2 / tk), (unsigned)a.ny, (unsigned)a.nf);
  fs_adj_z_kernel<T, NZ><<<grid, (unsigned)(tk * Cfg::TPL), smem, s>>>(a, tm);
  return cudaGetLastError();
}

// y pass over the adjoint's slots: the steps' in FP64; in FP32 the same kernel
// with the adjoint's transform.
template <typename T>
cudaError_t adj_ypass_t(const KArgs& a, const CUtensorMap& tm, int dir, int nslots, cudaStream_t s) {
  if constexpr (sizeof(T) == 8) {
    return ypass_launch_f64(a, tm, dir, a.nz, nslots, s);
  } else {
    switch (a.ny) {
#define FS_CASE(n)                                                                                                  \
  case n:                                                                                                           \
    return dir < 0 ? ypass_launch_tk<T, n, -1, TC_NONE, 0, true>(a, tm, a.nz, nslots, line_tk<T, n>(a.nx), s)       \
                   : ypass_launch_tk<T, n, 1, TC_NONE, 0, true>(a, tm, a.nz, nslots, line_tk<T, n>(a.nx), s);
      FS_LINE_SIZES(FS_CASE)
#undef FS_CASE
      default: return cudaErrorInvalidValue;
    }
  }
}

// Adjoint of one 3D step (five launches): x forward of lam', u, f(u) (the
// 2D adjoint's row kernel over ny nz rows), y forward of the 3 nf slots (the
// step's y pass), the z part (fs_adj_z_kernel), y inverse of the 2 nf result
// slots, x inverse with the pointwise Hessian product.  tm_y: [slot nz + z][y]
// [kx] over the adjoint slots; tm_z: [slot][z][y][kx].
template <typename T>
cudaError_t adjoint3_launch_t(const KArgs& a0, const CUtensorMap& tm_y, const CUtensorMap& tm_z, void* lam_out,
                              cudaStream_t s) {
  cudaError_t e = cudaErrorInvalidValue;
  switch (a0.nx) {
#define FS_CASE(n) \
  case n: e = adj_row_n<T, n>(a0, false, s); break;
    FS_ADJ_SIZES(FS_CASE)
#undef FS_CASE
    default: break;
  }
  if (e != cudaSuccess) return e;
  KArgs b = a0;
  b.carry3 = 0;  // plain y transforms of every slot (no carried c)
  b.plane0 = 0;
  b.tc = 0;
  e = adj_ypass_t<T>(b, tm_y, -1, 3 * a0.nf, s);
  if (e != cudaSuccess) return e;
  e = cudaErrorInvalidValue;
  switch (a0.nz) {
#define FS_CASE(n) \
  case n: e = adj_z_n<T, n>(b, tm_z, s); break;
    FS_LINE_SIZES(FS_CASE)
#undef FS_CASE
    default: break;
  }
  if (e != cudaSuccess) return e;
  e = adj_ypass_t<T>(b, tm_y, 1, 2 * a0.nf, s);
  if (e != cudaSuccess) return e;
  KArgs a1 = a0;
  a1.real = lam_out;
  e = cudaErrorInvalidValue;
  switch (a0.nx) {
#define FS_CASE(n) \
  case n: e = adj_row_n<T, n>(a1, true, s); break;
    FS_ADJ_SIZES(FS_CASE)
#undef FS_CASE
    default: break;
  }
  return e;
}

}  // namespace fs
