// FP32 instantiations of the warp-per-line row (pair form) and column passes:
// lines of 64 to 1024 points held by one warp (G = 1, tables tw_row2 /
// tw_col2) or, from 128 points, by two warps (G = 2, tables tw_row2w /
// tw_col2w; columns up to 2048 points).
#include "fs_k2d_v2.cuh"

namespace fs {
static bool v2_size(int n) { return n == 64 || n == 128 || n == 256 || n == 512 || n == 1024; }
bool row2_supported(int nx, int nf) { return v2_size(nx) && nf >= 1 && nf <= 5; }
bool col2_supported(int ny, int nf) { return (v2_size(ny) || ny == 2048) && nf >= 1 && nf <= 5; }

template <int NX, int G>
static cudaError_t row2_launch_n(const KArgs& a, cudaStream_t s) {
  if (G == 1 && a.nf == 3) return row2_launch_nw<float, NX, G, 3>(a, s);
  return row2_launch_nw<float, NX, G, 5>(a, s);
}
template <int G>
cudaError_t row2_launch_g(const KArgs& a, cudaStream_t s) {
  switch (a.nx) {
    case 64: if constexpr (G == 1) return row2_launch_n<64, G>(a, s); else return cudaErrorNotSupported;
    case 128: return row2_launch_n<128, G>(a, s);
    case 256: return row2_launch_n<256, G>(a, s);
    case 512: return row2_launch_n<512, G>(a, s);
    case 1024: return row2_launch_n<1024, G>(a, s);
    default: return cudaErrorNotSupported;
  }
}
// Column CTAs.  One warp per line: mixed CTAs of four lines (two columns of
// {df/dc, c}, four of an eta_i), which load and store a third fewer tile rows
// than pairs of columns throughout; from 1024 points and 1024-point rows on,
// where the tiles are many, four columns of {df/dc, c} or two eta_i in CTAs of
// eight lines (half the tile rows) -- but with p = 1, whose eta CTAs would
// have idle lines.  Per step, pairs / mixed / wide: 1024^2 p = 2 24.6 / 24.0 /
// 22.9 us, p = 4 36.2 / 35.1 / 33.6, p = 1 20.0 / 19.0 / 21.4; 256^2 p = 4 8.1 /
// 7.3 / 7.7; 512^2 p = 2 10.5 / 10.2 / 11.4.  Two warps per line keep pairs
// (2048^2 p = 4 133 / 136 / 156: a wide CTA has an SM to itself).
template <int NY, int G>
static cudaError_t col2_launch_tk(const KArgs& a, const CUtensorMap& tm2, const CUtensorMap& tm4, cudaStream_t s) {
  if constexpr (G == 1) {
    if constexpr (NY >= 1024) {
      if (a.nx >= 1024 && a.nf != 2) return col2_launch_n<float, NY, G, 4, 2>(a, tm4, s);
    }
    if (a.nx >= 16) return col2m_launch_n<NY, G>(a, tm2, tm4, s);  // whole blocks of four columns, two of them
  }
  return col2_launch_n<float, NY, G, 2, 2>(a, tm2, s);
}
template <int G>
cudaError_t col2_launch_g(const KArgs& a, const CUtensorMap& tm, const CUtensorMap& tm4, cudaStream_t s) {
  switch (a.ny) {
    case 64: if constexpr (G == 1) return col2_launch_tk<64, G>(a, tm, tm4, s); else return cudaErrorNotSupported;
    case 128: return col2_launch_tk<128, G>(a, tm, tm4, s);
    case 256: return col2_launch_tk<256, G>(a, tm, tm4, s);
    case 512: return col2_launch_tk<512, G>(a, tm, tm4, s);
    case 1024: return col2_launch_tk<1024, G>(a, tm, tm4, s);
    case 2048: if constexpr (G == 2) return col2_launch_tk<2048, G>(a, tm, tm4, s); else return cudaErrorNotSupported;
    default: return cudaErrorNotSupported;
  }
}

cudaError_t row2_launch_f32(const KArgs& a, cudaStream_t s) {
  if (a.mode > 2 || !row2_supported(a.nx, a.nf) || a.lines % 2) return cudaErrorNotSupported;
  if (a.tw_row2w) return row2_launch_g<2>(a, s);
  if (a.tw_row2) return row2_launch_g<1>(a, s);
  return cudaErrorNotSupported;
}
cudaError_t col2_launch_f32(const KArgs& a, const CUtensorMap& tm, const CUtensorMap& tm4, cudaStream_t s) {
  if (a.tc != 0 || a.nz != 1 || !col2_supported(a.ny, a.nf) || a.nx < 4) return cudaErrorNotSupported;
  if (a.tw_col2w) return col2_launch_g<2>(a, tm, tm4, s);
  if (a.tw_col2) return col2_launch_g<1>(a, tm, tm4, s);
  return cudaErrorNotSupported;
}
}  // namespace fs
