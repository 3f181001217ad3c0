// FP64 instantiations of the pair-form row pass and the warp-per-line column
// pass.
#include "fs_k2d_v2.cuh"

namespace fs {

// Warps per line.  An SM sub-core issues one FP64 warp instruction about every
// 64 cycles, so what matters is that every sub-core of the chip has a warp,
// and that a warp's own chain is short: few values per thread (2 at 64 points,
// 4 at 128 and 256, 8 above), which costs the fused butterflies almost no
// instructions (3 per value and radix-2 stage whatever the radix).
#define FS_ROW64_SIZES(X) X(64, 1) X(128, 1) X(256, 4) X(512, 4) X(1024, 4) X(2048, 8)
#define FS_COL64_SIZES(X) X(64, 1) X(128, 1) X(256, 2) X(512, 2) X(1024, 4) X(2048, 8)

int row2_g64(int nx) {
  switch (nx) {
#define FS_CASE(n, g) \
  case n: return g;
    FS_ROW64_SIZES(FS_CASE)
#undef FS_CASE
    default: return 0;
  }
}
int col2_g64(int ny) {
  switch (ny) {
#define FS_CASE(n, g) \
  case n: return g;
    FS_COL64_SIZES(FS_CASE)
#undef FS_CASE
    default: return 0;
  }
}

// Lines in flight per CTA: one per field, at most three where a line takes
// 256 threads (five would not fit a CTA) and for nf <= 3 at 128, whose CTAs
// then fit twice on an SM.
template <int NX, int G>
static cudaError_t row2_launch_n(const KArgs& a, cudaStream_t s) {
  if constexpr (G == 8) return row2_launch_nw<double, NX, G, 3>(a, s);
  else if constexpr (G == 4) {
    if (a.nf <= 3) return row2_launch_nw<double, NX, G, 3>(a, s);
  }
  if constexpr (G < 8) return row2_launch_nw<double, NX, G, 5>(a, s);
}

cudaError_t row2_launch_f64(const KArgs& a, cudaStream_t s) {
  if (a.mode > 2 || !a.tw_row2 || a.nf < 1 || a.nf > 5 || a.lines % 2) return cudaErrorNotSupported;
  switch (a.nx) {
#define FS_CASE(n, g) \
  case n: return row2_launch_n<n, g>(a, s);
    FS_ROW64_SIZES(FS_CASE)
#undef FS_CASE
    default: return cudaErrorNotSupported;
  }
}
cudaError_t col2_launch_f64(const KArgs& a, const CUtensorMap& tm, cudaStream_t s) {
  if (a.nz != 1 || !a.tw_col2 || a.nf < 1 || a.nf > 5 || a.nx < 4) return cudaErrorNotSupported;
  switch (a.ny) {
#define FS_CASE(n, g) \
  case n: return col2_launch_n<double, n, g, 1, 2>(a, tm, s);
    FS_COL64_SIZES(FS_CASE)
#undef FS_CASE
    default: return cudaErrorNotSupported;
  }
}

}  // namespace fs
