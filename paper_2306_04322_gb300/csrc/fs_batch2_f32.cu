// Ensemble (batched) launches of the warp-per-line forms, FP32: one CTA per
// item of the work list of all members -- row pairs for the row pass, (column
// pair, field group) for the column pass -- members ordered largest first,
// each item running the body instantiated for its member's size.  The plan's
// autotuner times these against the half-length / tile ensemble kernels and
// keeps the faster form per pass.
#include "fs_batch_impl.cuh"
#include "fs_k2d_v2.cuh"

namespace fs {

#define FS_V2_SIZES(X) X(64) X(128) X(256) X(512) X(1024)

__global__ void __launch_bounds__(Row2Cfg<float, 1024>::MAX_THREADS, 4)
    fs_row2_batch_kernel(const KArgs* __restrict__ mem, const long long* __restrict__ begin, int nm) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem_raw);
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  const long long item = blockIdx.x;
  const int m = find_member(begin, nm, item);
  const KArgs& a = mem[m];
  const long long rp = item - begin[m];
  switch (a.nx) {
#define FS_CASE(n) \
  case n: row2_body<float, n, 1, -1, true>(a, rp, smem_raw, bar, 0); break;
    FS_V2_SIZES(FS_CASE)
#undef FS_CASE
    default: break;
  }
}

__global__ void __launch_bounds__(128, 5)
    fs_col2_batch_kernel(const KArgs* __restrict__ mem, const CUtensorMap* __restrict__ maps,
                         const long long* __restrict__ begin, const int* __restrict__ pairs, int nm) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem_raw);
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  const long long item = blockIdx.x;
  const int m = find_member(begin, nm, item);
  const KArgs& a = mem[m];
  const int np = pairs[m];
  const int rem = (int)(item - begin[m]);
  const int group = rem / np, cp = rem % np;
  switch (a.ny) {
#define FS_CASE(n) \
  case n: col2_body<float, n, 1, 2, 2, true>(a, &maps[m], cp, group, smem_raw, bar, 0); break;
    FS_V2_SIZES(FS_CASE)
#undef FS_CASE
    default: break;
  }
}

size_t row2_smem_f32(int nx, int nf, int mode) {
  switch (nx) {
#define FS_CASE(n) \
  case n: return row2_smem_bytes<float, n>(nf, mode);
    FS_V2_SIZES(FS_CASE)
#undef FS_CASE
    default: return 0;
  }
}
size_t col2_smem_f32(int ny) {
  switch (ny) {
#define FS_CASE(n) \
  case n: return Col2Cfg<float, n, 1, 2, 2>::SMEM;
    FS_V2_SIZES(FS_CASE)
#undef FS_CASE
    default: return 0;
  }
}
int col2_groups(int nf) { return 1 + (nf - 1 + 1) / 2; }

cudaError_t row2_batch_launch_f32(const BatchArgs& b, cudaStream_t s) {
  static unsigned done = 0;
  cudaError_t e = allow_big_smem(fs_row2_batch_kernel, &done);
  if (e != cudaSuccess) return e;
  return launch_pdl(fs_row2_batch_kernel, dim3((unsigned)b.row2_total), dim3((unsigned)(32 * (b.nf1 - 1))),
                    b.row2_mode == 1 ? b.row2_smem1 : b.row2_smem, s, b.mem, b.row2_begin, b.nm);
}

cudaError_t col2_batch_launch_f32(const BatchArgs& b, cudaStream_t s) {
  static unsigned done = 0;
  cudaError_t e = allow_big_smem(fs_col2_batch_kernel, &done);
  if (e != cudaSuccess) return e;
  return launch_pdl(fs_col2_batch_kernel, dim3((unsigned)b.col2_total), dim3(128), b.col2_smem, s, b.mem_col, b.maps2,
                    b.col2_begin, b.col2_pairs, b.nm);
}

}  // namespace fs
