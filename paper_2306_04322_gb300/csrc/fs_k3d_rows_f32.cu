// FP32 instantiations of the x pass with several row pairs per CTA.
#include "fs_k2d_v2.cuh"

namespace fs {

bool row3_supported(int nx) { return nx == 64 || nx == 128 || nx == 256 || nx == 512; }

template <int NX>
static cudaError_t row3_launch_n(const KArgs& a, cudaStream_t s) {
  if (a.lines % (2 * Row3Cfg<NX>::PR)) return cudaErrorNotSupported;
  return a.nf <= 3 ? row3_launch_nw<NX, 3>(a, s) : row3_launch_nw<NX, 5>(a, s);
}

cudaError_t row3_launch_f32(const KArgs& a, cudaStream_t s) {
  if ((a.mode != 0 && a.mode != 2) || !a.tw_row3 || a.nf < 1 || a.nf > 5) return cudaErrorNotSupported;
  switch (a.nx) {
    case 64: return row3_launch_n<64>(a, s);
    case 128: return row3_launch_n<128>(a, s);
    case 256: return row3_launch_n<256>(a, s);
    case 512: return row3_launch_n<512>(a, s);
    default: return cudaErrorNotSupported;
  }
}

}  // namespace fs
