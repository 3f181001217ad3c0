// FP32 instantiations of the 3D x pass with several row pairs per CTA.
#include "fs_k2d_v2.cuh"

namespace fs {

bool row3_supported(int nx) { return nx == 64 || nx == 128 || nx == 256 || nx == 512; }

// Two warps per field, or one where that would leave fewer than four CTAs
// per SM (152 SMs).
template <int NX>
static cudaError_t row3_launch_n(const KArgs& a, cudaStream_t s) {
  const bool wide = a.lines % (2 * Row3Cfg<NX, 2>::PR) == 0 && a.lines / (2 * Row3Cfg<NX, 2>::PR) >= 608;
  if (!wide && a.lines % (2 * Row3Cfg<NX, 1>::PR)) return cudaErrorNotSupported;
  if (a.nf <= 3) return wide ? row3_launch_nw<NX, 2, 3>(a, s) : row3_launch_nw<NX, 1, 3>(a, s);
  return wide ? row3_launch_nw<NX, 2, 5>(a, s) : row3_launch_nw<NX, 1, 5>(a, s);
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
