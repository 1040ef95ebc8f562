// The register-resident QR, with column pivoting, in FP64.
#include "qr.cuh"

namespace ifmm {

bool qr_launch_f64_piv(int cls, const QrcpDesc* d, int nd, int R, int warps, size_t smem, cudaStream_t s, bool probe) {
  return qr_launch_c<double, true>(cls, d, nd, R, warps, smem, s, probe);
}
void qr_launch_warp_f64_piv(bool tall, const QrcpDesc* d, int nd, cudaStream_t s) { qr_launch_w<double, true>(tall, d, nd, s); }

}  // namespace ifmm
