// kernels_smw32.cu -- FP32 instances of the structured block-Jacobi apply (smw_sapply.cuh),
// in a file of their own so that the two precisions compile side by side.
#include "smw_sapply.cuh"

namespace sts {

sts_status smw_sapply32(sts_jac_s *h, int dir, const Vec<float> &x, const Vec<float> &z) {
    return smw_sapply_t<float>(h, dir, h->smw.ap32[dir], x, z);
}

}  // namespace sts
