// FP32 instances of the block-Jacobi apply with one thread per (element, row).
#include "pre1_rows.h"

namespace stdg {

cudaError_t launch_pre1_rows32(stdg_ctx* c, const float* r, float* z, const int* ridx, int64_t ld, int nshots) {
    return pre1_rows<float>(c, c->d_preV32, c->d_preB32, r, ridx, ld, z, nshots);
}

}  // namespace stdg
