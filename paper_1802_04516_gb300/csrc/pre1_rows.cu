// FP64 instances of the block-Jacobi apply with one thread per (element, row).
#include "pre1_rows.h"

namespace stdg {

cudaError_t launch_pre1_rows(stdg_ctx* c, const double* r, double* z, const int* ridx, int64_t ld, int nshots) {
    return pre1_rows<double>(c, c->d_preV, c->d_preB, r, ridx, ld, z, nshots);
}

}  // namespace stdg
