// 3D FP64 instances of the operator from assembled couplings (coupling_apply.h).
#include "coupling_apply.h"

namespace stdg {

template <typename R>
cudaError_t coupling_3d(stdg_ctx* c, const R* Ke, const R* Kf, const R* rhoJ, const R* x, const int* xidx, int64_t ld,
                        const R* base, const int* bidx, int64_t bld, R* y, double scale, int ns) {
    switch (c->Nphi) {
        case 4: return coupling_shape<R, 3, 4>(c, Ke, Kf, rhoJ, x, xidx, ld, base, bidx, bld, y, scale, ns);
        case 10: return coupling_shape<R, 3, 10>(c, Ke, Kf, rhoJ, x, xidx, ld, base, bidx, bld, y, scale, ns);
        case 20: return coupling_shape<R, 3, 20>(c, Ke, Kf, rhoJ, x, xidx, ld, base, bidx, bld, y, scale, ns);
        default: return cudaErrorInvalidValue;
    }
}

template cudaError_t coupling_3d<double>(stdg_ctx*, const double*, const double*, const double*, const double*, const int*, int64_t, const double*,
                                      const int*, int64_t, double*, double, int);

}  // namespace stdg
