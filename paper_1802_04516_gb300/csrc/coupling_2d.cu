// 2D FP64 instances of the operator from assembled couplings (coupling_apply.h).
#include "coupling_apply.h"

namespace stdg {

template <typename R>
cudaError_t coupling_2d(stdg_ctx* c, const R* Ke, const R* Kf, const R* rhoJ, const R* x, const int* xidx, int64_t ld,
                        const R* base, const int* bidx, int64_t bld, R* y, double scale, int ns) {
    switch (c->Nphi) {
        case 3: return coupling_shape<R, 2, 3>(c, Ke, Kf, rhoJ, x, xidx, ld, base, bidx, bld, y, scale, ns);
        case 6: return coupling_shape<R, 2, 6>(c, Ke, Kf, rhoJ, x, xidx, ld, base, bidx, bld, y, scale, ns);
        case 10: return coupling_shape<R, 2, 10>(c, Ke, Kf, rhoJ, x, xidx, ld, base, bidx, bld, y, scale, ns);
        case 15: return coupling_shape<R, 2, 15>(c, Ke, Kf, rhoJ, x, xidx, ld, base, bidx, bld, y, scale, ns);
        default: return cudaErrorInvalidValue;
    }
}

template cudaError_t coupling_2d<double>(stdg_ctx*, const double*, const double*, const double*, const double*, const int*, int64_t, const double*,
                                      const int*, int64_t, double*, double, int);

}  // namespace stdg
