// The fixed-point RHS with a spacing of its own on every axis.
#include "rhs_fixed_launch.cuh"

namespace acs {

acs_status launch_rhs_fixed_gen(const double* U, double* R, const Geom& g, const RhsConst& kf, const RhsConst& kc,
                                const RhsFix& fx, const acs_tile& t, cudaStream_t s) {
    return launch_rhs_fixed_form<false>(U, R, g, kf, kc, fx, t, s);
}

}  // namespace acs
