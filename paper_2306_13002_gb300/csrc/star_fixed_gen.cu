// The fixed-point star stencil with weights of its own on every axis.
#include "star_fixed_launch.cuh"

namespace acs {

acs_status launch_star_fixed_gen(const double* u, const double* a, double* out, const Geom& g, const StarCoef& c,
                                 const StarFix& fx, const acs_tile& t, cudaStream_t s) {
    return launch_star_fixed_kind<false>(u, a, out, g, c, fx, t, s);
}

}  // namespace acs
