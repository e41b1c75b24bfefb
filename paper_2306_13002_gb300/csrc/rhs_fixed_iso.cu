// The fixed-point RHS with equal spacing, the choice between the two spacing forms, and the constants.
#include "rhs_fixed_launch.cuh"

namespace acs {

// |c| = (h 2^31 + l) 2^(ex - 62), rounded to 62 bits (exact: a double has 53).
static void split62(double c, int& h, int& l, int& ex) {
    ex = std::ilogb(c) + 1;
    const long long n = std::llrint(std::ldexp(c, 62 - ex));
    h = (int)(n >> 31);
    l = (int)(n & 0x7fffffffll);
}

// The march takes positive spacings and dissipation (every term of R then has the sign it flips at
// the end), of magnitudes that leave its exponents room; other parameters keep the FP64 march.
void rhs_fix(const RhsConst& k, RhsFix& fx, RhsConst& kc) {
    std::memset(&fx, 0, sizeof(fx));
    kc = k;
    const double s[3] = {-k.sx, -k.sy, -k.sz};
    if (!(k.eps >= 0x1p-60 && k.eps <= 0x1p90) || !(std::fabs(k.g1) <= 0x1p20)) return;
    for (int d = 0; d < 3; ++d)
        if (!(s[d] >= 0x1p-90 && s[d] <= 0x1p90)) return;
    kc.sx = s[0];
    kc.sy = s[1];
    kc.sz = s[2];
    kc.nhg1s = k.nhg1 / s[0];
    split62(k.eps, fx.eh, fx.el, fx.ex_eps);
    for (int d = 0; d < 3; ++d) split62(s[d], fx.sh[d], fx.sl[d], fx.ex_s[d]);
    fx.g1 = (float)k.g1;
    fx.smax = (float)std::fmax(s[0], std::fmax(s[1], s[2])) * 1.001f;
    fx.smin = (float)std::fmin(s[0], std::fmin(s[1], s[2]));
    fx.eps = (float)k.eps;
    fx.ok = 1;
}

acs_status launch_rhs_fixed(const double* U, double* R, const Geom& g, const RhsConst& kf, const RhsConst& kc,
                            const RhsFix& fx, const acs_tile& t, cudaStream_t s) {
    return rhs_isotropic(kc) ? launch_rhs_fixed_form<true>(U, R, g, kf, kc, fx, t, s)
                             : launch_rhs_fixed_gen(U, R, g, kf, kc, fx, t, s);
}

}  // namespace acs
