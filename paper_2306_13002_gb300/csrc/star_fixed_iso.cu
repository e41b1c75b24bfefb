// The fixed-point star stencil with the same weights on every axis, the choice between the two weight
// forms, and the integer weights.
#include "star_fixed_launch.cuh"

namespace acs {

// Integer weights (see StarFix). The march needs weights of alternating sign (the centre's against
// the nearest ones', as second-derivative weights of every order have them; zeros may stand
// anywhere), sums that fit 64 bits, and a centre weight that carries a fair share of the sum (the
// point's own value is then a measure of its rounding errors), with the nearest x and y weights
// not lost against it. Spacing ratios up to about 8 pass; other weights keep the FP64 march.
void star_fix(const StarCoef& c, StarFix& fx) {
    std::memset(&fx, 0, sizeof(fx));
    bool iso = true;
    double sum = 0.0;
    const double sg = c.c0 < 0.0 ? 1.0 : -1.0;
    for (int q = 0; q < 12; ++q) {
        iso = iso && c.c[q] == c.c[q % 4];
        sum += 2.0 * std::fabs(c.c[q]);
        if (sg * c.c[q] * (q % 2 ? -1.0 : 1.0) < 0.0) return;
    }
    const double mid = std::fabs(c.c0);
    if (!(mid >= 0x1p-100 && mid <= 0x1p100) || mid < 0.25 * sum || std::fabs(c.c[0]) < mid / 64 ||
        std::fabs(c.c[4]) < mid / 64)
        return;
    const int LB = iso ? kStarIsoLB : kStarGenLB;
    int w = LB + 31 - std::ilogb(mid) + 2;
    while (std::ldexp(mid, w) >= std::ldexp(0.999, LB + 31) || std::ldexp(mid + sum, w) >= std::ldexp(0.999, LB + 32)) --w;
    // W = wh 2^LB + wl; the weights the march takes as negative (even distances and the centre) get a
    // negative wh even where they are 0.
    auto put = [&](int at, long long W) {
        const long long hi = at % 2 ? W >> LB : (W - 1) >> LB;
        fx.wh[at] = (unsigned)hi;
        fx.wl[at] = (unsigned)(W - (hi << LB));
    };
    long long total = 0;
    for (int q = 0; q < (iso ? 4 : 12); ++q) {
        const long long W = std::llrint(std::ldexp(sg * c.c[q], w));
        put(1 + q, W);
        total += W;
    }
    put(0, (iso ? -6 : -2) * total);
    fx.shift = LB + 29 - w;
    fx.neg = sg < 0.0;
    // The bound's reasoning takes a point's sum of |terms| for at least a nearest weight times the bound; Taylor
    // weights with the same spacing on every axis have 0.187 of the centre's there. Up to a power of
    // two (but for a tenth), 2^4 at most by the tests above (2^57, an eighth of the scale).
    double least = std::fmin(std::fabs(c.c[0]), std::fabs(c.c[4]));
    fx.zmask = std::fabs(c.c[8]) >= 0.5 * least ? ~0u : 0u;
    if (fx.zmask) least = std::fmin(least, std::fabs(c.c[8]));
    fx.small = kStarSmallHi << (least < 0.187 * mid ? std::ilogb(1.8 * 0.187 * mid / least) : 0);
    fx.kind = iso ? 1 : 2;
}

acs_status launch_star_fixed(const double* u, const double* a, double* out, const Geom& g, const StarCoef& c,
                             const StarFix& fx, const acs_tile& t, cudaStream_t s) {
    return fx.kind == 1 ? launch_star_fixed_kind<true>(u, a, out, g, c, fx, t, s)
                        : launch_star_fixed_gen(u, a, out, g, c, fx, t, s);
}

}  // namespace acs
