// March of the saturated RHS in block-scaled fixed point (fixed.cuh): the fluxes of a point are computed
// in FP64 as before (point_flux), everything that adds neighbours runs on the integer pipes.
//
//   R_c = -( sum of the flux differences + eps (S2 - 4 S1 + 18 U_c) )
//
// Of the 114 FP64 operations of a point (equal spacing) 23 remain; the 91 that difference fluxes and
// form the dissipation are sums of at most 13 terms with small whole weights, exact in 64-bit
// integers. The scale of the fluxes (|s| = 1/(2h)) is folded in where they are formed, for unequal
// spacing as well (30 operations).
//
// Scales: one exponent each for rho, the momenta and E, from the first planes of a segment, with
// the ranges of rho and E below them (they enter the bounds of the fluxes, and a point's own values
// must not lose their low bits); the fluxes' scales follow from these bounds. A plane that leaves
// the ranges ends the segment. The rule compares the bounds with the dissipation and the pressure (see
// segment), so it takes spacings near 1 (0.1 to 1 for the uniform and smooth states of perf/cases.py with a
// dissipation of 0.25, down to 0.03 with a spacing of 1) and refuses much finer or more uneven ones.
//
// Measured on GB300: 256^3 3237 us in FP64 (114 operations per point, 94 % of the FP64 pipe) -> 1113 us
// (element-wise staging 3403 -> 1252), three spacings 3293 -> 1410, 162^3 with three spacings 999 -> 444, 512^3
// of a smooth flow 25.7 -> 8.4 ms, 128^3 420 -> 168. Values that are refused: 256^3 3254 -> 3260, 128^3 420 -> 424,
// 64^3 70.3 -> 74.1 (the scan, 4 us per block). Error against 64 bits (2-norm): uniform state 2.2e-16 -> 4.9e-17,
// smooth flow 2.4e-15 -> 5.7e-16; no larger than FP64's in any octave of the points' own magnitudes, up to
// the ends of the ranges (momenta from 2^-30 to 2^-3, rho and E over 2^6). What bounds it now: a warp's own
// chains. About 1200 instructions per point (29 of them FP64, ring included: 70 % of that pipe's time) issue
// at 46 % of the peak rate, 16 warps per SM being what two rings of six planes and 128 registers leave room
// for; the stalls are FP64 and shared-memory results (2.1 cycles per instruction), fixed latencies (1.7)
// and the two barriers per plane (1.2).
#pragma once

#include "fixed.cuh"
#include "march.cuh"

namespace acs {

// 2^n; 0 below the normal floats, infinity above.
__device__ __forceinline__ float pow2f(int n) { return __int_as_float(min(max(n + 127, 0), 255) << 23); }

// t * 2^e2 rounded to FP64 (half away from zero) with its sign flipped, on the integer pipes. No
// branches here or in the flux: the five components' chains interleave.
__device__ __forceinline__ double minus_from_fixed(i64 t, int e2) {
    const u32 sg = (u32)((int)hi32((u64)t) >> 31);
    const u64 m = ((u64)t ^ pack64(sg, sg)) + (sg & 1u);
    const bool low = hi32(m) == 0;
    const u32 mh = low ? lo32(m) : hi32(m), ml = low ? 0u : lo32(m);
    // exponent field of a value with bit 63 (low: 31) set, less the hidden bit
    const int top = (low ? 1023 + 31 - 1 : 1023 + 63 - 1) + e2;
    const int lz = __clz((int)mh);
    const u32 nh = __funnelshift_l(ml, mh, lz), nl = ml << (lz & 31);
    const u64 r = pack64((nh >> 11) + ((u32)(top - lz) << 20), __funnelshift_r(nl, nh, 11)) + ((nl >> 10) & 1u);
    return mh == 0 ? 0.0 : __hiloint2double((int)(hi32(r) | (~sg & 0x80000000u)), (int)lo32(r));
}

// floor-like d * w / 2^63 for w = wh 2^31 + wl, both parts below 2^31 (error below two units).
__device__ __forceinline__ i64 mul63(i64 d, int wh, int wl) {
    const int dh = (int)hi32((u64)d);
    const u32 dl = lo32((u64)d);
    return (i64)dh * wh + (((i64)dh * wl) >> 31) + (i64)(((u64)dl * (u32)wh) >> 32);
}

// Fluxes of a point scaled by |s_d| per axis (unequal spacing), otherwise as point_flux.
__device__ __forceinline__ void point_flux_scaled(double rho, double mx, double my, double mz, double E,
                                                  const RhsConst& k, double fx[4], double fy[4], double fz[4]) {
    const Pipe& q = k.pp;
    const double r = rcp_inside(rho, q.one);
    const double vx = pmul(mx, r, q), vy = pmul(my, r, q), vz = pmul(mz, r, q);
    const double twoKE = fma(mz, vz, fma(my, vy, pmul(mx, vx, q)));
    const double P = fma(k.nhg1, twoKE, pmul(k.g1, E, q)), EP = padd(E, P, q);
    const double ax = pmul(vx, k.sx, q), ay = pmul(vy, k.sy, q), az = pmul(vz, k.sz, q);
    fx[0] = fma(mx, ax, pmul(P, k.sx, q));
    fx[1] = pmul(my, ax, q);
    fx[2] = pmul(mz, ax, q);
    fx[3] = pmul(EP, ax, q);
    fy[0] = pmul(mx, ay, q);
    fy[1] = fma(my, ay, pmul(P, k.sy, q));
    fy[2] = pmul(mz, ay, q);
    fy[3] = pmul(EP, ay, q);
    fz[0] = pmul(mx, az, q);
    fz[1] = pmul(my, az, q);
    fz[2] = fma(mz, az, pmul(P, k.sz, q));
    fz[3] = pmul(EP, az, q);
}

// Six ring slots of U (raw as they land, fixed point once their fluxes are formed), the x and y
// fluxes of one plane, constants, mbarriers and the scan's results.
template <int BX, int BY>
struct RhsFixShape {
    static constexpr int PX = BX + 4, PY = BY + 4, PLANE = PX * PY, CELLS = 5 * PLANE;
    static constexpr int NT = BX * BY, NSLOT = 6;
    static constexpr int NR = 2 * (BX + BY), NC = NT - NR;   // threads of the flux ring, and of the cells
    static constexpr int NE = (CELLS + NC - 1) / NC;
    static constexpr int FX_ELEMS = 4 * BY * (BX + 2), FY_ELEMS = 4 * (BY + 2) * BX;
    static constexpr int CONST_ELEMS = RhsShape<BX, BY>::CONST_ELEMS;
    // ... constants of the launch, mbarriers, the scan's results, constants of the segment
    static constexpr size_t BYTES = sizeof(u64) * ((size_t)NSLOT * CELLS + FX_ELEMS + FY_ELEMS + CONST_ELEMS + NSLOT + 4 + 10 + 3);
    static constexpr int MINB = NT <= 128 ? 4 : 2;
    static_assert((CELLS * sizeof(u64)) % 128 == 0, "every ring slot 128-byte aligned");
    static_assert(NT >= 2 * (BX + BY) && (2 * BX) % 32 == 0, "flux ring needs 2(BX+BY) threads, y-ring whole warps");
    static_assert(sizeof(RhsConst) <= CONST_ELEMS * sizeof(double), "constant staging area");
};

// A segment's constants, in shared memory: the march has few registers to spare.
struct RhsScale {
    int join[3][4];               // rho, momenta, E: RhsJoin
    int cu[3], lo[3];             // conversion exponents of U, least exponents (none for the momenta)
    int cf[2];                    // conversion exponents of the momentum and energy fluxes
    int seen[6];                  // exponent ranges of the planes marched so far (as the scan's; one spare)
};
static_assert(sizeof(RhsScale) == 104, "RhsFixShape reserves thirteen words");

// Shifts and exponent that join a component's flux sum a and dissipation d: z = (a >> sa) + (d >> sd),
// in units of 2^e.
struct RhsJoin {
    int sa, sd, e;
};
__device__ __forceinline__ RhsJoin rhs_join(int ea, int ed) {
    const int e = max(ea, ed) + 1;
    return RhsJoin{min(e - ea, 63), min(e - ed, 63), e};
}

// Whether the dissipation of a point's momenta has room for certain, from the upper halves of its values in
// three planes (addresses of rho's): 4.5 of the point's own and a quarter of the six at distance 2 are
// at most 12 2^59, so it takes six nearest values of the other sign that sum to 4 2^59 to exceed 2^63. A
// call of its own: inlined in the march, it took 30 us of 256^3 without being run.
template <int PX, int PLANE>
__device__ __noinline__ bool rhs_roomy(u32 below, u32 here, u32 above) {
    bool all = true;
#pragma unroll
    for (int c = 1; c < 4; ++c) {
        auto hi = [&](u32 a) { return lds_int(a + c * PLANE * 8 + 4); };
        const int h1 = (hi(here - 8) + hi(here + 8) + hi(here - 8 * PX)) + (hi(here + 8 * PX) + hi(below) + hi(above));
        all &= (hi(here) ^ h1) >= 0 || abs(h1) < (4 << 27) - 8;   // (8: their lower halves)
    }
    return all;
}

template <int BX, int BY, bool TMA, bool ISO>
struct RhsFixMarch {
    using S = RhsFixShape<BX, BY>;
    static constexpr int PX = S::PX, PLANE = S::PLANE, NE = S::NE, NC = S::NC, NSLOT = S::NSLOT;

    const double* __restrict__ U;
    double* __restrict__ R;
    const Geom& g;
    const RhsConst& kc;   // with |s_d| in place of s_d
    const RhsFix& fx;
    int i0, j0, k1;
    double* smem;
    const CUtensorMap* map;
    unsigned* tmo;

    __device__ __forceinline__ uint64_t* bar(int slot) const {
        return reinterpret_cast<uint64_t*>(smem + NSLOT * S::CELLS + S::FX_ELEMS + S::FY_ELEMS + S::CONST_ELEMS) + slot;
    }

    __device__ __forceinline__ RhsScale* scales() const { return reinterpret_cast<RhsScale*>(bar(NSLOT) + 4); }

    // Marches from plane k0; returns the first plane not finished, or k0 - 1 if the scanned planes do not
    // fit: the ring then holds planes k0-2 .. k0+3 (none past k1+1) as they are. `phase`, `flying`, `ok`: as
    // StarFixMarch::segment.
    __device__ __forceinline__ int segment(int k0, int tid, u32& phase, u32& flying, bool& ok) const {
        const u32 rs = smem_addr(smem), fxs = rs + NSLOT * S::CELLS * 8, fys = fxs + S::FX_ELEMS * 8;
        // [0] max rho, [1] min rho, [2] max m, [3] max E, [4] min E
        int* note = reinterpret_cast<int*>(bar(NSLOT));
        // Tiles cut by the grid's edges: points packed as in rhs_march, one halo column more than the
        // valid ones; rows up to the one past the last valid row.
        const int w = min(BX, g.nx - i0), h = min(BY, g.ny - j0);
        const int wf = w < BX ? w + 1 : BX;
        const int tx = w < BX ? tid % wf : tid % BX, ty = w < BX ? tid / wf : tid / BX;
        const bool fluxer = ty < BY && ty <= h && (tx < w || ty < h);   // not the corner past both edges
        const bool active = fluxer && tx < w && ty < h;
        constexpr u32 safe = (2 * PX + 2) * 8;   // the tile's first point
        const u32 own = ((ty + 2) * PX + tx + 2) * 8, mine = fluxer ? own : safe;

        // The first NR threads compute the ring's fluxes; the others stage and convert the cells.
        const int cell = tid - S::NR;
        u32 full = 0, core = 0;   // one bit per cell: read by some point on the segment's planes, and on others
        // (Away from the rim all cells are values of the flow: both stagings bring and convert the corners, too.)
        const bool rim = i0 == 0 || j0 == 0 || i0 + BX + 2 > g.nx || j0 + BY + 2 > g.ny;
        auto masks = [&]() {
            int xx = cell % PX, yy = cell / PX;
#pragma unroll 1
            for (int n = 0, e = cell; e >= 0 && e < S::CELLS; ++n, e += NC) {
                const bool xin = xx >= 2 && xx < w + 2, yin = yy >= 2 && yy < h + 2;
                if (xx < w + 4 && yy < h + 4 && (xin || yin)) full |= 1u << n;
                if (xin && yin) core |= 1u << n;
                xx += NC % PX;
                yy += NC / PX;
                if (xx >= PX) xx -= PX, ++yy;
                if (yy >= S::PY) yy -= S::PY;
            }
            if (!rim) full = ~0u;
        };
        if (!TMA) masks();
        auto keep = [&](int q) { return q >= k0 && q < k1 ? full : core; };
        auto slot_of = [&](int q) { return (q - k0 + 2) % NSLOT; };
        auto stage = [&](int q) {
            const int slot = slot_of(q);
            if (TMA) {
                flying |= 1u << slot;
                if (tid == 0) {
                    fence_proxy_async();
                    mbar_arrive_expect_tx(bar(slot), S::CELLS * 8);
                    tma_load_4d(smem + slot * S::CELLS, map, bar(slot), i0 - 2 + g.halo, j0 - 2 + g.halo, q + g.halo, 0);
                }
            } else {
                // Cell by cell, NC apart: the row and component steps are taken as they come (a division
                // per cell and 64-bit offsets of all of them at once ran the whole march 1.6 times longer).
                const double* base = U + (i64)(q + g.halo) * g.isz + (i64)(j0 - 2 + g.halo) * g.isy + (i0 - 2 + g.halo);
                u32 m = keep(q), dst = rs + (slot * S::CELLS + cell) * 8;
                int xx = cell % PX, yy = cell / PX;
                const double* at = base + yy * g.isy + xx;
#pragma unroll 1
                for (int e = cell; e >= 0 && e < S::CELLS; e += NC) {
                    cp_async8_or_zero(dst, (m & 1u) ? at : base, m & 1u);
                    m >>= 1;
                    dst += NC * 8;
                    at += (NC / PX) * g.isy + NC % PX;
                    xx += NC % PX;
                    yy += NC / PX;
                    if (xx >= PX) {
                        xx -= PX;
                        ++yy;
                        at += g.isy - PX;
                    }
                    if (yy >= S::PY) {
                        yy -= S::PY;
                        at += g.isc - S::PY * g.isy;
                    }
                }
                cp_async_commit();
            }
        };
        auto landed = [&](int slot) {
            if (!TMA || !ok) return;
            ok = mbar_wait_bounded(bar(slot), (phase >> slot) & 1u, tmo);
            if (ok) phase ^= 1u << slot, flying &= ~(1u << slot);
        };
        // f(n, cell, kind) over this thread's cells of a slot; kind 0 rho, 1 momentum, 2 E
        auto kind_of = [&](int n) {
            const int e = cell + n * NC;
            return (n + 1) * NC <= PLANE ? 0 : n * NC >= PLANE && (n + 1) * NC <= 4 * PLANE ? 1 : n * NC >= 4 * PLANE ? 2
                   : e < PLANE ? 0 : e < 4 * PLANE ? 1 : 2;
        };

        // Prologue: the first six planes under way; exponent ranges of the first five.
        int next = k0 - 2;
        for (; next < k0 + 4 && next < k1 + 2; ++next) stage(next);
        if (tid < 5) note[tid] = tid == 1 || tid == 4 ? 0x7ff : 0;
        __syncthreads();
        u32 rng[5] = {0, ~0u, 0, 0, ~0u};   // of the exponents, shifted up
        if (!TMA) {
            cp_async_wait_all();
            __syncthreads();
        }
        const int scanned = min(5, next - k0 + 2);
        {
            static_assert(PLANE <= 2 * S::NT, "two cells of a component and plane per thread");
            bool in[2], mid[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int r = tid + i * S::NT, yy = r / PX, xx = r - yy * PX;
                const bool xin = xx >= 2 && xx < w + 2, yin = yy >= 2 && yy < h + 2, is = r < PLANE;
                in[i] = is && (!rim || (xx < w + 4 && yy < h + 4 && (xin || yin)));
                mid[i] = is && xin && yin;
            }
            u32 at = rs + tid * 8 + 4;
#pragma unroll 1
            for (int p = 0; p < scanned; ++p) {
                landed(p);
                const bool inner = k0 - 2 + p >= k0 && k0 - 2 + p < k1;
                const bool a0 = inner ? in[0] : mid[0], a1 = inner ? in[1] : mid[1];
#pragma unroll
                for (int c = 0; c < 5; ++c, at += PLANE * 8) {
                    const u32 e0 = a0 ? (u32)lds_int(at) << 1 : 0u, e1 = a1 ? (u32)lds_int(at + S::NT * 8) << 1 : 0u;
                    const u32 top = max(e0, e1), low = min(a0 ? e0 : ~0u, a1 ? e1 : ~0u);
                    if (c == 0) {
                        rng[0] = max(rng[0], top);
                        rng[1] = min(rng[1], low);
                    } else if (c < 4) {
                        rng[2] = max(rng[2], top);
                    } else {
                        rng[3] = max(rng[3], top);
                        rng[4] = min(rng[4], low);
                    }
                }
            }
        }
#pragma unroll
        for (int n = 0; n < 5; ++n) {
            const bool mn = n == 1 || n == 4;
            const int v = (int)((mn ? __reduce_min_sync(0xffffffffu, rng[n]) : __reduce_max_sync(0xffffffffu, rng[n])) >> 21);
            if ((tid & 31) == 0) {
                if (mn)
                    atomicMin(note + n, v);
                else
                    atomicMax(note + n, v);
            }
        }
        if (!ok) note[0] = 0x7ff;
        // The exponent ranges of the planes marched before, widened by this segment's: a flow that swings
        // over a power of two then ends one segment by it, not one per swing.
        RhsScale* const scale = scales();
        int seen[5];
#pragma unroll
        for (int n = 0; n < 5; ++n) seen[n] = scale->seen[n];
        __syncthreads();
        // Exponents: |rho| in [2^rlo, 2^rhi), |m| < 2^mhi, |E| in [2^elo, 2^ehi), of all planes so far or,
        // where these range too far, of the scanned ones.
        int rhi = 0, rlo = 0, mhi = 0, ehi = 0, elo = 0, efm = 0, efe = 0;
        bool fits = false, more = true;
#pragma unroll 1
        for (int t = 0; t < 2 && !fits && more; ++t) {
            more = false;   // whether the planes before widen the ranges
#pragma unroll
            for (int n = 0; n < 5; ++n) {
                const int now = note[n];
                seen[n] = t ? now : n == 1 || n == 4 ? min(seen[n], now) : max(seen[n], now);
                more |= seen[n] != now;
            }
            rhi = seen[0] - 1022;
            rlo = seen[1] - 1023 - 1;
            mhi = max(seen[2], 1023 + rlo - 60) - 1022;
            ehi = seen[3] - 1022;
            elo = seen[4] - 1023 - 1;
            fits = seen[0] < 0x7ff && seen[2] < 0x7ff && seen[3] < 0x7ff && abs(rhi) < 200 && abs(ehi) < 200 &&
                   abs(mhi) < 200 && rhi - rlo <= 8 && ehi - elo <= 8;
            if (!fits) continue;
            // Bounds of the fluxes, and whether quantising against them stays below what FP64 rounds
            // anyway at the least rho and E: the dissipation (eps 18 U 2^-53) for the mass and energy
            // components, the pressure ((gamma - 1) E 2^-53) for the momenta. All relative to 2^ehi, so that
            // the floats hold them whatever the unit of U is.
            const float g1 = fabsf(fx.g1), vmax = pow2f(mhi - rlo), mv = pow2f(2 * mhi - rlo - ehi), el = pow2f(elo - ehi);
            const float P = g1 * (1.f + 1.5f * mv);
            const float bm = (mv + P) * fx.smax * 1.01f, be = (1.f + P) * vmax * fx.smax * 1.01f, pl = fx.smin * g1 * el;
            fits = bm > 0x1p-100f && bm < 0x1p100f && be > 0x1p-100f && be < 0x1p100f && fx.eps >= fx.smax * vmax * 0x1p-10f &&
                   fx.eps * el >= be * 0x1p-10f && pl >= bm * 0x1p-8f && pl * 0x1p5f >= fx.eps * pow2f(mhi - ehi);
            efm = (__float_as_int(bm) >> 23) - 126 + ehi;
            efe = (__float_as_int(be) >> 23) - 126 + ehi;
        }
        if (!fits) {
            for (int p = scanned; p < next - k0 + 2; ++p) landed(p);
            return k0 - 1;
        }
        if (TMA) masks();
        // Conversion exponents (leading bit at 59) and the units of the sums. U has one more bit of room, so
        // that a flow may double on the way: the dissipation, 6/4 + 6 + 4.5 times the largest value, is
        // below 12 2^59 for values as scanned and for values of one sign (a negative rho or E ends the
        // segment), and may need more than 63 bits for larger momenta of both (see roomy).
        const int cr = rhi + 1023, cm = mhi + 1023, ce = ehi + 1023, cfm = efm + 1022, cfe = efe + 1022;
        const int ur = rhi - 59, um = mhi - 59, ue = ehi - 59;
        const int dx = 2 + 1 + fx.ex_eps;   // dissipation / 4, mul63
        const int es = max(max(fx.ex_s[0], fx.ex_s[1]), fx.ex_s[2]);
        const u32 sc = smem_addr(scale);
        if (tid == 0) {
            const RhsJoin j[3] = {rhs_join(um + 1 + es + (ISO ? 0 : 2), ur + dx), rhs_join(efm - 60, um + dx),
                                  rhs_join(efe - 60, ue + dx)};
            for (int n = 0; n < 3; ++n) {
                scale->join[n][0] = j[n].sa;
                scale->join[n][1] = j[n].sd;
                scale->join[n][2] = j[n].e;
                scale->cu[n] = n == 0 ? cr : n == 1 ? cm : ce;
                scale->lo[n] = n == 0 ? rlo + 1023 : n == 1 ? 0 : elo + 1023;
            }
            scale->cf[0] = cfm;
            scale->cf[1] = cfe;
            for (int n = 0; n < 5; ++n) scale->seen[n] = seen[n];
        }
        __syncthreads();

        auto raw = [&](u32 at) { return __longlong_as_double((long long)lds1(at)); };
        auto flux = [&](u32 at, double* fxv, double* fyv, double* fzv) {
            const RhsConst k = stage_consts_read<RhsConst>(smem + NSLOT * S::CELLS + S::FX_ELEMS + S::FY_ELEMS);
            const double rho = raw(at), mx = raw(at + PLANE * 8), my = raw(at + 2 * PLANE * 8), mz = raw(at + 3 * PLANE * 8),
                         E = raw(at + 4 * PLANE * 8);
            if (ISO)
                point_flux<true, true>(rho, mx, my, mz, E, k, fxv, fyv, fzv);
            else
                point_flux_scaled(rho, mx, my, mz, E, k, fxv, fyv, fzv);
        };
        int bad = 0;
        auto fixm = [&](double v) { return to_fixed((u64)__double_as_longlong(v), lds_int(sc + 72), 0, bad); };
        auto fixe = [&](double v) { return to_fixed((u64)__double_as_longlong(v), lds_int(sc + 76), 0, bad); };

        u64 pa[4] = {0, 0, 0, 0}, pb[4] = {0, 0, 0, 0}, fzp[4] = {0, 0, 0, 0};   // flux sums of q-1 and q-2, F_z of q-1
        u64 ix[4], iy[4], iz[4], rg[4];   // fluxes of plane q: the thread's own point, its ring point
        int cur = 0;   // slot of plane q
        int q = k0 - 2;
        auto back = [&](int d) { return rs + (cur - d < 0 ? cur - d + NSLOT : cur - d) * (S::CELLS * 8); };
        auto z_plane = [&](int p) { return p >= k0 - 1 && p <= k1; };
        auto xy_plane = [&](int p) { return p >= k0 && p < k1; };
        // The ring's point outside the tile: rows -1 and BY for the first 2 BX threads, columns -1 and BX
        // for the next 2 BY. Threads without a point take a cell that every tile has.
        const int ring = tid < 2 * BX ? 1 : tid < 2 * (BX + BY) ? 2 : 0;
        int rat = -1;   // where its fluxes go
        u32 rfrom = safe;
        if (ring == 1) {
            const int rx = tid >> 1, ry = (tid & 1) ? BY : -1;
            if (rx < w && (ry < 0 || h == BY)) {
                rat = (ry + 1) * BX + rx;
                rfrom = ((ry + 2) * PX + rx + 2) * 8;
            }
        } else if (ring == 2) {
            const int t = tid - 2 * BX, ry = t >> 1, rx = (t & 1) ? BX : -1;
            if (ry < h && (rx < 0 || w == BX)) {
                rat = ry * (BX + 2) + rx + 1;
                rfrom = ((ry + 2) * PX + rx + 2) * 8;
            }
        }
        auto ring_flux = [&](u32 sn) {   // of the plane at sn
            double a[4], b[4], c[4];
            flux(sn + rfrom, a, b, c);
            if (ring == 1) {
#pragma unroll
                for (int n = 0; n < 4; ++n) rg[n] = n < 3 ? fixm(b[n]) : fixe(b[n]);
            } else {
#pragma unroll
                for (int n = 0; n < 4; ++n) rg[n] = n < 3 ? fixm(a[n]) : fixe(a[n]);
            }
        };
        auto own_flux = [&](u32 sn) {
            double a[4], b[4], c[4];
            flux(sn + mine, a, b, c);
            ix[0] = fixm(a[0]), ix[1] = fixm(a[1]), ix[2] = fixm(a[2]), ix[3] = fixe(a[3]);
            iy[0] = ISO ? ix[1] : fixm(b[0]), iy[1] = fixm(b[1]), iy[2] = fixm(b[2]), iy[3] = fixe(b[3]);
            iz[0] = ISO ? ix[2] : fixm(c[0]), iz[1] = ISO ? iy[2] : fixm(c[1]), iz[2] = fixm(c[2]), iz[3] = fixe(c[3]);
        };
        // x and y flux differences of plane q; the flux sums move on by one plane.
        u64 po[4];   // the complete flux sums of plane q-2
        auto gather = [&](bool xy, bool zflux) {
#pragma unroll
            for (int n = 0; n < 4; ++n) {
                u64 pc = 0;
                if (xy) {
                    const u32 xr = fxs + ((n * BY + ty) * (BX + 2) + tx) * 8, yr = fys + (n * (BY + 2) + ty) * BX * 8 + tx * 8;
                    pc = (lds1(xr + 16) - lds1(xr)) + (lds1(yr + 2 * BX * 8) - lds1(yr)) - fzp[n];
                }
                po[n] = pb[n];
                pb[n] = pa[n] + (zflux ? iz[n] : 0);
                pa[n] = pc;
                if (zflux) fzp[n] = iz[n];
            }
        };
        u64 old[5];   // the thread's own values at plane q-4: its slot is being filled again
        auto emit = [&]() {   // the result at plane q-2
            const int kk = q - 2;
            const u32 s0 = back(2) + own, sm1 = back(3) + own, sp1 = back(1) + own, sp2 = back(0) + own;
            double* Rp = R + (i64)kk * g.osz + (i64)(j0 + ty) * g.osy + (i0 + tx);
            i64 z[5];
            int ze[5];
#pragma unroll
            for (int c = 0; c < 5; ++c) {
                constexpr int C = PLANE * 8;
                const u64 mid = lds1(s0 + c * C), below = lds1(sm1 + c * C);
                const u64 s2 = (lds1(s0 + c * C - 16) + lds1(s0 + c * C + 16) + lds1(s0 + c * C - 16 * PX)) +
                               (lds1(s0 + c * C + 16 * PX) + old[c] + lds1(sp2 + c * C));
                const u64 s1 = (lds1(s0 + c * C - 8) + lds1(s0 + c * C + 8) + lds1(s0 + c * C - 8 * PX)) +
                               (lds1(s0 + c * C + 8 * PX) + below + lds1(sp1 + c * C));
                old[c] = below;
                const u64 d4 = (u64)((i64)s2 >> 2) - s1 + (mid << 2) + (u64)((i64)mid >> 1);
                const i64 ds = mul63((i64)d4, fx.eh, fx.el);
                i64 a;
                if (c == 0) {
                    const u64 ax = lds1(s0 + C + 8) - lds1(s0 + C - 8), ay = lds1(s0 + 2 * C + 8 * PX) - lds1(s0 + 2 * C - 8 * PX),
                              az = lds1(sp1 + 3 * C) - lds1(sm1 + 3 * C);
                    if (ISO)
                        a = mul63((i64)(ax + ay + az), fx.sh[0], fx.sl[0]);
                    else
                        a = (mul63((i64)ax, fx.sh[0], fx.sl[0]) >> min(es - fx.ex_s[0] + 2, 63)) +
                            (mul63((i64)ay, fx.sh[1], fx.sl[1]) >> min(es - fx.ex_s[1] + 2, 63)) +
                            (mul63((i64)az, fx.sh[2], fx.sl[2]) >> min(es - fx.ex_s[2] + 2, 63));
                } else {
                    a = (i64)po[c - 1];
                }
                const int4 j = lds_int4(sc + (c == 0 ? 0 : c == 4 ? 32 : 16));
                z[c] = (a >> j.x) + (ds >> j.y);
                ze[c] = j.z;
            }
#pragma unroll
            for (int c = 0; c < 5; ++c) Rp[(i64)c * g.osc] = minus_from_fixed(z[c], ze[c]);
        };
        bool wide = false;   // a momentum is larger than those scanned
        const bool whole = w == BX && h == BY;
#pragma unroll 1
        for (; q < k1 + 2; ++q) {
            const u32 sq = rs + cur * (S::CELLS * 8);
            const int nslot = cur + 1 == NSLOT ? 0 : cur + 1;
            const u32 sn = rs + nslot * (S::CELLS * 8);
            const bool zflux = z_plane(q), xy = xy_plane(q);
            if (!TMA) cp_async_wait_all();   // this thread's copies up to plane q+1, visible after the barrier
            __syncthreads();   // plane q's raw values, plane q-1's fluxes and plane q-4 have been read
            if (next < k1 + 2 && next <= q + 2) stage(next++);
            if (xy) {
                if (fluxer) {
#pragma unroll
                    for (int n = 0; n < 4; ++n) {
                        sts1(fxs + ((n * BY + ty) * (BX + 2) + tx + 1) * 8, ix[n]);
                        sts1(fys + ((n * (BY + 2) + ty + 1) * BX + tx) * 8, iy[n]);
                    }
                }
                if (rat >= 0) {
#pragma unroll
                    for (int n = 0; n < 4; ++n)
                        sts1(ring == 1 ? fys + (n * (BY + 2) * BX + rat) * 8 : fxs + (n * BY * (BX + 2) + rat) * 8, rg[n]);
                }
            }
            if (q + 1 < k1 + 2 && q + 1 >= k0 + 3) landed(nslot);
            bool grew = false;
            // The ring's fluxes of plane q+1 in FP64, beside the other threads' conversion of plane q.
            if (ring) {
                if (xy_plane(q + 1)) ring_flux(sn);
            } else {   // plane q to fixed point, in place
                const u32 m = rim || !xy ? keep(q) : ~0u;
                u64 v[NE];
#pragma unroll
                for (int n = 0; n < NE; ++n)
                    v[n] = (n + 1) * NC <= S::CELLS || cell + n * NC < S::CELLS ? lds1(sq + (cell + n * NC) * 8) : 0ull;
                if (m != ~0u) {
#pragma unroll
                    for (int n = 0; n < NE; ++n) {   // cells no point reads: a value in range
                        const int kd = kind_of(n);
                        if (!((m >> n) & 1u)) v[n] = kd == 1 ? 0ull : (u64)(u32)lds_int(sc + 60 + 4 * kd) << 52;
                    }
                }
                int room = 1;
#pragma unroll
                for (int n = 0; n < NE; ++n) {
                    const int kd = kind_of(n);
                    const int cu = lds_int(sc + 48 + 4 * kd);
                    if ((n + 1) * NC <= S::CELLS || cell + n * NC < S::CELLS) {
                        if ((n + 1) * NC > 4 * PLANE || n * NC < PLANE)
                            bad |= ((int)((hi32(v[n]) << 1) >> 21) - lds_int(sc + 60 + 4 * kd)) | (kd == 1 ? 0 : (int)hi32(v[n]));
                        int s;
                        sts1(sq + (cell + n * NC) * 8, to_fixed_by(v[n], cu, 0, s));
                        if (n * NC >= PLANE && (n + 1) * NC <= 4 * PLANE) {
                            room = min(room, s);
                        } else {
                            bad |= s;
                            if ((n + 1) * NC > PLANE && n * NC < 4 * PLANE && kd == 1) room = min(room, s);
                        }
                    }
                }
                bad |= room;
                grew = room == 0 && !wide;
                if (TMA) fence_proxy_async();
            }
            if (wide && active && q - 2 >= k0 && !rhs_roomy<PX, PLANE>(back(3) + own, back(2) + own, back(1) + own)) bad = -1;
            if (!ok) bad = -1;
            // Plane q in fixed point, its fluxes; a value out of range ends the segment before it is used, and so
            // does a point of plane q-2 whose dissipation may not fit.
            if (__syncthreads_or(bad < 0 || grew)) {
                if (__syncthreads_or(bad < 0)) break;
                wide = true;
            }
            bad = 0;
            // Then plane q-2's result from integers and plane q+1's fluxes in FP64: independent, and in one
            // stretch of code where the whole tile takes part, so that the two pipes work at once.
            if (whole && q - 2 >= k0 && q + 1 < k1) {
                gather(true, true);
                emit();
                own_flux(sn);
            } else {
                if (active) {
                    gather(xy, zflux);
                    if (q - 2 >= k0) {
                        emit();
                    } else if (q == k0 + 1) {
#pragma unroll
                        for (int c = 0; c < 5; ++c) old[c] = lds1(back(3) + own + c * PLANE * 8);
                    }
                }
                // (Of the planes before and after the segment only points of the tile: their edges are not
                // staged, and an empty cell's flux would end the segment.)
                if (xy_plane(q + 1) ? fluxer : active && z_plane(q + 1)) own_flux(sn);
            }
            cur = nslot;
        }
        // Copies not waited for yet: planes after q + 1 that a segment cut short had under way.
        for (int p = max(q + 2, k0 + 3), s = slot_of(p); p < next; ++p, s = s + 1 == NSLOT ? 0 : s + 1) landed(s);
        if (!TMA) cp_async_wait_all();
        return min(max(q - 2, k0), k1);
    }
};

// One block's work: the BX x BY column tile at (i0, j0), z-planes [k0, k1). Ends with all threads past
// a barrier after their last shared-memory access. Returns the first plane that is left for the FP64
// march (k1 if none); `raw`: the ring holds planes from two below that one on, as rhs_rest takes them.
//
// The FP64 march follows where nothing of this one lives any more, after a block's last unit. Called from
// here it got what registers the loops over segments and units left it, and spilled: 256^3 with
// values that never fit ran 3730 us in the balanced kernel, against 3255 for the FP64 kernel.
//
// `tid`: the thread's number. How it comes about decides what the compiler carries in registers across the
// loops, and is as measured: read anew per segment (FRESH) in the batch kernel (32 grids 390 us, 425 otherwise),
// read once by tid_x and tid_y in the balanced kernel (256^3 1113 us, 1160).
template <int BX, int BY, bool TMA, bool ISO, bool FRESH = false>
__device__ __forceinline__ int rhs_fixed_march(const double* __restrict__ U, double* __restrict__ R, const Geom& g,
                                               const RhsConst& kc, const RhsFix& fx, int i0, int j0, int k0, int k1,
                                               double* smem, const CUtensorMap* map, unsigned* tmo, int tid, bool& raw) {
    using S = RhsFixShape<BX, BY>;
    const RhsFixMarch<BX, BY, TMA, ISO> m{U, R, g, kc, fx, i0, j0, k1, smem, map, tmo};
    stage_consts_write(smem + S::NSLOT * S::CELLS + S::FX_ELEMS + S::FY_ELEMS, kc, tid);
    if (tid < 5) m.scales()->seen[tid] = tid == 1 || tid == 4 ? 0x7ff : 0;
    if (TMA && tid == 0) {
        for (int s = 0; s < S::NSLOT; ++s) mbar_init(m.bar(s), 1);
        fence_mbar_init();
    }
    __syncthreads();
    u32 phase = 0, flying = 0;
    bool ok = !TMA || (smem_addr(smem) & 127u) == 0;
    int kk = k0;
    raw = false;
    for (int left = 4; kk < k1 && ok; --left) {
        const int done = m.segment(kk, FRESH ? tid_y() * BX + tid_x() : tid, phase, flying, ok);
        ok = block_ok(ok);   // (a barrier: shared memory is free again)
        raw = done < kk;
        if (raw) break;
        left += (done - kk) / 16;
        const bool stop = done == kk || left <= 0;
        kk = done;
        if (stop) break;
    }
    if (TMA) {
        if (tid == 0 && !ok)   // as star_fixed_march
            for (int s = 0; s < S::NSLOT; ++s)
                if ((flying >> s) & 1u) mbar_wait_bounded(m.bar(s), (phase >> s) & 1u, tmo);
        __syncthreads();
        if (tid == 0)
            for (int s = 0; s < S::NSLOT; ++s) mbar_inval(m.bar(s));
        __syncthreads();
    }
    raw = raw && ok;
    return kk;
}

// The planes [k0, k1) of a column in the FP64 march.
template <int BX, int BY, bool TMA, bool ISO>
__device__ __forceinline__ void rhs_rest(const double* __restrict__ U, double* __restrict__ R, const Geom& g, const RhsConst& kf,
                                         int i0, int j0, int k0, int k1, double* smem, const CUtensorMap* map, unsigned* tmo,
                                         bool raw) {
    rhs_march<BX, BY, TMA, ISO, RhsFixShape<BX, BY>>(U, R, g, kf, i0, j0, k0, k1, smem, map, tmo, raw);
    __syncthreads();
}

}  // namespace acs
