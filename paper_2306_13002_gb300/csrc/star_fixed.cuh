// March of the saturated star stencil in block-scaled fixed point (fixed.cuh).
//
//   out(p) = a(p) * (C0 u(p) + sum_d sum_o c[d][o] (u(p+o e_d) + u(p-o e_d)))
//
// With the same four weights on every axis the 24 neighbours are first summed per distance and
// five products remain; with distinct weights the 12 symmetric pairs are summed and 13 remain.
// The weights are 59- or 60-bit integers with W0 = -(sum of the others), so a common offset of all
// inputs (the bias, which keeps the integers unsigned) drops out of the sum exactly.
//
// Measured on GB300, tensor copies: 384^3 with 16 x 8 tiles 2388 us in FP64 (26 operations per point, 98 %
// of the FP64 pipe) -> 562 us; 768^3, a smooth wave with distinct weights per axis, 19.0 -> 6.33 ms. Fields
// whose every point is left to FP64 (values 2^40 apart): 384^3 2405 -> 2420, 160^3 186 -> 195, 61 x 47 x 53
// 21.0 -> 20.8.
// Error against 64 bits (2-norm): uniform values 3.1e-16 -> 8.1e-17, a smooth wave 5.8e-15 -> 9.6e-17. What
// bounds it now: about 240 instructions per point (127 on the ALU pipe, 63 on the FMA pipe) issued at 56 % of
// the peak rate, 16 warps per SM at 128 registers waiting on each other's results; launch bounds for
// more warps spill and run 1.1 to 2 times longer. The 2 FP64 additions and one multiplication left
// per point take 40 % of the FP64 pipe, memory 1.4 GB at a third of its rate.
#pragma once

#include "acs_internal.cuh"
#include "fixed.cuh"
#include "tma.cuh"

namespace acs {

// A point is small if u(p) and its +x, +y and +z neighbours, all four, are below 2^53 units (2^-6 to 2^-7 of
// the segment's largest value): it is evaluated in FP64. The conversion's errors (0.3 unit of each input,
// so mostly the centre weight's share, 2.7 units for Taylor weights) are then no larger than FP64's
// roundings at any other point, relative to its sum of |terms|: a host emulation of both sums gives,
// with all inputs just above the bound, 4.5e-17 against 8.1e-17 (of one sign and alike 2.9e-17 against
// 4.0e-17), and with one input there and the others far below, 1.5e-16 (+x or +y) and 1.1e-16 (centre)
// against 1.4e-16 to 1.7e-16. Weights whose nearest ones are a smaller share of the centre's raise the bound by
// that (StarFix::small), or leave +z out.
constexpr u32 kStarBiasHi = 1u << 28;            // 2^60: the offset that keeps inputs unsigned
constexpr u32 kStarSmallHi = 1u << 21;           // 2^53
constexpr int kStarIsoLB = 29, kStarGenLB = 28;  // bits of Wl (see StarFix)

// The sum at one point in FP64, from global memory: the saturated form's operations in their order.
static __device__ __noinline__ double star_point(const double* __restrict__ p, i64 isy, i64 isz, const StarCoef& cf) {
    double t = cf.c0 * __ldg(p);
#pragma unroll
    for (int o = 1; o <= 4; ++o) t = fma(cf.c[o - 1], __ldg(p + o) + __ldg(p - o), t);
#pragma unroll
    for (int o = 1; o <= 4; ++o) t = fma(cf.c[4 + o - 1], __ldg(p + o * isy) + __ldg(p - o * isy), t);
#pragma unroll
    for (int o = 1; o <= 4; ++o) t = fma(cf.c[8 + o - 1], __ldg(p + o * isz) + __ldg(p - o * isz), t);
    return t;
}

// A tile of BX x BY points; a thread owns two neighbours along x (16-byte shared loads) and takes two
// planes per iteration. Eight ring slots: the planes kk .. kk+5 in fixed point, and kk+6, kk+7, which
// are on their way from memory while planes kk and kk+1 are computed and converted in place after that.
// The four planes below kk sit in registers.
template <int BX, int BY>
struct StarFixShape {
    static constexpr int PX = BX + 8, PY = BY + 8, PLANE = PX * PY;
    static constexpr int NT = BX * BY / 2;
    static constexpr int NE = (PLANE + NT - 1) / NT;   // plane cells staged per thread
    static constexpr int NSLOT = 8;
    static constexpr int LIST = 4 * NT;   // points of one iteration
    // Ring, one mbarrier per slot, two shared words, the list, and 128 bytes to align the ring.
    static constexpr size_t BYTES = sizeof(u64) * ((size_t)NSLOT * PLANE + NSLOT + 1) + sizeof(u32) * LIST + 128;
    static_assert((PLANE * sizeof(u64)) % 128 == 0, "every ring slot 128-byte aligned");
};

template <int BX, int BY, bool TMA, bool ISO>
struct StarFixMarch {
    using S = StarFixShape<BX, BY>;
    static constexpr int PX = S::PX, PLANE = S::PLANE, NE = S::NE, NT = S::NT;

    const double* __restrict__ u;
    const double* __restrict__ a;
    double* __restrict__ out;
    const Geom& g;
    const StarCoef& cf;
    const StarFix& fx;
    int i0, j0, k1;
    u64* ring;
    u64* bars;
    u32* note;   // shared: [0] largest exponent word, [1] length of the list
    u32* list;   // shared: points that are evaluated in FP64 at the segment's end
    const CUtensorMap* map;
    unsigned* tmo;
    int tid, w, h, tx, ty;

    __device__ __forceinline__ bool valid(int c) const { return ty < h && tx + c < w; }

    __device__ __forceinline__ bool at_rim() const { return i0 == 0 || j0 == 0 || i0 + BX + 4 > g.nx || j0 + BY + 4 > g.ny; }
    // The cells of a plane that count, one bit each. In tiles at the grid's rim those that some point reads: a
    // caller may leave the others (corners of the halo) unset. Elsewhere all of them, since tensor copies
    // bring them all and both stagings have to find the same scale. On planes past the segment's end only
    // the columns themselves (core).
    __device__ __forceinline__ void cells_read(u32& full, u32& core, u32 (&off)[NE]) const {
        full = core = 0;
#pragma unroll
        for (int n = 0; n < NE; ++n) {
            const int e = tid + n * NT;
            const int yy = e / PX, xx = e - yy * PX;
            const bool xin = xx >= 4 && xx < w + 4, yin = yy >= 4 && yy < h + 4;
            const bool in = xx < w + 8 && yy < h + 8 && e < PLANE && (xin || yin || (!TMA && !at_rim()));
            off[n] = in ? (u32)(yy * (int)g.isy + xx) : 0u;
            if (in) full |= 1u << n;
            if (xin && yin) core |= 1u << n;
        }
    }
    // Stages plane q (raw values) into its slot: one tensor copy, or this thread's cells with
    // cp.async (zeros for the cells no point reads).
    __device__ __forceinline__ void stage(int q, int slot, const u32 (&off)[NE], u32 keep, u32& flying) const {
        u64* dst = ring + slot * PLANE;
        if (TMA) {
            flying |= 1u << slot;
            if (tid == 0) {
                fence_proxy_async();
                uint64_t* bar = reinterpret_cast<uint64_t*>(bars + slot);
                mbar_arrive_expect_tx(bar, PLANE * sizeof(u64));
                tma_load_3d(dst, map, bar, i0 - 4 + g.halo, j0 - 4 + g.halo, q + g.halo);
            }
        } else {
            const double* base = u + (i64)(q + g.halo) * g.isz + (i64)(j0 - 4 + g.halo) * g.isy + (i0 - 4 + g.halo);
#pragma unroll
            for (int n = 0; n < NE; ++n)
                if (NE * NT == PLANE || n + 1 < NE || tid + n * NT < PLANE)
                    cp_async8_or_zero(smem_addr(dst + tid + n * NT), base + off[n], (keep >> n) & 1u);
            cp_async_commit();
        }
    }

    // Marches from plane k0 at one scale; returns the first plane it did not finish, or k0 - 1 if the planes
    // do not suit a scale: the ring then holds planes k0 .. k0+5 (none past k1+3) as they are.
    // `crowded`: it ended since its list was full. `phase`: the parity of each slot's next tensor copy (one bit per slot; every thread waits
    // for every copy once); `flying`: the slots with a copy not waited for yet. `ok` turns false when a
    // wait runs out.
    __device__ __forceinline__ int segment(int k0, u32& phase, u32& flying, bool& ok, bool& crowded) const {
        crowded = false;
        u32 full, core, off[NE];
        cells_read(full, core, off);
        const bool rim = TMA && at_rim();
        if (TMA && !rim) full = ~0u;
        auto keep = [&](int q) { return q < k1 ? full : core; };
        const bool work = ty < h;
        const u32 rs = smem_addr(ring), mine = rs + ((ty + 4) * PX + tx + 4) * 8;
        const double* col0 = u + (i64)(k0 + g.halo) * g.isz + (i64)(j0 + ty + g.halo) * g.isy + (i0 + tx + g.halo);
        auto below = [&](int q, int c) {   // the column's value q planes below k0 (0 for -0, which converts to -1)
            const u64 v = valid(c) ? (u64)__double_as_longlong(__ldg(col0 - q * g.isz + c)) : 0ull;
            return (v << 1) ? v : 0ull;
        };
        auto cells = [&](int slot, auto&& f) {   // f(bit, cell) over this thread's cells of a slot
            const u32 c = rs + (slot * PLANE + tid) * 8;
#pragma unroll
            for (int n = 0; n < NE; ++n)
                if (NE * NT == PLANE || n + 1 < NE || tid + n * NT < PLANE) {
                    u64 v = lds1(c + 8 * n * NT);
                    f(n, v);
                    sts1(c + 8 * n * NT, v);
                }
        };
        auto landed = [&](int slot) {
            if (!TMA || !ok) return;
            ok = mbar_wait_bounded(reinterpret_cast<uint64_t*>(bars + slot), (phase >> slot) & 1u, tmo);
            if (ok) phase ^= 1u << slot, flying &= ~(1u << slot);
        };

        // Prologue: planes k0 .. k0+5 under way; the largest exponent in them and in the
        // column's four values below.
        int next = k0;   // the next plane to stage
        for (; next < k0 + 6 && next < k1 + 4; ++next) stage(next, next - k0, off, keep(next), flying);
        if (tid < 2) note[tid] = 0;
        u32 top = 0;
        auto see = [&](u64 v) { top = max(top, (hi32(v) & 0x7fffffffu) | (lo32(v) != 0 ? 1u : 0u)); };
        u64 past[4][2];   // [distance below - 1][column]
#pragma unroll
        for (int q = 1; q <= 4; ++q)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                past[q - 1][c] = below(q, c);
                see(past[q - 1][c]);
            }
        if (!TMA) cp_async_wait_all();
#pragma unroll 1
        for (int q = 0; q < next - k0; ++q) {
            landed(q);
            const u32 m = keep(k0 + q);
            cells(q, [&](int n, u64& v) {
                if (!TMA || (m >> n) & 1u) see(v);
            });
        }
        top = __reduce_max_sync(0xffffffffu, top);
        __syncthreads();
        if ((tid & 31) == 0) atomicMax(note, top);
        __syncthreads();
        if (!ok) note[0] = 0x7fffffffu;
        __syncthreads();
        top = note[0];
        const bool zero = top == 0;
        int E0 = (int)(top >> 20);
        if (!zero && (E0 < kFixMinExp || E0 > kFixMaxExp)) return k0 - 1;   // so, too, if a wait ran out
        if (!zero) {
            // Mostly small values: the list would be longer than the rest is worth.
            int seen = 0, few = 0;
            const int low = ISO ? 6 : 59 - (63 - __clz((int)fx.small));   // 2^53: 6 below the leading bit
            for (int q = 0; q < next - k0 && k0 + q < k1; ++q)
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    if (!valid(c)) continue;
                    ++seen;
                    few += (int)((u32)lds_int(mine + q * (PLANE * 8) + c * 8 + 4) << 1 >> 21) < E0 - low;
                }
            const int crowd = __syncthreads_count(2 * few > seen), all = __syncthreads_count(seen > 0);
            if (2 * crowd > all) return k0 - 1;
        }
        if (zero) E0 = kFixMinExp;
        int bad = 0;
        const u32 bound = ISO ? kStarSmallHi : fx.small, bias = kStarBiasHi + bound;
        // This thread's cells of plane q from raw to fixed point, in place.
        auto convert = [&](int slot, int q) {
            if (zero) {
                const u32 m = keep(q);
                cells(slot, [&](int n, u64& v) {
                    if ((v << 1) != 0 && (!TMA || (m >> n) & 1u)) bad = -1;
                    v = (u64)bias << 32;
                });
            } else if (rim || (TMA && q >= k1)) {
                const u32 m = keep(q);
                cells(slot, [&](int n, u64& v) { v = to_fixed((m >> n) & 1u ? v : 0ull, E0, bias, bad); });
            } else {
                cells(slot, [&](int, u64& v) { v = to_fixed(v, E0, bias, bad); });
            }
            if (TMA) fence_proxy_async();
        };
        int kk = k0;
#pragma unroll 1
        for (int q = 0; q < next - k0; ++q) convert(q, k0 + q);
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int c = 0; c < 2; ++c) past[q][c] = to_fixed(past[q][c], E0, bias, bad);
        const FixOut fo = fix_out(E0 - 1023 - 59 + fx.shift, fx.neg != 0);
        const u32 small = zero ? 0u : 2 * bound;
        // + 1: the two floors in the joined sum lose half a unit each on average.
        const u64 round = zero ? 0 : 1;
        const i64 at0 = (i64)(k0 + g.halo) * g.isz + (i64)(j0 + ty + g.halo) * g.isy + (i0 + tx + g.halo);
        const double* ap = a + at0;
        double* op = out + (i64)k0 * g.osz + (i64)(j0 + ty) * g.osy + i0 + tx;
        const bool v0 = valid(0), v1 = valid(1);
        // Pairs of a and out as 16-byte accesses where their addresses allow it (tx is even).
        auto even = [](const void* at, i64 sy, i64 sz) { return ((uintptr_t)at & 15) == 0 && ((sy | sz) & 1) == 0; };
        const bool a16 = even(a + at0 - tx - ty * g.isy, g.isy, g.isz), o16 = even(op - tx - ty * g.osy, g.osy, g.osz);
        int cur = 0;   // the slot of plane kk
        __syncthreads();
#pragma unroll 1
        for (; kk < k1; kk += 2) {
            const bool two = kk + 1 < k1;
            double av[2][2];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                av[j][0] = av[j][1] = 0.0;
                if (j && !two) continue;
                if (v1 && a16) {
                    const double2 t = __ldg(reinterpret_cast<const double2*>(ap + j * g.isz));
                    av[j][0] = t.x;
                    av[j][1] = t.y;
                } else if (v0) {
                    av[j][0] = __ldg(ap + j * g.isz);
                    if (v1) av[j][1] = __ldg(ap + j * g.isz + 1);
                }
            }
#pragma unroll
            for (int j = 0; j < 2; ++j)   // planes kk+6 and kk+7 into the slots of kk-2 and kk-1
                if (next + j < k1 + 4) stage(next + j, (cur + 6 + j) & 7, off, keep(next + j), flying);
            next = min(next + 2, k1 + 4);
            if (work) {
                u32 s[6];   // planes kk .. kk+5 at the thread's points
#pragma unroll
                for (int j = 0; j < 6; j += 2) {
                    s[j] = mine + ((cur + j) & 7) * (PLANE * 8);
                    s[j + 1] = s[j] + PLANE * 8;
                }
                u64 here[2][2];
                u32 least = ~0u;
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    u64 row[10];
#pragma unroll
                    for (int x = 0; x < 10; x += 2) {
                        const U64x2 t = lds2(s[j] + (x - 4) * 8);
                        row[x] = t.x;
                        row[x + 1] = t.y;
                    }
                    here[j][0] = row[4];
                    here[j][1] = row[5];
                    FixAcc t[2] = {{0, 0, 0, 0}, {0, 0, 0, 0}};
                    u32 nh[2], nl[2];
#pragma unroll
                    for (int o = 1; o <= 4; ++o) {
                        const U64x2 yp2 = lds2(s[j] + o * PX * 8), ym2 = lds2(s[j] - o * PX * 8);
                        const U64x2 zp2 = lds2(s[j + o]);
#pragma unroll
                        for (int c = 0; c < 2; ++c) {
                            const u64 xp = row[4 + c + o], xm = row[4 + c - o];
                            const u64 yp = c ? yp2.y : yp2.x, ym = c ? ym2.y : ym2.x;
                            const u64 zp = c ? zp2.y : zp2.x;
                            const u64 zm = o <= j ? here[0][c] : past[o - 1 - j][c];
                            if (o == 1) {
                                nh[c] = hi32(row[4 + c]);
                                nl[c] = lo32(row[4 + c]);
                                least = min(least, (nh[c] ^ kStarBiasHi) | (hi32(xp) ^ kStarBiasHi) | (hi32(yp) ^ kStarBiasHi));
                            }
                            if (ISO) {
                                const u64 sm = (xp + xm + yp) + (ym + zp + zm);
                                fix_mac(t[c], sm, fx.wh[o], fx.wl[o]);
                                if (o % 2 == 0) {
                                    nh[c] += hi32(sm);
                                    nl[c] += lo32(sm);
                                }
                            } else {
                                const u64 sx = xp + xm, sy = yp + ym, sz = zp + zm;
                                fix_mac(t[c], sx, fx.wh[o], fx.wl[o]);
                                fix_mac(t[c], sy, fx.wh[4 + o], fx.wl[4 + o]);
                                fix_mac(t[c], sz, fx.wh[8 + o], fx.wl[8 + o]);
                                if (o % 2 == 0) {
                                    nh[c] += hi32(sx) + hi32(sy) + hi32(sz);
                                    nl[c] += lo32(sx) + lo32(sy) + lo32(sz);
                                }
                            }
                        }
                    }
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        fix_mac(t[c], row[4 + c], fx.wh[0], fx.wl[0]);
                        fix_neg(t[c], nh[c], nl[c]);
                        constexpr int LB = ISO ? kStarIsoLB : kStarGenLB;
                        const u64 sum = (t[c].hh << 3) + ((t[c].hl + hi32(t[c].ll)) >> (LB - 3)) +
                                        (u64)((i64)t[c].lh >> 29) + round;
av[j][c] *= from_fixed((i64)sum, fo);
                    }
                    if (j && !two) continue;
                    if (v1 && o16) {
                        *reinterpret_cast<double2*>(op + j * g.osz) = make_double2(av[j][0], av[j][1]);
                    } else if (v0) {
                        op[j * g.osz] = av[j][0];
                        if (v1) op[j * g.osz + 1] = av[j][1];
                    }
                }
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    past[3][c] = past[1][c];
                    past[2][c] = past[0][c];
                    past[1][c] = here[0][c];
                    past[0][c] = here[1][c];
                }
                if (least < small) {   // some of the four points may go on the list
#pragma unroll 1
                    for (int p = 0; p < 4; ++p) {
                        const int j = p >> 1, c = p & 1;
                        if (!(c ? v1 : v0) || (j && !two)) continue;
                        const u32 q = mine + (((cur + j) & 7) * PLANE + c) * 8, qz = mine + (((cur + j + 1) & 7) * PLANE + c) * 8;
                        if (((hi32(lds1(q)) ^ kStarBiasHi) | (hi32(lds1(q + 8)) ^ kStarBiasHi) |
                             (hi32(lds1(q + PX * 8)) ^ kStarBiasHi) | ((hi32(lds1(qz)) ^ kStarBiasHi) & (ISO ? ~0u : fx.zmask))) >= small)
                            continue;
                        const u32 at = atomicAdd(note + 1, 1u);
                        if (at < (u32)S::LIST)
                            list[at] = ((u32)(kk + j - k0) * BY + ty) * BX + tx + c;
                        else
                            bad = -1;
                    }
                }
            }
            // Planes kk+6 and kk+7 to fixed point (read from the next iteration on).
            if (!TMA) cp_async_wait_all();
#pragma unroll 1
            for (int j = 6; j < 8; ++j)
                if (kk + j < k1 + 4) {
                    landed((cur + j) & 7);
                    convert((cur + j) & 7, kk + j);
                }
            if (!ok) bad = -1;
            ap += 2 * g.isz;
            op += 2 * g.osz;
            cur = (cur + 2) & 7;
            if (__syncthreads_or(bad < 0)) {
                if (note[1] <= (u32)S::LIST) kk += 2;   // else these two planes are done again
                break;
            }
        }
        kk = min(kk, k1);
        // The listed points (of finished planes), by all threads.
        __syncthreads();
        const u32 listed = min(note[1], (u32)S::LIST);
        crowded = note[1] > (u32)S::LIST;
        for (u32 n = tid; n < listed; n += NT) {
            const int x = list[n] % BX, y = list[n] / BX % BY, q = k0 + (int)(list[n] / (BX * BY));
            if (q >= kk) continue;
            const i64 at = (i64)(q + g.halo) * g.isz + (i64)(j0 + y + g.halo) * g.isy + (i0 + x + g.halo);
            out[(i64)q * g.osz + (i64)(j0 + y) * g.osy + i0 + x] = __ldg(a + at) * star_point(u + at, g.isy, g.isz, cf);
        }
        return kk;
    }
};

// One block's work: the BX x BY column tile at (i0, j0), z-planes [k0, k1). Ends with all threads past a
// barrier after their last shared-memory access. A segment that meets a value beyond its scale (or too
// many points below it) ends early and the next one starts with a scale of its own. Returns the first
// plane that is left for star_rest (k1 if none): after several short segments, after one that filled its
// list within 16 planes (an eighth of its points), or where the planes at hand do not suit a scale;
// `raw`: the ring then holds them.
template <int BX, int BY, bool TMA, bool ISO>
__device__ __forceinline__ int star_fixed_march(const double* __restrict__ u, const double* __restrict__ a,
                                                double* __restrict__ out, const Geom& g, const StarCoef& cf,
                                                const StarFix& fx, int i0, int j0, int k0, int k1, double* smem,
                                                const CUtensorMap* map, unsigned* tmo, int tid, bool& raw) {
    using S = StarFixShape<BX, BY>;
    raw = false;
    if (g.isy >= (1 << 22)) return k0;   // staging offsets are 32 bits
    // A tile cut by the grid's x edge packs its column pairs into the first threads (see star_march).
    const int w = min(BX, g.nx - i0), h = min(BY, g.ny - j0), wp = (w + 1) / 2;
    u64* ring = reinterpret_cast<u64*>(align128(smem));
    u64* bars = ring + S::NSLOT * S::PLANE;
    const StarFixMarch<BX, BY, TMA, ISO> m{u,    a,   out, g,   cf,  fx, i0, j0, k1, ring,
                                           bars, reinterpret_cast<u32*>(bars + S::NSLOT), reinterpret_cast<u32*>(bars + S::NSLOT + 1), map, tmo, tid, w, h,
                                           2 * (w == BX ? tid % (BX / 2) : tid % wp),
                                           w == BX ? tid / (BX / 2) : tid / wp};
    if (TMA) {
        if (tid == 0) {
            for (int s = 0; s < S::NSLOT; ++s) mbar_init(reinterpret_cast<uint64_t*>(bars + s), 1);
            fence_mbar_init();
        }
        __syncthreads();
    }
    u32 phase = 0, flying = 0;
    bool ok = true;
    int kk = k0;
    for (int left = 4; kk < k1 && ok; --left) {
        bool crowded;
        const int done = m.segment(kk, phase, flying, ok, crowded);
        ok = block_ok(ok);   // (a barrier: the ring and the notes are free again)
        raw = done < kk;
        if (raw) break;
        const bool stop = done == kk || (crowded && done - kk < 16);
        left += (done - kk) / 16;
        kk = done;
        if (stop || left <= 0) break;
    }
    if (TMA) {
        // Copies may still be in flight after a wait of thread 0 ran out (another thread's: it has seen them
        // land): one more bounded wait each.
        if (tid == 0 && !ok)
            for (int s = 0; s < S::NSLOT; ++s)
                if ((flying >> s) & 1u) mbar_wait_bounded(reinterpret_cast<uint64_t*>(bars + s), (phase >> s) & 1u, tmo);
        __syncthreads();
        if (tid == 0)
            for (int s = 0; s < S::NSLOT; ++s) mbar_inval(reinterpret_cast<uint64_t*>(bars + s));
        __syncthreads();
    }
    raw = raw && ok;
    return kk;
}

// The planes [k0, k1) of a column in FP64, with star_march's operations in their order: two neighbours along x
// per thread and the ring of eight planes above, staged three steps ahead. A function of its own: inlined, it
// cost the fixed-point march registers (384^3 595 -> 645 us). `raw`: planes k0 .. k0+5 are in
// slots 0 .. 5, and no copy is in flight. Bound by the FP64 pipe like star_march; a field whose every
// point comes here (384^3, see star_fixed_march) runs as fast as in that kernel.
template <int BX, int BY, bool TMA>
__device__ __noinline__ void star_rest(const double* __restrict__ u, const double* __restrict__ a, double* __restrict__ out,
                                          const Geom& g, const StarCoef& cfc, int i0, int j0, int k0, int k1,
                                          const CUtensorMap* map, unsigned* tmo, bool raw) {
    extern __shared__ __align__(128) double smem[];
    using S = StarFixShape<BX, BY>;
    constexpr int PX = S::PX, PLANE = S::PLANE, HELD = 6;
    static_assert(S::LIST * sizeof(u32) >= sizeof(StarCoef), "the weights take the list's place");
    const int tid = tid_x();
    const int w = min(BX, g.nx - i0), h = min(BY, g.ny - j0), wp = (w + 1) / 2;
    const int tx = 2 * (w == BX ? tid % (BX / 2) : tid % wp), ty = w == BX ? tid / (BX / 2) : tid / wp;
    const bool v0 = ty < h && tx < w, v1 = ty < h && tx + 1 < w;
    double* ring = align128(smem);
    uint64_t* bars = reinterpret_cast<uint64_t*>(ring + S::NSLOT * PLANE);
    double* Cs = reinterpret_cast<double*>(bars + S::NSLOT + 1);
    const u32 own = v0 ? ((ty + 4) * PX + tx + 4) * 8 : (4 * PX + 4) * 8, rs = smem_addr(ring);
    const int top = k1 + 3;   // the last plane needed
    auto slot = [&](int q) { return (q - k0) & 7; };
    // Fills of a slot are counted from the barriers' start: the planes at hand are none.
    auto parity = [&](int q) { return (u32)(((q - k0) >> 3) - (raw && slot(q) < HELD)) & 1u; };
    bool ok = true;
    int lost = 0x7fffffff, issued = 0;   // thread 0: the plane whose wait ran out, the last one under way
    auto stage = [&](int q) {
        if (TMA) {
            if (tid == 0 && ok) {
                fence_proxy_async();
                mbar_arrive_expect_tx(bars + slot(q), PLANE * 8);
                tma_load_3d(ring + slot(q) * PLANE, map, bars + slot(q), i0 - 4 + g.halo, j0 - 4 + g.halo, q + g.halo);
                issued = q;
            }
        } else {
            const double* base = u + (i64)(q + g.halo) * g.isz + (i64)(j0 - 4 + g.halo) * g.isy + (i0 - 4 + g.halo);
            const int xlim = min(PX, g.nx + 8 - i0), ylim = min(S::PY, g.ny + 8 - j0);
#pragma unroll 1
            for (int e = tid; e < PLANE; e += S::NT) {
                const int yy = e / PX, xx = e - yy * PX;
                if (xx < xlim && yy < ylim) cp_async8(ring + slot(q) * PLANE + e, base + (i64)yy * g.isy + xx);
            }
        }
    };
    auto landed = [&](int q) {
        if (!TMA || !ok) return;
        ok = mbar_wait_bounded(bars + slot(q), parity(q), tmo);
        if (!ok) lost = q;
    };
    stage_consts_write(Cs, cfc, tid);
    if (TMA) {
        if (tid == 0) {
            for (int s = 0; s < S::NSLOT; ++s) mbar_init(bars + s, 1);
            fence_mbar_init();
        }
        __syncthreads();
    }
    // (Element-wise: planes k0 .. k0+4 in one group, each further one in a group of its own.)
    for (int q = raw ? k0 + HELD : k0; q <= k0 + 6; ++q) {
        if (q <= top) stage(q);
        if (!TMA && q >= k0 + 4) cp_async_commit();
    }
    if (!raw) {
        for (int q = k0; q <= k0 + 4; ++q) landed(q);
        if (!TMA) cp_async_wait_group2();
    }
    __syncthreads();
    const StarCoef cf = stage_consts_read<StarCoef>(Cs);
    const Pipe& p = cf.pp;
    auto pair = [&](u32 at, double (&v)[2]) {
        const U64x2 t = lds2(at);
        v[0] = __longlong_as_double((long long)t.x);
        v[1] = __longlong_as_double((long long)t.y);
    };
    double zq[9][2];   // the columns' values at planes kk-4 .. kk+4
    const i64 at0 = (i64)(k0 + g.halo) * g.isz + (i64)(j0 + ty + g.halo) * g.isy + (i0 + tx + g.halo);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        zq[m][0] = v0 ? __ldg(u + at0 + (m - 4) * g.isz) : 0.0;
        zq[m][1] = v1 ? __ldg(u + at0 + (m - 4) * g.isz + 1) : 0.0;
    }
#pragma unroll
    for (int m = 4; m < 9; ++m) pair(rs + slot(k0 + m - 4) * (PLANE * 8) + own, zq[m]);
    const double* ap = a + at0;
    double* op = out + (i64)k0 * g.osz + (i64)(j0 + ty) * g.osy + i0 + tx;
#pragma unroll 1
    for (int kk = k0; kk < k1; ++kk) {
        if (kk + 7 <= top) stage(kk + 7);   // into the slot of plane kk-1
        if (!TMA) cp_async_commit();
        if (v0) {
            const u32 s0 = rs + slot(kk) * (PLANE * 8) + own;
            double row[10];
#pragma unroll
            for (int x = 0; x < 10; x += 2) {
                double v[2];
                pair(s0 + (x - 4) * 8, v);
                row[x] = v[0];
                row[x + 1] = v[1];
            }
            double t[2];
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                t[c] = pmul(cf.c0, zq[4][c], p);
#pragma unroll
                for (int o = 1; o <= 4; ++o) t[c] = fma(cf.c[o - 1], padd(row[4 + c + o], row[4 + c - o], p), t[c]);
            }
#pragma unroll
            for (int o = 1; o <= 4; ++o) {
                double yp[2], ym[2];
                pair(s0 + o * PX * 8, yp);
                pair(s0 - o * PX * 8, ym);
#pragma unroll
                for (int c = 0; c < 2; ++c) t[c] = fma(cf.c[4 + o - 1], padd(yp[c], ym[c], p), t[c]);
            }
#pragma unroll
            for (int o = 1; o <= 4; ++o)
#pragma unroll
                for (int c = 0; c < 2; ++c) t[c] = fma(cf.c[8 + o - 1], padd(zq[4 + o][c], zq[4 - o][c], p), t[c]);
            op[0] = pmul(__ldg(ap), t[0], p);
            if (v1) op[1] = pmul(__ldg(ap + 1), t[1], p);
        }
        ap += g.isz;
        op += g.osz;
        if (kk + 5 <= top && !(raw && kk + 5 < k0 + HELD)) landed(kk + 5);
        if (!TMA) cp_async_wait_group2();   // every group but the last two steps': plane kk+5 is there
        __syncthreads();
#pragma unroll
        for (int m = 0; m < 8; ++m)
#pragma unroll
            for (int c = 0; c < 2; ++c) zq[m][c] = zq[m + 1][c];
        if (kk + 1 < k1) pair(rs + slot(kk + 5) * (PLANE * 8) + own, zq[8]);
    }
    if (TMA) {
        if (tid == 0 && !ok && lost != 0x7fffffff)   // copies that may still be in flight: one more bounded wait each
            for (int q = lost; q <= issued; ++q) mbar_wait_bounded(bars + slot(q), parity(q), tmo);
        __syncthreads();
        if (tid == 0)
            for (int s = 0; s < S::NSLOT; ++s) mbar_inval(bars + s);
    } else {
        cp_async_wait_all();
    }
    __syncthreads();
}

}  // namespace acs
