// Kernels and launchers of the fixed-point star march; star_fixed_iso.cu and star_fixed_gen.cu each
// compile one of its two weight forms.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstring>

#include "star_fixed.cuh"

namespace acs {
namespace {

// z-chunk of a launch: the work per resident slot plus a third of a chunk for the uneven end, each
// chunk paying about three plane steps for its prologue (384^3, 32 x 8: chunks of 64 ran 632 us, of
// 128 686 us, though both fill 95 % of their waves; 561 us now).
int star_fixed_kchunk(int nz, i64 columns, i64 slots) {
    static const int cand[] = {4, 6, 8, 12, 16, 24, 32, 48, 64, 96, 128};
    int best = nz;
    double best_cost = 1e300;
    for (int kc : cand) {
        if (kc > nz && kc != cand[0]) break;
        const double full = (double)columns * ((nz + kc - 1) / kc) / (double)(slots > 0 ? slots : 1);
        const double cost = (full > 1.0 ? full + 0.35 : 1.0) * ((kc < nz ? kc : nz) + 3.0);
        if (cost < best_cost - 1e-9) {
            best_cost = cost;
            best = kc < nz ? kc : nz;
        }
    }
    // A launch of one wave: the columns in as many parts as there are slots for, so that the SMs hold the same
    // number of blocks (160^3 of shells, where FP64 runs all of it, in chunks of 32 and 28: 16 x 8 204 -> 195 us,
    // 16 x 16 with distinct weights 222 -> 195, FP64 kernel 186; uniform values 59 -> 53 and 78 -> 70).
    if (columns * ((nz + best - 1) / best) <= slots) {
        const int parts = (int)(slots / columns);
        const int even = ((nz + parts - 1) / parts + 1) & ~1;   // (the march takes two planes at a time)
        best = std::max(std::min(best, 4), std::min(even, best));
    }
    return best < 1 ? 1 : best;
}

template <int BX, int BY, int MINB, bool TMA, bool ISO>
__global__ void __launch_bounds__(BX* BY / 2, MINB)
    star_fixed_kernel(const double* __restrict__ u, const double* __restrict__ a, double* __restrict__ out,
                      const __grid_constant__ Geom g, const __grid_constant__ StarCoef cf,
                      const __grid_constant__ StarFix fx, int kchunk, const __grid_constant__ CUtensorMap map, unsigned* tmo) {
    extern __shared__ __align__(128) double smem[];
    const int i0 = blockIdx.x * BX, j0 = blockIdx.y * BY, k0 = blockIdx.z * kchunk, k1 = min(k0 + kchunk, g.nz);
    bool raw;
    const int left = star_fixed_march<BX, BY, TMA, ISO>(u, a, out, g, cf, fx, i0, j0, k0, k1, smem, &map, tmo, threadIdx.x, raw);
    if (left < k1) star_rest<BX, BY, TMA>(u, a, out, g, cf, i0, j0, left, k1, &map, tmo, raw);
}

template <int BX, int BY, int MINB, bool TMA, bool ISO>
__global__ void __launch_bounds__(BX* BY / 2, MINB)
    star_fixed_balanced_kernel(const double* __restrict__ u, const double* __restrict__ a, double* __restrict__ out,
                               const __grid_constant__ Geom g, const __grid_constant__ StarCoef cf,
                               const __grid_constant__ StarFix fx, const __grid_constant__ BalancedPlan plan,
                               const __grid_constant__ CUtensorMap map, unsigned* tmo) {
    extern __shared__ __align__(128) double smem[];
    __shared__ BlockLeft list[kBlockLeft];
    i64 col;
    int z0, z1, n = 0, count = 0;
    bool raw = false;
    for (; count < kBlockLeft && balanced_segment(plan, blockIdx.x, n, col, z0, z1); ++n) {
        const int i0 = (int)col % plan.ntx * BX, j0 = (int)col / plan.ntx * BY;
        const int left = star_fixed_march<BX, BY, TMA, ISO>(u, a, out, g, cf, fx, i0, j0, z0, z1, smem, &map, tmo, threadIdx.x, raw);
        if (left < z1) {
            if (threadIdx.x == 0) list[count] = BlockLeft{i0, j0, left, z1};
            ++count;
        }
    }
    __syncthreads();
    // As in rhs_fixed_balanced_kernel.
    for (int i = count - 1; i >= 0 || count == kBlockLeft; --i, raw = false) {
        BlockLeft l;
        if (i >= 0) {
            l = list[i];
        } else {
            if (!balanced_segment(plan, blockIdx.x, n++, col, z0, z1)) break;
            l = BlockLeft{(int)col % plan.ntx * BX, (int)col / plan.ntx * BY, z0, z1};
        }
        star_rest<BX, BY, TMA>(u, a, out, g, cf, l.i0, l.j0, l.from, l.to, &map, tmo, raw);
    }
}

template <int BX, int BY, int MINB, bool TMA, bool ISO>
acs_status launch_star_fixed_t(const double* u, const double* a, double* out, const Geom& g, const StarCoef& c,
                               const StarFix& fx, int kchunk, int flags, const CUtensorMap& map, cudaStream_t s) {
    using S = StarFixShape<BX, BY>;
    unsigned* tmo = wait_timeout_counter();
    if (!tmo) return fail(ACS_ERR_CUDA, "cannot address the wait-timeout counter");
    const int ntx = (g.nx + BX - 1) / BX, nty = (g.ny + BY - 1) / BY;
    if (flags & ACS_TILE_BALANCED) {
        const void* fb = (const void*)star_fixed_balanced_kernel<BX, BY, MINB, TMA, ISO>;
        acs_status st = ensure_smem(fb, S::BYTES);
        if (st != ACS_OK) return st;
        const i64 C = (i64)ntx * nty;
        i64 G = resident_blocks(fb, S::NT, S::BYTES);
        if (G <= 0) return fail(ACS_ERR_CUDA, "occupancy query failed for star_fixed_balanced_kernel");
        if (G > C * g.nz) G = C * g.nz;
        const BalancedPlan plan = balanced_plan(C, ntx, g.nz, (int)G);
        star_fixed_balanced_kernel<BX, BY, MINB, TMA, ISO><<<(unsigned)G, S::NT, S::BYTES, s>>>(u, a, out, g, c, fx, plan, map, tmo);
        return launch_status("star_fixed_balanced_kernel");
    }
    const void* fn = (const void*)star_fixed_kernel<BX, BY, MINB, TMA, ISO>;
    acs_status st = ensure_smem(fn, S::BYTES);
    if (st != ACS_OK) return st;
    if (kchunk <= 0) kchunk = star_fixed_kchunk(g.nz, (i64)ntx * nty, resident_blocks(fn, S::NT, S::BYTES));
    dim3 grid(ntx, nty, (g.nz + kchunk - 1) / kchunk);
    star_fixed_kernel<BX, BY, MINB, TMA, ISO><<<grid, S::NT, S::BYTES, s>>>(u, a, out, g, c, fx, kchunk, map, tmo);
    return launch_status("star_fixed_kernel");
}

template <int BX, int BY, int MINB, bool ISO>
acs_status launch_star_fixed_tile(const double* u, const double* a, double* out, const Geom& g, const StarCoef& c,
                             const StarFix& fx, const acs_tile& t, cudaStream_t s) {
    CUtensorMap map;
    memset(&map, 0, sizeof(map));
    if ((t.flags & ACS_TILE_TMA) && encode_plane_map(u, g, 1, BX + 8, BY + 8, &map) == ACS_OK)
        return launch_star_fixed_t<BX, BY, MINB, true, ISO>(u, a, out, g, c, fx, t.kchunk, t.flags, map, s);
    return launch_star_fixed_t<BX, BY, MINB, false, ISO>(u, a, out, g, c, fx, t.kchunk, t.flags, map, s);
}


template <bool ISO>
acs_status launch_star_fixed_kind(const double* u, const double* a, double* out, const Geom& g, const StarCoef& c,
                                  const StarFix& fx, const acs_tile& t, cudaStream_t s) {
    if (t.bx == 32 && t.by == 8) return launch_star_fixed_tile<32, 8, 4, ISO>(u, a, out, g, c, fx, t, s);
    if (t.bx == 32 && t.by == 4) return launch_star_fixed_tile<32, 4, 8, ISO>(u, a, out, g, c, fx, t, s);
    if (t.bx == 32 && t.by == 16) return launch_star_fixed_tile<32, 16, 2, ISO>(u, a, out, g, c, fx, t, s);
    if (t.bx == 64 && t.by == 4) return launch_star_fixed_tile<64, 4, 4, ISO>(u, a, out, g, c, fx, t, s);
    if (t.bx == 64 && t.by == 8) return launch_star_fixed_tile<64, 8, 2, ISO>(u, a, out, g, c, fx, t, s);
    if (t.bx == 16 && t.by == 16) return launch_star_fixed_tile<16, 16, 4, ISO>(u, a, out, g, c, fx, t, s);
    if (t.bx == 16 && t.by == 8) return launch_star_fixed_tile<16, 8, 8, ISO>(u, a, out, g, c, fx, t, s);
    return fail(ACS_ERR_UNSUPPORTED, "stencil tile %dx%d is not built", t.bx, t.by);
}

}  // namespace
}  // namespace acs
