// Kernels and launchers of the fixed-point RHS march; rhs_fixed_iso.cu and rhs_fixed_gen.cu each compile
// one of its two spacing forms.
#pragma once

#include <cmath>
#include <cstring>

#include "rhs_fixed.cuh"

namespace acs {
namespace {

template <int BX, int BY, bool TMA, bool ISO>
__global__ void __launch_bounds__(BX* BY, RhsFixShape<BX, BY>::MINB)
    rhs_fixed_kernel(const double* __restrict__ U, double* __restrict__ R, const __grid_constant__ Geom g,
                     const __grid_constant__ RhsConst kf, const __grid_constant__ RhsConst kc,
                     const __grid_constant__ RhsFix fx, int kchunk, const __grid_constant__ CUtensorMap map,
                     unsigned* tmo) {
    extern __shared__ __align__(128) double smem[];
    const int i0 = blockIdx.x * BX, j0 = blockIdx.y * BY, k0 = blockIdx.z * kchunk, k1 = min(k0 + kchunk, g.nz);
    bool raw;
    const int tid = TMA ? threadIdx.y * BX + threadIdx.x : tid_y() * BX + tid_x();   // (as measured: 1207 / 1243, 1383 / 1427 us)
    const int left = rhs_fixed_march<BX, BY, TMA, ISO>(U, R, g, kc, fx, i0, j0, k0, k1, smem, &map, tmo, tid, raw);
    if (left < k1) rhs_rest<BX, BY, TMA, ISO>(U, R, g, kf, i0, j0, left, k1, smem, &map, tmo, raw);
}

template <int BX, int BY, bool TMA, bool ISO>
__global__ void __launch_bounds__(BX* BY, RhsFixShape<BX, BY>::MINB)
    rhs_fixed_balanced_kernel(const double* __restrict__ U, double* __restrict__ R, const __grid_constant__ Geom g,
                              const __grid_constant__ RhsConst kf, const __grid_constant__ RhsConst kc,
                              const __grid_constant__ RhsFix fx, const __grid_constant__ BalancedPlan plan,
                              const __grid_constant__ CUtensorMap map, unsigned* tmo) {
    extern __shared__ __align__(128) double smem[];
    __shared__ BlockLeft list[kBlockLeft];
    i64 col;
    int z0, z1, n = 0, count = 0;
    bool raw = false;
    for (; count < kBlockLeft && balanced_segment(plan, blockIdx.x, n, col, z0, z1); ++n) {
        const int i0 = (int)col % plan.ntx * BX, j0 = (int)col / plan.ntx * BY;
        const int left = rhs_fixed_march<BX, BY, TMA, ISO>(U, R, g, kc, fx, i0, j0, z0, z1, smem, &map, tmo, tid_y() * BX + tid_x(), raw);
        if (left < z1) {
            if (threadIdx.x == 0 && threadIdx.y == 0) list[count] = BlockLeft{i0, j0, left, z1};
            ++count;
        }
    }
    __syncthreads();
    // The listed planes, the last ones first (their ring may still hold them); a block with a full list
    // runs its other segments in FP64, too.
    for (int i = count - 1; i >= 0 || count == kBlockLeft; --i, raw = false) {
        BlockLeft l;
        if (i >= 0) {
            l = list[i];
        } else {
            if (!balanced_segment(plan, blockIdx.x, n++, col, z0, z1)) break;
            l = BlockLeft{(int)col % plan.ntx * BX, (int)col / plan.ntx * BY, z0, z1};
        }
        rhs_rest<BX, BY, TMA, ISO>(U, R, g, kf, l.i0, l.j0, l.from, l.to, smem, &map, tmo, raw);
    }
}

template <int BX, int BY, bool TMA, bool ISO>
acs_status launch_rhs_fixed_t(const double* U, double* R, const Geom& g, const RhsConst& kf, const RhsConst& kc,
                              const RhsFix& fx, int kchunk, int flags, const CUtensorMap& map, cudaStream_t s) {
    using S = RhsFixShape<BX, BY>;
    unsigned* tmo = wait_timeout_counter();
    if (!tmo) return fail(ACS_ERR_CUDA, "cannot address the wait-timeout counter");
    const int ntx = (g.nx + BX - 1) / BX, nty = (g.ny + BY - 1) / BY;
    const dim3 block(BX, BY, 1);
    if (flags & ACS_TILE_BALANCED) {
        const void* fn = (const void*)rhs_fixed_balanced_kernel<BX, BY, TMA, ISO>;
        acs_status st = ensure_smem(fn, S::BYTES);
        if (st != ACS_OK) return st;
        const i64 C = (i64)ntx * nty;
        i64 G = resident_blocks(fn, S::NT, S::BYTES);
        if (G <= 0) return fail(ACS_ERR_CUDA, "occupancy query failed for rhs_fixed_balanced_kernel");
        if (G > C * g.nz) G = C * g.nz;
        const BalancedPlan plan = balanced_plan(C, ntx, g.nz, (int)G);
        rhs_fixed_balanced_kernel<BX, BY, TMA, ISO><<<(unsigned)G, block, S::BYTES, s>>>(U, R, g, kf, kc, fx, plan, map, tmo);
        return launch_status("rhs_fixed_balanced_kernel");
    }
    const void* fn = (const void*)rhs_fixed_kernel<BX, BY, TMA, ISO>;
    acs_status st = ensure_smem(fn, S::BYTES);
    if (st != ACS_OK) return st;
    if (kchunk <= 0) kchunk = default_kchunk(g.nz, (i64)ntx * nty, S::MINB);
    const dim3 grid(ntx, nty, (g.nz + kchunk - 1) / kchunk);
    rhs_fixed_kernel<BX, BY, TMA, ISO><<<grid, block, S::BYTES, s>>>(U, R, g, kf, kc, fx, kchunk, map, tmo);
    return launch_status("rhs_fixed_kernel");
}

// 16 x 16 columns, with the tile's schedule and staging.
template <bool ISO>
acs_status launch_rhs_fixed_form(const double* U, double* R, const Geom& g, const RhsConst& kf, const RhsConst& kc,
                                 const RhsFix& fx, const acs_tile& t, cudaStream_t s) {
    constexpr int BX = 16, BY = 16;
    CUtensorMap map;
    memset(&map, 0, sizeof(map));
    if ((t.flags & ACS_TILE_TMA) && encode_plane_map(U, g, 5, BX + 4, BY + 4, &map) == ACS_OK)
        return launch_rhs_fixed_t<BX, BY, true, ISO>(U, R, g, kf, kc, fx, t.kchunk, t.flags, map, s);
    return launch_rhs_fixed_t<BX, BY, false, ISO>(U, R, g, kf, kc, fx, t.kchunk, t.flags, map, s);
}

}  // namespace
}  // namespace acs
