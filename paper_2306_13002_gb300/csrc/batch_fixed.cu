// The batched persistent launch with the fixed-point marches (star_fixed.cuh, rhs_fixed.cuh): the same
// queue of units as batch_kernel. Measured on GB300: 64 star grids with sides of 16 to 160 680 -> 235 us,
// 32 RHS grids with sides of 16 to 96 912 -> 390 us (small grids: a third of the steps of an RHS unit are
// its start, and its element-wise staging has to serve any row pitch).
#include "batch_desc.cuh"
#include "rhs_fixed.cuh"
#include "star_fixed.cuh"

namespace acs {
namespace {

template <int BX, int BY, bool TMA, bool ISO, int MINB>
__global__ void __launch_bounds__(BX* BY / 2, MINB)
    batch_star_fixed_kernel(const unsigned char* __restrict__ ws, unsigned long long* counter,
                            const __grid_constant__ StarCoef cf, const __grid_constant__ StarFix fx, unsigned* tmo) {
    extern __shared__ __align__(128) double smem[];
    __shared__ long long s_unit;
    const BatchView b = batch_view(ws);
    for (;;) {
        BatchUnit u;
        if (!batch_next(b, counter, &s_unit, threadIdx.x == 0, u)) break;
        const BatchDesc& d = b.items[u.item];
        const Geom g = d.g;
        const int i0 = u.tx * BX, j0 = u.ty * BY;
        const CUtensorMap* map = nullptr;
        if (TMA) {
            map = reinterpret_cast<const CUtensorMap*>(ws + b.head->maps_off) + u.item;
            if (threadIdx.x == 0) tensormap_acquire(map);
        }
        bool raw;
        const int left = star_fixed_march<BX, BY, TMA, ISO>(d.in0, d.in1, d.out, g, cf, fx, i0, j0, u.k0, u.k1, smem, map, tmo,
                                                            tid_x(), raw);
        if (left < u.k1) star_rest<BX, BY, TMA>(d.in0, d.in1, d.out, g, cf, i0, j0, left, u.k1, map, tmo, raw);
    }
}

template <int BX, int BY, bool ISO>
__global__ void __launch_bounds__(BX* BY, RhsFixShape<BX, BY>::MINB)
    batch_rhs_fixed_kernel(const unsigned char* __restrict__ ws, unsigned long long* counter,
                           const __grid_constant__ RhsConst kf, const __grid_constant__ RhsConst kc,
                           const __grid_constant__ RhsFix fx) {
    extern __shared__ __align__(128) double smem[];
    __shared__ long long s_unit;
    const BatchView b = batch_view(ws);
    const bool leader = threadIdx.x == 0 && threadIdx.y == 0;
    bool raw = false;
    int left = 0;
    BatchUnit u;
    for (;;) {
        if (!batch_next(b, counter, &s_unit, leader, u)) return;
        const BatchDesc& d = b.items[u.item];
        const Geom g = d.g;
        // (Little work: no planes for this march, since the FP64 one starts sooner. As a branch of its own the
        // test cost 32 grids 10 to 40 us of 390, by the registers it moved.)
        const int k1 = b.head->plain ? u.k0 : u.k1;
        left = rhs_fixed_march<BX, BY, false, ISO, true>(d.in0, d.out, g, kc, fx, u.tx * BX, u.ty * BY, u.k0, k1, smem, nullptr,
                                                   nullptr, threadIdx.y * BX + threadIdx.x, raw);
        if (left < u.k1) break;
    }
    // A block that met values that do not fit takes its further units in FP64 as well: what does not fit in
    // one grid mostly does not in the others (the parameters decide), and the queue evens out the time.
    u.k0 = left;
    do {
        const BatchDesc& d = b.items[u.item];
        const Geom g = d.g;
        rhs_rest<BX, BY, false, ISO>(d.in0, d.out, g, kf, u.tx * BX, u.ty * BY, u.k0, u.k1, smem, nullptr, nullptr, raw);
        raw = false;
    } while (batch_next(b, counter, &s_unit, leader, u));
}

template <class K, class... A>
acs_status launch_batch(K kernel, dim3 block, size_t smem, const BatchPlanHost& p, cudaStream_t s, const char* name, A... args) {
    acs_status st = ensure_smem((const void*)kernel, smem);
    if (st != ACS_OK) return st;
    i64 blocks = resident_blocks((const void*)kernel, block.x * block.y, smem);
    if (blocks < 1) return fail(ACS_ERR_CUDA, "occupancy query failed for %s", name);
    if (blocks > p.total) blocks = p.total;
    kernel<<<(unsigned)blocks, block, smem, s>>>(p.ws, args...);
    return launch_status(name);
}

template <int BX, int BY, int MINB>
acs_status launch_star_t(const BatchPlanHost& p, unsigned long long* counter, const StarCoef& sc, const StarFix& fx,
                         cudaStream_t s) {
    unsigned* tmo = wait_timeout_counter();
    if (!tmo) return fail(ACS_ERR_CUDA, "cannot address the wait-timeout counter");
    using S = StarFixShape<BX, BY>;
    auto run = [&](auto kernel) { return launch_batch(kernel, dim3(S::NT), S::BYTES, p, s, "batch_star_fixed_kernel", counter, sc, fx, tmo); };
    if (p.tile.flags & ACS_TILE_TMA)   // all grids have tensor maps (batch_pack)
        return fx.kind == 1 ? run(batch_star_fixed_kernel<BX, BY, true, true, MINB>) : run(batch_star_fixed_kernel<BX, BY, true, false, MINB>);
    return fx.kind == 1 ? run(batch_star_fixed_kernel<BX, BY, false, true, MINB>) : run(batch_star_fixed_kernel<BX, BY, false, false, MINB>);
}

template <int BX, int BY>
acs_status launch_rhs_t(const BatchPlanHost& p, unsigned long long* counter, const RhsConst& rk, const RhsConst& kc,
                        const RhsFix& fx, cudaStream_t s) {
    using S = RhsFixShape<BX, BY>;
    return rhs_isotropic(kc) ? launch_batch(batch_rhs_fixed_kernel<BX, BY, true>, dim3(BX, BY), S::BYTES, p, s,
                                            "batch_rhs_fixed_kernel", counter, rk, kc, fx)
                             : launch_batch(batch_rhs_fixed_kernel<BX, BY, false>, dim3(BX, BY), S::BYTES, p, s,
                                            "batch_rhs_fixed_kernel", counter, rk, kc, fx);
}

}  // namespace

// Runs the batch in fixed point if its weights or parameters suit (false: the FP64 kernel takes it).
bool batch_fixed_launch(const BatchPlanHost& p, unsigned long long* counter, const RhsConst& rk, const StarCoef& sc,
                        cudaStream_t s, acs_status& st) {
    const int bx = p.tile.bx, by = p.tile.by;
    if (p.kind == ACS_KIND_STENCIL) {
        StarFix fx;
        star_fix(sc, fx);
        if (!fx.kind) return false;
        if (bx == 32 && by == 8) st = launch_star_t<32, 8, 4>(p, counter, sc, fx, s);
        else if (bx == 32 && by == 4) st = launch_star_t<32, 4, 8>(p, counter, sc, fx, s);
        else if (bx == 32 && by == 16) st = launch_star_t<32, 16, 2>(p, counter, sc, fx, s);
        else if (bx == 64 && by == 4) st = launch_star_t<64, 4, 4>(p, counter, sc, fx, s);
        else if (bx == 64 && by == 8) st = launch_star_t<64, 8, 2>(p, counter, sc, fx, s);
        else if (bx == 16 && by == 16) st = launch_star_t<16, 16, 4>(p, counter, sc, fx, s);
        else if (bx == 16 && by == 8) st = launch_star_t<16, 8, 8>(p, counter, sc, fx, s);
        else return false;
        return true;
    }
    RhsFix fx;
    RhsConst kc;
    rhs_fix(rk, fx, kc);
    if (!fx.ok) return false;
    if (bx != 16 || by != 16) return false;
    st = launch_rhs_t<16, 16>(p, counter, rk, kc, fx, s);
    return true;
}

}  // namespace acs
