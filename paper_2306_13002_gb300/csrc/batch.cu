// Batched persistent launch: many grids of uneven sizes in one kernel launch.
//
// Every grid of the batch is cut into work units (BX x BY column tile, z-chunk of kchunk
// planes). A persistent grid of blocks (as many as fit on the GPU at once) pops units from
// an atomic counter in the caller's workspace and runs the same tile march as the
// single-grid saturated kernels (march.cuh), so the batch needs one launch however many
// grids it holds. Grids are ordered largest first, so the long units start early and the
// small ones fill the tail (longest-processing-time order); the last grids in that order
// take shorter z-chunks (guided self-scheduling), so the blocks run dry closer together.
//
// Workspace layout (device memory owned by the caller, 16-byte aligned):
//   [0, 64)                BatchHeader (the work counter, the unit total, the shape)
//   [64, 64 + n*D)         BatchDesc per grid, in processing order
//   [.., + 8 (n+1))        prefix sums of the grids' unit counts
//   [maps, + 128 n)        star-stencil batches with ACS_TILE_TMA all of whose grids TMA can copy: a
//                          tensor map per grid, in processing order, at the first 128-byte aligned
//                          address after the prefix sums (the header records the offset).
// acs_batch_prepare uploads everything but the counter; acs_batch_launch zeroes the
// counter with a memset on the stream and launches, so a prepared batch can be launched
// repeatedly and captured in a CUDA graph (a memset node plus a kernel node).
#include <algorithm>
#include <cstring>
#include <numeric>
#include <vector>

#include "batch_desc.cuh"
#include "march.cuh"

namespace acs {

namespace {

// The star stencil stages planes two steps ahead here (StarShape DEPTH 2): small grids give
// many edge tiles whose few active warps cannot hide one plane's copy latency per step.
constexpr int kBatchStarDepth = 2;

template <int BX, int BY, int KIND>
__global__ void __launch_bounds__(BX * BY, KIND == ACS_KIND_RHS ? RhsShape<BX, BY>::MINB
                                                                 : StarShape<BX, BY, kBatchStarDepth>::MINB)
    batch_kernel(const unsigned char* __restrict__ ws, unsigned long long* counter, RhsConst rk, StarCoef sc,
                 unsigned* tmo) {
    extern __shared__ __align__(128) double smem[];
    __shared__ long long s_unit;
    const BatchView b = batch_view(ws);
    const bool leader = threadIdx.x == 0 && threadIdx.y == 0;
    for (;;) {
        BatchUnit u;
        if (!batch_next(b, counter, &s_unit, leader, u)) break;
        const BatchDesc d = b.items[u.item];
        const int tx = u.tx, ty = u.ty, k0 = u.k0, k1 = u.k1;
        if (KIND == ACS_KIND_RHS) {
            if (rhs_isotropic(rk))   // uniform over the launch: the batch shares one set of constants
                rhs_march<BX, BY, false, true>(d.in0, d.out, d.g, rk, tx * BX, ty * BY, k0, k1, smem, nullptr, nullptr);
            else
                rhs_march<BX, BY, false, false>(d.in0, d.out, d.g, rk, tx * BX, ty * BY, k0, k1, smem, nullptr,
                                                nullptr);
        } else if (d.tma) {
            const CUtensorMap* map = reinterpret_cast<const CUtensorMap*>(ws + b.head->maps_off) + u.item;
            if (leader) tensormap_acquire(map);
            star_march<BX, BY, true, kBatchStarDepth>(d.in0, d.in1, d.out, d.g, sc, tx * BX, ty * BY, k0, k1, smem,
                                                       map, tmo);
        } else {
            star_march<BX, BY, false, kBatchStarDepth>(d.in0, d.in1, d.out, d.g, sc, tx * BX, ty * BY, k0, k1, smem,
                                                        nullptr, nullptr);
        }
    }
}

template <int BX, int BY, int KIND>
acs_status launch_batch_t(const BatchPlanHost& p, unsigned long long* counter, const RhsConst& rk,
                          const StarCoef& sc, cudaStream_t s) {
    const size_t smem = KIND == ACS_KIND_RHS ? RhsShape<BX, BY>::BYTES : StarShape<BX, BY, kBatchStarDepth>::BYTES;
    const void* fn = (const void*)batch_kernel<BX, BY, KIND>;
    acs_status st = ensure_smem(fn, smem);
    if (st != ACS_OK) return st;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batch_kernel<BX, BY, KIND>, BX * BY, smem) != cudaSuccess)
        return launch_status("cudaOccupancyMaxActiveBlocksPerMultiprocessor");
    if (per_sm < 1) return fail(ACS_ERR_UNSUPPORTED, "batch kernel %dx%d does not fit on an SM", BX, BY);
    long long blocks = (long long)per_sm * num_sms();
    if (blocks > p.total) blocks = p.total;
    unsigned* tmo = wait_timeout_counter();
    if (!tmo) return fail(ACS_ERR_CUDA, "cannot address the wait-timeout counter");
    batch_kernel<BX, BY, KIND><<<(unsigned)blocks, dim3(BX, BY, 1), smem, s>>>(p.ws, counter, rk, sc, tmo);
    return launch_status("batch_kernel");
}

// Blocks of the batch kernel resident on the whole device at once (0 if the query fails).
template <int BX, int BY, int KIND>
long long resident_t() {
    const size_t smem = KIND == ACS_KIND_RHS ? RhsShape<BX, BY>::BYTES : StarShape<BX, BY, kBatchStarDepth>::BYTES;
    if (ensure_smem((const void*)batch_kernel<BX, BY, KIND>, smem) != ACS_OK) return 0;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batch_kernel<BX, BY, KIND>, BX * BY, smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return (long long)per_sm * num_sms();
}

acs_status dispatch(const BatchPlanHost& p, unsigned long long* counter, const RhsConst& rk, const StarCoef& sc,
                    cudaStream_t s) {
    constexpr int K = ACS_KIND_STENCIL;
    const int bx = p.tile.bx, by = p.tile.by;
    if (p.kind == ACS_KIND_RHS) {   // always 16 x 16 columns (batch_prepare_host)
        if (bx == 16 && by == 16) return launch_batch_t<16, 16, ACS_KIND_RHS>(p, counter, rk, sc, s);
    } else {
        if (bx == 32 && by == 8) return launch_batch_t<32, 8, K>(p, counter, rk, sc, s);
        if (bx == 32 && by == 4) return launch_batch_t<32, 4, K>(p, counter, rk, sc, s);
        if (bx == 32 && by == 16) return launch_batch_t<32, 16, K>(p, counter, rk, sc, s);
        if (bx == 64 && by == 4) return launch_batch_t<64, 4, K>(p, counter, rk, sc, s);
        if (bx == 64 && by == 8) return launch_batch_t<64, 8, K>(p, counter, rk, sc, s);
        if (bx == 16 && by == 16) return launch_batch_t<16, 16, K>(p, counter, rk, sc, s);
        if (bx == 16 && by == 8) return launch_batch_t<16, 8, K>(p, counter, rk, sc, s);
    }
    return fail(ACS_ERR_UNSUPPORTED, "batch tile %dx%d is not built", bx, by);
}

// (Of the FP64 kernel, whose blocks per SM the chunk rules of batch_pack were measured with; which kernel runs
// is known at the launch only.)
long long resident_batch_blocks(int kind, const acs_tile& t) {
    constexpr int K = ACS_KIND_STENCIL;
    long long r = 0;
    const int bx = t.bx, by = t.by;
    if (kind == ACS_KIND_RHS) {
        if (bx == 16 && by == 16) r = resident_t<16, 16, ACS_KIND_RHS>();
    } else {
        if (bx == 32 && by == 8) r = resident_t<32, 8, K>();
        if (bx == 32 && by == 4) r = resident_t<32, 4, K>();
        if (bx == 32 && by == 16) r = resident_t<32, 16, K>();
        if (bx == 64 && by == 4) r = resident_t<64, 4, K>();
        if (bx == 64 && by == 8) r = resident_t<64, 8, K>();
        if (bx == 16 && by == 16) r = resident_t<16, 16, K>();
        if (bx == 16 && by == 8) r = resident_t<16, 8, K>();
    }
    // unknown (no device, or an unbuilt tile rejected later): the former estimate
    return r > 0 ? r : (long long)num_sms() * (kind == ACS_KIND_RHS ? 2 : 4);
}

}  // namespace

// Header, descriptors and prefix sums; the tensor maps follow at a 128-byte aligned address.
static size_t batch_table_bytes(int n) { return kHeader + desc_bytes(n) + sizeof(long long) * (size_t)(n + 1); }

size_t batch_ws_bytes(int n) { return n < 1 ? 0 : batch_table_bytes(n) + 128 + sizeof(CUtensorMap) * (size_t)n; }

// Host half of acs_batch_prepare: geometry already validated; builds the packed image.
// Clears ACS_TILE_TMA in the tile if not every grid can be staged so.
acs_status batch_pack(const acs_batch_item* items, const Geom* geo, int n, int kind, acs_tile& tile, bool plain,
                      uintptr_t ws_addr, std::vector<unsigned char>& image, long long& total) {
    std::vector<int> order(n);
    std::iota(order.begin(), order.end(), 0);
    auto points = [&](int q) { return (long long)geo[q].nx * geo[q].ny * geo[q].nz; };
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return points(x) > points(y); });
    // z-chunks of a batch with little work are shortened, so that the queue still holds a few units per
    // resident block (RHS: two; star stencil, whose blocks are smaller: one) but no shorter than what a
    // unit's start is worth. 8 RHS grids with sides of 16 to 96: chunks of 24 / 16 / 8 / 6 ran 404 / 297 /
    // 206 / 205 us, 16 grids 410 / 302 / 311 / 328 (by this rule and with the march as it is now 149 and 223); 8 star grids 32 / 16 / 8: 72 / 57 / 62 us.
    const long long resident = resident_batch_blocks(kind, tile);
    auto unit_count = [&](int q, int kc) {
        const Geom& g = geo[q];
        const long long ntx = (g.nx + tile.bx - 1) / tile.bx, nty = (g.ny + tile.by - 1) / tile.by;
        return ntx * nty * ((g.nz + kc - 1) / kc);
    };
    long long planes = 0;
    for (int q = 0; q < n; ++q) planes += unit_count(q, 1);
    const bool rhs = kind == ACS_KIND_RHS;
    // plain: the FP64 march, which starts at once
    const int kc = plain ? std::min(tile.kchunk, 16)
                         : (int)std::min<long long>(tile.kchunk, std::max<long long>(rhs ? 8 : 16, planes / (resident * (rhs ? 2 : 1))));
    // Guided z-chunks: the grids at the end of the order, whose units make up the last two
    // waves of the queue (two units per resident block), take z-chunks a quarter as long, so
    // the blocks run out of work closer together.
    const long long waves = 2LL * resident;
    const int tail_kchunk = std::min(kc, std::max(plain ? 1 : 4, kc / 4));
    // The fixed-point RHS march starts four planes early, so a grid's planes are split evenly instead of
    // leaving a last chunk of a few planes: 32 grids with sides of 16 to 96 611 -> 592 us, 20 of 60 to 96
    // 1283 -> 1234 us (with cut tiles still in the FP64 march, 398 and 881 us now), smaller batches and the
    // star stencil within 1 % either way.
    auto split = [&](int q, int c) {
        const int m = (geo[q].nz + c - 1) / c;
        return rhs && !plain ? (geo[q].nz + m - 1) / m : c;
    };
    std::vector<int> kchunk(n);
    for (int q = 0; q < n; ++q) kchunk[q] = split(q, kc);
    std::vector<long long> units(n);
    long long tail = 0;
    for (int r = n - 1; r >= 0; --r) {
        const int q = order[r];
        tail += unit_count(q, split(q, tail_kchunk));
        if (tail > waves) break;
        kchunk[q] = split(q, tail_kchunk);
    }
    for (int q = 0; q < n; ++q) units[q] = unit_count(q, kchunk[q]);
    image.assign(batch_ws_bytes(n), 0);
    BatchHeader h;
    std::memset(&h, 0, sizeof(h));
    h.n = n;
    h.kind = kind;
    h.bx = tile.bx;
    h.by = tile.by;
    h.kchunk = tile.kchunk;
    h.plain = plain;
    BatchDesc* d = reinterpret_cast<BatchDesc*>(image.data() + kHeader);
    long long* prefix = reinterpret_cast<long long*>(image.data() + kHeader + desc_bytes(n));
    // Tensor maps of a star-stencil batch staged by TMA: at the first 128-byte aligned device
    // address after the table.
    // All grids or none: blocks that run both stagings by turns crowd the instruction cache (64 grids, half
    // of them of even pitch: 293 us mixed, 257 us element-wise, 245 us if all can be copied).
    bool tma = (tile.flags & ACS_TILE_TMA) && kind == ACS_KIND_STENCIL;
    std::vector<CUtensorMap> map(tma ? n : 0);
    for (int q = 0; q < n && tma; ++q) {
        std::memset(&map[q], 0, sizeof(CUtensorMap));
        if (encode_plane_map(items[q].in0, geo[q], 1, tile.bx + 8, tile.by + 8, &map[q]) != ACS_OK) {
            tma = false;   // an odd pitch or a misaligned base
            set_error("%s", "");
        }
    }
    if (!tma) tile.flags &= ~ACS_TILE_TMA;
    if (tma) {
        const uintptr_t first = (ws_addr + batch_table_bytes(n) + 127) & ~(uintptr_t)127;
        h.maps_off = (int)(first - ws_addr);
    }
    long long acc = 0;
    for (int r = 0; r < n; ++r) {
        const int q = order[r];
        const Geom& g = geo[q];
        BatchDesc e;
        std::memset(&e, 0, sizeof(e));
        e.in0 = items[q].in0;
        e.in1 = items[q].in1;
        e.out = items[q].out;
        e.g = g;
        e.ntx = (g.nx + tile.bx - 1) / tile.bx;
        e.nty = (g.ny + tile.by - 1) / tile.by;
        e.nkc = (g.nz + kchunk[q] - 1) / kchunk[q];
        e.kchunk = kchunk[q];
        if (tma) {
            e.tma = 1;
            std::memcpy(image.data() + h.maps_off + (size_t)r * sizeof(CUtensorMap), &map[q], sizeof(CUtensorMap));
        }
        d[r] = e;
        prefix[r] = acc;
        acc += units[q];
    }
    prefix[n] = acc;
    h.total = acc;
    std::memcpy(image.data(), &h, sizeof(h));
    total = acc;
    return ACS_OK;
}

acs_status batch_prepare_host(const acs_batch_item* items, const Geom* geo, int n, int kind, const acs_tile& asked,
                              unsigned char* ws, size_t ws_bytes, cudaStream_t s, BatchPlanHost& plan) {
    // Columns of an RHS batch are 16 x 16, the shape the fixed-point march is built for (whether the
    // parameters suit it is known at the launch only).
    acs_tile tile = asked;
    bool plain = false;
    if (kind == ACS_KIND_RHS) {
        tile.bx = tile.by = 16;
        // Few planes per resident block: the FP64 march (4 grids with sides of 16 to 60, 3.2 planes: 87 us
        // against 95 to 105; 12 grids, 8.9 planes: 223 against 165).
        long long planes = 0;
        for (int q = 0; q < n; ++q) planes += (i64)((geo[q].nx + 15) / 16) * ((geo[q].ny + 15) / 16) * geo[q].nz;
        plain = planes < 5 * resident_batch_blocks(kind, tile);
    }
    std::vector<unsigned char> image;
    long long total = 0;
    acs_status st = batch_pack(items, geo, n, kind, tile, plain, (uintptr_t)ws, image, total);
    if (st != ACS_OK) return st;
    if (image.size() > ws_bytes) return fail(ACS_ERR_WORKSPACE, "workspace %zu bytes < %zu needed", ws_bytes, image.size());
    if (cudaMemcpyAsync(ws, image.data(), image.size(), cudaMemcpyHostToDevice, s) != cudaSuccess)
        return launch_status("cudaMemcpyAsync");
    if (cudaStreamSynchronize(s) != cudaSuccess) return launch_status("cudaStreamSynchronize");
    plan.ws = ws;
    plan.ws_bytes = ws_bytes;
    plan.kind = kind;
    plan.n = n;
    plan.tile = tile;
    plan.total = total;
    return ACS_OK;
}

acs_status batch_launch(const BatchPlanHost& p, const RhsConst& rk, const StarCoef& sc, cudaStream_t s) {
    unsigned long long* counter = reinterpret_cast<unsigned long long*>(p.ws);
    if (cudaMemsetAsync(counter, 0, sizeof(unsigned long long), s) != cudaSuccess) return launch_status("cudaMemsetAsync");
    acs_status st;
    if (batch_fixed_launch(p, counter, rk, sc, s, st)) return st;
    return dispatch(p, counter, rk, sc, s);
}

}  // namespace acs
