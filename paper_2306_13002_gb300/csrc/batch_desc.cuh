// The unit table of a batch (layout in batch.cu) as its kernels read it.
#pragma once

#include "acs_internal.cuh"

namespace acs {

struct BatchDesc {
    const double* in0;  // U (RHS) or u (stencil)
    const double* in1;  // unused (RHS) or a (stencil)
    double* out;
    Geom g;
    int ntx, nty, nkc, kchunk;   // this grid's z-chunk (see batch_pack)
    int tma, pad;                // tma: this grid's planes are staged by its tensor map
};
static_assert(sizeof(BatchDesc) <= 112, "the static batch scratch is sized for 112-byte descriptors");

struct BatchHeader {
    unsigned long long counter;
    long long total;
    int n, kind, bx, by, kchunk, maps_off;   // maps_off: byte offset of the tensor maps (0: none)
    int plain, pad;                          // plain: too little work for the fixed-point RHS march
    long long pad1[2];
};
static_assert(sizeof(BatchHeader) == 64, "batch header is 64 bytes");

constexpr size_t kHeader = 64;

__host__ __device__ inline size_t desc_bytes(int n) { return ((size_t)n * sizeof(BatchDesc) + 15) & ~(size_t)15; }

__device__ __forceinline__ int find_item(const long long* __restrict__ prefix, int n, long long u) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (prefix[mid] <= u)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

struct BatchView {
    const BatchHeader* head;
    const BatchDesc* items;
    const long long* prefix;
};
__device__ __forceinline__ BatchView batch_view(const unsigned char* __restrict__ ws) {
    const BatchHeader* h = reinterpret_cast<const BatchHeader*>(ws);
    return BatchView{h, reinterpret_cast<const BatchDesc*>(ws + kHeader),
                     reinterpret_cast<const long long*>(ws + kHeader + desc_bytes(h->n))};
}

struct BatchUnit {
    int item, tx, ty, k0, k1;
};
// The block's next unit from the queue; false when it is empty. Holds two barriers.
__device__ __forceinline__ bool batch_next(const BatchView& b, unsigned long long* counter, long long* slot, bool leader,
                                           BatchUnit& out) {
    if (leader) *slot = (long long)atomicAdd(counter, 1ULL);
    __syncthreads();
    const long long u = *slot;
    __syncthreads();
    if (u >= b.head->total) return false;
    out.item = find_item(b.prefix, b.head->n, u);
    const BatchDesc& d = b.items[out.item];
    long long lu = u - b.prefix[out.item];
    out.tx = (int)(lu % d.ntx);
    lu /= d.ntx;
    out.ty = (int)(lu % d.nty);
    out.k0 = (int)(lu / d.nty) * d.kchunk;
    out.k1 = min(out.k0 + d.kchunk, d.g.nz);
    return true;
}

}  // namespace acs
