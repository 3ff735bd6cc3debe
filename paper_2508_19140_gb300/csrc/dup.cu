// K2 + K3 + K5: copies of each point per touched tile, and per-tile ranges.
//
// Second half of the split sort of Sec. 3.2 ("Tiled Rendering"): after the
// points are sorted by depth, each point (in depth order) writes one copy per
// tile its footprint touches, keyed by the global tile id. Writing the copies
// in depth order and sorting them stably by tile id afterwards yields the
// (tile, depth, point index) order. The copy offsets come from an exclusive
// scan of the per-point tile counts in depth order; the total D stays on the
// device and is clamped to the workspace capacity (overflow sets the
// capacity bit of the error word; no write ever leaves the buffers).
#include "rast_internal.cuh"

namespace rast {
namespace {

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t x) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

template <int NT>
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t x, uint32_t* s_warp, uint32_t& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int NW = NT / 32;
    const uint32_t inc = warp_incl_scan(x);
    if (lane == 31) s_warp[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = lane < NW ? s_warp[lane] : 0u;
        const uint32_t wi = warp_incl_scan(w);
        if (lane < NW) s_warp[lane] = wi - w;
        if (lane == NW - 1) s_warp[32] = wi;
    }
    __syncthreads();
    const uint32_t res = s_warp[warp] + inc - x;
    total = s_warp[32];
    __syncthreads();
    return res;
}

constexpr int kT = 256;
constexpr int kPer = kScanItems / kT;  // consecutive items per thread
static_assert(kPer % 4 == 0, "items move as 16-byte vectors");

// kPer consecutive u32 / uint2 items starting at s0 (vector loads and stores
// when the whole run is in range; `fill` past the end).
__device__ __forceinline__ void load_u32s(const uint32_t* __restrict__ p, int64_t s0, int64_t n, uint32_t v[kPer],
                                          uint32_t fill) {
    if (s0 + kPer <= n) {
#pragma unroll
        for (int j = 0; j < kPer; j += 4) {
            const uint4 q = *reinterpret_cast<const uint4*>(p + s0 + j);
            v[j] = q.x; v[j + 1] = q.y; v[j + 2] = q.z; v[j + 3] = q.w;
        }
    } else {
#pragma unroll
        for (int j = 0; j < kPer; ++j) v[j] = s0 + j < n ? p[s0 + j] : fill;
    }
}

__device__ __forceinline__ void store_rects(uint2* __restrict__ p, int64_t s0, int64_t n, const uint2 r[kPer]) {
    if (s0 + kPer <= n) {
#pragma unroll
        for (int j = 0; j < kPer; j += 2)
            *reinterpret_cast<uint4*>(p + s0 + j) = make_uint4(r[j].x, r[j].y, r[j + 1].x, r[j + 1].y);
    } else {
#pragma unroll
        for (int j = 0; j < kPer; ++j)
            if (s0 + j < n) p[s0 + j] = r[j];
    }
}

// Sorted-order rects of a block of kScanItems points (gathered once, kept for
// k_dup_write) and the block's copy count. If the depth sort failed (its
// look-back wait ran out: the error word is set before this kernel starts),
// every point counts as empty, so no copy is made from a partial order; an
// index outside [0, n) is treated the same way. P4: bilinear packed 4-byte
// rects (the gather's array is half the size). CARRIED: the depth sort has
// brought the rects along (rectS is complete unless it failed; k_dup_write
// sees the same bit), nothing is gathered: 32 M points 332 -> 34 us, 4 M 27 -> 8 us (the
// sort's passes then move the code in bits they carry anyway).
template <bool P4, bool CARRIED>
__global__ void __launch_bounds__(kT) k_dup_count(const uint32_t* __restrict__ sorted_pts,
                                                  const void* __restrict__ rect, void* __restrict__ rectS,
                                                  int64_t n, uint32_t* __restrict__ blk,
                                                  const WsHeader* __restrict__ hdr) {
    dependency_sync(sorted_pts, rectS, hdr);
    __shared__ uint32_t s_warp[33];
    const int64_t s0 = (int64_t)blockIdx.x * kScanItems + (int64_t)threadIdx.x * kPer;
    const bool failed = (hdr->error & kErrTimeout) != 0u;
    uint32_t gi[kPer];
    if (!CARRIED) load_u32s(sorted_pts, s0, n, gi, 0xffffffffu);
    uint32_t c = 0;
    if constexpr (CARRIED) {
        if (!failed) {
            if constexpr (P4) {
                uint32_t r[kPer];
                load_u32s(static_cast<const uint32_t*>(rectS), s0, n, r, kRect4Empty);
#pragma unroll
                for (int j = 0; j < kPer; ++j) c += rect4_count(r[j]);
            } else {
                const uint2* rs = static_cast<const uint2*>(rectS);
#pragma unroll
                for (int j = 0; j < kPer; j += 2) {
                    uint4 q = make_uint4(1u, 0u, 1u, 0u);
                    if (s0 + j + 2 <= n) q = *reinterpret_cast<const uint4*>(rs + s0 + j);
                    else if (s0 + j < n) q.x = rs[s0 + j].x, q.y = rs[s0 + j].y;
                    c += rect_count(make_uint2(q.x, q.y)) + rect_count(make_uint2(q.z, q.w));
                }
            }
        }
    } else if constexpr (P4) {
        const uint32_t* r4 = static_cast<const uint32_t*>(rect);
        uint32_t r[kPer];
#pragma unroll
        for (int j = 0; j < kPer; ++j) r[j] = (!failed && (int64_t)gi[j] < n) ? r4[gi[j]] : kRect4Empty;
#pragma unroll
        for (int j = 0; j < kPer; ++j) c += rect4_count(r[j]);
        uint32_t* out = static_cast<uint32_t*>(rectS);
        if (s0 + kPer <= n) {
#pragma unroll
            for (int j = 0; j < kPer; j += 4)
                *reinterpret_cast<uint4*>(out + s0 + j) = make_uint4(r[j], r[j + 1], r[j + 2], r[j + 3]);
        } else {
#pragma unroll
            for (int j = 0; j < kPer; ++j)
                if (s0 + j < n) out[s0 + j] = r[j];
        }
    } else {
        const uint2* r8 = static_cast<const uint2*>(rect);
        uint2 r[kPer];
#pragma unroll
        for (int j = 0; j < kPer; ++j) r[j] = (!failed && (int64_t)gi[j] < n) ? r8[gi[j]] : make_uint2(1u, 0u);
#pragma unroll
        for (int j = 0; j < kPer; ++j) c += rect_count(r[j]);
        store_rects(static_cast<uint2*>(rectS), s0, n, r);
    }
    uint32_t tot;
    block_excl_scan<kT>(c, s_warp, tot);
    if (threadIdx.x == 0) blk[blockIdx.x] = tot;
}

// Per-point copy counts, kPer consecutive points from s0: the count array
// (Gaussian), or the packed bilinear rects (P4; an empty rect counts 0).
template <bool P4>
__device__ __forceinline__ void load_counts(const uint32_t* __restrict__ p, int64_t s0, int64_t n, uint32_t v[kPer]) {
    load_u32s(p, s0, n, v, P4 ? kRect4Empty : 0u);
    if constexpr (P4) {
#pragma unroll
        for (int j = 0; j < kPer; ++j) v[j] = rect4_count(v[j]);
    }
}

// The untiled baseline's copies a block and, with them scanned, a point's first copy.
__global__ void __launch_bounds__(kT) k_count_blocks(const uint32_t* __restrict__ rect4, int64_t n,
                                                     uint32_t* __restrict__ blk) {
    __shared__ uint32_t s_warp[33];
    const int64_t s0 = (int64_t)blockIdx.x * kScanItems + (int64_t)threadIdx.x * kPer;
    uint32_t v[kPer];
    load_counts<true>(rect4, s0, n, v);
    uint32_t sum = 0;
#pragma unroll
    for (int j = 0; j < kPer; ++j) sum += v[j];
    uint32_t tot;
    block_excl_scan<kT>(sum, s_warp, tot);
    if (threadIdx.x == 0) blk[blockIdx.x] = tot;
}

__global__ void __launch_bounds__(1024) k_scan_blocks(uint32_t* __restrict__ blk, int64_t nb,
                                                      WsHeader* hdr, int64_t cap) {
    dependency_sync(blk);
    __shared__ uint32_t s_warp[33];
    __shared__ unsigned long long s_wtot[32];
    const int64_t per = (nb + 1023) / 1024;
    const int64_t lo = threadIdx.x * per;
    const int64_t hi = lo + per < nb ? lo + per : nb;
    unsigned long long s = 0;
    for (int64_t t = lo; t < hi; ++t) s += blk[t];
    // 64-bit total: warp shuffle reduction, then one value per warp
    unsigned long long ws = s;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ws += __shfl_xor_sync(0xffffffffu, ws, o);
    if ((threadIdx.x & 31) == 0) s_wtot[threadIdx.x >> 5] = ws;
    uint32_t tot;
    uint32_t run = block_excl_scan<1024>((uint32_t)s, s_warp, tot);  // exact whenever total <= cap
    for (int64_t t = lo; t < hi; ++t) {
        const uint32_t c = blk[t];
        blk[t] = run;
        run += c;
    }
    if (threadIdx.x == 0) {
        unsigned long long total = 0;
        for (int w = 0; w < 32; ++w) total += s_wtot[w];
        const bool over = total > (unsigned long long)cap;
        hdr->n_copies_raw = total > 0xffffffffull ? 0xffffffffu : (uint32_t)total;
        hdr->n_copies = over ? 0u : (uint32_t)total;
        if (over) atomicOr(&hdr->error, kErrCapacity);
    }
}

// Writes the copies: key = global tile id, value = global point index.
// Copies of a block of kScanItems depth-ordered points: 2 * kT threads with
// half as many items each as the counting kernels (the per-item copy loops
// are the long part here, so more threads beat more items per thread).
constexpr int kTW = 2 * kT;
constexpr int kPerW = kScanItems / kTW;
static_assert(kPerW == 4, "the packed-rect path loads four rects as one 16-byte vector");
// Copies a block stages in shared memory before writing them out in coalesced
// runs (a block with more writes them directly): four a point for Gaussians
// (about two on average), one and a half for bilinear points (1.1 to 1.3), whose
// one, two or four copies are written without loops: 4 M points 38 -> 25 us, 32 M
// 203 -> 145 us, 62 M in 8 images 483 -> 381 us (staging alone, behind the loops,
// was 34, 219 and 512 us, direct stores without loops 39, 209 and 439 us).
template <bool P4>
constexpr int stage_cap() { return P4 ? 3 * kScanItems / 2 : 4 * kScanItems; }
template <bool P4>
constexpr size_t dup_write_smem() { return sizeof(uint32_t) * 2 * stage_cap<P4>(); }

template <bool P4>
__global__ void __launch_bounds__(kTW) k_dup_write(const ViewTable vt, const uint32_t* __restrict__ sorted_pts,
                                                   const void* __restrict__ rectS, int64_t n,
                                                   const uint32_t* __restrict__ blk,
                                                   uint32_t* __restrict__ keys, uint32_t* __restrict__ vals,
                                                   int64_t cap, const WsHeader* __restrict__ hdr) {
    dependency_sync(sorted_pts, rectS, blk, hdr);
    __shared__ uint32_t s_warp[33];
    if (hdr->error & kErrTimeout) return;  // set by an earlier kernel: no copy is made from a partial order
    extern __shared__ uint32_t s_copy[];  // [kStageCap] tile ids, then [kStageCap] point indices
    const int64_t s0 = (int64_t)blockIdx.x * kScanItems + (int64_t)threadIdx.x * kPerW;
    uint2 r[kPerW];
    uint32_t gi[kPerW];
    if (s0 + kPerW <= n) {
        if constexpr (P4) {
            const uint4 q = *reinterpret_cast<const uint4*>(static_cast<const uint32_t*>(rectS) + s0);
            r[0] = rect4_unpack(q.x); r[1] = rect4_unpack(q.y); r[2] = rect4_unpack(q.z); r[3] = rect4_unpack(q.w);
        } else {
            const uint2* rs = static_cast<const uint2*>(rectS);
#pragma unroll
            for (int j = 0; j < kPerW; j += 2) {
                const uint4 q = *reinterpret_cast<const uint4*>(rs + s0 + j);
                r[j] = make_uint2(q.x, q.y);
                r[j + 1] = make_uint2(q.z, q.w);
            }
        }
#pragma unroll
        for (int j = 0; j < kPerW; j += 4) {
            const uint4 q = *reinterpret_cast<const uint4*>(sorted_pts + s0 + j);
            gi[j] = q.x; gi[j + 1] = q.y; gi[j + 2] = q.z; gi[j + 3] = q.w;
        }
    } else {
#pragma unroll
        for (int j = 0; j < kPerW; ++j) {
            const bool ok = s0 + j < n;
            if constexpr (P4) r[j] = ok ? rect4_unpack(static_cast<const uint32_t*>(rectS)[s0 + j]) : make_uint2(1u, 0u);
            else r[j] = ok ? static_cast<const uint2*>(rectS)[s0 + j] : make_uint2(1u, 0u);
            gi[j] = ok ? sorted_pts[s0 + j] : 0u;
        }
    }
    uint32_t c[kPerW], sum = 0;
#pragma unroll
    for (int j = 0; j < kPerW; ++j) {
        c[j] = rect_count(r[j]);
        sum += c[j];
    }
    uint32_t tot;
    const uint32_t ex = block_excl_scan<kTW>(sum, s_warp, tot);
    const uint32_t blk0 = blk[blockIdx.x];
    // The block's copies fill one contiguous range of the output: staged in
    // shared memory, they leave in coalesced runs instead of one scattered
    // 4-byte store per copy and array.
    constexpr int kStageCap = stage_cap<P4>();
    const bool staged = tot <= (uint32_t)kStageCap;
    uint32_t o = staged ? ex : blk0 + ex;
#pragma unroll
    for (int j = 0; j < kPerW; ++j) {
        if (c[j] == 0) continue;
        const ViewDev& V = vt.v[view_of_point(vt, gi[j])];
        const int tx0 = r[j].x & 0xffff, ty0 = r[j].x >> 16, tx1 = r[j].y & 0xffff, ty1 = r[j].y >> 16;
        if constexpr (P4) {
            // at most two by two tiles: no loops
            auto put = [&](uint32_t at, uint32_t tile, uint32_t g) {
                if (staged) {
                    s_copy[at] = tile;
                    s_copy[kStageCap + at] = g;
                } else if ((int64_t)at < cap) {
                    keys[at] = tile;
                    vals[at] = g;
                }
            };
            const uint32_t tiles_x = (uint32_t)V.tiles_x, w = (uint32_t)(tx1 - tx0);
            const uint32_t first = (uint32_t)V.tile_off + (uint32_t)ty0 * tiles_x + (uint32_t)tx0;
            put(o, first, gi[j]);
            if (w) put(o + 1, first + 1, gi[j]);
            if (ty1 != ty0) {
                put(o + 1 + w, first + tiles_x, gi[j]);
                if (w) put(o + 3, first + tiles_x + 1, gi[j]);
            }
            o += c[j];
        } else {
            for (int ty = ty0; ty <= ty1; ++ty) {
                const uint32_t row = (uint32_t)(V.tile_off + (int64_t)ty * V.tiles_x);
                for (int tx = tx0; tx <= tx1; ++tx) {
                    if (staged) {
                        s_copy[o] = row + (uint32_t)tx;
                        s_copy[kStageCap + o] = gi[j];
                    } else if ((int64_t)o < cap) {
                        keys[o] = row + (uint32_t)tx;
                        vals[o] = gi[j];
                    }
                    ++o;
                }
            }
        }
    }
    if (!staged) return;  // block-uniform
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < tot; i += kTW) {
        const int64_t g = (int64_t)blk0 + i;
        if (g < cap) {
            keys[g] = s_copy[i];
            vals[g] = s_copy[kStageCap + i];
        }
    }
}

__global__ void __launch_bounds__(kT) k_scan_apply(const uint32_t* __restrict__ rect4, int64_t n,
                                                   const uint32_t* __restrict__ blk,
                                                   uint32_t* __restrict__ base) {
    __shared__ uint32_t s_warp[33];
    const int64_t s0 = (int64_t)blockIdx.x * kScanItems + (int64_t)threadIdx.x * kPer;
    uint32_t v[kPer];
    load_counts<true>(rect4, s0, n, v);
    uint32_t sum = 0;
#pragma unroll
    for (int j = 0; j < kPer; ++j) sum += v[j];
    uint32_t tot;
    uint32_t o = blk[blockIdx.x] + block_excl_scan<kT>(sum, s_warp, tot);
    uint32_t r[kPer];
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        r[j] = o;
        o += v[j];
    }
    if (s0 + kPer <= n) {
#pragma unroll
        for (int j = 0; j < kPer; j += 4)
            *reinterpret_cast<uint4*>(base + s0 + j) = make_uint4(r[j], r[j + 1], r[j + 2], r[j + 3]);
    } else {
#pragma unroll
        for (int j = 0; j < kPer; ++j)
            if (s0 + j < n) base[s0 + j] = r[j];
    }
}

__global__ void k_bwd_init(WsHeader* hdr) {
    hdr->needed_bwd = 0ull;
    hdr->slots = 0u;
}

// First partial-gradient slot of every point (backward): a block takes one run
// of slots for its points with a single addition, in whatever order the blocks
// come (which slot a row lies in has no effect on any value), where a count, a
// scan and a second pass over the points gave them in point order: 4 M points
// 26.2 -> 12.3 us, 16 M 55 -> 29 us, 62 M 159 -> 84 us. Bilinear points with one copy need none (their
// row is indexed by point), so the rows in use lie closer together (the blend
// that writes them 234 -> 220 us, the reduction that reads them 66.5 -> 60.8 us).
template <bool P4>
__global__ void __launch_bounds__(kT) k_point_slots(const uint32_t* __restrict__ cnt, int64_t n, WsHeader* hdr,
                                                    uint32_t* __restrict__ base) {
    dependency_sync(cnt);
    __shared__ uint32_t s_warp[33];
    __shared__ uint32_t s_first;
    const int64_t s0 = (int64_t)blockIdx.x * kScanItems + (int64_t)threadIdx.x * kPer;
    uint32_t v[kPer], sum = 0;
    load_counts<P4>(cnt, s0, n, v);
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        if (P4 && v[j] == 1u) v[j] = 0u;
        sum += v[j];
    }
    uint32_t tot;
    uint32_t o = block_excl_scan<kT>(sum, s_warp, tot);
    if (threadIdx.x == 0) s_first = tot ? atomicAdd(&hdr->slots, tot) : 0u;
    __syncthreads();
    o += s_first;
    uint32_t r[kPer];
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        r[j] = o;
        o += v[j];
    }
    if (s0 + kPer <= n) {
#pragma unroll
        for (int j = 0; j < kPer; j += 4)
            *reinterpret_cast<uint4*>(base + s0 + j) = make_uint4(r[j], r[j + 1], r[j + 2], r[j + 3]);
    } else {
#pragma unroll
        for (int j = 0; j < kPer; ++j)
            if (s0 + j < n) base[s0 + j] = r[j];
    }
}

// Tiles by list length, for the blends' heaviest-first order: bucket of
// floor(log2(length)) + 1, 0 for an empty list.
__device__ __forceinline__ int len_bucket(uint32_t len) { return len ? 32 - __clz(len) : 0; }

// Tile ranges found tile by tile: one thread a tile looks for its first copy
// among the sorted keys, WAYS - 1 probes a step, and neighbours share their ends
// (the last thread of a block only serves its neighbour). It touches a few dozen
// keys a tile instead of all of them, and needs no cleared ranges. The tiles'
// buckets (see k_tile_scatter) are counted on the way. If the tile sort's
// look-back wait ran out, the keys are a partial order: every range is empty, so
// the blends read no copy of it.
template <int WAYS>
__global__ void __launch_bounds__(kT) k_ranges_search(const uint32_t* __restrict__ keys,
                                                      const WsHeader* __restrict__ hdr, int64_t tiles,
                                                      uint2* __restrict__ ranges, uint32_t* __restrict__ buckets) {
    dependency_sync(keys, hdr);
    __shared__ uint32_t s_first[kT];
    __shared__ uint32_t s_cnt[33];
    if (threadIdx.x < 33) s_cnt[threadIdx.x] = 0;
    const uint32_t D = (hdr->error & kErrTimeout) ? 0u : hdr->n_copies;
    const int64_t t = (int64_t)blockIdx.x * (kT - 1) + threadIdx.x;
    // first position whose key is >= t: in [lo, hi]
    uint32_t lo = 0, hi = D;
    while (lo < hi) {
        uint32_t m[WAYS - 1], k[WAYS - 1];  // probes, ascending, in [lo, hi)
#pragma unroll
        for (int j = 0; j < WAYS - 1; ++j) m[j] = lo + (uint32_t)((uint64_t)(hi - lo) * (j + 1) / WAYS);
#pragma unroll
        for (int j = 0; j < WAYS - 1; ++j) k[j] = keys[m[j]];
        uint32_t nlo = lo, nhi = hi;
#pragma unroll
        for (int j = 0; j < WAYS - 1; ++j) {
            if ((int64_t)k[j] < t) nlo = m[j] + 1;
            else nhi = min(nhi, m[j]);
        }
        lo = nlo;
        hi = nhi;
    }
    s_first[threadIdx.x] = lo;
    __syncthreads();
    if (threadIdx.x < kT - 1 && t < tiles) {
        const uint2 r = make_uint2(lo, s_first[threadIdx.x + 1]);
        ranges[t] = r;
        atomicAdd(&s_cnt[len_bucket(r.y - r.x)], 1u);
    }
    __syncthreads();
    if (threadIdx.x < 33 && s_cnt[threadIdx.x]) atomicAdd(&buckets[threadIdx.x], s_cnt[threadIdx.x]);
}

__global__ void __launch_bounds__(kT) k_tile_buckets(const uint2* __restrict__ ranges, int64_t tiles,
                                                     uint32_t* __restrict__ buckets) {
    __shared__ uint32_t s_cnt[33];
    if (threadIdx.x < 33) s_cnt[threadIdx.x] = 0;
    __syncthreads();
    for (int64_t t = (int64_t)blockIdx.x * kT + threadIdx.x; t < tiles; t += (int64_t)gridDim.x * kT)
        atomicAdd(&s_cnt[len_bucket(ranges[t].y - ranges[t].x)], 1u);
    __syncthreads();
    if (threadIdx.x < 33 && s_cnt[threadIdx.x]) atomicAdd(&buckets[threadIdx.x], s_cnt[threadIdx.x]);
}

// Tile ranges from one read of the sorted tile keys, for lists too short for a
// search per tile (the untiled baselines: a tile a pixel). If the tile sort's look-back wait ran
// out, the keys are a partial order: the ranges are left empty (cleared before
// this kernel), so the blends read no copy of it.
__global__ void __launch_bounds__(kT) k_ranges(const uint32_t* __restrict__ keys,
                                               const WsHeader* __restrict__ hdr,
                                               uint2* __restrict__ ranges) {
    if (hdr->error & kErrTimeout) return;
    const int64_t D = hdr->n_copies;
    // Four consecutive keys per thread (one 16-byte load) plus the keys just
    // before and after them; a range starts or ends where neighbours differ.
    for (int64_t p0 = ((int64_t)blockIdx.x * kT + threadIdx.x) * 4; p0 < D; p0 += (int64_t)gridDim.x * kT * 4) {
        uint32_t k[6];  // keys p0-1 .. p0+4 (sentinels outside [0, D))
        k[0] = p0 > 0 ? keys[p0 - 1] : 0xffffffffu;
        if (p0 + 4 <= D) {
            const uint4 q = *reinterpret_cast<const uint4*>(keys + p0);
            k[1] = q.x; k[2] = q.y; k[3] = q.z; k[4] = q.w;
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) k[1 + j] = p0 + j < D ? keys[p0 + j] : 0xffffffffu;
        }
        k[5] = p0 + 4 < D ? keys[p0 + 4] : 0xffffffffu;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int64_t p = p0 + j;
            if (p >= D) break;
            const uint32_t t = k[1 + j];
            if (p == 0 || k[j] != t) ranges[t].x = (uint32_t)p;
            if (p + 1 == D || k[2 + j] != t) ranges[t].y = (uint32_t)(p + 1);
        }
    }
}

// ---- untiled baseline with one 64-bit-key sort (the arrangement Sec. 3.2
// "Tiled Rendering" starts from) ------------------------------------------
// Copies in POINT order, one per in-image pixel of the point's 2x2 box (the
// projection's rect with one-pixel tiles): the low key word is the point's
// depth key, the high word its pixel id; the point index goes with them. A
// stable LSD radix sort over the 64-bit key [pixel | depth] then yields the
// per-pixel lists in (depth, point index) order, ties falling back to the
// point order the copies were written in.
__global__ void __launch_bounds__(kT) k_untiled_copies(const ViewTable vt, const uint32_t* __restrict__ rect4,
                                                       const uint32_t* __restrict__ dkey,
                                                       const uint32_t* __restrict__ base,
                                                       uint32_t* __restrict__ key_lo, uint32_t* __restrict__ key_hi,
                                                       uint32_t* __restrict__ pt, int64_t cap) {
    const int64_t gi = (int64_t)blockIdx.x * kT + threadIdx.x;
    if (gi >= vt.n_total) return;
    const uint2 r = rect4_unpack(rect4[gi]);  // bilinear only: packed rects
    if (rect_count(r) == 0) return;
    const ViewDev& V = vt.v[view_of_point(vt, gi)];
    const int x0 = r.x & 0xffff, y0 = r.x >> 16, x1 = r.y & 0xffff, y1 = r.y >> 16;
    const uint32_t k = dkey[gi];
    int64_t o = base[gi];
    for (int y = y0; y <= y1; ++y)
        for (int x = x0; x <= x1; ++x, ++o) {
            if (o >= cap) return;
            key_lo[o] = k;
            key_hi[o] = (uint32_t)(V.tile_off + (int64_t)y * V.tiles_x + x);
            pt[o] = (uint32_t)gi;
        }
}

// Between the low-word and high-word digit passes of the 64-bit sort: the
// high key word and the point index of every copy, fetched by the copy id the
// low-word passes carried (a copy id outside [0, D) yields an empty key past
// every pixel; after a timed-out pass the count is treated as zero).
__global__ void __launch_bounds__(kT) k_gather_hi(const uint32_t* __restrict__ cid,
                                                  const uint32_t* __restrict__ key_hi,
                                                  const uint32_t* __restrict__ pt,
                                                  const WsHeader* __restrict__ hdr,
                                                  uint32_t* __restrict__ kout, uint32_t* __restrict__ vout) {
    if (hdr->error & kErrTimeout) return;
    const int64_t D = hdr->n_copies;
    for (int64_t j = (int64_t)blockIdx.x * kT + threadIdx.x; j < D; j += (int64_t)gridDim.x * kT) {
        const uint32_t c = cid[j];
        const bool ok = (int64_t)c < D;
        kout[j] = ok ? key_hi[c] : 0xffffffffu;
        vout[j] = ok ? pt[c] : 0u;
    }
}

}  // namespace

cudaError_t launch_untiled_copies(const ViewTable& vt, const Bufs& b, const uint32_t* dkey, uint32_t* key_lo,
                                  uint32_t* key_hi, uint32_t* pt, cudaStream_t s) {
    const int64_t n = vt.n_total;
    const int64_t nb = (n + kScanItems - 1) / kScanItems;
    if (nb == 0) return cudaSuccess;
    {
        ProfScope ps("dup.count", s);
        k_count_blocks<<<(unsigned)nb, kT, 0, s>>>(b.rect4, n, b.blk);
    }
    {
        ProfScope ps("dup.scan", s);
        k_scan_blocks<<<1, 1024, 0, s>>>(b.blk, nb, b.hdr, b.copy_cap);
        k_scan_apply<<<(unsigned)nb, kT, 0, s>>>(b.rect4, n, b.blk, b.base);
    }
    {
        ProfScope ps("dup.write", s);
        k_untiled_copies<<<(unsigned)((n + kT - 1) / kT), kT, 0, s>>>(vt, b.rect4, dkey, b.base, key_lo, key_hi, pt,
                                                                      b.copy_cap);
    }
    return cudaGetLastError();
}

cudaError_t launch_gather_hi(const Bufs& b, const uint32_t* cid, const uint32_t* key_hi, const uint32_t* pt,
                             uint32_t* kout, uint32_t* vout, cudaStream_t s) {
    if (b.copy_cap == 0) return cudaSuccess;
    int64_t g = (b.copy_cap + kT - 1) / kT;
    const int64_t gmax = (int64_t)device_sm_count() * 16;
    if (g > gmax) g = gmax;
    ProfScope ps("sort64.gather_hi", s);
    k_gather_hi<<<(unsigned)g, kT, 0, s>>>(cid, key_hi, pt, b.hdr, kout, vout);
    return cudaGetLastError();
}

cudaError_t launch_duplicate(const ViewTable& vt, const Bufs& b, const uint32_t* sorted_pts, bool carried,
                             cudaStream_t s) {
    const int64_t n = vt.n_total;
    const int64_t nb = (n + kScanItems - 1) / kScanItems;
    if (nb == 0) return cudaSuccess;  // the header was zeroed at the start of the pass
    {
        ProfScope ps(carried ? "dup.count" : "dup.gather", s);
        auto kern = vt.mode == 0 ? (carried ? k_dup_count<true, true> : k_dup_count<true, false>)
                                 : (carried ? k_dup_count<false, true> : k_dup_count<false, false>);
        const void* in = vt.mode == 0 ? (const void*)b.rect4 : (const void*)b.rect;
        void* out = vt.mode == 0 ? (void*)b.rect4S : (void*)b.rectS;
        const cudaError_t e = launch_dependent(kern, (unsigned)nb, kT, 0, s, sorted_pts, in, out, n, b.blk, b.hdr);
        if (e != cudaSuccess) return e;
    }
    {
        ProfScope ps("dup.scan", s);
        const cudaError_t e = launch_dependent(k_scan_blocks, 1, 1024, 0, s, b.blk, nb, b.hdr, b.copy_cap);
        if (e != cudaSuccess) return e;
    }
    {
        static PerDevice attr;
        const cudaError_t e = per_device(attr, nullptr, [](int, int*) {
            return cudaFuncSetAttribute(k_dup_write<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)dup_write_smem<false>());
        });
        if (e != cudaSuccess) return e;
        ProfScope ps("dup.write", s);
        if (vt.mode == 0)
            return launch_dependent(k_dup_write<true>, (unsigned)nb, kTW, dup_write_smem<true>(), s, vt, sorted_pts,
                                    b.rect4S, n, b.blk,
                                    b.keyC[0], b.valC[0], b.copy_cap, b.hdr);
        return launch_dependent(k_dup_write<false>, (unsigned)nb, kTW, dup_write_smem<false>(), s, vt, sorted_pts,
                                b.rectS, n,
                                b.blk, b.keyC[0], b.valC[0], b.copy_cap, b.hdr);
    }
}

cudaError_t launch_ranges(const ViewTable& vt, const Bufs& b, const uint32_t* sorted_tiles, int64_t expect,
                          cudaStream_t s) {
    // A search reads about 40 keys a tile, spread out; a scan clears the ranges
    // and reads every key, in order, and the tiles' buckets are counted by a
    // third kernel. The search where one round of blocks covers the grid (it is
    // then a matter of latency: 64 tiles 6.6 us against 2 + 6.5 + 6.6) and where
    // lists are long (16640 tiles, 5.3 M copies 9.1 against 2 + 10.2 + 5.7 us;
    // 8160 tiles, 37 M copies 12.3 against 2 + 39.3 + 6.0; 143 k tiles, 77 M
    // copies 24.7 against 3 + 69.9 + 6.3); the scan for large, sparsely covered
    // images and for the untiled baselines (a tile a pixel). Eight ways on
    // smaller grids, whose time is the steps' latency, four on larger ones,
    // whose time is the probes.
    const int64_t tiles = vt.tiles_total;
    uint32_t* const buckets = b.order + tiles;
    if (tiles <= 16384 || 32 * tiles <= expect) {
        if (tiles == 0) return cudaSuccess;
        ProfScope ps("ranges", s);
        return launch_dependent(tiles <= 32768 ? k_ranges_search<8> : k_ranges_search<4>,
                                (unsigned)((tiles + kT - 2) / (kT - 1)), kT, 0, s, sorted_tiles, b.hdr, tiles, b.ranges,
                                buckets);
    }
    cudaError_t e = cudaMemsetAsync(b.ranges, 0, sizeof(uint2) * tiles, s);
    if (e != cudaSuccess) return e;
    if (b.copy_cap > 0) {
        int64_t g = (b.copy_cap + kT - 1) / kT;
        const int64_t gmax = (int64_t)device_sm_count() * 8;
        if (g > gmax) g = gmax;
        ProfScope ps("ranges.scan", s);
        k_ranges<<<(unsigned)g, kT, 0, s>>>(sorted_tiles, b.hdr, b.ranges);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    if (vt.tile == 1) return cudaSuccess;  // the untiled blends take the pixels in order
    const int64_t want = (tiles + kT - 1) / kT;
    ProfScope ps("tile_order.count", s);
    k_tile_buckets<<<(unsigned)(want < 1024 ? want : 1024), kT, 0, s>>>(b.ranges, tiles, buckets);
    return cudaGetLastError();
}

cudaError_t launch_point_slots(const ViewTable& vt, const Bufs& b, cudaStream_t s) {
    {
        ProfScope ps("bwd_init", s);
        k_bwd_init<<<1, 1, 0, s>>>(b.hdr);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    const int64_t n = vt.n_total;
    const int64_t nb = (n + kScanItems - 1) / kScanItems;
    if (nb == 0) return cudaSuccess;
    ProfScope ps("point_slots", s);
    return launch_dependent(vt.mode == 0 ? k_point_slots<true> : k_point_slots<false>, (unsigned)nb, kT, 0, s,
                            vt.mode == 0 ? b.rect4 : b.cnt, n, b.hdr, b.base);
}

}  // namespace rast
