// K6: front-to-back blend per tile (Eq. 1), one CTA per tile (16x16 or 8x8
// pixels), one thread per pixel.
//
// F = sum_i T_i a_i f_i, T_i = prod_{j<i} (1 - a_j), over the pixel's covering
// fragments in (depth, point index) order, stopping before the first fragment
// that would take T below t_min. Each CTA walks its tile's sorted list in
// batches of D records (the blend depth: tile^2 x RPT): every thread gathers
// its RPT records with 16-byte cp.async copies into a shared-memory ring (two
// or three batches deep, padded stride against bank conflicts), and each pixel
// composites the records of the batch that cover it, in list order. The copies
// of the next batches (and the point indices of the ones after) are in flight
// while a batch is composited, so the gather latency overlaps the compositing
// instead of adding to every batch of the tile's serial chain.
//
// Bilinear splats touch at most 4 pixels, so testing every record against
// every pixel would make the kernel ALU-bound. Instead the record's thread
// computes its four slot alphas once (the oracle's FP32 operations) and sets
// one bit per covered pixel in a per-pixel D-bit mask (shared-memory atomicOr,
// order-free and therefore deterministic); each pixel visits only its set bits
// in ascending order = list order.
//
// Gaussian splats cover many pixels; there each warp owns an 8x4 sub-tile,
// ballots the records whose pixel box meets its two 4x4 halves, and each half
// composites its own, 16 lanes in lockstep; the records are staged once for the
// tile's warps, which run through them without CTA barriers.
//
// Tiles are visited heaviest first (k_tile_scatter): the
// blend's duration is bounded below by its longest tile list, so that list
// must start at once. The CTA stops reading as soon as every in-image pixel
// has terminated (__syncthreads_count), which is where early termination saves
// HBM traffic. Saved for the backward pass: T_final and the 1-based list
// position of the last blended fragment per pixel. The per-tile count of
// records the method had to read (every record if some pixel never terminated,
// else up to the last terminating fragment) is summed into the workspace
// header. The untiled baseline's per-pixel kernel (k_blend_fwd_pixel) is at
// the end of the file.
#include "blend_common.cuh"

namespace rast {
namespace {

// Tiles in descending order of list length, bucketed by floor(log2(len)): the
// ranges kernel has counted the tiles of every bucket; k_tile_scatter turns the
// 33 counts into bucket starts (heaviest bucket first) and places each tile at
// its bucket's next free position. The order inside a bucket depends on timing
// and only affects scheduling: every tile is blended the same way.
__device__ __forceinline__ int len_bucket(uint2 r) {
    const uint32_t len = r.y - r.x;
    return len ? 32 - __clz(len) : 0;  // 0..32
}

__global__ void __launch_bounds__(256) k_tile_scatter(const uint2* __restrict__ ranges, int64_t P,
                                                      const uint32_t* __restrict__ counts,
                                                      uint32_t* __restrict__ cursor, uint32_t* __restrict__ order) {
    dependency_sync(ranges, counts);
    __shared__ uint32_t s_start[33];  // global start of each bucket
    __shared__ uint32_t s_cnt[33];    // this block's tiles per bucket, then its next free slot
    if (threadIdx.x == 0) {
        uint32_t run = 0;
        for (int bk = 32; bk >= 0; --bk) {
            s_start[bk] = run;
            run += counts[bk];
        }
    }
    if (threadIdx.x < 33) s_cnt[threadIdx.x] = 0;
    __syncthreads();
    // This block's contiguous chunk of tiles: count, reserve one range per
    // bucket with a single global atomic, then place.
    const int64_t chunk = (P + gridDim.x - 1) / gridDim.x;
    const int64_t lo = (int64_t)blockIdx.x * chunk, hi = lo + chunk < P ? lo + chunk : P;
    for (int64_t t = lo + threadIdx.x; t < hi; t += blockDim.x) atomicAdd(&s_cnt[len_bucket(ranges[t])], 1u);
    __syncthreads();
    if (threadIdx.x < 33) {
        const uint32_t c = s_cnt[threadIdx.x];
        s_cnt[threadIdx.x] = s_start[threadIdx.x] + (c ? atomicAdd(&cursor[threadIdx.x], c) : 0u);
    }
    __syncthreads();
    for (int64_t t = lo + threadIdx.x; t < hi; t += blockDim.x)
        order[atomicAdd(&s_cnt[len_bucket(ranges[t])], 1u)] = (uint32_t)t;
}

// cp.async ring depth (batches in flight per CTA): three batches for 16x16
// tiles with one record per thread; two otherwise (deeper batches hide more
// latency each, and 8x8 tiles gain more from the extra CTAs per SM that a
// smaller ring leaves room for).
template <int TS, int RPT>
constexpr int stages_for() { return TS == 16 && RPT == 1 ? 3 : 2; }

template <int TS, int RPT, int C, bool BF16>
constexpr size_t bilinear_fwd_smem() {
    return sizeof(uint32_t) * stages_for<TS, RPT>() * TS * TS * RPT * ring_stride(RecLayout<0, C, BF16>::words) + 128;
}

// RPT = records each thread stages per batch: the batch ("blend depth") is
// D = TS * TS * RPT records; every pixel composites the records of a batch
// that cover it between two barriers, so a deeper batch spends fewer barriers
// per record and evens out the pixels' per-batch fragment counts.
template <int TS, int RPT, int C, bool BF16>
__global__ void __launch_bounds__(TS * TS) k_blend_fwd_bilinear(
    const ViewTable vt, const uint2* __restrict__ ranges, const uint32_t* __restrict__ order,
    const uint32_t* __restrict__ pts, const uint32_t* __restrict__ rec, uint32_t* __restrict__ rec_tile,
    float* __restrict__ t_final, uint32_t* __restrict__ last_out, WsHeader* __restrict__ hdr,
    unsigned long long* __restrict__ trace) {
    dependency_sync(ranges, order);
    constexpr int NT = TS * TS;     // threads = pixels
    constexpr int D = NT * RPT;     // records per batch
    constexpr int MW = D / 32;      // mask words per pixel
    constexpr int kStages = stages_for<TS, RPT>();
    const unsigned long long t_start = global_ns();
    const long long c_start = clock64();
    constexpr int RW = RecLayout<0, C, BF16>::words;
    constexpr int RS = ring_stride(RW);
    constexpr int FW = RecLayout<0, C, BF16>::feat_word;
    extern __shared__ __align__(128) uint32_t s_dyn[];
    uint32_t* const s_ring = align128(s_dyn);  // [kStages][D][RS] raw records
    __shared__ uint32_t s_mask[NT][MW + 1];    // MW words + 1 pad: conflict-free row reads
    // Per record: the alphas of its 2x2 box (FP32, pinned ops), indexed by the
    // parity (x & 1) + 2 (y & 1) of the covered pixel, and its depth. A 2x2 box
    // holds each parity once, so a pixel finds its own alpha at an offset that
    // is fixed for the thread: one 4-byte load, with no anchor to compare.
    __shared__ float4 s_alpha4[D];
    __shared__ float s_z[D];
    __shared__ uint32_t s_maxstop;

    const int64_t tile = order[blockIdx.x];
    const ViewDev& V = vt.v[view_of_tile(vt, tile)];
    const int64_t lt = tile - V.tile_off;
    const int tx = (int)(lt % V.tiles_x), ty = (int)(lt / V.tiles_x);
    const int tid = threadIdx.x, lane = tid & 31;
    const int lx = tid & (TS - 1), ly = tid / TS;
    const int px = tx * TS + lx, py = ty * TS + ly;
    const bool inside = px < V.W && py < V.H;
    const uint2 rg = ranges[tile];
    const uint32_t len = rg.y - rg.x;
    const uint32_t nbatch = (len + D - 1) / D;
    const float amax = vt.alpha_max, tmin = vt.t_min;
    const float* const my_alpha = reinterpret_cast<const float*>(s_alpha4) + ((lx & 1) | ((ly & 1) << 1));

    float T = 1.f, A = 0.f, Dp = 0.f;
    float F[C];
#pragma unroll
    for (int c = 0; c < C; ++c) F[c] = 0.f;
    uint32_t last = 0, stop = 0;
    bool done = !inside;
#pragma unroll
    for (int w = 0; w < MW; ++w) s_mask[tid][w] = 0;
    if (tid == 0) s_maxstop = 0;
    // Every row must be clear before any record thread sets bits in another
    // pixel's row (the first batch's atomicOr).
    __syncthreads();

    // Thread t copies records t, t + NT, ... of every batch. idx[s] = point
    // indices of batch j + kStages + s while batch j is processed (the copies
    // are issued kStages batches ahead, the indices read kStages further).
    auto point_of = [&](uint32_t j, int k) -> uint32_t {
        const uint32_t r = j * D + k * NT + tid;
        return r < len ? pts[rg.x + r] : 0xffffffffu;
    };
    auto issue = [&](uint32_t j, const uint32_t (&gi)[RPT]) {
#pragma unroll
        for (int k = 0; k < RPT; ++k) {
            if (gi[k] != 0xffffffffu) {
                uint32_t* dst = s_ring + ((size_t)(j % kStages) * D + k * NT + tid) * RS;
                const uint32_t* src = rec + (size_t)gi[k] * RW;
#pragma unroll
                for (int q = 0; q < RW; q += 4) cp_async16(dst + q, src + q);
            }
        }
        cp_async_commit();
    };
    uint32_t idx[kStages][RPT];
#pragma unroll
    for (int st = 0; st < kStages; ++st)
#pragma unroll
        for (int k = 0; k < RPT; ++k) idx[st][k] = point_of(st, k);
#pragma unroll
    for (int st = 0; st < kStages; ++st) {
        issue(st, idx[st]);
#pragma unroll
        for (int k = 0; k < RPT; ++k) idx[st][k] = point_of(st + kStages, k);
    }

    for (uint32_t j = 0; j < nbatch; ++j) {
        const uint32_t* ring = s_ring + (size_t)(j % kStages) * D * RS;
        cp_async_wait<kStages - 1>();  // this thread's copies of batch j have landed
        const uint32_t rel0 = j * D;
#pragma unroll
        for (int k = 0; k < RPT; ++k) {
            const int r = k * NT + tid;
            if (rel0 + r < len) {
                // Per record: the four fragment alphas of its 2x2 box (weights and
                // clamp in rounded operations, the same FP32 bits for every pixel)
                // and one mask bit per covered pixel of this tile.
                const uint4 g = *reinterpret_cast<const uint4*>(ring + r * RS);
                if (rec_tile) {
                    // The record, in list order, for the backward's sequential reads
                    // (coalesced: consecutive threads write consecutive records).
                    uint4* dst = reinterpret_cast<uint4*>(rec_tile + (size_t)(rg.x + rel0 + r) * RW);
                    dst[0] = g;
#pragma unroll
                    for (int q = 1; q < RW / 4; ++q)
                        dst[q] = *reinterpret_cast<const uint4*>(ring + r * RS + 4 * q);
                }
                const BilinGeom bg = bilin_geom(__uint_as_float(g.x), __uint_as_float(g.y));
                const float o = __uint_as_float(g.w);
                const float ax = __fsub_rn(1.f, bg.a), by = __fsub_rn(1.f, bg.b);
                const int X0 = bg.i0 - tx * TS, Y0 = bg.j0 - ty * TS;
                // weights of the even and the odd column and row of the box
                const float we = (X0 & 1) ? bg.a : ax, wo = (X0 & 1) ? ax : bg.a;
                const float he = (Y0 & 1) ? bg.b : by, ho = (Y0 & 1) ? by : bg.b;
                s_alpha4[r] = make_float4(fminf(__fmul_rn(o, __fmul_rn(we, he)), amax),
                                          fminf(__fmul_rn(o, __fmul_rn(wo, he)), amax),
                                          fminf(__fmul_rn(o, __fmul_rn(we, ho)), amax),
                                          fminf(__fmul_rn(o, __fmul_rn(wo, ho)), amax));
                s_z[r] = __uint_as_float(g.z);
                const uint32_t bit = 1u << lane;
                const int word = r >> 5;
#pragma unroll
                for (int dy = 0; dy < 2; ++dy) {
                    const int Y = Y0 + dy;
                    if ((unsigned)Y >= (unsigned)TS) continue;
#pragma unroll
                    for (int dx = 0; dx < 2; ++dx) {
                        const int X = X0 + dx;
                        if ((unsigned)X < (unsigned)TS) atomicOr(&s_mask[Y * TS + X][word], bit);
                    }
                }
            }
        }
        if (__syncthreads_count(!done) == 0) break;
        if (!done) {
            // One loop over every set bit of the pixel's D-bit mask, in order.
            MaskWalk<MW, true> walk(s_mask[tid]);
#pragma unroll 1
            while (walk.more()) {
                const int r = walk.next();
                const float alpha = my_alpha[4 * r];
                const float z = s_z[r];
                const float nT = __fmul_rn(T, __fsub_rn(1.f, alpha));
                if (nT < tmin) {
                    done = true;
                    stop = rel0 + r + 1;
                    break;
                }
                const uint32_t* rp = ring + r * RS;
                float f[C];
                load_features<C, BF16>(rp + FW, f);
                const float ta = T * alpha;
#pragma unroll
                for (int c = 0; c < C; ++c) F[c] = fmaf(ta, f[c], F[c]);
                Dp = fmaf(ta, z, Dp);
                A += ta;
                T = nT;
                last = rel0 + r + 1;
            }
        }
#pragma unroll
        for (int w = 0; w < MW; ++w) s_mask[tid][w] = 0;
        __syncthreads();
        // Slot j % kStages is free: refill it with batch j + kStages.
        issue(j + kStages, idx[0]);
#pragma unroll
        for (int st = 0; st + 1 < kStages; ++st)
#pragma unroll
            for (int k = 0; k < RPT; ++k) idx[st][k] = idx[st + 1][k];
#pragma unroll
        for (int k = 0; k < RPT; ++k) idx[kStages - 1][k] = point_of(j + 2 * kStages, k);
    }
    cp_async_wait<0>();  // no copy may land after the CTA has exited

    if (inside) {
        const int64_t pix = (int64_t)py * V.W + px;
        float* of = V.out_feat + pix * C;
        if (C % 4 == 0) {
#pragma unroll
            for (int c = 0; c < C; c += 4)
                *reinterpret_cast<float4*>(of + c) = make_float4(F[c], F[c + 1], F[c + 2], F[c + 3]);
        } else {
#pragma unroll
            for (int c = 0; c < C; ++c) of[c] = F[c];
        }
        if (V.out_alpha) V.out_alpha[pix] = A;
        if (V.out_depth) V.out_depth[pix] = Dp;
        t_final[V.pix_off + pix] = T;
        last_out[V.pix_off + pix] = last;
    }
    const int open = __syncthreads_or(inside && stop == 0);
    if (stop) atomicMax(&s_maxstop, stop);
    __syncthreads();
    if (tid == 0) {
        atomicAdd(&hdr->needed, (unsigned long long)(open ? (rg.y - rg.x) : s_maxstop));
        trace_tile(trace, tile, 0, t_start, c_start);
    }
}

// Gaussian: every warp owns an 8x4 sub-tile and goes through the tile's list
// with no CTA-wide barrier. The records are staged once for all of the tile's
// warps, in a ring of kFwdStages batches: one warp copies a batch
// (cp.async) and the batch's mbarrier tells the others when it has landed; the
// last warp to be done with a batch refills its slot with the batch kFwdStages
// further on (whose point indices one of the warps has read meanwhile), so warps
// may drift apart. Of every 32 records a warp ballots those whose box meets the
// left and the right 4x4 half of its sub-tile, and each half composites its own
// records, 16 lanes in lockstep, beside the other half's. A warp whose 32 pixels
// have terminated only keeps count, also of the rest of its batch (looked at
// every 32 records: where splats of 50 pixels end the lists early, 288 -> 262
// us); once all of the tile's warps have, nothing more is staged.
// Bound by issue slots (90 % busy, about 15 instructions a record and warp).
// Before, every warp gathered every record itself (three scattered 16-byte loads
// a record and warp: the L1 pipe 70 % busy) and walked the records that met its
// whole sub-tile (of 32 records with 3-pixel boxes about 9; a half meets 6): 16 M
// Gaussians, BF16, 703 -> 566 us; 2 M at 1599x899 397 -> 311 us. Halves alone
// were 660 and 356 us, the ring with batches of 32 records 611 and 357, of 64
// 571 and 325 us, of 128 566 and 311 us.
// On 8x8 tiles the ring of 128 records, shared by two warps, is what limits the
// CTAs on an SM. Where tiles are many times what fits, CTAs count more than long
// batches, and a batch has 64 records; up to ten times what fits with 128, the
// longest lists count, and it has 128. 1599x899 (22600 tiles, 13 times), 2 M, FP32:
// C = 4 332 us with 128, 279 with 64, 283 with 32 (every warp on its own 319 us),
// C = 16 634, 376, 342 us (510 us); 1200x720 (8 times), C = 4, 0.26 M / 1.2 M / 4.3 M
// Gaussians: 103 / 209 / 296 us with 128, 117 / 214 / 272 us with 64; 660x396 (2.5
// times): 69 / 184 / 250 and 72 / 201 / 271 us.
constexpr int kFwdStages = 3;
constexpr int kFwdBatch = 128, kFwdShortBatch = 64;
constexpr uint32_t kGaussStop = 2u;  // s_abort: every warp has finished

template <int GB, int C, bool BF16>
constexpr size_t gauss_fwd_smem() {
    return 128 + sizeof(uint32_t) * kFwdStages * GB * gauss_ring_stride<C, BF16>();
}

// GB: records per batch. STALL: test hook, batch 1 is never staged and the waits
// are short, so those on it run out (a kernel of its own: a limit that is not a
// constant cost the 8-channel blends 4 %).
template <int TS, int GB, int C, bool BF16, bool STALL>
__global__ void __launch_bounds__(TS * TS) k_blend_fwd_gauss(
    const ViewTable vt, const uint2* __restrict__ ranges, const uint32_t* __restrict__ order,
    const uint32_t* __restrict__ pts, const uint32_t* __restrict__ rec, float* __restrict__ t_final,
    uint32_t* __restrict__ last_out, WsHeader* __restrict__ hdr) {
    dependency_sync(ranges, order);
    constexpr int NT = TS * TS;
    constexpr int NW = NT / 32;      // warps = 8x4 sub-tiles
    constexpr int WPR = TS / 8;      // warps per row of 8x4 sub-tiles
    constexpr int R = kFwdStages;
    constexpr int NG = GB / 32;      // ballots per batch
    constexpr int RW = RecLayout<1, C, BF16>::words;
    constexpr int RS = gauss_ring_stride<C, BF16>();
    constexpr int FW = RecLayout<1, C, BF16>::feat_word;
    extern __shared__ __align__(128) uint32_t s_dyn[];
    uint32_t* const s_ring = align128(s_dyn);      // [R][GB][RS]
    __shared__ uint32_t s_pnext[R][GB];            // point indices of the batch a slot takes next
    __shared__ uint32_t s_done[R];                 // warps done with the slot's batch
    __shared__ __align__(8) uint64_t s_mbar[R];    // slot filled (32 arrivals: the staging lanes)
    __shared__ uint32_t s_fin;                     // warps whose pixels have all terminated
    __shared__ uint32_t s_abort;                   // kGaussStop, or 1 after a wait that ran out
    __shared__ uint32_t s_maxstop;

    const int64_t tile = order[blockIdx.x];
    const ViewDev& V = vt.v[view_of_tile(vt, tile)];
    const int64_t lt = tile - V.tile_off;
    const int tx = (int)(lt % V.tiles_x), ty = (int)(lt / V.tiles_x);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int sx0 = tx * TS + (warp % WPR) * 8, sy0 = ty * TS + (warp / WPR) * 4;
    const int px = sx0 + (lane >> 4) * 4 + (lane & 3), py = sy0 + ((lane >> 2) & 3);
    const bool inside = px < V.W && py < V.H;
    const uint2 rg = ranges[tile];
    const float amax = vt.alpha_max, tmin = vt.t_min;
    const float fpx = (float)px, fpy = (float)py;
    const float fx0 = (float)sx0, fy0 = (float)sy0;

    if (tid < R) {
        s_done[tid] = 0;
        mbar_init(&s_mbar[tid], 32);
    }
    if (tid == 0) {
        s_fin = 0;
        s_abort = 0;
        s_maxstop = 0;
    }
    mbar_init_fence();
    __syncthreads();

    float T = 1.f, A = 0.f, Dp = 0.f;
    float F[C];
#pragma unroll
    for (int c = 0; c < C; ++c) F[c] = 0.f;
    uint32_t last = 0, stop = 0;
    bool done = !inside, counted = false;
    const uint32_t nb = (rg.y - rg.x + GB - 1) / GB;

    // Stages batch j (all 32 lanes of one warp). Batches j >= R take their point
    // indices from s_pnext.
    auto stage = [&](uint32_t j) {
        if (STALL && j == 1) return;
        const int st = (int)(j % R);
#pragma unroll
        for (int k = 0; k < NG; ++k) {
            const uint32_t q = rg.x + j * GB + k * 32 + lane;
            if (q < rg.y) {
                const uint32_t gi = j < (uint32_t)R ? pts[q] : s_pnext[st][k * 32 + lane];
                uint32_t* dst = s_ring + ((size_t)st * GB + k * 32 + lane) * RS;
                const uint32_t* src = rec + (size_t)gi * RW;
#pragma unroll
                for (int w = 0; w < RS; w += 4) cp_async16(dst + w, src + w);
            }
        }
        cp_async_mbar_arrive_noinc(&s_mbar[st]);
    };
    if (warp == 0) {
        for (uint32_t j = 0; j < (uint32_t)R && j < nb; ++j) stage(j);
    }

    uint32_t phase = 0;  // parity of the next phase to wait for, per slot
#pragma unroll 1
    for (uint32_t j = 0; j < nb; ++j) {
        const int st = (int)(j % R);
        const uint32_t fin = __ballot_sync(0xffffffffu, done);
        if (fin == 0xffffffffu && !counted) {
            counted = true;
            if (lane == 0) atomicAdd(&s_fin, 1u);
        }
        if (!__all_sync(0xffffffffu, mbar_wait_or_abort(&s_mbar[st], (phase >> st) & 1u, &s_abort, STALL ? 64u : kMbarPolls))) {
            if (lane == 0 && *(volatile uint32_t*)&s_abort != kGaussStop) {
                s_abort = 1u;
                atomicOr(&hdr->error, kErrTimeout);
            }
            break;
        }
        if (__any_sync(0xffffffffu, *(volatile uint32_t*)&s_abort == kGaussStop)) break;
        phase ^= 1u << st;
        // One warp per batch reads the point indices of batch j + R now and
        // stores them before it counts itself done.
        const bool pref = warp == (int)(j % NW) && j + R < nb;
        uint32_t pnext[NG];
        if (pref) {
#pragma unroll
            for (int k = 0; k < NG; ++k) {
                const uint32_t q = rg.x + (j + R) * GB + k * 32 + lane;
                pnext[k] = q < rg.y ? pts[q] : 0u;
            }
        }
#pragma unroll 1
        for (int k = 0; k < NG && fin != 0xffffffffu; ++k) {
            const uint32_t* ring = s_ring + ((size_t)st * GB + k * 32) * RS;
            const uint32_t rel0 = j * GB + k * 32;
            bool hit = false, hit2 = false;  // this lane's record meets the left, the right half
            if (rg.x + rel0 + lane < rg.y) {
                const uint32_t* rp = ring + lane * RS;
                const GaussBounds bx = gauss_bounds(__fsub_rn(__uint_as_float(rp[0]), 0.5f),
                                                    __fsub_rn(__uint_as_float(rp[1]), 0.5f), __uint_as_float(rp[7]));
                hit = meets(bx, fx0, fx0 + 3.f, fy0, fy0 + 3.f);
                hit2 = meets(bx, fx0 + 4.f, fx0 + 7.f, fy0, fy0 + 3.f);
            }
            const uint32_t left = __ballot_sync(0xffffffffu, hit), right = __ballot_sync(0xffffffffu, hit2);
            uint32_t m = lane < 16 ? left : right;
            if (((lane < 16 ? fin : fin >> 16) & 0xffffu) == 0xffffu) m = 0;  // this half has finished
            __syncwarp();
            // As many rounds as the longer half has records, all lanes together.
            const int rounds = max(__popc(__shfl_sync(0xffffffffu, m, 0)), __popc(__shfl_sync(0xffffffffu, m, 16)));
#pragma unroll 1
            for (int it = 0; it < rounds; ++it) {
                const int r = (__ffs(m) - 1) & 31;
                const bool any = m != 0;
                m &= m - 1;
                const uint32_t* rp = ring + r * RS;
                const uint4 g = *reinterpret_cast<const uint4*>(rp);      // u, v, z, opacity
                const uint4 h = *reinterpret_cast<const uint4*>(rp + 4);  // conic, radius
                const float um = __fsub_rn(__uint_as_float(g.x), 0.5f), vm = __fsub_rn(__uint_as_float(g.y), 0.5f);
                const float dx = __fsub_rn(fpx, um), dy = __fsub_rn(fpy, vm);
                const float mm = gauss_m(dx, dy, __uint_as_float(h.x), __uint_as_float(h.y), __uint_as_float(h.z));
                if (any && mm <= 9.f && !done && meets(gauss_bounds(um, vm, __uint_as_float(h.w)), fpx, fpx, fpy, fpy)) {
                    const float alpha = fminf(__fmul_rn(__uint_as_float(g.w), gauss_value(mm)), amax);
                    const float nT = __fmul_rn(T, __fsub_rn(1.f, alpha));
                    if (nT < tmin) {
                        done = true;
                        stop = rel0 + r + 1;
                    } else {
                        float fr[C];
                        load_features<C, BF16>(rp + FW, fr);
                        const float ta = T * alpha;
#pragma unroll
                        for (int c = 0; c < C; ++c) F[c] = fmaf(ta, fr[c], F[c]);
                        Dp = fmaf(ta, __uint_as_float(g.z), Dp);
                        A += ta;
                        T = nT;
                        last = rel0 + r + 1;
                    }
                }
            }
            if (__all_sync(0xffffffffu, done)) break;
        }
        if (pref) {
#pragma unroll
            for (int k = 0; k < NG; ++k) s_pnext[st][k * 32 + lane] = pnext[k];
        }
        // Done with the batch: the last of the warps refills its slot, unless
        // every warp has finished.
        __syncwarp();
        __threadfence_block();
        uint32_t prev = 0;
        if (lane == 0) prev = atomicAdd(&s_done[st], 1u);
        prev = __shfl_sync(0xffffffffu, prev, 0);
        if (prev != (uint32_t)(NW - 1)) continue;
        __threadfence_block();
        if (__any_sync(0xffffffffu, *(volatile uint32_t*)&s_fin == (uint32_t)NW)) {
            // Nothing more is blended: warps that wait for the next batch of
            // this slot (none can wait for a later one) are let through to the flag.
            if (lane == 0) s_abort = kGaussStop;
            __syncwarp();
            __threadfence_block();
            if (j + R < nb) mbar_arrive(&s_mbar[st]);
            break;
        }
        if (lane == 0) s_done[st] = 0;
        __syncwarp();
        __threadfence_block();
        if (j + R < nb) stage(j + R);
    }
    cp_async_wait_all();  // no copy may land after the CTA has exited

    if (inside) {
        const int64_t pix = (int64_t)py * V.W + px;
        store_row<C>(V.out_feat + pix * C, F);
        if (V.out_alpha) V.out_alpha[pix] = A;
        if (V.out_depth) V.out_depth[pix] = Dp;
        t_final[V.pix_off + pix] = T;
        last_out[V.pix_off + pix] = last;
    }
    const int open = __syncthreads_or(inside && stop == 0);
    if (stop) atomicMax(&s_maxstop, stop);
    __syncthreads();
    if (tid == 0)
        atomicAdd(&hdr->needed, (unsigned long long)(open ? (rg.y - rg.x) : s_maxstop));
}

template <int TS, int C, bool BF16>
cudaError_t launch_fwd_gauss(const ViewTable& vt, const Bufs& b, const uint32_t* pts, cudaStream_t s) {
    constexpr size_t smem = gauss_fwd_smem<kFwdBatch, C, BF16>(), small = gauss_fwd_smem<kFwdShortBatch, C, BF16>();
    static_assert(smem <= 48 * 1024, "within the default dynamic shared memory");
    constexpr int64_t per_sm = 227 * 1024 / (smem + 3 * 1024);  // CTAs on an SM, with the static and the system's share
    const unsigned grid = (unsigned)vt.tiles_total;
    const bool short_batch = TS == 8 && vt.tiles_total > 10 * per_sm * device_sm_count();
    constexpr int GS = TS == 8 ? kFwdShortBatch : kFwdBatch;
    auto kern = short_batch ? k_blend_fwd_gauss<TS, GS, C, BF16, false> : k_blend_fwd_gauss<TS, kFwdBatch, C, BF16, false>;
    if constexpr (C == 4 && !BF16) {
        if (vt.flags & RAST_FLAG_TEST_FWD_BLEND_STALL)
            kern = short_batch ? k_blend_fwd_gauss<TS, GS, C, BF16, true> : k_blend_fwd_gauss<TS, kFwdBatch, C, BF16, true>;
    }
    ProfScope ps("blend_fwd", s);
    return launch_dependent(kern, grid, TS * TS, short_batch ? small : smem, s, vt, b.ranges, b.order, pts, b.rec, b.t_final,
                            b.last, b.hdr);
}

template <int TS, int RPT, int C, bool BF16>
cudaError_t launch_fwd_t(const ViewTable& vt, const Bufs& b, const uint32_t* pts, cudaStream_t s) {
    const unsigned grid = (unsigned)vt.tiles_total;
    if (vt.mode == 0) {
        constexpr size_t smem = bilinear_fwd_smem<TS, RPT, C, BF16>();
        static PerDevice attr;
        const cudaError_t e = per_device(attr, nullptr, [](int, int*) {
            return cudaFuncSetAttribute(k_blend_fwd_bilinear<TS, RPT, C, BF16>,
                                        cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        });
        if (e != cudaSuccess) return e;
        ProfScope ps("blend_fwd", s);
        return launch_dependent(k_blend_fwd_bilinear<TS, RPT, C, BF16>, grid, TS * TS, smem, s, vt, b.ranges, b.order,
                                pts, b.rec, b.rec_tile, b.t_final, b.last, b.hdr, b.trace);
    }
    return launch_fwd_gauss<TS, C, BF16>(vt, b, pts, s);
}

template <int TS, int C, bool BF16>
cudaError_t launch_fwd_d(const ViewTable& vt, const Bufs& b, const uint32_t* pts, cudaStream_t s) {
    const int rpt = vt.mode == 0 ? vt.blend_depth / (TS * TS) : 1;
    if constexpr (TS == 8) {
        if (rpt == 4) return launch_fwd_t<TS, 4, C, BF16>(vt, b, pts, s);
    }
    if (rpt == 2) return launch_fwd_t<TS, 2, C, BF16>(vt, b, pts, s);
    return launch_fwd_t<TS, 1, C, BF16>(vt, b, pts, s);
}

template <int C>
cudaError_t launch_fwd_c(const ViewTable& vt, const Bufs& b, const uint32_t* pts, cudaStream_t s) {
    if (vt.tile == 8)
        return vt.bf16 ? launch_fwd_d<8, C, true>(vt, b, pts, s) : launch_fwd_d<8, C, false>(vt, b, pts, s);
    return vt.bf16 ? launch_fwd_d<16, C, true>(vt, b, pts, s) : launch_fwd_d<16, C, false>(vt, b, pts, s);
}

}  // namespace

bool channels_supported(int C) {
    return C == 1 || C == 2 || C == 3 || C == 4 || C == 8 || C == 16;
}

cudaError_t launch_tile_order(const ViewTable& vt, const Bufs& b, cudaStream_t s) {
    const int64_t P = vt.tiles_total;
    if (P == 0) return cudaSuccess;
    uint32_t* counts = b.order + P;  // 33 bucket counts, then 33 cursors (cleared at the start of the pass)
    const int64_t want = (P + 255) / 256;
    const unsigned grid = (unsigned)(want < 1024 ? want : 1024);
    ProfScope ps("tile_order.scatter", s);
    return launch_dependent(k_tile_scatter, grid, 256, 0, s, b.ranges, P, counts, counts + 33, b.order);
}

namespace {

// Untiled baseline (the per-pixel lists of the original INPC rasterizer that
// Sec. 3.2 "Tiled Rendering" replaces): the copies are per-pixel fragments
// sorted by (pixel, depth, point index), and one thread composites its
// pixel's list front to back, gathering every fragment's record from memory.
// Same FP32 operations as the tiled kernel, so the images are identical.
template <int C, bool BF16>
__global__ void __launch_bounds__(256) k_blend_fwd_pixel(const ViewTable vt, const uint2* __restrict__ ranges,
                                                         const uint32_t* __restrict__ pts,
                                                         const uint32_t* __restrict__ rec,
                                                         float* __restrict__ t_final, uint32_t* __restrict__ last_out,
                                                         WsHeader* __restrict__ hdr) {
    constexpr int RW = RecLayout<0, C, BF16>::words;
    constexpr int FW = RecLayout<0, C, BF16>::feat_word;
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;  // global pixel ("tile") id
    const bool valid = p < vt.tiles_total;
    uint32_t need = 0;
    if (valid) {
        const ViewDev& V = vt.v[view_of_tile(vt, p)];
        const int64_t lp = p - V.tile_off;
        const int px = (int)(lp % V.W), py = (int)(lp / V.W);
        const uint2 rg = ranges[p];
        const float amax = vt.alpha_max, tmin = vt.t_min;
        float T = 1.f, A = 0.f, Dp = 0.f;
        float F[C];
#pragma unroll
        for (int c = 0; c < C; ++c) F[c] = 0.f;
        uint32_t last = 0, stop = 0;
#pragma unroll 1
        for (uint32_t q = rg.x; q < rg.y; ++q) {
            const uint32_t* rp = rec + (size_t)pts[q] * RW;
            const uint4 g = *reinterpret_cast<const uint4*>(rp);
            const BilinGeom bg = bilin_geom(__uint_as_float(g.x), __uint_as_float(g.y));
            const float o = __uint_as_float(g.w);
            const float wx = px == bg.i0 ? __fsub_rn(1.f, bg.a) : bg.a;
            const float wy = py == bg.j0 ? __fsub_rn(1.f, bg.b) : bg.b;
            const float alpha = fminf(__fmul_rn(o, __fmul_rn(wx, wy)), amax);
            const float nT = __fmul_rn(T, __fsub_rn(1.f, alpha));
            if (nT < tmin) {
                stop = q - rg.x + 1;
                break;
            }
            float f[C];
            load_features<C, BF16>(rp + FW, f);
            const float ta = T * alpha;
#pragma unroll
            for (int c = 0; c < C; ++c) F[c] = fmaf(ta, f[c], F[c]);
            Dp = fmaf(ta, __uint_as_float(g.z), Dp);
            A += ta;
            T = nT;
            last = q - rg.x + 1;
        }
        const int64_t pix = (int64_t)py * V.W + px;
        float* of = V.out_feat + pix * C;
#pragma unroll
        for (int c = 0; c < C; ++c) of[c] = F[c];
        if (V.out_alpha) V.out_alpha[pix] = A;
        if (V.out_depth) V.out_depth[pix] = Dp;
        t_final[V.pix_off + pix] = T;
        last_out[V.pix_off + pix] = last;
        need = stop ? stop : rg.y - rg.x;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) need += __shfl_xor_sync(0xffffffffu, need, o);
    if ((threadIdx.x & 31) == 0 && need) atomicAdd(&hdr->needed, (unsigned long long)need);
}

// The same per-pixel lists composited by one warp per pixel (the layout of
// the untiled rasterizer Sec. 3.2 starts from): the lanes gather 32
// consecutive fragments' records at once and compute their alphas; the
// transmittance then steps through the 32 alphas in list order with the
// per-thread walk's FP32 operations (every lane runs the same serial chain on
// shuffled alphas, so the termination decision and T_final are those of the
// serial walk bit for bit); the chunk's F, depth and alpha sums are warp
// reductions (tree order: within FP32 rounding of the serial sums, not bit
// for bit).
__device__ __forceinline__ float warp_sum_f(float x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

template <int C, bool BF16>
__global__ void __launch_bounds__(256) k_blend_fwd_pixel_warp(const ViewTable vt, const uint2* __restrict__ ranges,
                                                              const uint32_t* __restrict__ pts,
                                                              const uint32_t* __restrict__ rec,
                                                              float* __restrict__ t_final,
                                                              uint32_t* __restrict__ last_out,
                                                              WsHeader* __restrict__ hdr) {
    constexpr int RW = RecLayout<0, C, BF16>::words;
    constexpr int FW = RecLayout<0, C, BF16>::feat_word;
    const int64_t p = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;  // global pixel ("tile") id
    const int lane = threadIdx.x & 31;
    if (p >= vt.tiles_total) return;  // uniform per warp
    const ViewDev& V = vt.v[view_of_tile(vt, p)];
    const int64_t lp = p - V.tile_off;
    const int px = (int)(lp % V.W), py = (int)(lp / V.W);
    const uint2 rg = ranges[p];
    const float amax = vt.alpha_max, tmin = vt.t_min;
    float T = 1.f, A = 0.f, Dp = 0.f;
    float F[C];
#pragma unroll
    for (int c = 0; c < C; ++c) F[c] = 0.f;
    uint32_t last = 0, stop = 0;
#pragma unroll 1
    for (uint32_t q0 = rg.x; q0 < rg.y; q0 += 32) {
        const uint32_t q = q0 + lane;
        const int nv = (int)min(32u, rg.y - q0);
        float alpha = 0.f, z = 0.f;
        float f[C];
#pragma unroll
        for (int c = 0; c < C; ++c) f[c] = 0.f;
        if (q < rg.y) {
            const uint32_t* rp = rec + (size_t)pts[q] * RW;
            const uint4 g = *reinterpret_cast<const uint4*>(rp);
            const BilinGeom bg = bilin_geom(__uint_as_float(g.x), __uint_as_float(g.y));
            const float o = __uint_as_float(g.w);
            const float wx = px == bg.i0 ? __fsub_rn(1.f, bg.a) : bg.a;
            const float wy = py == bg.j0 ? __fsub_rn(1.f, bg.b) : bg.b;
            alpha = fminf(__fmul_rn(o, __fmul_rn(wx, wy)), amax);
            load_features<C, BF16>(rp + FW, f);
            z = __uint_as_float(g.z);
        }
        // Serial transmittance over the chunk: T_k before fragment k in lane k.
        float Tk = 0.f;
        int kstop = nv;
        for (int k = 0; k < nv; ++k) {
            const float ak = __shfl_sync(0xffffffffu, alpha, k);
            const float nT = __fmul_rn(T, __fsub_rn(1.f, ak));
            if (nT < tmin) {
                kstop = k;
                break;
            }
            if (lane == k) Tk = T;
            T = nT;
        }
        const float ta = lane < kstop ? Tk * alpha : 0.f;
#pragma unroll
        for (int c = 0; c < C; ++c) F[c] += warp_sum_f(ta * f[c]);
        Dp += warp_sum_f(ta * z);
        A += warp_sum_f(ta);
        if (kstop > 0) last = q0 - rg.x + (uint32_t)kstop;
        if (kstop < nv) {
            stop = q0 - rg.x + (uint32_t)kstop + 1;
            break;
        }
    }
    if (lane == 0) {
        const int64_t pix = (int64_t)py * V.W + px;
        store_row<C>(V.out_feat + pix * C, F);
        if (V.out_alpha) V.out_alpha[pix] = A;
        if (V.out_depth) V.out_depth[pix] = Dp;
        t_final[V.pix_off + pix] = T;
        last_out[V.pix_off + pix] = last;
        const uint32_t need = stop ? stop : rg.y - rg.x;
        if (need) atomicAdd(&hdr->needed, (unsigned long long)need);
    }
}

template <int C>
cudaError_t launch_pixel_warp_c(const ViewTable& vt, const Bufs& b, const uint32_t* pts, cudaStream_t s) {
    const unsigned grid = (unsigned)((vt.tiles_total * 32 + 255) / 256);
    ProfScope ps("blend_fwd_pixel_warp", s);
    if (vt.bf16)
        k_blend_fwd_pixel_warp<C, true><<<grid, 256, 0, s>>>(vt, b.ranges, pts, b.rec, b.t_final, b.last, b.hdr);
    else
        k_blend_fwd_pixel_warp<C, false><<<grid, 256, 0, s>>>(vt, b.ranges, pts, b.rec, b.t_final, b.last, b.hdr);
    return cudaGetLastError();
}

template <int C>
cudaError_t launch_pixel_c(const ViewTable& vt, const Bufs& b, const uint32_t* pts, cudaStream_t s) {
    const unsigned grid = (unsigned)((vt.tiles_total + 255) / 256);
    ProfScope ps("blend_fwd_pixel", s);
    if (vt.bf16) k_blend_fwd_pixel<C, true><<<grid, 256, 0, s>>>(vt, b.ranges, pts, b.rec, b.t_final, b.last, b.hdr);
    else k_blend_fwd_pixel<C, false><<<grid, 256, 0, s>>>(vt, b.ranges, pts, b.rec, b.t_final, b.last, b.hdr);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_blend_fwd_pixel(const ViewTable& vt, const Bufs& b, const uint32_t* pts, cudaStream_t s) {
    if (vt.tiles_total == 0) return cudaSuccess;
    switch (vt.C) {
        case 1: return launch_pixel_c<1>(vt, b, pts, s);
        case 2: return launch_pixel_c<2>(vt, b, pts, s);
        case 3: return launch_pixel_c<3>(vt, b, pts, s);
        case 4: return launch_pixel_c<4>(vt, b, pts, s);
        case 8: return launch_pixel_c<8>(vt, b, pts, s);
        case 16: return launch_pixel_c<16>(vt, b, pts, s);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_blend_fwd_pixel_warp(const ViewTable& vt, const Bufs& b, const uint32_t* pts, cudaStream_t s) {
    if (vt.tiles_total == 0) return cudaSuccess;
    switch (vt.C) {
        case 1: return launch_pixel_warp_c<1>(vt, b, pts, s);
        case 2: return launch_pixel_warp_c<2>(vt, b, pts, s);
        case 3: return launch_pixel_warp_c<3>(vt, b, pts, s);
        case 4: return launch_pixel_warp_c<4>(vt, b, pts, s);
        case 8: return launch_pixel_warp_c<8>(vt, b, pts, s);
        case 16: return launch_pixel_warp_c<16>(vt, b, pts, s);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_blend_fwd(const ViewTable& vt, const Bufs& b, const uint32_t* pts, cudaStream_t s) {
    if (vt.tiles_total == 0) return cudaSuccess;
    switch (vt.C) {
        case 1: return launch_fwd_c<1>(vt, b, pts, s);
        case 2: return launch_fwd_c<2>(vt, b, pts, s);
        case 3: return launch_fwd_c<3>(vt, b, pts, s);
        case 4: return launch_fwd_c<4>(vt, b, pts, s);
        case 8: return launch_fwd_c<8>(vt, b, pts, s);
        case 16: return launch_fwd_c<16>(vt, b, pts, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace rast
