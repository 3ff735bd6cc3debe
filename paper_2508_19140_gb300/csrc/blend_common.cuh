// Shared pieces of the blend kernels (K6 forward, K7 backward).
//
// A record is gathered once per (tile, batch) by one thread and staged in
// shared memory; the per-pixel work then reads only shared memory. The
// per-fragment alpha and the coverage test are single device functions used
// by both passes, so the backward replays the forward's FP32 decisions bit for
// bit (round-to-nearest intrinsics, no contraction):
//   bilinear:  a = (u - 1/2) - floor(u - 1/2), w = wx * wy with wx = 1 - a at
//              the anchor column and a at the next one, alpha = min(o w, amax);
//   Gaussian:  d = (px - (u - 1/2), py - (v - 1/2)),
//              m = ((a dx) dx + 2 (b dx) dy) + (c dy) dy, covered iff the pixel
//              is in the box of radius r and m <= 9, alpha = min(o exp(-m/2), amax);
//   step:      T' = T (1 - alpha); the fragment is excluded and the pixel stops
//              once T' < t_min.
#pragma once

#include "rast_internal.cuh"

namespace rast {

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// ---- cp.async (LDGSTS) staging ----------------------------------------------
// Each thread copies its own record into a shared-memory ring slot; copies are
// grouped per batch and retired with wait_group, so several batches are in
// flight per CTA without any spin-wait.

__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gmem_src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(smem_dst)), "l"(gmem_src)
                 : "memory");
}

__device__ __forceinline__ void cp_async4(void* smem_dst, const void* gmem_src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(smem_dst)), "l"(gmem_src)
                 : "memory");
}

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }

__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Arrives on `bar` once every cp.async this thread has issued so far has
// landed (counted as one of the barrier's expected arrivals).
__device__ __forceinline__ void cp_async_mbar_arrive_noinc(uint64_t* bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_addr(bar)) : "memory");
}

template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// 1 / x with the hardware reciprocal (rcp.approx: at most 1 ulp off, where an
// IEEE-rounded reciprocal is a multi-instruction sequence). The backward's
// replay T_k = T_{k+1} / (1 - alpha_k) uses it: 1 - alpha >= 1 - alpha_max
// = 0.01, so x is never tiny, and each replay step then carries about 1.5 ulp
// instead of 1 (the gradients' tolerance covers replays of thousands of steps).
__device__ __forceinline__ float rcp_fast(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// ---- TMA bulk copies completed on an mbarrier ---------------------------------
// One thread arms the barrier with the batch's byte count and issues a single
// global -> shared bulk copy of a contiguous run of records; every thread then
// waits on the barrier's phase. Each wait is bounded: after kMbarPolls polls
// it reports failure (the caller raises the timeout bit of the error word and
// stops) instead of spinning on.

constexpr uint32_t kMbarPolls = 1u << 20;

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

// Makes the barriers' initialisation visible to the copy engine (follow with
// a CTA barrier before the first copy).
__device__ __forceinline__ void mbar_init_fence() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// Orders this thread's accesses to shared memory before bulk copies that a
// later barrier releases.
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Arms `bar` for `bytes` and copies them from global `src` to shared `dst`
// (both 16-byte aligned, bytes a multiple of 16).
__device__ __forceinline__ void bulk_copy_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    const uint32_t b = smem_addr(bar);
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(b), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_addr(dst)),
                 "l"(src), "r"(bytes), "r"(b)
                 : "memory");
}

// Waits until the phase of `bar` with this parity has completed; false if it
// did not within `polls` polls.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, uint32_t polls = kMbarPolls) {
    const uint32_t b = smem_addr(bar);
    for (uint32_t i = 0; i < polls; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(b), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}

// Record stride (u32 words) for a mode, channel count and feature type; the
// host computes the same value (rec_words). A power of two of at least 8
// words (32 bytes): every record is 16-byte aligned for cp.async and no record
// straddles a 64-byte DRAM burst, so each gather costs one burst.
template <int MODE, int C, bool BF16>
struct RecLayout {
    static constexpr int feat_word = MODE == 0 ? 4 : 8;
    static constexpr int feat_words = BF16 ? (C + 1) / 2 : C;
    static constexpr int need = feat_word + feat_words;
    static constexpr int words = need <= 8 ? 8 : (need <= 16 ? 16 : 32);
};

// Shared-memory stride (words) of a staged record: 4 words more than its
// global stride, so consecutive records start in 8 different 4-bank groups
// (a stride of 8, 16 or 32 words would start them in at most 4) and the
// per-fragment reads of random records conflict less; still a multiple of 16
// bytes for cp.async.
__host__ __device__ constexpr int ring_stride(int rw) { return rw + 4; }

// Staged words of a record: the used prefix (u, v, z, o, conic, radius,
// features) rounded to 16 bytes. A stride of 12 words keeps the lane-parallel
// reads of the ballot step free of bank conflicts.
template <int C, bool BF16>
__host__ __device__ constexpr int gauss_ring_stride() {
    return (RecLayout<1, C, BF16>::need + 3) & ~3;
}
// Polls `bar` for the phase of this parity, giving up after `polls` polls or
// once another warp of the CTA has given up (abort flag).
__device__ __forceinline__ bool mbar_wait_or_abort(uint64_t* bar, uint32_t parity, const volatile uint32_t* abort,
                                                   uint32_t polls) {
    const uint32_t b = smem_addr(bar);
    for (uint32_t i = 0; i < polls; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(b), "r"(parity)
            : "memory");
        if (ok) return true;
        if ((i & 63u) == 63u && *abort) return false;
    }
    return false;
}

// 128-byte aligned view of a dynamic shared-memory buffer (allocated with
// 128 spare bytes).
__device__ __forceinline__ uint32_t* align128(uint32_t* p) {
    const uintptr_t a = reinterpret_cast<uintptr_t>(p);
    const uint32_t sa = smem_addr(p);
    return reinterpret_cast<uint32_t*>(a + ((128u - (sa & 127u)) & 127u));
}

// Stores N floats at dst: 16-byte vector stores when N is a multiple of 4 and
// dst is 16-byte aligned, scalar stores otherwise.
template <int N>
__device__ __forceinline__ void store_row(float* dst, const float* v) {
    if constexpr (N % 4 == 0) {
        if ((reinterpret_cast<uintptr_t>(dst) & 15u) == 0) {
#pragma unroll
            for (int k = 0; k < N; k += 4)
                *reinterpret_cast<float4*>(dst + k) = make_float4(v[k], v[k + 1], v[k + 2], v[k + 3]);
            return;
        }
    }
#pragma unroll
    for (int k = 0; k < N; ++k) dst[k] = v[k];
}

// Features of one record as FP32 registers.
template <int C, bool BF16>
__device__ __forceinline__ void load_features(const uint32_t* __restrict__ rp, float (&f)[C]) {
    if (!BF16) {
        if (C % 4 == 0) {
#pragma unroll
            for (int c = 0; c < C; c += 4) {
                const uint4 q = *reinterpret_cast<const uint4*>(rp + c);
                f[c] = __uint_as_float(q.x);
                f[c + 1] = __uint_as_float(q.y);
                f[c + 2] = __uint_as_float(q.z);
                f[c + 3] = __uint_as_float(q.w);
            }
        } else {
#pragma unroll
            for (int c = 0; c < C; ++c) f[c] = __uint_as_float(rp[c]);
        }
    } else {
        if (C % 8 == 0) {
#pragma unroll
            for (int c = 0; c < C; c += 8) {
                const uint4 q = *reinterpret_cast<const uint4*>(rp + c / 2);
                f[c] = bf16lo(q.x); f[c + 1] = bf16hi(q.x);
                f[c + 2] = bf16lo(q.y); f[c + 3] = bf16hi(q.y);
                f[c + 4] = bf16lo(q.z); f[c + 5] = bf16hi(q.z);
                f[c + 6] = bf16lo(q.w); f[c + 7] = bf16hi(q.w);
            }
        } else {
#pragma unroll
            for (int c = 0; c < C; c += 2) {
                const uint32_t w = rp[c / 2];
                f[c] = bf16lo(w);
                if (c + 1 < C) f[c + 1] = bf16hi(w);
            }
        }
    }
}

// Walk over the set bits of a pixel's batch mask (MW words, in shared memory),
// ascending or descending. Two words stay in registers as one; of more, only
// those that are not empty are taken, the next one already loaded (a loop over
// empty words costs every lane of the warp the longest lane's steps, a load at
// the change of words its latency). Against a scanning loop, forward / backward:
// 16x16 tiles, 20 k points 57 -> 54 us, 60 k 41 -> 37 / 44 -> 42, 500 k 94 -> 83,
// 8 M 258 -> 222; 8x8 tiles, 4 M 128 -> 121 / 220 -> 211.
template <int MW, bool UP>
struct MaskWalk {
    const uint32_t* row;
    uint32_t m, next_m, rest;  // bits left in the current word; the next word; words after it
    int w, next_w;

    __device__ __forceinline__ void prefetch() {
        next_m = 0;
        if (rest) {
            next_w = UP ? __ffs(rest) - 1 : 31 - __clz(rest);
            rest &= ~(1u << next_w);
            next_m = row[next_w];
        }
    }

    __device__ __forceinline__ explicit MaskWalk(const uint32_t* row_) : row(row_) {
        rest = 0;
#pragma unroll
        for (int k = 0; k < MW; ++k) rest |= row[k] ? 1u << k : 0u;
        next_w = 0;
        prefetch();
        m = next_m;
        w = next_w;
        prefetch();
    }

    // Whether bits are left; next() takes one.
    __device__ __forceinline__ bool more() const { return (m | next_m) != 0u; }
    __device__ __forceinline__ int next() {
        if (m == 0) {
            m = next_m;
            w = next_w;
            prefetch();
        }
        const int b = UP ? __ffs(m) - 1 : 31 - __clz(m);
        m &= ~(1u << b);
        return w * 32 + b;
    }
};

template <bool UP>
struct MaskWalk<2, UP> {
    unsigned long long m;
    __device__ __forceinline__ explicit MaskWalk(const uint32_t* row) : m(row[0] | (unsigned long long)row[1] << 32) {}
    __device__ __forceinline__ bool more() const { return m != 0ull; }
    __device__ __forceinline__ int next() {
        const int b = UP ? __ffsll(m) - 1 : 63 - __clzll(m);
        m &= ~(1ull << b);
        return b;
    }
};

// Bilinear anchor and fractions from the screen position (exact in FP32).
struct BilinGeom {
    int i0, j0;
    float a, b;
};

__device__ __forceinline__ BilinGeom bilin_geom(float u, float v) {
    const float um = __fsub_rn(u, 0.5f), vm = __fsub_rn(v, 0.5f);
    const float fi = floorf(um), fj = floorf(vm);
    BilinGeom g;
    g.i0 = (int)fi;
    g.j0 = (int)fj;
    g.a = __fsub_rn(um, fi);
    g.b = __fsub_rn(vm, fj);
    return g;
}

// Gaussian pixel box from the record's radius r (inclusive, unclipped).
struct GaussBox {
    int x0, x1, y0, y1;
};

__device__ __forceinline__ GaussBox gauss_box(float um, float vm, float r) {
    GaussBox bx;
    bx.x0 = (int)ceilf(__fsub_rn(um, r));
    bx.x1 = (int)floorf(__fadd_rn(um, r));
    bx.y0 = (int)ceilf(__fsub_rn(vm, r));
    bx.y1 = (int)floorf(__fadd_rn(vm, r));
    return bx;
}

// The same box as bounds in FP32: an integer p is at least ceil(x) exactly when
// p >= x, and at most floor(x) when p <= x, so the comparisons decide as with
// the rounded bounds, without rounding them. (A NaN bound covers no pixel here;
// its record's distance is NaN as well and excludes every pixel either way.)
struct GaussBounds {
    float x0, x1, y0, y1;
};

__device__ __forceinline__ GaussBounds gauss_bounds(float um, float vm, float r) {
    return GaussBounds{__fsub_rn(um, r), __fadd_rn(um, r), __fsub_rn(vm, r), __fadd_rn(vm, r)};
}

// Whether the box meets the pixels [x, x1] x [y, y1].
__device__ __forceinline__ bool meets(const GaussBounds& b, float x, float x1, float y, float y1) {
    return b.x0 <= x1 && b.x1 >= x && b.y0 <= y1 && b.y1 >= y;
}

// Mahalanobis distance squared of pixel (px, py) (FP32, fixed order).
__device__ __forceinline__ float gauss_m(float dx, float dy, float ca, float cb, float cc) {
    const float t0 = __fmul_rn(__fmul_rn(ca, dx), dx);
    const float t1 = __fmul_rn(__fmul_rn(cb, dx), dy);
    const float t2 = __fmul_rn(__fmul_rn(cc, dy), dy);
    return __fadd_rn(__fadd_rn(t0, __fadd_rn(t1, t1)), t2);
}

__device__ __forceinline__ float gauss_value(float m) { return expf(__fmul_rn(-0.5f, m)); }

}  // namespace rast
