// K4: stable LSD radix sort of (u32 key, u32 value) pairs, one kernel per digit.
//
// The split sort of Sec. 3.2 ("Tiled Rendering") runs this twice: first over
// the points by depth key, then over the point-tile copies by tile id. Both
// sorts must be stable: stability is what makes ties in depth fall back to
// point index, and what keeps the depth order inside every tile after the
// second sort.
//
// Structure (single-sweep LSD with decoupled look-back):
//   k_digit_hist  one read of all keys counts the digits of every pass at once
//                 (digit counts do not depend on the order), and clears the
//                 per-pass tile counters and look-back status words;
//   k_sweep       per pass, persistent CTAs take tiles of 256 * IPT keys in
//                 input order from an atomic counter; keys and values arrive by
//                 bulk copies. Each warp counts the digits of its own keys in
//                 shared memory (one increment a key), the tile's counts are
//                 published, and the warps' counters become the tile-local
//                 start of every (digit, warp). A key's place in the tile is
//                 then its digit's running counter plus the number of lower
//                 lanes with the same digit, and key and value go to shared
//                 memory there at once. After the threads have looked back for
//                 the counts of all earlier tiles, both leave shared memory in
//                 digit order, in runs.
// Look-back in two levels: a tile publishes its counts on their own and adds
// them to its group's sums (kGroup tiles; the word also counts the arrivals),
// and the group's last tile publishes the inclusive prefix. A tile sums the
// tiles before it in its group (one round of loads) and walks back over whole
// groups, so hundreds of tiles that start together wait on a few round trips
// rather than on a chain through all of them.
// A tile only waits on tiles that running CTAs took before it, so the waits
// always end; each wait is still bounded, and on expiry the kernel raises the
// timeout bit of the workspace error word and carries on with the partial
// prefix instead of spinning on. The element count may live on the device (copies
// are counted on the GPU): launch shapes depend only on the capacity and on
// the count the caller expects.
#include "blend_common.cuh"

namespace rast {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kGroup = 16;                  // tiles per look-back group
constexpr int kGroupWindow = 8;             // groups read per look-back step
constexpr uint32_t kFlag = 1u << 31;        // word published (tile counts, group prefixes)
constexpr uint32_t kValueMask = (1u << 30) - 1;
constexpr uint32_t kArrival = 1u << 24;     // group sums: one arrival; the sum (at most kGroup tiles) below it
static_assert(kGroup * kThreads * 16 < (1 << 24) && kGroup < 128, "group sums and arrivals share a word");

__device__ __forceinline__ int64_t read_count(int64_t n_host, const uint32_t* d_n) {
    return d_n ? (int64_t)(*d_n) : n_host;
}

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t x) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

// Exclusive scan across a block of NT threads (NT <= 1024); returns the
// thread's exclusive prefix, `total` gets the block sum. Uses s_warp[33]:
// [0, 32) the warps' exclusive prefixes, [32] the total (kept apart so a
// 32-warp block does not overwrite warp 31's prefix with it).
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

// Look-back words of one pass: per tile its digit counts, then per group the
// (inclusive prefix, sum and arrivals) pairs. A single tile has none.
struct StatusLayout {
    int64_t tiles, groups;
    int64_t pass_words;  // words of one pass
};
template <int BITS>
__host__ __device__ inline StatusLayout status_layout(int64_t cap, int tile_keys) {
    StatusLayout l;
    l.tiles = (cap + tile_keys - 1) / tile_keys;
    if (l.tiles == 1) l.tiles = 0;
    l.groups = (l.tiles + kGroup - 1) / kGroup;
    l.pass_words = (l.tiles + 2 * l.groups) << BITS;
    return l;
}

// Clears the passes' tile counters and the look-back words of n elements (thread
// t0 of dt).
template <int BITS>
__device__ __forceinline__ void clear_status(int64_t n, int64_t cap, int tile_keys, int passes,
                                             uint32_t* __restrict__ counters, uint32_t* __restrict__ status,
                                             int64_t t0, int64_t dt) {
    if (t0 < kMaxSortPasses) counters[t0] = 0;
    const StatusLayout full = status_layout<BITS>(cap, tile_keys), used = status_layout<BITS>(n, tile_keys);
    for (int p = 0; p < passes; ++p) {
        uint32_t* st = status + p * full.pass_words;
        for (int64_t i = t0; i < used.tiles << BITS; i += dt) st[i] = 0;
        uint32_t* gr = st + (full.tiles << BITS);
        for (int64_t i = t0; i < (2 * used.groups) << BITS; i += dt) gr[i] = 0;
    }
}

// Digit counts of every pass with one read of the keys; clears the tile
// counters and the look-back words the passes will use.
template <int BITS>
__global__ void __launch_bounds__(kThreads) k_digit_hist(const uint32_t* __restrict__ keys, int64_t n_host,
                                                         const uint32_t* d_n, int passes,
                                                         uint32_t* __restrict__ ghist,
                                                         uint32_t* __restrict__ counters,
                                                         uint32_t* __restrict__ status, int64_t cap, int tile_keys) {
    dependency_sync(keys, d_n);
    constexpr int BINS = 1 << BITS;
    __shared__ uint32_t s_h[kMaxSortPasses * BINS];
    const int64_t n = read_count(n_host, d_n);
    for (int i = threadIdx.x; i < passes * BINS; i += kThreads) s_h[i] = 0;
    clear_status<BITS>(n, cap, tile_keys, passes, counters, status, (int64_t)blockIdx.x * kThreads + threadIdx.x,
                       (int64_t)gridDim.x * kThreads);
    __syncthreads();
    // Eight independent loads in flight per thread before the shared-memory
    // counting (one load at a time leaves the kernel waiting on latency).
    constexpr int U = 8;
    const int64_t stride = (int64_t)gridDim.x * kThreads;
    for (int64_t i0 = (int64_t)blockIdx.x * kThreads + threadIdx.x; i0 < n; i0 += U * stride) {
        uint32_t k[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t i = i0 + u * stride;
            k[u] = i < n ? keys[i] : 0u;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (i0 + u * stride >= n) break;
            for (int p = 0; p < passes; ++p)
                atomicAdd(&s_h[p * BINS + ((k[u] >> (p * BITS)) & (BINS - 1))], 1u);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < passes * BINS; i += kThreads)
        if (s_h[i]) atomicAdd(&ghist[i], s_h[i]);
}

__device__ __forceinline__ uint32_t ld_relaxed(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ uint2 ld_relaxed2(const uint2* p) {
    uint2 v;
    asm volatile("ld.relaxed.gpu.global.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_relaxed(uint32_t* p, uint32_t v) {
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// The same for many keys: every lane counts in a column of its own, so that an
// increment never meets another lane's in a bank (32 random digits do: 3.4
// shared-memory passes an increment), 16-byte key loads, and the columns are
// added up once per block.
// 32 M keys, four 7-bit digits 67 -> 48 us; 62 M, four 8-bit digits 125 -> 98 us; 77 M,
// two 9-bit digits 119 -> 98 us; 4 M 17.2 -> 14.9 us; 0.9 M 10.0 against 10.3 us and
// 20 k 8.5 against 10.0 us (clearing and adding up the columns): from 1 Mi keys on.
constexpr int kWideThreads = 1024;
constexpr int64_t kWideExpect = 1 << 20;
template <int BITS>
__global__ void __launch_bounds__(kWideThreads) k_digit_hist_wide(const uint32_t* __restrict__ keys, int64_t n_host,
                                                                  const uint32_t* d_n, int passes,
                                                                  uint32_t* __restrict__ ghist,
                                                                  uint32_t* __restrict__ counters,
                                                                  uint32_t* __restrict__ status, int64_t cap,
                                                                  int tile_keys) {
    dependency_sync(keys, d_n);
    constexpr int BINS = 1 << BITS;
    extern __shared__ __align__(128) uint32_t s_col[];  // [passes][BINS][32]
    const int64_t n = read_count(n_host, d_n);
    const int tid = threadIdx.x, lane = tid & 31;
    for (int i = tid; i < passes * BINS * 8; i += kWideThreads)
        reinterpret_cast<uint4*>(s_col)[i] = make_uint4(0u, 0u, 0u, 0u);
    const int64_t t0 = (int64_t)blockIdx.x * kWideThreads + tid, dt = (int64_t)gridDim.x * kWideThreads;
    clear_status<BITS>(n, cap, tile_keys, passes, counters, status, t0, dt);
    __syncthreads();
    auto count = [&](uint32_t k) {
#pragma unroll
        for (int p = 0; p < kMaxSortPasses; ++p)
            if (p < passes) atomicAdd(&s_col[((p * BINS + ((k >> (p * BITS)) & (BINS - 1))) << 5) + lane], 1u);
    };
    const int64_t n4 = n / 4;  // whole 16-byte vectors
    const uint4* k4 = reinterpret_cast<const uint4*>(keys);
    int64_t i = t0;
    for (; i + dt < n4; i += 2 * dt) {  // two vectors in flight
        const uint4 a = k4[i], b = k4[i + dt];
        count(a.x); count(a.y); count(a.z); count(a.w);
        count(b.x); count(b.y); count(b.z); count(b.w);
    }
    if (i < n4) {
        const uint4 a = k4[i];
        count(a.x); count(a.y); count(a.z); count(a.w);
    }
    if (t0 < n - 4 * n4) count(keys[4 * n4 + t0]);
    __syncthreads();
    for (int b = tid; b < passes * BINS; b += kWideThreads) {
        uint32_t sum = 0;
#pragma unroll 8
        for (int c = 0; c < 32; ++c) sum += s_col[(b << 5) + ((c + lane) & 31)];
        if (sum) atomicAdd(&ghist[b], sum);
    }
}

// Counts of one digit over all tiles before `tile` (look-back). status points
// at the digit's word of tile 0, groups at its pair of group 0; rows are BINS
// apart. The words of the tiles before it in its group and of the nearest
// groups are read in one round; whole groups are then added nearest first
// until one has its inclusive prefix. Gives up after `limit` polls: the
// partial sum, with *err raised.
template <int BINS>
__device__ __forceinline__ uint32_t look_back(int64_t tile, const uint32_t* status, const uint2* groups,
                                              uint32_t limit, uint32_t* err) {
    const int left = (int)(tile & (kGroup - 1));
    const uint32_t* st = status + (tile - left) * BINS;
    int64_t q = tile / kGroup - 1;  // next group to add
    uint32_t spins = 0, sum = 0, own = 0;
    bool own_done = left == 0;
    for (;;) {
        uint32_t w[kGroup - 1];
        uint2 g[kGroupWindow];
        if (!own_done) {
#pragma unroll
            for (int j = 0; j < kGroup - 1; ++j) w[j] = j < left ? ld_relaxed(st + j * BINS) : kFlag;
        }
        if (q >= 0) {
#pragma unroll
            for (int j = 0; j < kGroupWindow; ++j)
                g[j] = q - j >= 0 ? ld_relaxed2(groups + (q - j) * BINS) : make_uint2(kFlag, 0u);
        }
        bool waits = false;  // a word that is not there yet
        if (!own_done) {
            uint32_t all = kFlag;
            own = 0;
#pragma unroll
            for (int j = 0; j < kGroup - 1; ++j) {
                all &= w[j];
                own += w[j] & kValueMask;
            }
            own_done = all != 0u;
            waits = !own_done;
        }
        if (q >= 0) {
            bool open = true;
#pragma unroll
            for (int j = 0; j < kGroupWindow; ++j) {
                if (!open) continue;
                if (g[j].x & kFlag) {
                    sum += g[j].x & kValueMask;
                    q = -1;
                    open = false;
                } else if (g[j].y >= kGroup * kArrival) {
                    sum += g[j].y & (kArrival - 1);
                    --q;
                } else {
                    waits = true;
                    open = false;
                }
            }
        }
        if (own_done && q < 0) return sum + own;
        if (waits) {
            if (++spins > limit) {
                atomicOr(err, kErrTimeout);
                return sum + own;
            }
            __nanosleep(20);
        }
    }
}

template <int BITS, int IPT>
constexpr size_t sweep_smem() {
    return 128 + sizeof(uint32_t) * (3 * kThreads * IPT + (2 * kWarps + 2) * (1 << BITS));
}

// What a sweep moves with its keys.
enum SweepKind {
    kPairs = 0,     // values as they are
    kIdentity = 1,  // the input values are their positions (not read from memory)
    kCarryIn = 2,   // first depth pass: the values are positions, their rects are read and packed with them
    kCarryOut = 3   // last depth pass: writes the point indices and the rects
};

// A key and a value as the first pass of a sort that carries rects writes
// them: the key without its first digit below the code's low bits, the index
// within the image below the code's high bits.
__device__ __forceinline__ uint2 carry_pack(const RectCarry& rc, uint32_t key, uint32_t gi, uint32_t code) {
    const uint32_t off = rc.img_bits ? rc.img_off[key >> rc.img_shift] : 0u;
    return make_uint2((key >> rc.first_bits) | (code << rc.rem_bits),
                      (gi - off) | ((code >> (32 - rc.rem_bits)) << rc.idx_bits));
}

__device__ __forceinline__ void carry_unpack(const RectCarry& rc, uint32_t k, uint32_t v, uint32_t& gi, uint32_t& code) {
    const uint32_t rem = k & ((1u << rc.rem_bits) - 1u);
    const uint32_t off = rc.img_bits ? rc.img_off[rem >> (rc.rem_bits - rc.img_bits)] : 0u;
    gi = (v & ((1u << rc.idx_bits) - 1u)) + off;
    code = ((k >> rc.rem_bits) | ((v >> rc.idx_bits) << (32 - rc.rem_bits))) & ((1u << rc.bits) - 1u);
}

// Tiles arrive by TMA bulk copies, one for the keys and one for the values,
// into three shared buffers that change roles from tile to tile: the keys are
// read into registers and sorted in place, the values go from their buffer to
// the spare one, the next tile's keys are fetched into the emptied values
// buffer while this tile is written out, and its values into the spare one
// after that. No thread holds values or waits on a global load.
//
// Bound by the L1 data pipe (about one shared-memory wavefront a key: counting,
// ranking and scattering by digit; 74 % of its cycles on 8 M keys), then by the integer
// pipe. The ranking takes the lane masks of every other round from ballots
// (integer pipe) and of the rounds between from a shared atomic OR (memory
// pipe): all rounds from ballots were 172 us, all from the OR 159 us, both in
// turn 151 us a pass over 32 M keys. Three CTAs on an SM (80 registers, 57 KB)
// with the next tile on its way beat four without: 147 us. The whole pass went
// 217 -> 147 us (32 M keys, 7-bit digits; 3.6 TB/s moved), 36.6 -> 27 us (4 M
// keys), 433 -> 322 us (62 M keys, 8-bit), 630 -> 493 us (77 M keys, 9-bit; a thread's
// two bins 256 apart: 553 us with neighbouring ones, whose counters share banks).
// Carrying the tile rects costs the 32 M depth passes 147 -> 163 us (sum 65 us) and
// saves the duplication's random gather of them (0.33 -> 0.03 ms).
template <int BITS, int IPT, int KIND>
__global__ void __launch_bounds__(kThreads, IPT == 16 ? 3 : 4) k_sweep(
    const uint32_t* __restrict__ kin, const uint32_t* __restrict__ vin, uint32_t* __restrict__ kout,
    uint32_t* __restrict__ vout, int64_t n_host, const uint32_t* d_n, int64_t cap, int shift,
    uint32_t mask, const uint32_t* __restrict__ ghist_pass, uint32_t* __restrict__ counter,
    uint32_t* __restrict__ status, uint32_t* __restrict__ err, int stall, const CarryIo carry) {
    dependency_sync(ghist_pass, err, d_n);
    constexpr bool IDV = KIND == kIdentity;
    constexpr int BINS = 1 << BITS;
    constexpr int VPT = BINS > kThreads ? BINS / kThreads : 1;  // bins per thread: tid, tid + kThreads
    constexpr int TILE = kThreads * IPT;
    extern __shared__ __align__(128) uint32_t s_dyn[];
    uint32_t* s_k = align128(s_dyn);  // TILE: the tile's keys, then its keys in digit order
    uint32_t* s_v = s_k + TILE;       // TILE: the tile's values, then the next tile's keys
    uint32_t* s_s = s_v + TILE;       // TILE: values in digit order, then the next tile's values
    uint2* const s_tab = reinterpret_cast<uint2*>(s_s + TILE);  // kWarps * BINS: (lanes, count, then running position)
    uint32_t* const s_goff = reinterpret_cast<uint32_t*>(s_tab + kWarps * BINS);  // BINS: global digit starts
    uint32_t* const s_ofs = s_goff + BINS;                      // BINS: global minus tile-local digit start
    __shared__ uint32_t s_warp[33];
    __shared__ uint32_t s_tile;
    __shared__ __align__(8) uint64_t s_mbar[2];  // keys arrived, values arrived
    // A pass after one whose look-back wait ran out does nothing: its input
    // is a partial order whose digit counts no longer match the histogram,
    // so its scatter positions could leave the buffers. (Within the pass that
    // gave up, a partial prefix only lowers positions: they stay in [0, n).)
    if (__syncthreads_or((*err & kErrTimeout) != 0u)) return;
    const int64_t n = read_count(n_host, d_n);
    const int64_t ntiles = (n + TILE - 1) / TILE;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t lt = lanemask_lt();
    uint2* const groups = reinterpret_cast<uint2*>(status + (status_layout<BITS>(cap, TILE).tiles << BITS));
    uint2* const tab = s_tab + warp * BINS;
    const int w0 = warp * (32 * IPT) + lane;  // this lane's first key in a tile

    // One bulk copy of tile t's words (rounded up to 16 bytes: the arrays are
    // padded to 256), by thread 0.
    auto fetch = [&](uint32_t* dst, const uint32_t* src, int64_t t, uint64_t* bar) {
        const int64_t left = n - t * TILE;
        const uint32_t words = ((uint32_t)(left < TILE ? left : TILE) + 3u) & ~3u;
        bulk_copy_g2s(dst, src + t * TILE, words * 4u, bar);
    };
    if (tid == 0) {
        mbar_init(&s_mbar[0], 1);
        mbar_init(&s_mbar[1], 1);
        mbar_init_fence();
        s_tile = atomicAdd(counter, 1u);
        if (s_tile < ntiles) {
            // (test hooks: the first tile's keys or values never arrive)
            if (stall != kStallKeys || s_tile != 0) fetch(s_k, kin, s_tile, &s_mbar[0]);
            if (!IDV && (stall != kStallValues || s_tile != 0)) fetch(s_v, vin, s_tile, &s_mbar[1]);
        }
    }
    // Global start of every digit in this pass.
    {
        uint32_t before = 0;
#pragma unroll
        for (int q = 0; q < VPT; ++q) {
            const int bin = tid + q * kThreads;
            uint32_t all;
            const uint32_t ex = block_excl_scan<kThreads>(bin < BINS ? ghist_pass[bin] : 0u, s_warp, all);
            if (bin < BINS) s_goff[bin] = before + ex;
            before += all;
        }
    }
    __syncthreads();
    int64_t tile = s_tile;
    uint32_t phase = 0;
    const uint32_t limit = stall ? 64u : (1u << 22);
    while (tile < ntiles) {
        const int64_t base = tile * TILE;
        const int cnt = (int)(n - base < TILE ? n - base : TILE);
#pragma unroll
        for (int i = 0; i < (BINS + 31) / 32; ++i)
            if (i * 32 + lane < BINS) tab[i * 32 + lane] = make_uint2(0u, 0u);
        const uint32_t key_polls = stall == kStallKeys && tile == 0 ? 64u : kMbarPolls;
        const uint32_t val_polls = stall == kStallValues && tile == 0 ? 64u : kMbarPolls;
        bool failed = !mbar_wait(&s_mbar[0], phase, key_polls);
        // Keys past the end are all ones: they have the highest digit and come
        // last in input order, so they rank behind every real key.
        uint32_t k[IPT];
        if (cnt == TILE) {
#pragma unroll
            for (int r = 0; r < IPT; ++r) k[r] = s_k[w0 + r * 32];
        } else {
#pragma unroll
            for (int r = 0; r < IPT; ++r) k[r] = w0 + r * 32 < cnt ? s_k[w0 + r * 32] : 0xffffffffu;
        }
        __syncwarp();
#pragma unroll
        for (int r = 0; r < IPT; ++r) atomicAdd(&tab[(k[r] >> shift) & mask].y, 1u);
        if (__syncthreads_or(failed)) {  // a copy never arrived: report it, let the other land, stop
            if (tid == 0) atomicOr(err, kErrTimeout);
            mbar_wait(&s_mbar[0], phase, key_polls);
            if (!IDV) mbar_wait(&s_mbar[1], phase);
            break;
        }

        // Publish the tile's counts (test hook: with kStallCounts the first tile
        // publishes nothing, so its successor's wait runs out), and turn the
        // warps' counts into tile-local positions (digit, then warp).
        const bool publish = ntiles > 1 && !(stall == kStallCounts && tile == 0);
        uint32_t tot[VPT];           // the tile's count of this thread's bins, keys past the end left out
        uint32_t c[VPT][kWarps];     // each warp's count
        uint32_t local[VPT], inc[VPT];  // all of them, and their sums over the warp's lanes
#pragma unroll
        for (int q = 0; q < VPT; ++q) {
            const int bin = tid + q * kThreads;
            uint32_t sum = 0;
            if (bin < BINS) {
#pragma unroll
                for (int w = 0; w < kWarps; ++w) {
                    c[q][w] = s_tab[w * BINS + bin].y;
                    sum += c[q][w];
                }
                tot[q] = sum - (bin == (int)mask ? (uint32_t)(TILE - cnt) : 0u);
                if (publish) {
                    st_relaxed(status + tile * BINS + bin, kFlag | tot[q]);
                    atomicAdd(&groups[(tile / kGroup) * BINS + bin].y, kArrival | tot[q]);
                }
            }
            local[q] = sum;
            inc[q] = warp_incl_scan(sum);
            if (lane == 31) s_warp[q * kWarps + warp] = inc[q];
        }
        __syncthreads();
        uint32_t start[VPT], before = 0;
#pragma unroll
        for (int q = 0; q < VPT; ++q) {
            const int bin = tid + q * kThreads;
            uint32_t run = before + inc[q] - local[q];
#pragma unroll
            for (int w = 0; w < kWarps; ++w) {
                const uint32_t x = s_warp[q * kWarps + w];
                run += w < warp ? x : 0u;
                before += x;
            }
            start[q] = run;
            if (bin < BINS) {
#pragma unroll
                for (int w = 0; w < kWarps; ++w) {
                    s_tab[w * BINS + bin].y = run;
                    run += c[q][w];
                }
            }
        }
        if (!IDV) failed = !mbar_wait(&s_mbar[1], phase, val_polls);
        if (__syncthreads_or(failed)) {
            if (tid == 0) atomicOr(err, kErrTimeout);
            mbar_wait(&s_mbar[1], phase, val_polls);
            break;
        }
        phase ^= 1u;

        // Stable rank: rounds in input order, lanes in order within a round.
#pragma unroll
        for (int r = 0; r < IPT; ++r) {
            const uint32_t d = (k[r] >> shift) & mask;
            uint32_t peers, pre;  // lanes holding the same digit; the digit's next position
            if (r & 1) {
                peers = 0xffffffffu;
#pragma unroll
                for (int bb = 0; bb < BITS; ++bb) {
                    const bool set = (d >> bb) & 1u;
                    const uint32_t m = __ballot_sync(0xffffffffu, set);
                    peers &= set ? m : ~m;
                }
                pre = tab[d].y;
            } else {
                atomicOr(&tab[d].x, 1u << lane);
                __syncwarp();
                const uint2 t = tab[d];
                peers = t.x;
                pre = t.y;
            }
            const uint32_t below = __popc(peers & lt);
            __syncwarp();
            if (below == 0) tab[d] = make_uint2(0u, pre + __popc(peers));
            __syncwarp();
            s_k[pre + below] = k[r];
            uint32_t v;
            if constexpr (KIND == kIdentity) {
                v = (uint32_t)base + (uint32_t)(w0 + r * 32);
            } else {
                v = s_v[w0 + r * 32];
                if constexpr (KIND == kCarryIn) {
                    // the rect's code and the key's position in the tile
                    if (!carry.coded)
                        v = v == kRect4Empty ? rect_code_empty(carry.rc)
                                             : rect_code(carry.rc, v & 0xffffu, (v >> 16) & 0x3fffu, (v >> 30) & 1u, v >> 31);
                    v = (v << 12) | (uint32_t)(w0 + r * 32);
                }
            }
            s_s[pre + below] = v;
        }
        // The next tile is taken before the look-back and its keys are fetched
        // while this one is written out. (Every wait is on tiles taken earlier,
        // whose counts are published before any wait of theirs: the look-backs
        // still end.)
        uint32_t next = 0;
        if (tid == 0) next = atomicAdd(counter, 1u);
#pragma unroll
        for (int q = 0; q < VPT; ++q) {
            const int bin = tid + q * kThreads;
            if (bin >= BINS) continue;
            const uint32_t excl = look_back<BINS>(tile, status + bin, groups + bin, limit, err);
            if ((tile & (kGroup - 1)) == kGroup - 1)  // more than one tile
                st_relaxed(&groups[(tile / kGroup) * BINS + bin].x, kFlag | (excl + tot[q]));
            s_ofs[bin] = s_goff[bin] + excl - start[q];
        }
        if (tid == 0) s_tile = next;
        fence_proxy_async();  // this thread's accesses to the buffers come before the copies into them
        __syncthreads();
        tile = s_tile;
        if (tid == 0 && tile < ntiles) fetch(s_v, kin, tile, &s_mbar[0]);

        auto put = [&](uint32_t key, uint32_t val, uint32_t dst) {
            if constexpr (KIND == kCarryIn) {
                const uint2 e = carry_pack(carry.rc, key, (uint32_t)base + (val & 4095u), val >> 12);
                kout[dst] = e.x;
                vout[dst] = e.y;
            } else if constexpr (KIND == kCarryOut) {
                const RectCarry& rc = carry.rc;
                uint32_t gi, code;
                carry_unpack(rc, key, val, gi, code);
                vout[dst] = gi;
                const uint32_t tx0 = code & ((1u << rc.tx_bits) - 1u), ty0 = (code >> rc.tx_bits) & ((1u << rc.ty_bits) - 1u);
                const uint32_t span = code >> (rc.tx_bits + rc.ty_bits);
                if (!carry.coded) {
                    static_cast<uint32_t*>(carry.out)[dst] =
                        code == rect_code_empty(rc) ? kRect4Empty : tx0 | (ty0 << 16) | (span << 30);
                } else {
                    uint2 q = make_uint2(1u, 0u);
                    if (code != rect_code_empty(rc)) {
                        const uint32_t w = span & 3u, h = span >> 2;
                        q = w == 3u ? ((int64_t)gi < n ? carry.full[gi] : q)
                                    : make_uint2(tx0 | (ty0 << 16), (tx0 + w) | ((ty0 + h) << 16));
                    }
                    static_cast<uint2*>(carry.out)[dst] = q;
                }
            } else {
                if (kout) kout[dst] = key;
                vout[dst] = val;
            }
        };
        if (cnt == TILE) {
            constexpr int U = 4;
#pragma unroll 1
            for (int j0 = tid; j0 < TILE; j0 += U * kThreads) {
                uint32_t key[U], val[U], dst[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    key[u] = s_k[j0 + u * kThreads];
                    val[u] = s_s[j0 + u * kThreads];
                }
#pragma unroll
                for (int u = 0; u < U; ++u)
                    dst[u] = s_ofs[(key[u] >> shift) & mask] + (uint32_t)(j0 + u * kThreads);
#pragma unroll
                for (int u = 0; u < U; ++u) put(key[u], val[u], dst[u]);
            }
        } else {
            for (int j = tid; j < cnt; j += kThreads) {
                const uint32_t key = s_k[j];
                const uint32_t dst = s_ofs[(key >> shift) & mask] + (uint32_t)j;
                put(key, s_s[j], dst);
            }
        }
        fence_proxy_async();
        __syncthreads();  // the tile's keys, values and offsets are read
        if (!IDV && tid == 0 && tile < ntiles) fetch(s_s, vin, tile, &s_mbar[1]);
        uint32_t* const free_buf = s_k;
        s_k = s_v;
        s_v = s_s;
        s_s = free_buf;
    }
}

// Keys per thread of the sweeps, by the count a sort is expected to have: tiles
// of 4096 keys, which spend the least on counts and look-back (4 M points 27.3
// us a pass, with 1024-key tiles 42.3 us; 500 k points 10.8 against 12.8 us),
// unless so few keys would occupy only a part of the SMs (20 k points 8.7
// against 10.1 us, 60 k points 9.3 against 10.4 us). Copies are counted on the
// device and can be far more than expected (large Gaussians), up to the
// capacity: small tiles only below 2 Mi, where they cost little if so (both
// tile sort passes of 0.12 M Gaussians, small / large tiles: 0.2 M copies 34 / 38
// us, 1.4 M 53 / 42 us, 4.4 M 119 / 73 us, 9.5 M 237 / 115 us).
int sweep_ipt(int64_t expect, int64_t cap) { return expect <= 256 * 1024 && cap <= 2 * 1024 * 1024 ? 4 : 16; }

template <int BITS, int IPT>
cudaError_t sort_t(uint32_t* keys[2], uint32_t* vals[2], int64_t n, const uint32_t* d_n, int64_t cap, int64_t expect,
                   const SortPlan& plan, const SortScratch& sc, cudaStream_t s, int* result_buf,
                   const char* const names[2], bool identity_vals, bool keys_out, const CarryIo* carry) {
    constexpr int BINS = 1 << BITS;
    constexpr int TILE = kThreads * IPT;
    // Launch attributes and the resident CTAs per SM of the sweep, once per
    // device: persistent grid = as many CTAs as fit on the GPU at once (every
    // CTA resident, so a look-back never waits on a tile no running CTA holds).
    static PerDevice setup;
    constexpr size_t smem = sweep_smem<BITS, IPT>();
    int per_sm = 1;
    cudaError_t e = per_device(setup, &per_sm, [](int, int* v) {
        *v = 1;
        cudaError_t r = cudaSuccess;
        for (auto kern : {k_sweep<BITS, IPT, kPairs>, k_sweep<BITS, IPT, kIdentity>, k_sweep<BITS, IPT, kCarryIn>,
                          k_sweep<BITS, IPT, kCarryOut>})
            if (r == cudaSuccess)
                r = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (r != cudaSuccess) return r;
        int occ = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_sweep<BITS, IPT, kPairs>, kThreads, smem) ==
                cudaSuccess && occ >= 1)
            *v = occ;
        return cudaSuccess;
    });
    if (e != cudaSuccess) return e;
    const StatusLayout sl = status_layout<BITS>(cap, TILE);
    const int sms = device_sm_count();
    {
        ProfScope ps(names[0], s);
        if (expect >= kWideExpect) {
            const size_t cols = (size_t)plan.passes * BINS * 32 * sizeof(uint32_t);
            static PerDevice wide;
            e = per_device(wide, nullptr, [](int, int*) {
                return cudaFuncSetAttribute(k_digit_hist_wide<BITS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)(kSortHistWords * 32 * sizeof(uint32_t)));
            });
            if (e != cudaSuccess) return e;
            const int per_sm = cols <= 64 * 1024 ? 2 : 1;  // 2048 threads an SM; 228 KB
            e = launch_dependent(k_digit_hist_wide<BITS>, (unsigned)(sms * per_sm), kWideThreads, cols, s, keys[0], n, d_n,
                                 plan.passes, sc.ghist, sc.counters, sc.status, cap, TILE);
            if (e != cudaSuccess) return e;
        } else {
            int64_t g = (cap + kThreads * 16 - 1) / (kThreads * 16);
            if (g > (int64_t)sms * 4) g = (int64_t)sms * 4;
            if (g < 1) g = 1;
            e = launch_dependent(k_digit_hist<BITS>, (unsigned)g, kThreads, 0, s, keys[0], n, d_n, plan.passes, sc.ghist,
                                 sc.counters, sc.status, cap, TILE);
            if (e != cudaSuccess) return e;
        }
    }
    const int64_t resident = (int64_t)sms * per_sm;
    const int64_t tiles = sl.tiles > 0 ? sl.tiles : 1;
    const unsigned gs = (unsigned)(tiles < resident ? tiles : resident);
    int cur = 0;
    for (int k = 0; k < plan.passes; ++k) {
        ProfScope ps(names[1], s);
        const bool last = k + 1 == plan.passes;
        auto kern = k_sweep<BITS, IPT, kPairs>;
        const uint32_t* vin = vals[cur];
        int shift = plan.shift[k];
        uint32_t mask = BINS - 1;
        if (carry) {
            // after the first pass the key's first digit is gone, and other bits stand above the key
            const int left = plan.bits - plan.shift[k];
            if (left < BITS) mask = (1u << left) - 1u;
            if (k > 0) shift -= plan.digit_bits[0];
            if (k == 0) vin = carry->in;
            if (k == 0) kern = k_sweep<BITS, IPT, kCarryIn>;
            else if (last) kern = k_sweep<BITS, IPT, kCarryOut>;
        } else if (k == 0 && identity_vals) {
            kern = k_sweep<BITS, IPT, kIdentity>;
        }
        uint32_t* kout = (last && !keys_out) ? nullptr : keys[cur ^ 1];
        e = launch_dependent(kern, gs, kThreads, smem, s, keys[cur], vin, kout, vals[cur ^ 1], n, d_n, cap, shift, mask,
                             sc.ghist + k * BINS, sc.counters + k, sc.status + k * sl.pass_words, sc.err,
                             k == 0 ? sc.stall : (int)kNoStall, carry ? *carry : CarryIo{});
        if (e != cudaSuccess) return e;
        cur ^= 1;
    }
    *result_buf = cur;
    return cudaSuccess;
}

template <int BITS>
cudaError_t sort_b(uint32_t* keys[2], uint32_t* vals[2], int64_t n, const uint32_t* d_n, int64_t cap, int64_t expect,
                   const SortPlan& plan, const SortScratch& sc, cudaStream_t s, int* result_buf,
                   const char* const names[2], bool identity_vals, bool keys_out, const CarryIo* carry) {
    if (sweep_ipt(expect, cap) == 4)
        return sort_t<BITS, 4>(keys, vals, n, d_n, cap, expect, plan, sc, s, result_buf, names, identity_vals, keys_out, carry);
    return sort_t<BITS, 16>(keys, vals, n, d_n, cap, expect, plan, sc, s, result_buf, names, identity_vals, keys_out, carry);
}

}  // namespace

SortPlan make_sort_plan(int bits) {
    SortPlan p{};
    if (bits <= 0) {
        p.passes = 0;
        return p;
    }
    // Up to 9-bit digits for short keys (tile ids); 7-bit digits for long keys
    // (depth): measured, four 7-bit passes over 27-bit depth keys beat three
    // 9-bit ones (4.4 against 6.4 ps a key and pass: four times the counts to
    // publish and look back for, shorter runs, fewer CTAs per SM).
    // Keys wider than 28 bits (a far/near ratio beyond about 2^29) take four
    // wider digits: the scratch buffers hold at most kMaxSortPasses passes.
    int passes = bits > 18 ? (bits + 6) / 7 : (bits + 8) / 9;
    if (passes > kMaxSortPasses) passes = kMaxSortPasses;
    int per = (bits + passes - 1) / passes;
    if (per < 4) per = 4;
    int shift = 0;
    for (int k = 0; k < passes; ++k) {
        p.digit_bits[k] = per;
        p.shift[k] = shift;
        shift += per;
    }
    p.passes = passes;
    p.bits = bits;
    return p;
}

int64_t sort_status_words(const SortPlan& plan, int64_t cap, int64_t expect) {
    if (plan.passes == 0) return 0;
    const StatusLayout l = status_layout<0>(cap, kThreads * sweep_ipt(expect, cap));
    return plan.passes * (l.pass_words << plan.digit_bits[0]);
}

cudaError_t radix_sort(uint32_t* keys[2], uint32_t* vals[2], int64_t n, const uint32_t* d_n, int64_t cap,
                       int64_t expect, const SortPlan& plan, const SortScratch& sc, cudaStream_t s, int* result_buf,
                       const char* const names[2], bool identity_vals, bool keys_out, const CarryIo* carry) {
    *result_buf = 0;
    if (plan.passes == 0 || cap == 0) return cudaSuccess;
    if (plan.passes > kMaxSortPasses) return cudaErrorInvalidValue;
    switch (plan.digit_bits[0]) {
        case 4: return sort_b<4>(keys, vals, n, d_n, cap, expect, plan, sc, s, result_buf, names, identity_vals, keys_out, carry);
        case 5: return sort_b<5>(keys, vals, n, d_n, cap, expect, plan, sc, s, result_buf, names, identity_vals, keys_out, carry);
        case 6: return sort_b<6>(keys, vals, n, d_n, cap, expect, plan, sc, s, result_buf, names, identity_vals, keys_out, carry);
        case 7: return sort_b<7>(keys, vals, n, d_n, cap, expect, plan, sc, s, result_buf, names, identity_vals, keys_out, carry);
        case 8: return sort_b<8>(keys, vals, n, d_n, cap, expect, plan, sc, s, result_buf, names, identity_vals, keys_out, carry);
        case 9: return sort_b<9>(keys, vals, n, d_n, cap, expect, plan, sc, s, result_buf, names, identity_vals, keys_out, carry);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace rast
