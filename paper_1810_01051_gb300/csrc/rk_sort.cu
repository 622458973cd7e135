// A6: ascending order of the match keys key = (id << 40) | x, which is the
// ascending (pattern id, offset) order the match list is defined in.
//
// Up to 32 tiles of 2048 keys per resident CTA: one cooperative launch that
// sorts by cells (sort_cells below): the keys' bits that can be non-zero, as
// one compact number, are cut into a few cells per key by their top bits;
// the keys are counted and ranked per cell, scattered to their cell, and put
// in order within it by comparison.  Keys crowded into few cells (kCrowdedMean)
// are sorted by the radix passes below instead, in the same launch.
//
// Radix passes: least significant digit first over 8-bit digits, only those
// that can be non-zero: those of the offset field (bits below ceil(log2(n)))
// and of the id field (bits 40.. up to ceil(log2(k))).  Above the cooperative
// launch's size:
//   1. one histogram kernel reads the keys once and counts every pass's
//      digits (the totals do not depend on the order), and clears the
//      per-tile status words of the passes;
//   2. one kernel per pass: each CTA takes the next tile of 2048 keys from a
//      counter, ranks its keys stably (ballot multisplit + per-warp digit counters),
//      publishes its digit counts, adds up the counts of the tiles before it
//      by looking back through their published words (decoupled look-back),
//      and scatters.  Look-back waits are bounded: a wait that runs out
//      records RK_ETIMEOUT in d_info[1].
//
// Every kernel reads the key count from d_info on the device, so nothing
// returns to the host between the scan and the sorted list.
#include <algorithm>
#include <mutex>

#include "rk_internal.cuh"
#include "rk_sortws.cuh"

namespace rk {
namespace {

constexpr uint32_t kThreads = 256;
constexpr uint32_t kWarps = kThreads / 32;
constexpr uint32_t kPerWarp = kSortTile / kWarps;  // 512 consecutive keys per warp
constexpr uint64_t kFlagAgg = 1ull << 62;          // tile's own counts published
constexpr uint64_t kFlagInc = 2ull << 62;          // inclusive prefix published
constexpr uint64_t kCountMask = (1ull << 62) - 1;
constexpr uint64_t kLookbackTimeoutNs = 2000000000ull;

__device__ __forceinline__ bool sort_count(const unsigned long long *info, uint64_t cap,
                                           uint64_t *m, uint32_t *tiles) {
    const uint64_t M = info[0];
    if (M > cap || M < 2 || info[1] != RK_OK) return false;
    *m = M;
    *tiles = (uint32_t)((M + kSortTile - 1) / kSortTile);
    return true;
}

// Lanes holding a valid key whose 8-bit digit equals this lane's: one ballot
// per digit bit, a fixed cost whatever the number of distinct digits (a
// warp match instruction takes longer the more distinct values there are).
__device__ __forceinline__ uint32_t digit_peers(uint32_t d, bool valid) {
    uint32_t peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
    for (uint32_t b = 0; b < 8; ++b) {
        const bool bit = (d >> b) & 1u;
        const uint32_t bal = __ballot_sync(0xffffffffu, bit);
        peers &= bit ? bal : ~bal;
    }
    return peers;
}

struct Shifts {
    uint32_t s[kMaxSortPasses];
    uint32_t n;
};

__global__ void __launch_bounds__(kThreads) rk_sort_hist_kernel(const uint64_t *keys,
                                                                const unsigned long long *info,
                                                                uint64_t cap, Shifts sh,
                                                                uint32_t *ghist,
                                                                uint64_t *status,
                                                                uint64_t tiles_max) {
    uint64_t M;
    uint32_t T;
    if (!sort_count(info, cap, &M, &T)) return;
    __shared__ uint32_t h[kMaxSortPasses][256];
    for (uint32_t p = 0; p < sh.n; ++p) h[p][threadIdx.x] = 0;
    __syncthreads();
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < M; i += stride) {
        const uint64_t k = keys[i];
        for (uint32_t p = 0; p < sh.n; ++p) atomicAdd(&h[p][(uint32_t)(k >> sh.s[p]) & 255u], 1u);
    }
    // clear the look-back words of every pass (tiles actually used)
    const uint64_t per_pass = (uint64_t)T * 256u;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < sh.n * per_pass;
         i += stride)
        status[(i / per_pass) * tiles_max * 256u + i % per_pass] = 0;
    __syncthreads();
    for (uint32_t p = 0; p < sh.n; ++p)
        if (h[p][threadIdx.x]) atomicAdd(&ghist[p * 256 + threadIdx.x], h[p][threadIdx.x]);
}

__global__ void __launch_bounds__(kThreads) rk_sort_pass_kernel(
    const uint64_t *in, uint64_t *out, unsigned long long *info, uint64_t cap, uint32_t shift,
    const uint32_t *ghist, uint64_t *status, uint32_t *counter) {
    uint64_t M;
    uint32_t T;
    if (!sort_count(info, cap, &M, &T)) return;
    __shared__ uint32_t wcnt[kWarps][256];  // per-warp digit counts, then exclusive offsets
    __shared__ uint32_t dbase[256];         // global start of each digit in this tile
    __shared__ uint32_t s_tile;
    __shared__ int s_abort;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t lt = (1u << lane) - 1u;

    // exclusive prefix of this pass's digit totals (thread d owns digit d):
    // shuffle scan within each warp, then over the 8 warp totals
    uint32_t gbase;
    {
        __shared__ uint32_t wsum[kWarps];
        const uint32_t v = ghist[tid];
        uint32_t incl = v;
#pragma unroll
        for (uint32_t d = 1; d < 32; d <<= 1) {
            const uint32_t o = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += o;
        }
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        uint32_t before = 0;
        for (uint32_t w = 0; w < warp; ++w) before += wsum[w];
        gbase = before + incl - v;
    }
    for (;;) {
        __syncthreads();
        if (tid == 0) {
            s_tile = atomicAdd(counter, 1u);
            s_abort = 0;
        }
        for (uint32_t w = 0; w < kWarps; ++w) wcnt[w][tid] = 0;
        __syncthreads();
        const uint32_t tile = s_tile;
        if (tile >= T) return;

        // stable local ranks: warp w takes keys [w*512, (w+1)*512) of the tile
        const uint64_t base = (uint64_t)tile * kSortTile + (uint64_t)warp * kPerWarp;
        uint64_t key[kPerWarp / 32];
        uint32_t rank[kPerWarp / 32];
        // all of this warp's keys first (independent loads in flight together)
#pragma unroll
        for (uint32_t r = 0; r < kPerWarp / 32; ++r) {
            const uint64_t idx = base + r * 32 + lane;
            key[r] = idx < M ? __ldcg(in + idx) : 0;
        }
#pragma unroll
        for (uint32_t r = 0; r < kPerWarp / 32; ++r) {
            const uint64_t idx = base + r * 32 + lane;
            const bool valid = idx < M;
            const uint32_t d = (uint32_t)(key[r] >> shift) & 255u;
            const uint32_t peers = digit_peers(d, valid);
            const uint32_t before = valid ? wcnt[warp][d] : 0;
            rank[r] = before + __popc(peers & lt);
            __syncwarp();
            if (valid && (peers & lt) == 0) wcnt[warp][d] = before + __popc(peers);
            __syncwarp();
        }
        __syncthreads();
        // thread d: per-warp exclusive offsets and the tile's count of digit d
        uint32_t cnt = 0;
        for (uint32_t w = 0; w < kWarps; ++w) {
            const uint32_t c = wcnt[w][tid];
            wcnt[w][tid] = cnt;
            cnt += c;
        }
        // decoupled look-back over the tiles before this one
        uint64_t *st = status + (uint64_t)tile * 256u + tid;
        uint64_t excl = 0;
        if (tile == 0) {
            *reinterpret_cast<volatile uint64_t *>(st) = kFlagInc | cnt;
        } else {
            *reinterpret_cast<volatile uint64_t *>(st) = kFlagAgg | cnt;
            // read kWindow predecessors per step (loads in flight together),
            // add their counts back to the first inclusive prefix
            constexpr int kWindow = 16;
            int64_t j = (int64_t)tile - 1;
            uint64_t t0 = 0;
            bool done = false;
            while (!done && j >= 0) {
                uint64_t v[kWindow];
#pragma unroll
                for (int u = 0; u < kWindow; ++u)
                    v[u] = j - u >= 0 ? *reinterpret_cast<volatile const uint64_t *>(
                                            status + (uint64_t)(j - u) * 256u + tid)
                                      : kFlagInc;
                int consumed = 0;
                bool stalled = false;
#pragma unroll
                for (int u = 0; u < kWindow; ++u) {
                    if (done || stalled) continue;
                    if (v[u] & kFlagInc) {
                        excl += v[u] & kCountMask;
                        done = true;
                    } else if (v[u] & kFlagAgg) {
                        excl += v[u] & kCountMask;
                        ++consumed;
                    } else {
                        stalled = true;  // not published yet (claimed earlier, so it runs)
                    }
                }
                j -= consumed;
                if (stalled) {
                    if (t0 == 0) t0 = globaltimer_ns();
                    else if (globaltimer_ns() - t0 > kLookbackTimeoutNs) {
                        info[1] = RK_ETIMEOUT;
                        s_abort = 1;
                        break;
                    }
                }
            }
            __threadfence();
            *reinterpret_cast<volatile uint64_t *>(st) = kFlagInc | (excl + cnt);
        }
        dbase[tid] = gbase + (uint32_t)excl;
        __syncthreads();
        if (s_abort) return;
#pragma unroll
        for (uint32_t r = 0; r < kPerWarp / 32; ++r) {
            const uint64_t idx = base + r * 32 + lane;
            if (idx < M) {
                const uint32_t d = (uint32_t)(key[r] >> shift) & 255u;
                out[dbase[d] + wcnt[warp][d] + rank[r]] = key[r];
            }
        }
    }
}

// Arrival with release semantics (gpu scope): the CTA's writes ordered
// before it by the preceding __syncthreads are visible to any thread that
// acquires the counter value.
__device__ __forceinline__ void arrive_release(unsigned int *ctr) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(ctr) : "memory");
}

__device__ __forceinline__ unsigned int load_acquire(const unsigned int *ctr) {
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ctr) : "memory");
    return v;
}

// Grid-wide barrier of a cooperative launch (every CTA resident): one
// arrival counter in global memory, target = barriers passed x CTAs; a
// release arrival and acquire loads order the phases' memory.  The wait is
// bounded; on a timeout RK_ETIMEOUT is recorded and false returned.
__device__ __forceinline__ bool grid_sync(unsigned int *ctr, unsigned int target,
                                          unsigned long long *info, int *s_ok) {
    __syncthreads();
    if (threadIdx.x == 0) {
        arrive_release(ctr);
        int ok = 1;
        uint64_t t0 = 0;
        while (load_acquire(ctr) < target) {
            const uint64_t now = globaltimer_ns();
            if (t0 == 0) {
                t0 = now;
            } else if (now - t0 > kLookbackTimeoutNs) {
                info[1] = RK_ETIMEOUT;
                ok = 0;
                break;
            }
        }
        *s_ok = ok;
    }
    __syncthreads();
    return *s_ok != 0;
}

// Inclusive sum of v over the lanes up to this one.
__device__ __forceinline__ uint32_t warp_incl(uint32_t v, uint32_t lane) {
#pragma unroll
    for (uint32_t d = 1; d < 32; d <<= 1) {
        const uint32_t o = __shfl_up_sync(0xffffffffu, v, d);
        if (lane >= d) v += o;
    }
    return v;
}

// Stable ranks of one tile's keys (warp w: keys [w*256, (w+1)*256) of the
// tile): key[r] and rank[r] per lane, the warp's digit counts in wc.
__device__ __forceinline__ void rank_tile(const uint64_t *src, uint64_t M, uint64_t base,
                                          uint32_t shift, uint64_t (&key)[kPerWarp / 32],
                                          uint32_t (&rank)[kPerWarp / 32], uint32_t *wc,
                                          uint32_t lane, uint32_t lt) {
#pragma unroll
    for (uint32_t r = 0; r < kPerWarp / 32; ++r) {
        const uint64_t idx = base + r * 32 + lane;
        key[r] = idx < M ? __ldcg(src + idx) : 0;
    }
#pragma unroll
    for (uint32_t r = 0; r < kPerWarp / 32; ++r) {
        const bool valid = base + r * 32 + lane < M;
        const uint32_t d = (uint32_t)(key[r] >> shift) & 255u;
        const uint32_t peers = digit_peers(d, valid);
        const uint32_t bef = valid ? wc[d] : 0;
        rank[r] = bef + __popc(peers & lt);
        __syncwarp();
        if (valid && (peers & lt) == 0) wc[d] = bef + __popc(peers);
        __syncwarp();
    }
}

// Every pass over a single tile (at most kSortTile keys) in one CTA: the keys
// stay in registers (warp w: keys [w*256, (w+1)*256)), each pass ranks them,
// scatters them to their place in the pass's order in shared memory and
// reads them back.  No grid barrier, no global round trip between passes.
__device__ __forceinline__ void sort_one_tile(uint64_t *keys, uint64_t M, const Shifts &sh,
                                              uint64_t *sbuf, uint32_t (&wcnt)[kWarps][256],
                                              uint32_t *dbase, uint32_t *wsum) {
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    const uint32_t base = warp * kPerWarp;
    uint64_t key[kPerWarp / 32];
    uint32_t rank[kPerWarp / 32];
#pragma unroll
    for (uint32_t r = 0; r < kPerWarp / 32; ++r) {
        const uint32_t idx = base + r * 32 + lane;
        key[r] = idx < M ? __ldcg(keys + idx) : 0;
    }
    for (uint32_t p = 0; p < sh.n; ++p) {
        const uint32_t shift = sh.s[p];
        for (uint32_t w = 0; w < kWarps; ++w) wcnt[w][tid] = 0;
        __syncthreads();
#pragma unroll
        for (uint32_t r = 0; r < kPerWarp / 32; ++r) {
            const bool valid = base + r * 32 + lane < M;
            const uint32_t d = (uint32_t)(key[r] >> shift) & 255u;
            const uint32_t peers = digit_peers(d, valid);
            const uint32_t bef = valid ? wcnt[warp][d] : 0;
            rank[r] = bef + __popc(peers & lt);
            __syncwarp();
            if (valid && (peers & lt) == 0) wcnt[warp][d] = bef + __popc(peers);
            __syncwarp();
        }
        __syncthreads();
        uint32_t c = 0;  // digit tid: per-warp exclusive offsets, tile count
        for (uint32_t w = 0; w < kWarps; ++w) {
            const uint32_t x = wcnt[w][tid];
            wcnt[w][tid] = c;
            c += x;
        }
        const uint32_t incl = warp_incl(c, lane);
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        uint32_t before = 0;
        for (uint32_t w = 0; w < warp; ++w) before += wsum[w];
        dbase[tid] = before + incl - c;
        __syncthreads();
#pragma unroll
        for (uint32_t r = 0; r < kPerWarp / 32; ++r)
            if (base + r * 32 + lane < M) {
                const uint32_t d = (uint32_t)(key[r] >> shift) & 255u;
                sbuf[dbase[d] + wcnt[warp][d] + rank[r]] = key[r];
            }
        __syncthreads();
#pragma unroll
        for (uint32_t r = 0; r < kPerWarp / 32; ++r)
            if (base + r * 32 + lane < M) key[r] = sbuf[base + r * 32 + lane];
        __syncthreads();
    }
#pragma unroll
    for (uint32_t r = 0; r < kPerWarp / 32; ++r) {
        const uint32_t idx = base + r * 32 + lane;
        if (idx < M) keys[idx] = key[r];
    }
}

// ---- sort by cells -------------------------------------------------------
// compact(key) has the key's order in shape.lo_bits + shape.hi_bits bits; a
// cell holds the keys that share its top bits.  With about one cell per key
// (2^cb in (M/2, M]) a cell of evenly spread keys holds a few, whatever the
// number of digits: five grid barriers in place of three per digit, and each
// key is read four times and written twice, mostly in L2.
//
// The comparisons within a cell cost its size squared: kCrowdedMean is the mean
// size (as a key meets it) from which on they cost more than the radix passes,
// which take over there.  Whole sorts, radix passes / cells: 20 K keys at 100 to a
// cell 60 / 48 us, at 200 60 / 67; 500 K at 78 72 / 67, at 625 70 / 184; 5 M at 97
// 390 / 340, at 780 368 / 1560.  It is estimated from samples before the keys are
// counted (without: 5 M keys at 8000 to a cell 348 -> 520 us, spent on noticing);
// kCellMax is the most in one cell that the count can meet after that (ranks have
// 16 bits).
// Measured against the radix passes in one cooperative launch, as whole
// searches: 10 M keys (4 GiB of bytes, 10,000 patterns) 4.38 -> 3.82 ms, 0.7 M
// keys (64 MB of words) 270 -> 235 us, 78,000 keys (33 MB) 103 -> 77 us, 400
// keys (1 MiB of DNA, one CTA) 37.9 -> 29.6 us.
constexpr uint32_t kCellMax = 1024;
constexpr uint32_t kCrowdedMean = 110;
// Shorter lists are not sampled (1 us of some 35): with two keys to a thread at
// most, even kCellMax keys to a cell cost about what the passes do.
constexpr uint32_t kSampledKeys = 1u << 17;
constexpr uint32_t kOneCellBits = 12;  // cells of the one-CTA sort
constexpr uint32_t kOneCellMax = 96;   // and the most keys it compares in one

// The bits of a key that its shape says are zero.  A list with one of them set
// (keys of another table or a longer text) is sorted by the radix passes, whose
// digits stay in range whatever the key: its cell would lie past the counts.
__device__ __forceinline__ uint64_t outside_shape(const SortShape &s) {
    const uint64_t lo = s.lo_bits >= 64 ? ~0ull : (1ull << s.lo_bits) - 1ull;
    return ~(s.hi_bits ? lo | (((1ull << s.hi_bits) - 1ull) << s.hi_shift) : lo);
}

// (of a key without such bits)
__device__ __forceinline__ uint64_t compact_key(uint64_t k, const SortShape &s) {
    const uint64_t lo = s.lo_bits >= 64 ? k : k & ((1ull << s.lo_bits) - 1ull);
    return s.hi_bits ? ((k >> s.hi_shift) << s.lo_bits) | lo : lo;
}

// Sum of v over the CTA, in every thread.
__device__ __forceinline__ uint32_t cta_sum(uint32_t v, uint32_t *wsum, uint32_t lane,
                                            uint32_t warp) {
#pragma unroll
    for (uint32_t d = 16; d; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
    __syncthreads();
    if (lane == 0) wsum[warp] = v;
    __syncthreads();
    uint32_t t = 0;
#pragma unroll
    for (uint32_t w = 0; w < kWarps; ++w) t += wsum[w];
    return t;
}

// Exclusive sum of v over the CTA's threads before this one; *total: of all.
__device__ __forceinline__ uint32_t cta_excl(uint32_t v, uint32_t *wsum, uint32_t lane,
                                             uint32_t warp, uint32_t *total) {
    const uint32_t incl = warp_incl(v, lane);
    __syncthreads();
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    uint32_t before = 0, t = 0;
#pragma unroll
    for (uint32_t w = 0; w < kWarps; ++w) {
        before += w < warp ? wsum[w] : 0u;
        t += wsum[w];
    }
    *total = t;
    return before + incl - v;
}

// The keys before key k, which lies at tmp[own], in its cell [b, e): the smaller
// ones, and of equal ones those at lower places (counted again, as they are rare;
// a test of j < own in the one loop: 5 M keys, 97 to a cell, 397 us, this 340,
// smaller keys alone 303; 1.2 to a cell 196, 196, 192).  Only a list that a caller
// made has equal keys: the library's own are told to be distinct.
__device__ __forceinline__ uint32_t place_in_cell(const uint64_t *tmp, uint32_t b, uint32_t e,
                                                  uint32_t own, uint64_t k, bool distinct) {
    uint32_t less = 0, same = 0;
    if (distinct) {
        for (uint32_t j = b; j < e; ++j) less += tmp[j] < k;
        return less;
    }
    for (uint32_t j = b; j < e; ++j) {
        const uint64_t v = tmp[j];
        less += v < k;
        same += v == k;
    }
    if (same > 1)
        for (uint32_t j = b; j < own; ++j) less += tmp[j] == k;
    return less;
}

// Up to kSortTile keys in one CTA, cells in shared memory.  Returns false,
// with the keys untouched, when a cell holds too many or a key is outside the
// shape.
__device__ __forceinline__ bool sort_one_cells(uint64_t *keys, uint32_t M, const SortShape &shape,
                                               uint64_t *sbuf, uint32_t *cell, uint32_t *wsum,
                                               bool distinct) {
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr uint32_t kCells = 1u << kOneCellBits, kPer = kCells / kThreads;
    constexpr uint32_t kKeys = kSortTile / kThreads;
    const uint32_t tb = shape.lo_bits + shape.hi_bits;
    const uint32_t cs = tb > kOneCellBits ? tb - kOneCellBits : 0;
    const uint64_t outside = outside_shape(shape);
    uint64_t key[kKeys];
    uint32_t cr[kKeys];  // cell << 16 | rank in it
#pragma unroll
    for (uint32_t r = 0; r < kKeys; ++r) {
        const uint32_t i = r * kThreads + tid;
        key[r] = i < M ? __ldcg(keys + i) : 0;
    }
    for (uint32_t i = tid; i < kCells / 4; i += kThreads)
        reinterpret_cast<uint4 *>(cell)[i] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    bool crowded = false;
#pragma unroll
    for (uint32_t r = 0; r < kKeys; ++r)
        if (r * kThreads + tid < M && (key[r] & outside)) {
            crowded = true;
        } else if (r * kThreads + tid < M) {
            const uint32_t c = (uint32_t)(compact_key(key[r], shape) >> cs);
            const uint32_t k = atomicAdd(&cell[c], 1u);
            crowded |= k >= kOneCellMax;
            cr[r] = (c << 16) | k;
        }
    if (__syncthreads_or(crowded)) return false;
    uint32_t v[kPer], sum = 0, total;
#pragma unroll
    for (uint32_t j = 0; j < kPer; ++j) {
        v[j] = cell[tid * kPer + j];
        sum += v[j];
    }
    uint32_t at = cta_excl(sum, wsum, lane, warp, &total);
#pragma unroll
    for (uint32_t j = 0; j < kPer; ++j) {
        cell[tid * kPer + j] = at;
        at += v[j];
    }
    if (tid == 0) cell[kCells] = M;
    __syncthreads();
#pragma unroll
    for (uint32_t r = 0; r < kKeys; ++r)
        if (r * kThreads + tid < M) sbuf[cell[cr[r] >> 16] + (cr[r] & 0xFFFFu)] = key[r];
    __syncthreads();
#pragma unroll
    for (uint32_t r = 0; r < kKeys; ++r)
        if (r * kThreads + tid < M) {
            const uint32_t b = cell[cr[r] >> 16], e = cell[(cr[r] >> 16) + 1];
            keys[b + place_in_cell(sbuf, b, e, b + (cr[r] & 0xFFFFu), key[r], distinct)] = key[r];
        }
    return true;
}

// Cells per key (at most; a compact key's fields are rounded up to whole bits,
// so up to three in four cells are empty): eight up to kManyCells keys, where
// clearing and adding up the counts costs little and a pattern with most of
// the matches has more cells to itself, two up to kTwoCells, then one, as the
// counts outgrow L2.  One cell -> this rule: 10 K keys 27 -> 21 us, 31 K of
// mostly one pattern 54 -> 23 us, 1 M 120 -> 83 us, 2.5 M 153 -> 124 us; two
// cells at 10 M: 370 -> 394 us.
constexpr uint64_t kManyCells = 1u << 18, kTwoCells = 1u << 22;
constexpr uint32_t kKeysPerCta = 512;

enum CellsResult { kCellsDone, kCellsCrowded, kCellsTimeout };

// Pairs of keys in one cell among the CTA's samples k, one per thread.  seen:
// kSeen zero words.
constexpr uint32_t kSeen = 8 * kThreads;
static_assert(kSeen == kWarps * 256, "the digit counters' shared memory");

__device__ __forceinline__ uint32_t sample_pairs(uint64_t k, const SortShape &shape, uint32_t cs,
                                                 uint64_t outside, uint32_t *seen, uint32_t *wsum,
                                                 uint32_t lane, uint32_t warp) {
    __syncthreads();  // seen is zero
    uint32_t before = 0;
    if (!(k & outside)) {
        const uint32_t c = (uint32_t)(compact_key(k, shape) >> cs) + 1u;
        uint32_t s = (c * 0x9E3779B1u) >> 22;  // one of kSeen / 2: four per sample
        for (;;) {
            const uint32_t o = atomicCAS(seen + s, 0u, c);
            if (o == 0 || o == c) break;
            s = (s + 1) % (kSeen / 2);
        }
        before = atomicAdd(seen + kSeen / 2 + s, 1u);
    }
    return cta_sum(before, wsum, lane, warp);
}

// M keys over G CTAs of a cooperative launch.  cnt: 2^cb + 1 words (cb >= 11),
// rank: M half words, part: G words of workspace, seen: kSeen words of shared
// memory; flag[0], flag[1] (sampled pairs) and *bar start at zero.
// kCellsCrowded (the same in every CTA; the cells hold too many keys, or a key
// is outside the shape): the keys are untouched.
__device__ __forceinline__ CellsResult sort_cells(uint64_t *keys, uint64_t *tmp, uint64_t M,
                                                  const SortShape &shape, uint32_t *cnt,
                                                  uint16_t *rank, uint32_t *part, uint32_t cb,
                                                  uint32_t *flag, unsigned int *bar, uint32_t G,
                                                  unsigned int *passed, unsigned long long *info,
                                                  uint32_t *seen, uint32_t *wsum, int *s_ok,
                                                  bool distinct) {
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t C = 1u << cb;
    const uint32_t tb = shape.lo_bits + shape.hi_bits;
    const uint32_t cs = tb > cb ? tb - cb : 0;
    const uint64_t outside = outside_shape(shape);
    const uint64_t gid = blockIdx.x * (uint64_t)kThreads + tid, stride = (uint64_t)G * kThreads;
    constexpr uint32_t kU = 8;  // keys in flight per thread

    // a CTA's samples are spread over the whole list: neighbours in it come from
    // one stretch of text, so a run of them would look crowded
    const bool sampled = M > kSampledKeys;
    uint64_t sample = 0;
    if (sampled) {
        sample = __ldcg(keys + ((uint64_t)tid * G + blockIdx.x) * M / ((uint64_t)kThreads * G));
        for (uint32_t i = tid; i < kSeen; i += kThreads) seen[i] = 0;
    }
    for (uint64_t i = gid; i < C / 4; i += stride)
        __stcg(reinterpret_cast<uint4 *>(cnt) + i, make_uint4(0, 0, 0, 0));
    if (sampled) {
        const uint32_t pairs = sample_pairs(sample, shape, cs, outside, seen, wsum, lane, warp);
        if (tid == 0 && pairs) atomicAdd(flag + 1, pairs);
    }
    if (!grid_sync(bar, ++*passed * G, info, s_ok)) return kCellsTimeout;
    // two keys share a cell with a chance of (mean size - 1) / M
    if (sampled && (uint64_t)__ldcg(flag + 1) * M >
        (uint64_t)G * (kThreads * (kThreads - 1) / 2) * (kCrowdedMean - 1))
        return kCellsCrowded;

    // count, and rank each key in its cell; the first key of every thread
    // alone, so that crowded keys are noticed before they queue up on a cell
    if (gid < M) {
        const uint64_t k = __ldcg(keys + gid);
        const uint32_t r =
            k & outside ? kCellMax : atomicAdd(cnt + (uint32_t)(compact_key(k, shape) >> cs), 1u);
        rank[gid] = (uint16_t)r;
        if (r >= kCellMax) *reinterpret_cast<volatile uint32_t *>(flag) = 1;
    }
    for (uint64_t i0 = gid + stride; i0 < M; i0 += kU * stride) {
        if (*reinterpret_cast<volatile uint32_t *>(flag)) break;
        uint64_t k[kU];
        uint32_t r[kU];
#pragma unroll
        for (uint32_t u = 0; u < kU; ++u) k[u] = i0 + u * stride < M ? __ldcg(keys + i0 + u * stride) : 0;
#pragma unroll
        for (uint32_t u = 0; u < kU; ++u)
            r[u] = i0 + u * stride >= M ? 0u
                   : k[u] & outside
                       ? kCellMax
                       : atomicAdd(cnt + (uint32_t)(compact_key(k[u], shape) >> cs), 1u);
#pragma unroll
        for (uint32_t u = 0; u < kU; ++u)
            if (i0 + u * stride < M) {
                rank[i0 + u * stride] = (uint16_t)r[u];
                if (r[u] >= kCellMax) *reinterpret_cast<volatile uint32_t *>(flag) = 1;
            }
    }
    if (!grid_sync(bar, ++*passed * G, info, s_ok)) return kCellsTimeout;
    if (__ldcg(flag)) return kCellsCrowded;

    // exclusive sums of the counts: each CTA a run of cells, blocks of 1024
    const uint32_t run = (C + G * 1024u - 1u) / (G * 1024u) * 1024u;
    const uint32_t lo = min(C, blockIdx.x * run), hi = min(C, lo + run);
    uint32_t mine = 0;
    for (uint32_t i = lo + tid * 4; i < hi; i += kThreads * 4) {
        const uint4 v = __ldcg(reinterpret_cast<const uint4 *>(cnt + i));
        mine += v.x + v.y + v.z + v.w;
    }
    mine = cta_sum(mine, wsum, lane, warp);
    if (tid == 0) part[blockIdx.x] = mine;
    if (!grid_sync(bar, ++*passed * G, info, s_ok)) return kCellsTimeout;
    uint32_t carry = 0;
    for (uint32_t b = tid; b < blockIdx.x; b += kThreads) carry += __ldcg(part + b);
    carry = cta_sum(carry, wsum, lane, warp);
    for (uint32_t i0 = lo; i0 < hi; i0 += kThreads * 4) {
        const uint32_t i = i0 + tid * 4;
        uint4 v = make_uint4(0, 0, 0, 0);
        if (i < hi) v = __ldcg(reinterpret_cast<const uint4 *>(cnt + i));
        uint32_t total;
        const uint32_t at = carry + cta_excl(v.x + v.y + v.z + v.w, wsum, lane, warp, &total);
        if (i < hi)
            __stcg(reinterpret_cast<uint4 *>(cnt + i),
                   make_uint4(at, at + v.x, at + v.x + v.y, at + v.x + v.y + v.z));
        carry += total;
    }
    if (gid == 0) cnt[C] = (uint32_t)M;
    if (!grid_sync(bar, ++*passed * G, info, s_ok)) return kCellsTimeout;

    // scatter every key to its cell
    for (uint64_t i0 = gid; i0 < M; i0 += kU * stride) {
        uint64_t k[kU];
        uint32_t at[kU];
#pragma unroll
        for (uint32_t u = 0; u < kU; ++u) {
            const uint64_t i = i0 + u * stride;
            k[u] = i < M ? __ldcg(keys + i) : 0;
            at[u] = i < M ? __ldcg(rank + i) : 0;
        }
#pragma unroll
        for (uint32_t u = 0; u < kU; ++u)
            at[u] += __ldcg(cnt + (uint32_t)(compact_key(k[u], shape) >> cs));
#pragma unroll
        for (uint32_t u = 0; u < kU; ++u)
            if (i0 + u * stride < M) tmp[at[u]] = k[u];
    }
    if (!grid_sync(bar, ++*passed * G, info, s_ok)) return kCellsTimeout;

    // each key's place in its cell: the number of smaller keys there, and of
    // equal ones before it
    constexpr uint32_t kV = 4;
    for (uint64_t i0 = gid; i0 < M; i0 += kV * stride) {
        uint64_t k[kV];
        uint32_t b[kV], e[kV];
#pragma unroll
        for (uint32_t u = 0; u < kV; ++u) k[u] = i0 + u * stride < M ? __ldcg(tmp + i0 + u * stride) : 0;
#pragma unroll
        for (uint32_t u = 0; u < kV; ++u) {
            const uint32_t c = (uint32_t)(compact_key(k[u], shape) >> cs);
            b[u] = __ldcg(cnt + c);
            e[u] = __ldcg(cnt + c + 1);
        }
#pragma unroll
        for (uint32_t u = 0; u < kV; ++u)
            if (i0 + u * stride < M) {
                const uint32_t own = (uint32_t)(i0 + u * stride);
                keys[b[u] + place_in_cell(tmp, b[u], e[u], own, k[u], distinct)] = k[u];
            }
    }
    return kCellsDone;
}

// The sort in one cooperative launch, for outputs of a few thousand tiles: by
// cells, or by every radix pass when the keys are crowded.  For the passes
// cnt holds, digit-major, the count of digit d among the keys of tile t at
// [d * pitch + t].  Per pass:
//   A  each CTA ranks its tile's keys stably (per-warp digit counters) and
//      publishes the tile's digit counts;
//   B  one warp per digit turns its row into exclusive prefixes over the
//      tiles (in place) and a total;
//   C  each CTA scatters its keys to (start of the digit) + (prefix of the
//      tile) + (rank within the tile);
// with a grid barrier after each phase.  With one tile per CTA the keys,
// ranks and counters stay on chip from A to C; with more, C ranks again.
// A single tile is sorted by one CTA alone, without barriers.
// A fixed number of barriers replaces the chain of look-back waits, whose
// length grows with the tile count.  An odd pass count ends with a copy
// back from the second buffer.  CTAs that the list is too short for leave at
// once.
__global__ void __launch_bounds__(kThreads) rk_sort_fused_kernel(
    uint64_t *keys, uint64_t *tmp, unsigned long long *info, uint64_t cap, Shifts sh,
    SortShape shape, uint32_t *cnt, uint64_t cnt_bytes, uint32_t pitch, uint32_t *totals,
    unsigned int *bar, uint32_t *flag, bool distinct) {
    uint64_t M;
    uint32_t T;
    if (!sort_count(info, cap, &M, &T)) return;
    // CTAs taking part: one per kKeysPerCta keys, so that a short list is not
    // left to a few SMs (64 K keys, with the cells: 34 -> 27 us)
    const uint32_t G =
        T == 1 ? 1u : (uint32_t)min((uint64_t)gridDim.x, (M + kKeysPerCta - 1) / kKeysPerCta);
    if (blockIdx.x >= G) return;
    __shared__ uint32_t wcnt[kWarps][256];
    __shared__ uint32_t dbase[256];
    __shared__ uint32_t wsum[kWarps];
    __shared__ int s_ok;
    if (T == 1) {
        __shared__ uint64_t sbuf[kSortTile];
        __shared__ __align__(16) uint32_t cell[(1u << kOneCellBits) + 4];
        if (!sort_one_cells(keys, (uint32_t)M, shape, sbuf, cell, wsum, distinct))
            sort_one_tile(keys, M, sh, sbuf, wcnt, dbase, wsum);
        return;
    }
    unsigned int passed = 0;
    {
        // 2^cb cells (words), then M ranks (half words), then a word per CTA, in
        // the look-back words' space (16 KiB per tile of the capacity)
        uint32_t cb = 31u - __clz((uint32_t)M);
        for (uint32_t more = M <= kManyCells ? 3u : M <= kTwoCells ? 1u : 0u; more; --more)
            if ((8ull << cb) + 2 * M + 4ull * gridDim.x + 64 <= cnt_bytes) ++cb;
        uint16_t *rank = reinterpret_cast<uint16_t *>(cnt + (1u << cb) + 4);
        uint32_t *part = reinterpret_cast<uint32_t *>(rank + (M + 1) / 2 * 2);
        const CellsResult r = sort_cells(keys, tmp, M, shape, cnt, rank, part, cb, flag, bar, G,
                                         &passed, info, &wcnt[0][0], wsum, &s_ok, distinct);
        if (r != kCellsCrowded) return;
    }
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    const bool one = T <= G;  // one tile per CTA: state kept from A to C
    uint64_t key[kPerWarp / 32];
    uint32_t rank[kPerWarp / 32];
    for (uint32_t p = 0; p < sh.n; ++p) {
        const uint64_t *src = (p & 1) ? tmp : keys;
        uint64_t *dst = (p & 1) ? keys : tmp;
        const uint32_t shift = sh.s[p];

        // A: rank each tile, publish its digit counts
        for (uint32_t t = blockIdx.x; t < T; t += G) {
            for (uint32_t w = 0; w < kWarps; ++w) wcnt[w][tid] = 0;
            __syncthreads();
            rank_tile(src, M, (uint64_t)t * kSortTile + (uint64_t)warp * kPerWarp, shift, key,
                      rank, wcnt[warp], lane, lt);
            __syncthreads();
            uint32_t c = 0;
            for (uint32_t w = 0; w < kWarps; ++w) c += wcnt[w][tid];
            cnt[(uint64_t)tid * pitch + t] = c;
            __syncthreads();
        }
        if (!grid_sync(bar, ++passed * G, info, &s_ok)) return;

        // B: per digit, exclusive prefix over the tiles (in place) and total:
        // under 32 tiles one thread per digit (its loads issued together),
        // else one warp per digit (256 warps or more take part)
        if (T < 32) {
            if (blockIdx.x == 0) {
                uint32_t *row = cnt + (uint64_t)tid * pitch;
                uint32_t v[32];
#pragma unroll
                for (uint32_t t = 0; t < 32; ++t) v[t] = t < T ? __ldcg(row + t) : 0u;
                uint32_t sum = 0;
#pragma unroll
                for (uint32_t t = 0; t < 32; ++t)
                    if (t < T) {
                        row[t] = sum;
                        sum += v[t];
                    }
                totals[tid] = sum;
            }
        } else
        for (uint32_t d = blockIdx.x * kWarps + warp; d < 256; d += G * kWarps) {
            uint32_t *row = cnt + (uint64_t)d * pitch;
            uint32_t carry = 0;
            for (uint32_t t0 = 0; t0 < T; t0 += 8 * 32) {
                uint32_t v[8];
#pragma unroll
                for (uint32_t j = 0; j < 8; ++j) {
                    const uint32_t t = t0 + 32 * j + lane;
                    v[j] = t < T ? __ldcg(row + t) : 0u;
                }
#pragma unroll
                for (uint32_t j = 0; j < 8; ++j) {
                    const uint32_t t = t0 + 32 * j + lane;
                    const uint32_t incl = warp_incl(v[j], lane);
                    if (t < T) row[t] = carry + incl - v[j];
                    carry += __shfl_sync(0xffffffffu, incl, 31);
                }
            }
            if (lane == 0) totals[d] = carry;
        }
        if (!grid_sync(bar, ++passed * G, info, &s_ok)) return;

        // C: scatter
        for (uint32_t t = blockIdx.x; t < T; t += G) {
            const uint32_t tot = __ldcg(totals + tid);
            const uint32_t tpre = __ldcg(cnt + (uint64_t)tid * pitch + t);
            const uint64_t base = (uint64_t)t * kSortTile + (uint64_t)warp * kPerWarp;
            if (!one) {
                for (uint32_t w = 0; w < kWarps; ++w) wcnt[w][tid] = 0;
                __syncthreads();
                rank_tile(src, M, base, shift, key, rank, wcnt[warp], lane, lt);
                __syncthreads();
            }
            // per-warp exclusive offsets of digit tid within the tile
            uint32_t c = 0;
            for (uint32_t w = 0; w < kWarps; ++w) {
                const uint32_t x = wcnt[w][tid];
                wcnt[w][tid] = c;
                c += x;
            }
            const uint32_t incl = warp_incl(tot, lane);
            if (lane == 31) wsum[warp] = incl;
            __syncthreads();
            uint32_t before = 0;
            for (uint32_t w = 0; w < warp; ++w) before += wsum[w];
            dbase[tid] = before + incl - tot + tpre;
            __syncthreads();
#pragma unroll
            for (uint32_t r = 0; r < kPerWarp / 32; ++r) {
                if (base + r * 32 + lane < M) {
                    const uint32_t d = (uint32_t)(key[r] >> shift) & 255u;
                    dst[dbase[d] + wcnt[warp][d] + rank[r]] = key[r];
                }
            }
            __syncthreads();
        }
        if (p + 1 < sh.n || (sh.n & 1))
            if (!grid_sync(bar, ++passed * G, info, &s_ok)) return;
    }
    if (sh.n & 1)
        for (uint64_t i = blockIdx.x * (uint64_t)kThreads + tid; i < M; i += (uint64_t)G * kThreads)
            keys[i] = __ldcg(tmp + i);
}

__global__ void rk_sort_copy_kernel(const uint64_t *in, uint64_t *out,
                                    const unsigned long long *info, uint64_t cap) {
    uint64_t M;
    uint32_t T;
    if (!sort_count(info, cap, &M, &T)) return;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < M;
         i += (uint64_t)gridDim.x * blockDim.x)
        out[i] = in[i];
}

uint32_t bits_for(uint64_t max_value) {
    uint32_t b = 0;
    while (b < 64 && (max_value >> b)) ++b;
    return b;
}

// CTAs of the fused sort: at most two per SM, all resident (0: the kernel
// does not fit on this device).
uint32_t fused_grid(int sm_count) {
    constexpr int kMaxDevices = 64;
    static std::mutex mu;
    static bool dev_seen[kMaxDevices] = {};
    static uint32_t per_sm[kMaxDevices];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return 0;
    std::lock_guard<std::mutex> lk(mu);
    if (!dev_seen[dev]) {
        int nb = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, rk_sort_fused_kernel, kThreads, 0) !=
            cudaSuccess)
            nb = 0;
        per_sm[dev] = (uint32_t)std::max(0, std::min(nb, 2));
        dev_seen[dev] = true;
    }
    return per_sm[dev] * (uint32_t)sm_count;
}

// Most tiles of 2048 keys per resident CTA that the fused sort takes: with
// more than one per CTA, phases A and C loop over them (C ranks again).
constexpr uint64_t kFusedTilesPerCta = 32;

// CTAs of the fused sort for an output of `capacity` keys (0: the look-back
// kernels are used instead).
uint32_t fused_ctas(int sm_count, uint64_t capacity) {
    const uint32_t gmax = fused_grid(sm_count);
    const uint64_t tiles = sort_ws_layout(capacity).tiles;
    if (!gmax || tiles > kFusedTilesPerCta * gmax) return 0;
    return (uint32_t)std::min<uint64_t>(tiles, gmax);
}

// The fields of a plain search's keys that can be non-zero.
SortShape plain_shape(uint64_t n, uint32_t k) {
    return SortShape{bits_for(n - 1), RK_KEY_OFFSET_BITS, bits_for(k - 1)};
}

// The radix passes' digit shifts for a key shape, least significant first.
Shifts shifts_of(const SortShape &shape) {
    Shifts sh{};
    for (uint32_t s = 0; s < shape.lo_bits; s += 8) sh.s[sh.n++] = s;
    for (uint32_t s = 0; s < shape.hi_bits; s += 8) sh.s[sh.n++] = shape.hi_shift + s;
    return sh;
}

}  // namespace

uint64_t sort_workspace_bytes(uint64_t capacity) { return sort_ws_bytes(capacity); }

int launch_sort_shape(int sm_count, const SortShape &shape_in, uint64_t *d_keys,
                      uint64_t capacity, const uint64_t *d_info, void *d_ws, uint64_t ws_bytes,
                      cudaStream_t stream, bool cleared, bool distinct) {
    SortShape shape = shape_in;
    Shifts sh = shifts_of(shape);
    if (capacity < 2 || sh.n == 0) return RK_OK;
    if (ws_bytes < sort_ws_bytes(capacity)) return RK_EINVAL;
    const SortWsLayout L = sort_ws_layout(capacity);
    uint8_t *ws = reinterpret_cast<uint8_t *>(d_ws);
    uint64_t *tmp = reinterpret_cast<uint64_t *>(ws + L.tmp_off);
    uint32_t *counters = reinterpret_cast<uint32_t *>(ws + L.ctrl_off);
    uint32_t *ghist = reinterpret_cast<uint32_t *>(ws + L.ghist_off);
    uint64_t *status = reinterpret_cast<uint64_t *>(ws + L.status_off);
    unsigned long long *info =
        reinterpret_cast<unsigned long long *>(const_cast<uint64_t *>(d_info));

    // up to kFusedTilesPerCta tiles per CTA: one cooperative launch
    if (const uint32_t g = fused_ctas(sm_count, capacity)) {
        // its barrier and flag are the control words; cell counts and ranks,
        // or digit-major counts (256 x tiles), go to the look-back words' space
        if (!cleared &&
            cudaMemsetAsync(counters, 0, L.ghist_off - L.ctrl_off, stream) != cudaSuccess)
            return RK_ECUDA;
        uint32_t *cnt = reinterpret_cast<uint32_t *>(status);
        uint64_t cnt_bytes = L.total - L.status_off;
        uint32_t pitch = (uint32_t)L.tiles;
        uint32_t *totals = ghist;
        unsigned int *bar = counters + 32;
        uint32_t *flag = counters;
        void *args[] = {&d_keys, &tmp,       &info,  &capacity, &sh,  &shape,
                        &cnt,    &cnt_bytes, &pitch, &totals,   &bar, &flag, &distinct};
        if (cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(rk_sort_fused_kernel), g,
                                        kThreads, args, 0, stream) != cudaSuccess) {
            cudaGetLastError();
            return RK_ECUDA;
        }
        return RK_OK;
    }
    if (cudaMemsetAsync(ws + L.ctrl_off, 0, L.status_off - L.ctrl_off, stream) != cudaSuccess)
        return RK_ECUDA;
    // histogram grid: about one CTA per 4096 keys of the capacity, at most 4 per SM
    const uint32_t grid =
        (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>((uint64_t)sm_count * 4,
                                                           (capacity + 4095) / 4096));
    const uint64_t tiles = L.tiles;
    rk_sort_hist_kernel<<<grid, kThreads, 0, stream>>>(d_keys, info, capacity, sh, ghist, status,
                                                       tiles);
    for (uint32_t p = 0; p < sh.n; ++p) {
        const uint64_t *src = (p & 1) ? tmp : d_keys;
        uint64_t *dst = (p & 1) ? d_keys : tmp;
        const uint32_t pgrid = (uint32_t)std::min<uint64_t>(tiles, (uint64_t)sm_count * 8);
        rk_sort_pass_kernel<<<pgrid, kThreads, 0, stream>>>(
            src, dst, info, capacity, sh.s[p], ghist + p * 256, status + (uint64_t)p * tiles * 256,
            counters + p);
    }
    if (sh.n & 1)
        rk_sort_copy_kernel<<<(uint32_t)sm_count * 4, 256, 0, stream>>>(tmp, d_keys, info, capacity);
    return cudaGetLastError() == cudaSuccess ? RK_OK : RK_ECUDA;
}

int launch_sort(const rk_table *t, uint64_t n, uint64_t *d_keys, uint64_t capacity,
                const uint64_t *d_info, void *d_ws, uint64_t ws_bytes, cudaStream_t stream,
                bool cleared, bool distinct) {
    if (n == 0 || t->dev.n_patterns == 0) return RK_OK;
    return launch_sort_shape(t->sm_count, plain_shape(n, t->dev.n_patterns), d_keys, capacity,
                             d_info, d_ws, ws_bytes, stream, cleared, distinct);
}

ZeroWords sort_control(int sm_count, uint64_t capacity, void *d_ws) {
    if (capacity < 2 || !d_ws || !fused_ctas(sm_count, capacity)) return {};
    const SortWsLayout L = sort_ws_layout(capacity);
    return {reinterpret_cast<uint32_t *>(reinterpret_cast<uint8_t *>(d_ws) + L.ctrl_off),
            (uint32_t)(L.ghist_off - L.ctrl_off) / 4};
}

ZeroWords sort_control(const rk_table *t, uint64_t n, uint64_t capacity, void *d_ws) {
    if (n == 0 || t->dev.n_patterns == 0) return {};
    return sort_control(t->sm_count, capacity, d_ws);
}

uint32_t sort_launches(const rk_table *t, uint64_t n, uint64_t capacity) {
    if (n == 0 || t->dev.n_patterns == 0 || capacity < 2) return 0;
    const uint32_t ns = shifts_of(plain_shape(n, t->dev.n_patterns)).n;
    if (ns == 0) return 0;
    if (fused_ctas(t->sm_count, capacity)) return 1;
    return 1 + ns + (ns & 1);  // histogram, one kernel per pass, copy back
}

}  // namespace rk
