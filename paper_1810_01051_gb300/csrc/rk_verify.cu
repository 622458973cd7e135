// Second pass of a deferred scan: A4 verify (A2 hash and A3 probe before it
// where patterns share prefix and length) and A5 emit
// for every candidate the tiled scan listed (a window whose exact q-byte
// prefix starts some pattern and whose next four bytes pass that prefix's
// fingerprint set).  The scan kernel handles one tile at a time, so its
// survivor rounds hold only the few candidates of one warp's share of a
// tile and a warp pays for the longest window among them; here every warp
// takes 32 listed candidates at a time; a window's first 8 bytes come with
// the candidate, longer windows read the rest from the text in global memory.
#include "rk_scan_body.cuh"
#include "rk_sortws.cuh"

namespace rk {
namespace {

constexpr uint32_t kVerifyThreads = 256;
constexpr uint32_t kVerifyBlocks = 5;  // per SM
constexpr uint32_t kVerifyWarps = kVerifyThreads / 32;
constexpr uint32_t kVerifySmemMax = 32u << 10;  // survivor tables staged in shared memory

// A window from the list: compared 32 bytes at a time, the text's loads and the
// pattern's issued together, so that a pattern of up to 40 bytes costs one
// round trip.  Here the loads' latency is what there is to save (10 M
// candidates of 8..64 bytes: 616 -> 446 us); in the scans, whose few survivor
// warps are short of issue slots, the extra instructions cost more (1 GiB of
// words 1393 -> 1441 us).
struct LText : WText {};

__device__ __forceinline__ bool verify(const LText &w, uint64_t pos, const uint8_t *pat,
                                       uint32_t L) {
    const uint64_t *pw = reinterpret_cast<const uint64_t *>(pat);
    const uint64_t last = (pos + L - 1) >> 2;  // the last word that holds a window byte
    const uint32_t s = (uint32_t)(pos & 3u) * 8u;
    uint64_t d = w.first8 ^ pw[0];
    if (L < 8) d &= (1ull << (8u * L)) - 1ull;
    for (uint32_t i = 8; i < L; i += 32) {
        const uint64_t a = (pos + i) >> 2;
        const uint32_t *tw = reinterpret_cast<const uint32_t *>(w.g.base) + a;
        const uint32_t lim = (uint32_t)(last - a);
        uint32_t t[9];
        uint64_t p[4];
#pragma unroll
        for (uint32_t j = 0; j < 9; ++j) t[j] = __ldg(tw + min(j, lim));
#pragma unroll
        for (uint32_t b = 0; b < 4; ++b) p[b] = i + 8u * b < L ? pw[i / 8u + b] : 0;
#pragma unroll
        for (uint32_t b = 0; b < 4; ++b) {
            const uint32_t o = i + 8u * b;
            if (o >= L) continue;
            const uint32_t lo = __funnelshift_r(t[2 * b], t[2 * b + 1], s),
                           hi = __funnelshift_r(t[2 * b + 1], t[2 * b + 2], s);
            uint64_t x = (((uint64_t)hi << 32) | lo) ^ p[b];
            if (L - o < 8) x &= (1ull << (8u * (L - o))) - 1ull;
            d |= x;
        }
        if (d) return false;
    }
    return d == 0;
}

struct VerifyParams {
    DevTable tab;
    GText text;         // 16-byte aligned base at or before the text start
    uint64_t mis;       // text start - base
    uint64_t n;         // text length
    const ulonglong2 *list;
    uint64_t cap;
    const unsigned long long *count;
    uint64_t *keys;
    uint64_t capacity;
    unsigned long long *info;
};

// S2S: the survivor tables (P.tab.s2_bytes) are first copied to the block's
// dynamic shared memory, so each candidate's chain of table loads stays on
// chip; otherwise they are read through L1/L2.  Five blocks per SM: the kernel
// waits on chains of global loads (candidate, slot, run, pattern and text), and
// the registers that keep a comparison's loads in flight together are worth
// more than the warps (10 M candidates: six blocks 502 us, five 446 us).
template <bool S2S>
__global__ void __launch_bounds__(kVerifyThreads, kVerifyBlocks)
    rk_verify_kernel(const __grid_constant__ VerifyParams P) {
    extern __shared__ __align__(128) uint8_t ss2[];
    __shared__ uint32_t mcount[kVerifyWarps];
    __shared__ uint64_t mbuf[kVerifyWarps][kMatchCap];
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) mcount[warp] = 0;
    if (S2S) {
        const uint4 *src = reinterpret_cast<const uint4 *>(P.tab.s2_base);
        uint4 *dst = reinterpret_cast<uint4 *>(ss2);
        for (uint32_t i = threadIdx.x; i < (P.tab.s2_bytes + 15u) / 16u; i += kVerifyThreads)
            dst[i] = src[i];
    }
    __syncthreads();
    WarpCtx w{mcount + warp, mbuf[warp], P.keys, P.capacity, P.info};
    WinCtx C{};
    C.s2 = make_s2<false>(P.tab, S2S ? ss2 : P.tab.s2_base);
    C.mis = P.mis;
    C.n = P.n;
    C.key_prefix = 0;
    C.pid_shift = RK_KEY_OFFSET_BITS;
    C.q = P.tab.q;
    C.gram_bits = P.tab.gram_bits;
    C.gram_mult = P.tab.gram_mult;
    C.base_log2 = P.tab.base_log2;
    C.n_lengths = P.tab.n_lengths;

    const uint64_t nc = min((uint64_t)*P.count, P.cap);
    const uint64_t stride = (uint64_t)gridDim.x * kVerifyThreads;
    // warp-uniform loop: every lane reaches the flushes
    for (uint64_t i0 = (uint64_t)blockIdx.x * kVerifyThreads + warp * 32; i0 < nc; i0 += stride) {
        const uint64_t i = i0 + lane;
        if (i < nc) {
            const ulonglong2 c = P.list[i];
            const uint64_t x = cand_x(c.x);
            const LText win{{P.text, x + P.mis, c.y}};
            probe_slot(C, w, win, x + P.mis, x, cand_slot(c.x), cand_class(c.x));
        }
        __syncwarp();
        if (warp_read(w.mcount) >= kMatchCap - 32) flush(w, lane);
    }
    flush(w, lane);
}

}  // namespace

int launch_verify(const rk_table *t, const uint8_t *d_text, uint64_t n, const CandList &cand,
                  uint64_t *d_keys, uint64_t capacity, uint64_t *d_info, cudaStream_t stream) {
    if (n == 0 || t->dev.n_patterns == 0) return RK_OK;
    VerifyParams p{};
    p.tab = t->dev;
    const uintptr_t addr = reinterpret_cast<uintptr_t>(d_text);
    p.mis = addr & 15u;
    p.text = GText{reinterpret_cast<const uint8_t *>(addr & ~uintptr_t(15)),
                   (p.mis + n + 15) & ~uint64_t(15)};
    p.n = n;
    p.list = cand.list;
    p.cap = cand.cap;
    p.count = cand.count;
    p.keys = d_keys;
    p.capacity = capacity;
    p.info = reinterpret_cast<unsigned long long *>(d_info);
    const uint32_t grid = (uint32_t)t->sm_count * kVerifyBlocks;
    // tables up to 32 KiB go to shared memory (with the static 8 KiB, at
    // least five blocks of 256 threads per SM); larger ones stay in L2
    const uint32_t s2 = t->dev.s2_bytes;
    if (s2 <= kVerifySmemMax) {
        rk_verify_kernel<true><<<grid, kVerifyThreads, (s2 + 15u) / 16u * 16u, stream>>>(p);
    } else {
        rk_verify_kernel<false><<<grid, kVerifyThreads, 0, stream>>>(p);
    }
    return cudaGetLastError() == cudaSuccess ? RK_OK : RK_ECUDA;
}

}  // namespace rk
