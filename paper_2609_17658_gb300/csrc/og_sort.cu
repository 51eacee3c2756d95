// og_sort.cu -- stable LSD radix sort of (63-bit Morton key, u32 index) pairs.
//
// The paper builds its tree by inserting the particles one after another in
// Peano-Hilbert order (Sect. 4.1.1); here the order is a Morton order made by a
// least-significant-digit radix sort, 8 bits per pass.  Each pass is
//   1. upsweep:   per 2048-key tile, a 256-bin digit histogram (shared-memory
//                 atomics, one sub-histogram per warp), stored digit-major;
//   2. scan:      exclusive scan over (digit, tile) -> global offsets;
//   3. downsweep: stable in-tile ranking by warp peer masks (each warp owns
//                 256 consecutive keys, 8 rounds of 32), keys staged in shared
//                 memory in digit order, then written out so that runs of one
//                 digit stay contiguous in global memory.
// Passes whose digit is the same for every key (found from one histogram of
// all passes, read by the pass kernels themselves: no host round trip) only
// copy their input.  Sorts of at most kOneSweepMaxTiles tiles (small sorts
// are bound by launch latency) run each pass as one kernel instead: the
// global digit bases come from that histogram, and a tile's offsets within
// its digit from a look-back over the counts the tiles before it publish.  Up to
// kClusterMax keys all passes are one launch (k_cluster_sort).
#include <map>
#include <mutex>
#include <vector>

#include "og_internal.h"

namespace og {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kItems = 8;
constexpr int kTile = kThreads * kItems;        // 2048 keys per tile
constexpr int kPerWarp = 32 * kItems;           // 256 consecutive keys per warp
constexpr int kRadix = 256;
// sorts of at most this many tiles run each pass as one kernel (k_onesweep);
// larger ones as a count, a scan and a scatter per pass
constexpr int64_t kOneSweepMaxTiles = 384;
static_assert(kThreads == kRadix, "one thread per digit in the pass kernels");

// true in every thread of the block when all n keys share the digit of this
// pass (hist8: the digit histograms of all passes)
__device__ __forceinline__ bool trivial_pass(const uint32_t *hist8, int shift, int64_t n) {
    return __syncthreads_or(hist8 && hist8[(shift / 8) * kRadix + threadIdx.x] == (uint64_t)n) != 0;
}

// exclusive scan of one value per thread over the block (kThreads values)
__device__ __forceinline__ uint32_t block_exclusive(uint32_t v, uint32_t *warp_tot) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t inc = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t o = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= d) inc += o;
    }
    if (lane == 31) warp_tot[warp] = inc;
    __syncthreads();
    uint32_t wpre = 0;
    for (int w = 0; w < warp; ++w) wpre += warp_tot[w];
    __syncthreads();
    return wpre + inc - v;
}

__global__ void __launch_bounds__(kThreads) k_upsweep(const uint64_t *__restrict__ keys, int64_t n,
                                                      int shift, uint32_t *counts,
                                                      int64_t ntiles, const uint32_t *hist8) {
    pdl_wait();
    __shared__ uint32_t hist[kWarps][kRadix];
    const int warp = threadIdx.x >> 5;
    if (trivial_pass(hist8, shift, n)) return;
    for (int i = threadIdx.x; i < kWarps * kRadix; i += kThreads) (&hist[0][0])[i] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kTile;
#pragma unroll 4
    for (int k = 0; k < kItems; ++k) {
        int64_t i = base + (int64_t)k * kThreads + threadIdx.x;
        if (i < n) atomicAdd(&hist[warp][(uint32_t)(keys[i] >> shift) & 0xffu], 1u);
    }
    __syncthreads();
    uint32_t tot = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) tot += hist[w][threadIdx.x];
    counts[(int64_t)threadIdx.x * ntiles + blockIdx.x] = tot;
}

// histogram of all eight digit positions over all keys (to skip trivial passes)
__global__ void __launch_bounds__(kThreads) k_all_digits(const uint64_t *__restrict__ keys,
                                                         int64_t n, uint32_t *hist8) {
    pdl_wait();
    __shared__ uint32_t h[8][kRadix];
    for (int i = threadIdx.x; i < 8 * kRadix; i += kThreads) (&h[0][0])[i] = 0;
    __syncthreads();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        uint64_t k = keys[i];
#pragma unroll
        for (int p = 0; p < 8; ++p) atomicAdd(&h[p][(uint32_t)(k >> (8 * p)) & 0xffu], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 8 * kRadix; i += kThreads) {
        uint32_t v = (&h[0][0])[i];
        if (v) atomicAdd(&hist8[i], v);
    }
}

struct DownSmem {
    uint64_t keys[kTile];
    uint32_t vals[kTile];
    uint32_t wcnt[kWarps][kRadix];
    uint32_t dstart[kRadix];
    uint32_t gofs[kRadix];
    uint32_t warp_tot[kWarps];
    uint32_t warp_tot2[kWarps];
};

__global__ void __launch_bounds__(kThreads, 4) k_downsweep(const uint64_t *__restrict__ kin,
                                                        const uint32_t *__restrict__ vin,
                                                        uint64_t *__restrict__ kout,
                                                        uint32_t *__restrict__ vout, int64_t n,
                                                        int shift, const uint32_t *offsets,
                                                        int64_t ntiles, const uint32_t *hist8) {
    pdl_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    DownSmem &S = *reinterpret_cast<DownSmem *>(smem_raw);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt_mask = (1u << lane) - 1u;
    if (trivial_pass(hist8, shift, n)) {
        // every key has this digit: the stable order is the input order
        const int64_t b0 = (int64_t)blockIdx.x * kTile;
        const int64_t e0 = (n - b0) < kTile ? n : b0 + kTile;
        for (int64_t i = b0 + threadIdx.x; i < e0; i += kThreads) {
            kout[i] = kin[i];
            vout[i] = vin[i];
        }
        return;
    }
    for (int i = threadIdx.x; i < kWarps * kRadix; i += kThreads) (&S.wcnt[0][0])[i] = 0;
    __syncthreads();

    const int64_t base = (int64_t)blockIdx.x * kTile;
    uint64_t k[kItems];
    uint32_t v[kItems];
    uint32_t rank[kItems];
#pragma unroll
    for (int r = 0; r < kItems; ++r) {
        int64_t i = base + warp * kPerWarp + r * 32 + lane;
        bool valid = i < n;
        k[r] = valid ? kin[i] : 0ull;
        v[r] = valid ? vin[i] : 0u;
    }
#pragma unroll
    for (int r = 0; r < kItems; ++r) {
        int64_t i = base + warp * kPerWarp + r * 32 + lane;
        uint32_t d = (i < n) ? ((uint32_t)(k[r] >> shift) & 0xffu) : (uint32_t)kRadix;
        // lanes with the same digit (9 bits: 256 marks an invalid key), from
        // one ballot per bit plane
        unsigned peers = 0xffffffffu;
#pragma unroll
        for (int bit = 0; bit < 9; ++bit) {
            const bool on = (d >> bit) & 1u;
            const unsigned bb = __ballot_sync(0xffffffffu, on);
            peers &= on ? bb : ~bb;
        }
        int leader = __ffs(peers) - 1;
        uint32_t before = (d < kRadix) ? S.wcnt[warp][d] : 0u;
        __syncwarp();
        if (lane == leader && d < kRadix) S.wcnt[warp][d] = before + __popc(peers);
        __syncwarp();
        rank[r] = before + __popc(peers & lt_mask);
    }
    __syncthreads();
    // per digit: exclusive offsets of the warps, then the digit's tile total
    const int t = threadIdx.x;  // one thread per digit
    uint32_t run = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
        uint32_t c = S.wcnt[w][t];
        S.wcnt[w][t] = run;
        run += c;
    }
    // block exclusive scan of the digit totals
    uint32_t inc = run;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        uint32_t o = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= d) inc += o;
    }
    if (lane == 31) S.warp_tot[warp] = inc;
    __syncthreads();
    uint32_t wpre = 0;
    for (int w = 0; w < warp; ++w) wpre += S.warp_tot[w];
    S.dstart[t] = wpre + inc - run;
    S.gofs[t] = offsets[(int64_t)t * ntiles + blockIdx.x];
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kItems; ++r) {
        int64_t i = base + warp * kPerWarp + r * 32 + lane;
        if (i < n) {
            uint32_t d = (uint32_t)(k[r] >> shift) & 0xffu;
            uint32_t pos = S.dstart[d] + S.wcnt[warp][d] + rank[r];
            S.keys[pos] = k[r];
            S.vals[pos] = v[r];
        }
    }
    __syncthreads();
    const int64_t cnt = (n - base) < kTile ? (n - base) : kTile;
    for (int p = threadIdx.x; p < cnt; p += kThreads) {
        uint64_t key = S.keys[p];
        uint32_t d = (uint32_t)(key >> shift) & 0xffu;
        uint32_t g = S.gofs[d] + ((uint32_t)p - S.dstart[d]);
        kout[g] = key;
        vout[g] = S.vals[p];
    }
}

// One pass of the sort in a single kernel: the tile's digit counts are
// published, the counts of the tiles before it are gathered by a look-back
// (decoupled: a tile's word first holds its own count, then the inclusive
// count of the tiles up to it), and the digit bases come from the histograms
// of all passes taken before the first pass.  Tiles are numbered in the order
// their blocks start, so every tile waits only on tiles whose blocks already
// run.  A look word: flag (2 bits: 1 own count, 2 inclusive), pass tag
// (6 bits, pass + 1, so that words of the previous pass read as not ready),
// count (low 32 bits).
constexpr unsigned long long kLookOwn = 1ull << 62, kLookInc = 2ull << 62;
constexpr int kLookSpinLimit = 1 << 20;

__device__ __forceinline__ void st_look(unsigned long long *p, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long ld_look(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__global__ void __launch_bounds__(kThreads, 4) k_onesweep(const uint64_t *__restrict__ kin,
                                                       const uint32_t *__restrict__ vin,
                                                       uint64_t *__restrict__ kout,
                                                       uint32_t *__restrict__ vout, int64_t n, int pass,
                                                       const uint32_t *hist8, unsigned long long *look,
                                                       uint32_t *tile_ctr, uint32_t *status) {
    pdl_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    DownSmem &S = *reinterpret_cast<DownSmem *>(smem_raw);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt_mask = (1u << lane) - 1u;
    const int shift = 8 * pass;
    if (threadIdx.x == 0) S.warp_tot2[0] = atomicAdd(&tile_ctr[pass], 1u);
    __syncthreads();
    const int64_t tile = S.warp_tot2[0];
    const int64_t base = tile * kTile;
    if (trivial_pass(hist8, shift, n)) {
        // every key has this digit: the stable order is the input order
        const int64_t e0 = (n - base) < kTile ? n : base + kTile;
        for (int64_t i = base + threadIdx.x; i < e0; i += kThreads) {
            kout[i] = kin[i];
            vout[i] = vin[i];
        }
        return;
    }
    for (int i = threadIdx.x; i < kWarps * kRadix; i += kThreads) (&S.wcnt[0][0])[i] = 0;
    __syncthreads();

    uint64_t k[kItems];
    uint32_t v[kItems];
    uint32_t rank[kItems];
#pragma unroll
    for (int r = 0; r < kItems; ++r) {
        int64_t i = base + warp * kPerWarp + r * 32 + lane;
        bool valid = i < n;
        k[r] = valid ? kin[i] : 0ull;
        v[r] = valid ? vin[i] : 0u;
    }
#pragma unroll
    for (int r = 0; r < kItems; ++r) {
        int64_t i = base + warp * kPerWarp + r * 32 + lane;
        uint32_t d = (i < n) ? ((uint32_t)(k[r] >> shift) & 0xffu) : (uint32_t)kRadix;
        // lanes with the same digit (9 bits: 256 marks an invalid key)
        unsigned peers = 0xffffffffu;
#pragma unroll
        for (int bit = 0; bit < 9; ++bit) {
            const bool on = (d >> bit) & 1u;
            const unsigned bb = __ballot_sync(0xffffffffu, on);
            peers &= on ? bb : ~bb;
        }
        int leader = __ffs(peers) - 1;
        uint32_t before = (d < kRadix) ? S.wcnt[warp][d] : 0u;
        __syncwarp();
        if (lane == leader && d < kRadix) S.wcnt[warp][d] = before + __popc(peers);
        __syncwarp();
        rank[r] = before + __popc(peers & lt_mask);
    }
    __syncthreads();
    // per digit (one thread each): offsets of the warps, the tile's count
    const int t = threadIdx.x;
    uint32_t run = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
        uint32_t c = S.wcnt[w][t];
        S.wcnt[w][t] = run;
        run += c;
    }
    // publish this tile's count, then gather the counts of the tiles before it
    const unsigned long long tag = (unsigned long long)(pass + 1) << 56;
    const unsigned long long tag_mask = 0x3full << 56;
    uint32_t excl = 0;
    if (tile == 0) {
        st_look(&look[t], kLookInc | tag | run);
    } else {
        st_look(&look[tile * kRadix + t], kLookOwn | tag | run);
        int64_t j = tile - 1;
        int spins = 0;
        while (j >= 0) {
            const unsigned long long w = ld_look(&look[j * kRadix + t]);
            if ((w & tag_mask) != tag || (w >> 62) == 0ull) {
                if (++spins > kLookSpinLimit) {  // a tile that never publishes: give up
                    atomicOr(status, ST_TIMEOUT);
                    break;
                }
                if (spins > 32) __nanosleep(64);
                continue;
            }
            excl += (uint32_t)w;
            if ((w >> 62) == 2ull) break;
            --j;
        }
        st_look(&look[tile * kRadix + t], kLookInc | tag | (excl + run));
    }
    // block exclusive scan of the tile's digit counts
    uint32_t inc = run;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        uint32_t o = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= d) inc += o;
    }
    if (lane == 31) S.warp_tot[warp] = inc;
    __syncthreads();
    uint32_t wpre = 0;
    for (int w = 0; w < warp; ++w) wpre += S.warp_tot[w];
    S.dstart[t] = wpre + inc - run;
    // where this tile's keys of digit t go: the keys of smaller digits (all
    // tiles) plus the keys of digit t in the tiles before this one
    S.gofs[t] = block_exclusive(hist8[pass * kRadix + t], S.warp_tot2) + excl;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kItems; ++r) {
        int64_t i = base + warp * kPerWarp + r * 32 + lane;
        if (i < n) {
            uint32_t d = (uint32_t)(k[r] >> shift) & 0xffu;
            uint32_t pos = S.dstart[d] + S.wcnt[warp][d] + rank[r];
            S.keys[pos] = k[r];
            S.vals[pos] = v[r];
        }
    }
    __syncthreads();
    const int64_t cnt = (n - base) < kTile ? (n - base) : kTile;
    for (int p = threadIdx.x; p < cnt; p += kThreads) {
        uint64_t key = S.keys[p];
        uint32_t d = (uint32_t)(key >> shift) & 0xffu;
        uint32_t g = S.gofs[d] + ((uint32_t)p - S.dstart[d]);
        kout[g] = key;
        vout[g] = S.vals[p];
    }
}

// ---- small sorts: all passes in one kernel of one cluster
//
// A pass of a small sort is a chain of latencies (launch, tile ticket, loads, ranking,
// look-back, stores) of some 7 us that does not get shorter with fewer keys.  Up to
// kClusterMax keys the whole sort is one launch of a cluster of 16 blocks: the keys
// stay in the blocks' shared memory, a block sends its digit counts and then its keys
// into the others' (asynchronous stores to distributed shared memory, counted by a
// barrier of the receiver), and 9-bit digits take 63-bit keys in 7 passes instead
// of 8.  Block c owns the slots [c slice, (c + 1) slice) of every pass's input.
// Builds of 4k, 10k, 32k and 65k particles: 107, 114, 122 and 133 us with the passes,
// 76, 81, 97 and 124 this way (the sort itself 22 us at 4k, 41 at 32k).  A pass's
// latencies are 2 us (ranking 0.4, the exchange of counts and of keys 0.4 each); above
// 16k keys 16 SMs' ranking and sending take over, and from some 90k on the passes on
// the whole chip win.
// Tried: keys through global memory with two cluster barriers per pass (46 us at 4k;
// the barrier's release waits for the stores), synchronous remote stores (28 us).
//
// What keeps a block from writing where another still reads: it sends counts of
// pass p + 2, which go where those of pass p were, after it has all counts of pass
// p + 1, and a block sends those after it has read the ones of pass p; it sends
// keys of pass p after it has all counts of pass p, and a block sends those after it
// has sent on the keys of pass p - 1, whose buffer the new ones take.
//
// A wait that runs out: the block sends and stores nothing from then on, so no block
// takes a record that never arrived (those it would have reached run out in turn), and
// what it leaves in keys and vals are the pairs that came in.  It still takes part in
// the last cluster barrier, after which nothing more is sent to it, and then waits
// (again with a limit) for what is on its way into its own shared memory.
constexpr int kClBlocks = 16, kClThreads = 1024, kClWarps = kClThreads / 32;
constexpr int kClBits = 9, kClRadix = 1 << kClBits, kClPairs = kClRadix / 2;
constexpr int kClMaxRounds = 4;        // keys per thread
constexpr int64_t kClusterMax = (int64_t)kClBlocks * kClThreads * kClMaxRounds;
// tries of a wait; each suspends the thread for about kClTryNs at most, so a wait that runs
// out takes some 65 ms
constexpr int kClWaitLimit = 1 << 16;
constexpr uint32_t kClTryNs = 1000;
constexpr int kClDrainLimit = 1 << 10;
// test hook (sort_wait_timeout_probe): the block that keeps back its counts of the first
// pass, or with kHoldKeys its keys
constexpr uint32_t kHoldNone = 0xffffffffu, kHoldKeys = 0x100u;
static_assert(kClThreads == 4 * kClPairs && kClThreads == kClBlocks * kClPairs / 4 &&
                  kClThreads * kClMaxRounds < 65536,
              "a thread per digit pair and quarter, and per four pairs and block");

template <int kIt>
struct ClusterSmem {
    uint4 rec[2][kClThreads * kIt];                // key, value: this pass's input, the next one's
    uint32_t cnt[2][kClBlocks][kClPairs];          // every block's digit counts (pairs of 16 bits), by parity of the pass
    uint32_t wcnt[kClWarps][kClPairs];             // per warp: counts, then offsets within the quarter's 8 warps
    uint32_t quarter[4][kClPairs];                 // per 8 warps: counts
    uint32_t qpre[4][kClPairs];                    // those of the quarters before
    uint32_t own[kClPairs];                        // this block's counts
    uint32_t base[kClRadix];                       // where this block's keys of the digit go
    uint32_t wsum[kClPairs / 32];
    uint32_t gave_up;                              // a wait for counts ran out
    unsigned long long cnt_bar[2], rec_bar;        // received counts, by parity; received keys
};

__device__ __forceinline__ uint32_t shared_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
// the same place in block `rank` of the cluster
__device__ __forceinline__ uint32_t cluster_addr(const void *p, uint32_t rank) {
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(shared_addr(p)), "r"(rank));
    return a;
}
// 16 bytes into another block, counted by a barrier of that block
__device__ __forceinline__ void cluster_send(uint32_t a, uint32_t bar, uint4 v) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(a),
                 "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void bar_expect(void *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(shared_addr(bar)), "r"(bytes) : "memory");
}
// false: the wait ran out
__device__ __forceinline__ bool bar_wait(void *bar, uint32_t phase, int limit = kClWaitLimit) {
    const uint32_t a = shared_addr(bar);
    for (int it = 0; it < limit; ++it) {
        uint32_t ok;
        asm volatile("{\n\t.reg .pred p;\n\t"
                     "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok)
                     : "r"(a), "r"(phase), "r"(kClTryNs)
                     : "memory");
        if (ok) return true;
    }
    return false;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// in place: keys, vals (indices below n)
template <int kIt>
__global__ void __launch_bounds__(kClThreads, 1) k_cluster_sort(uint64_t *keys, uint32_t *vals, uint32_t n,
                                                                uint32_t slice, int rounds, int npasses,
                                                                uint32_t *status, uint32_t hold) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ClusterSmem<kIt> &S = *reinterpret_cast<ClusterSmem<kIt> *>(smem_raw);
    const uint32_t t = threadIdx.x, lane = t & 31u, warp = t >> 5;
    const unsigned lt_mask = (1u << lane) - 1u;
    uint32_t cta;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(cta));
    const uint32_t lo = cta * slice;
    const uint32_t mine = lo < n ? (n - lo < slice ? n - lo : slice) : 0u;   // keys of this block
    const uint32_t wfirst = warp * 32u * (uint32_t)rounds;                   // the warp's first slot
    const uint32_t pair = t & (kClPairs - 1u), qt = t / kClPairs;            // of the per-digit work
    if (t == 0) {
        S.gave_up = 0u;
        for (void *b : {(void *)&S.cnt_bar[0], (void *)&S.cnt_bar[1], (void *)&S.rec_bar})
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(shared_addr(b)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    cluster_sync();                                // every block has started and its barriers are there
    pdl_wait();
    for (uint32_t r = t; r < mine; r += kClThreads) {
        const uint64_t k = keys[lo + r];
        S.rec[0][r] = make_uint4((uint32_t)k, (uint32_t)(k >> 32), vals[lo + r], 0u);
    }
    int cur = 0;
    uint32_t moved = 0;                            // passes that moved the keys
    bool stored = false, gave_up = false;
    int pass = 0;
    for (; pass < npasses; ++pass) {
        const int shift = kClBits * pass, par = pass & 1;
        for (uint32_t i = t; i < kClWarps * kClPairs; i += kClThreads) (&S.wcnt[0][0])[i] = 0u;
        if (t == 0) bar_expect(&S.cnt_bar[par], kClBlocks * kClPairs * 4u);
        gave_up = __syncthreads_or(moved && !bar_wait(&S.rec_bar, (moved - 1u) & 1u));
        if (gave_up) break;
        uint16_t *wc = reinterpret_cast<uint16_t *>(S.wcnt[warp]);
        uint4 rec[kIt];
        uint32_t rank[kIt];
        // rank of every key among its warp's keys of the same digit
#pragma unroll
        for (int r = 0; r < kIt; ++r) {
            if (r >= rounds || wfirst + 32u * (uint32_t)r >= mine) break;
            const uint32_t p = wfirst + 32u * (uint32_t)r + lane;
            const bool ok = p < mine;
            rec[r] = ok ? S.rec[cur][p] : make_uint4(0u, 0u, 0u, 0u);
            const uint64_t key = rec[r].x | (uint64_t)rec[r].y << 32;
            const uint32_t d = (uint32_t)(key >> shift) & (kClRadix - 1u);
            unsigned peers = __ballot_sync(0xffffffffu, ok);
#pragma unroll
            for (int bit = 0; bit < kClBits; ++bit) {
                const bool on = (d >> bit) & 1u;
                const unsigned bb = __ballot_sync(0xffffffffu, on);
                peers &= on ? bb : ~bb;
            }
            const uint32_t before = wc[d];
            __syncwarp();
            if (ok && (peers & lt_mask) == 0u) wc[d] = (uint16_t)(before + __popc(peers));
            __syncwarp();
            rank[r] = before + __popc(peers & lt_mask);
        }
        __syncthreads();
        // offsets of the warps within their quarter (pairs of 16-bit sums: a block has
        // fewer than 2^16 keys), the quarters' counts
        {
            uint32_t c[8], run = 0;
#pragma unroll
            for (int w = 0; w < 8; ++w) c[w] = S.wcnt[qt * 8 + w][pair];
#pragma unroll
            for (int w = 0; w < 8; ++w) {
                S.wcnt[qt * 8 + w][pair] = run;
                run += c[w];
            }
            S.quarter[qt][pair] = run;
        }
        __syncthreads();
        {
            uint32_t own = 0, pre = 0;
#pragma unroll
            for (uint32_t q = 0; q < 4; ++q) {
                const uint32_t c = S.quarter[q][pair];
                pre += q < qt ? c : 0u;
                own += c;
            }
            S.qpre[qt][pair] = pre;
            if (qt == 0) S.own[pair] = own;
        }
        __syncthreads();
        {
            // four pairs to one block
            const uint32_t b = t / (kClPairs / 4), q = 4u * (t & (kClPairs / 4 - 1u));
            if (hold != cta) cluster_send(cluster_addr(&S.cnt[par][cta][q], b), cluster_addr(&S.cnt_bar[par], b),
                         *reinterpret_cast<const uint4 *>(&S.own[q]));
        }
        if (!bar_wait(&S.cnt_bar[par], (uint32_t)(pass >> 1) & 1u)) S.gave_up = 1u;
        // the digits' counts in all blocks and in those before this one, and their scan
        uint32_t all_lo = 0, all_hi = 0, bef_lo = 0, bef_hi = 0, sum = 0;
        if (qt == 0) {
#pragma unroll
            for (uint32_t b = 0; b < kClBlocks; ++b) {
                const uint32_t c = S.cnt[par][b][pair];
                all_lo += c & 0xffffu;
                all_hi += c >> 16;
                bef_lo += b < cta ? c & 0xffffu : 0u;
                bef_hi += b < cta ? c >> 16 : 0u;
            }
            sum = all_lo + all_hi;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t o = __shfl_up_sync(0xffffffffu, sum, d);
                if (lane >= (uint32_t)d) sum += o;
            }
            if (lane == 31u) S.wsum[warp] = sum;
        }
        // one digit holds every key: the order stays
        stored = !__syncthreads_or(all_lo == n || all_hi == n);
        gave_up = S.gave_up != 0u;                 // written before the barrier only
        if (gave_up) break;
        if (!stored) continue;
        const bool last = pass == npasses - 1;
        if (t == 0 && !last) bar_expect(&S.rec_bar, mine * 16u);
        if (qt == 0) {
            uint32_t at = sum - all_lo - all_hi;
#pragma unroll
            for (uint32_t w = 0; w < kClPairs / 32; ++w) at += w < warp ? S.wsum[w] : 0u;
            S.base[2 * pair] = at + bef_lo;
            S.base[2 * pair + 1] = at + all_lo + bef_hi;
        }
        __syncthreads();
        const uint16_t *qp = reinterpret_cast<const uint16_t *>(S.qpre[warp >> 3]);
#pragma unroll
        for (int r = 0; r < kIt; ++r) {
            if (r >= rounds || wfirst + 32u * (uint32_t)r + lane >= mine) break;
            const uint64_t key = rec[r].x | (uint64_t)rec[r].y << 32;
            const uint32_t d = (uint32_t)(key >> shift) & (kClRadix - 1u);
            const uint32_t g = S.base[d] + qp[d] + wc[d] + rank[r];
            if (g >= n) {                          // cannot be: the counts are whole
                atomicOr(status, ST_INTERNAL);
            } else if (last) {
                keys[g] = key;
                vals[g] = rec[r].z;
            } else if (hold != (cta | kHoldKeys)) {
                const uint32_t b = g / slice;
                cluster_send(cluster_addr(&S.rec[cur ^ 1][g - b * slice], b), cluster_addr(&S.rec_bar, b), rec[r]);
            }
        }
        cur ^= 1;
        ++moved;
        // the next pass clears the warps' counts, which every thread has read
        __syncthreads();
    }
    if (gave_up) {
        if (t == 0) atomicOr(status, ST_TIMEOUT);
    } else if (!stored) {
        // the last pass had nothing to move: the keys are here
        for (uint32_t r = t; r < mine; r += kClThreads) {
            const uint4 v = S.rec[cur][r];
            keys[lo + r] = v.x | (uint64_t)v.y << 32;
            vals[lo + r] = v.z;
        }
    }
    cluster_sync();                                // no block ends while others may send to it
    if (gave_up && t == 0) {
        // What others sent before they stopped: a barrier that never completes only
        // takes the limit.  The wait that ran out was for the keys of the pass before
        // (then this pass's counts may be on their way) ...
        if (!S.gave_up) bar_wait(&S.rec_bar, (moved - 1u) & 1u, kClDrainLimit);
        bar_wait(&S.cnt_bar[pass & 1], (uint32_t)(pass >> 1) & 1u, kClDrainLimit);
        if (S.gave_up) {
            // ... or for this pass's counts (then its keys and the next one's counts)
            bar_expect(&S.rec_bar, mine * 16u);
            bar_wait(&S.rec_bar, moved & 1u, kClDrainLimit);
            bar_expect(&S.cnt_bar[(pass + 1) & 1], kClBlocks * kClPairs * 4u);
            bar_wait(&S.cnt_bar[(pass + 1) & 1], (uint32_t)((pass + 1) >> 1) & 1u, kClDrainLimit);
        }
    }
}

struct ClusterLaunch {
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg;
    ClusterLaunch(size_t smem, cudaStream_t s) : attr(), cfg() {
        cfg.gridDim = kClBlocks;
        cfg.blockDim = kClThreads;
        cfg.dynamicSmemBytes = smem;
        cfg.stream = s;
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim = {kClBlocks, 1, 1};
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 2;
    }
};

template <int kIt>
bool cluster_prepare() {
    auto kern = k_cluster_sort<kIt>;
    const size_t smem = sizeof(ClusterSmem<kIt>);
    ClusterLaunch l(smem, nullptr);
    l.cfg.numAttrs = 1;
    int count = 0;
    const bool ok = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) == cudaSuccess &&
                    cudaOccupancyMaxActiveClusters(&count, kern, &l.cfg) == cudaSuccess && count > 0;
    if (!ok) cudaGetLastError();
    return ok;
}

// whether a sort of n pairs takes the cluster kernel: asked once per device, since
// one without room for such a cluster takes the passes
bool cluster_fits(int64_t n) {
    if (n > kClusterMax) return false;
    static std::mutex mu;
    static std::map<int, bool> fits;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lk(mu);
    auto it = fits.find(dev);
    if (it == fits.end())
        it = fits.emplace(dev, cluster_prepare<1>() && cluster_prepare<2>() && cluster_prepare<4>()).first;
    return it->second;
}

template <int kIt>
void cluster_sort(uint64_t *keys, uint32_t *vals, int64_t n, int rounds, int npasses, uint32_t *status, cudaStream_t s,
                  uint32_t hold = kHoldNone) {
    ClusterLaunch l(sizeof(ClusterSmem<kIt>), s);
    const int64_t chunk = 32 * rounds;     // a warp's keys
    const uint32_t slice = (uint32_t)((((n + kClBlocks - 1) / kClBlocks + chunk - 1) / chunk) * chunk);
    cudaLaunchKernelEx(&l.cfg, k_cluster_sort<kIt>, keys, vals, (uint32_t)n, slice, rounds, npasses, status,
                       hold);
    note_launch();
}

}  // namespace

og_status sort_wait_timeout_probe(og_ctx *c, int64_t n, bool keys_held) {
    if (n < kClBlocks || !cluster_fits(n)) {
        set_error("og_debug_sort_wait_timeout: n must lie in [%d, %lld], on a device with room for the cluster",
                  kClBlocks, (long long)kClusterMax);
        return OG_ERR_ARG;
    }
    cudaStream_t s = c->stream;
    std::vector<uint64_t> k((size_t)n), k_in((size_t)n);
    std::vector<uint32_t> v((size_t)n);
    for (int64_t i = 0; i < n; ++i) {
        k_in[(size_t)i] = k[(size_t)i] = ((uint64_t)(i + 1) * 0x9e3779b97f4a7c15ull) >> 1;
        v[(size_t)i] = (uint32_t)i;
    }
    void *buf = nullptr;
    cudaError_t e = dev_malloc_async(&buf, (size_t)n * 12, s);
    if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? OG_ERR_OOM : cuda_fail(e, "cudaMallocAsync (probe)");
    uint64_t *dk = static_cast<uint64_t *>(buf);
    uint32_t *dv = reinterpret_cast<uint32_t *>(dk + n);
    cudaMemcpyAsync(dk, k.data(), (size_t)n * 8, cudaMemcpyHostToDevice, s);
    cudaMemcpyAsync(dv, v.data(), (size_t)n * 4, cudaMemcpyHostToDevice, s);
    const uint32_t hold = keys_held ? kHoldKeys : 0u;   // block 0 has keys at any n
    const int rounds = (int)((n + kClBlocks * kClThreads - 1) / (kClBlocks * kClThreads));
    const int np = (63 + kClBits - 1) / kClBits;
    if (rounds <= 1) cluster_sort<1>(dk, dv, n, rounds, np, c->d_status, s, hold);
    else if (rounds <= 2) cluster_sort<2>(dk, dv, n, rounds, np, c->d_status, s, hold);
    else cluster_sort<4>(dk, dv, n, rounds, np, c->d_status, s, hold);
    cudaMemcpyAsync(k.data(), dk, (size_t)n * 8, cudaMemcpyDeviceToHost, s);
    cudaMemcpyAsync(v.data(), dv, (size_t)n * 4, cudaMemcpyDeviceToHost, s);
    cudaFreeAsync(buf, s);
    e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail(e, "sort probe");
    // whatever was moved: pairs that came in, at places inside the arrays
    for (int64_t i = 0; i < n; ++i)
        if (v[(size_t)i] >= n || k[(size_t)i] != k_in[v[(size_t)i]]) {
            set_error("og_debug_sort_wait_timeout: pair %lld is none of those sorted", (long long)i);
            return OG_ERR_STATE;
        }
    return OG_OK;
}

size_t radix_sort_scratch_bytes(int64_t n) {
    int64_t ntiles = (n + kTile - 1) / kTile;
    // every-pass sort: per-tile counts and their scan
    size_t counts = (size_t)kRadix * ntiles * sizeof(uint32_t);
    size_t every = counts + scan_scratch_bytes((int64_t)kRadix * ntiles) + 8 * kRadix * sizeof(uint32_t) +
                   1024;
    // one-kernel passes: histograms, tile counters, one look word per tile and digit
    size_t one = 8 * kRadix * sizeof(uint32_t) + 256 + (size_t)kRadix * ntiles * sizeof(unsigned long long) +
                 1024;
    // large sorts: histograms, counters, the count scans' look words, counts, scan scratch
    size_t large = 8 * kRadix * sizeof(uint32_t) + 256 + scan_look_words((int64_t)kRadix * ntiles) * 8 + 256 +
                   counts + scan_scratch_bytes((int64_t)kRadix * ntiles) + 1024;
    if (large > one) one = large;
    return every > one ? every : one;
}

// word offset of the look words: the digit histograms and 64 tile counters before them
constexpr int64_t kLookAt = (8 * kRadix * sizeof(uint32_t) + 256) / sizeof(unsigned long long);

unsigned long long *radix_sort_clear(int64_t n, void *scratch, int64_t *words) {
    const int64_t ntiles = (n + kTile - 1) / kTile;
    if (cluster_fits(n)) {
        *words = 0;
        return nullptr;
    }
    // one-kernel passes: a look word per tile and digit; large sorts: the look words of
    // the tile counts' one-kernel scans (one tag per pass), the counts follow them
    *words = kLookAt + (ntiles > kOneSweepMaxTiles ? (int64_t)scan_look_words((int64_t)kRadix * ntiles)
                                                   : (int64_t)kRadix * ntiles);
    return reinterpret_cast<unsigned long long *>((reinterpret_cast<uintptr_t>(scratch) + 255) & ~(uintptr_t)255);
}

void radix_sort_pairs(uint64_t *keys, uint32_t *vals, uint64_t *keys_alt, uint32_t *vals_alt,
                      int64_t n, int bits, void *scratch, cudaStream_t s, bool *result_in_alt,
                      uint32_t *status, bool cleared) {
    *result_in_alt = false;
    if (n <= 1) return;
    if (cluster_fits(n)) {
        const int rounds = (int)((n + kClBlocks * kClThreads - 1) / (kClBlocks * kClThreads));
        const int np = (bits + kClBits - 1) / kClBits;
        if (rounds <= 1) cluster_sort<1>(keys, vals, n, rounds, np, status, s);
        else if (rounds <= 2) cluster_sort<2>(keys, vals, n, rounds, np, status, s);
        else cluster_sort<4>(keys, vals, n, rounds, np, status, s);
        return;
    }
    int64_t ntiles = (n + kTile - 1) / kTile;
    int64_t nclear;
    unsigned long long *p = radix_sort_clear(n, scratch, &nclear);
    uint32_t *hist8 = reinterpret_cast<uint32_t *>(p);
    uint32_t *tile_ctr = hist8 + 8 * kRadix;
    unsigned long long *look = p + kLookAt;
    const size_t scan_words = scan_look_words((int64_t)kRadix * ntiles);

    // the digit histograms of all passes (they give every pass its digit
    // bases and show which passes are trivial); counters and look words cleared
    if (!cleared) cudaMemsetAsync(p, 0, (size_t)nclear * sizeof(unsigned long long), s);
    int grid = (int)((n + kThreads * 16 - 1) / (kThreads * 16));
    if (grid > 1184) grid = 1184;
    launch_pdl(k_all_digits, grid, kThreads, 0, s, keys, n, hist8);

    static bool attr_set = false;
    if (!attr_set) {
        cudaFuncSetAttribute(k_downsweep, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(DownSmem));
        cudaFuncSetAttribute(k_onesweep, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(DownSmem));
        attr_set = true;
    }
    uint64_t *kin = keys, *kout = keys_alt;
    uint32_t *vin = vals, *vout = vals_alt;
    int npasses = (bits + 7) / 8;
    if (ntiles > kOneSweepMaxTiles) {
        // many tiles: the look-back's waits cost more than the count and scan
        // launches they save
        uint32_t *counts = reinterpret_cast<uint32_t *>(
            (reinterpret_cast<uintptr_t>(look + scan_words) + 255) & ~(uintptr_t)255);
        void *scan_scratch = counts + (size_t)kRadix * ntiles;   // the two-kernel form's tile totals
        for (int pass = 0; pass < npasses; ++pass) {
            const int shift = 8 * pass;
            launch_pdl(k_upsweep, (unsigned)ntiles, kThreads, 0, s, (const uint64_t *)kin, n, shift, counts,
                       ntiles, (const uint32_t *)hist8);
            scan_exclusive_u32_look(counts, counts, (int64_t)kRadix * ntiles, nullptr, look, tile_ctr + 8 + pass,
                                    (uint32_t)(pass + 1), status, scan_scratch, s);
            launch_pdl(k_downsweep, (unsigned)ntiles, kThreads, sizeof(DownSmem), s, (const uint64_t *)kin,
                       (const uint32_t *)vin, kout, vout, n, shift, (const uint32_t *)counts, ntiles,
                       (const uint32_t *)hist8);
            uint64_t *tk = kin; kin = kout; kout = tk;
            uint32_t *tv = vin; vin = vout; vout = tv;
        }
        *result_in_alt = (kin == keys_alt);
        return;
    }
    for (int pass = 0; pass < npasses; ++pass) {
        launch_pdl(k_onesweep, (unsigned)ntiles, kThreads, sizeof(DownSmem), s, (const uint64_t *)kin,
                   (const uint32_t *)vin, kout, vout, n, pass, (const uint32_t *)hist8, look, tile_ctr, status);
        uint64_t *tk = kin; kin = kout; kout = tk;
        uint32_t *tv = vin; vin = vout; vout = tv;
    }
    *result_in_alt = (kin == keys_alt);
}

void radix_sort_pairs_every_pass(uint64_t *keys, uint32_t *vals, uint64_t *keys_alt,
                                 uint32_t *vals_alt, int64_t n, int bits, void *scratch,
                                 cudaStream_t s) {
    if (n <= 1) return;
    int64_t ntiles = (n + kTile - 1) / kTile;
    char *p = static_cast<char *>(scratch);
    uint32_t *counts = reinterpret_cast<uint32_t *>(p);
    p += (size_t)kRadix * ntiles * sizeof(uint32_t);
    p += 8 * kRadix * sizeof(uint32_t);
    void *scan_scratch = p;
    cudaFuncSetAttribute(k_downsweep, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)sizeof(DownSmem));
    uint64_t *kin = keys, *kout = keys_alt;
    uint32_t *vin = vals, *vout = vals_alt;
    const int npasses = (bits + 7) / 8;
    for (int pass = 0; pass < npasses; ++pass) {
        const int shift = 8 * pass;
        launch_pdl(k_upsweep, (unsigned)ntiles, kThreads, 0, s, kin, n, shift, counts, ntiles, nullptr);
        scan_exclusive_u32(counts, counts, (int64_t)kRadix * ntiles, nullptr, scan_scratch, s);
        launch_pdl(k_downsweep, (unsigned)ntiles, kThreads, sizeof(DownSmem), s, kin, vin, kout, vout, n,
                                                                         shift, counts, ntiles, nullptr);
        uint64_t *tk = kin; kin = kout; kout = tk;
        uint32_t *tv = vin; vin = vout; vout = tv;
    }
}

}  // namespace og
