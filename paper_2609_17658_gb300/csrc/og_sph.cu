// og_sph.cu -- grouped neighbour search and SPH density at given smoothing
// lengths (Sect. 3.4 "Neighbour search", Sect. 6 "Smoothed Particle
// Hydrodynamics").
//
// rho_i = sum_j m_j W(|x_i - x_j|, h_i) over the particles j (i included)
// closer than h_i, with the cubic spline W = 8 / (pi h^3) w(r / h),
// w(q) = 1 - 6 q^2 + 6 q^3 below 1/2, 2 (1 - q)^3 up to 1.
//
// The search is done once per walk group (at most 32 particles that are
// neighbours in key order), as the paper does: one warp per group walks the
// tree from the root with a shared-memory stack of child ranges.  A node is
// opened unless its cell lies farther from the group's integer box than the
// group's largest h (exact 64-bit squared gaps, with a small margin: the
// margin only adds candidates); a particle within that distance of the box is
// a candidate and goes to the warp's shared chunk.  When the chunk fills,
// every lane (one target each) runs over it: j is a neighbour of i iff
// r2 < h2 in float32, r2 = (fx fx + fy fy) + fz fz from the exact integer
// separations and h2 = hg hg, hg = float32(h 2^32 / L), each operation
// rounded on its own, so the neighbour count is the same integer the oracle
// computes.  The density sums w in float32 and is scaled in float64.
//
// A round takes whole ranges from the top of the stack while they hold at most
// 32 child records together (a first range with more, a bucket of coincident
// particles, gives 32 and keeps the rest), one record per lane, so the records
// are loaded at once.  Stack depth: a round pushes at most 32 ranges, so while
// the depth is at most kSphDeep it ends at most 31 above; beyond kSphDeep a
// round takes a single range (one node, at most 8 child nodes), a plain depth-
// first walk that adds at most 7 entries per tree level, 7 x 21 for the
// deepest path: 31 + 147 < 200 entries above kSphDeep.  A push past the
// capacity would still only set the stack-overflow status and drop the range.
// The round count is bounded by the number of nodes plus the buckets' extra
// rounds.  Groups with very many candidates go to a block each (k_sph_long).
#include <cmath>
#include <map>
#include <mutex>

#include "og_internal.h"

namespace og {
namespace {

constexpr int kSphWarps = 4;      // warps (groups) per block: 20 KB of shared memory
constexpr int kSphStack = 512;    // child ranges per warp: first entry | count << 32
constexpr int kSphDeep = kSphStack - 200;  // above this depth a round takes one range
constexpr int kSphChunk = 64;     // candidate particles per warp
constexpr int kSphSmem = kSphWarps * (kSphStack * 8 + kSphChunk * 16);
static_assert(kSphSmem <= 48 * 1024, "shared memory of one block");

struct SphArgs {
    const CRec *crec;
    const uint32_t *ncbeg, *nccnt;
    const uint32_t *gbeg, *gend, *gbox;
    const uint32_t *px, *py, *pz;
    const uint32_t *perm;   // outputs to the caller's order; null: key order
    const uint8_t *done;    // null, or per particle (key order): converged, skip
    const float *hg;        // smoothing length in grid units, sorted order
    int64_t ngroups;
    uint32_t *longs;        // groups left to a block each: their number, then their ids
    int limit;              // candidates above which a group is left to a block
    const uint32_t *many;   // null, or the groups expected above the limit (k_sph_expect)
    uint32_t max_many;      // more than this: no group is left to a block
    int64_t max_rounds;     // nodes + 2 + buckets' extra rounds (<= n / 32)
    double dens;            // 8 / pi * (2^32 / L)^3
    float *rho;             // caller order (key order without perm)
    uint32_t *nngb;         // same order, or null
    uint32_t *status;
};

// interval [lo, lo + len] on the circle of 2^32 grid units
__device__ __forceinline__ uint32_t gap_point(uint32_t c, uint32_t lo, uint32_t len) {
    const uint32_t d = c - lo;
    if (d <= len) return 0u;
    const uint32_t fwd = d - len, back = 0u - d;
    return fwd < back ? fwd : back;
}

__device__ __forceinline__ uint32_t gap_boxes(uint32_t alo, uint32_t la, uint32_t blo, uint32_t lb) {
    if (blo - alo <= la || alo - blo <= lb) return 0u;
    const uint32_t a = blo - (alo + la), b = alo - (blo + lb);
    return a < b ? a : b;
}

__device__ __forceinline__ unsigned long long sq(uint32_t g) {
    return (unsigned long long)g * (unsigned long long)g;
}

// smoothing lengths to grid units in key order; 0 < h < L / 2
__global__ void k_sph_prep(int64_t n, const uint32_t *__restrict__ perm, const float *__restrict__ h,
                           double to_grid, float *__restrict__ hg, uint32_t *status) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double v = (double)h[perm ? perm[i] : (uint32_t)i];
    if (!(v > 0.0) || !(v * to_grid < 2147483648.0)) {   // also false for NaN
        atomicOr(status, ST_BAD_INPUT);
        hg[i] = 0.0f;
        return;
    }
    hg[i] = __double2float_rn(v * to_grid);
}

// A group that finds more than `limit` candidates (SphArgs) is left to a block
// (k_sph_long): a few groups of sparse particles beside a halo's core find tens of
// thousands, and one warp took as long for one of them as the rest of the GPU
// for all other groups (315 on average).  One warp searches 2048 in about 0.3 ms;
// the fewer the groups, the sooner the rest is done and the lower the limit pays.
// A call on clustered sets, start and with a limit of 512 / 1024 / 2048:
// 10k particles 472 -> 188 / 248 / 370 us; 100k 1456 -> 538 / 446 / 554 us; 2.1M
// 2.88 -> 2.55 (1024) / 2.28 (2048) / 2.33 ms (3072).
inline int candidate_limit(int64_t ngroups) { return ngroups < 2000 ? 512 : ngroups < 20000 ? 1024 : 2048; }

// the targets of a group, one per lane, and the search region
struct SphTargets {
    uint32_t me, xi, yi, zi;
    bool active;
    float hgi, h2i, inv_h;
    unsigned long long hm2;
    uint32_t lo[3], gl[3];
};
__device__ __forceinline__ SphTargets sph_targets(const SphArgs &a, int64_t g, unsigned lane) {
    SphTargets t;
    t.me = a.gbeg[g] + lane;
    t.active = t.me < a.gend[g];
    t.xi = t.active ? a.px[t.me] : 0u;
    t.yi = t.active ? a.py[t.me] : 0u;
    t.zi = t.active ? a.pz[t.me] : 0u;
    t.hgi = t.active ? a.hg[t.me] : 0.0f;
    t.h2i = __fmul_rn(t.hgi, t.hgi);
    t.inv_h = t.active && t.hgi > 0.0f ? 1.0f / t.hgi : 0.0f;
    // the group's search radius: the largest h, widened by a margin
    const float hmax = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(t.hgi)));
    const unsigned long long hm = (unsigned long long)(hmax * 1.0001f) + 2ull;
    t.hm2 = hm * hm;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        t.lo[k] = a.gbox[6 * g + k];
        t.gl[k] = a.gbox[6 * g + 3 + k] - t.lo[k];
    }
    return t;
}

// nc candidates for this lane's target
__device__ __forceinline__ void sph_pairs(const uint4 *chunk, int nc, const SphTargets &g, float &sum, uint32_t &cnt) {
    for (int t = 0; t < nc; ++t) {
        const uint4 c = chunk[t];
        const float fx = (float)(int32_t)(c.x - g.xi), fy = (float)(int32_t)(c.y - g.yi),
                    fz = (float)(int32_t)(c.z - g.zi);
        const float r2 = __fadd_rn(__fadd_rn(__fmul_rn(fx, fx), __fmul_rn(fy, fy)), __fmul_rn(fz, fz));
        if (r2 < g.h2i) {
            ++cnt;
            const float q = sqrtf(r2) * g.inv_h;
            const float u = 1.0f - q;
            const float w = q < 0.5f ? 1.0f - 6.0f * q * q * u : 2.0f * u * u * u;
            sum = fmaf(__uint_as_float(c.w), w, sum);
        }
    }
}

// a child record: a node to open, a candidate, or neither
__device__ __forceinline__ void sph_test(const CRec &rec, bool has, const SphTargets &t, bool &push, bool &app) {
    const bool node = has && !(rec.info >> 31);
    push = app = false;
    if (node) {
        const uint32_t lev = (rec.info >> 26) & 31u;
        const uint32_t side = 1u << (32u - lev);    // lev >= 1 for a child node
        const uint32_t msk = ~(side - 1u);
        const unsigned long long g2 = sq(gap_boxes(t.lo[0], t.gl[0], rec.x & msk, side - 1u)) +
                                      sq(gap_boxes(t.lo[1], t.gl[1], rec.y & msk, side - 1u)) +
                                      sq(gap_boxes(t.lo[2], t.gl[2], rec.z & msk, side - 1u));
        push = g2 <= t.hm2;
    } else if (has) {
        const unsigned long long g2 = sq(gap_point(rec.x, t.lo[0], t.gl[0])) +
                                      sq(gap_point(rec.y, t.lo[1], t.gl[1])) +
                                      sq(gap_point(rec.z, t.lo[2], t.gl[2]));
        app = g2 <= t.hm2;
    }
}

__device__ __forceinline__ void sph_store(const SphArgs &a, const SphTargets &t, float sum, uint32_t cnt) {
    if (!t.active) return;
    const uint32_t i = a.perm ? a.perm[t.me] : t.me;
    const double hd = (double)t.hgi;
    a.rho[i] = __double2float_rn(a.dens * (double)sum / (hd * hd * hd));
    if (a.nngb) a.nngb[i] = cnt;
}

// A group by a block of kLongWarps warps: every round takes up to one record per
// thread off one stack, and the chunk's candidates are shared out, warp w the w-th
// part of them for all targets.  The rounds are ordered by block barriers and every
// position by prefix sums, so the sums do not depend on the schedule.  Stack depth
// as in k_sph_density: a round adds at most kLongThreads ranges, beyond kLongDeep
// one range at a time.
constexpr int kLongWarps = 16, kLongThreads = 32 * kLongWarps;
constexpr int kLongStack = 2048, kLongDeep = kLongStack - kLongThreads - 200;
constexpr int kLongChunk = 1024;

// exclusive prefix over the block and its total; every thread calls it
__device__ __forceinline__ uint32_t block_prefix(uint32_t v, uint32_t *tot, uint32_t &total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t inc = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t o = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= d) inc += o;
    }
    __syncthreads();
    if (lane == 31) tot[warp] = inc;
    __syncthreads();
    uint32_t before = 0u;
    total = 0u;
#pragma unroll
    for (int k = 0; k < kLongWarps; ++k) {
        const uint32_t x = tot[k];
        if (k < warp) before += x;
        total += x;
    }
    return before + inc - v;
}

__global__ void __launch_bounds__(kLongThreads) k_sph_long(SphArgs a) {
    __shared__ unsigned long long stk[kLongStack];
    __shared__ uint4 chunk[kLongChunk];
    __shared__ uint32_t recs[kLongThreads], tot[kLongWarps];
    __shared__ float psum[kLongWarps][32];
    __shared__ uint32_t pcnt[kLongWarps][32];
    const int warp = threadIdx.x >> 5, tid = threadIdx.x;
    const unsigned lane = threadIdx.x & 31u;
    const uint32_t nlong = a.longs[0];
    for (uint32_t q = blockIdx.x; q < nlong; q += gridDim.x) {
        const int64_t g = a.longs[1 + q];
        const SphTargets t = sph_targets(a, g, lane);
        if (a.done && __all_sync(0xffffffffu, !t.active || a.done[t.me] != 0)) continue;  // the whole block
        float sum = 0.0f;
        uint32_t cnt = 0;
        int sp = 1, nc = 0;
        __syncthreads();
        if (tid == 0) stk[0] = (unsigned long long)a.ncbeg[0] | ((unsigned long long)a.nccnt[0] << 32);
        __syncthreads();
        for (int64_t round = 0; sp > 0 && round < a.max_rounds; ++round) {
            // the top ranges of the stack, whole while they fit in the block; a first
            // range that does not fit (a bucket) gives what does
            const int top = sp > kLongDeep ? 1 : (sp < kLongThreads ? sp : kLongThreads);
            const unsigned long long r = tid < top ? stk[sp - 1 - tid] : 0ull;
            const uint32_t beg = (uint32_t)r, c = (uint32_t)(r >> 32);
            uint32_t all;
            const uint32_t cc = c <= (uint32_t)kLongThreads ? c : (uint32_t)kLongThreads + 1u;
            const uint32_t excl = block_prefix(tid < top ? cc : 0u, tot, all);
            const bool whole = tid < top && excl + cc <= (uint32_t)kLongThreads;
            const bool bucket = tid == 0 && cc > (uint32_t)kLongThreads;
            const int take = __syncthreads_count(whole);
            if (whole)
                for (uint32_t k = 0; k < c; ++k) recs[excl + k] = beg + k;
            if (bucket) {
                for (uint32_t k = 0; k < (uint32_t)kLongThreads; ++k) recs[k] = beg + k;
                stk[sp - 1] = (unsigned long long)(beg + kLongThreads) | ((unsigned long long)(c - kLongThreads) << 32);
            }
            uint32_t total;
            (void)block_prefix(whole ? c : bucket ? (uint32_t)kLongThreads : 0u, tot, total);
            sp -= take;
            CRec rec{};
            const bool has = (uint32_t)tid < total;
            if (has) rec = a.crec[recs[tid]];
            bool push, app;
            sph_test(rec, has, t, push, app);
            // both counts in one prefix sum: pushes above, candidates below
            uint32_t both;
            const uint32_t at = block_prefix((push ? 1u << 16 : 0u) + (app ? 1u : 0u), tot, both);
            if (push) {
                const int pos = sp + (int)(at >> 16);
                if (pos < kLongStack) stk[pos] = (unsigned long long)rec.ref | ((unsigned long long)(rec.info & 0x3ffffffu) << 32);
                else atomicOr(a.status, ST_STACK_OVF);
            }
            if (app) chunk[nc + (int)(at & 0xffffu)] = make_uint4(rec.x, rec.y, rec.z, __float_as_uint(rec.m));
            sp += (int)(both >> 16);
            if (sp > kLongStack) sp = kLongStack;
            nc += (int)(both & 0xffffu);
            __syncthreads();
            if (nc > kLongChunk - kLongThreads || sp == 0) {
                const int b = nc * warp / kLongWarps, e = nc * (warp + 1) / kLongWarps;
                sph_pairs(chunk + b, e - b, t, sum, cnt);
                nc = 0;
                __syncthreads();
            }
        }
        if (sp > 0 && tid == 0) atomicOr(a.status, ST_INTERNAL);   // the round bound was reached
        psum[warp][lane] = sum;
        pcnt[warp][lane] = cnt;
        __syncthreads();
        if (warp == 0) {
            float v = psum[0][lane];
            uint32_t k = pcnt[0][lane];
            for (int w = 1; w < kLongWarps; ++w) {
                v = __fadd_rn(v, psum[w][lane]);
                k += pcnt[w][lane];
            }
            sph_store(a, t, v, k);
        }
    }
}

__global__ void __launch_bounds__(32 * kSphWarps) k_sph_density(SphArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int warp = threadIdx.x >> 5;
    const unsigned lane = threadIdx.x & 31u;
    const unsigned lt = (1u << lane) - 1u;
    const int64_t g = (int64_t)blockIdx.x * kSphWarps + warp;
    if (g >= a.ngroups) return;  // the whole warp
    const int limit = a.many && *a.many > a.max_many ? 0x7fffffff : a.limit;
    unsigned long long *stk = reinterpret_cast<unsigned long long *>(smem_raw) + (size_t)warp * kSphStack;
    uint4 *chunk = reinterpret_cast<uint4 *>(smem_raw + (size_t)kSphWarps * kSphStack * 8) +
                   (size_t)warp * kSphChunk;

    const SphTargets t = sph_targets(a, g, lane);
    if (a.done && __all_sync(0xffffffffu, !t.active || a.done[t.me] != 0)) return;  // nothing to redo
    float sum = 0.0f;
    uint32_t cnt = 0;
    auto flush = [&](int nc) {
        __syncwarp();
        sph_pairs(chunk, nc, t, sum, cnt);
        __syncwarp();
    };

    int sp = 0, nc = 0, found = 0;
    if (lane == 0) stk[0] = (unsigned long long)a.ncbeg[0] | ((unsigned long long)a.nccnt[0] << 32);
    sp = 1;
    __syncwarp();
    for (int64_t round = 0; sp > 0 && round < a.max_rounds; ++round) {
        // the top ranges of the stack (lane l holds the l-th from the top) and
        // the running record count over them
        const int top = sp > kSphDeep ? 1 : (sp < 32 ? sp : 32);
        unsigned long long r = 0ull;
        if ((int)lane < top) r = stk[sp - 1 - (int)lane];
        const uint32_t beg = (uint32_t)r, c = (uint32_t)(r >> 32);
        uint32_t incl = c;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t v = __shfl_up_sync(0xffffffffu, incl, d);
            if ((int)lane >= d) incl += v;
        }
        const uint32_t excl = incl - c;    // records of the ranges above this one
        // whole ranges while they fit in 32 records; a first range of more than
        // 32 records (a bucket) gives 32 and keeps the rest on the stack
        const unsigned fit = __ballot_sync(0xffffffffu, (int)lane < top && incl <= 32u);
        int take = __popc(fit);            // ranges taken whole (a prefix of the lanes)
        uint32_t total;
        if (take == 0) {
            total = 32;
            if (lane == 0) stk[sp - 1] = (unsigned long long)(beg + 32u) | ((unsigned long long)(c - 32u) << 32);
            take = 1;
        } else {
            total = __shfl_sync(0xffffffffu, incl, take - 1);
            sp -= take;
        }
        __syncwarp();
        // record t of the round belongs to the range l with excl(l) <= t < incl(l):
        // mark where each taken range starts (every range holds a record) and
        // count the starts at or below t
        const unsigned starts = __reduce_or_sync(0xffffffffu, (int)lane < take ? 1u << excl : 0u);
        const uint32_t owner = (uint32_t)__popc(starts & (0xffffffffu >> (31u - lane))) - 1u;
        const uint32_t obeg = __shfl_sync(0xffffffffu, beg, owner);
        const uint32_t oexcl = __shfl_sync(0xffffffffu, excl, owner);
        const bool has = lane < total;
        CRec rec{};
        if (has) rec = a.crec[obeg + (lane - oexcl)];
        bool push, app;
        sph_test(rec, has, t, push, app);
        const unsigned bp = __ballot_sync(0xffffffffu, push);
        if (push) {
            const int pos = sp + __popc(bp & lt);
            if (pos < kSphStack) stk[pos] = (unsigned long long)rec.ref | ((unsigned long long)(rec.info & 0x3ffffffu) << 32);
            else atomicOr(a.status, ST_STACK_OVF);
        }
        sp += __popc(bp);
        if (sp > kSphStack) sp = kSphStack;
        const unsigned ba = __ballot_sync(0xffffffffu, app);
        if (app) chunk[nc + __popc(ba & lt)] = make_uint4(rec.x, rec.y, rec.z, __float_as_uint(rec.m));
        nc += __popc(ba);
        if (nc > kSphChunk - 32) {
            found += nc;
            if (found > limit) {
                if (lane == 0) a.longs[1 + atomicAdd(&a.longs[0], 1u)] = (uint32_t)g;
                return;
            }
            flush(nc);
            nc = 0;
        }
        __syncwarp();
    }
    if (sp > 0) atomicOr(a.status, ST_INTERNAL);   // the round bound was reached
    flush(nc);
    sph_store(a, t, sum, cnt);
}

// One step of the smoothing-length iteration for every particle not yet
// converged (key order): N_eff = (4 pi / 3) h^3 rho / m against the target N.
// Within tol N it is done; else the step keeps a bracket [lo, hi] of h (lo:
// too few neighbours, hi: too many), expands or shrinks h by 1.26 until both
// ends are known, then bisects in volume, h = cbrt((lo^3 + hi^3) / 2).  A
// particle whose h would reach the cap (just below L / 2) stops there.
__global__ void k_sph_update(int64_t n, double nt, double tol, double hcap, const double *__restrict__ m,
                             const float *__restrict__ rho, float *__restrict__ h, float *__restrict__ lo,
                             float *__restrict__ hi, uint8_t *__restrict__ done,
                             unsigned long long *__restrict__ left) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n || done[i]) return;
    const double hh = (double)h[i];
    if (!(m[i] > 0.0)) {   // a massless particle has no neighbour relation to meet
        done[i] = 1;
        return;
    }
    const double neff = (4.0 * M_PI / 3.0) * hh * hh * hh * (double)rho[i] / m[i];
    if (fabs(neff - nt) <= tol * nt) {
        done[i] = 1;
        return;
    }
    double l = (double)lo[i], u = (double)hi[i];
    if (neff < nt) l = hh; else u = hh;
    double next;
    if (l > 0.0 && u > 0.0) next = cbrt(0.5 * (l * l * l + u * u * u));
    else next = (neff < nt) ? hh * 1.26 : hh / 1.26;
    lo[i] = (float)l;
    hi[i] = (float)u;
    if (next >= hcap) {
        next = hcap;
        if (hh >= hcap) {   // already at the cap and still too few neighbours
            done[i] = 1;
            return;
        }
    }
    h[i] = (float)next;
    atomicAdd(left, 1ull);
}

__global__ void k_sph_to_caller(int64_t n, const uint32_t *__restrict__ perm, const float *__restrict__ hs,
                                const float *__restrict__ rs, const uint32_t *__restrict__ cs,
                                float *__restrict__ h, float *__restrict__ rho, uint32_t *__restrict__ cnt) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint32_t j = perm[i];
    h[j] = hs[i];
    rho[j] = rs[i];
    if (cnt) cnt[j] = cs[i];
}

__global__ void k_sph_gather(int64_t n, const uint32_t *__restrict__ perm, const float *__restrict__ h,
                             float *__restrict__ hs) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    hs[i] = h[perm[i]];
}

inline unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

// How many groups to expect above the limit, from the group's own density over its
// search region: with smoothing lengths far too large (a solver's first steps from one
// mean length) nearly all are, and a block each costs more than a warp each.  The
// count depends on the lengths alone, so a call's bits do not depend on its timing.
// 11 us from a cold cache for the 99k groups of 2.1M particles, whose call takes 2.26 ms.
__global__ void k_sph_expect(SphArgs a, uint32_t *many) {
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    bool above = false;
    if (g < a.ngroups) {
        const uint32_t b = a.gbeg[g], e = a.gend[g];
        float h = 0.0f;
        bool todo = !a.done;
        for (uint32_t i = b; i < e; ++i) {
            h = fmaxf(h, a.hg[i]);
            todo = todo || a.done[i] == 0;
        }
        uint32_t side = 0;
        for (int k = 0; k < 3; ++k) side = max(side, a.gbox[6 * g + 3 + k] - a.gbox[6 * g + k]);
        const float x = side ? 1.0f + 2.0f * h / (float)side : 0.0f;
        above = todo && (float)(e - b) * (x * x * x) > (float)a.limit;
    }
    const unsigned m = __ballot_sync(0xffffffffu, above);
    if ((threadIdx.x & 31u) == 0u && m) atomicAdd(many, (uint32_t)__popc(m));
}

// From this many groups on a call asks k_sph_expect, and leaves no group to a block
// where it expects more than an eighth above the limit.  Below, a block each pays even
// where all groups are long.  From the mean length for every particle to 32 neighbours,
// a warp each always / a block each always / this rule: 100k particles (4.7k groups) 21.3 /
// 14.0 / 14.0 ms, 400k (19k) 55.9 / 56.0 / 46.6, 2.1M (99k) 187 / 311 / 180 (a quarter
// instead of an eighth 197, a half 245, a sixteenth 179 but 50.6 at 400k).
constexpr int64_t kExpectMin = 16384;

// scratch of a search: the long groups' number and list, the expected number
inline size_t long_bytes(int64_t ng) { return (size_t)(ng + 2) * 4; }

// blocks of k_sph_long that the device holds at once, asked once per device
int64_t resident_long() {
    static std::mutex mu;
    static std::map<int, int64_t> blocks;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lk(mu);
    auto it = blocks.find(dev);
    if (it == blocks.end()) {
        int sms = 1, per = 1;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_sph_long, kLongThreads, 0);
        it = blocks.emplace(dev, (int64_t)sms * (per < 1 ? 1 : per)).first;
    }
    return it->second;
}

// the density of every group of the tree, at a.hg
void search(SphArgs &a, char *scratch, cudaStream_t s) {
    if (a.ngroups < 1) return;
    uint32_t *many = reinterpret_cast<uint32_t *>(scratch);
    a.longs = many + 1;
    a.limit = candidate_limit(a.ngroups);
    a.many = nullptr;
    a.max_many = (uint32_t)(a.ngroups / 8);
    cudaMemsetAsync(many, 0, 8, s);
    if (a.ngroups >= kExpectMin) {
        k_sph_expect<<<nblk(a.ngroups, 256), 256, 0, s>>>(a, many); note_launch();
        a.many = many;
    }
    k_sph_density<<<nblk(a.ngroups, kSphWarps), 32 * kSphWarps, kSphSmem, s>>>(a); note_launch();
    // four times as many blocks as fit: the groups' lengths differ, and a block that has
    // none left makes room (300k particles to 64 neighbours: 845 us with the 304 that fit,
    // 835 with 456, 760 with 1216; 2.1M to 32: 2.36, 2.35 and 2.32 ms)
    const int64_t most = a.ngroups < 4 * resident_long() ? a.ngroups : 4 * resident_long();
    k_sph_long<<<(unsigned)most, kLongThreads, 0, s>>>(a); note_launch();
}

}  // namespace
}  // namespace og

using namespace og;

extern "C" og_status og_tree_sph_density(og_tree *t, const float *h, float *rho, uint32_t *n_ngb) {
    if (!t || !h || !rho) { set_error("og_tree_sph_density: NULL argument"); return OG_ERR_ARG; }
    if (t->nseg != 1) { set_error("og_tree_sph_density: a tree of one box only"); return OG_ERR_ARG; }
    if (t->refit) { set_error("og_tree_sph_density: a refitted tree (rebuild it)"); return OG_ERR_STATE; }
    og_ctx *c = t->ctx;
    cudaSetDevice(c->device);
    cudaStream_t s = c->stream;
    const int64_t n = t->n;
    if (n == 0) return OG_OK;
    const bool dev = (t->prm.flags & OG_DEVICE_PTRS) != 0;
    const double half = 0.5 * t->prm.box;
    if (!dev)
        for (int64_t i = 0; i < n; ++i)
            if (!(h[i] > 0.0f) || !((double)h[i] < half)) {
                set_error("og_tree_sph_density: h[%lld] = %g is not in (0, L/2)", (long long)i, (double)h[i]);
                return OG_ERR_ARG;
            }
    const size_t bh = (size_t)n * sizeof(float);
    // scratch: hg (sorted) [+ host staging: h in, rho and counts out]
    const size_t off_in = (bh + 255) & ~(size_t)255;
    const size_t off_long = off_in + (dev ? 0 : 3 * off_in);
    const size_t total = off_long + long_bytes(t->ngroups);
    char *buf = nullptr;
    cudaError_t e = dev_malloc_async(&buf, total, s);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMallocAsync (sph)");
    float *hg = reinterpret_cast<float *>(buf);
    const float *d_h = h;
    float *d_rho = rho;
    uint32_t *d_cnt = n_ngb;
    if (!dev) {
        float *hin = reinterpret_cast<float *>(buf + off_in);
        cudaMemcpyAsync(hin, h, bh, cudaMemcpyHostToDevice, s);
        d_h = hin;
        d_rho = reinterpret_cast<float *>(buf + 2 * off_in);
        d_cnt = n_ngb ? reinterpret_cast<uint32_t *>(buf + 3 * off_in) : nullptr;
    }
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    cudaEventRecord(e0, s);
    const double to_grid = 4294967296.0 / t->prm.box;
    k_sph_prep<<<nblk(n, 256), 256, 0, s>>>(n, t->perm, d_h, to_grid, hg, c->d_status); note_launch();
    SphArgs a;
    a.crec = t->crec;
    a.ncbeg = t->ncbeg;
    a.nccnt = t->nccnt;
    a.gbeg = t->gbeg;
    a.gend = t->gend;
    a.gbox = t->gbox;
    a.px = t->px;
    a.py = t->py;
    a.pz = t->pz;
    a.perm = t->perm;
    a.done = nullptr;
    a.hg = hg;
    a.ngroups = t->ngroups;
    a.max_rounds = t->nnodes + 2 + (n + 31) / 32;
    a.dens = 8.0 / M_PI * to_grid * to_grid * to_grid;
    a.rho = d_rho;
    a.nngb = d_cnt;
    a.status = c->d_status;
    search(a, buf + off_long, s);
    cudaEventRecord(e1, s);
    if (!dev) {
        cudaMemcpyAsync(rho, d_rho, bh, cudaMemcpyDeviceToHost, s);
        if (n_ngb) cudaMemcpyAsync(n_ngb, d_cnt, (size_t)n * sizeof(uint32_t), cudaMemcpyDeviceToHost, s);
    }
    cudaFreeAsync(buf, s);
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) {
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
        return cuda_fail(e, "sph density");
    }
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    t->ms_sph = ms;
    return check_status(c);
}

extern "C" og_status og_tree_sph_smoothing(og_tree *t, double n_target, double tol, int32_t max_iter,
                                           float *h, float *rho, uint32_t *n_ngb, int32_t *iters) {
    if (!t || !h || !rho) { set_error("og_tree_sph_smoothing: NULL argument"); return OG_ERR_ARG; }
    if (t->nseg != 1) { set_error("og_tree_sph_smoothing: a tree of one box only"); return OG_ERR_ARG; }
    if (t->refit) { set_error("og_tree_sph_smoothing: a refitted tree (rebuild it)"); return OG_ERR_STATE; }
    if (!(n_target > 32.0 / 3.0) || !std::isfinite(n_target) || !(tol > 0.0) || !(tol < 1.0) ||
        max_iter < 1 || max_iter > 1000) {
        set_error("og_tree_sph_smoothing: need N > 32/3 (the self term), 0 < tol < 1, 1 <= max_iter <= 1000");
        return OG_ERR_ARG;
    }
    og_ctx *c = t->ctx;
    cudaSetDevice(c->device);
    cudaStream_t s = c->stream;
    const int64_t n = t->n;
    const bool dev = (t->prm.flags & OG_DEVICE_PTRS) != 0;
    const double half = 0.5 * t->prm.box;
    if (!dev)
        for (int64_t i = 0; i < n; ++i)
            if (!(h[i] > 0.0f) || !((double)h[i] < half)) {
                set_error("og_tree_sph_smoothing: h[%lld] = %g is not in (0, L/2)", (long long)i, (double)h[i]);
                return OG_ERR_ARG;
            }
    // key-order state: h, lo, hi, grid h, rho, counts (4 B each), done (1 B); a
    // counter; host staging of h in/out, rho and counts out
    const size_t b4 = ((size_t)n * 4 + 255) & ~(size_t)255, b1 = ((size_t)n + 255) & ~(size_t)255;
    const size_t off_long = 6 * b4 + b1 + 256 + (dev ? 0 : 3 * b4);
    const size_t total = off_long + long_bytes(t->ngroups);
    char *buf = nullptr;
    cudaError_t e = dev_malloc_async(&buf, total, s);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMallocAsync (sph smoothing)");
    float *hs = reinterpret_cast<float *>(buf), *lo = reinterpret_cast<float *>(buf + b4);
    float *hi = reinterpret_cast<float *>(buf + 2 * b4), *hg = reinterpret_cast<float *>(buf + 3 * b4);
    float *rs = reinterpret_cast<float *>(buf + 4 * b4);
    uint32_t *cs = reinterpret_cast<uint32_t *>(buf + 5 * b4);
    uint8_t *done = reinterpret_cast<uint8_t *>(buf + 6 * b4);
    unsigned long long *left = reinterpret_cast<unsigned long long *>(buf + 6 * b4 + b1);
    float *d_h = h, *d_rho = rho;
    uint32_t *d_cnt = n_ngb;
    if (!dev) {
        char *st = buf + 6 * b4 + b1 + 256;
        d_h = reinterpret_cast<float *>(st);
        d_rho = reinterpret_cast<float *>(st + b4);
        d_cnt = n_ngb ? reinterpret_cast<uint32_t *>(st + 2 * b4) : nullptr;
        cudaMemcpyAsync(d_h, h, (size_t)n * 4, cudaMemcpyHostToDevice, s);
    }
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    cudaEventRecord(e0, s);
    k_sph_gather<<<nblk(n, 256), 256, 0, s>>>(n, t->perm, d_h, hs); note_launch();
    cudaMemsetAsync(lo, 0, 2 * b4, s);   // lo and hi: no bracket yet
    cudaMemsetAsync(done, 0, b1, s);
    const double to_grid = 4294967296.0 / t->prm.box;
    SphArgs a;
    a.crec = t->crec;
    a.ncbeg = t->ncbeg;
    a.nccnt = t->nccnt;
    a.gbeg = t->gbeg;
    a.gend = t->gend;
    a.gbox = t->gbox;
    a.px = t->px;
    a.py = t->py;
    a.pz = t->pz;
    a.perm = nullptr;
    a.done = done;
    a.hg = hg;
    a.ngroups = t->ngroups;
    a.max_rounds = t->nnodes + 2 + (n + 31) / 32;
    a.dens = 8.0 / M_PI * to_grid * to_grid * to_grid;
    a.rho = rs;
    a.nngb = cs;
    a.status = c->d_status;
    const double hcap = std::nextafter((float)(half * 0.999), 0.0f);
    int32_t it = 0;
    og_status st = OG_OK;
    while (it < max_iter) {
        k_sph_prep<<<nblk(n, 256), 256, 0, s>>>(n, nullptr, hs, to_grid, hg, c->d_status); note_launch();
        search(a, buf + off_long, s);
        ++it;
        cudaMemsetAsync(left, 0, sizeof(unsigned long long), s);
        k_sph_update<<<nblk(n, 256), 256, 0, s>>>(n, n_target, tol, hcap, t->pm64, rs, hs, lo, hi, done, left);
        note_launch();
        unsigned long long h_left = 0;
        cudaMemcpyAsync(&h_left, left, sizeof(h_left), cudaMemcpyDeviceToHost, s);
        if ((e = cudaStreamSynchronize(s)) != cudaSuccess) { st = cuda_fail(e, "sph smoothing"); break; }
        if (h_left == 0) break;
    }
    if (st == OG_OK) {
        // the densities and counts at the final h (a particle that moved in the
        // last step needs them at its new h)
        a.done = nullptr;
        k_sph_prep<<<nblk(n, 256), 256, 0, s>>>(n, nullptr, hs, to_grid, hg, c->d_status); note_launch();
        search(a, buf + off_long, s);
        k_sph_to_caller<<<nblk(n, 256), 256, 0, s>>>(n, t->perm, hs, rs, cs, d_h, d_rho, d_cnt); note_launch();
        cudaEventRecord(e1, s);
        if (!dev) {
            cudaMemcpyAsync(h, d_h, (size_t)n * 4, cudaMemcpyDeviceToHost, s);
            cudaMemcpyAsync(rho, d_rho, (size_t)n * 4, cudaMemcpyDeviceToHost, s);
            if (n_ngb) cudaMemcpyAsync(n_ngb, d_cnt, (size_t)n * 4, cudaMemcpyDeviceToHost, s);
        }
    }
    cudaFreeAsync(buf, s);
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess && st == OG_OK) st = cuda_fail(e, "sph smoothing");
    float ms = 0.f;
    if (st == OG_OK) cudaEventElapsedTime(&ms, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (st) return st;
    t->ms_sph = ms;
    if (iters) *iters = it;
    return check_status(c);
}
