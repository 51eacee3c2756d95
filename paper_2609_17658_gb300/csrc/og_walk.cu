// og_walk.cu -- group-wise tree walk and force evaluation (Sect. 4.1.2, 4.1.3, 4.2).
//
// The paper walks the tree once per target particle with a threaded
// (nextnode / sibling) loop and, on GPUs, processes neighbours in chunks of
// 32.  Here one warp walks the tree once for a whole group of up to 32
// spatially close targets and shares the resulting interaction list:
//
//   list building   the warp keeps a stack of child-array ranges of opened
//                   nodes in shared memory.  Each round the 32 lanes take the
//                   next 64 child records (32-byte records, coalesced loads;
//                   two independent records per lane), and each lane
//                   classifies its records against the group's integer
//                   bounding box:
//                     particle -> PP entry unless beyond the prune distance;
//                     node     -> pruned, opened (range pushed), or PN entry.
//                   Prune and boundary tests are exact integer geometry.  The
//                   Barnes-Hut / relative test is decided in FP32 when the
//                   FP32 value is farther from the threshold than its proven
//                   error bound, and otherwise by the exact FP64 expression
//                   (fixed operation order, no fused operations), so every
//                   decision equals the FP64 decision of the oracle.
//   evaluation      entries (x, y, z, m) go to one of two shared-memory chunks:
//                   "far" entries (integer distance from the group box >= h,
//                   so no target can need the softened kernel) and "near"
//                   entries.  A full chunk is evaluated by every lane for its
//                   two targets: exact int32 minimum-image separations,
//                   converted to FP32, r^2 by FMA, cutoff, rsqrt, erfc split
//                   factor, spline softening for near entries only, FP32
//                   accumulation over the chunk, then a compensated (Kahan) add
//                   into the totals.  A group of g targets takes P = ceil(g / 2)
//                   lanes; 32 / P replicas of them split the chunk's entries,
//                   and the replicas' totals are added in a fixed order at the end,
//                   with their compensations.
//
// What bounds it (2.1M clustered, Barnes-Hut pass, 2.7 ms): instruction issue
// (74 % of cycles) and the pipes behind it.  2.4 G warp instructions, 1.3 G of
// them the far loop: 42 a pair of interactions, beside which the pair keeps the
// multi-function pipe 40 cycles and the FMA pipe 36 busy, so no one unit can be
// relieved alone: forcing the integer differences to the other pipe, registers
// for 6 or 8 blocks per SM, or 2 to 8 entries in flight all measured within 2 %.
// The list building is the other 1 G, about 390 a round of 64 slots.  Two targets
// a lane, the straight-line classification and the erfc from 1 / r took the pass
// from 3.40 to 2.75 ms and the two-pass walk from 7.10 to 5.73 ms (5.69 now).
//
// Work distribution: persistent blocks; warps take groups from a global
// atomic counter, in decreasing order of the previous pass's list length
// when that is known (longest first shortens the tail of the launch), and in
// parts where a list is much longer than the others (kQuota).
#include <algorithm>
#include <map>
#include <mutex>
#include <type_traits>
#include <utility>
#include <vector>

#include "og_internal.h"

namespace og {
namespace {

constexpr int kMaxWarps = 8;       // warps per block: 1..kMaxWarps, chosen at launch
// Stack of child ranges per warp.  A round that takes several ranges may leave at most
// kStackSafe on it: from there a plain depth-first walk, one range (one node, at most 8
// child nodes) a round, ends within the stack, as it adds at most 7 ranges per tree
// level, 7 x 21 on the deepest path.  A round that would leave more is undone and taken
// again with half as many ranges; the next ones take twice as many again.  (One range a round from 172
// on, without trying: walks that open much of a large tree, on trees refitted after
// drifts of a tenth of the box, 48 ms where 768 entries and no such rule took 30.)
// One entry more keeps the range that a round takes in part.
constexpr int kStackCap = 383;
constexpr int kStackSafe = kStackCap - 7 * kLevels;
// A round appends at most 64 entries to either chunk, and a chunk is evaluated
// after the round that takes it above a limit: kNearFlush entries, or `chunk`
// far ones (WalkArgs::chunk, chosen at launch; 64 fewer with two replicas, far_limit in
// k_walk).  Both have room for that round and for the padding of an evaluation:
// fewer than kMaxRep entries in the near chunk, kMaxRep x kFarStep in the far one.  The
// 32 replicas of one pair of targets pad the near chunk to 128 at most, and the far one,
// evaluated 64 entries sooner, to chunk + 127.
constexpr int kMaxRep = 16;        // replicas of a group's targets at most (one or two targets: 32)
constexpr int kFarStep = 4;        // far entries in flight per lane
constexpr int kNearChunk = 128;
constexpr int kNearFlush = kNearChunk - 64 - kMaxRep;
constexpr int kFarPad = 64 + kMaxRep * kFarStep;
constexpr int kMaxChunk = 1024;
static_assert((kNearFlush + 64 + 31) / 32 * 32 <= kNearChunk && 32 * kFarStep - 1 <= kFarPad, "32 replicas' padding");

// Long walks in parts.  The relative criterion gives a few groups (large boxes,
// small accelerations) lists 15 times the mean, and one warp needs 0.3-0.5 ms for
// such a list, however idle the rest of the GPU is.  A walk that is not done
// after kQuota rounds leaves what its stack then holds to kParts - 1 further parts,
// which a second launch walks.  This depends on nothing but the group's own
// walk, so a group's sums are the same whatever else is in the launch.
// Only for boxes of 2049 to 196608 particles: below, no walk gets that far; above,
// the other groups fill the time and the parts cost more than they save.  The rule looks
// at the box and not at the launch, for the same reason; boxes of that size in a batch that
// fills the GPU pay for it: 64 boxes of 4k to 65k 2.80 ms with parts, 2.69 without, both
// passes 4.32 and 4.07; 128 boxes of 4k to 262k 11.96 and 11.92.
// Clustered, accelerations given: 32k 197 -> 154 us, 100k 356 -> 262, 131k 433 ->
// 309, 262k 499 -> 522 (not split); both passes: 65k 901 -> 554, 131k 785 -> 658,
// 2.1M 5.71 -> 6.08 ms (not split).  A quota of 32, 40 or 64 rounds, or 16 and 32
// parts: 262-302 us at 100k.  The Barnes-Hut lists are even enough that splitting
// them gained nothing at any size (131k 258 -> 265-280 us).
constexpr uint32_t kQuota = 48, kParts = 8;
constexpr int kSpill = 240;            // ranges a walk can leave (with more it goes on until they are fewer)
static_assert(kSpill >= kStackSafe && kSpill <= kStackCap, "above kStackSafe a walk soon comes back below it");
constexpr int64_t kSplitMin = 2048, kSplitMax = 196608;
// What a group leaves goes to a slot; the groups take slots as they come.  Mostly few do (1 to 2 in
// 100 groups of a clustered system of 10k to 190k, 1812 of 370k in a batch of 8M particles),
// without the force split nearly all.  A group that finds no slot left walks its parts one
// after another in its own warp and adds them up in the same order, so its sums are the
// same; a launch with that many of them is a full one anyhow.  65k uniform particles without
// the split: 485 us with a slot for every group, 788 with 204 slots, 851 without parts.
// At most 83 MB of slots (groups of 32) and 13 MB of the warps' own places, where a place per
// group and partial sums per particle took 250 B a particle of the whole forest.
constexpr int64_t kSlotMax = 8192;
constexpr int kWarpsPerSm = 21;        // resident ones at most (96 registers a thread)

// shared memory of one warp: its stack, near chunk and far chunk
__host__ __device__ constexpr size_t warp_smem(int chunk) {
    return (kStackCap + 1) * sizeof(uint2) + ((size_t)chunk + kNearChunk + kFarPad) * sizeof(uint4);
}
constexpr size_t kMaxBlockSmem = kMaxWarps * warp_smem(kMaxChunk);
static_assert(kMaxBlockSmem <= 227 * 1024, "walk block exceeds the shared memory of an SM");

// erfc(u) exp(u^2) by Abramowitz & Stegun 7.1.26 (t = 1 / (1 + p u), a polynomial
// a1 t + ... + a5 t^5; the split factor S(u) = exp(-u^2) (erfc(u) exp(u^2) +
// (2 / sqrt(pi)) u) to 7.4e-6 up to the usual cutoff u = 2.25), written in v = 1 - t:
// c0 + v (c1 + ... + v c5), v = p u / (1 + p u) in [0, 1), which comes from 1 / r, so r
// itself is not formed.  A least-maximum fit of S in the same form (p = 0.455) is good
// to 1e-7 at the same cost; it moved a group's smallest acceleration by 2.6e-7 on
// average (p99 2.4e-6, this form 7e-8 and 4e-7), and so a first pass near the threshold
// of the relative criterion to other lists in the second (25 particles of 2.1M by
// more than 1e-5, none this way), and is not used.
constexpr float kErfP = 0.3275911f;
constexpr float kErf0 = 0.999999999f, kErf1 = -3.44449638f, kErf2 = 5.874886615f;
constexpr float kErf3 = -6.222859923f, kErf4 = 3.853875118f, kErf5 = -1.061405429f;
constexpr float kTwoOverSqrtPi = 1.1283791670955126f;

// relative margin of the FP32 opening filter (the FP32 evaluation errs by
// less than 2^-20; inside this band the FP64 expression decides)
constexpr float kFilterHi = 1.0f + 1.0f / 65536.0f;
constexpr float kFilterLo = 1.0f - 1.0f / 65536.0f;
constexpr float kFilterEps = 1.0f / 65536.0f;


// One tree as the walk sees it (a forest counts as one tree).
struct TreeView {
    int64_t n, ngroups;
    const uint32_t *gbeg, *gend, *gbox;
    const uint32_t *gorder;       // processing order of the groups, or null (key order)
    uint32_t *gcost;              // out: list length per group
    const CRec *crec;
    const CExt *cext;             // node extents after a refit (kRefit), else unused
    int64_t nchild, max_rounds;
    const uint32_t *gseg;         // box of each group
    const uint32_t *ncbeg, *nccnt;  // child range of each node (the roots are nodes 0..B-1)
    const WalkParams *segp;       // per-box parameters
    const uint32_t *px, *py, *pz;
    const float *a_old;           // [3][n] sorted, relative criterion only
    float *acc;                   // [3][n] sorted, out
    float *pot;                   // [n] sorted, out (potential launches only)
    uint32_t *npp, *npn;          // [n] sorted, out
    int has_cost;                 // gcost holds the list lengths of a previous pass
    int64_t nall;                 // groups of the tree (ngroups: those to walk)
};

// Places of groups walked in parts, in scratch of the pass: slots that the groups
// take, then one place per warp for the groups that find none.
struct Parts {
    uint32_t slots, own;          // their numbers
    uint32_t pairs;               // of targets in a group at most
    unsigned long long *taken;    // groups that asked for a slot (null: no walks in parts)
    uint2 *head;                  // [slot, then warp] group, ranges left
    uint32_t *done;               // [slot, then warp] further parts finished
    uint2 *spill;                 // [slot, then warp][kSpill] child ranges
    uint2 *cnt;                   // [slot][part] PP and PN entries
    float4 *sums;                 // [slot][part][axis][pair]: two targets' totals, two compensations
    uint2 *own_cnt;               // [warp], summed over the parts so far
    float4 *own_sums;             // [warp][axis][pair], summed over the parts so far
};

struct WalkArgs {
    TreeView tree0;               // the tree of a single-tree launch
    const TreeView *trees;        // several trees: descriptors in device memory
    const uint64_t *goff;         // several trees: first item of each tree, plus the total
    const uint32_t *items;        // several trees: item order (longest list first), or null
    int64_t ntrees, nitems;
    uint32_t *lists;              // debug dump: (group, child slot) pairs
    unsigned long long *list_cursor;
    int64_t list_cap;
    unsigned long long *work;     // item counter
    int warps, chunk;             // launch shape: warps per block, far-chunk entries
    Parts parts;
    int second;                   // the launch that walks the further parts
    int one_seg;                  // a single tree of one box: its parameters are p0
    // The pass that only supplies the relative criterion's previous accelerations: plain
    // sums of whole chunks and of replicas.  Its error of some 2e-7 moves no more than a few
    // decisions of the second pass either way, and the list of a group does not change with
    // how the second pass rounds its sums.
    int plain;
    WalkParams p0;                // the box's parameters, in the launch's own argument space
    unsigned long long *inter;    // interactions evaluated
    unsigned long long *tree_inter;  // several trees: interactions per tree, or null
    uint32_t *status;
};

// multi-function-unit approximations (PTX .approx with flush-to-zero); the
// operands here are never subnormal: r^2 >= 1 in grid units, see eval_near
__device__ __forceinline__ float rsqrt_ftz(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rcp_ftz(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float ex2_ftz(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Intervals on the circle of 2^32 grid units are [lo, hi] with length
// hi - lo (mod 2^32); a drifted interval may wrap through 0.
// point c to the interval [lo, lo + len]
__device__ __forceinline__ uint32_t point_gap(uint32_t c, uint32_t lo, uint32_t len) {
    const uint32_t d = c - lo;
    if (d <= len) return 0u;
    const uint32_t fwd = d - len, back = 0u - d;
    return fwd < back ? fwd : back;
}

// interval [alo, alo + la] to interval [blo, blo + lb]
__device__ __forceinline__ uint32_t box_gap(uint32_t alo, uint32_t la, uint32_t blo, uint32_t lb) {
    if (blo - alo <= la || alo - blo <= lb) return 0u;
    const uint32_t a = blo - (alo + la), b = alo - (blo + lb);
    return a < b ? a : b;
}

__device__ __forceinline__ unsigned long long sq64(uint32_t g) {
    return (unsigned long long)g * (unsigned long long)g;
}

__device__ __forceinline__ float2 dup(float v) { return make_float2(v, v); }

// A lane's two targets: their fixed-point positions.
struct Targets {
    uint32_t x0, y0, z0, x1, y1, z1;
};

// Separations of one entry from a lane's two targets: exact 32-bit minimum-image
// differences, each rounded once to FP32; r^2 by FMA.
__device__ __forceinline__ void separations(const uint4 &s, const Targets &t, float2 &fx, float2 &fy, float2 &fz,
                                            float2 &r2) {
    fx = make_float2((float)(int)(s.x - t.x0), (float)(int)(s.x - t.x1));
    fy = make_float2((float)(int)(s.y - t.y0), (float)(int)(s.y - t.y1));
    fz = make_float2((float)(int)(s.z - t.z0), (float)(int)(s.z - t.z1));
    r2 = __ffma2_rn(fx, fx, __ffma2_rn(fy, fy, __fmul2_rn(fz, fz)));
}

// erfc(u) exp(u^2) from 1 / r (y), u = r / (2 r_s): v = 1 / (1 + y / (p / 2 r_s))
__device__ __forceinline__ float2 erfc_poly(float2 y, float ky) {
    const float2 den = __ffma2_rn(y, dup(ky), dup(1.0f));
    const float2 v = make_float2(rcp_ftz(den.x), rcp_ftz(den.y));
    float2 q = __ffma2_rn(v, dup(kErf5), dup(kErf4));
    q = __ffma2_rn(v, q, dup(kErf3));
    q = __ffma2_rn(v, q, dup(kErf2));
    q = __ffma2_rn(v, q, dup(kErf1));
    return __ffma2_rn(v, q, dup(kErf0));
}

// sums of a lane's two targets over its share of a chunk
struct Sums {
    float2 x, y, z, p;
};

// A lane holds two targets and takes its replica's q consecutive entries of the
// chunk: one shared-memory load serves both, and the two go through the
// arithmetic together as FP32 pairs (the f32x2 operations of sm_100 and later;
// each half is the same IEEE operation as the scalar one).  The chunk is padded
// with massless entries (pad_chunk), so q is the same for every replica and a
// multiple of the unrolling: no bounds test per entry and no remainder loop.
//
// Near entries (closer than h to the group box: the softened kernel may
// apply).  r^2 is guarded from below by 1 (a nonzero integer separation has
// r^2 >= 1 in grid units); a zero separation then contributes f * 0 = 0 exactly,
// the self term included.
// kPot: also the short-range potential sum of m erfc(r / 2 r_s) psi(r), psi the
// potential kernel of the spline (1/r beyond h); the self term (r = 0) is left
// out explicitly, it has no force to vanish with.
template <bool kSplit, bool kPot>
__device__ __forceinline__ Sums eval_near(const uint4 *ch, int q, const Targets &t, const WalkParams &p) {
    Sums a{};
    const float h = p.h, inv_h = p.inv_h, rc2 = p.rc2;
    const float hinv3 = inv_h * inv_h * inv_h;
#pragma unroll 1
    for (const uint4 *end = ch + q; ch != end; ++ch) {
        const uint4 s = *ch;
        float2 fx, fy, fz, r2;
        separations(s, t, fx, fy, fz, r2);
        const float m = __uint_as_float(s.w);
        float2 m2 = dup(m);
        if (kSplit) m2 = make_float2(r2.x < rc2 ? m : 0.0f, r2.y < rc2 ? m : 0.0f);
        const float2 r2c = make_float2(fmaxf(r2.x, 1.0f), fmaxf(r2.y, 1.0f));
        const float2 y = make_float2(rsqrt_ftz(r2c.x), rsqrt_ftz(r2c.y));
        const float2 r = __fmul2_rn(r2c, y);
        float2 mS = m2, erfcv = dup(1.0f);
        if (kSplit) {
            const float2 ec = erfc_poly(y, p.erf_ky);
            const float2 arg = __fmul2_rn(r2c, dup(p.kexp));
            const float2 ex = make_float2(ex2_ftz(arg.x), ex2_ftz(arg.y));
            mS = __fmul2_rn(m2, __fmul2_rn(ex, __ffma2_rn(dup(p.erf_c), r, ec)));
            if (kPot) erfcv = __fmul2_rn(ex, ec);
        }
        const float2 u = __fmul2_rn(r, dup(inv_h));
        const float2 u2 = __fmul2_rn(u, u);
        float2 g = __fmul2_rn(y, __fmul2_rn(y, y));
        if (kPot) {
            const float2 pin = __ffma2_rn(
                u2, __ffma2_rn(u2, __ffma2_rn(u, dup(-32.0f / 5.0f), dup(48.0f / 5.0f)), dup(-16.0f / 3.0f)),
                dup(14.0f / 5.0f));
            float2 pout = __ffma2_rn(u, dup(32.0f / 15.0f), dup(-48.0f / 5.0f));
            pout = __ffma2_rn(u, pout, dup(16.0f));
            pout = __ffma2_rn(u, pout, dup(-32.0f / 3.0f));
            pout = __ffma2_rn(u2, pout, dup(16.0f / 5.0f));
            pout.x -= (1.0f / 15.0f) * rcp_ftz(u.x);
            pout.y -= (1.0f / 15.0f) * rcp_ftz(u.y);
            const float px = r.x < h ? inv_h * (u.x < 0.5f ? pin.x : pout.x) : y.x;
            const float py = r.y < h ? inv_h * (u.y < 0.5f ? pin.y : pout.y) : y.y;
            a.p.x = fmaf((r2.x > 0.0f ? m2.x : 0.0f) * erfcv.x, px, a.p.x);
            a.p.y = fmaf((r2.y > 0.0f ? m2.y : 0.0f) * erfcv.y, py, a.p.y);
        }
        // cubic-spline softened kernel inside h (Monaghan 1985 form); the target
        // itself (r = 0) takes no force whatever its kernel
        if ((r.x < h && r2.x > 0.0f) || (r.y < h && r2.y > 0.0f)) {
            const float2 gin = __fmul2_rn(
                dup(hinv3), __ffma2_rn(u2, __ffma2_rn(u, dup(32.0f), dup(-192.0f / 5.0f)), dup(32.0f / 3.0f)));
            float2 go = __ffma2_rn(u, dup(-32.0f / 3.0f), dup(192.0f / 5.0f));
            go = __ffma2_rn(u, go, dup(-48.0f));
            go = __ffma2_rn(u, go, dup(64.0f / 3.0f));
            const float2 u3 = __fmul2_rn(u2, u);
            go = __ffma2_rn(make_float2(rcp_ftz(u3.x), rcp_ftz(u3.y)), dup(-1.0f / 15.0f), go);
            go = __fmul2_rn(dup(hinv3), go);
            g = make_float2(r.x < h ? (u.x < 0.5f ? gin.x : go.x) : g.x,
                            r.y < h ? (u.y < 0.5f ? gin.y : go.y) : g.y);
        }
        const float2 f = __fmul2_rn(mS, g);
        a.x = __ffma2_rn(f, fx, a.x);
        a.y = __ffma2_rn(f, fy, a.y);
        a.z = __ffma2_rn(f, fz, a.z);
    }
    return a;
}

// Far entries: every target of the group is at least h away (the entry lies
// outside the group box by more than h, and by at least one grid unit), so
// no softening applies and r^2 >= 1 needs no guard.
template <bool kSplit, bool kPot>
__device__ __forceinline__ Sums eval_far(const uint4 *ch, int q, const Targets &t, const WalkParams &p) {
    Sums a{};
    const float rc2 = p.rc2;
#pragma unroll 1
    for (const uint4 *end = ch + q; ch != end; ch += kFarStep) {
#pragma unroll
        for (int k = 0; k < kFarStep; ++k) {
            const uint4 s = ch[k];
            float2 fx, fy, fz, r2;
            separations(s, t, fx, fy, fz, r2);
            const float m = __uint_as_float(s.w);
            float2 m2 = dup(m);
            if (kSplit) m2 = make_float2(r2.x < rc2 ? m : 0.0f, r2.y < rc2 ? m : 0.0f);
            const float2 y = make_float2(rsqrt_ftz(r2.x), rsqrt_ftz(r2.y));
            float2 f;
            if (kSplit) {
                // S(r) r^-3 = (ec + (2 / sqrt(pi)) u) exp(-u^2) r^-3, with the second
                // term's r r^-1 taken as 1: (ec / r + c) exp(-u^2) r^-2
                const float2 ec = erfc_poly(y, p.erf_ky);
                const float2 arg = __fmul2_rn(r2, dup(p.kexp));
                const float2 mex = __fmul2_rn(m2, make_float2(ex2_ftz(arg.x), ex2_ftz(arg.y)));
                if (kPot) a.p = __ffma2_rn(__fmul2_rn(mex, ec), y, a.p);
                f = __fmul2_rn(mex, __fmul2_rn(__ffma2_rn(ec, y, dup(p.erf_c)), __fmul2_rn(y, y)));
            } else {
                if (kPot) a.p = __ffma2_rn(m2, y, a.p);
                f = __fmul2_rn(m2, __fmul2_rn(y, __fmul2_rn(y, y)));
            }
            a.x = __ffma2_rn(f, fx, a.x);
            a.y = __ffma2_rn(f, fy, a.y);
            a.z = __ffma2_rn(f, fz, a.z);
        }
    }
    return a;
}

// Massless entries behind the cnt entries of a chunk, so that R replicas take q
// each; returns q, a multiple of `step`.  They lie one grid unit outside the
// group box, so every target is at r >= 1 and they add an exact 0.  (A box that
// is the whole circle on every axis has no outside, but then every entry is
// near, and near entries guard r themselves.)
__device__ __forceinline__ int pad_chunk(uint4 *ch, int cnt, uint32_t R, uint32_t step, int lane,
                                         const uint32_t *hi) {
    const uint32_t q = ((uint32_t)cnt + R * step - 1u) / (R * step) * step;
    for (uint32_t k = (uint32_t)cnt + (uint32_t)lane; k < R * q; k += 32u)
        ch[k] = make_uint4(hi[0] + 1u, hi[1] + 1u, hi[2] + 1u, 0u);
    return (int)q;
}

// a - b, each half rounded once
__device__ __forceinline__ float2 sub2(const float2 &a, const float2 &b) { return __ffma2_rn(b, dup(-1.0f), a); }

// v into the compensated totals sum - comp of a lane's two targets
__device__ __forceinline__ void kahan_add(float2 &sum, float2 &comp, const float2 &v) {
    const float2 y = sub2(v, comp);
    const float2 t = __fadd2_rn(sum, y);
    comp = sub2(sub2(t, sum), y);
    sum = t;
}

// (s - k) + (os - ok) into s and k, exact but for the rounding of k
__device__ __forceinline__ void pair_add(float2 &s, float2 &k, const float2 &os, const float2 &ok) {
    const float2 t = __fadd2_rn(s, os);
    const float2 b = sub2(t, s);
    const float2 e = __fadd2_rn(sub2(s, sub2(t, b)), sub2(os, b));   // s + os - t, exactly
    k = sub2(__fadd2_rn(k, ok), e);
    s = t;
}

// compensated totals of a lane's two targets: s - k
struct Acc {
    float2 sx{0.f, 0.f}, sy{0.f, 0.f}, sz{0.f, 0.f}, kx{0.f, 0.f}, ky{0.f, 0.f}, kz{0.f, 0.f};
    __device__ __forceinline__ void add(const Sums &t) {
        kahan_add(sx, kx, t.x);
        kahan_add(sy, ky, t.y);
        kahan_add(sz, kz, t.z);
    }
};

// The squared distance of the gaps (gx, gy, gz) in single precision: each
// gap rounded once, then fma(fx, fx, fma(fy, fy, fz * fz)).  Its relative
// error is below 5 * 2^-24.
__device__ __forceinline__ float dist2f(uint32_t gx, uint32_t gy, uint32_t gz) {
    const float fx = (float)gx, fy = (float)gy, fz = (float)gz;
    return fmaf(fx, fx, fmaf(fy, fy, fz * fz));
}

// Barnes-Hut: open iff l2 > th2 * d2 with d2 = (dx*dx + dy*dy) + dz*dz in FP64.
// The FP32 value d2f decides when it is farther from the threshold than its
// error bound; inside that band the FP64 expression does.
__device__ __forceinline__ bool open_bh(uint32_t gx, uint32_t gy, uint32_t gz, float d2f, float l2f,
                                        double l2, const WalkParams &p) {
    const float q = p.th2f * d2f;
    if (l2f > q * kFilterHi) return true;
    if (l2f < q * kFilterLo) return false;
    const double dx = (double)gx, dy = (double)gy, dz = (double)gz;
    const double d2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
    return l2 > __dmul_rn(p.th2, d2);
}

// relative: open iff (G M) l2 > arel (d2 d2), arel = (alpha a_min) s^2, in FP64.
__device__ __forceinline__ bool open_rel(uint32_t gx, uint32_t gy, uint32_t gz, float d2f, float l2f,
                                         double l2, float Mf, double M, float arelf, double arel,
                                         const WalkParams &p) {
    const float lhs = (p.Gf * Mf) * l2f;
    const float rhs = (arelf * d2f) * d2f;
    const bool normal = lhs >= 1e-30f && lhs <= 1e30f && rhs >= 1e-30f && rhs <= 1e30f;
    if (normal) {
        if (lhs > rhs * kFilterHi) return true;
        if (lhs < rhs * kFilterLo) return false;
    }
    const double dx = (double)gx, dy = (double)gy, dz = (double)gz;
    const double d2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
    return __dmul_rn(__dmul_rn(p.G, M), l2) > __dmul_rn(arel, __dmul_rn(d2, d2));
}

// Gap between a node's cell and the group box on one axis, from the cell's
// centre c (cell [c - s2, c + s2 - 1], s2 = half the side).  d = c - lo on
// the circle; outside the box the centre is fwd = d - len past its far end or
// back = -d before its near end.  The centre's own gap is dc = min(fwd, back)
// (0 inside); the cell's gap is dc - s2 when the box lies before the cell
// (fwd side) and dc - s2 + 1 when it lies after it (back side, the cell ends
// at c + s2 - 1), and 0 when that is not positive (they meet).  Equal to the
// interval gap of the cell and the box, exactly.
__device__ __forceinline__ void cell_gap(uint32_t c, uint32_t lo, uint32_t len, uint32_t s2,
                                         uint32_t &dc, uint32_t &cg) {
    const uint32_t d = c - lo;
    const uint32_t fwd = d - len, back = 0u - d;
    const bool inside = d <= len;
    const bool onback = back < fwd;
    dc = inside ? 0u : (onback ? back : fwd);
    const int e = (int)(dc - s2 + (onback ? 1u : 0u));
    cg = e > 0 ? (uint32_t)e : 0u;
}

// x >> n with n >= 32 giving 0 (the hardware shift clamps; C++ leaves it undefined)
__device__ __forceinline__ uint32_t shr(uint32_t x, uint32_t n) {
    uint32_t r;
    asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(n));
    return r;
}

// One child record against the group box: PP / PN entry, opened node (its
// child range to push), or nothing (pruned, or no record in this slot).
struct Cls {
    bool emit, open, isnode, near;
    uint4 ent;
    uint32_t push_ref, push_cnt;
};

// the group box: [lo, hi] per axis on the circle
struct Box {
    uint32_t lo[3], hi[3];
};

// The opening decision in FP64, from gaps on the circle (the rare case where
// single precision, or the short form of the gaps, does not settle it).
template <int kOpen>
__device__ __forceinline__ bool open_exact(const uint4 &c, const Box &b, double l2, double M, double arel,
                                           const WalkParams &p, float &d2f) {
    const uint32_t gx = point_gap(c.x, b.lo[0], b.hi[0] - b.lo[0]);
    const uint32_t gy = point_gap(c.y, b.lo[1], b.hi[1] - b.lo[1]);
    const uint32_t gz = point_gap(c.z, b.lo[2], b.hi[2] - b.lo[2]);
    d2f = dist2f(gx, gy, gz);
    const double dx = (double)gx, dy = (double)gy, dz = (double)gz;
    const double d2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
    if (kOpen == OG_OPEN_BH) return l2 > __dmul_rn(p.th2, d2);
    return __dmul_rn(__dmul_rn(p.G, M), l2) > __dmul_rn(arel, __dmul_rn(d2, d2));
}

// The general form: intervals on the circle, any box, node extents after a refit.
template <int kOpen, bool kSplit, bool kRefit>
__device__ __forceinline__ Cls classify(const TreeView &T, uint32_t ci, bool has, const Box &b,
                                        const WalkParams &p, float arelf, double arel) {
    const uint32_t *lo = b.lo;
    const uint32_t gl[3] = {b.hi[0] - b.lo[0], b.hi[1] - b.lo[1], b.hi[2] - b.lo[2]};
    bool emit = false, open = false, isnode = false, near = false;
    uint4 ent = make_uint4(0u, 0u, 0u, 0u);
    uint32_t push_ref = 0u, push_cnt = 0u;
    if (has && ci < T.nchild) {
        const CRec r = T.crec[ci];
        ent = make_uint4(r.x, r.y, r.z, __float_as_uint(r.m));
        isnode = (r.info >> 31) == 0u;
        // gaps of the particle, or of the node's centre of mass, to the group box
        const uint32_t gx = point_gap(r.x, lo[0], gl[0]);
        const uint32_t gy = point_gap(r.y, lo[1], gl[1]);
        const uint32_t gz = point_gap(r.z, lo[2], gl[2]);
        if (!isnode) {
            const unsigned long long pg2 = sq64(gx) + sq64(gy) + sq64(gz);
            near = pg2 < p.hnear2;
            emit = !kSplit || pg2 <= p.rprune;
        } else {
            bool pruned = false, bnear;
            float l2f;
            double l2;
            if (kRefit) {
                // the node's extent: its cell joined with its drifted members
                const CExt e = T.cext[ci];
                const unsigned long long ell =
                    (unsigned long long)max(e.lx, max(e.ly, e.lz)) + 1ull;
                l2 = (double)ell * (double)ell;
                l2f = (float)l2;
                if (kSplit) {
                    const unsigned long long g2 = sq64(box_gap(lo[0], gl[0], e.sx, e.lx)) +
                                                  sq64(box_gap(lo[1], gl[1], e.sy, e.ly)) +
                                                  sq64(box_gap(lo[2], gl[2], e.sz, e.lz));
                    pruned = g2 > p.rprune;
                }
                // boundary check: the box meets the cube of side 1.2 ell
                // centred on the extent: 10 g <= 6 ell, i.e. g <= floor(3 ell / 5)
                // (ell <= 2^32, so the limit fits in 32 bits)
                const uint32_t blim = (uint32_t)((3ull * ell) / 5ull);
                bnear = point_gap(e.sx + (uint32_t)(((unsigned long long)e.lx + 1ull) >> 1), lo[0], gl[0]) <= blim &&
                        point_gap(e.sy + (uint32_t)(((unsigned long long)e.ly + 1ull) >> 1), lo[1], gl[1]) <= blim &&
                        point_gap(e.sz + (uint32_t)(((unsigned long long)e.lz + 1ull) >> 1), lo[2], gl[2]) <= blim;
            } else {
                // the node's cell, from its level and centre of mass: half side
                // s2 = 2^(31 - lev), centre = (COM with the low 32 - lev bits
                // cleared) + s2
                const uint32_t lev = (r.info >> 26) & 31u;
                const uint32_t s2 = 0x80000000u >> lev;
                const uint32_t keep = ~(2u * s2 - 1u);
                l2f = __uint_as_float((uint32_t)(127 + 64 - 2 * lev) << 23);
                l2 = __longlong_as_double((long long)(1023 + 64 - 2 * lev) << 52);
                uint32_t dcx, dcy, dcz, cgx, cgy, cgz;
                cell_gap((r.x & keep) | s2, lo[0], gl[0], s2, dcx, cgx);
                cell_gap((r.y & keep) | s2, lo[1], gl[1], s2, dcy, cgy);
                cell_gap((r.z & keep) | s2, lo[2], gl[2], s2, dcz, cgz);
                if (kSplit) pruned = sq64(cgx) + sq64(cgy) + sq64(cgz) > p.rprune;
                // boundary check: the box meets the cell enlarged to 0.6 side,
                // 10 dc <= 6 side, i.e. dc <= floor(6 s2 / 5) = s2 + floor(s2 / 5)
                const uint32_t blim = s2 + (__umulhi(s2, 0xCCCCCCCDu) >> 2);
                bnear = dcx <= blim && dcy <= blim && dcz <= blim;
            }
            if (!pruned) {
                const float d2f = dist2f(gx, gy, gz);
                if (bnear) {
                    open = true;
                } else {
                    if (kOpen == OG_OPEN_BH) open = open_bh(gx, gy, gz, d2f, l2f, l2, p);
                    else open = open_rel(gx, gy, gz, d2f, l2f, l2, r.m, r.M, arelf, arel, p);
                }
                emit = !open;
                // conservative: in single precision with a margin above its error
                near = !(d2f >= p.hnear2f);
                push_ref = r.ref;
                push_cnt = r.info & 0x3ffffffu;
            }
        }
    }
    return Cls{emit, open, isnode, near, ent, push_ref, push_cnt};
}

// The short form, for a group whose box sides are in [1, 2^29) grid units and
// whose prune distance is below 2^29: signed differences to the near and far
// sides, no wrap to tell apart, and one straight line for particles and nodes,
// so that the two records of a lane overlap.  About 60 instructions a record,
// where the interval form above takes about 100 in two divergent branches.
//
// With a = lo - c and b = c - hi (signed), the gap of c is max(a, b, 0).  It
// differs from the gap on the circle only where both a and b are positive,
// i.e. for a c within len of the far side of the circle, where it takes the larger
// one; both are above 2^31 - 2^29 there (and with len >= 1 they are never both
// -2^31).  A particle or a cell (half side
// s2 <= 2^30) there is beyond the prune distance either way.  The centre of mass
// of a cell that is not pruned is at most 2 s2 further, so it can be there
// only for a node of level 1; those take the exact branch.
//
// A cell's centre is c = (COM with the low 32 - lev bits cleared) + s2 and its
// gap max(a + 1 - s2, b - s2, 0) = max(max(b - 1, a) - (s2 - 1), 0), as it spans
// [c - s2, c + s2 - 1].  The level of a particle reads as 32 or more: s2 = 0, and
// without the ones the cell is the point itself.
// Boundary check: the box meets the cell enlarged to 0.6 side, max(a, b) <=
// floor(6 s2 / 5) on every axis; 6/5 = 1.0011 0011..., so for s2 = 2^(31 - lev)
// that is 0x99999999 >> lev.
//
// After a refit (kRefit) a node spans its extent [s, s + l] instead, and the gap is
// max(lo - (s + l), s - hi, 0); an extent of 2^30 or more on some axis takes the
// general form.  The centre of mass of members on either side of the box's face is
// the plain mean of their coordinates, far outside the extent, so its gap is taken
// on the circle.  200k particles, Barnes-Hut: 384 -> 345 us.
template <int kOpen, bool kSplit, bool kRefit>
__device__ __forceinline__ Cls classify_short(const TreeView &T, uint32_t ci, bool has, const Box &b,
                                              const WalkParams &p, float arelf, double arel) {
    const uint4 *rec = reinterpret_cast<const uint4 *>(T.crec + (has ? ci : 0u));
    const uint4 q0 = rec[0], q1 = rec[1];
    const uint32_t info = q1.z, lev = info >> 26;
    const bool isnode = (int)info >= 0;
    unsigned long long g2 = 0ull;
    int dc;
    uint32_t g[3], blim, side = 0u;
    bool odd;                  // a node that the short form does not cover
    float l2f;
    const uint32_t c[3] = {q0.x, q0.y, q0.z};
    if (kRefit) {
        const uint4 *ext = reinterpret_cast<const uint4 *>(T.cext + (has ? ci : 0u));
        const uint4 x0 = ext[0], x1 = ext[1];
        const uint32_t es[3] = {x0.x, x0.y, x0.z}, el[3] = {x1.x, x1.y, x1.z};   // zeros for a particle
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const uint32_t s = isnode ? es[k] : c[k], cc = s + ((el[k] + 1u) >> 1);
            const int a = (int)(b.lo[k] - cc), d = (int)(cc - b.hi[k]);
            dc = k == 0 ? max(a, d) : __vimax3_s32(dc, a, d);
            g2 += sq64((uint32_t)__vimax_s32_relu((int)(b.lo[k] - (s + el[k])), (int)(s - b.hi[k])));
            g[k] = point_gap(c[k], b.lo[k], b.hi[k] - b.lo[k]);
        }
        side = max(el[0], max(el[1], el[2])) + 1u;
        odd = side - 1u >= (1u << 30);
        blim = __umulhi(3u * side, 0xCCCCCCCDu) >> 2;   // floor(3 ell / 5)
        const float ell = (float)side;
        l2f = ell * ell;
    } else {
        const int isn = isnode ? 1 : 0;
        const uint32_t mask = shr(0xffffffffu, lev), s2 = shr(0x80000000u, lev);
        blim = shr(0x99999999u, lev);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const uint32_t cc = (c[k] & ~mask) | s2;
            const int a = (int)(b.lo[k] - cc), d = (int)(cc - b.hi[k]);
            dc = k == 0 ? max(a, d) : __vimax3_s32(dc, a, d);
            const uint32_t cg = (uint32_t)__viaddmax_s32_relu(__viaddmax_s32(d, -isn, a), isn - (int)s2, 0);
            g2 += sq64(cg);
            g[k] = (uint32_t)__vimax_s32_relu((int)(b.lo[k] - c[k]), (int)(c[k] - b.hi[k]));
        }
        odd = lev == 1u;
        l2f = __uint_as_float(0x5f800000u - (lev << 24));   // 2^(64 - 2 lev)
    }
    float d2f = dist2f(g[0], g[1], g[2]);
    const bool keep = has && g2 <= p.rprune;
    const bool bnear = dc <= (int)blim;
    bool op, sure;
    if (kOpen == OG_OPEN_BH) {
        const float q = p.th2f * d2f, t = l2f - q;
        op = t > 0.0f;
        sure = fabsf(t) > q * kFilterEps;
    } else {
        const float lhs = (p.Gf * __uint_as_float(q0.w)) * l2f, rhs = (arelf * d2f) * d2f, t = lhs - rhs;
        op = t > 0.0f;
        sure = fabsf(t) > rhs * kFilterEps && fminf(lhs, rhs) >= 1e-30f && fmaxf(lhs, rhs) <= 1e30f;
    }
    if (kRefit) {
        if (__builtin_expect(has && isnode && odd, 0))
            return classify<kOpen, kSplit, kRefit>(T, ci, has, b, p, arelf, arel);
    }
    if (__builtin_expect(keep && isnode && !bnear && (!sure || (!kRefit && odd)), 0)) {
        const double l2 = kRefit ? (double)side * (double)side
                                 : __longlong_as_double((long long)(1023 + 64 - 2 * lev) << 52);
        op = open_exact<kOpen>(q0, b, l2, __hiloint2double((int)q1.y, (int)q1.x), arel, p, d2f);
    }
    const bool open = keep && isnode && (bnear || op);
    // near: in single precision with a margin above its error
    return Cls{keep && !open, open, isnode, !(d2f >= p.hnear2f), q0, q1.w, info & 0x3ffffffu};
}

// kOneSeg: a single tree of one box, whose parameters come from the launch
// argument (constant operands) instead of a per-box record in global memory.
// Registers: at most 96 per thread (64 KB / (96 x 128) gives 5 blocks of 4
// warps per SM, as many as their shared memory allows), 128 with the
// potential output; a block of kMaxWarps warps fits either way.
template <int kOpen, bool kSplit, bool kDump, bool kRefit, bool kMulti, bool kPot = false,
          bool kOneSeg = false>
__global__ void __maxnreg__(kPot ? 128 : 96) k_walk(WalkArgs a);

template <int kOpen, bool kSplit, bool kDump, bool kRefit, bool kMulti, bool kPot, bool kOneSeg>
__global__ void __maxnreg__(kPot ? 128 : 96) k_walk(WalkArgs a) {
    // walks in parts: the relative criterion, one tree
    constexpr bool kParted = kOpen == OG_OPEN_REL && !kMulti;
    // (read from the arguments where it is used: held over the walk it costs a spill)
    auto plain = [&] { return kOpen == OG_OPEN_BH && !kMulti && a.plain != 0; };
    extern __shared__ __align__(16) unsigned char smem[];
    // layout: per warp, its stack, near chunk and far chunk (warp_smem bytes);
    // blockDim.x = 32 * a.warps and the launch sizes smem to match
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int chunk = a.chunk;
    unsigned char *wbase = smem + (size_t)warp * warp_smem(chunk);
    uint2 *stk = reinterpret_cast<uint2 *>(wbase);
    uint4 *chn = reinterpret_cast<uint4 *>(wbase + (kStackCap + 1) * sizeof(uint2));
    uint4 *chf = chn + kNearChunk;
    const unsigned FULL = 0xffffffffu;
    const unsigned lt = (1u << lane) - 1u;

    pdl_wait();
    // Items: the groups, or in the second launch the further parts.  A warp's first
    // item is its own number (neighbours on different SMs), the rest come from a
    // counter: the first ones taken there too would queue every warp of the launch
    // on one address.
    const uint32_t nitems =
        kParted && a.second ? (uint32_t)min(*a.parts.taken, (unsigned long long)a.parts.slots) * (kParts - 1u)
                            : (uint32_t)(kMulti ? a.nitems : a.tree0.ngroups);
    uint32_t item = gridDim.x * (uint32_t)warp + blockIdx.x;
    auto advance = [&] {
        const uint32_t nwarps = gridDim.x * (blockDim.x >> 5);
        if (nitems <= nwarps) return false;
        uint32_t k = 0;
        if (lane == 0) k = (uint32_t)atomicAdd(a.work + (kParted && a.second ? 4 : 0), 1ull);
        item = nwarps + __shfl_sync(FULL, k, 0);
        return true;
    };
    uint32_t job = 0;              // a further part of a group (kParted): its place << 3 | part
    static_assert(kParts == 8, "a job's low three bits");
    for (bool more = true; more && item < nitems; more = (kParted && !a.second && job) || advance()) {
        int64_t g;
        int64_t ti = 0;
        if (kParted && a.second) job = item / (kParts - 1u) << 3 | (1u + item % (kParts - 1u));
        if (kParted && job) {
            g = a.parts.head[job >> 3].x;
        } else if (kMulti) {
            const uint64_t it = a.items ? min(a.items[item], nitems - 1u) : item;   // (as below)
            int64_t lo_t = 0, hi_t = a.ntrees;  // goff[lo_t] <= item < goff[hi_t]
            while (hi_t - lo_t > 1) {
                const int64_t mid = (lo_t + hi_t) >> 1;
                if (a.goff[mid] <= it) lo_t = mid; else hi_t = mid;
            }
            ti = lo_t;
            g = (int64_t)(it - a.goff[ti]);
        } else {
            // (the limit holds after a sort whose wait ran out: ST_TIMEOUT is set)
            g = a.tree0.gorder ? (int64_t)min(a.tree0.gorder[item], (uint32_t)a.tree0.nall - 1u) : (int64_t)item;
        }
        const TreeView &T = kMulti ? a.trees[ti] : a.tree0;
        const uint32_t seg = kOneSeg ? 0u : T.gseg[g];
        const WalkParams &p = kOneSeg ? a.p0 : T.segp[seg];
        const uint32_t gb = T.gbeg[g], ge = T.gend[g];
        const uint32_t gsize = ge - gb;
        Box box;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            box.lo[k] = T.gbox[6 * g + k];
            box.hi[k] = T.gbox[6 * g + 3 + k];
        }
        // the short form of the tests (see classify_short)
        bool compact = kSplit && p.rprune < (1ull << 58);
#pragma unroll
        for (int k = 0; k < 3; ++k) compact = compact && box.hi[k] - box.lo[k] - 1u < (1u << 29) - 1u;
        // Lane -> (target pair, replica): P lanes hold the group's targets, two
        // each, and R = 32 / P replicas of them split the entries.  Two targets a
        // lane fill the warp better than one (P need not be a power of two: a
        // group of 20 keeps 30 of 32 lanes busy, where one target a lane kept 20)
        // and halve the shared-memory loads.
        const uint32_t P = (gsize + 1u) >> 1;
        const uint32_t rep = ((uint32_t)lane * (65536u / P + 1u)) >> 16;   // lane / P
        const uint32_t tl = (uint32_t)lane - rep * P;
        const uint32_t R = P == 1u && !plain() ? 32u : min(32u / P, (uint32_t)kMaxRep);
        const uint32_t share = min(rep, R - 1u);    // the lanes left over repeat the last share, unused
        // far entries after which the chunk is evaluated: a lane's plain sum of one
        // evaluation takes at most chunk / 2 terms (two replicas: 64 entries short of the
        // chunk, as a round may add 64; more replicas: the chunk).  Sums of 2000 terms of
        // one sign in groups of 32 err by 1.9 roundings this way and 2.1 with the whole chunk
        // for all; the time is within 1 %.
        // Groups of one or two targets take every lane (262k particles in groups of 1: 2.72 ms
        // with 16 replicas, 2.58 with 32, 2.69 with one target a lane).
        const int far_limit = plain() ? chunk : P == 1u ? chunk - 64 : min(chunk, (chunk >> 1) * (int)R - 64);
        const uint32_t i0 = gb + 2u * tl;
        const bool two = 2u * tl + 1u < gsize;
        const uint32_t i1 = two ? i0 + 1u : i0;
        const Targets tg = {T.px[i0], T.py[i0], T.pz[i0], T.px[i1], T.py[i1], T.pz[i1]};
        // relative criterion: arel = (alpha * a_min) * s^2, a_min = min over the group
        // of |a_old| in FP64 of the single-precision components
        double arel = 0.0;
        float arelf = 0.0f;
        if (kOpen == OG_OPEN_REL) {
            double an = __longlong_as_double(0x7ff0000000000000ll);  // +inf
            const uint32_t i = gb + (uint32_t)lane;
            if ((uint32_t)lane < gsize) {
                double ax0 = T.a_old[i], ay0 = T.a_old[T.n + i], az0 = T.a_old[2 * T.n + i];
                an = __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(ax0, ax0), __dmul_rn(ay0, ay0)),
                                          __dmul_rn(az0, az0)));
            }
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) an = fmin(an, __shfl_xor_sync(FULL, an, d));
            arel = __dmul_rn(__dmul_rn(p.alpha, an), p.s2);
            arelf = __double2float_rn(arel);
        }

        // the root's children, or this part's share of what the first part left
        int sp = 1, cf = 0, cn = 0;
        const uint32_t part = job & 7u;
        if (kParted && part > 0u) {
            const uint32_t left = a.parts.head[job >> 3].y;
            sp = left >= part ? (int)((left - part) / (kParts - 1u)) + 1 : 0;
            for (int k = lane; k < sp; k += 32)
                stk[k] = a.parts.spill[(uint64_t)(job >> 3) * kSpill + part - 1u + (uint32_t)k * (kParts - 1u)];
        } else if (lane == 0) {
            stk[0] = make_uint2(T.ncbeg[seg], T.nccnt[seg]);
        }
        __syncwarp();
        const uint32_t quota = !kParted || part > 0u || !p.split_long ? 0xffffffffu : kQuota;
        bool leave = false;
        uint32_t rounds = 0;
        int most = 32;                        // ranges the next round takes at most
        const uint32_t nchild = (uint32_t)T.nchild, max_rounds = (uint32_t)T.max_rounds;
        uint32_t cnt_all = 0, my_pn = 0;      // entries (warp), node entries (this lane)
        Acc acc;
        float2 psum = make_float2(0.f, 0.f), pcomp = psum;   // potential totals (kPot), compensated
        bool overflow = false;

        while (true) {
            // every round that is not undone consumes at least one child record and a
            // record is visited at most once per walk: more rounds than that is a bug
            if (++rounds > max_rounds) {
                overflow = true;
                if (lane == 0) atomicOr(a.status, ST_INTERNAL);
                break;
            }
            // a round takes up to 64 child records from the top ranges of the
            // stack: slot l and slot l + 32 go to lane l
            const int nr = min(sp, most);
            uint2 Rg = make_uint2(0u, 0u);
            if (lane < nr) Rg = stk[sp - 1 - lane];
            const uint32_t cnt = Rg.y;
            uint32_t incl = cnt;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                uint32_t o = __shfl_up_sync(FULL, incl, d);
                if (lane >= d) incl += o;
            }
            const uint32_t excl = incl - cnt;
            const bool mine = lane < nr;
            const unsigned fullm = __ballot_sync(FULL, mine && incl <= 64u);
            const int nfull = __popc(fullm);
            const uint32_t total = __shfl_sync(FULL, incl, 31);
            const int ntake = total < 64u ? (int)total : 64;
            // first slot of every range that starts in this round, slots 0..31 and 32..63
            const unsigned slo = __reduce_or_sync(FULL, mine && excl < 32u ? 1u << excl : 0u);
            const unsigned shi = __reduce_or_sync(FULL, mine && excl >= 32u && excl < 64u ? 1u << (excl - 32u) : 0u);
            __syncwarp();
            sp -= nfull;
            if (lane == nfull && mine) {
                stk[kStackCap] = Rg;               // in case the round is undone
                if (excl < 64u) {
                    const uint32_t used = 64u - excl;
                    stk[sp - 1] = make_uint2(Rg.x + used, Rg.y - used);
                }
            }
            // this lane's two child slots: the range of a slot is the last one
            // starting at or before it
            const unsigned upm = lt | (1u << lane);
            const int rj0 = __popc(slo & upm) - 1;
            const int rj1 = __popc(slo) + __popc(shi & upm) - 1;
            const uint32_t base = Rg.x - excl;
            const uint32_t ci0 = __shfl_sync(FULL, base, rj0) + (uint32_t)lane;
            const uint32_t ci1 = __shfl_sync(FULL, base, rj1) + (uint32_t)lane + 32u;
            const bool has0 = lane < ntake && ci0 < nchild, has1 = lane + 32 < ntake && ci1 < nchild;
            // (the two forms as two copies of all that follows from them: their
            // results merged after a branch cost more than the tests)
            auto take = [&](auto form) {
                constexpr bool kShort = decltype(form)::value;
                const Cls c0 = kShort ? classify_short<kOpen, kSplit, kRefit>(T, ci0, has0, box, p, arelf, arel)
                                      : classify<kOpen, kSplit, kRefit>(T, ci0, has0, box, p, arelf, arel);
                const Cls c1 = kShort ? classify_short<kOpen, kSplit, kRefit>(T, ci1, has1, box, p, arelf, arel)
                                      : classify<kOpen, kSplit, kRefit>(T, ci1, has1, box, p, arelf, arel);
                // push opened ranges (the stage Records has checked that every node has
                // children, inside the child array)
                const unsigned bo0 = __ballot_sync(FULL, c0.open), bo1 = __ballot_sync(FULL, c1.open);
                const int np0 = __popc(bo0), npush = np0 + __popc(bo1);
                if (sp + npush > (most > 1 ? kStackSafe : kStackCap)) return false;
                if (c0.open) stk[sp + __popc(bo0 & lt)] = make_uint2(c0.push_ref, c0.push_cnt);
                if (c1.open) stk[sp + np0 + __popc(bo1 & lt)] = make_uint2(c1.push_ref, c1.push_cnt);
                sp += npush;
                // append entries to the far / near chunks (at most 64 each per round)
                const unsigned be0 = __ballot_sync(FULL, c0.emit), be1 = __ballot_sync(FULL, c1.emit);
                const unsigned bq0 = __ballot_sync(FULL, c0.emit && c0.near);
                const unsigned bq1 = __ballot_sync(FULL, c1.emit && c1.near);
                const unsigned bf0 = be0 & ~bq0, bf1 = be1 & ~bq1;
                const int nf0 = __popc(bf0), nq0 = __popc(bq0);
                const int nfar = nf0 + __popc(bf1), nnear = nq0 + __popc(bq1);
                if (c0.emit && c0.isnode) ++my_pn;
                if (c1.emit && c1.isnode) ++my_pn;
                // the chunks are adjacent: far entry k is chn[kNearChunk + k]
                const int at0 = (c0.near ? cn : kNearChunk + cf) + __popc((c0.near ? bq0 : bf0) & lt);
                const int at1 = (c1.near ? cn + nq0 : kNearChunk + cf + nf0) + __popc((c1.near ? bq1 : bf1) & lt);
                if (c0.emit) chn[at0] = c0.ent;
                if (c1.emit) chn[at1] = c1.ent;
                if (kDump && nfar + nnear > 0) {
                    unsigned long long d = 0;
                    if (lane == 0) d = atomicAdd(a.list_cursor, (unsigned long long)(nfar + nnear));
                    d = __shfl_sync(FULL, d, 0);
                    auto dump = [&](unsigned long long at, uint32_t ci) {
                        if (at < (unsigned long long)a.list_cap) {
                            a.lists[2 * at] = (uint32_t)g;
                            a.lists[2 * at + 1] = ci;
                        } else {
                            atomicOr(a.status, ST_LIST_OVF);
                        }
                    };
                    if (c0.emit) dump(d + __popc(be0 & lt), ci0);
                    if (c1.emit) dump(d + __popc(be0) + __popc(be1 & lt), ci1);
                }
                cf += nfar;
                cn += nnear;
                cnt_all += (uint32_t)(nfar + nnear);
                return true;
            };
            bool ok;
            if (kSplit && __builtin_expect(compact, 1)) ok = take(std::integral_constant<bool, true>{});
            else ok = take(std::integral_constant<bool, false>{});
            if (__builtin_expect(!ok, 0)) {
                if (most == 1) {
                    overflow = true;
                    break;
                }
                // undo: the ranges taken whole still lie above sp
                const int taken = min(sp + nfull, most);
                __syncwarp();
                if (nfull < taken && lane == 0) stk[sp - 1] = stk[kStackCap];
                __syncwarp();
                sp += nfull;
                most = taken >> 1;
                continue;
            }
            most = sp > kStackSafe ? 1 : min(2 * most, 32);
            __syncwarp();
            // a chunk above its limit, or the walk's end, is evaluated; flushes are
            // rare, so they are hinted off the round's path
            leave = kParted && rounds >= quota && sp > 0 && sp <= kSpill;
            const bool done = sp == 0 || leave;
            if (__builtin_expect(done || cn > kNearFlush, 0)) {
                const int q = pad_chunk(chn, cn, R, 1u, lane, box.hi);
                __syncwarp();
                const Sums t = eval_near<kSplit, kPot>(chn + share * (uint32_t)q, q, tg, p);
                acc.add(t);
                if (kPot) kahan_add(psum, pcomp, t.p);
                cn = 0;
                __syncwarp();
            }
            if (__builtin_expect(done || cf > far_limit, 0)) {
                const int q = pad_chunk(chf, cf, R, (uint32_t)kFarStep, lane, box.hi);
                __syncwarp();
                const Sums t = eval_far<kSplit, kPot>(chf + share * (uint32_t)q, q, tg, p);
                acc.add(t);
                if (kPot) kahan_add(psum, pcomp, t.p);
                cf = 0;
                __syncwarp();
            }
            if (done) break;
        }
        if (overflow) {
            if (lane == 0) atomicOr(a.status, ST_STACK_OVF);
            job = 0u;
            __syncwarp();
            continue;
        }
        uint32_t cnt_pn = __reduce_add_sync(FULL, my_pn), cnt_pp = cnt_all - cnt_pn;
        // replicas of a target: fixed-order pairwise sums, replica r with r + o, their
        // compensations carried along (plain sums: rounded away)
        auto settle = [&](float2 &v, float2 &k) {
            if (plain()) {
                v = sub2(v, k);
                k = dup(0.0f);
            }
        };
        settle(acc.sx, acc.kx); settle(acc.sy, acc.ky); settle(acc.sz, acc.kz);
        for (uint32_t o = 1; o < R; o <<= 1) {
            const bool in = rep + o < R;
            auto fold = [&](float2 &v, float2 &k) {
                float2 ov, ok, nv = v, nk = k;
                ov.x = __shfl_down_sync(FULL, v.x, o * P); ov.y = __shfl_down_sync(FULL, v.y, o * P);
                ok.x = __shfl_down_sync(FULL, k.x, o * P); ok.y = __shfl_down_sync(FULL, k.y, o * P);
                pair_add(nv, nk, ov, ok);
                if (in) { v = nv; k = plain() ? dup(0.0f) : nk; }
            };
            fold(acc.sx, acc.kx); fold(acc.sy, acc.ky); fold(acc.sz, acc.kz);
            if (kPot) fold(psum, pcomp);
        }
        // A group in parts: every part leaves its sums and counts, and the one that
        // finishes last adds them up in the order of the parts.
        if (kParted && (leave || part > 0u)) {
            // per axis and lane one record of the two targets' totals
            const uint32_t pairs = a.parts.pairs, ax = (kPot ? 4u : 3u) * pairs;   // of one part
            const uint32_t slots = a.parts.slots;
            uint32_t slot = job >> 3;
            if (part == 0u) {
                unsigned long long k = 0;
                if (lane == 0) k = atomicAdd(a.parts.taken, 1ull);
                slot = __shfl_sync(FULL, (uint32_t)min(k, (unsigned long long)slots), 0);
                if (slot == slots) slot += blockIdx.x * (blockDim.x >> 5) + (uint32_t)warp;
                for (int q = lane; q < sp; q += 32) a.parts.spill[(uint64_t)slot * kSpill + q] = stk[q];
                if (lane == 0) {
                    a.parts.head[slot] = make_uint2((uint32_t)g, (uint32_t)sp);
                    a.parts.done[slot] = 0u;
                }
            }
            if (slot >= slots) {
                // no slot: the parts follow in this warp, as its next items
                float4 *w = a.parts.own_sums + (uint64_t)(slot - slots) * ax;
                auto run = [&](uint32_t axis, float2 &v, float2 &k) {
                    float4 &q = w[axis * pairs + tl];
                    if (part > 0u) pair_add(v, k, make_float2(q.x, q.y), make_float2(q.z, q.w));
                    q = make_float4(v.x, v.y, k.x, k.y);
                };
                if (rep == 0u) {
                    run(0u, acc.sx, acc.kx); run(1u, acc.sy, acc.ky); run(2u, acc.sz, acc.kz);
                    if (kPot) run(3u, psum, pcomp);
                }
                uint2 &c = a.parts.own_cnt[slot - slots];
                if (part > 0u) {
                    cnt_pp += c.x;
                    cnt_pn += c.y;
                }
                __syncwarp();
                if (lane == 0) c = make_uint2(cnt_pp, cnt_pn);
                job = part + 1u < kParts ? slot << 3 | (part + 1u) : 0u;
                __syncwarp();
                if (job) continue;
            } else {
                float4 *w = a.parts.sums + ((uint64_t)slot * kParts + part) * ax;
                if (rep == 0u) {
                    w[tl] = make_float4(acc.sx.x, acc.sx.y, acc.kx.x, acc.kx.y);
                    w[pairs + tl] = make_float4(acc.sy.x, acc.sy.y, acc.ky.x, acc.ky.y);
                    w[2u * pairs + tl] = make_float4(acc.sz.x, acc.sz.y, acc.kz.x, acc.kz.y);
                    if (kPot) w[3u * pairs + tl] = make_float4(psum.x, psum.y, pcomp.x, pcomp.y);
                }
                if (lane == 0) a.parts.cnt[(uint64_t)slot * kParts + part] = make_uint2(cnt_pp, cnt_pn);
                if (part == 0u) {          // the second launch walks the further parts
                    __syncwarp();
                    continue;
                }
                __threadfence();
                __syncwarp();
                uint32_t before = 0;
                if (lane == 0) before = atomicAdd(&a.parts.done[slot], 1u);
                before = __shfl_sync(FULL, before, 0);
                if (before + 2u != kParts) continue;
                __threadfence();
                w = a.parts.sums + (uint64_t)slot * kParts * ax;
                auto total = [&](uint32_t axis, float2 &v, float2 &k) {
                    v = k = make_float2(0.f, 0.f);
                    for (uint32_t q = 0; q < kParts; ++q) {
                        const float4 x = __ldcg(w + q * ax + axis * pairs + tl);
                        pair_add(v, k, make_float2(x.x, x.y), make_float2(x.z, x.w));
                    }
                };
                if (rep == 0u) {
                    total(0u, acc.sx, acc.kx); total(1u, acc.sy, acc.ky); total(2u, acc.sz, acc.kz);
                    if (kPot) total(3u, psum, pcomp);
                }
                cnt_pp = cnt_pn = 0u;
                for (uint32_t q = 0; q < kParts; ++q) {
                    const uint2 c = __ldcg(&a.parts.cnt[(uint64_t)slot * kParts + q]);
                    cnt_pp += c.x;
                    cnt_pn += c.y;
                }
            }
        }
        if (rep == 0u) {
            const float2 vx = __fmul2_rn(sub2(acc.sx, acc.kx), dup(p.out_scale));
            const float2 vy = __fmul2_rn(sub2(acc.sy, acc.ky), dup(p.out_scale));
            const float2 vz = __fmul2_rn(sub2(acc.sz, acc.kz), dup(p.out_scale));
            const float2 vp = kPot ? __fmul2_rn(sub2(psum, pcomp), dup(-p.pot_scale)) : vx;
            T.acc[i0] = vx.x;
            T.acc[T.n + i0] = vy.x;
            T.acc[2 * T.n + i0] = vz.x;
            T.npp[i0] = cnt_pp - 1u;
            T.npn[i0] = cnt_pn;
            if (kPot) T.pot[i0] = vp.x;
            if (two) {
                T.acc[i1] = vx.y;
                T.acc[T.n + i1] = vy.y;
                T.acc[2 * T.n + i1] = vz.y;
                T.npp[i1] = cnt_pp - 1u;
                T.npn[i1] = cnt_pn;
                if (kPot) T.pot[i1] = vp.y;
            }
        }
        if (lane == 0) {
            T.gcost[g] = cnt_pp + cnt_pn;
            const unsigned long long ni = (unsigned long long)gsize * (unsigned long long)(cnt_pp - 1u + cnt_pn);
            atomicAdd(a.inter, ni);
            if (kMulti && a.tree_inter) atomicAdd(a.tree_inter + ti, ni);
        }
        __syncwarp();
    }
}

template <int kOpen, bool kSplit, bool kDump, bool kRefit, bool kMulti, bool kPot = false,
          bool kOneSeg = false>
void launch_walk_t(const WalkArgs &a, int64_t nitems, cudaStream_t s, int sms) {
    const size_t smem = (size_t)a.warps * warp_smem(a.chunk);
    auto kern = k_walk<kOpen, kSplit, kDump, kRefit, kMulti, kPot, kOneSeg>;
    // resident blocks per SM of each launch shape, queried once per shape
    static std::mutex mu;
    static std::map<std::pair<int, int>, int> per_sm_of;
    int per_sm = 0;
    {
        std::lock_guard<std::mutex> lk(mu);
        auto it = per_sm_of.find({a.warps, a.chunk});
        if (it != per_sm_of.end()) {
            per_sm = it->second;
        } else {
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxBlockSmem);
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, a.warps * 32, smem);
            if (per_sm < 1) per_sm = 1;
            per_sm_of[{a.warps, a.chunk}] = per_sm;
        }
    }
    int64_t want = (nitems + a.warps - 1) / a.warps;
    int64_t grid = (int64_t)sms * per_sm;
    if (want < grid) grid = want;
    // every warp has a place of its own, where a group may find no slot
    if (a.parts.own && grid > a.parts.own / a.warps) grid = a.parts.own / a.warps;
    if (grid < 1) grid = 1;
    launch_pdl(kern, (unsigned)grid, (unsigned)a.warps * 32u, smem, s, a);
    if (kOpen == OG_OPEN_REL && a.parts.taken) {
        // the further parts: their number is known on the device only
        WalkArgs b = a;
        b.second = 1;
        const int64_t most = a.parts.slots * (int64_t)(kParts - 1u), all = (int64_t)sms * per_sm;
        grid = (most + a.warps - 1) / a.warps;
        launch_pdl(kern, (unsigned)(grid < all ? grid : all), (unsigned)a.warps * 32u, smem, s, b);
    }
}

template <int kOpen, bool kSplit>
void launch_walk(const WalkArgs &a, bool dump, bool refit, bool multi, bool pot, int64_t nitems,
                 cudaStream_t s, int sms) {
    if (pot) {
        // the potential is computed on single trees without list dumps
        if (refit) launch_walk_t<kOpen, kSplit, false, true, false, true, true>(a, nitems, s, sms);
        else launch_walk_t<kOpen, kSplit, false, false, false, true, true>(a, nitems, s, sms);
    } else if (multi) {
        // several trees: the serving loop's walks, Barnes-Hut
        if constexpr (kOpen == OG_OPEN_BH) {
            if (refit) launch_walk_t<kOpen, kSplit, false, true, true>(a, nitems, s, sms);
            else launch_walk_t<kOpen, kSplit, false, false, true>(a, nitems, s, sms);
        }
    } else if (dump) {
        if (refit) launch_walk_t<kOpen, kSplit, true, true, false>(a, nitems, s, sms);
        else launch_walk_t<kOpen, kSplit, true, false, false>(a, nitems, s, sms);
    } else if (a.one_seg) {
        if (refit) launch_walk_t<kOpen, kSplit, false, true, false, false, true>(a, nitems, s, sms);
        else launch_walk_t<kOpen, kSplit, false, false, false, false, true>(a, nitems, s, sms);
    } else {
        if (refit) launch_walk_t<kOpen, kSplit, false, true, false>(a, nitems, s, sms);
        else launch_walk_t<kOpen, kSplit, false, false, false>(a, nitems, s, sms);
    }
}

__global__ void k_cost_keys(int64_t ng, const uint32_t *__restrict__ gcost, uint64_t *keys,
                            uint32_t *vals) {
    int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= ng) return;
    // longest list first in coarse classes, a quarter octave of list length
    // each (the exponent and the next two bits of cost + 1), key order within
    // a class: the long groups still start first, and groups walked together
    // stay close in space, so more of their tree records are still in L2
    const uint32_t c = gcost[g] + 1u;
    const uint32_t e = 31u - __clz(c);
    const uint32_t code = (e << 2) | (e >= 2u ? ((c >> (e - 2u)) & 3u) : 0u);
    keys[g] = (uint64_t)(255u - code);
    vals[g] = (uint32_t)g;
}

// several trees: sort keys of every (tree, group) item, longest list first
__global__ void k_item_keys(int64_t nitems, int64_t ntrees, const uint64_t *__restrict__ goff,
                            const TreeView *__restrict__ trees, uint64_t *keys, uint32_t *vals) {
    int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= nitems) return;
    int64_t lo = 0, hi = ntrees;
    while (hi - lo > 1) {
        const int64_t mid = (lo + hi) >> 1;
        if (goff[mid] <= (uint64_t)q) lo = mid; else hi = mid;
    }
    const TreeView &T = trees[lo];
    const uint32_t cost = T.has_cost ? T.gcost[q - goff[lo]] : 0u;
    // the classes of k_cost_keys: longest first, tree and key order within
    const uint32_t c = cost + 1u;
    const uint32_t e = 31u - __clz(c);
    const uint32_t code = (e << 2) | (e >= 2u ? ((c >> (e - 2u)) & 3u) : 0u);
    keys[q] = (uint64_t)(255u - code);
    vals[q] = (uint32_t)q;
}

int sm_count() {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

template <int kOpen>
void dispatch(const WalkArgs &a, bool split, bool dump, bool refit, bool multi, bool pot,
              int64_t nitems, cudaStream_t s, int sms) {
    if (split) launch_walk<kOpen, true>(a, dump, refit, multi, pot, nitems, s, sms);
    else launch_walk<kOpen, false>(a, dump, refit, multi, pot, nitems, s, sms);
}

void launch(const WalkArgs &a, int opening, bool split, bool dump, bool refit, bool multi,
            int64_t nitems, cudaStream_t s, bool pot = false) {
    const int sms = sm_count();
    if (opening == OG_OPEN_BH) dispatch<OG_OPEN_BH>(a, split, dump, refit, multi, pot, nitems, s, sms);
    else dispatch<OG_OPEN_REL>(a, split, dump, refit, multi, pot, nitems, s, sms);
}

// The places of a pass of `groups` walks: one allocation, laid out by place().
struct PartsScratch {
    uint64_t slots, own, pairs, axes;
    PartsScratch(int64_t groups, int group_max, bool pot) : pairs((uint64_t)(group_max + 1) / 2), axes(pot ? 4u : 3u) {
        slots = (uint64_t)std::min(kSlotMax, groups);
        const int64_t warps = std::min<int64_t>(groups + kMaxWarps, (int64_t)sm_count() * kWarpsPerSm);
        own = kSlotMax >= groups ? 0u : (uint64_t)warps;
    }
    uint64_t place(char *base, Parts *p) const {
        uint64_t at = 0;
        auto take = [&](auto *&q, uint64_t count) {
            using T = std::remove_reference_t<decltype(*q)>;
            q = reinterpret_cast<T *>(base + at);
            at += (count * sizeof(T) + 255u) & ~(uint64_t)255u;
        };
        take(p->head, slots + own);
        take(p->done, slots + own);
        take(p->spill, (slots + own) * kSpill);
        take(p->cnt, slots * kParts);
        take(p->sums, slots * kParts * axes * pairs);
        take(p->own_cnt, own);
        take(p->own_sums, own * axes * pairs);
        p->slots = (uint32_t)slots;
        p->own = (uint32_t)own;
        p->pairs = (uint32_t)pairs;
        return at;
    }
};

// Per-box parameters of a pass (uploaded if the launch reads them as a table) and the tree's view.  The first
// pass of the relative criterion is Barnes-Hut with theta_first_pass.
og_status prepare_view(og_tree *t, int opening, bool first_pass, const float *a_old_sorted,
                       float *acc_sorted, bool table, TreeView *v, WalkParams *wp0, bool *split_long) {
    cudaStream_t s = t->ctx->stream;
    const int64_t B = t->nseg;
    t->h_wp.resize((size_t)B);
    for (int64_t b = 0; b < B; ++b) {
        const og_params &q = t->seg_prm[b];
        t->h_wp[b] = make_walk_params(q, opening, first_pass ? q.theta_first_pass : q.theta);
        if (first_pass) t->h_wp[b].dump = false;
        // FP64 output: the last pass stores the unscaled sums, scaled in FP64 later
        if (!first_pass && t->unscaled_out) t->h_wp[b].out_scale = 1.0f;
        const int64_t nb = (int64_t)t->h_seg_off[b + 1] - (int64_t)t->h_seg_off[b];
        t->h_wp[b].split_long = opening == OG_OPEN_REL && nb > kSplitMin && nb <= kSplitMax;
        if (t->h_wp[b].split_long) *split_long = true;
    }
    *wp0 = t->h_wp[0];
    WalkParams *dp = t->segp + (first_pass ? 0 : B);
    if (table) {
        cudaError_t err = cudaMemcpyAsync(dp, t->h_wp.data(), B * sizeof(WalkParams), cudaMemcpyHostToDevice, s);
        if (err != cudaSuccess) return cuda_fail(err, "walk setup");
    }
    TreeView &w = *v;
    w = TreeView{};
    w.n = t->n;
    w.ngroups = t->ngroups;
    w.nall = t->ngroups;
    w.gbeg = t->gbeg;
    w.gend = t->gend;
    w.gbox = t->gbox;
    w.gcost = t->gcost;
    w.gorder = nullptr;
    w.crec = t->crec;
    w.cext = t->cext;
    w.nchild = t->nchild;
    w.max_rounds = 6 * (t->nchild + 2);      // a round is undone five times at most (32 ranges, 16, .. 2)
    w.gseg = t->gseg;
    w.ncbeg = t->ncbeg;
    w.nccnt = t->nccnt;
    w.segp = dp;
    w.px = t->px;
    w.py = t->py;
    w.pz = t->pz;
    w.a_old = a_old_sorted;
    w.acc = acc_sorted;
    w.npp = t->npp_sorted;
    w.npn = t->npn_sorted;
    w.has_cost = t->have_cost ? 1 : 0;
    return OG_OK;
}

void fill_common(WalkArgs &a, og_ctx *c, og_tree *t) {
    // a tree's launch shape (zero fields take the defaults)
    a.warps = t && t->prm.walk_warps > 0 ? t->prm.walk_warps : kDefaultWalkWarps;
    a.chunk = t && t->prm.walk_chunk > 0 ? t->prm.walk_chunk : kDefaultWalkChunk;
    a.lists = t ? t->lists : nullptr;
    a.list_cap = t ? t->list_cap : 0;
    a.work = c->d_counters;
    a.inter = c->d_counters + 1;
    a.list_cursor = c->d_counters + 2;
    a.status = c->d_status;
}

}  // namespace

WalkParams make_walk_params(const og_params &p, int opening, double theta) {
    WalkParams w{};
    const double two32 = 4294967296.0;
    w.opening = opening;
    w.split = p.r_s > 0.0;
    w.dump = (p.flags & OG_DEBUG_DUMP_LISTS) != 0;
    w.th2 = theta * theta;
    w.th2f = (float)w.th2;
    w.G = p.G;
    w.Gf = (float)p.G;
    const double s = p.box / two32;
    w.s2 = s * s;
    w.alpha = p.alpha;
    if (w.split) {
        const double rcg = (p.rcut_over_rs * p.r_s) / p.box * two32;
        const double rsg = p.r_s / p.box * two32;
        w.rc2 = (float)(rcg * rcg);
        w.rprune = (unsigned long long)(rcg * rcg * (1.0 + 1.0 / 1024.0));
        // exp(-r^2 / (4 r_s^2)) = 2^(r^2 * kexp)
        w.kexp = (float)(-1.4426950408889634 / (4.0 * rsg * rsg));
        w.erf_ky = (float)(2.0 * rsg / (double)kErfP);
        w.erf_c = (float)((double)kTwoOverSqrtPi / (2.0 * rsg));
    } else {
        w.rc2 = __builtin_huge_valf();
        w.rprune = ~0ull;
        w.kexp = 0.0f;
        w.erf_ky = 0.0f;
        w.erf_c = 0.0f;
    }
    const double hg = 2.8 * p.eps / p.box * two32;
    w.h = (float)hg;
    w.inv_h = hg > 0.0 ? (float)(1.0 / hg) : 0.0f;
    // an entry is "near" when its integer distance to the group box is below
    // h (with a generous rounding margin); only near entries may need
    // softening.  An entry inside the group box (a member itself) is always
    // near, so a far entry is at r^2 >= 1 from every target.
    const double hn = hg * (1.0 + 1.0 / 256.0) + 2.0;
    w.hnear2 = hg > 0.0 ? (unsigned long long)(hn * hn) : 1ull;
    // the single-precision square of an integer distance errs by less than
    // 5 * 2^-24 relative, so d2f >= hnear2f implies an exact square >= hnear2
    w.hnear2f = nextafterf((float)((double)w.hnear2 * (1.0 + 1.0 / (1 << 20))), __builtin_huge_valf());
    w.out_scale = (float)(p.G * (two32 / p.box) * (two32 / p.box));
    w.pot_scale = (float)(p.G * (two32 / p.box));
    return w;
}

// The counters before a walk: cleared here, unless the last build or force call left
// them at zero (its last kernel clears them, which saves a memset between two kernels).
static void clear_counters(og_ctx *c) {
    if (!c->counters_zero) cudaMemsetAsync(c->d_counters, 0, kWalkCounters * sizeof(unsigned long long), c->stream);
    c->counters_zero = false;
}

static og_status finish_pass(og_ctx *c, cudaEvent_t e0, cudaEvent_t e1, float *ms_out,
                             unsigned long long h[3]) {
    cudaStream_t s = c->stream;
    cudaMemcpyAsync(h, c->d_counters, 3 * sizeof(unsigned long long), cudaMemcpyDeviceToHost, s);
    cudaError_t err = cudaStreamSynchronize(s);
    float ms = 0;
    cudaEventElapsedTime(&ms, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (err != cudaSuccess) return cuda_fail(err, "walk");
    if ((err = cudaGetLastError()) != cudaSuccess) return cuda_fail(err, "walk launch");
    if (ms_out) *ms_out = ms;
    return OG_OK;
}

// Replace the debug list buffer by one of at least `need` entries and clear
// the overflow bit the short buffer left in the status word.
static og_status grow_lists(og_tree *t, int64_t need) {
    cudaStream_t s = t->ctx->stream;
    cudaError_t e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return cuda_fail(e, "list buffer");
    cudaFree(t->lists);
    t->lists = nullptr;
    t->list_cap = 0;
    const int64_t cap = need + need / 8 + 1024;
    if ((e = cudaMalloc(&t->lists, (size_t)cap * 2 * sizeof(uint32_t))) != cudaSuccess) {
        t->lists = nullptr;
        return cuda_fail(e, "cudaMalloc (lists)");
    }
    t->list_cap = cap;
    uint32_t st = 0;
    if ((e = cudaMemcpy(&st, t->ctx->d_status, sizeof(st), cudaMemcpyDeviceToHost)) != cudaSuccess)
        return cuda_fail(e, "status read");
    st &= ~(uint32_t)ST_LIST_OVF;
    if ((e = cudaMemcpy(t->ctx->d_status, &st, sizeof(st), cudaMemcpyHostToDevice)) != cudaSuccess)
        return cuda_fail(e, "status write");
    return OG_OK;
}

og_status finish_deferred(og_tree *t, float *ms_walk) {
    og_status st = OG_OK;
    for (int k = 0; k < t->npend; ++k) {
        float ms = 0;
        if (cudaEventElapsedTime(&ms, t->pend_e0[k], t->pend_e1[k]) == cudaSuccess && ms_walk)
            *ms_walk += ms;
        cudaEventDestroy(t->pend_e0[k]);
        cudaEventDestroy(t->pend_e1[k]);
        t->pend_e0[k] = t->pend_e1[k] = nullptr;
        const unsigned long long *h = pinned_counters(t->ctx, k);
        t->interactions_last = (int64_t)h[1];
        t->interactions += (int64_t)h[1];
    }
    t->npend = 0;
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) st = cuda_fail(err, "walk launch");
    return st;
}

og_status walk_pass(og_tree *t, int opening, bool first_pass, const float *a_old_sorted,
                    float *acc_sorted, float *ms_out, bool use_order, const uint32_t *subset,
                    int64_t nsubset, float *pot_sorted, bool defer) {
    cudaStream_t s = t->ctx->stream;
    WalkArgs a{};
    WalkParams wp;
    bool split_long = false;
    // one box without list dumps: the parameters come with the launch
    const bool dump = (t->seg_prm[0].flags & OG_DEBUG_DUMP_LISTS) != 0 && !pot_sorted;
    og_status st = prepare_view(t, opening, first_pass, a_old_sorted, acc_sorted, t->nseg > 1 || dump, &a.tree0,
                                &wp, &split_long);
    if (st) return st;
    fill_common(a, t->ctx, t);
    a.one_seg = t->nseg == 1 ? 1 : 0;
    a.p0 = t->h_wp[0];
    a.plain = first_pass ? 1 : 0;
    cudaError_t err;
    void *sort_tmp = nullptr, *pass_tmp = nullptr;
    if (split_long) {
        const PartsScratch sc(subset ? nsubset : t->ngroups, t->prm.group_max, pot_sorted != nullptr);
        if ((err = dev_malloc_async(&pass_tmp, sc.place(nullptr, &a.parts), s)) != cudaSuccess)
            return cuda_fail(err, "cudaMallocAsync (walk parts)");
        sc.place(static_cast<char *>(pass_tmp), &a.parts);
        a.parts.taken = t->ctx->d_counters + 3;
    }
    auto release = [&] {
        if (pass_tmp) cudaFreeAsync(pass_tmp, s);
        if (sort_tmp) cudaFreeAsync(sort_tmp, s);
    };
    if (subset) {
        // only these groups, in this order (the walk takes them from gorder)
        a.tree0.gorder = subset;
        a.tree0.ngroups = nsubset;
    } else if (use_order && t->have_cost && t->ngroups > 1) {
        // longest list first, from the costs of the previous pass on this tree
        const int64_t ng = t->ngroups;
        size_t bytes = (size_t)ng * 24 + radix_sort_scratch_bytes(ng) + 1024;
        if ((err = dev_malloc_async(&sort_tmp, bytes, s)) != cudaSuccess) {
            release();
            return cuda_fail(err, "cudaMallocAsync (group order)");
        }
        char *q = static_cast<char *>(sort_tmp);
        uint64_t *k0 = reinterpret_cast<uint64_t *>(q);
        uint64_t *k1 = k0 + ng;
        uint32_t *v0 = reinterpret_cast<uint32_t *>(k1 + ng);
        uint32_t *v1 = v0 + ng;
        void *scr = v1 + ng + 64;
        k_cost_keys<<<(unsigned)((ng + 255) / 256), 256, 0, s>>>(ng, t->gcost, k0, v0); note_launch();
        bool alt = false;
        radix_sort_pairs(k0, v0, k1, v1, ng, 8, scr, s, &alt, t->ctx->d_status);
        cudaMemcpyAsync(t->gorder, alt ? v1 : v0, ng * sizeof(uint32_t), cudaMemcpyDeviceToDevice, s);
        a.tree0.gorder = t->gorder;
    }
    if (defer && !wp.dump && t->npend < 2) {
        // no host synchronisation: the counters go to page-locked slot npend and
        // the times to events, both read by finish_deferred
        const int k = t->npend;
        clear_counters(t->ctx);
        cudaEventCreate(&t->pend_e0[k]);
        cudaEventCreate(&t->pend_e1[k]);
        cudaEventRecord(t->pend_e0[k], s);
        a.tree0.pot = pot_sorted;
        launch(a, opening, wp.split, false, t->refit, false, a.tree0.ngroups, s, pot_sorted != nullptr);
        cudaEventRecord(t->pend_e1[k], s);
        // the last pass's counters are reported by the caller's last kernel
        if (first_pass)
            cudaMemcpyAsync(pinned_counters(t->ctx, k), t->ctx->d_counters, 3 * sizeof(unsigned long long),
                            cudaMemcpyDeviceToHost, s);
        t->npend = k + 1;
        release();
        // the next pass may take this one's list lengths: stream order makes them ready
        t->have_cost = true;
        if (ms_out) *ms_out = 0.0f;
        return OG_OK;
    }
    unsigned long long h[3] = {0, 0, 0};
    for (int attempt = 0; attempt < 2; ++attempt) {
        clear_counters(t->ctx);
        cudaEvent_t e0, e1;
        cudaEventCreate(&e0);
        cudaEventCreate(&e1);
        cudaEventRecord(e0, s);
        a.tree0.pot = pot_sorted;
        launch(a, opening, wp.split, wp.dump && !pot_sorted, t->refit, false, a.tree0.ngroups, s,
               pot_sorted != nullptr);
        cudaEventRecord(e1, s);
        st = finish_pass(t->ctx, e0, e1, ms_out, h);
        if (st) break;
        if (!wp.dump || h[2] <= (unsigned long long)t->list_cap) break;
        // debug lists only: the pass counted every entry it could not keep;
        // give the buffer that size and walk again (the pass is deterministic)
        st = grow_lists(t, (int64_t)h[2]);
        if (st) break;
        a.lists = t->lists;
        a.list_cap = t->list_cap;
    }
    release();
    if (st) return st;
    t->have_cost = true;
    t->interactions_last = (int64_t)h[1];
    t->interactions += (int64_t)h[1];
    if (wp.dump) t->list_len = (int64_t)(h[2] < (unsigned long long)t->list_cap ? h[2] : t->list_cap);
    return OG_OK;
}

og_status walk_multi(og_ctx *c, og_tree *const *trees, int64_t ntrees, float *const *acc_sorted, float *ms_out,
                     int64_t *interactions, int64_t *tree_interactions) {
    cudaStream_t s = c->stream;
    if (ntrees < 1) return OG_OK;
    std::vector<TreeView> hv((size_t)ntrees);
    std::vector<uint64_t> hoff((size_t)ntrees + 1);
    bool split = false, refit = false;
    uint64_t total = 0;
    for (int64_t k = 0; k < ntrees; ++k) {
        WalkParams wp;
        bool split_long = false;             // never with Barnes-Hut
        og_status st = prepare_view(trees[k], OG_OPEN_BH, false, nullptr, acc_sorted[k], true, &hv[k], &wp,
                                    &split_long);
        if (st) return st;
        if (k == 0) split = wp.split;
        else if (wp.split != split) {
            set_error("walk over several trees: split on/off must agree");
            return OG_ERR_ARG;
        }
        refit = refit || trees[k]->refit;
        hoff[k] = total;
        total += (uint64_t)trees[k]->ngroups;
    }
    hoff[ntrees] = total;
    if (refit) {
        // one instantiation for all trees: built trees read their cells as extents
        for (int64_t k = 0; k < ntrees; ++k) {
            if (!trees[k]->cext) {
                og_status st = cell_extents(trees[k]);
                if (st) return st;
            }
            hv[k].cext = trees[k]->cext;
        }
    }
    const int64_t nitems = (int64_t)total;
    size_t bytes = (size_t)ntrees * sizeof(TreeView) + (size_t)(ntrees + 1) * 8 + (size_t)nitems * 24 +
                   radix_sort_scratch_bytes(nitems) + (size_t)ntrees * 8 + 4096;
    void *tmp = nullptr;
    cudaError_t err;
    if ((err = dev_malloc_async(&tmp, bytes, s)) != cudaSuccess) return cuda_fail(err, "cudaMallocAsync (walk items)");
    char *q = static_cast<char *>(tmp);
    TreeView *dv = reinterpret_cast<TreeView *>(q);
    q += ((size_t)ntrees * sizeof(TreeView) + 255) & ~(size_t)255;
    uint64_t *doff = reinterpret_cast<uint64_t *>(q);
    q += ((size_t)(ntrees + 1) * 8 + 255) & ~(size_t)255;
    uint64_t *k0 = reinterpret_cast<uint64_t *>(q);
    uint64_t *k1 = k0 + nitems;
    uint32_t *v0 = reinterpret_cast<uint32_t *>(k1 + nitems);
    uint32_t *v1 = v0 + nitems;
    unsigned long long *tint = reinterpret_cast<unsigned long long *>(
        (reinterpret_cast<uintptr_t>(v1 + nitems) + 255) & ~(uintptr_t)255);
    void *scr = tint + ntrees + 32;
    cudaMemcpyAsync(dv, hv.data(), ntrees * sizeof(TreeView), cudaMemcpyHostToDevice, s);
    cudaMemcpyAsync(doff, hoff.data(), (ntrees + 1) * 8, cudaMemcpyHostToDevice, s);
    k_item_keys<<<(unsigned)((nitems + 255) / 256), 256, 0, s>>>(nitems, ntrees, doff, dv, k0, v0); note_launch();
    bool alt = false;
    radix_sort_pairs(k0, v0, k1, v1, nitems, 8, scr, s, &alt, c->d_status);
    WalkArgs a{};
    fill_common(a, c, nullptr);
    a.trees = dv;
    a.goff = doff;
    a.items = alt ? v1 : v0;
    a.ntrees = ntrees;
    a.nitems = nitems;
    a.tree_inter = tint;
    cudaMemsetAsync(tint, 0, (size_t)ntrees * sizeof(unsigned long long), s);
    clear_counters(c);
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    cudaEventRecord(e0, s);
    launch(a, OG_OPEN_BH, split, false, refit, true, nitems, s);
    cudaEventRecord(e1, s);
    std::vector<unsigned long long> hti(tree_interactions ? (size_t)ntrees : 0);
    if (tree_interactions)
        cudaMemcpyAsync(hti.data(), tint, (size_t)ntrees * sizeof(unsigned long long), cudaMemcpyDeviceToHost, s);
    cudaFreeAsync(tmp, s);
    unsigned long long h[3] = {0, 0, 0};
    og_status st = finish_pass(c, e0, e1, ms_out, h);
    if (st) return st;
    for (int64_t k = 0; k < ntrees; ++k) trees[k]->have_cost = true;
    if (interactions) *interactions = (int64_t)h[1];
    if (tree_interactions)
        for (int64_t k = 0; k < ntrees; ++k) tree_interactions[k] = (int64_t)hti[(size_t)k];
    return OG_OK;
}

}  // namespace og
