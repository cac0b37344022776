// Equal-sized subclustering (Algorithm 1 steps 2-5, repeated on the points left out as
// §II describes): round r builds the landmark L = per-attribute minimum of the
// remaining points, takes the N remaining points nearest to L as subcluster r and
// removes them.
//
// Membership is defined by the float64 distance
//     delta64_i = sum_{j ascending} (double(x_ij) - double(L_j))^2   (one rounding per op)
// with equal distances taken in ascending point index.
//
// Epochs.  L changes only when every remaining point that holds some attribute's minimum
// has been taken, and while L stays the distances stay: the round after r takes the next N
// points of the same order.  So one pass of distances serves an epoch of up to K rounds
// (K = rounds_per_pass, at most kMaxEpoch): with K boundaries at ranks N, 2N, ..., KN of
// the order by (delta64, index), every point left gets the round of the epoch it falls
// in, and the epoch commits its rounds up to the first one after which some attribute
// has no holder of its landmark value left.  The later rounds' assignments are dropped
// and the next epoch starts from the new landmark (a new pass of distances) or, when all
// K rounds committed, from the same one (no pass at all).  K itself is read off the keys:
// the holders' largest key per attribute bounds the round in which the landmark changes,
// so an epoch resolves only the boundaries up to there (phase B).  On 2^20 points of 16
// attributes in 256 rounds the landmark changes in 50 rounds or so, one epoch each.
//
// Each pass works in float32 and keeps exact arithmetic for thin bands around the
// boundaries:
//   A. delta32_i in float32 (FMA chains, a row's pieces summed across the lanes that read
//      it), kept as its bit pattern (order-preserving for non-negative floats), and a
//      2048-bin histogram of the keys, the bins fitted to the range the keys can lie in
//      (DigitMap).  Points equal to L in an attribute are counted per attribute and flagged
//      (the holders);
//   B. per boundary, the first-digit bin holding its rank, and 2048-bin histograms of
//      the keys inside those bins: each boundary's float32 key lies in a range [A, B] of a
//      few units in the last place;
//   C. |delta32 - delta64| <= eps*delta32 + ea with eps = key_roundings*2^-23, ea = 2^-120, so the
//      boundary's delta64 lies in [A(1-eps)-ea, B(1+eps)+ea]: a point whose bound lies
//      below that interval is certainly before the boundary, one above it certainly
//      after; the few in between form the boundary's band (boundaries whose bands overlap
//      form one group);
//   D. each group is settled by one CTA: compensated float32 distances of its entries
//      (within eps_ff of delta64) order all but the entries within that error of a cut,
//      and those (in practice exact ties) are ranked by float64 and index;
//   E. every CTA finds how many rounds the epoch commits from the grid's counts and takes
//      their points out of its list.
// A phase runs for a few microseconds once an epoch, so its code comes from beyond the
// instruction cache every time: rare work sits in rolled loops or out of line, and loops are
// unrolled only as far as their loads need (390 -> 240 KB in all; a fifth off an epoch).
// The partition is therefore exactly the float64 definition's, whatever float32 does.
//
// Most landmark changes move one or two attributes (the others keep a holder).  The pass
// after such a change reads only the attributes that moved: with J those attributes, o_j
// the old and l_j the new value, the squared distance changes by exactly
//     sum_{j in J} (l_j - o_j)(l_j + o_j - 2 x_j),
// which is added to every live key in float32.  The keys' error bound then takes the form
// |delta32 - delta64| <= eps*delta32 + ea with eps and ea carried from pass to pass: a
// full pass sets (eps0, ea0) = (key_roundings 2^-23, 2^-120), and an update with C = sum_J (l_j - o_j)
// gives eps' = eps + 2^-23 and ea' = ea + (5 eps + (16 + 4|J|) 2^-24) C (the update's own
// rounding, the old key's error carried to the new key, and the float64 definition's;
// scaled values lie in [0, 1]).  Phase C uses the carried bound; a full pass is taken
// instead when J spans many 32-byte sectors of a row, when more than kIncMax attributes
// moved, or when eps would pass 1.5 (d+4) 2^-23 or ea an eighth of (d+4) 2^-23 times the last epoch's
// first boundary key (the landmark sits at the corner of the minima, so the boundary keys
// are large and ea stays a small share of the bands' width).
//
// Points never move: CTA c owns the index slice [c n/G, (c+1) n/G) and keeps the ids of its
// points left in a list with their keys by list position: in shared memory while the slice
// fits (ascending), else in global memory, with gaps until a quarter of it is gone.  Every
// point gets its round in rnd[]; after the launch a stable counting sort by round packs
// the subclusters (ascending index inside each).  The next landmark differs from the last
// one only in the attributes that lost their last holder (the commit knows them), usually
// one to three: the compaction that drops the committed points is followed by a minimum of
// those attributes over the points it kept, the same columns the key update reads next.
// (Sorted bucket lists per attribute, built before the first epoch and walked from their low
// end, took 27-34 ms of atomics at 2^24 x 64, 1 ms at 400000 x 128, and 42 us an epoch of
// dependent loads on clustered 2-D data.)
//
// All epochs run in one persistent cooperative launch, the phases separated by grid
// barriers.  Every barrier wait is bounded; a CTA that gives up sets the abort flag, every
// other CTA then leaves at its next wait, and the host sees PSCL_ETIMEOUT.
#include <algorithm>
#include <cstddef>

#include "pscl_internal.cuh"

namespace pscl {
namespace {

constexpr int kThreads = 256;
constexpr int kW = kThreads / 32;
constexpr uint32_t kInfBits = 0x7f800000u;
constexpr uint32_t kGone = 0xFFFFFFFFu;       // key past the end of a list
constexpr uint32_t kNone = 0xFFFFFFFFu;       // round of a point not assigned (yet)
constexpr int kIncMax = 8;                     // moved attributes a pass may update keys for
constexpr int kKeyCache = 4096;               // keys and ids of a slice kept in shared memory, if it fits
constexpr int kSelBins = 2048;
constexpr int kSelList = 1024;
constexpr int kSelBatch = 8;
constexpr int kScrWords = 8192;
static_assert(kScrWords >= kHistBins, "phase A's histogram fits the scratch");
static_assert(kScrWords >= kSelBins + 3 * kSelList, "a selection's scratch fits");
constexpr int kPeelDynWords = kScrWords + 2 * kKeyCache + kKeyCache / 4;
// Settling a group in shared memory: the histogram of its distances, the bins marked, and the
// entries near a boundary (distance, id, float64 distance, two bytes of state); in place of a
// slice's key cache, where there is none, all entries' distances and ids.
constexpr int kRankBins = 2048;
constexpr int kNear = 1024;
constexpr int kStage = (2 * kKeyCache + kKeyCache / 4) / 3;
// Close entries ranked one by one, at most; more (tied data) are sorted.  Each of them against every
// near one takes their product: 10^6 x 1 with 1000 points a value 73.5 ms of peel, sorted 8.3.
constexpr int kRankOne = 128;
static_assert(kRankBins + kRankBins / 32 + 5 * kNear + kNear / 2 <= kScrWords, "settling fits the scratch");
constexpr int kQT = 4;                        // tiles of kThreads items per compaction scan
constexpr int kCB = 8;                        // keys per thread in flight when classifying
// list positions a thread has in flight in the passes that read attributes by id: a slice in
// shared memory has 16 a thread at most, and wants little code; one in global memory is bound by
// the loads in flight (2^24 x 64: landmark 63 -> 41 us, key update 77 -> 68 us an epoch)
constexpr int kLoadKc = 4, kLoadGlobal = 8;
constexpr int kHoldBatch = 8;                 // state bytes per thread in flight when finding holders
// State byte of each list position: bit 7 set once the point has held some attribute's
// landmark value (it then holds it while it is left); bits 0..6 its place in the current
// epoch: a round 0..kMaxEpoch-1 it is certainly in, kFlBand (in a band), kFlNone.
constexpr uint8_t kFlHold = 0x80;
constexpr uint8_t kFlBand = 0x7E;
constexpr uint8_t kFlNone = 0x7F;
constexpr uint32_t kPosMask = 0x7FFFFFFFu;    // a band entry's id; bit 31 carries its hold flag
constexpr int kDefaultRounds = 32;            // rounds per distance pass by default
constexpr uint32_t kAllResolve = 6;           // boundaries up to which every CTA resolves them itself
constexpr unsigned kDefaultSpin = 1u << 25;   // ~1-2 s of polling per barrier at most

// ------------------------------------------------------------------ block helpers
__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    return v;
}

// Exclusive scan over the block (blockDim.x == kThreads); `total` gets the block sum.
__device__ uint32_t block_excl_scan(uint32_t v, uint32_t &total)
{
    __shared__ uint32_t wsum[kW];
    __shared__ uint32_t wtot;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t inc = warp_incl_scan(v);
    if (lane == 31) wsum[w] = inc;
    __syncthreads();
    if (w == 0) {
        uint32_t s = lane < kW ? wsum[lane] : 0;
        uint32_t si = warp_incl_scan(s);
        if (lane < kW) wsum[lane] = si - s;
        if (lane == kW - 1) wtot = si;
    }
    __syncthreads();
    uint32_t r = wsum[w] + inc - v;
    total = wtot;
    __syncthreads();
    return r;
}

__device__ uint32_t block_sum(uint32_t v)
{
    uint32_t tot;
    block_excl_scan(v, tot);
    return tot;
}

__device__ __forceinline__ uint32_t warp_min(uint32_t v)
{
#pragma unroll
    for (int o = 16; o; o >>= 1) v = min(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

__device__ uint32_t block_min(uint32_t v)
{
    __shared__ uint32_t wm[kW];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    v = warp_min(v);
    if (lane == 0) wm[w] = v;
    __syncthreads();
    v = wm[0];
#pragma unroll
    for (int q = 1; q < kW; q++) v = min(v, wm[q]);
    __syncthreads();
    return v;
}

// ------------------------------------------------------------------ grid barriers
// Thread 0's bounded wait for the arrival counter to reach `target`.  Returns false if the
// launch is being aborted (or this wait gave up, which aborts it).
__device__ bool bar_wait(PeelCtl *ctl, uint32_t *flags, unsigned target, unsigned limit)
{
    unsigned spins = 0, v;
    for (;;) {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&ctl->bar_count) : "memory");
        if ((int)(v - target) >= 0) return true;
        if ((++spins & 63) == 0) {
            if (*(volatile unsigned *)&ctl->abort) return false;
            if (spins > limit) {
                atomicExch(&ctl->abort, 1u);
                atomicOr(&flags[1], 2u);               // timed out
                return false;
            }
            __nanosleep(32);
        }
    }
}

// Grid-wide barrier with a bounded wait: a monotonic arrival counter (release on arrival,
// acquire while polling), so no reset is needed within a launch.  `extra` arrivals more
// than the grid gives are awaited (a test of the give-up path; 0 otherwise).
__device__ __noinline__ bool grid_wait(PeelCtl *ctl, uint32_t *flags, unsigned target, unsigned limit, unsigned extra)
{
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        if (blockIdx.x == 0) ctl->barriers += 1;     // statistics (one writer)
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&ctl->bar_count) : "memory");
        ok = bar_wait(ctl, flags, target + extra, limit) ? 1 : 0;
    }
    __syncthreads();
    return ok != 0;
}

__device__ __forceinline__ bool grid_sync(PeelCtl *ctl, uint32_t *flags, unsigned &target, unsigned limit,
                                          unsigned extra = 0)
{
    target += gridDim.x;
    return grid_wait(ctl, flags, target, limit, extra);
}

// A grid barrier whose last arriving CTA runs work() (all its threads) before any CTA
// leaves: every CTA adds one arrival, the last one then runs the work and adds one more.
template <class Work>
__device__ bool grid_sync_last(PeelCtl *ctl, uint32_t *flags, unsigned &target, unsigned limit, Work work)
{
    __shared__ int ok, last;
    target += gridDim.x + 1;
    __syncthreads();
    if (threadIdx.x == 0) {
        if (blockIdx.x == 0) ctl->barriers += 1;     // statistics (one writer)
        unsigned old;
        asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(old) : "l"(&ctl->bar_count) : "memory");
        last = old == target - 2u;
    }
    __syncthreads();
    if (last) {
        work();
        __syncthreads();
        if (threadIdx.x == 0) {
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&ctl->bar_count) : "memory");
            ok = *(volatile unsigned *)&ctl->abort ? 0 : 1;
        }
    } else if (threadIdx.x == 0) {
        ok = bar_wait(ctl, flags, target, limit) ? 1 : 0;
    }
    __syncthreads();
    return ok != 0;
}

// ------------------------------------------------------------------ distances
// float32 distance of one row by one thread (the phase-A path for d not a multiple of 4,
// or below 8): t = RN(x - L), acc = RN(t*t + acc) (fused), ascending attributes.  `hz` is
// set when some attribute equals the landmark's.
template <int D>
__device__ __forceinline__ float dist32(const float *__restrict__ row, const float *Ls, int d, bool &hz)
{
    float acc = 0.0f;
    bool z = false;
    if (D > 0 && (D % 4) == 0) {
        const float4 *r4 = reinterpret_cast<const float4 *>(row);
#pragma unroll
        for (int q = 0; q < D / 4; q++) {
            float4 v = __ldg(&r4[q]);
            float t0 = __fsub_rn(v.x, Ls[4 * q + 0]);
            acc = __fmaf_rn(t0, t0, acc);
            float t1 = __fsub_rn(v.y, Ls[4 * q + 1]);
            acc = __fmaf_rn(t1, t1, acc);
            float t2 = __fsub_rn(v.z, Ls[4 * q + 2]);
            acc = __fmaf_rn(t2, t2, acc);
            float t3 = __fsub_rn(v.w, Ls[4 * q + 3]);
            acc = __fmaf_rn(t3, t3, acc);
            z |= (t0 == 0.0f) | (t1 == 0.0f) | (t2 == 0.0f) | (t3 == 0.0f);
        }
    } else {
        const int dd = D > 0 ? D : d;
#pragma unroll 4
        for (int j = 0; j < dd; j++) {
            float t = __fsub_rn(__ldg(&row[j]), Ls[j]);
            acc = __fmaf_rn(t, t, acc);
            z |= t == 0.0f;
        }
    }
    hz = z;
    return acc;
}

// float64 distance exactly as defined: diff, square, add, each rounded, no fusion.
__device__ __noinline__ double dist64(const float *__restrict__ row, const float *Ls, int d)
{
    double s = 0.0;
#pragma unroll 4
    for (int j = 0; j < d; j++) {
        double diff = __dsub_rn((double)__ldg(&row[j]), (double)Ls[j]);
        s = __dadd_rn(s, __dmul_rn(diff, diff));
    }
    return s;
}

// Compensated float32 distance (h + l, |l| <= ulp(h)/2): each difference is split exactly
// into s + e (TwoSum), s^2 is kept exactly as p + pe (FMA), 2*s*e is folded into the low
// part (e^2 <= 2^-48 s^2 is dropped) and the high parts are summed error-free (TwoSum).
// Its distance to the float64 definition is below eps_ff(d) * (h + l).
__device__ __forceinline__ void dist_ff(const float *__restrict__ row, const float *Ls, int d, float &h, float &l)
{
    float hi = 0.0f, lo = 0.0f;
#pragma unroll 4
    for (int j = 0; j < d; j++) {
        const float a = __ldg(&row[j]), b = Ls[j];
        const float s = __fsub_rn(a, b);
        const float bb = __fsub_rn(s, a);                       // TwoSum(a, -b)
        const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(-b, bb));
        const float p = __fmul_rn(s, s);
        const float pe = __fmaf_rn(s, s, -p);
        const float q = __fmaf_rn(__fmul_rn(2.0f, s), e, pe);
        const float t = __fadd_rn(hi, p);                       // TwoSum(hi, p)
        const float bv = __fsub_rn(t, hi);
        const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(t, bv)), __fsub_rn(p, bv));
        hi = t;
        lo = __fadd_rn(lo, __fadd_rn(err, q));
    }
    h = __fadd_rn(hi, lo);                                      // normalise (Fast2Sum)
    l = __fsub_rn(lo, __fsub_rn(h, hi));
}

// Bound on |dff - delta64| / delta64: (d^2 + 8d) u^2 for the compensated sum
// (u = 2^-24) plus (d + 2) 2^-53 for the float64 one, with a factor two of margin.
__device__ __forceinline__ float eps_ff(int d)
{
    return (float)((double)d * d + 8.0 * d + 1.0) * 0x1p-47f;
}

// The same by 8 lanes of a warp (sub = lane & 7, every lane of the warp taking part): lane sub
// sums the attributes sub, sub + 8, ..., then the partial sums are added pairwise, the high
// parts error-free.  Fewer roundings per term than the one chain the bound allows.
__device__ __forceinline__ void dist_ff8(const float *__restrict__ row, const float *Ls, int d, int sub, float &h,
                                         float &l)
{
    float hi = 0.0f, lo = 0.0f;
#pragma unroll 4
    for (int j = sub; j < d; j += 8) {
        const float a = __ldg(&row[j]), b = Ls[j];
        const float s = __fsub_rn(a, b);
        const float bb = __fsub_rn(s, a);
        const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(-b, bb));
        const float p = __fmul_rn(s, s);
        const float q = __fmaf_rn(__fmul_rn(2.0f, s), e, __fmaf_rn(s, s, -p));
        const float t = __fadd_rn(hi, p);
        const float bv = __fsub_rn(t, hi);
        const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(t, bv)), __fsub_rn(p, bv));
        hi = t;
        lo = __fadd_rn(lo, __fadd_rn(err, q));
    }
#pragma unroll
    for (int o = 4; o; o >>= 1) {
        const float p = __shfl_xor_sync(0xffffffffu, hi, o), pl = __shfl_xor_sync(0xffffffffu, lo, o);
        const float t = __fadd_rn(hi, p);
        const float bv = __fsub_rn(t, hi);
        const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(t, bv)), __fsub_rn(p, bv));
        hi = t;
        lo = __fadd_rn(__fadd_rn(lo, pl), err);
    }
    h = __fadd_rn(hi, lo);
    l = __fsub_rn(lo, __fsub_rn(h, hi));
}

__device__ __forceinline__ uint64_t ff_key(float h, float l)
{
    double v = __dadd_rn((double)h, (double)l);
    if (!(v > 0.0)) v = 0.0;
    return (uint64_t)__double_as_longlong(v);
}

// The compensated distance h + l rounded once to float64 (its bit pattern orders like
// the value), the key a group's entries are ranked by.
__device__ __forceinline__ uint64_t dff_key(const float *__restrict__ row, const float *Ls, int d)
{
    float h, l;
    dist_ff(row, Ls, d, h, l);
    return ff_key(h, l);
}

// The digits of the keys in one pass.  Every key left lies in [base, top] (the range's
// derivation: see its assignment in the kernel; a key below base only widens a band), cut
// into bins of 2^sh values (bin 0: the keys below base) and a bin into sub-bins of 2^ss (2^s0
// for bin 0).  With the range spread over the whole first digit (before, its bits were the
// key's top 11: two bits of mantissa, a few bins holding most points), the second digit
// reaches down to single keys or nearly, so the bands shrink to the float32 error, and few
// points share a boundary's bin: phase B counts 2000 keys instead of half of them.
struct DigitMap {
    uint32_t base;
    int sh, ss, s0;
    __device__ __forceinline__ uint32_t bin(uint32_t k) const
    {
        return k < base ? 0u : min((uint32_t)kHistBins - 1u, 1u + ((k - base) >> sh));
    }
    __device__ __forceinline__ uint32_t low(uint32_t b) const { return b ? base + ((b - 1u) << sh) : 0u; }
    __device__ __forceinline__ uint32_t sub(uint32_t k, uint32_t b) const
    {
        return min((uint32_t)kHistBins - 1u, (k - low(b)) >> (b ? ss : s0));
    }
    // the keys of a sub-bin: [A, B]
    __device__ __forceinline__ void range(uint32_t b, uint32_t sb, uint32_t &A, uint32_t &B) const
    {
        const int s = b ? ss : s0;
        A = low(b) + (sb << s);
        B = A + ((1u << s) - 1u);
        if (sb == (uint32_t)kHistBins - 1u) B = b == (uint32_t)kHistBins - 1u ? kInfBits - 1u : max(B, low(b + 1u) - 1u);
    }
};

__device__ __forceinline__ DigitMap digit_map(uint32_t base, uint32_t top)
{
    DigitMap m;
    m.base = base;
    const uint32_t span = top > base ? top - base : 0u;
    m.sh = max(0, 21 - __clz(span | 1u));                // span >> sh <= 2047 - 1
    if ((span >> m.sh) > (uint32_t)kHistBins - 3u) m.sh++;
    m.ss = max(0, m.sh - 11);
    m.s0 = max(0, 21 - __clz(base | 1u));
    return m;
}

// Cut-offs of phase C from the range [kA, kB] of a boundary's float32 key.
// With |delta32 - delta64| <= eps delta32 + ea (eps <= 1/3) the boundary's delta64 lies in
// [A(1-eps) - ea, B(1+eps) + ea]; a point is certainly before it if delta32 (1+eps) + ea
// is below that interval, which holds for delta32 < A(1-2eps) - 2ea, and certainly after
// it if delta32 (1-eps) - ea is above it, which holds for delta32 > B(1+3eps) + 3ea.  Both
// cut-offs are evaluated in float32 rounded towards the safe side.
__device__ void band_cutoffs(uint32_t kA, uint32_t kB, float eps, float ea, uint32_t &in_key, uint32_t &out_key)
{
    const float A = __uint_as_float(kA), B = __uint_as_float(kB);
    const float in_thr = __fsub_rd(__fmul_rd(A, __fsub_rd(1.0f, 2.0f * eps)), 2.0f * ea);
    const float out_thr = __fadd_ru(__fmul_ru(B, __fadd_ru(1.0f, __fmul_ru(3.0f, eps))), __fmul_ru(3.0f, ea));
    in_key = in_thr > 0.0f ? __float_as_uint(in_thr) : 0u;
    out_key = __float_as_uint(out_thr);
}

// ------------------------------------------------------------------ exact selection
// The `need`-th smallest (1-based) of nb entries by (key, position), key_at / pos_at giving
// entry i.  Single-block radix select with 8-bit digits over the 96-bit composite.
template <class KeyAt, class PosAt>
__device__ void select_radix(KeyAt key_at, PosAt pos_at, uint32_t nb, uint32_t need, uint64_t &K, uint32_t &Pp)
{
    __shared__ uint32_t h[256];
    __shared__ uint64_t pk;
    __shared__ uint32_t pp, rank;
    if (threadIdx.x == 0) {
        pk = 0;
        pp = 0;
        rank = need - 1;
    }
    __syncthreads();
    for (int pass = 0; pass < 12; pass++) {
        h[threadIdx.x] = 0;
        __syncthreads();
        const uint64_t cpk = pk;
        const uint32_t cpp = pp;
        for (uint32_t i = threadIdx.x; i < nb; i += kThreads) {
            const uint64_t k = key_at(i);
            const uint32_t p = pos_at(i);
            bool match;
            uint32_t digit;
            if (pass < 8) {
                match = pass == 0 || (k >> (64 - 8 * pass)) == (cpk >> (64 - 8 * pass));
                digit = (uint32_t)(k >> (56 - 8 * pass)) & 0xFFu;
            } else {
                const int q = pass - 8;
                match = k == cpk && (q == 0 || (p >> (32 - 8 * q)) == (cpp >> (32 - 8 * q)));
                digit = (p >> (24 - 8 * q)) & 0xFFu;
            }
            if (match) atomicAdd(&h[digit], 1u);
        }
        __syncthreads();
        const uint32_t v = h[threadIdx.x];
        uint32_t tot;
        const uint32_t before = block_excl_scan(v, tot);
        const uint32_t r = rank;
        __syncthreads();
        if (r >= before && r < before + v) {
            if (pass < 8) pk = cpk | ((uint64_t)threadIdx.x << (56 - 8 * pass));
            else pp = cpp | ((uint32_t)threadIdx.x << (24 - 8 * (pass - 8)));
            rank = r - before;
        }
        __syncthreads();
    }
    K = pk;
    Pp = pp;
    __syncthreads();
}

// The same selection in three passes when the keys spread: the smallest and largest key
// give the bits all keys share; an 11-bit histogram of the next bits finds the digit of
// the need-th entry; that digit's entries (at most kSelList) are gathered in shared memory
// and ranked there by (key, position).  Returns false, with nothing decided, when all keys
// are equal or the digit holds more entries: the caller then runs select_radix.
// scratch: kSelBins + 3 kSelList words of shared memory.
template <class KeyAt, class PosAt>
__device__ bool select_fast(KeyAt key_at, PosAt pos_at, uint32_t nb, uint32_t need, uint32_t *scratch, uint64_t &K,
                            uint32_t &Pp)
{
    __shared__ unsigned long long s_mn[kW], s_mx[kW];
    __shared__ uint32_t s_bin, s_rank, s_cnt, s_hit;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    uint32_t *h = scratch;
    uint64_t *lk = reinterpret_cast<uint64_t *>(scratch + kSelBins);      // 8-byte aligned: kSelBins is even
    uint32_t *lp = scratch + kSelBins + 2 * kSelList;
    unsigned long long mn = ~0ull, mx = 0ull;
    for (uint32_t i0 = t; i0 < nb; i0 += kSelBatch * kThreads) {
        unsigned long long kk[kSelBatch];
#pragma unroll
        for (int u = 0; u < kSelBatch; u++) {
            const uint32_t i = i0 + u * kThreads;
            kk[u] = i < nb ? key_at(i) : 0ull;
        }
#pragma unroll
        for (int u = 0; u < kSelBatch; u++) {
            if (i0 + u * kThreads < nb) {
                mn = min(mn, kk[u]);
                mx = max(mx, kk[u]);
            }
        }
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        mn = min(mn, __shfl_xor_sync(0xffffffffu, mn, o));
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    if (lane == 0) {
        s_mn[w] = mn;
        s_mx[w] = mx;
    }
    for (int b = t; b < kSelBins; b += kThreads) h[b] = 0;
    __syncthreads();
    mn = s_mn[0];
    mx = s_mx[0];
#pragma unroll
    for (int q = 1; q < kW; q++) {
        mn = min(mn, (unsigned long long)s_mn[q]);
        mx = max(mx, (unsigned long long)s_mx[q]);
    }
    __syncthreads();
    if (mn == mx) return false;                          // uniform across the block
    const int hb = 63 - __clzll((long long)(mn ^ mx));   // highest bit where keys differ
    const int sh = hb >= 10 ? hb - 10 : 0;               // digit = bits [sh, hb]
    for (uint32_t i0 = t; i0 < nb; i0 += kSelBatch * kThreads) {
        unsigned long long kk[kSelBatch];
#pragma unroll
        for (int u = 0; u < kSelBatch; u++) {
            const uint32_t i = i0 + u * kThreads;
            kk[u] = i < nb ? key_at(i) : 0ull;
        }
#pragma unroll
        for (int u = 0; u < kSelBatch; u++)
            if (i0 + u * kThreads < nb) atomicAdd(&h[(uint32_t)(kk[u] >> sh) & (kSelBins - 1)], 1u);
    }
    __syncthreads();
    {
        constexpr int per = kSelBins / kThreads;
        uint32_t loc = 0;
#pragma unroll
        for (int q = 0; q < per; q++) loc += h[t * per + q];
        uint32_t tot;
        const uint32_t before = block_excl_scan(loc, tot);
        const uint32_t target = need - 1;
        if (target >= before && target < before + loc) {
            uint32_t cc = before;
            for (int q = 0; q < per; q++) {
                const uint32_t v = h[t * per + q];
                if (target >= cc && target < cc + v) {
                    s_bin = (uint32_t)(t * per + q);
                    s_rank = target - cc;
                    s_cnt = v;
                }
                cc += v;
            }
        }
        if (t == 0) s_hit = 0;
    }
    __syncthreads();
    const uint32_t bin = s_bin, rank = s_rank, cnt = s_cnt;
    if (cnt > (uint32_t)kSelList) return false;          // uniform across the block
    for (uint32_t i0 = t; i0 < nb; i0 += kSelBatch * kThreads) {
        unsigned long long kk[kSelBatch];
#pragma unroll
        for (int u = 0; u < kSelBatch; u++) {
            const uint32_t i = i0 + u * kThreads;
            kk[u] = i < nb ? key_at(i) : 0ull;
        }
#pragma unroll
        for (int u = 0; u < kSelBatch; u++) {
            const uint32_t i = i0 + u * kThreads;
            if (i < nb && ((uint32_t)(kk[u] >> sh) & (kSelBins - 1)) == bin) {
                const uint32_t slot = atomicAdd(&s_hit, 1u);
                lk[slot] = kk[u];
                lp[slot] = pos_at(i);
            }
        }
    }
    __syncthreads();
    for (uint32_t q = t; q < cnt; q += kThreads) {
        const uint64_t kq = lk[q];
        const uint32_t pq = lp[q];
        uint32_t rk = 0;
        for (uint32_t o = 0; o < cnt; o++) rk += (lk[o] < kq) || (lk[o] == kq && lp[o] < pq);
        if (rk == rank) {
            s_mn[0] = kq;
            s_hit = pq;
        }
    }
    __syncthreads();
    K = s_mn[0];
    Pp = s_hit;
    __syncthreads();
    return true;
}

// Of entries in global memory: keys gk, ids gp (bit 31 is no part of an id).
__device__ __noinline__ void select_kth(const uint64_t *gk, const uint32_t *gp, uint32_t nb, uint32_t need,
                                        uint32_t *scratch, uint64_t &K, uint32_t &Pp)
{
    auto key_at = [&](uint32_t i) -> uint64_t { return __ldcg(&gk[i]); };
    auto pos_at = [&](uint32_t i) -> uint32_t { return __ldcg(&gp[i]) & kPosMask; };
    if (!select_fast(key_at, pos_at, nb, need, scratch, K, Pp)) select_radix(key_at, pos_at, nb, need, K, Pp);
}

// ------------------------------------------------------------------ the kernel
struct PeelArgs {
    const float *x;
    const float *xt;             // d x n: the points by attribute (or NULL: the updates read x)
    int d;
    int64_t n, N, S;
    uint32_t *rnd;
    uint8_t *pflag;              // 2 x n: the state byte of each list position
    uint32_t *lidx;              // 2 x n: per CTA slice, the ids of its points left (not kc; two lists)
    uint32_t *kpos;              // 2 x n: their keys by list position
    uint32_t *band_k32;
    uint32_t *band_pos;
    uint64_t *gkey;
    uint32_t *gpos;
    uint64_t *akey;
    uint32_t *apos;
    float *landmarks;            // S x d or NULL
    PeelCtl *ctl;
    uint32_t *flags;             // job flags: [1] |= 1 bound violated, 2 barrier timed out
    uint32_t kmax;               // rounds per distance pass
    uint32_t spin;               // polls of a barrier wait before it gives up
    uint32_t stall;              // test hook: the first barrier awaits one arrival too many
    int transpose;               // the launch writes xt itself (xt_out)
    float *xt_out;
};

// rows a thread keeps in flight at once (64 floats of rows at most)
template <int D>
__host__ __device__ constexpr int kPeelBatch()
{
    return D <= 0 ? 1 : (D >= 64 ? 1 : (64 / D > 4 ? 4 : 64 / D));
}

// Phase A reads a row with P = min(D/4, 32) lanes, one float4 each (F per lane when D > 128),
// so that one warp load covers 32/P whole rows instead of one 16-byte piece of 32 rows.
// Each lane sums its part of P rows (fused, ascending attributes) and a butterfly over the
// P lanes leaves every lane the whole sum of one row.  Every squared difference passes
// through at most D/P + log2 P roundings, fewer than the d of the recursive sum that the
// phase-C error bound allows.
template <int D>
__host__ __device__ constexpr bool kCoopRows()
{
    return D >= 8 && D % 4 == 0;
}

template <int D>
__host__ __device__ constexpr int kCoopLanes()
{
    return D / 4 < 32 ? D / 4 : 32;
}

// 32-row warp chunks a thread keeps in flight: about 16 float4 loads per lane
template <int D>
__host__ __device__ constexpr int kCoopBatch()
{
    return 16 / (D / 4) >= 4 ? 4 : (16 / (D / 4) >= 1 ? 16 / (D / 4) : 1);
}

// The key's error bound in units of 2^-23: the roundings a term passes through (its own
// difference's twice, the chain's, the butterfly's), with a factor two of margin.
template <int D>
__host__ __device__ constexpr int key_roundings(int d)
{
    if (!kCoopRows<D>()) return d + 4;
    int lg = 0;
    for (int p = kCoopLanes<D>(); p > 1; p >>= 1) lg++;
    return D / kCoopLanes<D>() + lg + 4;
}

__device__ __forceinline__ bool in_mask(const uint32_t *jm, int j)
{
    return (jm[j >> 5] >> (j & 31)) & 1u;
}

// A live point equal to the landmark in some attribute: counted per such attribute whose
// landmark value is new (jm; the counts of the others carry over) and flagged for the
// epochs' holder bookkeeping.
__device__ __forceinline__ void note_holder(const float *__restrict__ row, const float *Ls, int d, uint8_t *fl,
                                            uint32_t *chold, const uint32_t *jm)
{
    for (int j = 0; j < d; j++)
        if (__ldg(&row[j]) == Ls[j] && in_mask(jm, j)) atomicAdd(&chold[j], 1u);
    *fl |= kFlHold;
}

// Phase A: every live point's float32 key, stored by list position (shared memory when
// kc, else kpos: the slice's keys) and counted in the first-digit histogram sh (but in the
// first epoch); holders
// counted per attribute of jm and flagged in their position's state byte (pfl: the
// slice's, by list position).  Out of line, so that the register allocation of the
// kernel's other phases does not carry its loads in flight.
template <int D>
__device__ __noinline__ void phase_keys(const float *__restrict__ x, const float *Ls, int d, uint32_t n_live,
                                        uint32_t s0, bool first, bool kc, const uint32_t *sid, const uint32_t *glin,
                                        uint32_t *skey, uint32_t *kpos, uint32_t *sh, const DigitMap *dm,
                                        uint8_t *pfl, uint32_t *chold, const uint32_t *jm)
{
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const DigitMap mp = *dm;
    auto LID = [&](uint32_t q) -> uint32_t { return kc ? sid[q] : __ldcg(&glin[q]); };
    auto key_out = [&](bool live, uint32_t pos, uint32_t k) {
        if (live) {
            if (kc) skey[pos] = k;
            else kpos[pos] = k;
            if (!first) atomicAdd(&sh[mp.bin(k)], 1u);       // the first epoch fits the bins to its keys
        }
    };
    if constexpr (kCoopRows<D>()) {
        constexpr int P = kCoopLanes<D>();                 // lanes per row
        constexpr int F = D / (4 * P);                     // float4 per lane and row
        constexpr int RW = 32 / P;                         // rows per warp load
        constexpr int BC = kCoopBatch<D>();
        static_assert((P & (P - 1)) == 0 && P >= 2, "lanes per row: a power of two");
        const int g = lane / P, sl = lane % P;
        float4 Lq[F];
#pragma unroll
        for (int f = 0; f < F; f++) {
            const int j = 4 * (sl + P * f);
            Lq[f] = make_float4(Ls[j], Ls[j + 1], Ls[j + 2], Ls[j + 3]);
        }
#pragma unroll 1
        for (uint32_t base = 0; base < n_live; base += BC * kThreads) {
            // chunk q of this warp: list positions cb + [0, 32); lane i fetches the id of
            // position cb + i, and row u of its group is position cb + u*RW + g.  Past the
            // end and at gaps the id is the slice's first row (read again, an L1 hit).
            uint32_t myid[BC], live[BC];
#pragma unroll
            for (int q = 0; q < BC; q++) {
                const uint32_t pos = base + q * kThreads + w * 32 + lane;
                myid[q] = pos < n_live ? LID(pos) : kGone;
                live[q] = __ballot_sync(0xffffffffu, myid[q] != kGone);
                if (myid[q] == kGone) myid[q] = s0;
            }
            static_assert(BC * P <= 32, "a mask bit per row");
            uint32_t hzs = 0;                              // rows with a landmark value
            float4 v[BC][P][F];
#pragma unroll
            for (int q = 0; q < BC; q++)
#pragma unroll
                for (int u = 0; u < P; u++) {
                    const uint32_t id = __shfl_sync(0xffffffffu, myid[q], u * RW + g);
                    const float4 *r4 = reinterpret_cast<const float4 *>(x + (size_t)id * D) + sl;
#pragma unroll
                    for (int f = 0; f < F; f++) v[q][u][f] = __ldg(r4 + P * f);
                }
#pragma unroll
            for (int q = 0; q < BC; q++) {
                float ps[P];
                uint32_t hz = 0;
#pragma unroll
                for (int u = 0; u < P; u++) {
                    float acc = 0.0f;
                    bool z = false;
#pragma unroll
                    for (int f = 0; f < F; f++) {
                        const float t0 = __fsub_rn(v[q][u][f].x, Lq[f].x);
                        acc = __fmaf_rn(t0, t0, acc);
                        const float t1 = __fsub_rn(v[q][u][f].y, Lq[f].y);
                        acc = __fmaf_rn(t1, t1, acc);
                        const float t2 = __fsub_rn(v[q][u][f].z, Lq[f].z);
                        acc = __fmaf_rn(t2, t2, acc);
                        const float t3 = __fsub_rn(v[q][u][f].w, Lq[f].w);
                        acc = __fmaf_rn(t3, t3, acc);
                        z |= (t0 == 0.0f) | (t1 == 0.0f) | (t2 == 0.0f) | (t3 == 0.0f);
                    }
                    ps[u] = acc;
                    hz |= (uint32_t)z << u;
                }
                // butterfly: after the round with mask m a lane keeps the half of rows
                // whose index has its lane bit m; at the end ps[0] is row sl's sum
                constexpr int LP = P >= 32 ? 5 : P >= 16 ? 4 : P >= 8 ? 3 : P >= 4 ? 2 : 1;
#pragma unroll
                for (int lv = 1; lv <= LP; lv++) {
                    const int m = P >> lv;
                    const bool up = (sl & m) != 0;
#pragma unroll
                    for (int i = 0; i < m; i++) {
                        const float keep = up ? ps[i + m] : ps[i];
                        const float send = up ? ps[i] : ps[i + m];
                        ps[i] = __fadd_rn(keep, __shfl_xor_sync(0xffffffffu, send, m));
                    }
                }
                hzs |= hz << (q * P);
                const uint32_t src = (uint32_t)(sl * RW + g);
                key_out((live[q] >> src) & 1u, base + q * kThreads + w * 32 + src, __float_as_uint(ps[0]));
            }
            // rare: rows holding a landmark value in this lane's attributes
#pragma unroll 1
            while (hzs) {
                const int b = __ffs(hzs) - 1;
                hzs &= hzs - 1u;
                const uint32_t rpos = base + (uint32_t)(b / P) * kThreads + w * 32 + (uint32_t)(b % P) * RW + g;
                const uint32_t id = rpos < n_live ? LID(rpos) : kGone;
                if (id == kGone) continue;
                const float4 *r4 = reinterpret_cast<const float4 *>(x + (size_t)id * D) + sl;
#pragma unroll 1
                for (int f = 0; f < F; f++) {
                    const float4 vv = __ldg(r4 + P * f);
                    const int j = 4 * (sl + P * f);
                    if (vv.x == Ls[j + 0] && in_mask(jm, j + 0)) atomicAdd(&chold[j + 0], 1u);
                    if (vv.y == Ls[j + 1] && in_mask(jm, j + 1)) atomicAdd(&chold[j + 1], 1u);
                    if (vv.z == Ls[j + 2] && in_mask(jm, j + 2)) atomicAdd(&chold[j + 2], 1u);
                    if (vv.w == Ls[j + 3] && in_mask(jm, j + 3)) atomicAdd(&chold[j + 3], 1u);
                }
                pfl[rpos] |= kFlHold;
            }
        }
    } else {
        constexpr int B = kPeelBatch<D>();
#pragma unroll 1
        for (uint32_t base = 0; base < n_live; base += B * kThreads) {
            bool lv[B];
            uint32_t ids[B];
#pragma unroll
            for (int q = 0; q < B; q++) {
                const uint32_t qi = base + q * kThreads + t;
                ids[q] = qi < n_live ? LID(qi) : kGone;
                lv[q] = ids[q] != kGone;
                if (!lv[q]) ids[q] = s0;
            }
            // past the end and at gaps a thread reads the slice's first row (an L1 hit), so every
            // thread keeps B rows in flight without branching
            float dl[B];
            bool hz[B];
#pragma unroll
            for (int q = 0; q < B; q++) dl[q] = dist32<D>(x + (size_t)ids[q] * d, Ls, d, hz[q]);
            uint32_t hzs = 0;
#pragma unroll
            for (int q = 0; q < B; q++) {
                hzs |= (uint32_t)(lv[q] && hz[q]) << q;
                key_out(lv[q], base + q * kThreads + t, __float_as_uint(dl[q]));
            }
#pragma unroll 1
            while (hzs) {
                const uint32_t pos = base + (uint32_t)(__ffs(hzs) - 1) * kThreads + t;
                hzs &= hzs - 1u;
                note_holder(x + (size_t)LID(pos) * d, Ls, d, &pfl[pos], chold, jm);
            }
        }
    }
}

// Phase A after a landmark change in the nj attributes jj (ascending; old values jo, new
// values jl): every live key moves by the change of its squared distance,
// sum_i (jl_i - jo_i)(jl_i + jo_i - 2 x_{jj_i}) (FMA chain in float32), read from those
// attributes only; the result is clamped at 0, stored in place and counted in sh, and the
// holders of the new values are counted and flagged as in phase_keys.
// U: list positions per thread in flight (kLoadKc, kLoadGlobal).
template <int D, int U>
__device__ __noinline__ void phase_inc(const float *__restrict__ x, const float *__restrict__ xt, uint32_t n, int d,
                                       uint32_t n_live, bool kc, const uint32_t *sid, const uint32_t *glin,
                                       uint32_t *skey, uint32_t *kpos, uint32_t *sh, const DigitMap *dm,
                                       uint8_t *pfl, uint32_t *chold, uint32_t nj, const int *jj, const float *jo,
                                       const float *jl)
{
    const int t = threadIdx.x;
    const DigitMap mp = *dm;
    // attribute j of point i at src[i * ps + j * as]: the by-attribute copy (a CTA's ids
    // ascend, so a warp's loads fall close together) or the rows; read through L2, since this
    // launch may have written the copy
    const float *src = xt ? xt : x;
    const size_t ps = xt ? 1 : (size_t)(D > 0 ? D : d), as = xt ? (size_t)n : 1;
#pragma unroll 1
    for (uint32_t q0 = 0; q0 < n_live; q0 += U * kThreads) {          // block-uniform bound
        uint32_t id[U], key[U], hold = 0;
        float acc[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const uint32_t qi = q0 + u * kThreads + t;
            const bool v = qi < n_live;
            id[u] = v ? (kc ? sid[qi] : __ldcg(&glin[qi])) : kGone;
            key[u] = v ? (kc ? skey[qi] : __ldcg(&kpos[qi])) : 0u;
            acc[u] = 0.0f;
        }
        for (uint32_t i = 0; i < nj; i++) {
            const int j = jj[i];
            const float ln = jl[i], c = __fsub_rn(ln, jo[i]), sm = __fadd_rn(ln, jo[i]);
            float v[U];
#pragma unroll
            for (int u = 0; u < U; u++) v[u] = id[u] != kGone ? __ldcg(&src[(size_t)id[u] * ps + (size_t)j * as]) : ln;
#pragma unroll
            for (int u = 0; u < U; u++) {
                acc[u] = __fmaf_rn(c, __fmaf_rn(-2.0f, v[u], sm), acc[u]);
                if (v[u] == ln && id[u] != kGone) {
                    atomicAdd(&chold[j], 1u);
                    hold |= 1u << u;
                }
            }
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            const uint32_t qi = q0 + u * kThreads + t;
            const bool live = id[u] != kGone;
            const float kv = __fadd_rn(__uint_as_float(key[u]), acc[u]);
            const uint32_t k = kv > 0.0f ? __float_as_uint(kv) : 0u;
            if (live) {
                if (kc) skey[qi] = k;
                else kpos[qi] = k;
                if ((hold >> u) & 1u) pfl[qi] |= kFlHold;
                atomicAdd(&sh[mp.bin(k)], 1u);
            }
        }
    }
}

// The holders among a warp's 32 points (the lanes of m; ids by lane), one at a time by
// the whole warp: f(j, v) for every attribute j in which the point equals the landmark, v its
// lane's val.  A row is read in one coalesced load per 32 attributes, where a thread walking
// it alone held its warp for d loads (400000 x 128: 15 us of an epoch's key pass).
template <class F>
__device__ __forceinline__ void for_held(const float *__restrict__ x, const float *Ls, int d, uint32_t m, uint32_t id,
                                         uint32_t val, F f)
{
    const int lane = threadIdx.x & 31;
#pragma unroll 1
    while (m) {
        const int q = __ffs(m) - 1;
        m &= m - 1u;
        const float *row = x + (size_t)__shfl_sync(0xffffffffu, id, q) * d;
        const uint32_t vq = __shfl_sync(0xffffffffu, val, q);
#pragma unroll 1
        for (int j0 = 0; j0 < d; j0 += 128) {
            float v[4];
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const int j = j0 + 32 * u + lane;
                v[u] = j < d ? __ldg(&row[j]) : -1.0f;
            }
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const int j = j0 + 32 * u + lane;
                if (j < d && v[u] == Ls[j]) f(j, vq);
            }
        }
    }
}

// Many holders among a warp's points, few attributes: the lanes walk their points side by side (10^6 x
// 3 with 4 values an attribute, most of a band's 10^5 points holders and one CTA settling them: 9.0 ->
// 5.1 ms of peel).
__device__ __noinline__ void count_side(const float *__restrict__ x, const float *Ls, int d, bool hold, uint32_t id,
                                        uint32_t round, uint32_t (*hcnt)[kMaxEpoch])
{
    if (!hold) return;
    const float *row = x + (size_t)id * d;
#pragma unroll 4
    for (int j = 0; j < d; j++)
        if (__ldg(&row[j]) == Ls[j]) atomicAdd(&hcnt[j][round], 1u);
}

// The holders counted per attribute and round (out of line: rare, and three callers)
__device__ __noinline__ void count_held(const float *__restrict__ x, const float *Ls, int d, bool hold, uint32_t id,
                                        uint32_t round, uint32_t (*hcnt)[kMaxEpoch])
{
    const uint32_t m = __ballot_sync(0xffffffffu, hold);
    if (__popc(m) > max(4, d / 2)) return count_side(x, Ls, d, hold, id, round, hcnt);
    for_held(x, Ls, d, m, id, round, [&](int j, uint32_t r) { atomicAdd(&hcnt[j][r], 1u); });
}

// The largest key among the holders of each attribute
__device__ __noinline__ void max_held(const float *__restrict__ x, const float *Ls, int d, bool hold, uint32_t id,
                                      uint32_t key, uint32_t *hmax)
{
    for_held(x, Ls, d, __ballot_sync(0xffffffffu, hold), id, key, [&](int j, uint32_t k) { atomicMax(&hmax[j], k); });
}

// A group of more entries than fit in shared memory: each of its boundaries' cut by selection,
// then the entries within the cut's error ranked by float64 and index (see settle_group).
__device__ __noinline__ void settle_large(const PeelArgs &a, const float *Ls, uint32_t q1, uint32_t q2, uint32_t off,
                                          uint32_t ne, uint32_t before, uint32_t r0, uint32_t K,
                                          uint32_t (*hcnt)[kMaxEpoch], uint32_t *scr)
{
    PeelCtl *ctl = a.ctl;
    const int d = a.d;
    const uint32_t N = (uint32_t)a.N;
    const int t = threadIdx.x;
    __shared__ uint32_t s_na;
    __shared__ double s_lo[kMaxEpoch], s_hi[kMaxEpoch];
    __shared__ uint32_t s_need[kMaxEpoch], s_need3[kMaxEpoch], s_na3[kMaxEpoch], s_p3[kMaxEpoch];
    __shared__ unsigned long long s_k3[kMaxEpoch];
    __shared__ uint32_t s_bc[kMaxEpoch];
    const uint64_t *gk = a.gkey + off;
    const uint32_t *gp = a.gpos + off;
    uint64_t *ak = a.akey + off;
    uint32_t *ap = a.apos + off;
    if (t < kMaxEpoch) s_bc[t] = 0;
    __syncthreads();
    auto KA = [&](uint32_t i) -> uint64_t { return __ldcg(&gk[i]); };
    // an entry's id (bit 31 of the stored word is its hold flag)
    auto PA = [&](uint32_t i) -> uint32_t { return __ldcg(&gp[i]) & kPosMask; };
    const double win_rel = 4.0 * ((double)eps_ff(d) + 0x1p-52);
    for (uint32_t i = q1; i <= q2; i++) {
        const uint32_t bi = i - q1;
        const int64_t need_s = (int64_t)(i + 1) * N - (int64_t)before;
        uint32_t need = need_s < 0 ? 0u : (need_s > (int64_t)ne ? ne : (uint32_t)need_s);
        if (t == 0 && (need_s < 0 || need_s > (int64_t)ne)) atomicOr(&a.flags[1], 1u);
        if (need == 0 || need == ne) {
            if (t == 0) s_need[bi] = need;
            __syncthreads();
            continue;
        }
        uint64_t V;
        uint32_t Pv;
        select_kth(gk, gp, ne, need, scr, V, Pv);
        const double v = __longlong_as_double((long long)V);
        const double win = win_rel * v + 0x1p-110;
        const double lo = v - win, hi = v + win;
        if (t == 0) s_na = 0;
        __syncthreads();
        uint32_t below = 0;
        for (uint32_t e = t; e < ne; e += kThreads) {
            const double ke = __longlong_as_double((long long)KA(e));
            if (ke < lo) {
                below++;
            } else if (ke <= hi) {
                const uint32_t slot = atomicAdd(&s_na, 1u);
                ap[slot] = PA(e);
            }
        }
        below = block_sum(below);
        const uint32_t na = s_na;
        const uint32_t need3 = need >= below ? need - below : 0u;
        if (t == 0 && (need < below || need3 > na)) atomicOr(&a.flags[1], 1u);
        uint64_t K3 = 0;
        uint32_t P3 = 0;
        if (need3 > 0 && need3 < na) {
            // the entries within the error of the cut-off, ranked by float64 and index
            for (uint32_t e = t; e < na; e += kThreads) {
                const uint32_t pos = __ldcg(&ap[e]);
                ak[e] = (uint64_t)__double_as_longlong(dist64(a.x + (size_t)pos * d, Ls, d));
            }
            __syncthreads();
            select_kth(ak, ap, na, need3, scr, K3, P3);
        }
        if (t == 0) {
            s_need[bi] = need;
            s_lo[bi] = lo;
            s_hi[bi] = hi;
            s_need3[bi] = need3;
            s_na3[bi] = na;
            s_k3[bi] = K3;
            s_p3[bi] = P3;
        }
        __syncthreads();
    }
    // every entry's round: the first boundary of the group plus the boundaries it is after
    for (uint32_t e0 = 0; e0 < ne; e0 += kThreads) {            // block-uniform bound
        const uint32_t e = e0 + (uint32_t)t;
        const bool v = e < ne;
        const uint64_t kb = v ? KA(e) : 0ull;
        const uint32_t raw = v ? __ldcg(&gp[e]) : 0u;
        const uint32_t pos = raw & kPosMask;
        const double ke = __longlong_as_double((long long)kb);
        uint32_t after = 0;
        for (uint32_t bi = 0; v && bi <= q2 - q1; bi++) {
            const uint32_t need = s_need[bi];
            if (need == 0) {
                after++;
                continue;
            }
            if (need == ne || ke < s_lo[bi]) continue;
            if (ke > s_hi[bi]) {
                after++;
                continue;
            }
            const uint32_t n3 = s_need3[bi];
            if (n3 == 0) {
                after++;
            } else if (n3 < s_na3[bi]) {
                const uint64_t k64 = (uint64_t)__double_as_longlong(dist64(a.x + (size_t)pos * d, Ls, d));
                if (k64 > s_k3[bi] || (k64 == s_k3[bi] && pos > s_p3[bi])) after++;
            }
        }
        const uint32_t rr = q1 + after;
        if (v && rr < K) {
            a.rnd[pos] = r0 + rr;
            atomicAdd(&s_bc[rr], 1u);
        }
        const bool ch = v && rr < K && (raw & ~kPosMask);
        if (__any_sync(0xffffffffu, ch)) count_held(a.x, Ls, d, ch, pos, rr, hcnt);
    }
    __syncthreads();
    if (t < (int)K && s_bc[t]) atomicAdd(&ctl->bnd[t], s_bc[t]);
}

// The window k - W .. k + W of a distance k (bit patterns; see settle_group).
constexpr uint64_t kTiny = 963ull << 52;                                    // 2^-60
__device__ __forceinline__ uint64_t win_lo(uint64_t k, uint64_t W) { return k < kTiny + W ? 0ull : k - W; }
__device__ __forceinline__ uint64_t win_hi(uint64_t k, uint64_t W) { return (k < kTiny ? kTiny : k) + W; }

// The ranks of a group's nn (<= kNear) near entries by (float64 distance, id), where ties make most
// of them close: a bitonic network over their indexes, padded to a power of two by indexes past the
// last, then for each the entries before it: the near ones, and those of the bins below its window
// that are not marked.  mn, sh, hist, mark: settle_group's bins; W: its window.
__device__ __noinline__ void rank_many(const float *__restrict__ x, const float *Ls, int d, uint64_t mn, int sh,
                                       uint32_t nn, const uint64_t *nk, uint64_t *d64, const uint32_t *np,
                                       const uint32_t *hist, const uint32_t *mark, uint32_t *rank, uint64_t W)
{
    const uint32_t t = threadIdx.x, m = 1u << (32 - __clz((int)max(nn, 2u) - 1));
    uint32_t *idx = rank;
#pragma unroll 1
    for (uint32_t f = t; f < nn; f += kThreads)
        d64[f] = (uint64_t)__double_as_longlong(dist64(x + (size_t)(np[f] & kPosMask) * d, Ls, d));
#pragma unroll 1
    for (uint32_t i = t; i < m; i += kThreads) idx[i] = i;
    __syncthreads();
#pragma unroll 1
    for (uint32_t k = 2; k <= m; k *= 2)
#pragma unroll 1
        for (uint32_t j = k / 2; j; j /= 2) {
#pragma unroll 1
            for (uint32_t q = t; q < m / 2; q += kThreads) {
                const uint32_t lo = 2 * q - (q & (j - 1u)), hi = lo + j;
                const uint32_t a = idx[lo], b = idx[hi];
                bool less = b < nn;                       // b before a
                if (less && a < nn) {
                    const uint64_t ka = d64[a], kb = d64[b];
                    less = kb < ka || (kb == ka && (np[b] & kPosMask) < (np[a] & kPosMask));
                }
                if (less == ((lo & k) == 0u)) {
                    idx[lo] = b;
                    idx[hi] = a;
                }
            }
            __syncthreads();
        }
    uint32_t *rk = reinterpret_cast<uint32_t *>(d64);     // (done with)
#pragma unroll 1
    for (uint32_t p = t; p < nn; p += kThreads) {
        const uint32_t u = idx[p];
        const uint64_t lo = win_lo(nk[u], W);
        const uint32_t bl = lo <= mn ? 0u : (uint32_t)((lo - mn) >> sh);
        uint32_t before = p;
#pragma unroll 1
        for (uint32_t wd = 0; wd <= bl >> 5; wd++) {
            uint32_t un = ~mark[wd];
            if (wd == bl >> 5) un &= (1u << (bl & 31u)) - 1u;
            if (un == ~0u) {
                before += hist[32u * wd + 32u] - hist[32u * wd];
                continue;
            }
#pragma unroll 1
            for (; un; un &= un - 1u) {
                const uint32_t b = 32u * wd + (uint32_t)__ffs(un) - 1u;
                before += hist[b + 1u] - hist[b];
            }
        }
        rk[u] = before;
    }
    __syncthreads();
#pragma unroll 1
    for (uint32_t u = t; u < nn; u += kThreads) rank[u] = rk[u];
}

// Settles group g of the epoch's boundaries (one CTA): every band entry of the group gets
// its round, exactly by (delta64, index).  q1 .. q2: the group's boundaries; off, ne: its region
// of the regrouped entries; certs: the points certainly in rounds 0 .. q1; r0: the epoch's first
// round; K: its boundaries; stage: the entries that fit past the scratch (0: none).
//
// An entry's round follows from its rank among the group's by their compensated distances:
// the entries whose distance is smaller beyond the error window come before it, and where the
// window holds others and a boundary cuts through it, those of them that are smaller by float64
// and index.  The window of a distance with bits k: k +- W, W >= 4 (eps_ff + 2^-52) 2^53 (a
// relative step r moves a double's bits by at most r 2^53); below 2^-60 the absolute error of
// tiny squares counts too, so all of them are one window.  A histogram of the distances tells
// most entries' sides of every boundary; only those close to one (all, of a small group) are
// ranked one by one, a warp each, against the entries of the bins their windows touch: no
// selection, and few barriers (past kRankOne of them by rank_many).  Short rolled loops throughout: the CTA that settles a group is
// the only one that fetches this code, and the others wait for it.  (Every entry ranked against
// every other: 25 us for 1000 entries; the selection of larger groups: 130 to 170 us.)
__device__ __noinline__ void settle_group(const PeelArgs &a, const float *Ls, uint32_t g, uint32_t q1, uint32_t q2,
                                          uint32_t off, uint32_t ne, uint32_t certs, uint32_t r0, uint32_t K,
                                          uint32_t (*hcnt)[kMaxEpoch], uint32_t *scr, uint32_t stage)
{
    PeelCtl *ctl = a.ctl;
    const int d = a.d;
    const uint32_t N = (uint32_t)a.N;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    __shared__ uint32_t s_need[kMaxEpoch], s_bc[kMaxEpoch];
    __shared__ unsigned long long s_mn[kW], s_mx[kW];
    __shared__ uint32_t s_near, s_close, s_any;
    // points before the group: the certain ones and the entries of the groups before it
    const uint32_t before = certs + off, filled = __ldcg(&ctl->gfill[g]);
    uint32_t *hist = scr, *mark = hist + kRankBins;                         // entries before a bin; bins marked
    uint64_t *nk = reinterpret_cast<uint64_t *>(mark + kRankBins / 32);     // near entries: distance,
    uint64_t *d64 = nk + kNear;                                             // by float64,
    uint32_t *np = reinterpret_cast<uint32_t *>(d64 + kNear);               // id and hold flag,
    uint8_t *nst = reinterpret_cast<uint8_t *>(np + kNear), *e64 = nst + kNear;   // state, in a cut window
    // state: the entry's round is its rank's to find; a boundary cuts its window; else neither
    constexpr uint8_t kClose = 1, kCut = 2;
    uint64_t *stk = reinterpret_cast<uint64_t *>(scr + kScrWords);
    uint32_t *stp = reinterpret_cast<uint32_t *>(stk + kStage);
    const uint64_t *gk = a.gkey + off;
    const uint32_t *gp = a.gpos + off;
    const bool all = ne <= 64u, st = ne <= stage && !all;
    const uint32_t nq = q2 - q1 + 1u;
    if (t < kMaxEpoch) s_bc[t] = 0;
    if (t == 0 && filled != ne) atomicOr(&a.flags[1], 1u);
    if (t < (int)nq) {
        const int64_t need_s = (int64_t)(q1 + t + 1) * N - (int64_t)before;
        s_need[t] = need_s < 0 ? 0u : (need_s > (int64_t)ne ? ne : (uint32_t)need_s);
        if (need_s < 0 || need_s > (int64_t)ne) atomicOr(&a.flags[1], 1u);
    }
    if (t == 0) {
        s_any = s_close = 0;
        s_near = all ? ne : 0u;
    }
    const uint64_t W0 = 256ull * ((uint64_t)d * d + 8ull * d + 1ull) + 8ull, W = W0 + (W0 >> 4);
    auto KEY = [&](uint32_t e) -> uint64_t { return st ? stk[e] : __ldcg(&gk[e]); };
    auto RAW = [&](uint32_t e) -> uint32_t { return st ? stp[e] : __ldcg(&gp[e]); };
    auto settle = [&](bool v, uint32_t raw, uint32_t rr) {                  // a warp's entries with v set
        if (v && rr < K) {
            a.rnd[raw & kPosMask] = r0 + rr;
            atomicAdd(&s_bc[rr], 1u);
        }
        const bool ch = v && rr < K && (raw & ~kPosMask);
        if (__any_sync(0xffffffffu, ch)) count_held(a.x, Ls, d, ch, raw & kPosMask, rr, hcnt);
    };
    unsigned long long mn = ~0ull, mx = 0ull;
    int sh = 0;
    auto bin = [&](uint64_t k) { return k <= mn ? 0u : (uint32_t)(min(k, (uint64_t)mx) - mn >> sh); };
    // an entry's round from the bins alone; true if a boundary lies among those of its window
    auto close_to = [&](uint64_t k, uint32_t &rr, uint32_t &bl, uint32_t &bh) {
        bl = bin(win_lo(k, W));
        bh = bin(win_hi(k, W));
        const uint32_t least = hist[bl], most = bh + 1u < (uint32_t)kRankBins ? hist[bh + 1u] : ne;
        rr = q1;
        bool close = false;                                                 // the rank lies in [least, most)
#pragma unroll 1
        for (uint32_t b = 0; b < nq; b++) {
            rr += s_need[b] <= least;
            close |= s_need[b] > least && s_need[b] < most;
        }
        return close;
    };
    // f(e, key, whether e < ne) for every entry, by whole warps: the keys of four loaded at once
    auto each = [&](auto f) {
#pragma unroll 1
        for (uint32_t e0 = 0; e0 < ne; e0 += 4 * kThreads) {
            uint64_t k4[4];
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const uint32_t e = e0 + u * kThreads + t;
                k4[u] = e < ne ? KEY(e) : 0ull;
            }
#pragma unroll 1
            for (uint32_t u = 0; u < 4 && e0 + u * kThreads < ne; u++) {
                const uint32_t e = e0 + u * kThreads + t;
                f(e, u < 2 ? (u ? k4[1] : k4[0]) : (u == 2 ? k4[2] : k4[3]), e < ne);
            }
        }
    };
    if (all) {
        if (t < (int)ne) {
            nk[t] = __ldcg(&gk[t]);
            np[t] = __ldcg(&gp[t]);
            nst[t] = kClose;
            e64[t] = 0;
        }
    } else {
#pragma unroll 4
        for (uint32_t e = t; e < ne; e += kThreads) {
            const unsigned long long k = __ldcg(&gk[e]);
            if (st) {
                stk[e] = k;
                stp[e] = __ldcg(&gp[e]);
            }
            mn = min(mn, k);
            mx = max(mx, k);
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            mn = min(mn, __shfl_xor_sync(0xffffffffu, mn, o));
            mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        }
        if (lane == 0) {
            s_mn[w] = mn;
            s_mx[w] = mx;
        }
#pragma unroll 1
        for (int b = t; b < kRankBins + kRankBins / 32; b += kThreads) hist[b] = 0;
        __syncthreads();
#pragma unroll 1
        for (int q = 0; q < kW; q++) {
            mn = min(mn, s_mn[q]);
            mx = max(mx, s_mx[q]);
        }
        sh = max(0, 53 - __clzll((long long)((mx - mn) | 1ull)));           // (mx - mn) >> sh < kRankBins
        each([&](uint32_t, uint64_t k, bool v) {
            if (v) atomicAdd(&hist[bin(k)], 1u);
        });
        __syncthreads();
        {
            constexpr int per = kRankBins / kThreads;
            uint32_t c[per], sum = 0, tot;
#pragma unroll
            for (int q = 0; q < per; q++) {
                c[q] = hist[t * per + q];
                sum += c[q];
            }
            uint32_t ex = block_excl_scan(sum, tot);
#pragma unroll
            for (int q = 0; q < per; q++) {
                hist[t * per + q] = ex;
                ex += c[q];
            }
        }
        __syncthreads();
        // the bins of the close entries' windows, and the entries in those
        each([&](uint32_t, uint64_t k, bool v) {
            uint32_t rr, bl, bh;
            if (v && close_to(k, rr, bl, bh))
#pragma unroll 1
                for (uint32_t b = bl; b <= bh; b++)
                    if (!((mark[b >> 5] >> (b & 31u)) & 1u)) atomicOr(&mark[b >> 5], 1u << (b & 31u));
        });
        __syncthreads();
        each([&](uint32_t e, uint64_t k, bool v) {
            const uint32_t b = bin(k);
            if (v && ((mark[b >> 5] >> (b & 31u)) & 1u)) {
                const uint32_t slot = atomicAdd(&s_near, 1u);
                if (slot < (uint32_t)kNear) {
                    uint32_t rr, bl, bh;
                    const bool cl = close_to(k, rr, bl, bh);
                    nk[slot] = k;
                    np[slot] = RAW(e);
                    nst[slot] = cl ? kClose : (uint8_t)0;
                    e64[slot] = 0;
                    if (cl) atomicAdd(&s_close, 1u);
                }
            }
        });
    }
    __syncthreads();
    const uint32_t nn = s_near;
    if (nn > (uint32_t)kNear) {                                             // heavily tied
        settle_large(a, Ls, q1, q2, off, ne, before, r0, K, hcnt, scr);
        return;
    }
    // the close entries' ranks, among the near ones: every entry of the bins that a close one's
    // window touches is near
    __shared__ uint32_t s_rank[kNear];
    const bool many = s_close > (uint32_t)kRankOne;
    if (many) rank_many(a.x, Ls, d, mn, sh, nn, nk, d64, np, hist, mark, s_rank, W);
#pragma unroll 1
    for (uint32_t u = many ? nn : (uint32_t)w; u < nn; u += kW) {
        if (!(nst[u] & kClose)) continue;                                   // the warp's
        const uint64_t k = nk[u], lo = win_lo(k, W), hi = win_hi(k, W);
        const uint32_t bl = all ? 0u : bin(lo), base = all ? 0u : hist[bl];
        uint32_t below = 0, upto = 0;
#pragma unroll 2
        for (uint32_t f = (uint32_t)lane; f < nn; f += 32) {
            const uint64_t kf = nk[f];
            const bool in = all || bin(kf) >= bl;
            below += in && kf < lo;
            upto += in && kf <= hi;
        }
        below = base + __reduce_add_sync(0xffffffffu, below);
        upto = base + __reduce_add_sync(0xffffffffu, upto);
        // lane q: the group's boundary q
        const bool cut = __any_sync(0xffffffffu, (uint32_t)lane < nq && s_need[lane] > below && s_need[lane] < upto);
        if (lane == 0) {
            s_rank[u] = below;
            if (cut) nst[u] = kClose | kCut;
            if (cut) s_any = 1;
        }
        // the entries of a window that a boundary cuts are ranked by float64
        if (cut)
#pragma unroll 2
            for (uint32_t f = (uint32_t)lane; f < nn; f += 32)
                if (nk[f] >= lo && nk[f] <= hi) e64[f] = 1;
    }
    __syncthreads();
    if (s_any) {
#pragma unroll 1
        for (uint32_t f = t; f < nn; f += kThreads)
            if (e64[f]) d64[f] = (uint64_t)__double_as_longlong(dist64(a.x + (size_t)(np[f] & kPosMask) * d, Ls, d));
        __syncthreads();
#pragma unroll 1
        for (uint32_t u = (uint32_t)w; u < nn; u += kW) {
            if (!(nst[u] & kCut)) continue;                                 // the warp's
            const uint32_t pu = np[u] & kPosMask;
            const uint64_t k = nk[u], lo = win_lo(k, W), hi = win_hi(k, W), ku = d64[u];
            uint32_t more = 0;
#pragma unroll 2
            for (uint32_t f = (uint32_t)lane; f < nn; f += 32)
                if (nk[f] >= lo && nk[f] <= hi)
                    more += d64[f] < ku || (d64[f] == ku && (np[f] & kPosMask) < pu);
            more = __reduce_add_sync(0xffffffffu, more);
            if (lane == 0) s_rank[u] += more;
        }
        __syncthreads();
    }
    // the rounds: of the close entries by rank, of the others by their bins
#pragma unroll 1
    for (uint32_t u0 = 0; u0 < nn; u0 += kThreads) {                        // block-uniform bounds
        const uint32_t u = u0 + (uint32_t)t;
        const bool v = u < nn && (nst[u] & kClose);
        uint32_t rr = q1;
#pragma unroll 1
        for (uint32_t b = 0; v && b < nq; b++) rr += s_need[b] <= s_rank[u];
        settle(v, v ? np[u] : 0u, rr);
    }
    if (!all)
        each([&](uint32_t e, uint64_t k, bool in) {
            uint32_t rr = 0, bl, bh;
            const bool v = in && !close_to(k, rr, bl, bh);
            settle(v, v ? RAW(e) : 0u, rr);
        });
    __syncthreads();
    if (t < (int)K && s_bc[t]) atomicAdd(&ctl->bnd[t], s_bc[t]);
}

// The next landmark: in each attribute that lost its last holder (lost[0 .. nl), shared), the smallest
// value among the points left, here those of one CTA's list, kMinAttrs attributes and
// kMinBatch points per thread at a time (their loads issued together), added to the grid's
// minimum (values lie in [0, 1], so their bits order like them).
constexpr int kMinAttrs = 4;

template <int kMinBatch>
__device__ __noinline__ void lost_minima(const float *__restrict__ x, const float *__restrict__ xt, uint32_t n, int d,
                                         uint32_t n_live, bool kc, const uint32_t *sid, const uint32_t *glist,
                                         const uint16_t *lost, uint32_t nl, uint32_t *Lbits)
{
    __shared__ uint32_t s_min[kMinAttrs];
    const int t = threadIdx.x, lane = t & 31;
    const float *src = xt ? xt : x;
    const size_t ps = xt ? 1 : (size_t)d, as = xt ? (size_t)n : 1;
#pragma unroll 1
    for (uint32_t l0 = 0; l0 < nl; l0 += kMinAttrs) {
        const float *col[kMinAttrs];
        uint32_t mn[kMinAttrs];
#pragma unroll
        for (int i = 0; i < kMinAttrs; i++) {       // past the last one, the first of the group again
            const uint32_t j = lost[l0 + i < nl ? l0 + i : l0];
            col[i] = src + (size_t)j * as;
            mn[i] = kInfBits;
        }
        if (t < kMinAttrs) s_min[t] = kInfBits;
        __syncthreads();
        const uint32_t na = min((uint32_t)kMinAttrs, nl - l0);
#pragma unroll 1
        for (uint32_t q0 = 0; q0 < n_live; q0 += kMinBatch * kThreads) {
            uint32_t id[kMinBatch];
#pragma unroll
            for (int u = 0; u < kMinBatch; u++) {
                const uint32_t qi = q0 + u * kThreads + t;
                id[u] = qi < n_live ? (kc ? sid[qi] : __ldcg(&glist[qi])) : kGone;
            }
#pragma unroll
            for (int i = 0; i < kMinAttrs; i++)
                if (i < (int)na) {
#pragma unroll
                    for (int u = 0; u < kMinBatch; u++)
                        mn[i] = min(mn[i], id[u] != kGone ? __float_as_uint(__ldcg(&col[i][(size_t)id[u] * ps])) : kInfBits);
                }
        }
#pragma unroll
        for (int i = 0; i < kMinAttrs; i++) {
            const uint32_t m = __reduce_min_sync(0xffffffffu, mn[i]);
            if (lane == 0 && i < (int)na) atomicMin(&s_min[i], m);
        }
        __syncthreads();
        if (t < (int)na && s_min[t] != kInfBits) atomicMin(&Lbits[lost[l0 + t]], s_min[t]);
    }
}

// The same where many attributes lost theirs at once (correlated data: one point holds the minimum
// of most): each warp takes its own four attributes over all of the CTA's points, without a barrier
// between them, kManyBatch points a lane in flight (points on a line, each round's holding every
// minimum: 300000 x 128 in rounds of 1000 57 -> 26 ms of peel, 10^6 x 64 in rounds of 4000 43 -> 28,
// 200000 x 16 in rounds of 249 30 -> 27).
constexpr int kMinMany = 2 * kW, kManyBatch = 8;

__device__ __noinline__ void many_minima(const float *__restrict__ x, const float *__restrict__ xt, uint32_t n, int d,
                                         uint32_t n_live, bool kc, const uint32_t *sid, const uint32_t *glist,
                                         const uint16_t *lost, uint32_t nl, uint32_t *Lbits)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const float *src = xt ? xt : x;
    const size_t ps = xt ? 1 : (size_t)d, as = xt ? (size_t)n : 1;
#pragma unroll 1
    for (uint32_t l0 = (uint32_t)w * kMinAttrs; l0 < nl; l0 += kW * kMinAttrs) {
        const float *col[kMinAttrs];
        uint32_t mn[kMinAttrs];
#pragma unroll
        for (int i = 0; i < kMinAttrs; i++) {       // past the last one, the first of the group again
            col[i] = src + (size_t)lost[l0 + i < nl ? l0 + i : l0] * as;
            mn[i] = kInfBits;
        }
#pragma unroll 1
        for (uint32_t q0 = 0; q0 < n_live; q0 += kManyBatch * 32) {
            uint32_t id[kManyBatch];
#pragma unroll
            for (int u = 0; u < kManyBatch; u++) {
                const uint32_t qi = q0 + u * 32 + lane;
                id[u] = qi < n_live ? (kc ? sid[qi] : __ldcg(&glist[qi])) : kGone;
            }
#pragma unroll
            for (int i = 0; i < kMinAttrs; i++)
#pragma unroll
                for (int u = 0; u < kManyBatch; u++)
                    mn[i] = min(mn[i], id[u] != kGone ? __float_as_uint(__ldcg(&col[i][(size_t)id[u] * ps])) : kInfBits);
        }
#pragma unroll
        for (int i = 0; i < kMinAttrs; i++) {
            const uint32_t m = __reduce_min_sync(0xffffffffu, mn[i]);
            if (lane == 0 && l0 + i < nl && m != kInfBits) atomicMin(&Lbits[lost[l0 + i]], m);
        }
    }
}

// The epoch's groups of boundaries: group g's band holds the keys in [in, out], its last
// boundary is q2 (its first the one after group g - 1's).
struct GroupTab {
    uint32_t in[kMaxEpoch], out[kMaxEpoch], q2[kMaxEpoch], ng;
    float kref;                  // lower end of the first boundary's key range
};

// After phase B: each boundary's first-digit bin and rank inside it become its band cut-offs
// (second digit from the boundary's histogram), and boundaries whose bands overlap merge into
// groups (tab, in shared memory).  Every CTA does this for itself when the boundaries are
// few; otherwise the last CTA to arrive does it for all.  Warp w resolves boundaries w, w + kW,
// ...: lane i holds
// second-digit bins [64 i, 64 i + 64), a warp scan finds the lane holding the rank, and that
// lane counts its bins before it.
__device__ __noinline__ void resolve_cutoffs(PeelCtl *ctl, uint32_t K, float keps, float kabs, const DigitMap *dm,
                                             const uint32_t *sb, const uint32_t *sr, const uint32_t *sslot,
                                             GroupTab &tab)
{
    __shared__ uint32_t s_b1[kMaxEpoch];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const DigitMap mp = *dm;
    if (t < kMaxEpoch) s_b1[t] = 0;
    __syncthreads();
#pragma unroll 1
    for (uint32_t q = (uint32_t)w; q < K; q += kW) {
        const uint4 *h4 = reinterpret_cast<const uint4 *>(ctl->h1[sslot[q]] + lane * 64);
        uint4 h[16];
#pragma unroll
        for (int i = 0; i < 16; i++) h[i] = __ldcg(h4 + i);
        uint32_t ls = 0, hs[16];
#pragma unroll
        for (int i = 0; i < 16; i++) hs[i] = ls += h[i].x + h[i].y + h[i].z + h[i].w;
        const uint32_t ex = warp_incl_scan(ls) - ls;
        const uint32_t r = sr[q];
        if (r >= ex && r < ex + ls) {
            // the four bins that hold the rank, then the one of them
            uint32_t cc = ex, found = 0;
            uint4 at = h[0];
#pragma unroll
            for (int i = 0; i < 16; i++) {
                const uint32_t end = ex + hs[i];      // past the i-th four
                if (end <= r) {
                    found = 4u * (uint32_t)i + 4u;
                    cc = end;
                } else if (found == 4u * (uint32_t)i) {
                    at = h[i];
                }
            }
            found += (cc + at.x <= r) + (cc + at.x + at.y <= r) + (cc + at.x + at.y + at.z <= r);
            s_b1[q] = found + (uint32_t)lane * 64u;
        }
    }
    __syncthreads();
    static_assert(kMaxEpoch <= 32, "a lane per boundary");
    if (w == 0) {
        // lane q: boundary q's cut-offs, ascending with q; a boundary whose band starts past
        // the one before it ends opens a group
        uint32_t A = 0, B = 0, ik = 0, ok = 0;
        if (lane < (int)K) {
            mp.range(sb[lane], s_b1[lane], A, B);
            band_cutoffs(A, B, keps, kabs, ik, ok);
        }
        const uint32_t pk = __shfl_up_sync(0xffffffffu, ok, 1);
        const uint32_t open = __ballot_sync(0xffffffffu, lane < (int)K && (lane == 0 || ik > pk));
        if (lane < (int)K) {
            const uint32_t g = (uint32_t)__popc(open & ((2u << lane) - 1u)) - 1u;
            if ((open >> lane) & 1u) tab.in[g] = ik;
            if (lane == (int)K - 1 || ((open >> (lane + 1)) & 1u)) {
                tab.out[g] = ok;
                tab.q2[g] = (uint32_t)lane;
            }
        }
        if (lane == 0) {
            tab.ng = (uint32_t)__popc(open);
            tab.kref = __uint_as_float(A);
        }
    }
    __syncthreads();
}

// After phase D, in every CTA: how many rounds the epoch commits, up to the first round after
// which some attribute has no holder of its landmark value left (the landmark then changes);
// which attributes those are (s_lost); and the smallest key that a point left can have.  Each
// CTA forms them from the grid's counts (an L2 round trip; one CTA doing it for all would
// add another for its answer).  chold, the holders per attribute, is read here and its
// successor chold2 written by CTA 0; CTA 0 also checks that every round got exactly N points.
__device__ __noinline__ void commit_count(const PeelArgs &a, uint32_t K, const GroupTab &tab, const uint32_t *chold,
                                          uint32_t *chold2, const uint32_t (*hcnt)[kMaxEpoch], uint32_t &s_kcm,
                                          uint32_t &s_nl, uint32_t &s_klast, uint16_t *s_lost)
{
    PeelCtl *ctl = a.ctl;
    const int d = a.d;
    const int t = threadIdx.x;
    const bool own = blockIdx.x == 0;
    if (t == 0) s_nl = 0;
    if (own && t < (int)K && __ldcg(&ctl->cert[t]) + __ldcg(&ctl->bnd[t]) != (uint32_t)a.N) atomicOr(&a.flags[1], 1u);
    // per attribute: the first round after which no holder of L_j is left
    // (the counts are read all at once, then scanned in registers; those of a thread's first
    // attribute stay there for the second use)
    constexpr int RB = 8;
    uint32_t qs = kNone, hc[RB], ch = 0;
    for (int j0 = (d - 1) / kThreads * kThreads; j0 >= 0; j0 -= kThreads) {
        const int j = j0 + t;
        ch = j < d ? __ldcg(&chold[j]) : 0u;
        uint32_t acc = 0, qj = kNone;
#pragma unroll 1
        for (uint32_t q0 = 0; q0 < K; q0 += RB) {
#pragma unroll
            for (int r = 0; r < RB; r++) hc[r] = q0 + r < K && j < d ? __ldcg(&hcnt[j][q0 + r]) : 0u;
#pragma unroll
            for (int r = 0; r < RB; r++) {
                acc += hc[r];
                if (qj == kNone && q0 + r < K && j < d && acc >= ch) qj = q0 + (uint32_t)r;
            }
        }
        qs = min(qs, qj);
    }
    qs = block_min(qs);
    const uint32_t kc_ = qs < K ? qs + 1u : K;
    // the holders that leave with the committed rounds; an attribute that has none left gets
    // a new landmark value (the minimum over the points left, taken next) and its holders are
    // counted by the next pass
    for (int j = t; j < d; j += kThreads) {
        uint32_t gone = 0;
#pragma unroll 1
        for (uint32_t q0 = 0; q0 < kc_; q0 += RB) {
            if (j >= kThreads || K > (uint32_t)RB) {
#pragma unroll
                for (int r = 0; r < RB; r++) hc[r] = q0 + r < kc_ ? __ldcg(&hcnt[j][q0 + r]) : 0u;
            }
#pragma unroll
            for (int r = 0; r < RB; r++) gone += q0 + r < kc_ ? hc[r] : 0u;
        }
        const uint32_t left = (j >= kThreads ? __ldcg(&chold[j]) : ch) - gone;
        if (own) chold2[j] = left;
        if (left == 0u) s_lost[atomicAdd(&s_nl, 1u)] = (uint16_t)j;
    }
    // every point left lies at or past the start of the last committed boundary's band
    if (t < 32) {
        const uint32_t past = __ballot_sync(0xffffffffu, t < (int)tab.ng && tab.q2[t] >= kc_ - 1u);
        if (past && t == __ffs(past) - 1) s_klast = tab.in[t];
    }
    if (t == 0) s_kcm = kc_;
    __syncthreads();
}

// ------------------------------------------------------------------ the points by attribute
// x (n x d, by point) into xt (d x n, by attribute) for the landmark's minima and the key
// updates: 32 x 32 tiles through shared memory, so that both the reads (32 attributes of a
// point) and the writes (32 points of an attribute) are coalesced.  The peel's own launch
// makes it for small sets, whose few tiles per CTA cost less than another launch; larger ones
// take a launch of their own before it, at full occupancy (2^20 x 16: 240 us inside the
// peel's launch, 25 us outside).
constexpr size_t kTransposeBytes = size_t(1) << 20;

__device__ __forceinline__ void transpose_tiles(const float *__restrict__ x, int64_t n, int d, float *__restrict__ xt,
                                                float (*tile)[33])
{
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int64_t tiles_c = (d + 31) / 32;
    const int64_t tiles = (n + 31) / 32 * tiles_c;
    for (int64_t tt = blockIdx.x; tt < tiles; tt += gridDim.x) {
        const int64_t r0 = tt / tiles_c * 32;
        const int c0 = (int)(tt % tiles_c) * 32;
        for (int k = ty; k < 32; k += kThreads / 32) {
            const int64_t r = r0 + k;
            if (r < n && c0 + tx < d) tile[k][tx] = __ldg(&x[r * d + c0 + tx]);
        }
        __syncthreads();
        for (int k = ty; k < 32; k += kThreads / 32) {
            const int64_t r = r0 + tx;
            if (r < n && c0 + k < d) xt[(size_t)(c0 + k) * (size_t)n + (size_t)r] = tile[tx][k];
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kThreads) k_transpose(const float *__restrict__ x, int64_t n, int d,
                                                        float *__restrict__ xt)
{
    __shared__ float tile[32][33];
    transpose_tiles(x, n, d, xt, tile);
}

// The same for d a multiple of AT (4 to 32): tiles of AT attributes of 4096 / AT points, read four
// attributes at a time, four such loads in flight per thread.  (The 32 x 32 tiles, their loads
// of 4 bytes four in flight and half of their lanes without an attribute at d = 16: 2^20 x 16 72 -> 19 us, 2^24 x 64 2.67 -> 1.26 ms.)
template <int AT>
__global__ void __launch_bounds__(kThreads) k_transpose4(const float4 *__restrict__ x4, int64_t n, int d,
                                                         float *__restrict__ xt)
{
    constexpr int PT = 4096 / AT, A4 = AT / 4, PP = kThreads / A4;      // points a pass reads
    __shared__ float tile[AT][PT + 1];
    const int t = threadIdx.x, g = t % A4, pp = t / A4;
    const int64_t tiles_a = d / AT, tiles = (n + PT - 1) / PT * tiles_a;
    for (int64_t tt = blockIdx.x; tt < tiles; tt += gridDim.x) {
        const int64_t r0 = tt / tiles_a * PT;
        const int c0 = (int)(tt % tiles_a) * AT;
        float4 v[PT / PP];
#pragma unroll
        for (int u = 0; u < PT / PP; u++) {
            const int64_t r = r0 + u * PP + pp;
            if (r < n) v[u] = __ldg(&x4[(r * d + c0) / 4 + g]);
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < PT / PP; u++) {
            const int p = u * PP + pp;
            tile[4 * g][p] = v[u].x;
            tile[4 * g + 1][p] = v[u].y;
            tile[4 * g + 2][p] = v[u].z;
            tile[4 * g + 3][p] = v[u].w;
        }
        __syncthreads();
#pragma unroll 4
        for (int e = t; e < 4096; e += kThreads) {
            const int a = e / PT, p = e % PT;
            if (r0 + p < n) xt[(size_t)(c0 + a) * (size_t)n + (size_t)(r0 + p)] = tile[a][p];
        }
    }
}

template <int AT>
void transpose4_launch(const float *x, int64_t n, int d, float *xt, int sm_count, cudaStream_t st)
{
    constexpr int PT = 4096 / AT;
    const int64_t tiles = (n + PT - 1) / PT * (d / AT);
    k_transpose4<AT><<<(int)std::min<int64_t>(tiles, (int64_t)sm_count * 64), kThreads, 0, st>>>(
        reinterpret_cast<const float4 *>(x), n, d, xt);
}

void transpose_launch(const float *x, int64_t n, int d, float *xt, int sm_count, cudaStream_t st)
{
    if (d % 32 == 0) return transpose4_launch<32>(x, n, d, xt, sm_count, st);
    if (d % 16 == 0) return transpose4_launch<16>(x, n, d, xt, sm_count, st);
    if (d % 8 == 0) return transpose4_launch<8>(x, n, d, xt, sm_count, st);
    if (d % 4 == 0) return transpose4_launch<4>(x, n, d, xt, sm_count, st);
    const int64_t tiles = (n + 31) / 32 * ((d + 31) / 32);
    k_transpose<<<(int)std::min<int64_t>(tiles, (int64_t)sm_count * 64), kThreads, 0, st>>>(x, n, d, xt);
}

// A CTA's list of points left, by list position: ids, float32 keys and state bytes; in
// shared memory when the slice fits the key cache (kc), else in one of two global lists.
struct ListView {
    bool kc;
    const uint32_t *sid, *skey;
    uint8_t *sfl;
    const uint32_t *gid, *gkp;
    uint8_t *gfl;
    uint32_t *gid2, *gkp2;       // the other global list (compaction target)
    uint8_t *gfl2;
    __device__ __forceinline__ uint32_t id(uint32_t q) const { return kc ? sid[q] : __ldcg(&gid[q]); }
    __device__ __forceinline__ uint32_t key(uint32_t q) const { return kc ? skey[q] : __ldcg(&gkp[q]); }
    __device__ __forceinline__ uint8_t *fl() const { return kc ? sfl : gfl; }
};

// Phase C for one CTA's list: every live key classified against the epoch's groups (see
// the kernel); certain points get their round in rnd[] and counted in s_cc, band entries
// are listed (with their hold flag in bit 31 of the id) and counted per group in s_gc.  Only the
// keys of all points are read, kCB per thread in flight; each warp queues its few points of the
// epoch in shared memory and takes them 32 at a time, with full lanes and one round trip for
// their ids and state bytes.  For a list in global memory their positions are noted in gid2 (the
// other list, idle until a compaction) for the commit; returned: how many.  (Handled where they
// were found, unrolled, the phase was 48 KB of code, and fetching it bound the smaller jobs; in
// a rolled loop, a round trip for every few points bound 2^24 x 64: 38 us an epoch.)
constexpr int kQueue = 32 * (kCB + 1);        // a warp's queue: less than 32 left over, and a batch
static_assert(2 * kQueue * kW <= kScrWords, "the warps' queues fit the scratch");

__device__ __noinline__ uint32_t classify_live(const PeelArgs &a, const ListView &L, uint32_t n_live, const float *Ls,
                                              uint32_t r0, uint32_t K, const GroupTab &tab, uint32_t *s_cc,
                                              uint32_t *s_gc, uint32_t (*hcnt)[kMaxEpoch], uint32_t *scr)
{
    __shared__ uint32_t s_hits;
    PeelCtl *ctl = a.ctl;
    const int d = a.d;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    const uint32_t ng = tab.ng, last = tab.out[ng - 1];
    uint8_t *pfl = L.fl();
    uint32_t *qk = scr + w * 2 * kQueue, *qp = qk + kQueue;      // the warp's queue: keys, positions
    if (t == 0) s_hits = 0;
    __syncthreads();
    constexpr uint32_t kBandTag = 0x100u;
    uint32_t cnt = 0;
#pragma unroll 1
    for (uint32_t q0 = (uint32_t)w * 32; q0 < n_live; q0 += kCB * kThreads) {
        uint32_t kk[kCB];
#pragma unroll
        for (int u = 0; u < kCB; u++) {
            const uint32_t qi = q0 + u * kThreads + lane;
            kk[u] = qi < n_live ? L.key(qi) : kGone;
        }
#pragma unroll
        for (int u = 0; u < kCB; u++) {
            const bool in = kk[u] <= last;
            const uint32_t m = __ballot_sync(0xffffffffu, in);
            if (in) {
                const uint32_t o = cnt + __popc(m & lt);
                qk[o] = kk[u];
                qp[o] = q0 + u * kThreads + lane;
            }
            cnt += __popc(m);
        }
        __syncwarp();
        const bool end = q0 + kCB * kThreads >= n_live;           // what is left in the queue, too
#pragma unroll 1
        while (cnt >= 32u || (end && cnt)) {
            const uint32_t m = min(cnt, 32u);
            cnt -= m;
            // a key's class: its round r < K (certainly), kBandTag | g (in group g's band), or
            // kNone (after the epoch: the point keeps its state byte, kFlNone since the last commit)
            uint32_t cls = kNone, id = 0, fl = 0, k = 0;
            if ((uint32_t)lane < m) {
                k = qk[cnt + lane];
                const uint32_t qi = qp[cnt + lane];
                id = L.id(qi);
                fl = pfl[qi];
                uint32_t g = 0, cum = 0;
#pragma unroll 1
                while (g < ng && k > tab.out[g]) {
                    cum = tab.q2[g] + 1u;
                    g++;
                }
                if (g < ng && k >= tab.in[g]) cls = kBandTag | g;
                else if (cum < K) cls = cum;
                if (cls != kNone) pfl[qi] = (uint8_t)((fl & kFlHold) | (cls >= kBandTag ? kFlBand : cls));
            }
            __syncwarp();
            if (!L.kc) {
                const uint32_t hm = __ballot_sync(0xffffffffu, cls != kNone);
                uint32_t base = 0;
                if (lane == 0 && hm) base = atomicAdd(&s_hits, (uint32_t)__popc(hm));
                base = __shfl_sync(0xffffffffu, base, 0);
                if (cls != kNone) L.gid2[base + __popc(hm & lt)] = qp[cnt + lane];
            }
            const bool band = cls != kNone && cls >= kBandTag;
            const bool cert = cls < kBandTag;
            const uint32_t bm = __ballot_sync(0xffffffffu, band);
            if (bm) {
                uint32_t base = 0;
                const int leader = __ffs(bm) - 1;
                if (lane == leader) base = atomicAdd(&ctl->band_cnt, (uint32_t)__popc(bm));
                base = __shfl_sync(0xffffffffu, base, leader);
                if (band) {
                    const uint32_t slot = base + (uint32_t)__popc(bm & lt);
                    a.band_k32[slot] = k;
                    a.band_pos[slot] = id | ((fl & kFlHold) ? ~kPosMask : 0u);
                    atomicAdd(&s_gc[cls - kBandTag], 1u);
                }
            }
            if (cert) {
                a.rnd[id] = r0 + cls;
                atomicAdd(&s_cc[cls], 1u);
            }
            const bool ch = cert && (fl & kFlHold);
            if (__any_sync(0xffffffffu, ch)) count_held(a.x, Ls, d, ch, id, cls, hcnt);
        }
    }
    __syncthreads();
    return s_hits;
}

// Phase E for a list in shared memory (kc), compacted in place: the points whose round
// lies before live_from leave it; dropped assignments are reset; with the landmark kept,
// the committed keys leave the first-digit histogram.  Returns the points left.
__device__ __noinline__ uint32_t compact_shared(const PeelArgs &a, const ListView &L, uint32_t n_live, uint32_t r0,
                                                uint32_t live_from, bool changed, const DigitMap *dmp, uint32_t *scr)
{
    PeelCtl *ctl = a.ctl;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    const DigitMap dm = *dmp;
    uint8_t *pfl = L.sfl;
    if (!changed)
        for (int b = t; b < kHistBins; b += kThreads) scr[b] = 0;
    __syncthreads();
    constexpr int PER = kQT * kW / 32;
    static_assert(PER * 32 == kQT * kW, "one warp scans the tile counts");
    __shared__ uint32_t woff[kQT * kW + 1];
    uint32_t *kid = const_cast<uint32_t *>(L.sid), *kkey = const_cast<uint32_t *>(L.skey);
    uint32_t done = 0;
    // in place: a tile's ids, keys and state bytes are all read before any kept one
    // is written, and those land at or below the tile's own positions.  A position's
    // state byte tells its round in the epoch; only band entries read their round
    // (settled by another CTA) from rnd[].
#pragma unroll 1
    for (uint32_t cb = 0; cb < n_live; cb += kQT * kThreads) {
        // the positions kept, and of those the ones whose assignment is dropped
        uint32_t kp = 0, dropped = 0, out = 0, rv[kQT];
#pragma unroll
        for (int q = 0; q < kQT; q++) {
            const uint32_t qi = cb + q * kThreads + t;
            rv[q] = 0;                                       // past the end: leaves the list
            if (qi < n_live) {
                const uint32_t st = pfl[qi] & 0x7Fu;
                rv[q] = st == kFlBand ? __ldcg(&a.rnd[kid[qi]]) : st == kFlNone ? kNone : r0 + st;
                out |= 1u << q;
            }
        }
#pragma unroll
        for (int q = 0; q < kQT; q++) {
            const bool keep = ((out >> q) & 1u) && rv[q] >= live_from;
            kp |= (uint32_t)keep << q;
            dropped |= (uint32_t)(keep && rv[q] != kNone) << q;
        }
        out &= ~kp;
#pragma unroll
        for (int q = 0; q < kQT; q++) {
            const uint32_t b = __ballot_sync(0xffffffffu, (kp >> q) & 1u);
            if (lane == 0) woff[q * kW + w] = __popc(b);
        }
        // few: in rolled loops (the phase's time was the fetch of 19 KB of unrolled code)
#pragma unroll 1
        while (dropped) {                                    // an assignment dropped
            a.rnd[kid[cb + (__ffs(dropped) - 1) * kThreads + t]] = kNone;
            dropped &= dropped - 1u;
        }
#pragma unroll 1
        while (out && !changed) {
            // the next epoch keeps these keys: the committed ones leave the histogram
            atomicAdd(&scr[dm.bin(kkey[cb + (__ffs(out) - 1) * kThreads + t])], 1u);
            out &= out - 1u;
        }
        uint32_t ids[kQT], keys[kQT], fls[kQT];
#pragma unroll
        for (int q = 0; q < kQT; q++) {
            const uint32_t qi = cb + q * kThreads + t;
            if ((kp >> q) & 1u) {
                ids[q] = kid[qi];
                keys[q] = kkey[qi];
                fls[q] = pfl[qi];
            }
        }
        __syncthreads();
        if (w == 0) {
            uint32_t vk[PER], sk = 0;
#pragma unroll
            for (int e = 0; e < PER; e++) {
                vk[e] = woff[lane * PER + e];
                sk += vk[e];
            }
            const uint32_t ik = warp_incl_scan(sk);
            uint32_t ek = ik - sk;
#pragma unroll
            for (int e = 0; e < PER; e++) {
                woff[lane * PER + e] = ek;
                ek += vk[e];
            }
            if (lane == 31) woff[kQT * kW] = ik;
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kQT; q++) {
            const bool keep = (kp >> q) & 1u;
            const uint32_t b = __ballot_sync(0xffffffffu, keep);
            if (keep) {
                const uint32_t o = done + woff[q * kW + w] + __popc(b & lt);
                kid[o] = ids[q];
                kkey[o] = keys[q];
                pfl[o] = (uint8_t)((fls[q] & kFlHold) | kFlNone);
            }
        }
        done += woff[kQT * kW];
        __syncthreads();
    }

    if (!changed) {
        // the next epoch keeps these keys: the committed ones leave the histogram
        __syncthreads();
        for (int b = t; b < kHistBins; b += kThreads)
            if (scr[b]) atomicSub(&ctl->h0[b], scr[b]);
    }
    return done;
}

// Phase E for a list in global memory.  The epoch's points (n_hit positions noted in gid2 by
// the classification) are taken out in place: those that leave get kGone for their id and key,
// which every pass skips; dropped assignments are reset; with the landmark kept, the committed
// keys leave the first-digit histogram.  Once a quarter of the list is gone, each warp takes
// chunks of 32 kQT positions and appends what is left to the other list (the order does not
// matter: the subclusters are packed by a counting sort over rnd afterwards), claiming slots with
// one shared atomic per chunk.  (Copying the list every epoch moved 18 bytes a point: 44 us an
// epoch at 2^24 x 64.)  gone: the list's gaps, kept by the caller; returns whether the lists
// changed places.
__device__ __noinline__ bool commit_global(const PeelArgs &a, const ListView &L, uint32_t &n_live, uint32_t &gone,
                                           uint32_t n_hit, uint32_t r0, uint32_t live_from, bool changed,
                                           const DigitMap *dmp, uint32_t *scr)
{
    PeelCtl *ctl = a.ctl;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    const DigitMap dm = *dmp;
    uint32_t *gid = const_cast<uint32_t *>(L.gid), *gkp = const_cast<uint32_t *>(L.gkp);
    __shared__ uint32_t s_out;
    if (!changed)
#pragma unroll 1
        for (int b = t; b < kHistBins; b += kThreads) scr[b] = 0;
    if (t == 0) s_out = 0;
    __syncthreads();
    uint32_t left = 0;
#pragma unroll 1
    for (uint32_t h0 = 0; h0 < n_hit; h0 += kQT * kThreads) {
        uint32_t pos[kQT], ids[kQT], keys[kQT], fls[kQT];
#pragma unroll
        for (int q = 0; q < kQT; q++) {
            const uint32_t h = h0 + q * kThreads + t;
            pos[q] = h < n_hit ? __ldcg(&L.gid2[h]) : kGone;
        }
#pragma unroll
        for (int q = 0; q < kQT; q++)
            if (pos[q] != kGone) {
                ids[q] = __ldcg(&gid[pos[q]]);
                keys[q] = __ldcg(&gkp[pos[q]]);
                fls[q] = L.gfl[pos[q]];
            }
#pragma unroll
        for (int q = 0; q < kQT; q++)
            if (pos[q] != kGone) {
                const uint32_t st = fls[q] & 0x7Fu;
                const uint32_t rv = st == kFlBand ? __ldcg(&a.rnd[ids[q]]) : r0 + st;
                if (rv < live_from) {
                    gid[pos[q]] = kGone;
                    gkp[pos[q]] = kGone;
                    L.gfl[pos[q]] = kFlNone;
                    left++;
                    if (!changed) atomicAdd(&scr[dm.bin(keys[q])], 1u);
                } else {
                    L.gfl[pos[q]] = (uint8_t)((fls[q] & kFlHold) | kFlNone);
                    if (rv != kNone) a.rnd[ids[q]] = kNone;              // an assignment dropped
                }
            }
    }
    left = __reduce_add_sync(0xffffffffu, left);
    if (lane == 0 && left) atomicAdd(&s_out, left);
    __syncthreads();
    if (!changed) {
        // the next epoch keeps these keys: the committed ones leave the histogram
#pragma unroll 1
        for (int b = t; b < kHistBins; b += kThreads)
            if (scr[b]) atomicSub(&ctl->h0[b], scr[b]);
    }
    gone += s_out;
    if (gone < (n_live + 3u) / 4u) return false;
    __syncthreads();
    if (t == 0) s_out = 0;
    __syncthreads();
#pragma unroll 1
    for (uint32_t cb = (uint32_t)w * 32 * kQT; cb < n_live; cb += kW * 32 * kQT) {
        uint32_t ids[kQT], keys[kQT], fls[kQT], tot = 0;
#pragma unroll
        for (int q = 0; q < kQT; q++) {
            const uint32_t qi = cb + q * 32 + lane;
            const bool v = qi < n_live;
            ids[q] = v ? __ldcg(&gid[qi]) : kGone;
            keys[q] = v ? __ldcg(&gkp[qi]) : kGone;
            fls[q] = v ? L.gfl[qi] : (uint32_t)kFlNone;
        }
#pragma unroll
        for (int q = 0; q < kQT; q++) tot += __popc(__ballot_sync(0xffffffffu, ids[q] != kGone));
        uint32_t ob = 0;
        if (lane == 0 && tot) ob = atomicAdd(&s_out, tot);
        ob = __shfl_sync(0xffffffffu, ob, 0);
#pragma unroll
        for (int q = 0; q < kQT; q++) {
            const uint32_t b = __ballot_sync(0xffffffffu, ids[q] != kGone);
            if (ids[q] != kGone) {
                const uint32_t o = ob + __popc(b & lt);
                L.gid2[o] = ids[q];
                L.gkp2[o] = keys[q];
                L.gfl2[o] = (uint8_t)fls[q];
            }
            ob += __popc(b);
        }
    }
    __syncthreads();
    n_live = s_out;
    gone = 0;
    return true;
}

// (No bound on the CTAs per SM: k_peel<128> takes 255 registers, so an SM holds one, the others
// 128 and two.  Bounded to 128 it spills no more than they do and yet loses 8 us an epoch: 300000 x
// 128 2.85 -> 3.36 ms.  Whoever runs peels side by side sizes their grids by
// peel_least_ctas_per_sm.)
template <int D>
__global__ void __launch_bounds__(kThreads) k_peel(PeelArgs a)
{
    // dynamic shared memory: [scratch: phase A's histogram | selection scratch + staged
    // band entries] [keys by list position | ids by list position] (the latter when kc)
    extern __shared__ __align__(16) uint32_t dyn[];
    uint32_t *scr = dyn;
    uint32_t *skey = dyn + kScrWords;
    uint32_t *sid = skey + kKeyCache;
    uint8_t *sfl = reinterpret_cast<uint8_t *>(sid + kKeyCache);     // state bytes by list position (kc)
    __shared__ float Ls[D > 0 ? D : kMaxD];
    __shared__ uint32_t s_b[kMaxEpoch], s_r[kMaxEpoch], s_slot[kMaxEpoch], s_sbin[kMaxEpoch];
    __shared__ GroupTab s_tab;
    __shared__ uint32_t s_kcm, s_nl, s_klast, s_off[kMaxEpoch + 1], s_cert[kMaxEpoch];
    __shared__ uint16_t s_lost[D > 0 ? D : kMaxD];
    __shared__ uint32_t s_cc[kMaxEpoch], s_gc[kMaxEpoch];
    __shared__ uint32_t s_nslot, s_hold_end;
    __shared__ __align__(4) uint8_t s_map[kHistBins];
    // the previous epoch's landmark; the attributes whose landmark value is new (mask) and,
    // for an update of the keys, those attributes with their old and new values
    __shared__ float Lold[D > 0 ? D : kMaxD];
    __shared__ uint32_t s_jm[kMaxD / 32];
    __shared__ int s_ij[kIncMax];
    __shared__ float s_io[kIncMax], s_il[kIncMax];
    __shared__ uint32_t s_nj;
    __shared__ int s_inc;
    __shared__ float s_keps, s_kabs;
    __shared__ DigitMap s_dm;
    PeelCtl *ctl = a.ctl;
    const int d = a.d;
    const uint32_t n = (uint32_t)a.n, N = (uint32_t)a.N;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const unsigned G = gridDim.x, c = blockIdx.x;
    const unsigned lim = a.spin;
    const uint32_t s0 = (uint32_t)((uint64_t)c * n / G);
    const uint32_t s1 = (uint32_t)((uint64_t)(c + 1) * n / G);
    uint32_t n_live = s1 - s0;           // its list's length: the points of the slice left
    uint32_t gone = 0;                   // and (not kc) the gaps among them
    const bool kc = s1 - s0 <= (uint32_t)kKeyCache;   // the list and its keys stay in shared memory
    // slices beyond the key cache alternate between two lists in global memory
    uint32_t *gid = a.lidx + s0, *gid2 = a.lidx + n + s0;
    uint32_t *gkp = a.kpos + s0, *gkp2 = a.kpos + n + s0;
    uint8_t *gfl = a.pflag + s0, *gfl2 = a.pflag + n + s0;
    uint8_t *pfl = kc ? sfl : gfl;                      // the slice's state bytes by list position
    unsigned gen = 0;
    // ---- before the first epoch: the control block (but for its first words, cleared by the
    // host) and the slice's state; then the points by attribute where the launch makes them
    {
        uint32_t *cw = &ctl->h0[0];
        constexpr uint32_t words = (uint32_t)(offsetof(PeelCtl, Lbits) - offsetof(PeelCtl, h0)) / 4u;
#pragma unroll 1
        for (uint32_t b = c * kThreads + t; b < words; b += G * kThreads) cw[b] = 0;
#pragma unroll 1
        for (uint32_t j = c * kThreads + t; j < (uint32_t)kMaxD; j += G * kThreads) {
            ctl->Lbits[0][j] = 0u;
            ctl->Lbits[1][j] = kInfBits;
        }
#pragma unroll 1
        for (uint32_t q = t; q < s1 - s0; q += kThreads) {
            a.rnd[s0 + q] = kNone;
            pfl[q] = kFlNone;
            if (kc) sid[q] = s0 + q;
            else gid[q] = s0 + q;
        }
    }
    if (!grid_sync(ctl, a.flags, gen, lim, a.stall)) return;
    if (a.transpose) transpose_tiles(a.x, a.n, d, a.xt_out, reinterpret_cast<float(*)[33]>(scr));
    if (!grid_sync(ctl, a.flags, gen, lim)) return;
    bool first = true;           // the first epoch
    bool need_keys = true;       // the landmark changed: the keys must be computed
    uint32_t r0 = 0;             // the epoch's first round
    int lpar = 0, hpar = 0;      // the landmark's and the holder counts' current arrays
    // the keys' error bound |delta32 - delta64| <= k_eps delta32 + k_abs (thread 0 keeps it,
    // the same in every CTA) and the key updates since the last full pass
    const float eps_cap = (float)(d + 4) * 0x1p-23f, eps0 = (float)key_roundings<D>(d) * 0x1p-23f;
    float k_eps = eps0, k_abs = 0x1p-120f;
    for (;;) {
        const uint32_t nl_tot = n - r0 * N;
        auto LID = [&](uint32_t q) -> uint32_t { return kc ? sid[q] : __ldcg(&gid[q]); };
        auto LKEY = [&](uint32_t q) -> uint32_t { return kc ? skey[q] : __ldcg(&gkp[q]); };
        const ListView LV{kc, sid, skey, sfl, gid, gkp, gfl, gid2, gkp2, gfl2};
        // the landmark and the holder counts alternate between two arrays, so that no CTA
        // overwrites what a slower one still reads
        const uint32_t *Lcur = ctl->Lbits[lpar];
        uint32_t *chold = ctl->chold[hpar];
        uint32_t (*hcnt)[kMaxEpoch] = ctl->hcnt[hpar];
        const uint32_t e_kmax = __ldcg(&ctl->kmax);
#pragma unroll 1
        for (int j = t; j < d; j += kThreads) {
            Lold[j] = Ls[j];
            Ls[j] = __uint_as_float(__ldcg(&Lcur[j]));
        }
        __syncthreads();
        if (nl_tot <= N) {                            // the last subcluster: all that is left
#pragma unroll 1
            for (uint32_t q = t; q < n_live; q += kThreads) {
                const uint32_t id = LID(q);
                if (id != kGone) a.rnd[id] = r0;
            }
            if (c == 0 && a.landmarks)
#pragma unroll 1
                for (int j = t; j < d; j += kThreads) a.landmarks[(size_t)r0 * d + j] = Ls[j];
            break;
        }
        uint32_t Kb = min(a.kmax, (nl_tot + N - 1) / N - 1u);   // boundaries the epoch resolves, at most

        // ---- A: float32 distances of the points left, the first histogram, the holders
        if (need_keys) {
            // the attributes whose landmark value is new (all of them at first)
#pragma unroll 1
            for (int j0 = w * 32; j0 < d; j0 += kW * 32) {
                const int j = j0 + lane;
                const bool mv = j < d && (first || __float_as_uint(Ls[j]) != __float_as_uint(Lold[j]));
                const uint32_t m = __ballot_sync(0xffffffffu, mv);
                if (lane == 0) s_jm[j0 >> 5] = m;
            }
#pragma unroll 1
            for (int b = t; b < kHistBins; b += kThreads) scr[b] = 0;
            __syncthreads();
            if (t == 0) {
                // an update of the keys, or a full pass (the same choice in every CTA)
                // (float32 rounded up throughout: a float64 chain here held up every CTA; cs: the
                // moves of all attributes, for the keys' range.  Those of the first kIncMax alone left
                // keys below it, in one coarse bin, and a band of 10^5 points: 6 10^6 x 128 of 8
                // blobs 75 -> 22 ms of peel)
                uint32_t nj = 0, nsec = 0, last_sec = kGone;
                float cs = 0.0f;
                bool fin = true;
                for (int wd = 0; wd < (d + 31) / 32; wd++) {
                    uint32_t m = s_jm[wd];
                    while (m) {
                        const int j = wd * 32 + __ffs(m) - 1;
                        m &= m - 1u;
                        const float c = __fsub_rn(Ls[j], Lold[j]);
                        fin = fin && c >= 0.0f && c <= 1.0f;
                        cs = __fadd_ru(cs, c);
                        if (nj < (uint32_t)kIncMax) {
                            s_ij[nj] = j;
                            s_io[nj] = Lold[j];
                            s_il[nj] = Ls[j];
                        }
                        nj++;
                        if ((uint32_t)(j >> 3) != last_sec) {
                            nsec++;
                            last_sec = (uint32_t)(j >> 3);
                        }
                    }
                }
                cs = __fmul_ru(cs, 1.0f + 0x1p-20f);
                const float ne = __fadd_ru(k_eps, 0x1p-23f);
                const float na = __fadd_ru(
                    k_abs, __fmul_ru(__fadd_ru(__fmul_ru(5.0f, k_eps), (16.0f + 4.0f * (float)nj) * 0x1p-24f), cs));
                // the absolute term stays below an eighth of the relative one at the last
                // epoch's first boundary, so the bands widen little
                const bool inc = !first && fin && nj >= 1 && nj <= (uint32_t)kIncMax && nsec * 160u < 12u * (uint32_t)d &&
                                 ne <= 1.5f * eps_cap && na <= 0.125f * eps_cap * s_tab.kref;
                if (inc) {
                    k_eps = ne;
                    k_abs = na;
                } else {
                    k_eps = eps0;
                    k_abs = 0x1p-120f;
                }
                s_nj = inc ? nj : 0u;
                s_inc = inc ? 1 : 0;
                if (inc && c == 0) ctl->key_updates += 1;
                s_keps = k_eps;
                s_kabs = k_abs;
                // the range of the new keys: none was below klast, the landmark's move takes
                // at most 2 cs off a distance (c (2 x - l - o) <= 2 c per attribute, x <= 1) and
                // adds nothing (x >= l for every point left), so none is above the first
                // epoch's largest; a margin of 2^-12 for the roundings
                if (!first) {
                    const float lo = __uint_as_float(s_klast) * (1.0f - 0x1p-12f) - cs * (2.0f + 0x1p-12f);
                    s_dm = digit_map(lo > 0.0f ? __float_as_uint(lo) : 0u, e_kmax + 4096u);
                }
            }
            __syncthreads();
            if (s_inc && kc)
                phase_inc<D, kLoadKc>(a.x, a.xt, n, d, n_live, kc, sid, gid, skey, gkp, scr, &s_dm, pfl, chold, s_nj,
                                      s_ij, s_io, s_il);
            else if (s_inc)
                phase_inc<D, kLoadGlobal>(a.x, a.xt, n, d, n_live, kc, sid, gid, skey, gkp, scr, &s_dm, pfl, chold, s_nj,
                                          s_ij, s_io, s_il);
            else
                phase_keys<D>(a.x, Ls, d, n_live, s0, first, kc, sid, gid, skey, gkp, scr, &s_dm, pfl, chold, s_jm);
            __syncthreads();
            if (first) {
                // the first epoch's bins, from its own keys
                uint32_t mn = kGone, mx = 0;
#pragma unroll 4
                for (uint32_t q = t; q < n_live; q += kThreads) {
                    const uint32_t k = LKEY(q);
                    mn = min(mn, k);
                    mx = max(mx, k);
                }
                mn = __reduce_min_sync(0xffffffffu, mn);
                mx = __reduce_max_sync(0xffffffffu, mx);
                if (lane == 0 && n_live) {
                    atomicMax(&ctl->kmin, ~mn);
                    atomicMax(&ctl->kmax, mx);
                }
                if (!grid_sync(ctl, a.flags, gen, lim)) return;
                if (t == 0) s_dm = digit_map(~__ldcg(&ctl->kmin), __ldcg(&ctl->kmax) + 4096u);
                __syncthreads();
#pragma unroll 4
                for (uint32_t q = t; q < n_live; q += kThreads) atomicAdd(&scr[s_dm.bin(LKEY(q))], 1u);
                __syncthreads();
            }
            // each attribute's largest holder key (the holders are the flagged points left)
#pragma unroll 1
            for (uint32_t q0 = 0; q0 < n_live; q0 += kHoldBatch * kThreads) {
                uint32_t held = 0;
#pragma unroll
                for (int u = 0; u < kHoldBatch; u++) {
                    const uint32_t qi = q0 + u * kThreads + t;
                    held |= (uint32_t)(qi < n_live && (pfl[qi] & kFlHold)) << u;
                }
                uint32_t todo = __reduce_or_sync(0xffffffffu, held);
#pragma unroll 1
                while (todo) {
                    const int u = __ffs(todo) - 1;
                    todo &= todo - 1u;
                    const bool h = (held >> u) & 1u;
                    const uint32_t qi = q0 + u * kThreads + t;
                    max_held(a.x, Ls, d, h, h ? LID(qi) : 0u, h ? LKEY(qi) : 0u, ctl->hmax);
                }
            }
#pragma unroll 1
            for (int b = t; b < kHistBins; b += kThreads)
                if (scr[b]) atomicAdd(&ctl->h0[b], scr[b]);
            if (!grid_sync(ctl, a.flags, gen, lim)) return;
        }

        // ---- B: each boundary's first-digit bin (every CTA), then second-digit histograms
        {
            constexpr int per = kHistBins / kThreads;       // 8 bins per thread
            uint32_t l0[per];
            const uint4 *p = reinterpret_cast<const uint4 *>(ctl->h0 + t * per);
            const uint4 u = __ldcg(p), v = __ldcg(p + 1);
            l0[0] = u.x; l0[1] = u.y; l0[2] = u.z; l0[3] = u.w;
            l0[4] = v.x; l0[5] = v.y; l0[6] = v.z; l0[7] = v.w;
            uint32_t s = 0;
#pragma unroll
            for (int q = 0; q < per; q++) s += l0[q];
            uint32_t m = kGone;
#pragma unroll 1
            for (int j = t; j < d; j += kThreads) m = min(m, __ldcg(&ctl->hmax[j]));
            uint32_t tot;
            const uint32_t e0 = block_excl_scan(s, tot);
            // the rounds this landmark can serve: up to the one in which the last holder of
            // some attribute's landmark value leaves (the landmark changes after it).  That
            // holder's key m (the smallest over the attributes of their holders' largest key)
            // is at most the c-th smallest live key, c the points up to the end of m's bin, so
            // it leaves at the latest in round (c - 1) / N; the boundaries past that round are
            // not resolved (a prediction that falls short costs one more epoch)
            m = block_min(m);
            {
                const uint32_t mb = s_dm.bin(m);
                if ((uint32_t)t == mb / per) {
                    uint32_t cc = e0;
#pragma unroll
                    for (int i = 0; i < per; i++)
                        if ((uint32_t)i <= mb % per) cc += l0[i];
                    s_hold_end = cc;
                }
            }
            __syncthreads();
            Kb = min(Kb, (s_hold_end > 0u ? (s_hold_end - 1u) / N : 0u) + 1u);
            // boundary q's rank is (q + 1) N - 1: the boundaries inside this thread's bins
            for (uint32_t q = e0 / N; q < Kb && (q + 1) * N - 1u < e0 + s; q++) {
                const uint32_t target = (q + 1) * N - 1u;
                uint32_t cc = e0;
#pragma unroll
                for (int i = 0; i < per; i++) {
                    if (target >= cc && target < cc + l0[i]) {
                        s_b[q] = (uint32_t)(t * per + i);
                        s_r[q] = target - cc;
                    }
                    cc += l0[i];
                }
            }
#pragma unroll 1
            for (int b = t; b < kHistBins / 4; b += kThreads) reinterpret_cast<uint32_t *>(s_map)[b] = 0xFFFFFFFFu;
            __syncthreads();
            if (w == 0) {
                const bool v = lane < (int)Kb;
                const uint32_t b = v ? s_b[lane] : 0u;
                const uint32_t pb = __shfl_up_sync(0xffffffffu, b, 1);
                const uint32_t open = __ballot_sync(0xffffffffu, v && (lane == 0 || b != pb));
                if (v) {
                    const uint32_t sl = (uint32_t)__popc(open & ((2u << lane) - 1u)) - 1u;
                    s_slot[lane] = sl;
                    if ((open >> lane) & 1u) {
                        s_sbin[sl] = b;
                        s_map[b] = (uint8_t)sl;
                    }
                }
                if (lane == 0) {
                    s_nslot = (uint32_t)__popc(open);
                    if (tot != nl_tot) atomicOr(&a.flags[1], 1u);
                }
            }
            __syncthreads();
            // the keys in those bins, straight to the grid's histograms: few of them, but one
            // atomic per warp for the equal ones (tied data crowds them into one)
            const DigitMap mp = s_dm;
#pragma unroll 1
            for (uint32_t q0 = t - lane; q0 < n_live; q0 += 4 * kThreads) {       // warp-uniform bound
                uint32_t k4[4];
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    const uint32_t qi = q0 + lane + q * kThreads;
                    k4[q] = qi < n_live ? LKEY(qi) : kGone;
                }
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    const uint32_t b = mp.bin(k4[q]);
                    const uint32_t sl = k4[q] == kGone ? 0xFFu : s_map[b];
                    const uint32_t hit = __ballot_sync(0xffffffffu, sl != 0xFFu);
                    if (!hit) continue;
                    const uint32_t at = sl != 0xFFu ? sl * kHistBins + mp.sub(k4[q], b) : kGone;
                    const uint32_t peers = __match_any_sync(0xffffffffu, at);
                    if (at != kGone && lane == __ffs(peers) - 1)
                        atomicAdd(&ctl->h1[0][0] + at, (uint32_t)__popc(peers));
                }
            }
        }
        // each boundary's bins become its band cut-offs, and boundaries whose bands overlap
        // merge into groups
        const uint32_t K = Kb;                        // boundaries of the epoch
        if (K <= kAllResolve) {
            if (!grid_sync(ctl, a.flags, gen, lim)) return;
            resolve_cutoffs(ctl, K, s_keps, s_kabs, &s_dm, s_b, s_r, s_slot, s_tab);
        } else {
            if (!grid_sync_last(ctl, a.flags, gen, lim, [&]() {
                    resolve_cutoffs(ctl, K, s_keps, s_kabs, &s_dm, s_b, s_r, s_slot, s_tab);
#pragma unroll 1
                    for (uint32_t e = t; e < sizeof(GroupTab) / 4u; e += kThreads)
                        ctl->tab[e] = reinterpret_cast<const uint32_t *>(&s_tab)[e];
                }))
                return;
#pragma unroll 1
            for (uint32_t e = t; e < sizeof(GroupTab) / 4u; e += kThreads)
                reinterpret_cast<uint32_t *>(&s_tab)[e] = __ldcg(&ctl->tab[e]);
            __syncthreads();
        }

        // ---- C: classify every point left: certainly in a round of the epoch, in a band, or later
        const uint32_t ng = s_tab.ng;
        if (t < kMaxEpoch) {
            s_cc[t] = 0;
            s_gc[t] = 0;
        }
        __syncthreads();
        const uint32_t n_hit = classify_live(a, LV, n_live, Ls, r0, K, s_tab, s_cc, s_gc, hcnt, scr);
        if (t < (int)K && s_cc[t]) atomicAdd(&ctl->cert[t], s_cc[t]);
        if (t < (int)ng && s_gc[t]) atomicAdd(&ctl->gcnt[t], s_gc[t]);
        if (!grid_sync(ctl, a.flags, gen, lim)) return;

        // ---- D: the band entries regrouped by group with their compensated distances
        // (across the grid), then each group's band settled (CTA c takes groups c, c + G, ...)
        {
            const uint32_t nlist = __ldcg(&ctl->band_cnt);
            // each group's region in gkey / gpos, and the certain points up to each round
            if (t < 32) {
                const uint32_t v = __ldcg(&ctl->gcnt[t]), cv = __ldcg(&ctl->cert[t]);
                s_off[t + 1] = warp_incl_scan(v);
                s_cert[t] = warp_incl_scan(cv);
                if (t == 0) s_off[0] = 0;
            }
            __syncthreads();
            // one slot claim per warp and group: the entries of a pass crowd into a few
            // groups, whose fill counters would otherwise take one contended atomic each
            // (8 lanes per entry from 32 attributes on: a thread's chain over 128 took 15 us)
            if (d >= 32) {
                constexpr uint32_t EB = kThreads / 8;
#pragma unroll 1
                for (uint32_t b0 = c * EB; b0 < nlist; b0 += G * EB) {               // block-uniform bound
                    const uint32_t e = b0 + (uint32_t)t / 8u, sub = (uint32_t)t & 7u;
                    const bool v = e < nlist;
                    const uint32_t k = v ? __ldcg(&a.band_k32[e]) : 0u;
                    const uint32_t pos = v ? __ldcg(&a.band_pos[e]) : 0u;
                    uint32_t g = 0;
                    while (g + 1 < ng && k > s_tab.out[g]) g++;
                    const uint32_t peers = __match_any_sync(0xffffffffu, v && sub == 0u ? g : kGone);
                    const uint32_t leader = (uint32_t)__ffs(peers) - 1u;
                    uint32_t slot = 0;
                    if (v && sub == 0u && (uint32_t)lane == leader) slot = atomicAdd(&ctl->gfill[g], (uint32_t)__popc(peers));
                    float h, l;
                    dist_ff8(a.x + (size_t)(pos & kPosMask) * d, Ls, d, (int)sub, h, l);
                    slot = __shfl_sync(0xffffffffu, slot, (int)leader) + (uint32_t)__popc(peers & ((1u << lane) - 1u));
                    if (v && sub == 0u) {
                        a.gkey[s_off[g] + slot] = ff_key(h, l);
                        a.gpos[s_off[g] + slot] = pos;
                    }
                }
            } else for (uint32_t b0 = c * kThreads; b0 < nlist; b0 += G * kThreads) {     // warp-uniform bound
                const uint32_t e = b0 + (uint32_t)t;
                const bool v = e < nlist;
                const uint32_t k = v ? __ldcg(&a.band_k32[e]) : 0u;
                const uint32_t pos = v ? __ldcg(&a.band_pos[e]) : 0u;
                uint32_t g = 0;
                while (g + 1 < ng && k > s_tab.out[g]) g++;
                const uint32_t lane = (uint32_t)t & 31u;
                const uint32_t peers = __match_any_sync(0xffffffffu, v ? g : 0xFFFFFFFFu);
                const uint32_t leader = (uint32_t)__ffs(peers) - 1u;
                uint32_t slot = 0;
                if (v && lane == leader) slot = atomicAdd(&ctl->gfill[g], (uint32_t)__popc(peers));
                const uint64_t key = v ? dff_key(a.x + (size_t)(pos & kPosMask) * d, Ls, d) : 0ull;
                slot = __shfl_sync(0xffffffffu, slot, (int)leader) + (uint32_t)__popc(peers & ((1u << lane) - 1u));
                if (v) {
                    a.gkey[s_off[g] + slot] = key;
                    a.gpos[s_off[g] + slot] = pos;
                }
            }
            if (!grid_sync(ctl, a.flags, gen, lim)) return;
#pragma unroll 1
            for (uint32_t g = c; g < ng; g += G) {
                const uint32_t q1 = g ? s_tab.q2[g - 1] + 1u : 0u;
                settle_group(a, Ls, g, q1, s_tab.q2[g], s_off[g], s_off[g + 1] - s_off[g], s_cert[q1], r0, K, hcnt, scr,
                             kc ? 0u : (uint32_t)kStage);
            }
        }
        // how many rounds the epoch commits: up to the first round after which some attribute
        // has no holder of its landmark value left
        if (!grid_sync(ctl, a.flags, gen, lim)) return;
        commit_count(a, K, s_tab, chold, ctl->chold[hpar ^ 1], hcnt, s_kcm, s_nl, s_klast, s_lost);

        // ---- E: commit: the epoch's first kcm rounds leave the lists; the other
        // assignments are dropped; the next landmark if it changes
        const uint32_t n_lost = s_nl;
        uint32_t kcm = s_kcm;
        if (kcm < 1u || kcm > K) {                    // cannot happen; keeps the loop finite
            if (c == 0 && t == 0) atomicOr(&a.flags[1], 1u);
            kcm = 1u;
        }
        const bool changed = n_lost != 0u;
        if (c == 0 && t == 0) {
            ctl->epochs += 1;
            ctl->passes += need_keys ? 1u : 0u;
        }
        const uint32_t live_from = r0 + kcm;
        if (kc) {
            n_live = compact_shared(a, LV, n_live, r0, live_from, changed, &s_dm, scr);
        } else if (commit_global(a, LV, n_live, gone, n_hit, r0, live_from, changed, &s_dm, scr)) {
            uint32_t *ti = gid; gid = gid2; gid2 = ti;
            uint32_t *tk = gkp; gkp = gkp2; gkp2 = tk;
            uint8_t *tf = gfl; gfl = gfl2; gfl2 = tf;
            pfl = gfl;
        }
        // the epoch's scratch, cleared across the grid for the next one
        {
            if (changed) {                            // recomputed by the next pass
#pragma unroll 1
                for (uint32_t b = c * kThreads + t; b < (uint32_t)kHistBins; b += G * kThreads) ctl->h0[b] = 0;
                // the next landmark: the attributes that keep theirs here, the others' minima
                // below; this one's array becomes the one after's
                uint32_t *Lnext = ctl->Lbits[lpar ^ 1];
#pragma unroll 1
                for (uint32_t j = c * kThreads + t; j < (uint32_t)d; j += G * kThreads) {
                    ctl->hmax[j] = 0;
                    ctl->Lbits[lpar][j] = kInfBits;
                    bool keep = true;
                    for (uint32_t e = 0; e < n_lost; e++) keep = keep && s_lost[e] != (uint16_t)j;
                    if (keep) Lnext[j] = __float_as_uint(Ls[j]);
                }
            }
            if (a.landmarks)
#pragma unroll 1
                for (uint32_t e = c * kThreads + t; e < kcm * (uint32_t)d; e += G * kThreads)
                    a.landmarks[(size_t)(r0 + e / d) * d + e % d] = Ls[e % d];
            uint32_t *h1 = &ctl->h1[0][0];
#pragma unroll 1
            for (uint32_t b = c * kThreads + t; b < s_nslot * (uint32_t)kHistBins; b += G * kThreads) h1[b] = 0;
            uint32_t *hc = &ctl->hcnt[hpar ^ 1][0][0];        // the next epoch's
#pragma unroll 1
            for (uint32_t b = c * kThreads + t; b < (uint32_t)d * kMaxEpoch; b += G * kThreads) hc[b] = 0;
            if (c == 0 && t < kMaxEpoch) {
                ctl->cert[t] = 0;
                ctl->bnd[t] = 0;
                ctl->gcnt[t] = 0;
                ctl->gfill[t] = 0;
            }
            if (c == 0 && t == 0) ctl->band_cnt = 0;
        }
        if (changed && n_live && n_lost >= (uint32_t)kMinMany)
            many_minima(a.x, a.xt, n, d, n_live, kc, sid, gid, s_lost, n_lost, ctl->Lbits[lpar ^ 1]);
        else if (changed && n_live && kc)
            lost_minima<kLoadKc>(a.x, a.xt, n, d, n_live, kc, sid, gid, s_lost, n_lost, ctl->Lbits[lpar ^ 1]);
        else if (changed && n_live)
            lost_minima<kLoadGlobal>(a.x, a.xt, n, d, n_live, kc, sid, gid, s_lost, n_lost, ctl->Lbits[lpar ^ 1]);
        first = false;
        hpar ^= 1;
        if (changed) lpar ^= 1;
        need_keys = changed;
        r0 += kcm;
        if (!grid_sync(ctl, a.flags, gen, lim)) return;
    }
}

// ------------------------------------------------------------------ barrier cost
// The peel's grid barrier alone: `rounds` barriers in a row, in the peel's launch shape
// (the same block size, dynamic shared memory and CTAs per SM, so the same grid), timed
// to give the latency floor that the peel's barriers put under its epochs.
__global__ void __launch_bounds__(kThreads) k_barrier_bench(PeelCtl *ctl, uint32_t *flags, int rounds, unsigned lim)
{
    extern __shared__ __align__(16) uint32_t dyn[];
    if (threadIdx.x == 0 && rounds < 0) dyn[0] = 0;          // keeps the launch's shared memory
    unsigned gen = 0;
    for (int r = 0; r < rounds; r++)
        if (!grid_sync(ctl, flags, gen, lim)) return;
}

// ------------------------------------------------------------------ packing by round
// Stable counting sort of the points by round (8 bits of it per pass): the subclusters,
// each in ascending point index.  Chunk c of the items is [c m/G, (c+1) m/G).
constexpr int kPermThreads = kThreads;        // 256, a digit's values: block_excl_scan's block
static_assert(kPermThreads == 256, "a thread per digit value");

__global__ void __launch_bounds__(kPermThreads) k_perm_count(const uint32_t *__restrict__ rnd,
                                                             const uint32_t *__restrict__ src, uint32_t m, int sh,
                                                             uint32_t *__restrict__ cnt)
{
    __shared__ uint32_t h[256];
    const int t = threadIdx.x;
    const uint32_t G = gridDim.x, c = blockIdx.x;
    h[t] = 0;
    __syncthreads();
    const uint32_t lo = (uint32_t)((uint64_t)c * m / G), hi = (uint32_t)((uint64_t)(c + 1) * m / G);
    for (uint32_t i = lo + t; i < hi; i += kPermThreads) {
        const uint32_t id = src ? __ldg(&src[i]) : i;
        atomicAdd(&h[(__ldg(&rnd[id]) >> sh) & 255u], 1u);
    }
    __syncthreads();
    cnt[(size_t)t * G + c] = h[t];
}

// Inclusive scan of each digit's G counts over the chunks, in place: a block per digit, whose
// last value is the digit's total (the scatter adds the digits before).  One block for all 256 G
// was a chain of L2 round trips (2^20 points: 59 us).
__global__ void __launch_bounds__(kPermThreads) k_perm_scan(uint32_t *cnt, uint32_t G)
{
    uint32_t *c = cnt + (size_t)blockIdx.x * G;
    uint32_t run = 0;
    for (uint32_t b = 0; b < G; b += 4 * kPermThreads) {
        uint32_t v[4], s = 0, tot;
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const uint32_t e = b + 4 * threadIdx.x + q;
            v[q] = e < G ? c[e] : 0u;
            s += v[q];
        }
        uint32_t at = run + block_excl_scan(s, tot);
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const uint32_t e = b + 4 * threadIdx.x + q;
            at += v[q];
            if (e < G) c[e] = at;
        }
        run += tot;
    }
}

__global__ void __launch_bounds__(kPermThreads) k_perm_scatter(const uint32_t *__restrict__ rnd,
                                                               const uint32_t *__restrict__ src, uint32_t m, int sh,
                                                               const uint32_t *__restrict__ cnt,
                                                               uint32_t *__restrict__ dst)
{
    constexpr int W = kPermThreads / 32;
    __shared__ uint32_t base[256];
    __shared__ uint32_t wc[W][256];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const uint32_t G = gridDim.x, c = blockIdx.x;
    const uint32_t lt = (1u << lane) - 1u;
    {
        uint32_t all;
        const uint32_t before = block_excl_scan(__ldg(&cnt[(size_t)t * G + G - 1]), all);
        base[t] = before + (c ? __ldg(&cnt[(size_t)t * G + c - 1]) : 0u);
    }
    const uint32_t lo = (uint32_t)((uint64_t)c * m / G), hi = (uint32_t)((uint64_t)(c + 1) * m / G);
    for (uint32_t i0 = lo; i0 < hi; i0 += kPermThreads) {
        const uint32_t i = i0 + t;
        const bool valid = i < hi;
        const uint32_t id = valid ? (src ? __ldg(&src[i]) : i) : 0u;
        const uint32_t dg = valid ? (__ldg(&rnd[id]) >> sh) & 255u : 256u;
        for (int q = t; q < W * 256; q += kPermThreads) (&wc[0][0])[q] = 0;
        __syncthreads();
        const uint32_t peers = __match_any_sync(0xffffffffu, dg);
        if (valid && (peers & lt) == 0) wc[w][dg] = (uint32_t)__popc(peers);
        __syncthreads();
        if (valid) {
            uint32_t o = base[dg] + (uint32_t)__popc(peers & lt);
            for (int v = 0; v < w; v++) o += wc[v][dg];
            dst[o] = id;
        }
        __syncthreads();
        uint32_t add = 0;
#pragma unroll
        for (int v = 0; v < W; v++) add += wc[v][t];
        base[t] += add;
        __syncthreads();
    }
}

template <bool kVec4>
__global__ void k_gather_rows(const float *__restrict__ x, const uint32_t *__restrict__ perm,
                              int64_t n, int d, float *__restrict__ out)
{
    if (kVec4) {
        const int d4 = d / 4;
        const float4 *x4 = reinterpret_cast<const float4 *>(x);
        float4 *o4 = reinterpret_cast<float4 *>(out);
        for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n * d4;
             e += (int64_t)gridDim.x * blockDim.x) {
            int64_t p = e / d4;
            int q = (int)(e - p * d4);
            o4[e] = __ldg(&x4[(int64_t)perm[p] * d4 + q]);
        }
    } else {
        for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n * d;
             e += (int64_t)gridDim.x * blockDim.x) {
            int64_t p = e / d;
            int q = (int)(e - p * d);
            out[e] = __ldg(&x[(int64_t)perm[p] * d + q]);
        }
    }
}

// k_peel<D>'s CTAs per SM, its shared memory allowed.
template <int D>
cudaError_t peel_occupancy(int *per_sm)
{
    const size_t smem = kPeelDynWords * sizeof(uint32_t);
    const cudaError_t e = cudaFuncSetAttribute(k_peel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, k_peel<D>, kThreads, smem);
}

template <int D>
cudaError_t peel_launch(const PeelBuffers &b, int64_t n, int d, int64_t N, int sm_count,
                        cudaStream_t st, KTimer *kt)
{
    const int64_t S = (n + N - 1) / N;
    // all control state starts cleared (the launch clears the rest); the first landmark is
    // the origin (the scaled minimum of every attribute is exactly 0)
    cudaError_t e = cudaMemsetAsync(b.ctl, 0, offsetof(PeelCtl, h0), st);
    if (e != cudaSuccess) return e;
    const size_t smem = kPeelDynWords * sizeof(uint32_t);
    int per_sm = 0;
    e = peel_occupancy<D>(&per_sm);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    int64_t grid = (int64_t)sm_count * std::min(per_sm, 4);
    if (grid > kMaxPeelGrid) grid = kMaxPeelGrid;
    // one CTA per SM while its slice holds few points: fewer arrivals at the barriers
    // (200003 x 7: 861 against 820 us, 400000 x 128: 6.8 against 6.5 ms), where 2^20 x 16, with
    // 6900 points per SM, wants two (3.0 against 2.6 ms)
    if (n <= (int64_t)sm_count * 3072 && grid > sm_count) grid = sm_count;
    const int64_t want = (n + 63) / 64;             // at least ~64 points per CTA
    if (grid > want) grid = std::max<int64_t>(1, want);
    if (b.max_grid > 0 && grid > b.max_grid) grid = b.max_grid;
    PeelArgs a;
    a.x = b.x;
    // the points by attribute for the landmark's minima and the key updates, in xseg (idle
    // until the subclusters are gathered after the launch): they then read 4 bytes of each
    // point left instead of a 32-byte sector of its row
    a.xt = d >= 4 ? b.xseg : nullptr;
    a.xt_out = b.xseg;
    a.transpose = a.xt && (size_t)n * d * sizeof(float) <= kTransposeBytes;
    a.d = d;
    a.n = n;
    a.N = N;
    a.S = S;
    a.rnd = b.rnd;
    a.pflag = b.pflag;
    a.lidx = b.lidx;
    a.kpos = b.kpos;
    a.band_k32 = b.band_k32;
    a.band_pos = b.band_pos;
    a.gkey = b.gkey;
    a.gpos = b.gpos;
    a.akey = b.akey;
    a.apos = b.apos;
    a.landmarks = b.landmarks;
    a.ctl = b.ctl;
    a.flags = b.flags;
    a.kmax = (uint32_t)(b.rounds_per_pass > 0 ? std::min(b.rounds_per_pass, kMaxEpoch) : kDefaultRounds);
    a.spin = b.wait_limit ? b.wait_limit : kDefaultSpin;
    a.stall = b.stall_first_barrier ? 1u : 0u;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    kt->begin(st);
    if (a.xt && !a.transpose) {  // timed and counted with the peel it serves
        transpose_launch(b.x, n, d, b.xseg, sm_count, st);
        kt->launches[PSCL_K_PEEL]++;
    }
    e = cudaLaunchKernelEx(&cfg, k_peel<D>, a);
    kt->end(PSCL_K_PEEL, st);
    if (e != cudaSuccess) return e;
    // the subclusters packed by round: a stable counting sort, 8 bits of the round per pass
    int passes = 1;
    while (passes < 4 && (S - 1) >> (8 * passes)) passes++;
    const int pg = perm_grid(n, sm_count);
    const uint32_t m = (uint32_t)n;
    const uint32_t *src = nullptr;
    for (int p = 0; p < passes; p++) {
        uint32_t *dst = ((passes - 1 - p) & 1) ? b.gpos : b.perm;
        kt->begin(st);
        k_perm_count<<<pg, kPermThreads, 0, st>>>(b.rnd, src, m, 8 * p, b.pcnt);
        k_perm_scan<<<256, kPermThreads, 0, st>>>(b.pcnt, (uint32_t)pg);
        k_perm_scatter<<<pg, kPermThreads, 0, st>>>(b.rnd, src, m, 8 * p, b.pcnt, dst);
        kt->end(PSCL_K_GATHER, st);
        src = dst;
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_gather(b.x, b.perm, n, d, b.xseg, sm_count, st, kt);
}

}  // namespace

cudaError_t launch_gather(const float *x, const uint32_t *perm, int64_t n, int d, float *xseg, int sm_count,
                          cudaStream_t st, KTimer *kt)
{
    int64_t work = (d % 4 == 0) ? n * d / 4 : n * d;
    int64_t g = (work + 255) / 256;
    if (g > (int64_t)sm_count * 16) g = (int64_t)sm_count * 16;
    if (g < 1) g = 1;
    kt->begin(st);
    if (d % 4 == 0)
        k_gather_rows<true><<<(int)g, 256, 0, st>>>(x, perm, n, d, xseg);
    else
        k_gather_rows<false><<<(int)g, 256, 0, st>>>(x, perm, n, d, xseg);
    kt->end(PSCL_K_GATHER, st);
    return cudaGetLastError();
}

cudaError_t measure_grid_barrier(int sm_count, double *us, bool *timed_out)
{
    const size_t smem = kPeelDynWords * sizeof(uint32_t);
    cudaError_t e = cudaFuncSetAttribute(k_barrier_bench, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    // the peel's grid at full size: its CTAs per SM (capped at 4), as peel_launch sizes it
    int per_sm = 0;
    e = peel_occupancy<16>(&per_sm);
    if (e != cudaSuccess) return e;
    int bench_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bench_sm, k_barrier_bench, kThreads, smem);
    if (e != cudaSuccess) return e;
    per_sm = std::min(std::min(per_sm, 4), bench_sm);
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    const int grid = std::min(sm_count * per_sm, kMaxPeelGrid);
    PeelCtl *ctl = nullptr;
    uint32_t *flags = nullptr;
    cudaStream_t st = nullptr;
    cudaEvent_t t0 = nullptr, t1 = nullptr;
    constexpr int kRounds = 2000;
    float best = 0.0f;
    uint32_t hf[2] = {0u, 0u};
    if ((e = cudaMalloc(&ctl, sizeof(PeelCtl))) == cudaSuccess && (e = cudaMalloc(&flags, 8)) == cudaSuccess &&
        (e = cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking)) == cudaSuccess &&
        (e = cudaEventCreate(&t0)) == cudaSuccess && (e = cudaEventCreate(&t1)) == cudaSuccess) {
        for (int r = 0; r < 4 && e == cudaSuccess; r++) {        // the first a warm-up
            cudaMemsetAsync(ctl, 0, sizeof(PeelCtl), st);
            cudaMemsetAsync(flags, 0, 8, st);
            int rounds = kRounds;
            unsigned lim = kDefaultSpin;
            void *args[] = {&ctl, &flags, &rounds, &lim};
            cudaEventRecord(t0, st);
            e = cudaLaunchCooperativeKernel((const void *)k_barrier_bench, dim3(grid), dim3(kThreads), args, smem, st);
            cudaEventRecord(t1, st);
            if (e == cudaSuccess) e = cudaEventSynchronize(t1);
            if (e == cudaSuccess) e = cudaMemcpy(hf, flags, 8, cudaMemcpyDeviceToHost);
            float ms = 0.0f;
            if (e == cudaSuccess) cudaEventElapsedTime(&ms, t0, t1);
            if (r > 0 && (best == 0.0f || ms < best)) best = ms;
            if (hf[1]) break;
        }
    }
    if (t0) cudaEventDestroy(t0);
    if (t1) cudaEventDestroy(t1);
    if (st) cudaStreamDestroy(st);
    cudaFree(flags);
    cudaFree(ctl);
    if (e != cudaSuccess) return e;
    *timed_out = hf[1] != 0u;
    *us = 1e3 * (double)best / kRounds;
    return cudaSuccess;
}

int perm_grid(int64_t n, int sm_count)
{
    int64_t g = (n + 2047) / 2048;
    if (g > (int64_t)sm_count * 4) g = (int64_t)sm_count * 4;
    return (int)std::max<int64_t>(1, g);
}

cudaError_t peel_ctas_per_sm(int d, int *per_sm)
{
    switch (d) {
    case 2: return peel_occupancy<2>(per_sm);
    case 4: return peel_occupancy<4>(per_sm);
    case 8: return peel_occupancy<8>(per_sm);
    case 16: return peel_occupancy<16>(per_sm);
    case 32: return peel_occupancy<32>(per_sm);
    case 64: return peel_occupancy<64>(per_sm);
    case 128: return peel_occupancy<128>(per_sm);
    default: return peel_occupancy<0>(per_sm);
    }
}

cudaError_t peel_least_ctas_per_sm(int *per_sm)
{
    int least = 0;
    for (int d : {0, 2, 4, 8, 16, 32, 64, 128}) {           // launch_peel's widths
        int v = 0;
        if (const cudaError_t e = peel_ctas_per_sm(d, &v)) return e;
        least = d == 0 ? v : std::min(least, v);
    }
    *per_sm = least;
    return cudaSuccess;
}

cudaError_t launch_peel(const PeelBuffers &b, int64_t n, int d, int64_t N, int sm_count,
                        cudaStream_t st, KTimer *kt)
{
    switch (d) {
    case 2: return peel_launch<2>(b, n, d, N, sm_count, st, kt);
    case 4: return peel_launch<4>(b, n, d, N, sm_count, st, kt);
    case 8: return peel_launch<8>(b, n, d, N, sm_count, st, kt);
    case 16: return peel_launch<16>(b, n, d, N, sm_count, st, kt);
    case 32: return peel_launch<32>(b, n, d, N, sm_count, st, kt);
    case 64: return peel_launch<64>(b, n, d, N, sm_count, st, kt);
    case 128: return peel_launch<128>(b, n, d, N, sm_count, st, kt);
    default: return peel_launch<0>(b, n, d, N, sm_count, st, kt);
    }
}

}  // namespace pscl
