// Lloyd's k-means (§I) on many point sets at once: every subcluster of Algorithm 1
// step 4, and the pooled local centers of §V.
//
// Layout: the points of all sets are packed row-major one set after another (the
// paper's "flattening while subgrouping", §V); set s has seg_size[s] rows starting at
// seg_start[s] and k_eff[s] centers starting at cen_off[s] in one P x d center array.
// Work is cut into units of at most a few thousand rows of one set, so a launch keeps
// every SM busy whatever the mix of set sizes.
//
// One iteration = k_lloyd_assign (nearest center of every row, lowest index on ties,
// and the row's coordinates added to its center's sum) + k_lloyd_finalize (center =
// sum / count; an empty cluster keeps its center).  The sums are exact: coordinates
// (scaled to [0, 1]) are rounded once to 32.32 fixed point and added as 64-bit
// integers, first in shared memory, then with one global atomic per (center,
// attribute) and unit.  Integer addition is associative, so the result does not depend
// on how units are scheduled or batched with other work.
#include <algorithm>

#include "pscl_internal.cuh"
#include "sse.cuh"

namespace pscl {
namespace {

constexpr int kThreads = 256;
static_assert(kThreads == kSseThreads, "the SSE kernels' blocks");
constexpr float kFix = 4294967296.0f;                  // 2^32
constexpr size_t kSmemAccMax = 96 * 1024;              // shared accumulators up to this size
constexpr int kCenterChunkBytes = 48 * 1024;           // center chunk held in shared memory

// ---------------------------------------------------------------- SplitMix64
// Steele, Lea & Flood (OOPSLA 2014): the state advances by the golden-ratio constant
// and each output is the variant-13 mix of the state.
__device__ __forceinline__ uint64_t sm64_next(uint64_t &s)
{
    s += 0x9E3779B97F4A7C15ULL;
    uint64_t z = s;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}

// Initial centers of set s: the first k positions of a Fisher-Yates shuffle of its m
// rows (step i swaps i with j_i = i + r_i mod (m - i)), the stream keyed by (seed, stage, s):
// r_i is the mix of the key plus (i + 1) golden ratios, so every step's draw and its 64-bit
// remainder are formed in parallel.  What the shuffle leaves at position i is what position
// j_i held before step i: the row j_i itself, unless an earlier step t with j_t = j_i put
// there what position t held before step t, and so on.  A thread follows that chain back; the
// steps are found by their j in hash chains.  (One thread walking the steps in order, a
// remainder and two dependent look-ups each, took 109 us for k = 500.)
__global__ void k_lloyd_init(const float *__restrict__ pts, SegTable t, int d, float *centers,
                             unsigned long long *acc, int32_t *count2, int64_t P,
                             uint64_t seed, uint32_t stage, int first_k)
{
    extern __shared__ int32_t sh[];
    for (int s = blockIdx.x; s < t.n_seg; s += gridDim.x) {
        const int k = t.k_eff[s];
        const int32_t m = t.seg_size[s];
        int cap = 1;
        while (cap < k) cap <<= 1;
        int32_t *A = sh;                       // k: the rows picked
        int32_t *jt = sh + k;                  // k: j_i
        int32_t *nx = jt + k;                  // k: next step of the same hash chain (-1 = end)
        int32_t *head = nx + k;                // cap
        auto slot = [&](int32_t j) { return ((uint32_t)j * 0x9E3779B1u >> 16) & (uint32_t)(cap - 1); };
        for (int i = threadIdx.x; i < cap; i += blockDim.x) head[i] = -1;
        __syncthreads();
        uint64_t key = ((uint64_t)stage << 32) | (uint64_t)(uint32_t)s;
        const uint64_t st0 = seed ^ sm64_next(key);
        for (int i = threadIdx.x; i < k; i += blockDim.x) {
            uint64_t st = st0 + (uint64_t)i * 0x9E3779B97F4A7C15ULL;
            const uint64_t r = sm64_next(st);
            const int32_t j = first_k ? i : i + (int32_t)(r % (uint64_t)(m - i));
            jt[i] = j;
            nx[i] = atomicExch(&head[slot(j)], i);
        }
        __syncthreads();
        for (int i = threadIdx.x; i < k; i += blockDim.x) {
            int32_t p = jt[i], at = i;         // what position p held before step `at`
            for (;;) {
                int32_t q = -1;                // the last step before `at` that swapped p
                for (int32_t e = head[slot(p)]; e >= 0; e = nx[e])
                    if (jt[e] == p && e < at && e > q) q = e;
                if (q < 0) break;
                p = at = q;                    // it left there what position q held before step q
            }
            A[i] = p;
        }
        __syncthreads();
        const int64_t row0 = t.seg_start[s];
        const int64_t c0 = t.cen_off[s];
        for (int e = threadIdx.x; e < k * d; e += blockDim.x) {
            int j = e / d, a = e - j * d;
            centers[(c0 + j) * d + a] = pts[(row0 + A[j]) * d + a];
            acc[(c0 + j) * d + a] = 0ull;
        }
        for (int j = threadIdx.x; j < k; j += blockDim.x) {
            count2[c0 + j] = 0;
            count2[P + c0 + j] = 0;
        }
        __syncthreads();
    }
}

__device__ __forceinline__ unsigned long long to_fix(float v) { return fix_of(v); }

// Widths between the compiled ones run in the next wider kernel (D > d) on rows and centers
// padded with zeros: a padded attribute adds RN(0 * 0 + acc) = acc, so the distances are the
// same bits.  (Rows walked in global memory with a runtime width took 28 us an iteration at
// 200003 x 7, k = 40, where the padded kernel takes 8.)
constexpr int pad_width(int d)
{
    return d <= 2 ? 2 : d <= 4 ? 4 : d <= 8 ? 8 : d <= 12 ? 12 : d <= 16 ? 16 : d <= 24 ? 24 : d <= 32 ? 32
           : d <= 48 ? 48 : d <= 64 ? 64 : d <= 96 ? 96 : d <= 128 ? 128 : 0;
}

// A row of d <= D attributes into registers, zeros past d.
template <int D>
__device__ __forceinline__ void load_row(const float *__restrict__ xr, int d, float (&xv)[D])
{
    if (D % 4 == 0 && d == D && ((uintptr_t)xr & 15u) == 0) {        // a caller's points may lie anywhere
        const float4 *x4 = reinterpret_cast<const float4 *>(xr);
#pragma unroll
        for (int j4 = 0; j4 < D / 4; j4++) {
            const float4 v = __ldg(&x4[j4]);
            xv[4 * j4 + 0] = v.x;
            xv[4 * j4 + 1] = v.y;
            xv[4 * j4 + 2] = v.z;
            xv[4 * j4 + 3] = v.w;
        }
    } else {
#pragma unroll
        for (int j = 0; j < D; j++) xv[j] = j < d ? __ldg(&xr[j]) : 0.0f;
    }
}

// The float32 direct distance of a row of any width in global memory to a center in shared memory.
// From its first 32-byte boundary on the row is read a sector at a time, so that the rows of a
// block need not stay in L1 from one attribute to the next: read by attributes, rows of odd widths
// took twice as long whenever they did not (60000 x 129, k = 33: 46 % of the sectors hit, 1.42 ms an
// iteration, 75 % and 0.68 ms with other warps in the way; by sectors 0.57.  500 sets of 300 x 150
// 46 -> 13 ms, 200000 x 256 in sets of 10000 26 -> 8.8).
__device__ __forceinline__ float dist_any(const float *__restrict__ xr, const float *c, int d)
{
    float v = 0.0f;
    auto add = [&](float x, int a) {
        const float t = __fsub_rn(x, c[a]);
        v = __fmaf_rn(t, t, v);
    };
    const int head = min(d, (int)(8u - ((uint32_t)((uintptr_t)xr >> 2) & 7u)) & 7);
    // up to 7 attributes from a on, their loads together (one by one: one set of 20000 x 129, k = 300
    // 20.2 ms of a batch's ten iterations, together 18.5)
    auto part = [&](int a, int m) {
        float x[7];
#pragma unroll
        for (int q = 0; q < 7; q++) x[q] = q < m ? __ldg(&xr[a + q]) : 0.0f;
#pragma unroll
        for (int q = 0; q < 7; q++)
            if (q < m) add(x[q], a + q);
    };
    part(0, head);
    int a = head;
#pragma unroll 2
    for (; a + 8 <= d; a += 8) {
        const float4 p = __ldg(reinterpret_cast<const float4 *>(xr + a)), q = __ldg(reinterpret_cast<const float4 *>(xr + a + 4));
        add(p.x, a);
        add(p.y, a + 1);
        add(p.z, a + 2);
        add(p.w, a + 3);
        add(q.x, a + 4);
        add(q.y, a + 5);
        add(q.z, a + 6);
        add(q.w, a + 7);
    }
    part(a, d - a);
    return v;
}

// n centers of d attributes into shared memory at a stride of D >= d (D = 0: d), zeros past d, by
// NT threads (0: the block's; known, the strides are constants and the loads go out together: SSE
// of 20000 x 32, k = 300: 67 -> 45 us).
template <int D, int NT = 0>
__device__ __forceinline__ void load_centers(float *sc, const float *__restrict__ c, int n, int d)
{
    if (D == 0 || d == D) {
        for (int e = threadIdx.x; e < n * d; e += NT ? (unsigned)NT : blockDim.x) sc[e] = c[e];
    } else {
        for (int e = threadIdx.x; e < n * D; e += NT ? (unsigned)NT : blockDim.x) {
            const int j = e / D, a = e - j * D;
            sc[e] = a < d ? c[j * d + a] : 0.0f;
        }
    }
}

// Squared distances of R rows (registers) to one center (shared memory), float32
// direct form, ascending attributes; the center is read as float4 when D % 4 == 0.
template <int D, int R>
__device__ __forceinline__ void dist_rows(const float (&xv)[R][D], const float *c, float (&out)[R])
{
#pragma unroll
    for (int q = 0; q < R; q++) out[q] = 0.0f;
    if (D % 4 == 0) {
        const float4 *c4 = reinterpret_cast<const float4 *>(c);
#pragma unroll
        for (int j4 = 0; j4 < D / 4; j4++) {
            const float4 cv = c4[j4];
            const float cc[4] = {cv.x, cv.y, cv.z, cv.w};
#pragma unroll
            for (int e = 0; e < 4; e++) {
#pragma unroll
                for (int q = 0; q < R; q++) {
                    const float tq = __fsub_rn(xv[q][4 * j4 + e], cc[e]);
                    out[q] = __fmaf_rn(tq, tq, out[q]);
                }
            }
        }
    } else {
#pragma unroll
        for (int j = 0; j < D; j++) {
            const float cj = c[j];
#pragma unroll
            for (int q = 0; q < R; q++) {
                const float tq = __fsub_rn(xv[q][j], cj);
                out[q] = __fmaf_rn(tq, tq, out[q]);
            }
        }
    }
}

// The nearest of the n centers at sc (stride D, indices from base on) to R rows, folded into
// the best so far: strict comparisons in ascending order, so the lowest index wins equal
// distances.  Narrow rows against many centers take four at a time and keep only the smallest
// distance and its group of four (five instructions a group where a comparison and two
// selections per center took twelve, next to 8 D of arithmetic); the index is found at the
// end by scoring that group again, which only many centers repay (250000 x 2, k = 100: the
// local Lloyd 225 -> 177 us; 8 attributes or 16 centers: slower).  The others take two at a
// time, as independent sets of chains.
template <int D, int R>
__device__ __forceinline__ void scan_centers(const float (&xv)[R][D], const float *sc, int n, int base, float (&best)[R],
                                             int (&bj)[R])
{
    int j = 0;
    if (D <= 4 && n >= 32) {
        int grp[R];
#pragma unroll
        for (int q = 0; q < R; q++) grp[q] = -1;
        for (; j + 3 < n; j += 4) {
            float v[4][R];
#pragma unroll
            for (int e = 0; e < 4; e++) dist_rows<D, R>(xv, sc + (size_t)(j + e) * D, v[e]);
#pragma unroll
            for (int q = 0; q < R; q++) {
                const float mn = fminf(min3f(v[0][q], v[1][q], v[2][q]), v[3][q]);
                grp[q] = mn < best[q] ? j : grp[q];
                best[q] = fminf(best[q], mn);
            }
        }
#pragma unroll
        for (int q = 0; q < R; q++) {
            if (grp[q] >= 0) {
                const float *c = sc + (size_t)grp[q] * D;
                float x1[1][D], u[1];
#pragma unroll
                for (int a = 0; a < D; a++) x1[0][a] = xv[q][a];
                int e = 0;
                for (; e < 3; e++) {
                    dist_rows<D, 1>(x1, c + e * D, u);
                    if (u[0] == best[q]) break;
                }
                bj[q] = base + grp[q] + e;
            }
        }
    } else {
        for (; j + 1 < n; j += 2) {
            float v[R], w[R];
            dist_rows<D, R>(xv, sc + (size_t)j * D, v);
            dist_rows<D, R>(xv, sc + (size_t)(j + 1) * D, w);
#pragma unroll
            for (int q = 0; q < R; q++) {
                if (v[q] < best[q]) { best[q] = v[q]; bj[q] = base + j; }
                if (w[q] < best[q]) { best[q] = w[q]; bj[q] = base + j + 1; }
            }
        }
    }
    for (; j < n; j++) {
        float v[R];
        dist_rows<D, R>(xv, sc + (size_t)j * D, v);
#pragma unroll
        for (int q = 0; q < R; q++)
            if (v[q] < best[q]) { best[q] = v[q]; bj[q] = base + j; }
    }
}

// One assignment step over work units [unit_lo, unit_lo + gridDim.x).
//   D > 0: d <= D (see pad_width), each thread keeps R rows in registers and
//          reads every center once for all of them; D == 0: any d, one row at a time.
template <int D, int R, bool kSmemAcc>
__global__ void __launch_bounds__(kThreads)
k_lloyd_assign(const float *__restrict__ pts, SegTable t, int d, const float *__restrict__ centers,
               unsigned long long *acc, int32_t *count, int32_t *labels, int32_t *trace,
               int64_t trace_off, int unit_lo, int chunk_k, const int32_t *__restrict__ weights)
{
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int DR = D > 0 ? D : 1;
    const int u = unit_lo + blockIdx.x;
    const int s = t.unit_seg[u];
    const int k = t.k_eff[s];
    const int64_t c0 = t.cen_off[s];
    const int64_t row0 = t.seg_start[s] + t.unit_start[u];
    const int rows = t.unit_count[u];
    const int dd = D > 0 ? D : d;             // the centers' stride in shared memory

    // [center chunk | high sums | low sums | counts], each 16-byte aligned.  A fixed-point
    // value q <= 2^32 is added as q >> 11 (<= 2^21) and q & 0x7FF with two native 32-bit
    // shared atomics; a unit has at most 1024 rows, so neither sum can wrap, and the
    // flush recombines them exactly into the 64-bit global sums.  A center's sums take an
    // odd stride ds = d | 1, so that the lanes of a warp adding attribute a of different
    // centers fall in different banks (with stride 16 they shared two).
    const int ds = d | 1;
    const size_t c_bytes = ((size_t)min(chunk_k, k) * dd * 4 + 15) & ~(size_t)15;
    float *sc = reinterpret_cast<float *>(smem);
    uint32_t *shi = reinterpret_cast<uint32_t *>(smem + c_bytes);
    uint32_t *slo = shi + (size_t)k * ds;
    int32_t *scnt = reinterpret_cast<int32_t *>(slo + (size_t)k * ds);
    if (kSmemAcc) {
        for (int e = threadIdx.x; e < k * ds; e += kThreads) {
            shi[e] = 0u;
            slo[e] = 0u;
        }
        for (int j = threadIdx.x; j < k; j += kThreads) scnt[j] = 0;
    }
    chain_wait();
    const bool one_chunk = chunk_k >= k;
    // centers at .. at + n - 1: those of the compiled width at constant strides, so that their
    // loads go out together (ten iterations at 20000 x 128, k = 300: 4.89 -> 4.25 ms; 400000 x 16,
    // k = 64: 0.86 -> 0.81).  The padded ones are left at the block's: with both constant the
    // kernel for 64 attributes is scheduled worse, 2.26 -> 2.76 ms at 400000 x 64, k = 64.
    auto centers_in = [&](int64_t at, int n) {
        if (D > 0 && d != D) load_centers<D>(sc, centers + at * d, n, d);
        else for (int e = threadIdx.x; e < n * dd; e += kThreads) sc[e] = centers[at * dd + e];
    };
    if (one_chunk) centers_in(c0, k);
    __syncthreads();

    for (int p0 = 0; p0 < rows; p0 += kThreads * R) {
        float xv[R][DR];
        bool live[R];
        int prow[R];
#pragma unroll
        for (int q = 0; q < R; q++) {
            prow[q] = p0 + q * kThreads + threadIdx.x;
            live[q] = prow[q] < rows;
            if constexpr (D > 0) load_row<DR>(pts + (row0 + (live[q] ? prow[q] : 0)) * d, d, xv[q]);
        }
        float best[R];
        int bj[R];
#pragma unroll
        for (int q = 0; q < R; q++) {
            best[q] = __int_as_float(0x7f800000);
            bj[q] = 0;
        }
        // (a warp without a row left scores none: half of the warps of a unit of 128 rows; 25000 x 2,
        // k = 500: 14.5 -> 11.6 us an iteration.  Not where rows are walked in global memory: the
        // others' rows then leave L1 sooner; 20000 x 256, k = 300: 5.8 ms an iteration with them,
        // 6.5 without)
        const int kw = D > 0 && one_chunk && p0 + (threadIdx.x & ~31) >= rows ? 0 : k;
        for (int cb = 0; cb < kw; cb += chunk_k) {
            const int ce = min(k, cb + chunk_k);
            if (!one_chunk) {
                __syncthreads();
                centers_in(c0 + cb, ce - cb);
                __syncthreads();
            }
            if constexpr (D > 0) {
                scan_centers<DR, R>(xv, one_chunk ? sc + (size_t)cb * dd : sc, ce - cb, cb, best, bj);
            } else {
                const float *cbase = one_chunk ? sc + (size_t)cb * dd : sc;
                const float *xr = pts + (row0 + (live[0] ? prow[0] : 0)) * d;
                for (int j = cb; j < ce; j++) {
                    const float v = dist_any(xr, cbase + (size_t)(j - cb) * dd, d);
                    if (v < best[0]) { best[0] = v; bj[0] = j; }
                }
            }
        }
#pragma unroll
        for (int q = 0; q < R; q++) {
            if (!live[q]) continue;
            const int64_t row = row0 + prow[q];
            labels[row] = bj[q];
            if (trace) trace[trace_off + row] = bj[q];
            const float *xr = pts + row * d;
            if (kSmemAcc) {
                atomicAdd(&scnt[bj[q]], 1);
                const size_t e0 = (size_t)bj[q] * ds;
                if (D > 0) {
#pragma unroll
                    for (int j = 0; j < DR; j++) {
                        if (j < d) {
                            const unsigned long long v = to_fix(xv[q][j]);
                            atomicAdd(&shi[e0 + j], (uint32_t)(v >> 11));
                            atomicAdd(&slo[e0 + j], (uint32_t)(v & 0x7FFu));
                        }
                    }
                } else {
                    for (int j = 0; j < d; j++) {
                        const unsigned long long v = to_fix(__ldg(&xr[j]));
                        atomicAdd(&shi[e0 + j], (uint32_t)(v >> 11));
                        atomicAdd(&slo[e0 + j], (uint32_t)(v & 0x7FFu));
                    }
                }
            } else {
                // weighted rows (global sums only): w x and w; a zero weight adds nothing
                const unsigned long long w = weights ? (unsigned long long)(uint32_t)weights[row] : 1ull;
                if (w == 0ull) continue;
                atomicAdd(&count[c0 + bj[q]], (int)w);
                if (D > 0) {
#pragma unroll
                    for (int j = 0; j < DR; j++)
                        if (j < d) atomicAdd(&acc[(c0 + bj[q]) * d + j], to_fix(xv[q][j]) * w);
                } else {
                    for (int j = 0; j < d; j++) atomicAdd(&acc[(c0 + bj[q]) * d + j], to_fix(__ldg(&xr[j])) * w);
                }
            }
        }
    }
    if (kSmemAcc) {
        __syncthreads();
        for (int e = threadIdx.x; e < k * d; e += kThreads) {
            const int c = e / d, es = c * ds + (e - c * d);
            const unsigned long long v = ((unsigned long long)shi[es] << 11) + slo[es];
            if (v) atomicAdd(&acc[c0 * d + e], v);
        }
        for (int j = threadIdx.x; j < k; j += kThreads) {
            int v = scnt[j];
            if (v) atomicAdd(&count[c0 + j], v);
        }
    }
}

// ---------------------------------------------------------------- small sets: every iteration in one launch
// All iterations of a set of at most R blockDim rows by one CTA: its rows stay in registers
// (R per thread), its centers, exact sums and counts in shared memory, and an iteration costs
// two barriers instead of two launches.  The arithmetic is k_lloyd_assign's and
// k_lloyd_finalize's, so the results are the same bits.  After the first iteration only the
// rows that moved are added (and taken off their old center: the sums are integers, the two
// 32-bit halves of fix_parts modulo 2^32, exact for up to 65535 rows), only the centers they
// touched are formed again, and an iteration in which no row moved ends the set: its centers
// are a fixed point, so every later iteration would repeat it.  Lloyd of 16 sets of 256 x 4
// (k = 16, 20 iterations) 124 + 115 us of launches back to back -> 17 us; 300 sets of 40-600
// rows x 5 222 -> 42 us; 250 sets of 1000 x 2 (k = 100) 640 -> 177 us.
constexpr int kSetThreads = 1024;
constexpr size_t kSetSmemMax = 100 * 1024;

// rows per thread: 32 floats of rows at most, or one wider row (MAXT is 1024 only for sets that
// need as many threads: at 64 registers a thread the wider of them spill)
template <int D>
__host__ __device__ constexpr int kSetRows()
{
    return D >= 32 ? 1 : (32 / D > 4 ? 4 : 32 / D);
}

// the rows of a set that one CTA's registers hold
inline int set_rows(int D)
{
    return D <= 32 ? kSetThreads * (32 / D > 4 ? 4 : 32 / D) : D <= 64 ? 512 : 256;
}

// [centers k x D | high, low sums k x (d | 1) | reciprocals k (double) | counts k | touched k]
__host__ __device__ inline size_t set_smem(int D, int d, int k)
{
    const size_t c = ((size_t)k * D * 4 + (size_t)k * (d | 1) * 8 + 15) & ~(size_t)15;
    return c + (size_t)k * 8 + (size_t)k * 8;
}

template <int D, int R, int MAXT>
__global__ void __launch_bounds__(MAXT)
k_lloyd_sets(const float *__restrict__ pts, SegTable t, int d, float *centers, int32_t *count2, int64_t P,
             int32_t *labels, int32_t *trace, int64_t rows_all, int iters)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int s = blockIdx.x, tid = threadIdx.x, NT = blockDim.x;
    const int k = t.k_eff[s], rows = t.seg_size[s];
    const int64_t c0 = t.cen_off[s], row0 = t.seg_start[s];
    const int ds = d | 1;
    float *sc = reinterpret_cast<float *>(smem);
    uint32_t *shi = reinterpret_cast<uint32_t *>(sc + (size_t)k * D);
    uint32_t *slo = shi + (size_t)k * ds;
    double *srec = reinterpret_cast<double *>(smem + (((size_t)k * D * 4 + (size_t)k * ds * 8 + 15) & ~(size_t)15));
    int32_t *scnt = reinterpret_cast<int32_t *>(srec + k);
    int32_t *stouch = scnt + k;                // the last iteration (+ 1) that changed the center's members
    load_centers<D>(sc, centers + c0 * d, k, d);
    for (int e = tid; e < 2 * k * ds; e += NT) shi[e] = 0u;
    for (int j = tid; j < k; j += NT) scnt[j] = stouch[j] = 0;
    float xv[R][D];
    int lab[R];
#pragma unroll
    for (int q = 0; q < R; q++) {
        const int r = q * NT + tid;
        load_row<D>(pts + (row0 + (r < rows ? r : 0)) * d, d, xv[q]);
        lab[q] = -1;
    }
    __syncthreads();
    int it = 0;
    for (; it < iters; it++) {
        float best[R];
        int bj[R];
#pragma unroll
        for (int q = 0; q < R; q++) {
            best[q] = __int_as_float(0x7f800000);
            bj[q] = 0;
        }
        scan_centers<D, R>(xv, sc, k, 0, best, bj);
        bool moved = false;
#pragma unroll
        for (int q = 0; q < R; q++) {
            const int r = q * NT + tid;
            if (r >= rows) continue;
            if (trace) trace[(int64_t)it * rows_all + row0 + r] = bj[q];
            if (bj[q] == lab[q]) continue;
            moved = true;
            const int o = lab[q];
            atomicAdd(&scnt[bj[q]], 1);
            stouch[bj[q]] = it + 1;
            if (o >= 0) {
                atomicSub(&scnt[o], 1);
                stouch[o] = it + 1;
            }
            auto move = [&](float v, int a) {
                uint32_t hi, lo;
                fix_parts(v, hi, lo);
                atomicAdd(&shi[bj[q] * ds + a], hi);
                atomicAdd(&slo[bj[q] * ds + a], lo);
                if (o >= 0) {
                    atomicSub(&shi[o * ds + a], hi);
                    atomicSub(&slo[o * ds + a], lo);
                }
            };
            if constexpr (D <= 32) {
#pragma unroll
                for (int a = 0; a < D; a++)
                    if (a < d) move(xv[q][a], a);
            } else {                            // a wide row read again: unrolled, its sums spill
                const float *x = pts + (row0 + r) * d;
#pragma unroll 4
                for (int a = 0; a < d; a++) move(__ldg(&x[a]), a);
            }
            lab[q] = bj[q];
        }
        if (!__syncthreads_or(moved)) break;
        for (int c = tid; c < k; c += NT)
            if (stouch[c] == it + 1 && scnt[c] > 0) srec[c] = __drcp_rn((double)scnt[c]);
        __syncthreads();
        for (int e = tid; e < k * d; e += NT) {
            const int c = e / d, a = e - c * d;
            if (stouch[c] == it + 1 && scnt[c] > 0) {
                const long long sum = (long long)(((unsigned long long)shi[c * ds + a] << 16) + slo[c * ds + a]);
                sc[(size_t)c * D + a] = __double2float_rn(__dmul_rn(__dmul_rn((double)sum, 0x1p-32), srec[c]));
            }
        }
        __syncthreads();
    }
    // (a set that ended early: its remaining iterations repeat the last one)
#pragma unroll
    for (int q = 0; q < R; q++) {
        const int r = q * NT + tid;
        if (r < rows && iters > 0) {
            labels[row0 + r] = lab[q];
            if (trace)
                for (int i2 = it + 1; i2 < iters; i2++) trace[(int64_t)i2 * rows_all + row0 + r] = lab[q];
        }
    }
    for (int e = tid; e < k * d; e += NT) {
        const int c = e / d, a = e - c * d;
        centers[c0 * d + e] = sc[(size_t)c * D + a];
    }
    if (iters > 0) {
        int32_t *cnt = count2 + (size_t)((iters - 1) & 1) * P;
        for (int j = tid; j < k; j += NT) cnt[c0 + j] = scnt[j];
    }
}

// center = exact sum / count (double), rounded once to float; empty clusters keep their
// center.  Clears the sums and the other parity's counts for the next iteration, or with
// `keep` (a sums pass that adds only the rows that moved) leaves the sums and carries the
// counts over.  A thread
// takes EPT consecutive attributes of one center (d % EPT == 0) and forms the count's
// reciprocal once for them: float64 is the slow pipe of this GPU.  I is the element index
// type (32-bit whenever the elements fit, which avoids 64-bit division).
template <int EPT, typename I>
__global__ void k_lloyd_finalize(float *centers, unsigned long long *acc, const int32_t *count,
                                 int32_t *count_next, int64_t cen_lo, int64_t cen_hi, int d, bool keep)
{
    chain_wait();
    const I g0 = (I)(cen_lo * d / EPT), g1 = (I)(cen_hi * d / EPT), dd = (I)d;
    for (I g = g0 + (I)blockIdx.x * blockDim.x + threadIdx.x; g < g1; g += (I)gridDim.x * blockDim.x) {
        const I e = g * EPT;
        const I c = e / dd;
        const int32_t n = count[c];
        if (n > 0) {
            const double r = __drcp_rn((double)n);
#pragma unroll
            for (int q = 0; q < EPT; q++) {
                const long long sum = (long long)acc[e + q];
                centers[e + q] = __double2float_rn(__dmul_rn(__dmul_rn((double)sum, 0x1p-32), r));
            }
        }
        if (!keep) {
#pragma unroll
            for (int q = 0; q < EPT; q++) acc[e + q] = 0ull;
        }
        if (e - c * dd == 0) count_next[c] = keep ? n : 0;
    }
}

template <int EPT>
cudaError_t finalize_launch(const LloydBuffers &b, int32_t *count_next, int64_t cen_lo, int64_t cen_hi, int d,
                     int sm_count, bool keep, cudaStream_t st)
{
    const int64_t work = (cen_hi - cen_lo) * d / EPT;
    int64_t g = (work + 255) / 256;
    if (g > (int64_t)sm_count * 8) g = (int64_t)sm_count * 8;
    if (g < 1) g = 1;
    if (cen_hi * d < ((int64_t)1 << 31))
        return launch_chained(b.chain, k_lloyd_finalize<EPT, uint32_t>, g, 256, 0, st, b.centers, b.acc, b.count, count_next, cen_lo,
                              cen_hi, d, keep);
    return launch_chained(b.chain, k_lloyd_finalize<EPT, int64_t>, g, 256, 0, st, b.centers, b.acc, b.count, count_next, cen_lo, cen_hi,
                          d, keep);
}

// The nearest of a set's centers to R rows of one thread: float32 direct distances, two centers
// at a time (two independent sets of chains), the lowest index on equal ones.
template <int D, int R>
struct Nearest {
    float xv[R][D > 0 ? D : 1];
    const float *xr;
    float best[R];
    int bj[R];
    // rows i0, i0 + step, ... (those below n; past them the first row again)
    __device__ __forceinline__ void load(const float *__restrict__ x, int64_t i0, int64_t step, int64_t n, int d)
    {
#pragma unroll
        for (int q = 0; q < R; q++) {
            const int64_t i = i0 + q * step;
            const float *r = x + (i < n ? i : 0) * d;
            if constexpr (D > 0) load_row<D>(r, d, xv[q]);
            else xr = r;
            best[q] = __int_as_float(0x7f800000);
            bj[q] = 0;
        }
    }
    // centers cb .. ce - 1, sc holding them from cb on
    __device__ __forceinline__ void score(const float *sc, int cb, int ce, int d)
    {
        if constexpr (D > 0) {
            scan_centers<D, R>(xv, sc, ce - cb, cb, best, bj);
        } else {
            for (int j = cb; j < ce; j++) {
                const float acc = dist_any(xr, sc + (size_t)(j - cb) * d, d);
                if (acc < best[0]) { best[0] = acc; bj[0] = j; }
            }
        }
    }
};

// ---------------------------------------------------------------- wide rows: register tiles
// A thread with one wide row in registers reads 16 bytes of a center from shared memory per 8
// float32 instructions; shared memory returns 128 bytes a cycle to an SM, so those loads take
// twice the cycles of the arithmetic (1000003 x 64, k = 300: 19.6 of 37 TFLOP/s).  Here a
// block takes 256 rows in shared memory and a thread an 8 x 4 tile of (row, center) pairs:
// 12 such loads per 256 instructions.  The distances are the same chains (ascending
// attributes, one subtraction and one fused multiply-add each; zeros past d), and the lowest
// index wins ties.  Rows and centers lie at an odd number of 16-byte words, so that 8
// consecutive ones fall in different banks.
constexpr int kTileC = 64;                                 // centers in shared memory at a time
// Widths that take the tiles.  At d = 32 two rows per thread are faster for the units of independent
// sets (the uneven batch 7.1 against 9.5 ms), and the tiles for one set, whose few rows leave a
// thread one row and its two chains (6 x 32, k = 340: 62 us, tiles 40, one chain a thread 46; 400000 x
// 32, k = 64: 134, 89 and 169).
constexpr int kTiledMin = 32, kTiledMinUnits = 33, kTiledMax = 128;

constexpr int kTiledCenters = 24;                          // fewer leave the tile's 32 mostly empty

__host__ __device__ constexpr size_t tile_smem(int d) { return (size_t)(kThreads + kTileC) * tile_ld4(d) * 16; }

// The nearest of k centers to each of the block's rows (xs: kThreads rows, loaded and
// synchronised); cs: kTileC rows.  Thread t returns row t's.  Every thread of the block calls.
__device__ __forceinline__ void tile_nearest(const float4 *xs, float4 *cs, const float *__restrict__ centers, int k,
                                             int d, int ld4, float &rbest, int &rbj)
{
    __shared__ float s_best[kThreads];
    __shared__ int s_bj[kThreads];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, d4 = (d + 3) / 4;
    const int cg = lane & 7, rg = w * 4 + (lane >> 3);     // centers cg + 8 j, rows rg + 32 i
    float best[8];
    int bj[8];
#pragma unroll
    for (int i = 0; i < 8; i++) {
        best[i] = __int_as_float(0x7f800000);
        bj[i] = 0x7fffffff;
    }
    for (int cb = 0; cb < k; cb += kTileC) {
        const int nc = min(kTileC, k - cb);
        __syncthreads();
        tile_load(cs, centers + (int64_t)cb * d, nc, (nc + 31) & ~31, d, ld4);
        __syncthreads();
        for (int c0 = 0; c0 < nc; c0 += 32) {
            float acc[8][4];
#pragma unroll
            for (int i = 0; i < 8; i++)
#pragma unroll
                for (int j = 0; j < 4; j++) acc[i][j] = 0.0f;
            const float4 *xp = xs + rg * ld4, *cp = cs + (c0 + cg) * ld4;
            for (int q = 0; q < d4; q++) {
                float4 xr[8];
#pragma unroll
                for (int i = 0; i < 8; i++) xr[i] = xp[i * 32 * ld4 + q];
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    const float4 c = cp[j * 8 * ld4 + q];
#pragma unroll
                    for (int i = 0; i < 8; i++) {
                        float t = __fsub_rn(xr[i].x, c.x);
                        acc[i][j] = __fmaf_rn(t, t, acc[i][j]);
                        t = __fsub_rn(xr[i].y, c.y);
                        acc[i][j] = __fmaf_rn(t, t, acc[i][j]);
                        t = __fsub_rn(xr[i].z, c.z);
                        acc[i][j] = __fmaf_rn(t, t, acc[i][j]);
                        t = __fsub_rn(xr[i].w, c.w);
                        acc[i][j] = __fmaf_rn(t, t, acc[i][j]);
                    }
                }
            }
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const int c = c0 + cg + 8 * j;
                if (c < nc) {
#pragma unroll
                    for (int i = 0; i < 8; i++)
                        if (acc[i][j] < best[i]) {
                            best[i] = acc[i][j];
                            bj[i] = cb + c;
                        }
                }
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 8; i++) {
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) {
            const float ov = __shfl_xor_sync(0xffffffffu, best[i], o);
            const int oj = __shfl_xor_sync(0xffffffffu, bj[i], o);
            if (ov < best[i] || (ov == best[i] && oj < bj[i])) {
                best[i] = ov;
                bj[i] = oj;
            }
        }
        if (cg == 0) {
            s_best[rg + 32 * i] = best[i];
            s_bj[rg + 32 * i] = bj[i];
        }
    }
    __syncthreads();
    rbest = s_best[threadIdx.x];
    rbj = s_bj[threadIdx.x] < k ? s_bj[threadIdx.x] : 0;   // (no distance below infinity: center 0, as elsewhere)
}

// Nearest final center of every scaled point (original order) and the sum of squared
// errors: each point's float32 direct distance is added in double, per thread, then
// per block and over the blocks in a fixed tree.
// D > 0: d <= D, a thread keeps R of its rows (consecutive ones in its order, so the sums are
// the same whatever R) in registers and scores two centers at a time against them.
template <int D, int R>
__global__ void __launch_bounds__(kThreads)
k_final_sse(const float *__restrict__ x, int64_t n, int d, const float *__restrict__ centers,
            int k, int chunk_k, int32_t *labels, double *blk_sse, double *sse, uint32_t *ticket)
{
    sse_enter(ticket);
    extern __shared__ __align__(16) unsigned char smem[];
    float *sc = reinterpret_cast<float *>(smem);
    const bool one_chunk = chunk_k >= k;
    if (one_chunk) {
        load_centers<D, kThreads>(sc, centers, k, d);
        __syncthreads();
    }
    double part = 0.0;
    const int64_t stride = (int64_t)gridDim.x * kThreads;
    const int64_t nround = (n + stride - 1) / stride;
    for (int64_t it = 0; it < nround; it += R) {
        const int64_t i0 = it * stride + (int64_t)blockIdx.x * kThreads + threadIdx.x;
        Nearest<D, R> nb;
        nb.load(x, i0, stride, n, d);
        for (int cb = 0; cb < k; cb += chunk_k) {
            const int ce = min(k, cb + chunk_k);
            if (!one_chunk) {
                __syncthreads();
                load_centers<D, kThreads>(sc, centers + (size_t)cb * d, ce - cb, d);
                __syncthreads();
            }
            nb.score(sc, cb, ce, d);
        }
#pragma unroll
        for (int q = 0; q < R; q++)
            if (i0 + q * stride < n) {
                labels[i0 + q * stride] = nb.bj[q];
                part = __dadd_rn(part, (double)nb.best[q]);
            }
    }
    sse_reduce(part, blk_sse, sse, ticket);
}

// The same for wide rows (register tiles): a block's 256 rows are the tile, so every thread
// adds the same rows in the same order.
__global__ void __launch_bounds__(kThreads, 2)
k_final_sse_tiled(const float *__restrict__ x, int64_t n, int d, const float *__restrict__ centers, int k,
                  int32_t *labels, double *blk_sse, double *sse, uint32_t *ticket)
{
    sse_enter(ticket);
    extern __shared__ __align__(16) float4 tiles[];
    const int ld4 = tile_ld4(d);
    float4 *xs = tiles, *cs = tiles + kThreads * ld4;
    double part = 0.0;
    const int64_t stride = (int64_t)gridDim.x * kThreads;
    for (int64_t i0 = (int64_t)blockIdx.x * kThreads; i0 < n; i0 += stride) {
        const int rows = (int)min((int64_t)kThreads, n - i0);
        __syncthreads();
        tile_load(xs, x + i0 * d, rows, kThreads, d, ld4);
        float best;
        int bj;
        tile_nearest(xs, cs, centers, k, d, ld4, best, bj);
        if ((int)threadIdx.x < rows) {
            labels[i0 + threadIdx.x] = bj;
            part = __dadd_rn(part, (double)best);
        }
    }
    sse_reduce(part, blk_sse, sse, ticket);
}

int center_chunk(int d, int k)
{
    int c = kCenterChunkBytes / (d * 4);
    if (c < 1) c = 1;
    return c >= k ? k : c;
}

// Per work unit of independent sets: the nearest center of every row among its set's
// centers (float32 direct form, lowest index on ties) and the sum of those squared
// distances in double (per thread in row order, then a fixed tree over the block).
template <int D, int R>
__global__ void __launch_bounds__(kThreads)
k_seg_sse(const float *__restrict__ pts, SegTable t, int d, const float *__restrict__ centers, int chunk_k,
          int32_t *labels, double *unit_sse)
{
    extern __shared__ __align__(16) unsigned char smem[];
    float *sc = reinterpret_cast<float *>(smem);
    const int u = blockIdx.x;
    const int s = t.unit_seg[u];
    const int k = t.k_eff[s];
    const int64_t c0 = t.cen_off[s];
    const int64_t row0 = t.seg_start[s] + t.unit_start[u];
    const int rows = t.unit_count[u];
    const bool one_chunk = chunk_k >= k;
    if (one_chunk) {
        load_centers<D>(sc, centers + c0 * d, k, d);
        __syncthreads();
    }
    double part = 0.0;
    for (int p0 = 0; p0 < rows; p0 += R * kThreads) {
        Nearest<D, R> nb;
        nb.load(pts + row0 * d, p0 + (int)threadIdx.x, kThreads, rows, d);
        for (int cb = 0; cb < k; cb += chunk_k) {
            const int ce = min(k, cb + chunk_k);
            if (!one_chunk) {
                __syncthreads();
                load_centers<D>(sc, centers + (c0 + cb) * d, ce - cb, d);
                __syncthreads();
            }
            nb.score(sc, cb, ce, d);
        }
#pragma unroll
        for (int q = 0; q < R; q++) {
            const int p = p0 + q * kThreads + (int)threadIdx.x;
            if (p < rows) {
                labels[row0 + p] = nb.bj[q];
                part = __dadd_rn(part, (double)nb.best[q]);
            }
        }
    }
    const double b = block_tree_sum(part);
    if (threadIdx.x == 0) unit_sse[u] = b;
}

// The same for wide rows (register tiles).
__global__ void __launch_bounds__(kThreads, 2)
k_seg_sse_tiled(const float *__restrict__ pts, SegTable t, int d, const float *__restrict__ centers, int32_t *labels,
                double *unit_sse)
{
    extern __shared__ __align__(16) float4 tiles[];
    const int ld4 = tile_ld4(d);
    float4 *xs = tiles, *cs = tiles + kThreads * ld4;
    const int u = blockIdx.x, s = t.unit_seg[u], k = t.k_eff[s], rows = t.unit_count[u];
    const float *cen = centers + (int64_t)t.cen_off[s] * d;
    const int64_t row0 = t.seg_start[s] + t.unit_start[u];
    double part = 0.0;
    for (int p0 = 0; p0 < rows; p0 += kThreads) {
        const int nr = min(kThreads, rows - p0);
        __syncthreads();
        tile_load(xs, pts + (row0 + p0) * d, nr, kThreads, d, ld4);
        float best;
        int bj;
        tile_nearest(xs, cs, cen, k, d, ld4, best, bj);
        if ((int)threadIdx.x < nr) {
            labels[row0 + p0 + threadIdx.x] = bj;
            part = __dadd_rn(part, (double)best);
        }
    }
    const double b = block_tree_sum(part);
    if (threadIdx.x == 0) unit_sse[u] = b;
}

// SSE of every set: its units' sums in unit order.
__global__ void k_seg_sse_fold(const double *unit_sse, const int32_t *seg_unit0, int n_seg, double *seg_sse)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n_seg) return;
    double v = 0.0;
    for (int u = seg_unit0[s]; u < seg_unit0[s + 1]; u++) v = __dadd_rn(v, unit_sse[u]);
    seg_sse[s] = v;
}

// rows kept in registers per thread: 64 floats of rows at most
template <int D>
__host__ __device__ constexpr int kRowsPerThread()
{
    return D <= 0 ? 1 : (D >= 64 ? 1 : 64 / D > 4 ? 4 : 64 / D);
}

template <int D>
cudaError_t seg_sse_dispatch(const float *pts, const SegTable &t, int d, const float *centers, int kmax,
                             int32_t *labels, double *unit_sse, cudaStream_t st, KTimer *kt)
{
    const int chunk = center_chunk(D > 0 ? D : d, kmax);
    const size_t smem = (size_t)chunk * (D > 0 ? D : d) * 4;
    auto kern = k_seg_sse<D, kRowsPerThread<D>()>;
    if (const cudaError_t ea = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) return ea;
    kt->begin(st);
    kern<<<t.n_units, kThreads, smem, st>>>(pts, t, d, centers, chunk, labels, unit_sse);
    kt->end(PSCL_K_FINAL_SSE, st);
    return cudaGetLastError();
}

template <int D, int R>
cudaError_t assign_launch(const LloydBuffers &b, const SegTable &t, int d, int iter, int unit_lo,
                          int unit_hi, int kmax, cudaStream_t st, KTimer *kt)
{
    const int chunk = center_chunk(D > 0 ? D : d, kmax);
    const size_t acc_bytes = (size_t)kmax * (d | 1) * 8 + (size_t)kmax * 4;
    const size_t c_bytes = ((size_t)chunk * (D > 0 ? D : d) * 4 + 15) & ~(size_t)15;
    const bool smem_acc = !b.weights && acc_bytes <= kSmemAccMax;
    const size_t smem = (smem_acc ? acc_bytes : 0) + c_bytes;
    const int grid = unit_hi - unit_lo;
    if (grid <= 0) return cudaSuccess;
    cudaError_t e;
    if (smem_acc) {
        auto kern = k_lloyd_assign<D, R, true>;
        if (const cudaError_t ea = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) return ea;
        kt->begin(st);
        e = launch_chained(b.chain, kern, grid, kThreads, smem, st, b.pts, t, d, b.centers, b.acc, b.count, b.labels, b.trace,
                           (int64_t)iter * b.rows, unit_lo, chunk, b.weights);
        kt->end(PSCL_K_LLOYD_ASSIGN, st);
    } else {
        auto kern = k_lloyd_assign<D, R, false>;
        if (const cudaError_t ea = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) return ea;
        kt->begin(st);
        e = launch_chained(b.chain, kern, grid, kThreads, smem, st, b.pts, t, d, b.centers, b.acc, b.count, b.labels, b.trace,
                           (int64_t)iter * b.rows, unit_lo, chunk, b.weights);
        kt->end(PSCL_K_LLOYD_ASSIGN, st);
    }
    return e;
}

template <int D, int R, int MAXT>
cudaError_t sets_launch(const LloydBuffers &b, const SegTable &t, int d, int64_t P, int max_rows, int kmax, int iters,
                        cudaStream_t st, KTimer *kt)
{
    const size_t smem = set_smem(D, d, kmax);
    auto kern = k_lloyd_sets<D, R, MAXT>;
    if (const cudaError_t ea = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) return ea;
    const int threads = std::min(MAXT, ((max_rows + R - 1) / R + 31) / 32 * 32);
    kt->begin(st);
    kern<<<t.n_seg, threads, smem, st>>>(b.pts, t, d, b.centers, b.count, P, b.labels, b.trace, b.rows, iters);
    kt->end(PSCL_K_LLOYD_ASSIGN, st);
    return cudaGetLastError();
}

template <int D>
cudaError_t sets_dispatch(const LloydBuffers &b, const SegTable &t, int d, int64_t P, int max_rows, int kmax,
                          int iters, cudaStream_t st, KTimer *kt)
{
    // one row per thread for sets of up to 256 rows (more warps hide more latency), two of up to 8
    // attributes for sets of up to 2048 (300 sets of 40-600 rows x 5: the whole batch 126 -> 123
    // us), else as many as the registers hold (each center read from shared memory serves them all)
    constexpr int R = kSetRows<D>();
    if (max_rows <= 256) return sets_launch<D, 1, 256>(b, t, d, P, max_rows, kmax, iters, st, kt);
    if constexpr (R >= 4) {
        if (max_rows <= 1024) return sets_launch<D, 2, 512>(b, t, d, P, max_rows, kmax, iters, st, kt);
        if (max_rows <= 2048) return sets_launch<D, 2, 1024>(b, t, d, P, max_rows, kmax, iters, st, kt);
    } else if constexpr (D <= 64) {
        if (max_rows <= 512 * R) return sets_launch<D, R, 512>(b, t, d, P, max_rows, kmax, iters, st, kt);
    }
    if constexpr (D <= 32) return sets_launch<D, R, 1024>(b, t, d, P, max_rows, kmax, iters, st, kt);
    return cudaErrorInvalidValue;
}

// rows_per_thread: 0 = kRowsPerThread<D>(), 1 = one row per thread, 2 = eight rows per
// thread for d <= 16 (tuning choices; the result is the same)
template <int D>
cudaError_t assign_dispatch(const LloydBuffers &b, const SegTable &t, int d, int iter, int unit_lo,
                            int unit_hi, int kmax, int rows_per_thread, cudaStream_t st, KTimer *kt)
{
    if (rows_per_thread == 1 && kRowsPerThread<D>() > 1)
        return assign_launch<D, 1>(b, t, d, iter, unit_lo, unit_hi, kmax, st, kt);
    if (rows_per_thread == 2 && D > 0 && D <= 16)                 // 8 rows: half the center reads
        return assign_launch<D, (D > 0 && D <= 16 ? 8 : 1)>(b, t, d, iter, unit_lo, unit_hi, kmax, st, kt);
    return assign_launch<D, kRowsPerThread<D>()>(b, t, d, iter, unit_lo, unit_hi, kmax, st, kt);
}

// An SSE kernel; its blocks as one cluster where no ticket is given (see sse_reduce).
template <class... P, class... A>
cudaError_t sse_launch(void (*kern)(P...), int grid, size_t smem, bool cluster, cudaStream_t st, A... args)
{
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)grid;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(grid);
    c.blockDim = dim3(kThreads);
    c.dynamicSmemBytes = smem;
    c.stream = st;
    c.attrs = &at;
    c.numAttrs = cluster ? 1 : 0;
    return cudaLaunchKernelEx(&c, kern, static_cast<P>(args)...);
}

template <int D>
cudaError_t sse_dispatch(const float *x, int64_t n, int d, const float *centers, int k, int32_t *labels,
                         double *blk_sse, double *sse, uint32_t *ticket, int sm_count, cudaStream_t st,
                         KTimer *kt)
{
    const int chunk = center_chunk(D > 0 ? D : d, k);
    const size_t smem = (size_t)chunk * (D > 0 ? D : d) * 4;
    int64_t want = (n + kThreads - 1) / kThreads;
    int grid = (int)(want < (int64_t)sm_count * 8 ? want : (int64_t)sm_count * 8);
    if (grid < 1) grid = 1;
    // several rows per thread only where a thread has several
    auto kern = n > (int64_t)grid * kThreads ? k_final_sse<D, kRowsPerThread<D>()> : k_final_sse<D, 1>;
    if (const cudaError_t ea = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) return ea;
    kt->begin(st);
    const cudaError_t e = sse_launch(kern, grid, smem, ticket == nullptr, st, x, n, d, centers, k, chunk, labels, blk_sse,
                                     sse, ticket);
    kt->end(PSCL_K_FINAL_SSE, st);
    return e;
}

}  // namespace

bool small_sse(int64_t n) { return n <= (int64_t)kClusterSse * kThreads; }

int sse_grid(int64_t n, int sm_count)
{
    int64_t want = (n + kThreads - 1) / kThreads;
    return (int)(want < (int64_t)sm_count * 8 ? want : (int64_t)sm_count * 8);
}

cudaError_t launch_lloyd_init(const LloydBuffers &b, const SegTable &t, int d, int64_t P,
                              uint64_t seed, uint32_t stage, int first_k, int kmax, cudaStream_t st,
                              KTimer *kt)
{
    int cap = 1;
    while (cap < kmax) cap <<= 1;
    size_t smem = (3 * (size_t)kmax + (size_t)cap) * sizeof(int32_t);
    if (const cudaError_t ea = cudaFuncSetAttribute(k_lloyd_init, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) return ea;
    int grid = t.n_seg < 65535 ? t.n_seg : 65535;
    kt->begin(st);
    k_lloyd_init<<<grid, 256, smem, st>>>(b.pts, t, d, b.centers, b.acc, b.count, P, seed, stage, first_k);
    kt->end(PSCL_K_LLOYD_INIT, st);
    return cudaGetLastError();
}

// Whether small sets run all their iterations in one launch (k_lloyd_sets) rather than two
// launches an iteration.  Both score the same distances; per iteration the launches add about
// 11000 cycles on an idle GPU (2.5-3 us each) where the one launch's barriers add 1500, but a
// set then has one SM alone: rows k (2 D + 3) instructions at 60 % of 128 lanes (half of that
// with one wide row per thread, bound by reading the centers).  The launch pays while the largest set's time stays below the whole work spread over the SMs plus the
// difference.
bool sets_supported(const SegTable &t, int d, int max_rows, int kmax, double evals, int prec, const LloydBuffers &b,
                    int sm_count)
{
    const int D = pad_width(d);
    if (b.weights || D == 0 || max_rows > set_rows(D) || set_smem(D, d, kmax) > kSetSmemMax) return false;
    if (prec != PSCL_PREC_FP32 && b.tmask && t.split && tc_supported(d, kmax, prec, b.rows)) return false;
    const double per = (2.0 * D + 3.0) / (128.0 * (D <= 32 ? 0.6 : 0.3));
    return (double)max_rows * kmax * per <= evals * per / sm_count + 9500.0;
}

cudaError_t launch_lloyd_sets(const LloydBuffers &b, const SegTable &t, int d, int64_t P, int max_rows, int kmax,
                              int iters, cudaStream_t st, KTimer *kt)
{
    switch (pad_width(d)) {
    case 2: return sets_dispatch<2>(b, t, d, P, max_rows, kmax, iters, st, kt);
    case 4: return sets_dispatch<4>(b, t, d, P, max_rows, kmax, iters, st, kt);
    case 8: return sets_dispatch<8>(b, t, d, P, max_rows, kmax, iters, st, kt);
    case 12: return sets_dispatch<12>(b, t, d, P, max_rows, kmax, iters, st, kt);
    case 16: return sets_dispatch<16>(b, t, d, P, max_rows, kmax, iters, st, kt);
    case 24: return sets_dispatch<24>(b, t, d, P, max_rows, kmax, iters, st, kt);
    case 32: return sets_dispatch<32>(b, t, d, P, max_rows, kmax, iters, st, kt);
    case 48: return sets_dispatch<48>(b, t, d, P, max_rows, kmax, iters, st, kt);
    case 64: return sets_dispatch<64>(b, t, d, P, max_rows, kmax, iters, st, kt);
    case 96: return sets_dispatch<96>(b, t, d, P, max_rows, kmax, iters, st, kt);
    case 128: return sets_dispatch<128>(b, t, d, P, max_rows, kmax, iters, st, kt);
    default: return cudaErrorInvalidValue;
    }
}

// One Lloyd iteration over units [unit_lo, unit_hi) and centers [cen_lo, cen_hi).
// b.count must point at this iteration's count buffer; count_next at the other one.
cudaError_t launch_lloyd_iter(const LloydBuffers &b, int32_t *count_next, const SegTable &t, int d,
                              int iter, int unit_lo, int unit_hi, int64_t cen_lo, int64_t cen_hi,
                              int kmax, int prec, uint32_t *flags, int sm_count, cudaStream_t st,
                              KTimer *kt, int rows_per_thread)
{
    cudaError_t e;
    bool keep = false;
    if (prec != PSCL_PREC_FP32 && !b.weights && b.tmask && t.split && unit_lo == 0 && unit_hi == t.n_units &&
        tc_supported(d, kmax, prec, b.rows)) {
        e = launch_lloyd_assign_tc(b, t, d, iter, kmax, prec, flags, sm_count, st, kt);
        keep = b.raw != nullptr;
    } else if (prec != PSCL_PREC_FP32 && !b.weights && b.has_chunks && b.chunk_scratch && t.n_seg == 1 &&
               kmax > tc_chunk(d) && unit_lo == 0 && unit_hi == t.n_units && tc_sse_supported(d, kmax, prec, b.rows)) {
        e = launch_lloyd_chunks_tc(b, d, iter, kmax, prec, flags, sm_count, st, kt);
    } else switch (pad_width(d)) {
    case 2: e = assign_dispatch<2>(b, t, d, iter, unit_lo, unit_hi, kmax, rows_per_thread, st, kt); break;
    case 4: e = assign_dispatch<4>(b, t, d, iter, unit_lo, unit_hi, kmax, rows_per_thread, st, kt); break;
    case 8: e = assign_dispatch<8>(b, t, d, iter, unit_lo, unit_hi, kmax, rows_per_thread, st, kt); break;
    case 12: e = assign_dispatch<12>(b, t, d, iter, unit_lo, unit_hi, kmax, rows_per_thread, st, kt); break;
    case 16: e = assign_dispatch<16>(b, t, d, iter, unit_lo, unit_hi, kmax, rows_per_thread, st, kt); break;
    case 24: e = assign_dispatch<24>(b, t, d, iter, unit_lo, unit_hi, kmax, rows_per_thread, st, kt); break;
    case 32: e = assign_dispatch<32>(b, t, d, iter, unit_lo, unit_hi, kmax, rows_per_thread, st, kt); break;
    case 48: e = assign_dispatch<48>(b, t, d, iter, unit_lo, unit_hi, kmax, rows_per_thread, st, kt); break;
    case 64: e = assign_dispatch<64>(b, t, d, iter, unit_lo, unit_hi, kmax, rows_per_thread, st, kt); break;
    case 96: e = assign_dispatch<96>(b, t, d, iter, unit_lo, unit_hi, kmax, rows_per_thread, st, kt); break;
    case 128: e = assign_dispatch<128>(b, t, d, iter, unit_lo, unit_hi, kmax, rows_per_thread, st, kt); break;
    default: e = assign_dispatch<0>(b, t, d, iter, unit_lo, unit_hi, kmax, rows_per_thread, st, kt); break;
    }
    if (e != cudaSuccess) return e;
    kt->begin(st);
    if (d % 4 == 0) e = finalize_launch<4>(b, count_next, cen_lo, cen_hi, d, sm_count, keep, st);
    else if (d % 2 == 0) e = finalize_launch<2>(b, count_next, cen_lo, cen_hi, d, sm_count, keep, st);
    else e = finalize_launch<1>(b, count_next, cen_lo, cen_hi, d, sm_count, keep, st);
    kt->end(PSCL_K_LLOYD_FINALIZE, st);
    return e;
}

cudaError_t launch_seg_sse(const LloydBuffers &b, const SegTable &t, const int32_t *seg_unit0, int d, int kmax,
                           int prec, int32_t *labels, double *unit_sse, double *seg_sse, uint32_t *flags,
                           int sm_count, cudaStream_t st, KTimer *kt)
{
    const float *pts = b.pts, *centers = b.centers;
    cudaError_t e;
    if (seg_sse_tc_supported(b, t, d, kmax, prec)) {
        e = launch_seg_sse_tc(b, t, d, kmax, prec, labels, unit_sse, flags, sm_count, st, kt);
    } else if (d >= kTiledMinUnits && d <= kTiledMax && kmax >= kTiledCenters) {
        const size_t smem = tile_smem(d);
        if (const cudaError_t ea = cudaFuncSetAttribute(k_seg_sse_tiled, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) return ea;
        kt->begin(st);
        k_seg_sse_tiled<<<t.n_units, kThreads, smem, st>>>(pts, t, d, centers, labels, unit_sse);
        kt->end(PSCL_K_FINAL_SSE, st);
        e = cudaGetLastError();
    } else switch (pad_width(d)) {
    case 2: e = seg_sse_dispatch<2>(pts, t, d, centers, kmax, labels, unit_sse, st, kt); break;
    case 4: e = seg_sse_dispatch<4>(pts, t, d, centers, kmax, labels, unit_sse, st, kt); break;
    case 8: e = seg_sse_dispatch<8>(pts, t, d, centers, kmax, labels, unit_sse, st, kt); break;
    case 12: e = seg_sse_dispatch<12>(pts, t, d, centers, kmax, labels, unit_sse, st, kt); break;
    case 16: e = seg_sse_dispatch<16>(pts, t, d, centers, kmax, labels, unit_sse, st, kt); break;
    case 24: e = seg_sse_dispatch<24>(pts, t, d, centers, kmax, labels, unit_sse, st, kt); break;
    case 32: e = seg_sse_dispatch<32>(pts, t, d, centers, kmax, labels, unit_sse, st, kt); break;
    case 48: e = seg_sse_dispatch<48>(pts, t, d, centers, kmax, labels, unit_sse, st, kt); break;
    case 64: e = seg_sse_dispatch<64>(pts, t, d, centers, kmax, labels, unit_sse, st, kt); break;
    case 96: e = seg_sse_dispatch<96>(pts, t, d, centers, kmax, labels, unit_sse, st, kt); break;
    case 128: e = seg_sse_dispatch<128>(pts, t, d, centers, kmax, labels, unit_sse, st, kt); break;
    default: e = seg_sse_dispatch<0>(pts, t, d, centers, kmax, labels, unit_sse, st, kt); break;
    }
    if (e != cudaSuccess) return e;
    k_seg_sse_fold<<<(t.n_seg + 255) / 256, 256, 0, st>>>(unit_sse, seg_unit0, t.n_seg, seg_sse);
    return cudaGetLastError();
}

cudaError_t launch_final_sse(const float *x, int64_t n, int d, const float *centers, int k,
                             int32_t *labels, double *blk_sse, double *sse, uint32_t *ticket,
                             int sm_count, cudaStream_t st, KTimer *kt)
{
    if (d >= kTiledMin && d <= kTiledMax && k >= kTiledCenters) {
        const size_t smem = tile_smem(d);
        if (const cudaError_t ea = cudaFuncSetAttribute(k_final_sse_tiled, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) return ea;
        kt->begin(st);
        const cudaError_t e = sse_launch(k_final_sse_tiled, std::max(1, sse_grid(n, sm_count)), smem, ticket == nullptr, st,
                                         x, n, d, centers, k, labels, blk_sse, sse, ticket);
        kt->end(PSCL_K_FINAL_SSE, st);
        return e;
    }
    switch (pad_width(d)) {
    case 2: return sse_dispatch<2>(x, n, d, centers, k, labels, blk_sse, sse, ticket, sm_count, st, kt);
    case 4: return sse_dispatch<4>(x, n, d, centers, k, labels, blk_sse, sse, ticket, sm_count, st, kt);
    case 8: return sse_dispatch<8>(x, n, d, centers, k, labels, blk_sse, sse, ticket, sm_count, st, kt);
    case 12: return sse_dispatch<12>(x, n, d, centers, k, labels, blk_sse, sse, ticket, sm_count, st, kt);
    case 16: return sse_dispatch<16>(x, n, d, centers, k, labels, blk_sse, sse, ticket, sm_count, st, kt);
    case 24: return sse_dispatch<24>(x, n, d, centers, k, labels, blk_sse, sse, ticket, sm_count, st, kt);
    case 32: return sse_dispatch<32>(x, n, d, centers, k, labels, blk_sse, sse, ticket, sm_count, st, kt);
    case 48: return sse_dispatch<48>(x, n, d, centers, k, labels, blk_sse, sse, ticket, sm_count, st, kt);
    case 64: return sse_dispatch<64>(x, n, d, centers, k, labels, blk_sse, sse, ticket, sm_count, st, kt);
    case 96: return sse_dispatch<96>(x, n, d, centers, k, labels, blk_sse, sse, ticket, sm_count, st, kt);
    case 128: return sse_dispatch<128>(x, n, d, centers, k, labels, blk_sse, sse, ticket, sm_count, st, kt);
    default: return sse_dispatch<0>(x, n, d, centers, k, labels, blk_sse, sse, ticket, sm_count, st, kt);
    }
}

}  // namespace pscl
