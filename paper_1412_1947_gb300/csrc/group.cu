// Unequal-sized subclustering (Algorithm 2): after feature scaling, L and H are the
// points made of every attribute's lowest and highest value; the segment from L to H is
// cut into m equal pieces whose middles are the landmarks
//     l_i = float(L + ((i + 1/2) / m) (H - L))        (double arithmetic, stored as float)
// and every point joins its nearest landmark.  "Nearest" is the float64 squared distance
// of the peel (ascending attributes, one rounding per operation), the lower landmark index
// on ties.  As in the peel, each point's distances are computed in float32 with the bound
// |d32 - d64| <= eps d32 + 2^-120, eps = (d+4) 2^-23; only when that bound leaves more than
// one landmark in contention are those landmarks' float64 distances computed.
// The landmarks lie on a line at equal steps, so a point's projection on it leaves only the few
// around its place in contention (the bound: see k_group).  All m of them scored twice, each
// read once per point and attribute, took 0.8 ms at 500009 x 32 with 128 landmarks; the
// projection and three candidates leave the pass to the points' bytes.
//
// The subclusters are the groups in landmark order with their points in ascending index
// (a stable counting sort: per-tile histograms, a scan over (group, tile), and a stable
// scatter per tile with warp match), groups that nobody joins being left out.
#include "pscl_internal.cuh"

namespace pscl {
namespace {

constexpr int kTile = 1024;                  // points per tile of the counting sort

__global__ void k_landmarks(const double *mn, const double *mx, int d, int m, float *lm)
{
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < m * d; e += gridDim.x * blockDim.x) {
        const int i = e / d, a = e - i * d;
        const double t = __ddiv_rn((double)i + 0.5, (double)m);
        lm[e] = __double2float_rn(__dadd_rn(mn[a], __dmul_rn(t, __dsub_rn(mx[a], mn[a]))));
    }
}

template <int D>
__device__ __forceinline__ float dist32(const float *x, const float *l, int d)
{
    const int dd = D > 0 ? D : d;
    float acc = 0.0f;
#pragma unroll
    for (int a = 0; a < dd; a++) {
        const float t = __fsub_rn(x[a], l[a]);
        acc = __fmaf_rn(t, t, acc);
    }
    return acc;
}

__device__ __forceinline__ double dist64(const float *x, const float *l, int d)
{
    double s = 0.0;
    for (int a = 0; a < d; a++) {
        const double t = __dsub_rn((double)x[a], (double)l[a]);
        s = __dadd_rn(s, __dmul_rn(t, t));
    }
    return s;
}

// Group of every point, and per tile of kTile points the count of every group
// (cnt[g * ntiles + tile]).
//
// With c, e the first and last landmark and v = e - c, point x lies at p = (m - 1) (x - c) v /
// |v|^2 along the landmarks' indexes.  Landmark i is c + i v / (m - 1) but for its own rounding
// and the ends', at most 2^-23 M_a per attribute (M_a >= |L_a|, |H_a|; b their norm over the
// attributes), and |x - l_i| <= 2 |v| (x lies in the box of L and H, and |H - L| = m / (m - 1)
// |v|).  So with q >= |p' - p|, the error of the computed p', and i0 the landmark at p' (rounded,
// within 0 .. m - 1), one more than w steps away is farther than i0 by at least
//     |v|^2 / (m - 1)^2 (w + 1) (w - 2 q)  -  2 (4 |v| b + b^2 + 4 |v|^2 (d + 2) 2^-52),
// in float64 as defined, and cannot be the nearest where that is positive.  q: the differences
// and products round once each, the sum d times, and |v|^2 likewise: (3 d + 16) 2^-23 m.  All
// landmarks are scored where no w below m does (coincident ends), or one is all there are.
constexpr size_t kTableBytes = 100 * 1024;

template <int D>
__global__ void __launch_bounds__(256) k_group(const float *__restrict__ x, int64_t n, int d,
                                               const float *__restrict__ lm, int m, int32_t *group, uint32_t *cnt,
                                               int ntiles, int table)
{
    // [counts m | c, v: d each | the landmarks, d | 1 floats apart (table): lanes read several]
    extern __shared__ uint32_t hist[];
    __shared__ float s_vv[8], s_mm[8], s_scale;
    __shared__ int s_w, s_close;
    __shared__ uint16_t s_list[kTile];
    const int dd = D > 0 ? D : d, t = threadIdx.x, ds = dd | 1;
    float *sc = reinterpret_cast<float *>(hist + m), *sv = sc + dd, *sl = sv + dd;
    for (int g = t; g < m; g += blockDim.x) hist[g] = 0;
    float vv = 0.0f, mm = 0.0f;
    for (int a = t; a < dd; a += blockDim.x) {
        const float c = lm[a], e = lm[(size_t)(m - 1) * dd + a], v = __fsub_rn(e, c);
        sc[a] = c;
        sv[a] = v;
        vv = __fmaf_rn(v, v, vv);
        const float M = fmaxf(fabsf(c), fabsf(e)) + fabsf(v);
        mm = __fmaf_rn(M, M, mm);
    }
    if (table)
        for (int e = t; e < m * dd; e += blockDim.x) sl[e / dd * ds + e % dd] = lm[e];
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        vv += __shfl_xor_sync(0xffffffffu, vv, o);
        mm += __shfl_xor_sync(0xffffffffu, mm, o);
    }
    if ((t & 31) == 0) {
        s_vv[t >> 5] = vv;
        s_mm[t >> 5] = mm;
    }
    __syncthreads();
    if (t == 0) {
        vv = mm = 0.0f;
        for (int q = 0; q < 8; q++) {
            vv += s_vv[q];
            mm += s_mm[q];
        }
        // (float32 with a factor two of margin on the right-hand side)
        const float q2 = 2.0f * (float)(3 * dd + 16) * 0x1p-23f * (float)m;
        const float b = 0x1p-23f * sqrtf(mm / vv), r = (float)(m - 1) * (float)(m - 1);
        const float need = 2.0f * 2.0f * r * (4.0f * b + b * b + 4.0f * (float)(dd + 2) * 0x1p-52f);
        int w = m;
        if (m > 1 && vv > 0x1p-60f && need < r) {                  // NaN and coincident ends: all
            w = 1;
            while (w < m && !((float)(w + 1) * ((float)w - q2) >= need)) w++;
        }
        s_close = 0;
        s_w = w;
        s_scale = (float)(m - 1) / vv;
    }
    __syncthreads();
    const int w = s_w;
    const float scale = s_scale;
    const float eps = (float)(d + 4) * 0x1p-23f;
    const int64_t i0 = (int64_t)blockIdx.x * kTile;
    // point q of the tile; one whose best two the float32 bound cannot separate is put off
    // (exact: decided)
    auto place = [&](int q, bool exact) {
        const int64_t i = i0 + q;
        const float *xi = x + i * dd;
        float xv[D > 0 ? D : 1];
        if constexpr (D > 0 && D % 4 == 0) {
#pragma unroll
            for (int a = 0; a < D; a += 4) {
                const float4 v4 = __ldg(reinterpret_cast<const float4 *>(xi + a));
                xv[a] = v4.x;
                xv[a + 1] = v4.y;
                xv[a + 2] = v4.z;
                xv[a + 3] = v4.w;
            }
        } else if constexpr (D > 0) {
#pragma unroll
            for (int a = 0; a < D; a++) xv[a] = __ldg(&xi[a]);
        }
        const float *xp = D > 0 ? xv : xi;
        int lo = 0, hi = m - 1;
        if (w < m) {
            float p = 0.0f;
#pragma unroll
            for (int a = 0; a < dd; a++) p = __fmaf_rn(__fsub_rn(xp[a], sc[a]), sv[a], p);
            const int at = min(max(__float2int_rn(p * scale), 0), m - 1);
            lo = max(at - w, 0);
            hi = min(at + w, m - 1);
        }
        auto L = [&](int j) { return table ? sl + j * ds : lm + (size_t)j * dd; };
        float best = __int_as_float(0x7f800000), next = best;
        int bj = 0;
        for (int j = lo; j <= hi; j++) {
            const float v = dist32<D>(xp, L(j), dd);
            if (v < best) {
                next = best;
                best = v;
                bj = j;
            } else {
                next = fminf(next, v);
            }
        }
        // a landmark that the float32 bound cannot separate from the best: float64, as defined,
        // for those
        const float top = __fadd_ru(__fmul_ru(best, 1.0f + eps), 0x1p-120f);
        if (__fsub_rd(__fmul_rd(next, 1.0f - eps), 0x1p-120f) <= top) {
            if (!exact) {
                s_list[atomicAdd(&s_close, 1)] = (uint16_t)q;
                return;
            }
            double b64 = 0.0;
            int b = -1;
            for (int j = lo; j <= hi; j++) {
                const float v = dist32<D>(xp, L(j), dd);
                if (__fsub_rd(__fmul_rd(v, 1.0f - eps), 0x1p-120f) > top) continue;
                const double w64 = dist64(xi, lm + (size_t)j * dd, dd);
                if (b < 0 || w64 < b64) { b64 = w64; b = j; }
            }
            bj = b;
        }
        group[i] = bj;
        atomicAdd(&hist[bj], 1u);
    };
    const int rows = (int)min((int64_t)kTile, n - i0);
    for (int q = t; q < rows; q += blockDim.x) place(q, false);
    // those put off, side by side: found one at a time, the few of a tile took a float64 pass of
    // most of its warps (500009 x 32, m = 128: 106 -> 53 us)
    __syncthreads();
    for (int q = t; q < s_close; q += blockDim.x) place(s_list[q], true);
    __syncthreads();
    for (int g = t; g < m; g += blockDim.x) cnt[(size_t)g * ntiles + blockIdx.x] = hist[g];
}

// Exclusive scan of v over a block of 256 threads; total gets the sum.
__device__ __forceinline__ uint32_t scan256(uint32_t v, uint32_t &total)
{
    __shared__ uint32_t ws[8];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += u;
    }
    __syncthreads();
    if (lane == 31) ws[w] = inc;
    __syncthreads();
    uint32_t before = 0;
    total = 0;
#pragma unroll
    for (int q = 0; q < 8; q++) {
        if (q < w) before += ws[q];
        total += ws[q];
    }
    return before + inc - v;
}

// Exclusive scan of each group's counts over the tiles, in place, and its total: a block per
// group (one block for all of them took a barrier chain per 1024 counts: 62592 counts, 90 us).
__global__ void __launch_bounds__(256) k_group_scan(uint32_t *cnt, int m, int ntiles, uint32_t *total)
{
    for (int g = blockIdx.x; g < m; g += gridDim.x) {
        uint32_t *c = cnt + (size_t)g * ntiles;
        uint32_t run = 0;
        for (int b = 0; b < ntiles; b += 4 * 256) {
            uint32_t v[4], s = 0, tot;
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const int e = b + 4 * (int)threadIdx.x + q;
                v[q] = e < ntiles ? c[e] : 0u;
                s += v[q];
            }
            uint32_t at = run + scan256(s, tot);
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const int e = b + 4 * (int)threadIdx.x + q;
                if (e < ntiles) c[e] = at;
                at += v[q];
            }
            run += tot;
        }
        if (threadIdx.x == 0) total[g] = run;
    }
}

// Stable scatter of one tile: its points in order, 32 at a time (one warp, all its groups
// loaded first: a round trip for each 32 of them took 40 us).
__global__ void __launch_bounds__(32) k_group_scatter(const int32_t *group, int64_t n, const uint32_t *cnt,
                                                      const uint32_t *total, int m, int ntiles, uint32_t *perm)
{
    extern __shared__ uint32_t cur[];
    const int lane = threadIdx.x;
    const int64_t i0 = (int64_t)blockIdx.x * kTile;
    int gr[kTile / 32];
#pragma unroll
    for (int r = 0; r < kTile / 32; r++) {
        const int64_t i = i0 + r * 32 + lane;
        gr[r] = i < n ? __ldg(&group[i]) : -1;
    }
    uint32_t before = 0;                          // the points of the groups before
#pragma unroll 4
    for (int g0 = 0; g0 < m; g0 += 32) {
        const int g = g0 + lane;
        const uint32_t v = g < m ? __ldg(&total[g]) : 0u, c = g < m ? __ldg(&cnt[(size_t)g * ntiles + blockIdx.x]) : 0u;
        uint32_t inc = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t u = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += u;
        }
        if (g < m) cur[g] = before + inc - v + c;
        before += __shfl_sync(0xffffffffu, inc, 31);
    }
    __syncwarp();
#pragma unroll
    for (int r = 0; r < kTile / 32; r++) {
        const int g = gr[r];
        const uint32_t peers = __match_any_sync(0xffffffffu, g);
        if (g >= 0) perm[cur[g] + __popc(peers & ((1u << lane) - 1u))] = (uint32_t)(i0 + r * 32 + lane);
        __syncwarp();
        if (g >= 0 && lane == __ffs(peers) - 1) cur[g] += __popc(peers);
        __syncwarp();
    }
}

template <int D>
cudaError_t group_launch(const float *x, int64_t n, int d, const float *lm, int m, int32_t *group, uint32_t *cnt,
                         uint32_t *total, uint32_t *perm, cudaStream_t st)
{
    const int ntiles = (int)((n + kTile - 1) / kTile);
    const size_t hs = (size_t)m * sizeof(uint32_t), line = 2 * (size_t)d * sizeof(float);
    const size_t tab = (size_t)m * (d | 1) * sizeof(float);
    const int table = hs + line + tab <= kTableBytes;
    const size_t gs = hs + line + (table ? tab : 0);
    cudaError_t e = cudaFuncSetAttribute(k_group<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gs);
    if (e != cudaSuccess) return e;
    k_group<D><<<ntiles, 256, gs, st>>>(x, n, d, lm, m, group, cnt, ntiles, table);
    k_group_scan<<<m, 256, 0, st>>>(cnt, m, ntiles, total);
    e = cudaFuncSetAttribute(k_group_scatter, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)hs);
    if (e != cudaSuccess) return e;
    k_group_scatter<<<ntiles, 32, hs, st>>>(group, n, cnt, total, m, ntiles, perm);
    return cudaGetLastError();
}

}  // namespace

size_t group_cnt_words(int64_t n, int m) { return (size_t)m * (size_t)((n + kTile - 1) / kTile); }

cudaError_t launch_group_unequal(const float *x, int64_t n, int d, const double *lo, const double *hi, int m,
                                 float *lm, int32_t *group, uint32_t *cnt, uint32_t *total, uint32_t *perm,
                                 cudaStream_t st, KTimer *kt)
{
    kt->begin(st);
    k_landmarks<<<(m * d + 255) / 256, 256, 0, st>>>(lo, hi, d, m, lm);
    cudaError_t e;
    switch (d) {
    case 2: e = group_launch<2>(x, n, d, lm, m, group, cnt, total, perm, st); break;
    case 4: e = group_launch<4>(x, n, d, lm, m, group, cnt, total, perm, st); break;
    case 8: e = group_launch<8>(x, n, d, lm, m, group, cnt, total, perm, st); break;
    case 16: e = group_launch<16>(x, n, d, lm, m, group, cnt, total, perm, st); break;
    case 32: e = group_launch<32>(x, n, d, lm, m, group, cnt, total, perm, st); break;
    case 64: e = group_launch<64>(x, n, d, lm, m, group, cnt, total, perm, st); break;
    default: e = group_launch<0>(x, n, d, lm, m, group, cnt, total, perm, st); break;
    }
    kt->end(PSCL_K_PEEL, st);
    return e;
}

}  // namespace pscl
