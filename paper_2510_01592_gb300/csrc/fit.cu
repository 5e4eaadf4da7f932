// fit.cu -- cluster-parallel plane estimation (Sec. III.C, multi-plane
// estimation stages a-c), inlier refit and boundary polygons (Sec. III.C,
// boundary polygon generation), for all clusters of a batch at once.
//
//  k_hyp     stage a: one thread per (cluster, hypothesis): three sample
//            indices from Philox4x64-10, plane through the samples.
//  k_score   stage b: a persistent kernel; CTAs pull (cluster, point tile)
//            work items from an atomic queue, stage the tile in shared memory
//            and test every point against every hypothesis held in registers;
//            integer counts are summed in shared memory and added to global
//            memory with integer atomics (order-free, hence exact).  Large fits
//            take k_score_slab, which bounds most tests instead of making them.
//  k_select  stage c: max count, lowest hypothesis index on ties; in-plane
//            basis and hull origin.
//  k_extract inliers of the selected plane, centroid partial sums and the
//            extreme inliers along 16 integer directions (exact integer keys);
//            the CTA that completes a cluster forms its centroid and polygon.
//  k_filter  covariance partial sums; points strictly inside the 16-gon of
//            extreme points cannot be hull vertices and are dropped (the GPU
//            filtering step of the cited convex-hull method), the rest are
//            appended.
//  k_refit   per cluster: TLS refit from the partial sums (double-float sums,
//            adjugate power iteration).
//  k_hull    per cluster: a finer filter where many are left, then a sort of the
//            remaining quantised points in shared memory and Andrew's monotone
//            chain with exact int64 orientation tests (few points: a rank sort
//            and a test per point); gift wrapping over global memory when too
//            many remain for shared memory.
#include <climits>
#include <mutex>
#include <string>

#include "vm_internal.cuh"

namespace vmx {
namespace {

constexpr int kT = 256;
constexpr int kHullCap = 2048;   // hull candidates sorted in shared memory
constexpr int kSurvCap = 10240;  // first-filter survivors staged in shared memory: two CTAs of k_hull fit an SM

// ---------------------------------------------------------------- Philox
__device__ __forceinline__ void philox4x64_10(const unsigned long long ctr[4], const unsigned long long key[2],
                                              unsigned long long out[4]) {
    unsigned long long x0 = ctr[0], x1 = ctr[1], x2 = ctr[2], x3 = ctr[3];
    unsigned long long k0 = key[0], k1 = key[1];
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r) {
            k0 += 0x9E3779B97F4A7C15ull;
            k1 += 0xBB67AE8584CAA73Bull;
        }
        const unsigned long long m0 = 0xD2E7470EE14C6C93ull, m1 = 0xCA5A826395121157ull;
        const unsigned long long hi0 = __umul64hi(m0, x0), lo0 = m0 * x0;
        const unsigned long long hi1 = __umul64hi(m1, x2), lo1 = m1 * x2;
        x0 = hi1 ^ x1 ^ k0;
        x1 = lo1;
        x2 = hi0 ^ x3 ^ k1;
        x3 = lo0;
    }
    out[0] = x0; out[1] = x1; out[2] = x2; out[3] = x3;
}

__device__ __forceinline__ float plane_dist(float nx, float ny, float nz, float d, float px, float py, float pz) {
    return fabsf(__fmaf_rn(nz, pz, __fmaf_rn(ny, py, __fmaf_rn(nx, px, d))));
}

// Stage b for one point against a thread's R hypotheses: acc[r] += 1 when
// |n_r . p + d_r| <= eps (the fma chain of plane_dist).  The comparison is a
// set to all-ones / zero subtracted from the count: two instructions a test
// after the three fused multiply-adds.
template <int R>
__device__ __forceinline__ void count_point(const float4 (&pl)[R], float4 p, float eps, uint32_t (&acc)[R]) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const float dist = plane_dist(pl[r].x, pl[r].y, pl[r].z, pl[r].w, p.x, p.y, p.z);
        uint32_t t;
        asm("set.le.u32.f32 %0, %1, %2;" : "=r"(t) : "f"(dist), "f"(eps));
        acc[r] -= t;
    }
}

// Two points at once: the two masks come off the count in one three-input add.
template <int R>
__device__ __forceinline__ void count_points2(const float4 (&pl)[R], float4 p, float4 q, float eps,
                                              uint32_t (&acc)[R]) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const float a = plane_dist(pl[r].x, pl[r].y, pl[r].z, pl[r].w, p.x, p.y, p.z);
        const float b = plane_dist(pl[r].x, pl[r].y, pl[r].z, pl[r].w, q.x, q.y, q.z);
        uint32_t t, u;
        asm("set.le.u32.f32 %0, %1, %2;" : "=r"(t) : "f"(a), "f"(eps));
        asm("set.le.u32.f32 %0, %1, %2;" : "=r"(u) : "f"(b), "f"(eps));
        acc[r] = acc[r] - t - u;
    }
}

// The cluster of work item it: one load from the item -> cluster table k_hyp
// writes (item_cl), else a binary search over the item offsets.
__device__ __forceinline__ uint32_t find_cluster(const uint32_t* __restrict__ item_cl,
                                                 const uint32_t* __restrict__ item_off, uint32_t k, uint32_t it) {
    if (item_cl) return item_cl[it];
    uint32_t lo = 0, hi = k;  // largest c with item_off[c] <= it
    while (lo < hi) {
        const uint32_t mid = (lo + hi + 1) >> 1;
        if (item_off[mid] <= it) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// ---------------------------------------------------------------- stage a
// Also writes the item -> cluster table (item_cl, when not null): the thread
// of hypothesis 0 of each cluster fills its cluster's items.  from_all: the
// counts start at the cluster's size (k_score_slab takes the misses off).
__global__ void k_hyp(const float* __restrict__ pts, const uint32_t* __restrict__ off,
                      const uint32_t* __restrict__ labels, const uint32_t* __restrict__ kp, int H,
                      unsigned long long seed, uint32_t round, float4* __restrict__ hyp, uint8_t* __restrict__ valid,
                      uint32_t* __restrict__ counts, const uint32_t* __restrict__ item_off,
                      uint32_t* __restrict__ item_cl, uint32_t* __restrict__ lower, bool from_all) {
    pdl_gate();
    const uint32_t k = *kp;
    const size_t total = (size_t)k * H;
    for (size_t t = (size_t)blockIdx.x * kT + threadIdx.x; t < total; t += (size_t)gridDim.x * kT) {
        const uint32_t c = (uint32_t)(t / H), h = (uint32_t)(t % H);
        if (h == 0 && item_cl)
            for (uint32_t it = item_off[c], e = item_off[c + 1]; it < e; ++it) item_cl[it] = c;
        const uint32_t base = off[c], n = off[c + 1] - base;
        const uint32_t label = labels ? labels[c] : c;
        const unsigned long long ctr[4] = {label, h, round, 0ull}, key[2] = {seed, 0ull};
        unsigned long long r[4];
        philox4x64_10(ctr, key, r);
        const uint32_t i0 = (uint32_t)__umul64hi(r[0], n), i1 = (uint32_t)__umul64hi(r[1], n),
                       i2 = (uint32_t)__umul64hi(r[2], n);
        if (from_all && h == 0) lower[c] = 0;
        uint8_t ok = (i0 != i1) && (i0 != i2) && (i1 != i2);
        float4 pl = make_float4(0.0f, 0.0f, 0.0f, __int_as_float(0x7f800000));  // never an inlier
        if (ok) {
            const float* p0 = pts + 3 * ((size_t)base + i0);
            const float* p1 = pts + 3 * ((size_t)base + i1);
            const float* p2 = pts + 3 * ((size_t)base + i2);
            const float e1x = __fsub_rn(p1[0], p0[0]), e1y = __fsub_rn(p1[1], p0[1]), e1z = __fsub_rn(p1[2], p0[2]);
            const float e2x = __fsub_rn(p2[0], p0[0]), e2y = __fsub_rn(p2[1], p0[1]), e2z = __fsub_rn(p2[2], p0[2]);
            const float cx = __fmaf_rn(e1y, e2z, -__fmul_rn(e1z, e2y));
            const float cy = __fmaf_rn(e1z, e2x, -__fmul_rn(e1x, e2z));
            const float cz = __fmaf_rn(e1x, e2y, -__fmul_rn(e1y, e2x));
            const float nn = __fmaf_rn(cz, cz, __fmaf_rn(cy, cy, __fmul_rn(cx, cx)));
            if (nn > 0.0f) {
                const float inv = __fdiv_rn(1.0f, __fsqrt_rn(nn));
                const float nx = __fmul_rn(cx, inv), ny = __fmul_rn(cy, inv), nz = __fmul_rn(cz, inv);
                const float d = -__fmaf_rn(nz, p0[2], __fmaf_rn(ny, p0[1], __fmul_rn(nx, p0[0])));
                pl = make_float4(nx, ny, nz, d);
            } else {
                ok = 0;
            }
        }
        hyp[t] = pl;
        valid[t] = ok;
        counts[t] = from_all && fabsf(pl.w) < __int_as_float(0x7f800000) ? n : 0u;  // no point is near any other plane
    }
}

// ---------------------------------------------------------------- stage c
// The record of cluster c from its best (count << 32 | ~h) key (0: no valid
// hypothesis): the selected plane, the in-plane basis and the hull origin.
__device__ __forceinline__ void select_record(uint32_t c, unsigned long long best, const float* __restrict__ pts,
                                              const uint32_t* __restrict__ off, int H,
                                              const float4* __restrict__ hyp, FitCluster* __restrict__ cl) {
    FitCluster f;
    memset(&f, 0, sizeof(f));
    const uint32_t n = off[c + 1] - off[c];
    if (best != 0) {
        const int h = (int)(~(uint32_t)(best & 0xffffffffu));
        const float4 pl = hyp[(size_t)c * H + h];
        f.best_h = h;
        f.n[0] = pl.x; f.n[1] = pl.y; f.n[2] = pl.z; f.d = pl.w;
        f.inliers = (uint32_t)(best >> 32);
        const float nx = pl.x, ny = pl.y, nz = pl.z;
        float ux, uy, uz;
        if (fabsf(nx) < 0.9f) { ux = 0.0f; uy = -nz; uz = ny; }  // e_x cross n
        else { ux = nz; uy = 0.0f; uz = -nx; }                   // e_y cross n
        const float ul = __fmaf_rn(uz, uz, __fmaf_rn(uy, uy, __fmul_rn(ux, ux)));
        const float ui = __fdiv_rn(1.0f, __fsqrt_rn(ul));
        ux = __fmul_rn(ux, ui); uy = __fmul_rn(uy, ui); uz = __fmul_rn(uz, ui);
        f.u[0] = ux; f.u[1] = uy; f.u[2] = uz;
        f.v[0] = __fmaf_rn(ny, uz, -__fmul_rn(nz, uy));
        f.v[1] = __fmaf_rn(nz, ux, -__fmul_rn(nx, uz));
        f.v[2] = __fmaf_rn(nx, uy, -__fmul_rn(ny, ux));
    } else {
        f.best_h = -1;
    }
    if (n) {
        const float* p = pts + 3 * (size_t)off[c];
        f.o[0] = p[0]; f.o[1] = p[1]; f.o[2] = p[2];
    }
    cl[c] = f;
}

// This thread's best (count << 32 | ~h) key over hypotheses h = i, i + step,
// ... of cluster c (counts read from L2: other CTAs added them).
__device__ __forceinline__ unsigned long long best_key(uint32_t c, int i, int step, int H,
                                                       const uint8_t* __restrict__ valid,
                                                       const uint32_t* __restrict__ counts) {
    unsigned long long best = 0;  // 0 = none
    for (int h = i; h < H; h += step) {
        const size_t t = (size_t)c * H + h;
        if (valid[t]) {
            const unsigned long long key = ((unsigned long long)__ldcg(counts + t) << 32) | (uint32_t)(~(uint32_t)h);
            best = key > best ? key : best;
        }
    }
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
        const unsigned long long o = __shfl_xor_sync(0xffffffffu, best, s);
        best = o > best ? o : best;
    }
    return best;
}

// Stage c for cluster c by a whole CTA of kT threads (wbest: kT / 32 words
// of shared memory): maximum count, lowest hypothesis index on ties.
__device__ __forceinline__ void select_cta(uint32_t c, const float* __restrict__ pts, const uint32_t* __restrict__ off,
                                           int H, const float4* __restrict__ hyp, const uint8_t* __restrict__ valid,
                                           const uint32_t* __restrict__ counts, FitCluster* __restrict__ cl,
                                           unsigned long long* wbest) {
    unsigned long long best = best_key(c, threadIdx.x, kT, H, valid, counts);
    if ((threadIdx.x & 31) == 0) wbest[threadIdx.x >> 5] = best;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kT / 32; ++w) best = wbest[w] > best ? wbest[w] : best;
        select_record(c, best, pts, off, H, hyp, cl);
    }
    __syncthreads();
}

__global__ void k_select(const float* __restrict__ pts, const uint32_t* __restrict__ off,
                         const uint32_t* __restrict__ kp, int H, const float4* __restrict__ hyp,
                         const uint8_t* __restrict__ valid, const uint32_t* __restrict__ counts,
                         FitCluster* __restrict__ cl) {
    pdl_gate();
    const uint32_t k = *kp;
    __shared__ unsigned long long wbest[kT / 32];
    for (uint32_t c = blockIdx.x; c < k; c += gridDim.x) select_cta(c, pts, off, H, hyp, valid, counts, cl, wbest);
}

// Per-cluster completion: every work item of a cluster, after its results
// are visible device-wide, counts itself done; the CTA that completes the
// cluster's last item runs the cluster's next serial step (the centroid after
// extraction, the refit after the filter) in place of a kernel of its own.
// done: two counters a cluster, cleared before the fit.
__device__ __forceinline__ bool cta_last_item(uint32_t* done, uint32_t n_items, uint32_t* flag) {
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) *flag = atomicAdd(done, 1u) + 1u == n_items;
    __syncthreads();
    const bool last = *flag != 0u;
    if (last) __threadfence();
    return last;
}

// ---------------------------------------------------------------- stage b
template <int R>
__global__ void __launch_bounds__(kT) k_score(const float* __restrict__ pts, const uint32_t* __restrict__ off,
                                              const uint32_t* __restrict__ item_off,
                                              const uint32_t* __restrict__ item_cl, const uint32_t* __restrict__ kp,
                                              int H, const uint32_t* __restrict__ tile,
                                              const float4* __restrict__ hyp, uint32_t* __restrict__ counts,
                                              uint32_t* __restrict__ queue, float eps) {
    pdl_wait();
    const uint32_t k = *kp;
    const int T = (int)*tile;
    extern __shared__ float4 sp[];                // T staged points
    uint32_t* red = reinterpret_cast<uint32_t*>(sp + T);  // [P][G*R]
    __shared__ uint32_t s_item;
    const int G = (H + R - 1) / R;                // threads per point subset
    const int P = kT / G;                         // point subsets
    const int g = threadIdx.x / G, j = threadIdx.x % G;
    const bool active = g < P;
    const uint32_t n_items = item_off[k];
    for (int guard = 0; guard < kLoopCap; ++guard) {
        __syncthreads();
        if (threadIdx.x == 0) s_item = atomicAdd(queue, 1u);
        __syncthreads();
        const uint32_t it = s_item;
        if (it >= n_items) break;
        const uint32_t c = find_cluster(item_cl, item_off, k, it);
        const uint32_t start = off[c] + (it - item_off[c]) * (uint32_t)T;
        const uint32_t end = min(off[c + 1], start + (uint32_t)T);
        const int cnt = (int)(end - start);
        for (int q = threadIdx.x; q < cnt; q += kT) {
            const float* p = pts + 3 * ((size_t)start + q);
            sp[q] = make_float4(p[0], p[1], p[2], 0.0f);
        }
        float4 pl[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int h = j * R + r;
            pl[r] = (active && h < H) ? hyp[(size_t)c * H + h]
                                      : make_float4(0.0f, 0.0f, 0.0f, __int_as_float(0x7f800000));
        }
        __syncthreads();
        uint32_t acc[R];
#pragma unroll
        for (int r = 0; r < R; ++r) acc[r] = 0;
        if (active) {
            for (int q = g; q < cnt; q += P) count_point<R>(pl, sp[q], eps, acc);
#pragma unroll
            for (int r = 0; r < R; ++r) red[g * (G * R) + j * R + r] = acc[r];
        }
        __syncthreads();
        for (int h = threadIdx.x; h < H; h += kT) {
            uint32_t s = 0;
            for (int q = 0; q < P; ++q) s += red[q * (G * R) + h];
            if (s) atomicAdd(&counts[(size_t)c * H + h], s);
        }
    }
}

// In-plane coordinates relative to the origin in units of 2^-16 m, before
// rounding: quantise() rounds exactly these values, so each lies within half
// a unit of its quantised coordinate.
__device__ __forceinline__ float2 plane_coords(const FitCluster& f, float px, float py, float pz) {
    const float qx = __fsub_rn(px, f.o[0]), qy = __fsub_rn(py, f.o[1]), qz = __fsub_rn(pz, f.o[2]);
    const float a = __fmaf_rn(qz, f.u[2], __fmaf_rn(qy, f.u[1], __fmul_rn(qx, f.u[0])));
    const float b = __fmaf_rn(qz, f.v[2], __fmaf_rn(qy, f.v[1], __fmul_rn(qx, f.v[0])));
    return make_float2(__fmul_rn(a, 65536.0f), __fmul_rn(b, 65536.0f));
}

// Quantised in-plane coordinates (units of 2^-16 m) relative to the origin.
__device__ __forceinline__ int2 quantise(const FitCluster& f, float px, float py, float pz) {
    const float2 w = plane_coords(f, px, py, pz);
    return make_int2(__float2int_rn(w.x), __float2int_rn(w.y));
}

// The 16 filter directions, counter-clockwise: (1,0) (2,1) (1,1) (1,2) (0,1)
// (-1,2) (-1,1) (-2,1) (-1,0) (-2,-1) (-1,-1) (-1,-2) (0,-1) (1,-2) (1,-1) (2,-1);
// direction d + 8 is direction d negated.  With |X|, |Y| < 2^28 every value
// fits in int32.
__device__ __forceinline__ int32_t dir_value(int dir, int2 p) {
    const int a = (dir == 0 || dir == 2 || dir == 3 || dir == 14 || dir == 13) ? 1
                : (dir == 1 || dir == 15) ? 2
                : (dir == 4 || dir == 12) ? 0
                : (dir == 7 || dir == 9) ? -2 : -1;
    const int b = (dir == 0 || dir == 8) ? 0
                : (dir == 1 || dir == 2 || dir == 4 || dir == 6 || dir == 7) ? 1
                : (dir == 3 || dir == 5) ? 2
                : (dir == 11 || dir == 13) ? -2 : -1;
    return a * p.x + b * p.y;
}

__device__ __forceinline__ unsigned long long ext_key(int32_t v, uint32_t idx) {
    return ((unsigned long long)((uint32_t)v ^ 0x80000000u) << 32) | idx;
}

template <typename Tv>
__device__ __forceinline__ Tv block_sum(Tv v, Tv* sh) {
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) v += __shfl_xor_sync(0xffffffffu, v, s);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    Tv t = 0;
    if (threadIdx.x == 0)
        for (int w = 0; w < kT / 32; ++w) t += sh[w];
    return t;  // valid in thread 0
}

// Partial sums of the refit are formed per 256-point chunk of a cluster (one
// point per thread, a fixed reduction tree), whatever the work-item tile: the
// refit is then the same for every scoring schedule, and a cluster's result
// does not depend on the batch it is fitted in.
constexpr uint32_t kChunk = kT;

// Per-chunk sums in a fixed order without a barrier per chunk: each warp
// reduces its 32 values with a shuffle tree and parks the result in shared
// memory (wp[chunk][warp][value]); after the item's last chunk one barrier,
// then thread j adds chunk j's eight warp results in warp order.
constexpr int kMaxChunksPerItem = 16384 / (int)kChunk;

// The warp tree is the butterfly over lane offsets 16, 8, 4, 2, 1 for every
// value, transposed: at each of the first levels a lane keeps half of its
// values and sends the other half to its partner, which keeps the opposite
// half, so NV values (padded to P = 4 or 8) take 2 + 1 + 3 (P = 4) or
// 4 + 2 + 1 + 2 (P = 8) shuffles instead of 5 NV.  Each partial sum is
// the one the plain butterfly forms at that level (a + b = b + a exactly),
// so the totals are bit-identical to it.  Value e ends in the lanes whose top
// log2(P) lane bits equal e.
template <int NV>
__device__ __forceinline__ void warp_park(float (&v)[NV], float* wp, uint32_t j) {
    static_assert(NV == 4 || NV == 6, "4 or 6 values");
    constexpr int P = NV == 4 ? 4 : 8;
    constexpr int L = NV == 4 ? 2 : 3;  // log2(P): halving levels at offsets 16 .. 32 >> L
    const int lane = threadIdx.x & 31;
    float x[P];
#pragma unroll
    for (int e = 0; e < P; ++e) x[e] = e < NV ? v[e] : 0.0f;
#pragma unroll
    for (int lv = 0; lv < L; ++lv) {
        const int s = 16 >> lv, h = P >> (lv + 1);
        const bool up = (lane & s) != 0;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const float keep = up ? x[h + i] : x[i];
            const float send = up ? x[i] : x[h + i];
            x[i] = keep + __shfl_xor_sync(0xffffffffu, send, s);
        }
    }
#pragma unroll
    for (int s = 16 >> L; s > 0; s >>= 1) x[0] += __shfl_xor_sync(0xffffffffu, x[0], s);
    const int e = (lane >> (5 - L)) & (P - 1);
    if ((lane & ((32 >> L) - 1)) == 0 && e < NV) wp[(j * (kT / 32) + (threadIdx.x >> 5)) * NV + e] = x[0];
}

template <int NV>
__device__ __forceinline__ void chunks_out(const float* wp, uint32_t n_chunks, float* dst /* [chunk][10] */,
                                           int first) {
    __syncthreads();
    for (uint32_t j = threadIdx.x; j < n_chunks; j += kT) {
        float t[NV];
#pragma unroll
        for (int e = 0; e < NV; ++e) t[e] = 0.0f;
        for (int w = 0; w < kT / 32; ++w)
#pragma unroll
            for (int e = 0; e < NV; ++e) t[e] += wp[(j * (kT / 32) + w) * NV + e];
#pragma unroll
        for (int e = 0; e < NV; ++e) dst[(size_t)j * 10 + first + e] = t[e];
    }
    __syncthreads();
}

// Double-float arithmetic: a value is hi + lo with |lo| at most half an ulp of
// hi, about 46 significant bits, on the FP32 pipes (FP64 is a slow path on
// this part).  Built from the error-free transformations TwoSum (Knuth) and
// TwoProduct (Dekker; exact here with an fma).
struct df2 {
    float hi, lo;
};
__device__ __forceinline__ df2 df_two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ df2 df_fast_two_sum(float a, float b) {  // requires |a| >= |b| or a == 0
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ df2 df_add(df2 x, df2 y) {
    df2 s = df_two_sum(x.hi, y.hi);
    const df2 t = df_two_sum(x.lo, y.lo);
    s = df_fast_two_sum(s.hi, __fadd_rn(s.lo, t.hi));
    return df_fast_two_sum(s.hi, __fadd_rn(s.lo, t.lo));
}
__device__ __forceinline__ df2 df_neg(df2 x) { return {-x.hi, -x.lo}; }
__device__ __forceinline__ df2 df_sub(df2 x, df2 y) { return df_add(x, df_neg(y)); }
__device__ __forceinline__ df2 df_mul(df2 x, df2 y) {
    const float p = __fmul_rn(x.hi, y.hi);
    float e = __fmaf_rn(x.hi, y.hi, -p);
    e = __fmaf_rn(x.hi, y.lo, e);
    e = __fmaf_rn(x.lo, y.hi, e);
    return df_fast_two_sum(p, e);
}
__device__ __forceinline__ df2 df_mulf(df2 x, float y) { return df_mul(x, df2{y, 0.0f}); }
// x / n for a count n < 2^24 (exact in FP32): one quotient, its exact
// residual, one correction.
__device__ __forceinline__ df2 df_div_count(df2 x, uint32_t n) {
    const float fn = (float)n;
    const float q1 = __fdiv_rn(x.hi, fn);
    const df2 r = df_sub(x, df2{__fmul_rn(q1, fn), __fmaf_rn(q1, fn, -__fmul_rn(q1, fn))});
    return df_fast_two_sum(q1, __fdiv_rn(r.hi, fn));
}
__device__ __forceinline__ df2 df_shfl_xor(df2 x, int o) {
    return {__shfl_xor_sync(0xffffffffu, x.hi, o), __shfl_xor_sync(0xffffffffu, x.lo, o)};
}

// Sums NV double-float values over a CTA in a fixed order: a shuffle tree in
// each warp, then the warps' results in warp order, a thread per value.  The
// totals end in tot (shared, valid after the call's last barrier); sh: NV * (kT
// / 32) entries of shared memory.  Rolled loops: this code runs once a cluster,
// and fetching it unrolled (10 KB) took longer than running it.
template <int NV>
__device__ __forceinline__ void block_df_sum(df2 (&v)[NV], df2* sh, df2* tot) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll 1
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int e = 0; e < NV; ++e) v[e] = df_add(v[e], df_shfl_xor(v[e], o));
    if (lane == 0)
#pragma unroll
        for (int e = 0; e < NV; ++e) sh[e * (kT / 32) + w] = v[e];
    __syncthreads();
    if (threadIdx.x < NV) {
        const df2* s = sh + threadIdx.x * (kT / 32);
        df2 t = s[0];
#pragma unroll 1
        for (int q = 1; q < kT / 32; ++q) t = df_add(t, s[q]);
        tot[threadIdx.x] = t;
    }
    __syncthreads();
}

__device__ __forceinline__ long long cross3(int2 o, int2 a, int2 b) {
    return (long long)(a.x - o.x) * (long long)(b.y - o.y) - (long long)(a.y - o.y) * (long long)(b.x - o.x);
}

// Forms cluster c's polygon, by one warp: a lane per direction.  A cluster with
// inliers has an extreme in every direction, one without in none.  f: the
// cluster's plane; its extremes are read from L2 (other CTAs wrote them).
__device__ __forceinline__ void poly_warp(const FitCluster& f, const float* __restrict__ pts, uint32_t base,
                                          FitPoly* __restrict__ out) {
    const int lane = threadIdx.x & 31, d = lane & 15;
    const unsigned long long key = __ldcg(&f.ext[d]);
    int2 xy = make_int2(0, 0);
    if (key) {
        const float* p = pts + 3 * ((size_t)base + (uint32_t)(key & 0xffffffffu));
        xy = quantise(f, p[0], p[1], p[2]);
    }
    const int px = __shfl_sync(0xffffffffu, xy.x, d ? d - 1 : 0), py = __shfl_sync(0xffffffffu, xy.y, d ? d - 1 : 0);
    const uint32_t keep = __ballot_sync(0xffffffffu, key && lane < 16 && (d == 0 || xy.x != px || xy.y != py));
    int m = __popc(keep);
    // vertex i: the i-th kept direction's extreme
    uint32_t rest = keep;
    for (int i = 0; i < lane && i < kFiltDirs; ++i) rest &= rest - 1;
    const int src = rest ? __ffs(rest) - 1 : 0;
    const int ax = __shfl_sync(0xffffffffu, xy.x, src), ay = __shfl_sync(0xffffffffu, xy.y, src);
    const int lx = __shfl_sync(0xffffffffu, ax, m ? m - 1 : 0), ly = __shfl_sync(0xffffffffu, ay, m ? m - 1 : 0);
    const int fx = __shfl_sync(0xffffffffu, ax, 0), fy = __shfl_sync(0xffffffffu, ay, 0);
    if (m > 1 && lx == fx && ly == fy) --m;
    const int nx0 = __shfl_sync(0xffffffffu, ax, lane + 1 < m ? lane + 1 : 0);
    const int ny0 = __shfl_sync(0xffffffffu, ay, lane + 1 < m ? lane + 1 : 0);
    long long area2 = lane < m ? (long long)ax * ny0 - (long long)ay * nx0 : 0ll;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) area2 += __shfl_xor_sync(0xffffffffu, area2, o);
    if (m < 3 || area2 <= 0) m = 0;
    // |X|, |Y| of every inlier: at most the extremes along +-x (directions 0, 8), +-y (4, 12)
    int mx = key && !(d & 3) ? abs((int)((uint32_t)(key >> 32) ^ 0x80000000u)) : 0;
    mx = __reduce_max_sync(0xffffffffu, mx);
    const float sM = (float)mx + 1.0f;
    if (lane < kFiltDirs) {
        float4 e = make_float4(0.0f, 0.0f, 2.0f, 0.0f);
        if (lane < m) {
            const long long ex = (long long)nx0 - ax, ey = (long long)ny0 - ay;
            const long long cc = (long long)((unsigned long long)ex * (unsigned long long)(long long)ay -
                                             (unsigned long long)ey * (unsigned long long)(long long)ax);
            const float exf = (float)ex, eyf = (float)ey, cf = (float)cc;
            const float sum = fabsf(exf) + fabsf(eyf);
            const float E = 2.0f * (0.5f * sum + 4.76837158203125e-7f * (sum * sM + fabsf(cf)) + 1.0f);
            e = make_float4(__fdiv_rn(exf, E), -__fdiv_rn(eyf, E), -__fdiv_rn(cf, E), 0.0f);
            out->pt[lane] = make_int2(ax, ay);
            if (lane == m - 1) out->pt[m] = make_int2(fx, fy);
        }
        out->edge[lane] = e;
    }
    if (lane == 0) out->m = m;
}

// Inlier count and centroid of cluster c by a whole CTA: the per-chunk
// partial sums (read from L2: other CTAs wrote them) added in double-float in
// a fixed order (thread-strided, then block_df_sum), so the result does not
// depend on scheduling.  The centroid is kept as (hi, lo) per axis.  The last
// warp forms the filter polygon meanwhile.
struct CentroidShared {
    df2 sh[3 * (kT / 32)], tot[3];
    uint32_t n[kT / 32];
};
__device__ __forceinline__ void centroid_cta(uint32_t c, const float* __restrict__ pts,
                                             const uint32_t* __restrict__ off, const uint32_t* __restrict__ item_off,
                                             uint32_t cpt, const float* __restrict__ part,
                                             FitCluster* __restrict__ cl, float* __restrict__ cen,
                                             FitPoly* __restrict__ poly, CentroidShared& sm) {
    df2 v[3] = {{0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}};
    uint32_t n = 0;
    const uint32_t base = item_off[c] * cpt, nch = (off[c + 1] - off[c] + kChunk - 1) / kChunk;
#pragma unroll 2
    for (uint32_t j = threadIdx.x; j < nch; j += kT) {
        const float* pp = part + (size_t)(base + j) * 10;
        n += (uint32_t)__ldcg(pp);
        v[0] = df_add(v[0], df2{__ldcg(pp + 1), 0.0f});
        v[1] = df_add(v[1], df2{__ldcg(pp + 2), 0.0f});
        v[2] = df_add(v[2], df2{__ldcg(pp + 3), 0.0f});
    }
    n = __reduce_add_sync(0xffffffffu, n);
    if ((threadIdx.x & 31) == 0) sm.n[threadIdx.x >> 5] = n;
    block_df_sum<3>(v, sm.sh, sm.tot);
    FitCluster& f = cl[c];
    if (threadIdx.x >= kT - 32) poly_warp(f, pts, off[c], poly + c);
    if (threadIdx.x < 3) {
        n = 0;
#pragma unroll
        for (int q = 0; q < kT / 32; ++q) n += sm.n[q];
        df2 x{f.o[threadIdx.x], 0.0f};
        if (n) x = df_add(x, df_div_count(sm.tot[threadIdx.x], n));
        float* ce = cen + 6 * (size_t)c + 2 * threadIdx.x;
        ce[0] = x.hi;
        ce[1] = x.lo;
        f.c[threadIdx.x] = x.hi;
        if (threadIdx.x == 0) f.inliers = n;
    }
    __syncthreads();  // shared partials reused next
}

// After an extraction item of cluster c: the CTA that completes the cluster's
// last item computes its centroid (out of line: the item loop keeps its
// registers).
__device__ __noinline__ void extract_tail(uint32_t c, const float* __restrict__ pts, const uint32_t* __restrict__ off,
                                          const uint32_t* __restrict__ item_off, uint32_t cpt,
                                          const float* __restrict__ part, FitCluster* __restrict__ cl,
                                          float* __restrict__ cen, FitPoly* __restrict__ poly,
                                          uint32_t* __restrict__ done) {
    __shared__ CentroidShared sm;
    __shared__ uint32_t s_last;
    if (cta_last_item(done + 2 * (size_t)c, item_off[c + 1] - item_off[c], &s_last))
        centroid_cta(c, pts, off, item_off, cpt, part, cl, cen, poly, sm);
}

// Inliers, centroid partials (relative to the origin) and the extreme inliers
// along the 16 filter directions (reduced per CTA, then one atomicMax each: the
// items of a large cluster meet on its 16 words).
// kTail: the CTA that completes a cluster's last item computes its centroid
// (done: the per-cluster completion counters).  Loads in flight bound it, so
// registers are held to what lets a small fit's items, four an SM, all run at
// once (a walk map 13.2 -> 11 us, 16 clusters 14.2 -> 10.9), and a large fit's
// CTAs be five an SM (2,000 clusters 376 -> 349 us); the few spilled words cost
// less.
template <bool kTail>
__global__ void __launch_bounds__(kT, kTail ? 4 : 5)
k_extract(const float* __restrict__ pts, const uint32_t* __restrict__ off, const uint32_t* __restrict__ item_off,
          const uint32_t* __restrict__ item_cl, const uint32_t* __restrict__ kp, const uint32_t* __restrict__ tile,
          FitCluster* __restrict__ cl, uint8_t* __restrict__ inlier, float* __restrict__ part, float eps,
          uint32_t* __restrict__ err, uint32_t* __restrict__ done, float* __restrict__ cen,
          FitPoly* __restrict__ poly) {
    pdl_gate();
    const uint32_t k = *kp, T = *tile;
    __shared__ float wp[kMaxChunksPerItem * (kT / 32) * 4];
    __shared__ unsigned long long wext[kT / 32][kFiltDirs];
    const uint32_t n_items = item_off[k];
    const uint32_t cpt = T / kChunk;  // chunks per work item
    for (uint32_t it = blockIdx.x; it < n_items; it += gridDim.x) {
        const uint32_t c = find_cluster(item_cl, item_off, k, it);
        const FitCluster f = cl[c];
        const uint32_t start = off[c] + (it - item_off[c]) * T;
        const uint32_t end = min(off[c + 1], start + T);
        // per thread and direction d < 8: the largest value and its point (the
        // last one, i.e. the largest index, among equal values: points come in
        // index order), and the smallest value and its point; direction d + 8
        // is direction d negated, so its key is (-smallest, index)
        int vmax[kFiltDirs / 2], imax[kFiltDirs / 2], vmin[kFiltDirs / 2], imin[kFiltDirs / 2];
#pragma unroll
        for (int d = 0; d < kFiltDirs / 2; ++d) {
            vmax[d] = INT_MIN;
            vmin[d] = INT_MAX;
            imax[d] = imin[d] = 0;
        }
        bool big = false;
        // chunk within the item; its slot is it * cpt + j (item_off[c] * cpt + its chunk in the cluster)
        uint32_t j = 0;
#pragma unroll 4
        for (uint32_t q0 = start; q0 < end; q0 += kChunk, ++j) {  // unrolled: later chunks' loads go out early
            const uint32_t q = q0 + threadIdx.x;
            float v[4] = {0.0f, 0.0f, 0.0f, 0.0f};  // count, sum (p - o)
            if (q < end) {
                const float px = pts[3 * (size_t)q], py = pts[3 * (size_t)q + 1], pz = pts[3 * (size_t)q + 2];
                const bool in = f.best_h >= 0 && plane_dist(f.n[0], f.n[1], f.n[2], f.d, px, py, pz) <= eps;
                inlier[q] = in;
                if (in) {
                    v[0] = 1.0f;
                    v[1] = __fsub_rn(px, f.o[0]);
                    v[2] = __fsub_rn(py, f.o[1]);
                    v[3] = __fsub_rn(pz, f.o[2]);
                    const int2 xy = quantise(f, px, py, pz);
                    big |= (abs(xy.x) >= (1 << 28)) | (abs(xy.y) >= (1 << 28));
                    const int idx = (int)(q - off[c]);
#pragma unroll
                    for (int d = 0; d < kFiltDirs / 2; ++d) {
                        const int val = dir_value(d, xy);
                        if (val >= vmax[d]) { vmax[d] = val; imax[d] = idx; }
                        if (val <= vmin[d]) { vmin[d] = val; imin[d] = idx; }
                    }
                }
            }
            warp_park<4>(v, wp, j);
        }
        chunks_out<4>(wp, j, part + (size_t)it * cpt * 10, 0);  // slot 0 holds the count (at most 256: exact)
        if (big) atomicOr(err, kErrOverflow);
        // the warp's largest key per direction (the extreme value, then the
        // largest index among the lanes that hold it), then the CTA's
        const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
        for (int d = 0; d < kFiltDirs / 2; ++d) {
            const int wmax = __reduce_max_sync(0xffffffffu, vmax[d]);
            const int wimax = __reduce_max_sync(0xffffffffu, vmax[d] == wmax ? imax[d] : 0);
            const int wmin = __reduce_min_sync(0xffffffffu, vmin[d]);
            const int wimin = __reduce_max_sync(0xffffffffu, vmin[d] == wmin ? imin[d] : 0);
            if (lane == d) wext[w][d] = wmax != INT_MIN ? ext_key(wmax, (uint32_t)wimax) : 0ull;
            if (lane == d + 8) wext[w][d + 8] = wmin != INT_MAX ? ext_key(-wmin, (uint32_t)wimin) : 0ull;
        }
        __syncthreads();
        if (threadIdx.x < kFiltDirs) {
            unsigned long long key = 0;
#pragma unroll
            for (int q = 0; q < kT / 32; ++q) key = wext[q][threadIdx.x] > key ? wext[q][threadIdx.x] : key;
            if (key) atomicMax(&cl[c].ext[threadIdx.x], key);
        }
        __syncthreads();
        if constexpr (kTail) extract_tail(c, pts, off, item_off, cpt, part, cl, cen, poly, done);
    }
}

struct RefitShared {
    df2 sh[6 * (kT / 32)], tot[6];
};
__device__ __forceinline__ void refit_cta(uint32_t c, const uint32_t* __restrict__ off,
                                          const uint32_t* __restrict__ item_off, uint32_t cpt,
                                          const float* __restrict__ part, const float* __restrict__ cen,
                                          FitCluster* __restrict__ cl, RefitShared& sm);

// After a filter item of cluster c: the CTA that completes the cluster's last
// item refits its plane (out of line).
__device__ __noinline__ void filter_tail(uint32_t c, const uint32_t* __restrict__ off,
                                         const uint32_t* __restrict__ item_off, uint32_t cpt,
                                         const float* __restrict__ part, const float* __restrict__ cen,
                                         FitCluster* __restrict__ cl, uint32_t* __restrict__ done) {
    __shared__ RefitShared sm;
    __shared__ uint32_t s_last;
    if (cta_last_item(done + 2 * (size_t)c + 1, item_off[c + 1] - item_off[c], &s_last))
        refit_cta(c, off, item_off, cpt, part, cen, cl, sm);
}

// Covariance partials about the centroid, and the 16-gon filter: inliers
// strictly inside the polygon through the 16 extreme inliers cannot be hull
// vertices; the others are appended to the cluster's survivor list.  Each
// warp gathers its survivors in shared memory and reserves room in the list
// with one atomic per kSurvBuf survivors (usually one per work item) instead
// of one returned atomic per chunk on the loop's critical path.
//
// The polygon test runs in FP32 on the unrounded plane coordinates (af, bf)
// against each edge's line scaled by a bound E on the test's own error: with
// A -> B an edge (quantised ints, ex = B - A), c = ex A.y - ey A.x and the
// cluster's inliers within |X|, |Y| <= M - 1 (their extremes along +-x, +-y),
//   F = (ex bf - ey af - c) / E,  E = 2 (0.5 (|ex| + |ey|) + 2^-21 ((|ex| + |ey|) M + |c|) + 1),
// differs from the exact cross product (ex Y - ey X - c) / E by less than 0.5:
// af, bf lie within half a unit of X, Y, and the conversions, the divisions
// and the two fused multiply-adds add at most 2^-22 ((|ex| + |ey|) M + |c|).
// So min over the edges F > 1 means strictly inside every edge (the point is
// dropped) and F < -1 on some edge means outside it (a survivor); the few
// points in between take the exact integer test.  The polygon is formed once a
// cluster, with its centroid (poly_warp; one thread an item did it in 1.4 us).
// The edges' coefficients are read from shared memory once per kBatch chunks.
// Registers are held down as in k_extract, six CTAs an SM in a large fit (2,000
// clusters 376 -> 292 us).
template <bool kTail>
__global__ void __launch_bounds__(kT, kTail ? 4 : 6)
k_filter(const float* __restrict__ pts, const uint32_t* __restrict__ off, const uint32_t* __restrict__ item_off,
         const uint32_t* __restrict__ item_cl, const uint32_t* __restrict__ kp, const uint32_t* __restrict__ tile,
         FitCluster* __restrict__ cl, const uint8_t* __restrict__ inlier, const float* __restrict__ cen,
         const FitPoly* __restrict__ poly_of, float* __restrict__ part, int2* __restrict__ surv,
         uint32_t* __restrict__ done) {
    pdl_gate();
    const uint32_t k = *kp, T = *tile;
    constexpr int kSurvBuf = 128;
    constexpr int kBatch = 4;  // chunks a thread tests against the edges together
    __shared__ float wp[kMaxChunksPerItem * (kT / 32) * 6];
    __shared__ int2 poly[kFiltDirs + 1];
    __shared__ float4 edge[kFiltDirs];
    __shared__ int npoly;
    __shared__ int2 sbuf[kT / 32][kSurvBuf];
    int2* sb = sbuf[threadIdx.x >> 5];
    const uint32_t n_items = item_off[k];
    const int lane = threadIdx.x & 31;
    const uint32_t cpt = T / kChunk;
    for (uint32_t it = blockIdx.x; it < n_items; it += gridDim.x) {
        const uint32_t c = find_cluster(item_cl, item_off, k, it);
        const FitCluster f = cl[c];
        const uint32_t base = off[c];
        const uint32_t start = base + (it - item_off[c]) * T;
        const uint32_t end = min(off[c + 1], start + T);
        __syncthreads();
        const FitPoly* fp = poly_of + c;
        if (threadIdx.x < kFiltDirs) edge[threadIdx.x] = fp->edge[threadIdx.x];
        if (threadIdx.x >= 32 && threadIdx.x - 32 <= kFiltDirs) poly[threadIdx.x - 32] = fp->pt[threadIdx.x - 32];
        if (threadIdx.x == 64) npoly = fp->m;
        __syncthreads();
        const int m = npoly;
        const float cx = cen[6 * c], cy = cen[6 * c + 2], cz = cen[6 * c + 4];  // nearest floats of the centroid
        int cnt = 0;  // survivors in this warp's buffer (warp-uniform)
        auto flush = [&]() {
            uint32_t pos = 0;
            if (lane == 0) pos = atomicAdd(&cl[c].n_surv, (uint32_t)cnt);
            pos = __shfl_sync(0xffffffffu, pos, 0);
            for (int i = lane; i < cnt; i += 32) surv[base + pos + i] = sb[i];
            __syncwarp();
            cnt = 0;
        };
        uint32_t j = 0;
        for (uint32_t qb = start; qb < end; qb += kBatch * kChunk) {
            float px[kBatch], py[kBatch], pz[kBatch], af[kBatch], bf[kBatch], fmin[kBatch];
            bool live[kBatch];
#pragma unroll
            for (int u = 0; u < kBatch; ++u) {
                const uint32_t q = qb + u * kChunk + threadIdx.x;
                live[u] = q < end && inlier[q];
                px[u] = py[u] = pz[u] = af[u] = bf[u] = 0.0f;
                if (live[u]) {
                    px[u] = pts[3 * (size_t)q]; py[u] = pts[3 * (size_t)q + 1]; pz[u] = pts[3 * (size_t)q + 2];
                    const float2 w = plane_coords(f, px[u], py[u], pz[u]);
                    af[u] = w.x;
                    bf[u] = w.y;
                }
                fmin[u] = 2.0f;
            }
            if (m) {
#pragma unroll
                for (int i = 0; i < kFiltDirs; ++i) {
                    const float4 e = edge[i];
#pragma unroll
                    for (int u = 0; u < kBatch; ++u)
                        fmin[u] = fminf(fmin[u], __fmaf_rn(e.x, bf[u], __fmaf_rn(e.y, af[u], e.z)));
                }
            }
#pragma unroll
            for (int u = 0; u < kBatch; ++u) {
                if (qb + u * kChunk >= end) continue;  // uniform: past the item's last chunk
                bool keep = false;
                int2 xy = make_int2(0, 0);
                float v[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};  // centred second moments
                if (live[u]) {
                    const float rx = __fsub_rn(px[u], cx), ry = __fsub_rn(py[u], cy), rz = __fsub_rn(pz[u], cz);
                    v[0] = __fmul_rn(rx, rx); v[1] = __fmul_rn(ry, ry); v[2] = __fmul_rn(rz, rz);
                    v[3] = __fmul_rn(rx, ry); v[4] = __fmul_rn(rx, rz); v[5] = __fmul_rn(ry, rz);
                    keep = !m || !(fmin[u] > 1.0f);
                    if (keep) {
                        xy = make_int2(__float2int_rn(af[u]), __float2int_rn(bf[u]));
                        if (m && !(fmin[u] < -1.0f)) {  // within the error band of an edge: the exact test
                            for (int i = 0; i < m; ++i) {  // strictly inside every edge -> not a hull vertex
                                if (cross3(poly[i], poly[i + 1], xy) <= 0) break;
                                if (i == m - 1) keep = false;
                            }
                        }
                    }
                }
                const uint32_t b = __ballot_sync(0xffffffffu, keep);
                if (cnt + __popc(b) > kSurvBuf) flush();
                if (keep) sb[cnt + __popc(b & ((1u << lane) - 1u))] = xy;
                cnt += __popc(b);
                __syncwarp();
                warp_park<6>(v, wp, j);
                ++j;
            }
        }
        if (cnt) flush();
        chunks_out<6>(wp, j, part + (size_t)it * cpt * 10, 4);
        if constexpr (kTail) filter_tail(c, off, item_off, cpt, part, cen, cl, done);
    }
}

// Refit of cluster c by a whole CTA: total least squares on the inliers.  The
// covariance A about the centroid is summed in double-float over the
// per-chunk partials and scaled by its trace.  Its smallest eigenvector is the
// dominant eigenvector of its adjugate adj(A) (eigenvalues lambda_j lambda_k);
// the adjugate's cofactors, where the cancellation is, are formed in
// double-float and rounded, then six steps of power iteration in FP32 from
// the selected RANSAC normal converge by lambda_min / lambda_mid per step.
// n_z >= 0, d = -n . centroid (double-float); lambda_mid < 10 lambda_min
// (from the trace, the Rayleigh quotient in double-float and
// x^T adj(A) x = lambda_1 lambda_2) flags the plane ill-conditioned.
// The double-float steps run a lane per value (six entries, six cofactors,
// three rows), so that their code is short: it runs once a cluster, and
// written out for one thread its 13 KB took 3.5 us, most of it fetching.
__device__ __forceinline__ df2 df_shfl(df2 x, int src) {
    return {__shfl_sync(0xffffffffu, x.hi, src), __shfl_sync(0xffffffffu, x.lo, src)};
}
// Lane's pick of a small table packed in 4-bit fields.
__device__ __forceinline__ int nib(uint32_t table, int i) { return (int)((table >> (4 * i)) & 15u); }
__device__ __forceinline__ void refit_cta(uint32_t c, const uint32_t* __restrict__ off,
                                          const uint32_t* __restrict__ item_off, uint32_t cpt,
                                          const float* __restrict__ part, const float* __restrict__ cen,
                                          FitCluster* __restrict__ cl, RefitShared& sm) {
    df2 A[6];
#pragma unroll
    for (int e = 0; e < 6; ++e) A[e] = df2{0.0f, 0.0f};
    const uint32_t base = item_off[c] * cpt, nch = (off[c + 1] - off[c] + kChunk - 1) / kChunk;
#pragma unroll 2
    for (uint32_t j = threadIdx.x; j < nch; j += kT) {
        float v[6];
#pragma unroll
        for (int e = 0; e < 6; ++e) v[e] = __ldcg(part + (size_t)(base + j) * 10 + 4 + e);
#pragma unroll
        for (int e = 0; e < 6; ++e) A[e] = df_add(A[e], df2{v[e], 0.0f});
    }
    block_df_sum<6>(A, sm.sh, sm.tot);
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x, e6 = lane < 6 ? lane : 0, r3 = lane % 4 < 3 ? lane % 4 : 0;
        FitCluster& f = cl[c];
        uint32_t flags = 0;
        const float fx = f.n[0], fy = f.n[1], fz = f.n[2];
        const float tr = __fadd_rn(__fadd_rn(sm.tot[0].hi, sm.tot[1].hi), sm.tot[2].hi);
        const bool found = f.best_h >= 0 && f.inliers > 0;
        float x = fx, y = fy, z = fz;
        df2 S{0.0f, 0.0f};
        if (found && tr > 0.0f) {
            // A / tr: entries of magnitude at most 1 (the diagonal is non-negative); lane e holds entry e of
            // [[0 3 4] [3 1 5] [4 5 2]]
            S = df_mulf(sm.tot[e6], __fdiv_rn(1.0f, tr));
            // symmetric adjugate, lane e: S[i0] S[i1] - S[i2] S[i3] of m00, m11, m22, m01, m02, m12
            const df2 a0 = df_shfl(S, nib(0x334001u, e6)), a1 = df_shfl(S, nib(0x455122u, e6));
            const df2 a2 = df_shfl(S, nib(0x043345u, e6)), a3 = df_shfl(S, nib(0x512345u, e6));
            const float m = df_sub(df_mul(a0, a1), df_mul(a2, a3)).hi;
            const float m00 = __shfl_sync(0xffffffffu, m, 0), m11 = __shfl_sync(0xffffffffu, m, 1);
            const float m22 = __shfl_sync(0xffffffffu, m, 2), m01 = __shfl_sync(0xffffffffu, m, 3);
            const float m02 = __shfl_sync(0xffffffffu, m, 4), m12 = __shfl_sync(0xffffffffu, m, 5);
            bool ok = true;
#pragma unroll 1
            for (int it = 0; it < 6; ++it) {
                const float nx = __fmaf_rn(m02, z, __fmaf_rn(m01, y, __fmul_rn(m00, x)));
                const float ny = __fmaf_rn(m12, z, __fmaf_rn(m11, y, __fmul_rn(m01, x)));
                const float nz = __fmaf_rn(m22, z, __fmaf_rn(m12, y, __fmul_rn(m02, x)));
                const float q = __fmaf_rn(nz, nz, __fmaf_rn(ny, ny, __fmul_rn(nx, nx)));
                if (!(q > 1e-30f) || !(q < 1e30f)) { ok = false; break; }  // rank <= 1: keep the RANSAC normal
                const float sc = rsqrtf(q);
                x = __fmul_rn(nx, sc); y = __fmul_rn(ny, sc); z = __fmul_rn(nz, sc);
            }
            if (!ok) {
                x = fx; y = fy; z = fz;
                flags |= 1u;
            }
            // unit length to FP32 accuracy
            const float inv = __fdiv_rn(1.0f, __fsqrt_rn(__fmaf_rn(z, z, __fmaf_rn(y, y, __fmul_rn(x, x)))));
            x = __fmul_rn(x, inv); y = __fmul_rn(y, inv); z = __fmul_rn(z, inv);
            if (z < 0.0f || (z == 0.0f && (y < 0.0f || (y == 0.0f && x < 0.0f)))) { x = -x; y = -y; z = -z; }
            // eigenvalues (scaled by 1 / tr) for the conditioning flag: lanes 0 .. 2 hold the rows of A x, lanes 4
            // .. 6 the centroid; each times its component, summed in lanes 0 and 4
            const df2 s0 = df_shfl(S, nib(0x430u, r3)), s1 = df_shfl(S, nib(0x513u, r3)), s2 = df_shfl(S, nib(0x254u, r3));
            df2 row = df_add(df_add(df_mulf(s0, x), df_mulf(s1, y)), df_mulf(s2, z));
            if (lane & 4) row = df2{cen[6 * (size_t)c + 2 * r3], cen[6 * (size_t)c + 2 * r3 + 1]};
            row = df_mulf(row, r3 == 0 ? x : (r3 == 1 ? y : z));
            const df2 t1 = df_shfl(row, (lane & 4) + 1), t2 = df_shfl(row, (lane & 4) + 2);
            const float dot = df_add(df_add(row, t1), t2).hi;
            const float lmin = __shfl_sync(0xffffffffu, dot, 0), cd = __shfl_sync(0xffffffffu, dot, 4);
            const float p12 = x * (m00 * x + m01 * y + m02 * z) + y * (m01 * x + m11 * y + m12 * z) +
                              z * (m02 * x + m12 * y + m22 * z);
            const float Sx = 1.0f - lmin;
            const float disc = fmaxf(Sx * Sx - 4.0f * p12, 0.0f);
            const float lmax = 0.5f * (Sx + sqrtf(disc));
            const float lmid = lmax > 0.0f ? p12 / lmax : 0.0f;  // no cancellation
            if (!(lmid >= 10.0f * lmin)) flags |= 1u;
            if (lane == 0) {
                f.refit_n[0] = x; f.refit_n[1] = y; f.refit_n[2] = z;
                f.refit_d = -cd;
                f.flags = flags;
            }
        } else if (lane == 0) {
            float rd = 0.0f;
            x = y = z = 0.0f;
            if (found) {  // zero spread: no plane to fit; the RANSAC normal through the centroid
                flags = 1u;
                x = fx; y = fy; z = fz;
                const float* ce = cen + 6 * (size_t)c;
                rd = -df_add(df_add(df_mulf(df2{ce[0], ce[1]}, x), df_mulf(df2{ce[2], ce[3]}, y)),
                             df_mulf(df2{ce[4], ce[5]}, z)).hi;
            }
            f.refit_n[0] = x; f.refit_n[1] = y; f.refit_n[2] = z;
            f.refit_d = rd;
            f.flags = flags;
        }
    }
    __syncthreads();  // shared partials reused next
}

// The centroid and the refit of every cluster as kernels of their own (a CTA
// per cluster), for fits too large for the per-cluster completion counters
// to pay (launch_fit).
__global__ void __launch_bounds__(kT) k_centroid(const float* __restrict__ pts, const uint32_t* __restrict__ off,
                                                 const uint32_t* __restrict__ item_off, const uint32_t* __restrict__ kp,
                                                 const uint32_t* __restrict__ tile, const float* __restrict__ part,
                                                 FitCluster* __restrict__ cl, float* __restrict__ cen,
                                                 FitPoly* __restrict__ poly) {
    pdl_gate();
    const uint32_t k = *kp, cpt = *tile / kChunk;
    __shared__ CentroidShared sm;
    for (uint32_t c = blockIdx.x; c < k; c += gridDim.x) centroid_cta(c, pts, off, item_off, cpt, part, cl, cen, poly, sm);
}

__global__ void __launch_bounds__(kT) k_refit(const uint32_t* __restrict__ off, const uint32_t* __restrict__ item_off,
                                              const uint32_t* __restrict__ kp, const uint32_t* __restrict__ tile,
                                              const float* __restrict__ part, const float* __restrict__ cen,
                                              FitCluster* __restrict__ cl) {
    pdl_gate();
    const uint32_t k = *kp, cpt = *tile / kChunk;
    __shared__ RefitShared sm;
    for (uint32_t c = blockIdx.x; c < k; c += gridDim.x) refit_cta(c, off, item_off, cpt, part, cen, cl, sm);
}

__device__ __forceinline__ unsigned long long xy_key(int2 p) {
    return ((unsigned long long)((uint32_t)p.x ^ 0x80000000u) << 32) | ((uint32_t)p.y ^ 0x80000000u);
}
__device__ __forceinline__ int2 key_xy(unsigned long long k) {
    return make_int2((int32_t)((uint32_t)(k >> 32) ^ 0x80000000u), (int32_t)((uint32_t)k ^ 0x80000000u));
}

// Monotone chain over sorted unique points; one thread builds a chain.  The
// two top entries stay in registers so a pop costs one shared-memory load.
__device__ int chain(const unsigned long long* P, int u, bool upper, uint32_t* st) {
    int kk = 0;
    int2 t1 = make_int2(0, 0), t0 = make_int2(0, 0);  // top, second
    for (int s = 0; s < u; ++s) {
        const int i = upper ? (u - 1 - s) : s;
        const int2 p = key_xy(P[i]);
        while (kk >= 2 && cross3(t0, t1, p) <= 0) {
            --kk;
            t1 = t0;
            if (kk >= 2) t0 = key_xy(P[st[kk - 2]]);
        }
        st[kk] = (uint32_t)i;
        t0 = t1;
        t1 = p;
        ++kk;
    }
    return kk;
}

// "Better next vertex" from cur: more clockwise, or collinear and farther.
__device__ __forceinline__ bool jarvis_better(int2 cur, int2 a, bool a_ok, int2 b, bool b_ok) {
    if (!b_ok) return false;
    if (!a_ok) return true;
    const long long cr = cross3(cur, a, b);
    if (cr < 0) return true;
    if (cr > 0) return false;
    const long long da = (long long)(a.x - cur.x) * (a.x - cur.x) + (long long)(a.y - cur.y) * (a.y - cur.y);
    const long long db = (long long)(b.x - cur.x) * (b.x - cur.x) + (long long)(b.y - cur.y) * (b.y - cur.y);
    return db > da;
}

// Directions of the second hull filter: kHullDirs integer vectors
// (rint(1024 cos), rint(1024 sin)) of multiples of 360/kHullDirs degrees, in
// counter-clockwise order.  Any closed polygon through input points serves
// the filter (a point strictly left of every edge has winding number >= 1, so
// it lies in the convex hull of the polygon's vertices and is not an extreme
// point); the directions only decide how much it removes.
constexpr int kHullDirs = 128;
constexpr int kFewDirs = 32;
constexpr int kFewSurv = 96;    // survivors that are not worth a pass
constexpr int kFewCand = 128;   // candidates that are not worth a second one
constexpr int kSmallHull = kT;  // candidates ranked and tested in parallel, one a thread

// Per cluster hull of the first filter's survivors: (1) extreme survivors along
// kFewDirs or kHullDirs directions; (2) survivors strictly inside the polygon they span
// are dropped (none of them can be a hull vertex), the rest gathered in shared
// memory; when many are left, both once more with kHullDirs directions;
// (3) bitonic sort by (X, Y), duplicates removed; (4) monotone chain, lower
// and upper halves built concurrently by two threads.  If more than
// kHullCap points remain, gift wrapping runs over the survivors instead.
// Most clusters leave some 20 survivors, and these go straight to (3'): a pass
// costs 4 us however few they are.  A first pass of 32 directions is cheap where
// there are many survivors (1,500 cost 128 directions 10 us) and enough where
// there are few; in between, 128 at once spare a second pass.  16 clusters: 8.4 ->
// 7.5 us, 2,000 clusters 58 -> 43, the 5 x 5 x 5 m window 21.8 -> 14.5.
// hull_ctr: a word that is zero at launch; the last CTA to finish turns
// hull_cnt into the hulls' offsets (exclusive scan, the total at [k]) and
// zeroes the word again.
__global__ void __launch_bounds__(kT) k_hull(const uint32_t* __restrict__ off, const uint32_t* __restrict__ kp,
                                             const FitCluster* __restrict__ cl, const int2* __restrict__ surv,
                                             int2* __restrict__ hull, uint32_t* __restrict__ hull_cnt,
                                             uint32_t* __restrict__ err, uint32_t* __restrict__ hull_ctr) {
    pdl_gate();
    const uint32_t k = *kp;
    extern __shared__ unsigned long long sk[];              // kHullCap keys, then kHullCap unique
    unsigned long long* uq = sk + kHullCap;
    uint32_t* st_lo = reinterpret_cast<uint32_t*>(uq + kHullCap);
    uint32_t* st_hi = st_lo + kHullCap;
    int2* ssv = reinterpret_cast<int2*>(uq);  // kSurvCap staged survivors, done with before the unique keys
    __shared__ uint32_t wsum[kT / 32];
    __shared__ int s_klo, s_khi, s_m, s_cnt;
    __shared__ int2 poly[kHullDirs];       // the extreme point of each direction
    __shared__ int2 hpoly[kHullDirs + 1];  // the filter polygon
    __shared__ long long warea[kT / 32];
    __shared__ int2 sdir[kHullDirs];
    __shared__ int2 jcand[kT];
    __shared__ int jok[kT];
    __shared__ unsigned long long wmin[kT / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    bool dirs = false;  // sdir is there
    for (uint32_t c = blockIdx.x; c < k; c += gridDim.x) {
        __syncthreads();
        const uint32_t base = off[c];
        const int s = (int)cl[c].n_surv;
        int2* out = hull + base;
        // stage the survivors (when they fit) so the scans below read shared memory
        const int2* sv = surv + base;
        if (s <= kSurvCap) {
            for (int i = threadIdx.x; i < s; i += kT) ssv[i] = sv[i];
            sv = ssv;
        }
        if (s > kFewSurv && !dirs) {
            for (int j = threadIdx.x; j < kHullDirs; j += kT) {
                const float t = (float)j * (2.0f / kHullDirs);
                sdir[j] = make_int2(__float2int_rn(1024.0f * cospif(t)), __float2int_rn(1024.0f * sinpif(t)));
            }
            dirs = true;
        }
        __syncthreads();
        // (1), (2): from `from`, n points, to `to`; the candidates so far are cand[0 .. s2)
        const int2* cand = sv;
        int s2 = s;
        for (int pass = 0, D = s > 160 && s <= 512 ? kHullDirs : kFewDirs; pass < 2; ++pass, D = kHullDirs) {
            const int2* from = cand;
            int2* to = reinterpret_cast<int2*>(sk);
            int n = s2;
            if (pass == 0 ? s <= kFewSurv : s2 <= kFewCand) break;
            if (pass && s2 > kHullCap) {  // from the survivors again: the first polygon dropped too few
                from = sv;
                n = s;
            } else if (pass) {
                to = reinterpret_cast<int2*>(uq);  // the staged survivors are done with
            }
            // (1) extreme points along D directions, four a warp at a time.  The
            // projections are FP32: any closed polygon through input points
            // serves the filter below (which is exact), so an extreme point only
            // has to be an input point, not the exact maximiser.
            for (int d0 = 4 * w; d0 < D; d0 += 4 * (kT / 32)) {
                float dxq[4], dyq[4], bv[4];
                int bi[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int2 dir = sdir[(d0 + q) * (kHullDirs / D)];
                    dxq[q] = (float)dir.x;
                    dyq[q] = (float)dir.y;
                    bv[q] = -INFINITY;
                    bi[q] = -1;
                }
#pragma unroll 2
                for (int i = lane; i < n; i += 32) {
                    const int2 p = from[i];
                    const float fx = (float)p.x, fy = (float)p.y;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float v = fmaf(dxq[q], fx, dyq[q] * fy);
                        if (v > bv[q]) { bv[q] = v; bi[q] = i; }
                    }
                }
                // the warp's largest projection (its bits as an ordered integer), then the lowest index that has it
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int b = __float_as_int(bv[q]), key = b ^ ((b >> 31) & 0x7fffffff);
                    const int top = __reduce_max_sync(0xffffffffu, key);
                    const int at = __reduce_min_sync(0xffffffffu, key == top && bi[q] >= 0 ? bi[q] : INT_MAX);
                    if (lane == q) poly[d0 + q] = at != INT_MAX ? from[at] : make_int2(INT_MIN, INT_MIN);
                }
            }
            __syncthreads();
            // The polygon through the extremes, consecutive duplicates removed (and
            // the last vertex when it repeats the first), in parallel: a direction's
            // extreme is kept unless it repeats the previous direction's; a ballot
            // places the kept ones.  Every direction has an extreme: n > 0.
            int2 p = make_int2(0, 0);
            bool keep = false;
            if (threadIdx.x < D) {
                p = poly[threadIdx.x];
                const int2 q = poly[threadIdx.x ? threadIdx.x - 1 : 0];
                keep = threadIdx.x == 0 || p.x != q.x || p.y != q.y;
            }
            const uint32_t kb = __ballot_sync(0xffffffffu, keep);
            if (lane == 0) wsum[w] = __popc(kb);
            __syncthreads();
            uint32_t at = __popc(kb & ((1u << lane) - 1u)), m0 = 0;
            for (int q = 0; q < kT / 32; ++q) {
                at += q < w ? wsum[q] : 0u;
                m0 += wsum[q];
            }
            if (keep) hpoly[at] = p;
            __syncthreads();
            if (m0 > 1 && hpoly[m0 - 1].x == hpoly[0].x && hpoly[m0 - 1].y == hpoly[0].y) --m0;
            // twice the signed area: a degenerate (zero-area) polygon filters nothing
            long long a2 = 0;
            if (threadIdx.x < m0) {
                const int2 a = hpoly[threadIdx.x], bb = hpoly[threadIdx.x + 1 < m0 ? threadIdx.x + 1 : 0];
                a2 = (long long)a.x * bb.y - (long long)a.y * bb.x;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) a2 += __shfl_xor_sync(0xffffffffu, a2, o);
            if (lane == 0) warea[w] = a2;
            __syncthreads();
            if (threadIdx.x == 0) {
                long long area2 = 0;
                for (int q = 0; q < kT / 32; ++q) area2 += warea[q];
                s_m = (m0 >= 3 && area2 > 0) ? (int)m0 : 0;
                hpoly[m0] = hpoly[0];
                s_cnt = 0;
            }
            __syncthreads();
            const int m = s_m;
            // (2) drop the points strictly inside the polygon
            for (int i0 = 0; i0 < n; i0 += kT) {
                const int i = i0 + threadIdx.x;
                bool out_or_on = false;
                int2 pt = make_int2(0, 0);
                if (i < n) {
                    pt = from[i];
                    out_or_on = (m == 0);
#pragma unroll 4
                    for (int e = 0; e < m; ++e) out_or_on |= cross3(hpoly[e], hpoly[e + 1], pt) <= 0;
                }
                const uint32_t b = __ballot_sync(0xffffffffu, out_or_on);
                int pos = 0;
                if (lane == 0 && b) pos = atomicAdd(&s_cnt, __popc(b));
                pos = __shfl_sync(0xffffffffu, pos, 0) + __popc(b & ((1u << lane) - 1u));
                if (out_or_on && pos < kHullCap) to[pos] = pt;
            }
            __syncthreads();
            cand = to;
            s2 = s_cnt;
        }
        if (s2 <= kHullCap)
            for (int i = threadIdx.x; i < s2; i += kT) sk[i] = xy_key(cand[i]);
        __syncthreads();
        if (s2 <= kSmallHull) {
            // (3') at most kT candidates: rank sort with duplicates removed --
            // a candidate is kept if no earlier one has its key, and lands at
            // the number of kept keys below it
            // (few candidates share the threads, 4 or 2 to one)
            const int i = threadIdx.x, Lr = s2 <= kT / 4 ? 4 : (s2 <= kT / 2 ? 2 : 1), cr = i / Lr, sr = i % Lr;
            unsigned long long key = 0;
            int twin = 0;
            if (cr < s2) {
                key = sk[cr];
#pragma unroll 4
                for (int j = sr; j < cr; j += Lr) twin |= sk[j] == key;
            }
            for (int o = 1; o < Lr; o <<= 1) twin |= __shfl_xor_sync(0xffffffffu, twin, o);
            const bool uniq = cr < s2 && !twin, first = uniq && sr == 0;
            if (sr == 0) st_lo[cr] = first;
            __syncthreads();
            int rank = 0;
            if (uniq)
#pragma unroll 4
                for (int j = sr; j < s2; j += Lr) rank += (st_lo[j] != 0u) & (sk[j] < key);
            for (int o = 1; o < Lr; o <<= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
            const uint32_t b = __ballot_sync(0xffffffffu, first);
            if (lane == 0) wsum[w] = __popc(b);
            __syncthreads();
            int u = 0;
            for (int q = 0; q < kT / 32; ++q) u += (int)wsum[q];
            if (first) uq[rank] = key;
            __syncthreads();
            if (u < 3) {
                if (i < u) out[i] = key_xy(uq[i]);
                if (i == 0) hull_cnt[c] = (uint32_t)u;
            } else {
                // (4') Andrew's chains by a test per candidate: in the sorted
                // order, P_i is a vertex of the lower chain iff it is an end or
                // cross(P_j, P_i, P_k) > 0 for every j < i < k -- the directions
                // P_i - P_j and P_k - P_i lie in a half-plane (x >= 0, x = 0 only
                // upwards) where cross orders them by angle, so it is enough that
                // the most counter-clockwise P_i - P_j turns left into the most
                // clockwise P_k - P_i; of the upper chain iff the most clockwise
                // P_i - P_j lies right of the most counter-clockwise P_k - P_i.
                // Collinear points fail (cross = 0), as in the chains.  Few
                // candidates share the threads, 4 or 2 to a candidate (48
                // candidates took a thread each 4.3 us).
                const int L = u <= kT / 4 ? 4 : (u <= kT / 2 ? 2 : 1), ci = (int)threadIdx.x / L;
                const int sub = (int)threadIdx.x % L;
                bool lo = false, hi = false;
                const auto turn = [](int2 a, int2 b) { return (long long)a.x * b.y - (long long)a.y * b.x; };
                const int2 P = ci < u ? key_xy(uq[ci]) : make_int2(0, 0);
                int2 dc[2], dw[2];  // most counter-clockwise and most clockwise, before and after; (0, 0): none yet
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    int2 C = make_int2(0, 0), W = make_int2(0, 0);
                    const int q1 = ci < u ? (t ? u : ci) : 0;
                    int q = (t ? ci + 1 : 0) + sub;
                    if (q < q1) {
                        const int2 Q = key_xy(uq[q]);
                        C = W = t ? make_int2(Q.x - P.x, Q.y - P.y) : make_int2(P.x - Q.x, P.y - Q.y);
                    }
#pragma unroll 2
                    for (q += L; q < q1; q += L) {
                        const int2 Q = key_xy(uq[q]);
                        const int2 d = t ? make_int2(Q.x - P.x, Q.y - P.y) : make_int2(P.x - Q.x, P.y - Q.y);
                        if (turn(C, d) > 0) C = d;
                        if (turn(d, W) > 0) W = d;
                    }
                    for (int o = 1; o < L; o <<= 1) {
                        const int2 c2 = make_int2(__shfl_xor_sync(0xffffffffu, C.x, o), __shfl_xor_sync(0xffffffffu, C.y, o));
                        const int2 w2 = make_int2(__shfl_xor_sync(0xffffffffu, W.x, o), __shfl_xor_sync(0xffffffffu, W.y, o));
                        if (c2.x | c2.y) {
                            if (!(C.x | C.y) || turn(C, c2) > 0) C = c2;
                            if (!(W.x | W.y) || turn(w2, W) > 0) W = w2;
                        }
                    }
                    dc[t] = C;
                    dw[t] = W;
                }
                if (ci < u && sub == 0) {
                    const bool end = ci == 0 || ci == u - 1;
                    // the lower chain's last point opens the upper chain, whose last point is the lower's first
                    lo = ci < u - 1 && (end || turn(dc[0], dw[1]) > 0);
                    hi = ci > 0 && (end || turn(dc[1], dw[0]) > 0);
                }
                // lower vertices in increasing order, then upper vertices in decreasing order
                const uint32_t bl = __ballot_sync(0xffffffffu, lo), bh = __ballot_sync(0xffffffffu, hi);
                if (lane == 0) {
                    wsum[w] = __popc(bl);
                    st_hi[w] = __popc(bh);
                }
                __syncthreads();
                int klo = 0, khi = 0, plo = __popc(bl & ((1u << lane) - 1u)), phi = __popc(bh >> lane) - (hi ? 1 : 0);
                for (int q = 0; q < kT / 32; ++q) {
                    klo += (int)wsum[q];
                    khi += (int)st_hi[q];
                    plo += q < w ? (int)wsum[q] : 0;
                    phi += q > w ? (int)st_hi[q] : 0;
                }
                if (lo) out[plo] = P;
                if (hi) out[klo + phi] = P;
                if (i == 0) hull_cnt[c] = (uint32_t)(klo + khi);
            }
        } else if (s2 <= kHullCap) {
            int n2 = 1;
            while (n2 < s2) n2 <<= 1;
            for (int i = s2 + threadIdx.x; i < n2; i += kT) sk[i] = ~0ull;
            __syncthreads();
            // (3) bitonic sort, ascending
            for (int size = 2; size <= n2; size <<= 1) {
                for (int stride = size >> 1; stride > 0; stride >>= 1) {
                    for (int i = threadIdx.x; i < n2; i += kT) {
                        const int jdx = i ^ stride;
                        if (jdx > i) {
                            const bool up = (i & size) == 0;
                            const unsigned long long a = sk[i], b = sk[jdx];
                            if ((a > b) == up) { sk[i] = b; sk[jdx] = a; }
                        }
                    }
                    __syncthreads();
                }
            }
            // unique, order-preserving (block scan in chunks)
            int u = 0;
            for (int c0 = 0; c0 < s2; c0 += kT) {
                const int i = c0 + threadIdx.x;
                const uint32_t fl = (i < s2) && (i == 0 || sk[i] != sk[i - 1]);
                uint32_t inc = fl;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
                    if (lane >= o) inc += t;
                }
                if (lane == 31) wsum[w] = inc;
                __syncthreads();
                uint32_t wpre = 0, tot = 0;
                for (int q = 0; q < kT / 32; ++q) {
                    if (q < w) wpre += wsum[q];
                    tot += wsum[q];
                }
                if (fl) uq[u + wpre + inc - 1] = sk[i];
                u += (int)tot;
                __syncthreads();
            }
            // (4) monotone chain
            if (u < 3) {
                for (int i = threadIdx.x; i < u; i += kT) out[i] = key_xy(uq[i]);
                if (threadIdx.x == 0) hull_cnt[c] = (uint32_t)u;
            } else {
                if (threadIdx.x == 0) s_klo = chain(uq, u, false, st_lo);
                if (threadIdx.x == 32) s_khi = chain(uq, u, true, st_hi);
                __syncthreads();
                const int klo = s_klo - 1, khi = s_khi - 1;
                for (int i = threadIdx.x; i < klo + khi; i += kT)
                    out[i] = key_xy(uq[i < klo ? st_lo[i] : st_hi[i - klo]]);
                if (threadIdx.x == 0) hull_cnt[c] = (uint32_t)(klo + khi);
            }
        } else {
            // gift wrapping over all survivors in global memory
            unsigned long long bk = ~0ull;
            for (int i = threadIdx.x; i < s; i += kT) {
                const unsigned long long key = xy_key(sv[i]);
                bk = key < bk ? key : bk;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long t = __shfl_xor_sync(0xffffffffu, bk, o);
                bk = t < bk ? t : bk;
            }
            if (lane == 0) wmin[w] = bk;
            __syncthreads();
            if (threadIdx.x == 0) {
                for (int q = 1; q < kT / 32; ++q) bk = wmin[q] < bk ? wmin[q] : bk;
                wmin[0] = bk;
            }
            __syncthreads();
            const int2 start = key_xy(wmin[0]);
            int2 cur = start;
            int h = 0;
            if (threadIdx.x == 0) out[h] = cur;
            ++h;
            for (int guard = 0; guard <= s; ++guard) {
                int2 cand = make_int2(0, 0);
                bool ok = false;
                for (int i = threadIdx.x; i < s; i += kT) {
                    const int2 p = sv[i];
                    const bool pok = !(p.x == cur.x && p.y == cur.y);
                    if (jarvis_better(cur, cand, ok, p, pok)) { cand = p; ok = true; }
                }
                jcand[threadIdx.x] = cand;
                jok[threadIdx.x] = ok;
                __syncthreads();
                for (int r = kT / 2; r > 0; r >>= 1) {
                    if ((int)threadIdx.x < r) {
                        const int o = threadIdx.x + r;
                        if (jarvis_better(cur, jcand[threadIdx.x], jok[threadIdx.x], jcand[o], jok[o])) {
                            jcand[threadIdx.x] = jcand[o];
                            jok[threadIdx.x] = 1;
                        }
                    }
                    __syncthreads();
                }
                const int2 nxt = jcand[0];
                const bool nok = jok[0];
                __syncthreads();
                if (!nok || (nxt.x == start.x && nxt.y == start.y)) break;
                if (h >= s) {  // more vertices than points: only a broken invariant gets here
                    if (threadIdx.x == 0) atomicOr(err, kErrTimeout);
                    break;
                }
                if (threadIdx.x == 0) out[h] = nxt;
                ++h;
                cur = nxt;
            }
            if (threadIdx.x == 0) hull_cnt[c] = (uint32_t)h;
        }
    }
    // hull offsets, by the last CTA to finish
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_cnt = atomicAdd(hull_ctr, 1u) + 1u == gridDim.x;
    __syncthreads();
    if (!s_cnt) return;
    __threadfence();
    uint32_t carry = 0;
    for (uint32_t c0 = 0; c0 < k; c0 += kT) {
        const uint32_t c = c0 + threadIdx.x;
        const uint32_t v = c < k ? __ldcg(hull_cnt + c) : 0u;
        uint32_t inc = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        if (lane == 31) wsum[w] = inc;
        __syncthreads();
        uint32_t wpre = 0, tot = 0;
        for (int q = 0; q < kT / 32; ++q) {
            if (q < w) wpre += wsum[q];
            tot += wsum[q];
        }
        if (c < k) hull_cnt[c] = carry + wpre + inc - v;
        carry += tot;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        hull_cnt[k] = carry;
        *hull_ctr = 0;
    }
}

// The tile of a fit: the tuning's, or, when the fit may choose (adapt_ctas),
// the smallest multiple of a chunk that gives the points at most adapt_ctas
// work items, so that a small fit's scoring, extraction and filter passes
// spread over the GPU.  (240 thousand points of a walk map: 157 items of 2048
// on 152 SMs scored in 21 us, 490 of 512 in 12 us; one 17,000-point cluster: 9
// items in 14 us, 68 in 6 us.)  Results do not depend on the tile.
__device__ __forceinline__ uint32_t choose_tile(uint32_t T, uint32_t n, uint32_t adapt_ctas) {
    if (!adapt_ctas) return T;
    const uint32_t want = (n / adapt_ctas + kChunk) / kChunk * kChunk;
    return want < T ? want : T;
}

// Work items per cluster (scanned into the item offsets next) -- at least one,
// so that an empty cluster's per-cluster steps still run -- the work queue's
// heads and the per-cluster completion counters (done, may be null) cleared
// for the fit that follows; queue[1] receives the tile.
__global__ void k_items(const uint32_t* __restrict__ off, const uint32_t* __restrict__ kp, uint32_t tile,
                        uint32_t adapt_ctas, uint32_t* __restrict__ item_cnt, uint32_t* __restrict__ queue,
                        uint32_t* __restrict__ done) {
    pdl_gate();
    const uint32_t k = *kp, T = choose_tile(tile, off[k], adapt_ctas);
    if (blockIdx.x == 0 && threadIdx.x < 4) queue[threadIdx.x] = threadIdx.x == 1 ? T : 0u;
    for (uint32_t c = blockIdx.x * kT + threadIdx.x; c < k; c += gridDim.x * kT) {
        const uint32_t n = off[c + 1] - off[c];
        item_cnt[c] = n ? (n + T - 1) / T : 1u;
        if (done) done[2 * (size_t)c] = done[2 * (size_t)c + 1] = 0u;
    }
}

// The work items of up to kItemsScanMax clusters and their offsets in one
// CTA: counts as in k_items, an exclusive scan with a carry across rounds,
// the total at item_off[k].
constexpr int kItemsScanT = 1024;
constexpr uint32_t kItemsScanMax = 16384;
__global__ void __launch_bounds__(kItemsScanT) k_items_scan(const uint32_t* __restrict__ off,
                                                             const uint32_t* __restrict__ kp, uint32_t tile,
                                                             uint32_t adapt_ctas, uint32_t* __restrict__ item_off,
                                                             uint32_t* __restrict__ queue,
                                                             uint32_t* __restrict__ done) {
    pdl_gate();
    __shared__ uint32_t ws[kItemsScanT / 32];
    const uint32_t k = *kp, T = choose_tile(tile, off[k], adapt_ctas);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (threadIdx.x < 4) queue[threadIdx.x] = threadIdx.x == 1 ? T : 0u;
    uint32_t carry = 0;
    for (uint32_t c0 = 0; c0 < k; c0 += kItemsScanT) {
        const uint32_t c = c0 + threadIdx.x;
        uint32_t v = 0;
        if (c < k) {
            const uint32_t n = off[c + 1] - off[c];
            v = n ? (n + T - 1) / T : 1u;
            if (done) done[2 * (size_t)c] = done[2 * (size_t)c + 1] = 0u;
        }
        uint32_t inc = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        if (lane == 31) ws[w] = inc;
        __syncthreads();
        uint32_t wpre = 0, tot = 0;
        for (int q = 0; q < kItemsScanT / 32; ++q) {
            const uint32_t t = ws[q];
            wpre += q < w ? t : 0u;
            tot += t;
        }
        if (c < k) item_off[c] = carry + wpre + inc - v;
        carry += tot;
        __syncthreads();
    }
    if (threadIdx.x == 0) item_off[k] = carry;
}

__global__ void k_pack(const uint32_t* __restrict__ off, const uint32_t* __restrict__ labels,
                       const uint32_t* __restrict__ kp, const FitCluster* __restrict__ cl,
                       const int2* __restrict__ hull, const uint32_t* __restrict__ hull_off,
                       vm_plane* __restrict__ planes, int32_t* __restrict__ hull_xy, float* __restrict__ hull_xyz,
                       uint32_t hull_cap, HeaderArgs ha) {
    pdl_gate();
    const uint32_t k = *kp;
    if (ha.out && blockIdx.x == 0 && threadIdx.x == 0) write_header(ha);
    for (uint32_t c = blockIdx.x; c < k; c += gridDim.x) {
        const uint32_t ho = hull_off[c];
        pack_cluster(cl[c], labels ? labels[c] : c, off[c + 1] - off[c], hull + off[c], ho, hull_off[c + 1] - ho,
                     planes + c, hull_xy, hull_xyz, hull_cap);
    }
}

// Stage b with one warp per work item (the schedule for many small
// clusters): each warp pulls its own items from the queue and stages the
// item's points in its own slice of shared memory; lanes hold R hypotheses
// each, 32 / ceil(H / R) lanes groups split the points, and the groups' counts
// are combined with shuffles before the integer atomics.  No CTA barrier.
template <int R>
__global__ void __launch_bounds__(kT) k_score_warp(const float* __restrict__ pts, const uint32_t* __restrict__ off,
                                                   const uint32_t* __restrict__ item_off,
                                                   const uint32_t* __restrict__ item_cl,
                                                   const uint32_t* __restrict__ kp, int H,
                                                   const uint32_t* __restrict__ tile,
                                                   const float4* __restrict__ hyp, uint32_t* __restrict__ counts,
                                                   uint32_t* __restrict__ queue, float eps) {
    pdl_wait();
    const uint32_t k = *kp;
    const int T = (int)*tile;
    extern __shared__ float4 sp[];  // [kT / 32][T]
    const int lane = threadIdx.x & 31;
    float4* wp = sp + (size_t)(threadIdx.x >> 5) * T;
    const int G = (H + R - 1) / R;  // lanes per point group (<= 32, checked by the host)
    const int P = 32 / G;           // point groups per warp
    const int g = lane / G, j = lane % G;
    const bool active = g < P;
    const uint32_t n_items = item_off[k];
    for (int guard = 0; guard < kLoopCap; ++guard) {
        uint32_t it = 0;
        if (lane == 0) it = atomicAdd(queue, 1u);
        it = __shfl_sync(0xffffffffu, it, 0);
        if (it >= n_items) break;
        const uint32_t c = find_cluster(item_cl, item_off, k, it);
        const uint32_t start = off[c] + (it - item_off[c]) * (uint32_t)T;
        const uint32_t end = min(off[c + 1], start + (uint32_t)T);
        const int cnt = (int)(end - start);
        __syncwarp();
        for (int q = lane; q < cnt; q += 32) {
            const float* p = pts + 3 * ((size_t)start + q);
            wp[q] = make_float4(p[0], p[1], p[2], 0.0f);
        }
        float4 pl[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int h = j * R + r;
            pl[r] = (active && h < H) ? hyp[(size_t)c * H + h]
                                      : make_float4(0.0f, 0.0f, 0.0f, __int_as_float(0x7f800000));
        }
        __syncwarp();
        uint32_t acc[R];
#pragma unroll
        for (int r = 0; r < R; ++r) acc[r] = 0;
        if (active)
            for (int q = g; q < cnt; q += P) count_point<R>(pl, wp[q], eps, acc);
        for (int q = 1; q < P; ++q) {
            const int src = j + q * G;  // < 32 since P * G <= 32
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const uint32_t v = __shfl_sync(0xffffffffu, acc[r], src);
                if (g == 0) acc[r] += v;
            }
        }
        if (g == 0) {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int h = j * R + r;
                if (h < H && acc[r]) atomicAdd(&counts[(size_t)c * H + h], acc[r]);
            }
        }
    }
}

// ---------------------------------------------------------------- stage b, large fits
// The reference plane of each cluster for k_score_slab: the hypothesis with the
// most inliers among kRefPts points spread over the cluster (any plane serves;
// a good one decides more tiles at once).  Its normal frames the tiles' boxes and
// so has to be a unit vector: a hypothesis whose samples are closer than 1e-9 m, or
// farther than 1e9 m, apart has none, as the square of its cross product leaves the
// range of normal floats.  w is infinite when no hypothesis will do.  One CTA a
// cluster, a thread per hypothesis.
constexpr int kRefPts = 64;
__global__ void __launch_bounds__(kT) k_score_ref(const float* __restrict__ pts, const uint32_t* __restrict__ off,
                                                  const uint32_t* __restrict__ kp, int H,
                                                  const float4* __restrict__ hyp, float4* __restrict__ ref, float eps) {
    pdl_gate();
    const uint32_t k = *kp;
    __shared__ float4 sp[kRefPts];
    __shared__ unsigned long long wbest[kT / 32];
    for (uint32_t c = blockIdx.x; c < k; c += gridDim.x) {
        const uint32_t base = off[c], n = off[c + 1] - base, m = n < (uint32_t)kRefPts ? n : (uint32_t)kRefPts;
        __syncthreads();
        if (threadIdx.x < m) {
            const float* p = pts + 3 * ((size_t)base + (size_t)threadIdx.x * n / m);
            sp[threadIdx.x] = make_float4(p[0], p[1], p[2], 0.0f);
        }
        __syncthreads();
        unsigned long long best = 0;  // inliers + 1 << 32 | ~h
        for (int h = threadIdx.x; h < H; h += kT) {
            const float4 pl[1] = {hyp[(size_t)c * H + h]};
            const float n2 = pl[0].x * pl[0].x + pl[0].y * pl[0].y + pl[0].z * pl[0].z;
            if (!(fabsf(pl[0].w) < __int_as_float(0x7f800000)) || !(fabsf(n2 - 1.0f) < 9.5367431640625e-07f)) continue;
            uint32_t in[1] = {1u};
            for (uint32_t q = 0; q < m; ++q) count_point<1>(pl, sp[q], eps, in);
            const unsigned long long key = ((unsigned long long)in[0] << 32) | (uint32_t)~(uint32_t)h;
            best = key > best ? key : best;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long t = __shfl_xor_sync(0xffffffffu, best, o);
            best = t > best ? t : best;
        }
        if ((threadIdx.x & 31) == 0) wbest[threadIdx.x >> 5] = best;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int w = 1; w < kT / 32; ++w) best = wbest[w] > best ? wbest[w] : best;
            ref[c] = best ? hyp[(size_t)c * H + (int)(~(uint32_t)(best & 0xffffffffu))]
                          : make_float4(0.0f, 0.0f, 0.0f, __int_as_float(0x7f800000));
        }
    }
}

// A float's order as an integer's.
__device__ __forceinline__ int ord(float x) {
    const int b = __float_as_int(x);
    return b ^ ((b >> 31) & 0x7fffffff);
}
__device__ __forceinline__ float unord(int k) { return __int_as_float(k ^ ((k >> 31) & 0x7fffffff)); }

// The inliers of each cluster's reference plane: a lower bound of the best count.
__global__ void __launch_bounds__(kT) k_score_lower(const float* __restrict__ pts, const uint32_t* __restrict__ off,
                                                    const uint32_t* __restrict__ item_off,
                                                    const uint32_t* __restrict__ item_cl,
                                                    const uint32_t* __restrict__ kp, const uint32_t* __restrict__ tile,
                                                    const float4* __restrict__ ref, uint32_t* __restrict__ lower,
                                                    float eps) {
    pdl_gate();
    const uint32_t k = *kp, T = *tile, n_items = item_off[k];
    for (uint32_t it = blockIdx.x; it < n_items; it += gridDim.x) {
        const uint32_t c = find_cluster(item_cl, item_off, k, it);
        const uint32_t start = off[c] + (it - item_off[c]) * T, end = min(off[c + 1], start + T);
        const float4 r0[1] = {ref[c]};
        uint32_t in[1] = {0u};
#pragma unroll 4
        for (uint32_t q = start + threadIdx.x; q < end; q += kT)
            count_point<1>(r0, make_float4(pts[3 * (size_t)q], pts[3 * (size_t)q + 1], pts[3 * (size_t)q + 2], 0.0f), eps, in);
        in[0] = __reduce_add_sync(0xffffffffu, in[0]);
        if ((threadIdx.x & 31) == 0 && in[0]) atomicAdd(lower + c, in[0]);
    }
}

// Stage b for large fits: the best count, and every count that could be it, with
// far fewer tests than k_score.
// (1) A tile's points within eps / 2 of the cluster's reference plane (n0, d0),
// the near points, are bounded by their range of residuals and a box aligned
// with the plane and their longest direction.  For a hypothesis (n, d) the
// residual of a near point is its reference residual plus (n - n0) . p + (d -
// d0), which is linear, so the box bounds it; when the bound lies within eps
// every near point is an inlier, and when it lies beyond eps none is: no test
// is made.  The points off the plane (outliers) are tested against every
// hypothesis, the near points against those the bound leaves open.  All tests
// are count_point's, and the bound is widened by 2^-16 (|d| + |d0| + sum of the
// largest |coordinates|), over 250 rounding units of every quantity that enters
// it or the test (their sum stays below 150), so the counts are exact.  The
// in-plane axis is a difference, whose rounding leaves 2^-22 r / s of the normal
// in it when the farthest point lies r from the box's centre but only s from it
// in the plane: that costs 64 units more while the hypothesis leans from the
// reference by less than 16 s / r (angle t), and nothing beyond: no near point is
// farther than r from the centre, so one at an angle a from the farthest has a
// residual lower by r (1 - cos a), and the box adds r (1 - cos t) (1 + cos a) for
// it along the normal, together more than the r sin a sin t that it can lose, as
// cos(t - a) + cos t < 2.
// (2) counts start at the cluster's size and lose a tile's misses.  A
// hypothesis whose count has fallen below the reference plane's inliers cannot
// be selected any more and is dropped; its count stays below the best one.  The
// tiles of a cluster are taken spread over the launch, so that a poor
// hypothesis is dropped after a few of them.
// On the batch of 2,000 clusters (48 M points, 5 % outliers, H = 256, tile 2048)
// about a fifth of the tests remain (two fifths without (2)): 1.23 ms in place
// of 2.86 ms, and 0.11 ms for the two passes before it.
constexpr float kSlabErr = 1.52587890625e-05f;  // 2^-16
template <int R>
__global__ void __launch_bounds__(kT) k_score_slab(const float* __restrict__ pts, const uint32_t* __restrict__ off,
                                                   const uint32_t* __restrict__ item_off,
                                                   const uint32_t* __restrict__ item_cl,
                                                   const uint32_t* __restrict__ kp, int H,
                                                   const uint32_t* __restrict__ tile,
                                                   const float4* __restrict__ hyp, const float4* __restrict__ ref,
                                                   const uint32_t* __restrict__ lower, uint32_t* __restrict__ counts,
                                                   uint32_t* __restrict__ queue, float eps) {
    pdl_wait();
    const uint32_t k = *kp;
    const int T = (int)*tile;
    extern __shared__ float4 sp[];                         // T points: the near ones from the front, the others from the back
    uint32_t* hc = reinterpret_cast<uint32_t*>(sp + T);    // [H] inliers of the tile
    uint16_t* open = reinterpret_cast<uint16_t*>(hc + H);  // [H] hypotheses the bound leaves open
    uint16_t* alive = open + H;                            // [H] hypotheses still in the race
    __shared__ uint32_t s_item, s_near, s_far, s_open, s_alive, s_step;
    __shared__ int smin[kT / 32][4], smax[kT / 32][4];
    __shared__ unsigned long long sfar[kT / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    const uint32_t n_items = item_off[k];
    const float inf = __int_as_float(0x7f800000);
    if (threadIdx.x == 0) {
        uint32_t step = (uint32_t)(0.618034 * (double)n_items) | 1u;
        for (;; ++step) {  // ends: n_items + 1 is coprime to n_items
            uint32_t a = step, b = n_items;
            while (b) {
                const uint32_t t = a % b;
                a = b;
                b = t;
            }
            if (a == 1u || step > n_items) break;
        }
        s_step = step;
    }
    for (int guard = 0; guard < kLoopCap; ++guard) {
        __syncthreads();
        if (threadIdx.x == 0) {
            s_item = atomicAdd(queue, 1u);
            s_near = s_far = s_open = s_alive = 0;
        }
        for (int h = threadIdx.x; h < H; h += kT) hc[h] = 0;
        __syncthreads();
        if (s_item >= n_items) break;
        // a step coprime to the item count spreads each cluster's tiles over the launch
        const uint32_t it = (uint32_t)((unsigned long long)s_item * s_step % n_items);
        const uint32_t c = find_cluster(item_cl, item_off, k, it);
        const uint32_t start = off[c] + (it - item_off[c]) * (uint32_t)T;
        const int cnt = (int)(min(off[c + 1], start + (uint32_t)T) - start);
        const float4 r0 = ref[c];
        const float4* hy = hyp + (size_t)c * H;
        // near and other points; the near ones' bounds: x, y, z and the residual
        float lo[4] = {inf, inf, inf, inf}, hi[4] = {-inf, -inf, -inf, -inf};
#pragma unroll 4
        for (int q0 = 0; q0 < cnt; q0 += kT) {
            const int q = q0 + threadIdx.x;
            float v[4] = {0.0f, 0.0f, 0.0f, inf};
            if (q < cnt) {
                const float* p = pts + 3 * ((size_t)start + q);
                v[0] = p[0]; v[1] = p[1]; v[2] = p[2];
                v[3] = __fmaf_rn(r0.z, v[2], __fmaf_rn(r0.y, v[1], __fmaf_rn(r0.x, v[0], r0.w)));
            }
            const bool near = fabsf(v[3]) <= 0.5f * eps, far = q < cnt && !near;  // not a number: far
            const uint32_t bn = __ballot_sync(0xffffffffu, near), bf = __ballot_sync(0xffffffffu, far);
            uint32_t an = 0, af = 0;
            if (lane == 0) {
                if (bn) an = atomicAdd(&s_near, (uint32_t)__popc(bn));
                if (bf) af = atomicAdd(&s_far, (uint32_t)__popc(bf));
            }
            an = __shfl_sync(0xffffffffu, an, 0) + __popc(bn & lt);
            af = __shfl_sync(0xffffffffu, af, 0) + __popc(bf & lt);
            if (near | far) sp[near ? (int)an : T - 1 - (int)af] = make_float4(v[0], v[1], v[2], 0.0f);
            if (near)
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    lo[a] = fminf(lo[a], v[a]);
                    hi[a] = fmaxf(hi[a], v[a]);
                }
        }
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int l = __reduce_min_sync(0xffffffffu, ord(lo[a])), g = __reduce_max_sync(0xffffffffu, ord(hi[a]));
            if (lane == a) {
                smin[w][a] = l;
                smax[w][a] = g;
            }
        }
        __syncthreads();
        const int nn = (int)s_near, nf = (int)s_far;
        float ctr[3], half[3], sumM = 0.0f, rlo = 0.0f, rhi = 0.0f;
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            int l = smin[0][a], g = smax[0][a];
#pragma unroll
            for (int q = 1; q < kT / 32; ++q) {
                l = min(l, smin[q][a]);
                g = max(g, smax[q][a]);
            }
            const float fl = unord(l), fg = unord(g);
            if (a < 3) {
                ctr[a] = 0.5f * (fl + fg);
                half[a] = 0.5f * (fg - fl);
                sumM += fmaxf(fabsf(fl), fabsf(fg));
            } else {
                rlo = fl;
                rhi = fg;
            }
        }
        // the longest direction: towards the near point farthest from the box's centre
        unsigned long long best = 0;
        for (int q = threadIdx.x; q < nn; q += kT) {
            const float4 p = sp[q];
            const float dx = p.x - ctr[0], dy = p.y - ctr[1], dz = p.z - ctr[2];
            const unsigned long long key =
                ((unsigned long long)__float_as_uint(dx * dx + dy * dy + dz * dz) << 32) | (uint32_t)q;
            best = key > best ? key : best;
        }
        const uint32_t top = __reduce_max_sync(0xffffffffu, (uint32_t)(best >> 32));
        const uint32_t who = __reduce_max_sync(0xffffffffu, (uint32_t)(best >> 32) == top ? (uint32_t)best : 0u);
        if (lane == 0) sfar[w] = ((unsigned long long)top << 32) | who;
        __syncthreads();
        best = sfar[0];
#pragma unroll
        for (int q = 1; q < kT / 32; ++q) best = sfar[q] > best ? sfar[q] : best;
        float ax = 0.0f, ay = 0.0f, az = 0.0f;
        if (nn) {
            const float4 p = sp[(uint32_t)best];
            ax = p.x - ctr[0];
            ay = p.y - ctr[1];
            az = p.z - ctr[2];
        }
        const float along = ax * r0.x + ay * r0.y + az * r0.z;
        ax -= along * r0.x;
        ay -= along * r0.y;
        az -= along * r0.z;
        const float len2 = ax * ax + ay * ay + az * az;
        const bool framed = len2 > 1e-12f && len2 < 1e12f;  // else the axis-aligned box alone
        const float il = framed ? rsqrtf(len2) : 0.0f;
        ax *= il;
        ay *= il;
        az *= il;
        const float bx = r0.y * az - r0.z * ay, by = r0.z * ax - r0.x * az, bz = r0.x * ay - r0.y * ax;
        float ea = 0.0f, eb = 0.0f;
        for (int q = threadIdx.x; q < nn; q += kT) {
            const float4 p = sp[q];
            const float dx = p.x - ctr[0], dy = p.y - ctr[1], dz = p.z - ctr[2];
            ea = fmaxf(ea, fabsf(dx * ax + dy * ay + dz * az));
            eb = fmaxf(eb, fabsf(dx * bx + dy * by + dz * bz));
        }
        const uint32_t ua = __reduce_max_sync(0xffffffffu, __float_as_uint(ea));
        const uint32_t ub = __reduce_max_sync(0xffffffffu, __float_as_uint(eb));
        __syncthreads();  // smin / smax read above
        if (lane == 0) {
            smax[w][0] = (int)ua;
            smax[w][1] = (int)ub;
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kT / 32; ++q) {
            ea = fmaxf(ea, __int_as_float(smax[q][0]));
            eb = fmaxf(eb, __int_as_float(smax[q][1]));
        }
        const float rc = r0.x * ctr[0] + r0.y * ctr[1] + r0.z * ctr[2] + r0.w;
        const float er = fmaxf(fabsf(rhi - rc), fabsf(rlo - rc));
        // each hypothesis: out of the race, or all near points, none of them, or open
        const uint32_t least = lower[c];
        for (int h0 = 0; h0 < H; h0 += kT) {
            const int h = h0 + threadIdx.x;
            bool is_alive = false, is_open = false;
            if (h < H) {
                const float4 pl = hy[h];
                is_alive = fabsf(pl.w) < inf && __ldcg(counts + (size_t)c * H + h) >= least;
                if (is_alive && nn) {
                    const float dot = pl.x * r0.x + pl.y * r0.y + pl.z * r0.z, sg = dot < 0.0f ? -1.0f : 1.0f;
                    const float gx = sg * pl.x - r0.x, gy = sg * pl.y - r0.y, gz = sg * pl.z - r0.z;
                    const float mid = gx * ctr[0] + gy * ctr[1] + gz * ctr[2] + (sg * pl.w - r0.w);
                    float spread = fabsf(gx) * half[0] + fabsf(gy) * half[1] + fabsf(gz) * half[2];
                    if (framed)
                        spread = fminf(spread, fabsf(gx * ax + gy * ay + gz * az) * ea +
                                                   fabsf(gx * bx + gy * by + gz * bz) * eb +
                                                   fabsf(gx * r0.x + gy * r0.y + gz * r0.z) * er);
                    spread += kSlabErr * (fabsf(pl.w) + fabsf(r0.w) + sumM);
                    const float s_lo = rlo + mid - spread, s_hi = rhi + mid + spread;
                    if (s_lo >= -eps && s_hi <= eps) hc[h] = (uint32_t)nn;
                    else is_open = !(s_lo > eps || s_hi < -eps);
                }
            }
            const uint32_t bo = __ballot_sync(0xffffffffu, is_open), ba = __ballot_sync(0xffffffffu, is_alive);
            uint32_t ao = 0, aa = 0;
            if (lane == 0) {
                if (bo) ao = atomicAdd(&s_open, (uint32_t)__popc(bo));
                if (ba) aa = atomicAdd(&s_alive, (uint32_t)__popc(ba));
            }
            ao = __shfl_sync(0xffffffffu, ao, 0) + __popc(bo & lt);
            aa = __shfl_sync(0xffffffffu, aa, 0) + __popc(ba & lt);
            if (is_open) open[ao] = (uint16_t)h;
            if (is_alive) alive[aa] = (uint16_t)h;
        }
        __syncthreads();
        // the points off the plane against every live hypothesis, the near ones against the open ones
#pragma unroll 1
        for (int pass = 0; pass < 2; ++pass) {
            const int nh = (int)(pass ? s_open : s_alive), np = pass ? nn : nf;
            if (!nh || !np) continue;
            const int G = (nh + R - 1) / R, P = kT / G;  // threads per point subset, point subsets
            const int g = threadIdx.x / G, j = threadIdx.x % G;
            if (g >= P) continue;
            const float4* src = pass ? sp : sp + (T - nf);
            float4 pl[R];
            uint32_t acc[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int h = j * R + r;
                pl[r] = h < nh ? hy[pass ? open[h] : alive[h]] : make_float4(0.0f, 0.0f, 0.0f, inf);
                acc[r] = 0;
            }
            int q = g;
            for (; q + P < np; q += 2 * P) count_points2<R>(pl, src[q], src[q + P], eps, acc);
            if (q < np) count_point<R>(pl, src[q], eps, acc);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int h = j * R + r;
                if (h < nh && acc[r]) atomicAdd(&hc[pass ? (int)open[h] : (int)alive[h]], acc[r]);
            }
        }
        __syncthreads();
        for (uint32_t a = threadIdx.x; a < s_alive; a += kT) {
            const int h = alive[a];
            if (hc[h] < (uint32_t)cnt) atomicSub(&counts[(size_t)c * H + h], (uint32_t)cnt - hc[h]);
        }
    }
}

// The scoring launch's arguments (stage b).
struct ScoreArgs {
    const float* pts;
    const uint32_t* off;
    const uint32_t* item_off;
    const uint32_t* item_cl;  // item -> cluster table, or null for a binary search
    const uint32_t* kp;
    int H, T;              // T: the largest tile, which sizes shared memory
    const uint32_t* tile;  // the tile (device)
    const float4* hyp;
    uint32_t* counts;
    uint32_t* queue;
    float eps;
    int grid;
    bool early;  // launched while stage a runs (see launch_fit)
};

template <int R>
cudaError_t launch_score(const ScoreArgs& a, cudaStream_t s) {
    const int G = (a.H + R - 1) / R;
    const int P = kT / G;
    const size_t smem = (size_t)a.T * sizeof(float4) + (size_t)P * G * R * sizeof(uint32_t);
    launch_as(a.early, k_score<R>, dim3(a.grid), dim3(kT), smem, s, a.pts, a.off, a.item_off, a.item_cl, a.kp, a.H, a.tile,
                a.hyp, a.counts, a.queue, a.eps);
    return cudaGetLastError();
}

// Large fits: the reference planes and their inliers, then the slab scoring.
template <int R>
cudaError_t launch_score_slab(const ScoreArgs& a, float4* ref, uint32_t* lower, unsigned cgrid, unsigned igrid,
                              cudaStream_t s) {
    const size_t smem = (size_t)a.T * sizeof(float4) + (size_t)a.H * 8;
    launch_k(k_score_ref, dim3(cgrid), dim3(kT), 0, s, a.pts, a.off, a.kp, a.H, a.hyp, ref, a.eps);
    launch_full(k_score_lower, dim3(igrid), dim3(kT), 0, s, a.pts, a.off, a.item_off, a.item_cl, a.kp, a.tile, ref,
                lower, a.eps);
    launch_full(k_score_slab<R>, dim3(a.grid), dim3(kT), smem, s, a.pts, a.off, a.item_off, a.item_cl, a.kp, a.H,
                a.tile, a.hyp, ref, lower, a.counts, a.queue, a.eps);
    count_launch(2);
    return cudaGetLastError();
}

template <int R>
cudaError_t launch_score_warp(const ScoreArgs& a, cudaStream_t s) {
    const size_t smem = (size_t)(kT / 32) * a.T * sizeof(float4);
    launch_full(k_score_warp<R>, dim3(a.grid), dim3(kT), smem, s, a.pts, a.off, a.item_off, a.item_cl, a.kp, a.H,
                a.tile, a.hyp, a.counts, a.queue, a.eps);
    return cudaGetLastError();
}

__global__ void k_set_u32(uint32_t* __restrict__ p, uint32_t v) { pdl_gate(); *p = v; }

}  // namespace

FitTuning default_tuning() { return FitTuning{2048, 4, 4, 0, 1}; }

FitTuning tuning_of(const vm_fit_tuning& t) {
    FitTuning f{(int)t.tile, (int)t.hyp_per_thread, (int)t.ctas_per_sm, (int)t.schedule, 0};
    const FitTuning d = default_tuning();
    f.adapt = f.tile == d.tile && f.hyp_per_thread == d.hyp_per_thread && f.ctas_per_sm == d.ctas_per_sm &&
              f.schedule == d.schedule;
    return f;
}

// The scoring variant launch_fit picks for t and H: hypotheses per thread
// and whether the warp schedule applies.
static void score_variant(const FitTuning& t, int H, int& R, bool& warp) {
    R = t.hyp_per_thread;
    warp = t.schedule == 1 && H <= 256 && (size_t)(kT / 32) * t.tile * sizeof(float4) <= 200 * 1024;
    if (warp) {
        while (R < 8 && (H + R - 1) / R > 32) R <<= 1;
    } else {
        while (R < 8 && (H + R - 1) / R > kT) R <<= 1;
    }
}

int score_max_ctas_per_sm(const FitTuning& t, int H) {
    fit_init_attributes();
    int R;
    bool warp;
    score_variant(t, H, R, warp);
    const int G = (H + R - 1) / R;
    const size_t smem = warp ? (size_t)(kT / 32) * t.tile * sizeof(float4)
                             : (size_t)t.tile * sizeof(float4) + (size_t)(kT / G) * G * R * sizeof(uint32_t);
    int n = 0;
    cudaError_t e;
    if (warp) {
        switch (R) {
            case 1: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_score_warp<1>, kT, smem); break;
            case 2: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_score_warp<2>, kT, smem); break;
            case 4: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_score_warp<4>, kT, smem); break;
            default: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_score_warp<8>, kT, smem); break;
        }
    } else {
        switch (R) {
            case 1: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_score<1>, kT, smem); break;
            case 2: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_score<2>, kT, smem); break;
            case 8: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_score<8>, kT, smem); break;
            default: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_score<4>, kT, smem); break;
        }
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

size_t fit_hull_smem() {
    constexpr size_t chains = kHullCap * (sizeof(unsigned long long) + 2 * sizeof(uint32_t));
    constexpr size_t staged = kSurvCap * sizeof(int2);
    return kHullCap * sizeof(unsigned long long) + (chains > staged ? chains : staged);
}

void fit_init_attributes() {
    static std::once_flag once;  // maps on several host threads may reach here together
    std::call_once(once, [] {
        cudaFuncSetAttribute(k_hull, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fit_hull_smem());
        cudaFuncSetAttribute(k_score<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        cudaFuncSetAttribute(k_score<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        cudaFuncSetAttribute(k_score<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        cudaFuncSetAttribute(k_score<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        cudaFuncSetAttribute(k_score_warp<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        cudaFuncSetAttribute(k_score_slab<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, 208 * 1024);
        cudaFuncSetAttribute(k_score_warp<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        cudaFuncSetAttribute(k_score_slab<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, 208 * 1024);
        cudaFuncSetAttribute(k_score_warp<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        cudaFuncSetAttribute(k_score_slab<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, 208 * 1024);
        cudaFuncSetAttribute(k_score_warp<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        cudaFuncSetAttribute(k_score_slab<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, 208 * 1024);
    });
}

cudaError_t launch_fit(const float* pts, const uint32_t* off, const uint32_t* labels, const uint32_t* kp,
                       uint32_t kcap, const vm_segment_params& p, FitBuffers& fb, const FitTuning& t, int sms,
                       cudaStream_t s, StageHook* hk, uint32_t round) {
    if (kcap == 0) return cudaSuccess;
    fit_init_attributes();
    const int H = (int)p.n_hyp;
    const int T = (t.tile + (int)kChunk - 1) / (int)kChunk * (int)kChunk;  // callers validate; never below a chunk
    cudaError_t e;
    VM_STAGE_BEGIN(hk, kStHyp, s);
    const uint32_t adapt = t.adapt ? (uint32_t)(sms * t.ctas_per_sm) : 0u;
    const uint32_t* tile = fb.queue + 1;
    if (kcap <= kItemsScanMax) {
        launch_k(k_items_scan, dim3(1), dim3(kItemsScanT), 0, s, off, kp, (uint32_t)T, adapt, fb.item_off, fb.queue,
                 fb.done);
        count_launch(1);
    } else {
        const unsigned kgrid = (kcap + kT - 1) / kT < (uint32_t)sms * 8 ? (kcap + kT - 1) / kT : (uint32_t)sms * 8;
        launch_k(k_items, dim3(kgrid), dim3(kT), 0, s, off, kp, (uint32_t)T, adapt, fb.item_off, fb.queue, fb.done);
        e = exclusive_scan_dev(fb.item_off, fb.item_off, fb.tot, kp, kcap, fb.scan_tmp, s, fb.err, true);
        if (e != cudaSuccess) return e;
        count_launch(1);
    }
    // The warp schedule needs ceil(H / R) <= 32 lanes with R <= 8 and its
    // per-warp tiles within the shared-memory limit; otherwise the CTA one
    // runs, with at most one subset row of kT threads.
    int R;
    bool warp;
    score_variant(t, H, R, warp);
    // Small fits (a map's segmentation) compute each cluster's centroid and
    // refit in the kernel before them, triggered by per-cluster completion
    // counters: that removes two dependent launches.  In large batches the
    // counters' fences wait, per work item, for the item's contended atomics,
    // which costs more than the launches; they take the separate kernels.
    // Large fits also score by k_score_slab, which makes two passes more and
    // far fewer tests (small ones are bound by their launches).  Results are
    // the same.
    uint32_t* done = fb.large ? nullptr : fb.done;
    const bool slab = !done && !warp && p.eps < 1e6f;
    const size_t kh = (size_t)kcap * H;
    const unsigned hgrid = (unsigned)((kh + kT - 1) / kT < (size_t)sms * 16 ? (kh + kT - 1) / kT : (size_t)sms * 16);
    launch_k(k_hyp, dim3(hgrid), dim3(kT), 0, s, pts, off, labels, kp, H, p.seed, round, fb.hyp, fb.hyp_valid,
             fb.counts, fb.item_off, fb.item_cl, fb.lower, slab);
    VM_STAGE_END(hk, kStHyp, s);
    count_launch(1);
    const int grid = sms * t.ctas_per_sm;
    VM_STAGE_BEGIN(hk, kStScore, s);
    // Scoring launched while stage a runs lands unevenly beside stage a's CTAs (a walk map: 13.9 us for 12.1); where
    // those take at most half of the SMs it does not, and a direct fit gains the 2 us of a launch.
    const bool early = hgrid * 2 <= (unsigned)sms;
    const ScoreArgs sa{pts, off, fb.item_off, fb.item_cl, kp, H, T, tile, fb.hyp, fb.counts, fb.queue, p.eps, grid, early};
    const unsigned cgrid = kcap < (uint32_t)sms * 8 ? kcap : (uint32_t)sms * 8;
    // A small fit has about four items an SM.  Of a large fit's many a CTA takes few, so that the last ones to finish
    // leave little idle (2,000 clusters, extraction and filter: 776 us at 8 CTAs an SM, 740 at 64, 765 at 256).
    const unsigned igrid = (unsigned)sms * (done ? 8 : 64);
    if (warp) {
        switch (R) {
            case 1: e = launch_score_warp<1>(sa, s); break;
            case 2: e = launch_score_warp<2>(sa, s); break;
            case 4: e = launch_score_warp<4>(sa, s); break;
            default: e = launch_score_warp<8>(sa, s); break;
        }
    } else if (slab) {
        switch (R) {
            case 1: e = launch_score_slab<1>(sa, fb.ref, fb.lower, cgrid, igrid, s); break;
            case 2: e = launch_score_slab<2>(sa, fb.ref, fb.lower, cgrid, igrid, s); break;
            case 8: e = launch_score_slab<8>(sa, fb.ref, fb.lower, cgrid, igrid, s); break;
            default: e = launch_score_slab<4>(sa, fb.ref, fb.lower, cgrid, igrid, s); break;
        }
    } else {
        switch (R) {
            case 1: e = launch_score<1>(sa, s); break;
            case 2: e = launch_score<2>(sa, s); break;
            case 8: e = launch_score<8>(sa, s); break;
            default: e = launch_score<4>(sa, s); break;
        }
    }
    if (e != cudaSuccess) return e;
    VM_STAGE_END(hk, kStScore, s);
    count_launch(1);
    // stage c (k_select, a CTA per cluster), then the extraction; with the
    // completion counters the centroid runs in the extraction kernel and the
    // refit in the filter kernel, otherwise as kernels of their own
    VM_STAGE_BEGIN(hk, kStExtract, s);
    launch_k(k_select, dim3(cgrid), dim3(kT), 0, s, pts, off, kp, H, fb.hyp, fb.hyp_valid, fb.counts, fb.cl);
    count_launch(1);
    launch_as(done != nullptr, done ? k_extract<true> : k_extract<false>, dim3(igrid), dim3(kT), 0, s, pts, off, fb.item_off,
                fb.item_cl, kp, tile, fb.cl, fb.inlier, fb.part, p.eps, fb.err, done, fb.cen, fb.poly);
    if (!done) {
        launch_k(k_centroid, dim3(cgrid), dim3(kT), 0, s, pts, off, fb.item_off, kp, tile, fb.part, fb.cl,
                 fb.cen, fb.poly);
        count_launch(1);
    }
    launch_as(done != nullptr, done ? k_filter<true> : k_filter<false>, dim3(igrid), dim3(kT), 0, s, pts, off, fb.item_off,
                fb.item_cl, kp, tile, fb.cl, fb.inlier, fb.cen, fb.poly, fb.part, fb.surv, done);
    VM_STAGE_END(hk, kStExtract, s);
    count_launch(2);
    VM_STAGE_BEGIN(hk, kStHull, s);
    if (!done) {
        launch_k(k_refit, dim3(cgrid), dim3(kT), 0, s, off, fb.item_off, kp, tile, fb.part, fb.cen, fb.cl);
        count_launch(1);
    }
    // as many CTAs as run at once: a cluster takes about as long as another, and the last CTA's count of the finished ones
    // is shorter (a walk map 231 us for 234 with a CTA for every cluster the scratch has room for)
    const unsigned hull_grid = cgrid < (unsigned)sms * 2 ? cgrid : (unsigned)sms * 2;
    launch_k(k_hull, dim3(hull_grid), dim3(kT), fit_hull_smem(), s, off, kp, fb.cl, fb.surv, fb.hull, fb.hull_cnt, fb.err,
             fb.queue + 3);
    VM_STAGE_END(hk, kStHull, s);
    count_launch(1);
    return cudaGetLastError();
}

cudaError_t launch_pack(const FitBuffers& fb, const uint32_t* off, const uint32_t* labels, const uint32_t* kp,
                        uint32_t kcap, vm_plane* planes, int32_t* hull_xy, float* hull_xyz, uint32_t hull_cap,
                        cudaStream_t s, const HeaderArgs* header) {
    if (kcap == 0) return cudaSuccess;
    const HeaderArgs ha = header ? *header : HeaderArgs{};
    launch_k(k_pack, dim3(kcap < 4096 ? kcap : 4096), dim3(128), 0, s, off, labels, kp, fb.cl, fb.hull, fb.hull_cnt,
             planes, hull_xy, hull_xyz, hull_cap, ha);
    count_launch(1);
    return cudaGetLastError();
}

}  // namespace vmx

// ---------------------------------------------------------------- no-allocation RANSAC
// vm_ransac_static runs the same hypothesis / scoring / selection kernels as
// vm_fit_planes, but every scratch buffer lives in one file-scope device array
// instead of memory obtained from cudaMalloc.  It exists for callers that may
// not allocate device memory once they are running -- a control loop with a
// hard deadline (cudaMalloc can block on device-wide synchronisation for an
// unbounded time), or a host program whose device memory is owned up front by
// another allocator.  The array is sized for at most kStaticMaxClusters
// clusters and kStaticMaxSlots (clusters x hypotheses); every GPU that loads
// the library holds it (about 11 MiB) until the process exits.
namespace vmx {
namespace {

constexpr uint32_t kStaticMaxClusters = 4096;
constexpr uint32_t kStaticMaxSlots = 524288;  // clusters x hypotheses

constexpr size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }
constexpr size_t kOffHyp = 0;
constexpr size_t kOffCounts = kOffHyp + align256((size_t)kStaticMaxSlots * sizeof(float4));
constexpr size_t kOffValid = kOffCounts + align256((size_t)kStaticMaxSlots * sizeof(uint32_t));
constexpr size_t kOffCl = kOffValid + align256((size_t)kStaticMaxSlots);
constexpr size_t kOffItems = kOffCl + align256((size_t)kStaticMaxClusters * sizeof(FitCluster));
constexpr size_t kOffQueue = kOffItems + align256((size_t)(kStaticMaxClusters + 1) * sizeof(uint32_t));
constexpr size_t kOffScan = kOffQueue + 256;  // the queue area also holds the count and a scan total
constexpr size_t kScanWords = 64;
static_assert(kScanWords >= scan_tmp_words(kStaticMaxClusters + 1), "static scan scratch too small");
constexpr size_t kStaticBytes = kOffScan + align256(kScanWords * sizeof(uint32_t));

// Copies the selected plane, hypothesis index and inlier count of each cluster
// to the caller's arrays.
__global__ void k_static_out(const FitCluster* __restrict__ cl, const uint32_t* __restrict__ kp,
                             float* __restrict__ planes, int32_t* __restrict__ best_h, uint32_t* __restrict__ inliers) {
    pdl_gate();
    const uint32_t k = *kp;
    for (uint32_t c = blockIdx.x * kT + threadIdx.x; c < k; c += gridDim.x * kT) {
        const FitCluster f = cl[c];
        planes[4 * c + 0] = f.n[0];
        planes[4 * c + 1] = f.n[1];
        planes[4 * c + 2] = f.n[2];
        planes[4 * c + 3] = f.d;
        best_h[c] = f.best_h;
        inliers[c] = f.best_h >= 0 ? f.inliers : 0u;
    }
}

}  // namespace
}  // namespace vmx

static __device__ __align__(256) unsigned char g_ransac_scratch[vmx::kStaticBytes];

namespace {
// Device address of g_ransac_scratch per device ordinal, looked up once per
// device (with that device current) by the first call made on it.
constexpr int kMaxDevices = 64;
std::mutex g_static_mu;
void* g_static_addr[kMaxDevices] = {};
}  // namespace

extern "C" vm_status vm_ransac_static(const float* xyz, const uint32_t* off, const uint32_t* labels, uint32_t k,
                                      const vm_segment_params* params, void* stream, float* planes_out,
                                      int32_t* best_h_out, uint32_t* inliers_out) {
    using namespace vmx;
    if (!params || (k && (!xyz || !off || !planes_out || !best_h_out || !inliers_out))) {
        set_error("vm_ransac_static: null argument");
        return VM_ERR_INVALID_ARG;
    }
    if (params->n_hyp < 1 || params->n_hyp > 1024 || !(params->eps >= 0.0f) || params->planes_per_cluster > 1) {
        set_error("vm_ransac_static: n_hyp must be in [1, 1024], eps >= 0 and planes_per_cluster <= 1");
        return VM_ERR_INVALID_ARG;
    }
    if (k > kStaticMaxClusters || (uint64_t)k * params->n_hyp > kStaticMaxSlots) {
        set_error("vm_ransac_static: " + std::to_string(k) + " clusters x " + std::to_string(params->n_hyp) +
                  " hypotheses exceed the static scratch (at most " + std::to_string(kStaticMaxClusters) +
                  " clusters and " + std::to_string(kStaticMaxSlots) + " cluster-hypothesis pairs)");
        return VM_ERR_CAPACITY;
    }
    // The address lookup comes before the k == 0 return, so an empty call
    // serves as the set-up call that loads the array on this device.
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_status(e, "cudaGetDevice");
    if (dev < 0 || dev >= kMaxDevices) {
        set_error("vm_ransac_static: device ordinal out of range");
        return VM_ERR_INVALID_ARG;
    }
    char* base;
    {
        std::lock_guard<std::mutex> lk(g_static_mu);
        if (!g_static_addr[dev]) {
            void* p = nullptr;
            e = cudaGetSymbolAddress(&p, g_ransac_scratch);
            if (e != cudaSuccess) return cuda_status(e, "cudaGetSymbolAddress(g_ransac_scratch)");
            g_static_addr[dev] = p;
        }
        base = static_cast<char*>(g_static_addr[dev]);
    }
    if (k == 0) return VM_OK;
    const int H = (int)params->n_hyp;
    const FitTuning t = default_tuning();
    float4* hyp = reinterpret_cast<float4*>(base + kOffHyp);
    uint32_t* counts = reinterpret_cast<uint32_t*>(base + kOffCounts);
    uint8_t* valid = reinterpret_cast<uint8_t*>(base + kOffValid);
    FitCluster* cl = reinterpret_cast<FitCluster*>(base + kOffCl);
    uint32_t* item_off = reinterpret_cast<uint32_t*>(base + kOffItems);
    uint32_t* queue = reinterpret_cast<uint32_t*>(base + kOffQueue);
    uint32_t* kdev = queue + 8;
    uint32_t* total = queue + 9;
    uint32_t* scan_tmp = reinterpret_cast<uint32_t*>(base + kOffScan);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 1;
    fit_init_attributes();
    // the work queue starts at zero every call (k_items); counts are zeroed by k_hyp
    launch_k(k_set_u32, dim3(1), dim3(1), 0, s, kdev, k);
    launch_k(k_items, dim3((k + kT - 1) / kT), dim3(kT), 0, s, off, kdev, (uint32_t)t.tile, 0u, item_off, queue,
             static_cast<uint32_t*>(nullptr));
    if ((e = exclusive_scan_dev(item_off, item_off, total, kdev, k, scan_tmp, s, nullptr, true)) != cudaSuccess)
        return cuda_status(e, "scan");
    const size_t kh = (size_t)k * H;
    const unsigned hgrid = (unsigned)((kh + kT - 1) / kT < (size_t)sms * 16 ? (kh + kT - 1) / kT : (size_t)sms * 16);
    launch_k(k_hyp, dim3(hgrid), dim3(kT), 0, s, xyz, off, labels, kdev, H, params->seed, 0u, hyp, valid, counts,
             item_off, static_cast<uint32_t*>(nullptr), static_cast<uint32_t*>(nullptr), false);
    // The CTA-per-item schedule whatever the tuning asks for: with no
    // item -> cluster table here, the clusters of work items come from a
    // binary search, which only that schedule does.
    FitTuning tc = t;
    tc.schedule = 0;
    int R;
    bool warp;
    score_variant(tc, H, R, warp);
    const int grid = sms * t.ctas_per_sm;
    const ScoreArgs sa{xyz, off, item_off, nullptr, kdev, H, t.tile, queue + 1, hyp, counts, queue, params->eps, grid, false};
    switch (R) {
        case 1: e = launch_score<1>(sa, s); break;
        case 2: e = launch_score<2>(sa, s); break;
        case 8: e = launch_score<8>(sa, s); break;
        default: e = launch_score<4>(sa, s); break;
    }
    if (e != cudaSuccess) return cuda_status(e, "k_score");
    const unsigned cgrid = k < (uint32_t)sms * 8 ? k : (uint32_t)sms * 8;
    launch_k(k_select, dim3(cgrid), dim3(kT), 0, s, xyz, off, kdev, H, hyp, valid, counts, cl);
    launch_k(k_static_out, dim3((k + kT - 1) / kT), dim3(kT), 0, s, cl, kdev, planes_out, best_h_out, inliers_out);
    count_launch(6);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_status(e, "vm_ransac_static launch");
    return VM_OK;
}
