// segment.cu -- multi-plane segmentation up to the cluster point lists
// (Sec. III.C): mean positions from the exact sums, normals and steppable
// classification (Eq. 3, Eq. 4), clustering (Algorithm 1) and cluster
// formation.
//
// Layout.  About a fifth of the voxel slots of an allocated brick are occupied
// (surfaces), so every per-voxel array holds the occupied voxels only, in
// voxel-id order: bricks ranked by key, and inside a brick the set bits of its
// occupancy bitmap.  A neighbour's entry follows from its brick's record (one
// 128-byte line: bitmap, counts before each bitmap word, first entry) with a
// popcount.  At frame 300 of the 4 x 4 x 2 m trajectory at 0.01 m that is
// 0.28 M entries in place of 1.35 M slots, at 8 x 8 x 3 m 1.4 M in place of 8 M.
//
// Clustering works on components, not voxels: k_ccl_local joins voxels inside
// each brick, k_ccl_cross lists the pairs of in-brick components that touch
// across a border, and the forest over the components (a few per brick) is
// small enough for one SM's shared memory.  Components are numbered in the
// order of their smallest voxel, so a root with the smallest number holds the
// smallest voxel id -- the fixed point of Algorithm 1's min-label propagation.
#include <climits>
#include <cstddef>
#include <mutex>

#include "vm_internal.cuh"

namespace vmx {
namespace {

constexpr int kT = 256;
constexpr float kInvQ = 9.5367431640625e-07f;  // 2^-20

__device__ __forceinline__ void brick_coords(int32_t key, const Grid& g, int& bx, int& by, int& bz) {
    bx = key % g.nbx;
    by = (key / g.nbx) % g.nby;
    bz = key / (g.nbx * g.nby);
}

// Row (y, z) of a brick's halo, y, z in -1 .. 8: the occupied cells x = -1 .. 8
// as bits 0 .. 9, and the entries of cell -1, of the first occupied cell of x
// = 0 .. 7 and of cell 8 (meaningless where the cells are free).  nb: the ranks
// of the 27 bricks around.
__device__ __forceinline__ uint4 halo_row(const BrickRec* __restrict__ brec, const int32_t* nb, int y, int z) {
    const int by = y < 0 ? 0 : (y > 7 ? 2 : 1), bz = z < 0 ? 0 : (z > 7 ? 2 : 1);
    const int w = (z & 7) * 2 + ((y & 7) >> 2), sh = (y & 3) * 8;
    uint32_t byte[3] = {0u, 0u, 0u}, at[3] = {0u, 0u, 0u};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const int32_t rk = nb[bz * 9 + by * 3 + d];
        if (rk >= 0) {
            const BrickRec* b = brec + rk;
            const uint32_t m = b->mask[w];
            byte[d] = (m >> sh) & 0xffu;
            at[d] = b->base + b->pre[w] + __popc(m & ((1u << sh) - 1u));
        }
    }
    return make_uint4((byte[0] >> 7) | (byte[1] << 1) | ((byte[2] & 1u) << 9), at[0] + __popc(byte[0]) - 1u, at[1],
                      at[2]);
}

// The entries of cells x - 1, x, x + 1 of a halo row (x in 0 .. 7); win: which
// of them are occupied (bits 0 .. 2).
__device__ __forceinline__ void row_window(const uint4& row, int x, uint32_t& win, uint32_t idx[3]) {
    win = (row.x >> x) & 7u;
    const uint32_t at = row.z + __popc((row.x >> 1) & ((1u << x) - 1u));
    idx[0] = x > 0 ? at - 1u : row.y;
    idx[1] = at;
    idx[2] = x < 7 ? at + ((win >> 1) & 1u) : row.w;
}

// Mean of each occupied voxel: M = floor((2 S + c) / (2 c)), the exact integer
// mean in 2^-20 m units rounded half up (Eq. 1's mu up to that quantum).  A
// warp takes a brick: its bitmap is expanded to a list of voxel indices, then
// every lane has an occupied voxel (a lane per slot left four of five idle in
// the 64-bit divisions).  The warp also looks the 27 bricks around up and
// forms the brick's 10 x 10 halo rows (the occupied cells and their entries),
// which the window moments and the cross-brick joins read: one chain of
// dependent loads here in place of one in each of those.
constexpr int kFinWarps = kT / 32;
__global__ void __launch_bounds__(kT) k_finalize(SegCounters* __restrict__ ctr, uint32_t cap_b, Grid g,
                                                 const BrickRec* __restrict__ brec,
                                                 const int32_t* __restrict__ rank_table,
                                                 const unsigned long long* __restrict__ S,
                                                 const uint32_t* __restrict__ C, int4* __restrict__ M,
                                                 uint32_t* __restrict__ vox, int32_t* __restrict__ near,
                                                 uint4* __restrict__ rows) {
    pdl_gate();
    __shared__ uint16_t slist[kFinWarps][kBrickVox];
    __shared__ int32_t snb[kFinWarps][27];
    const uint32_t n_all = ctr->n_sorted, n_sorted = min(n_all, cap_b);
    // more bricks than the scratch was sized for: the kernels clamp to it, the
    // host regrows and reruns
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        ctr->n_vox = n_all > cap_b ? brec[cap_b].base : ctr->n_occ;
        if (n_all > cap_b) atomicOr(&ctr->err, kErrScratch);
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint16_t* list = slist[w];
    int32_t* nb = snb[w];
    const uint32_t lt = (1u << lane) - 1u;
    for (uint32_t r = blockIdx.x * kFinWarps + w; r < n_sorted; r += gridDim.x * kFinWarps) {
        const BrickRec* br = brec + r;
        const uint4 hd = *reinterpret_cast<const uint4*>(&br->base);  // base, n, key, slot
        const uint32_t mine = lane < 16 ? br->mask[lane] : 0u, pre = lane < 16 ? br->pre[lane] : 0u;
        int32_t rk = -1;
        if (lane < 27) {
            int x, y, z;
            brick_coords((int32_t)hd.z, g, x, y, z);
            x += lane % 3 - 1;
            y += (lane / 3) % 3 - 1;
            z += lane / 9 - 1;
            if (x >= 0 && y >= 0 && z >= 0 && x < g.nbx && y < g.nby && z < g.nbz)
                rk = rank_table[(z * g.nby + y) * g.nbx + x];
            if (rk >= (int32_t)n_sorted) rk = -1;  // beyond the scratch
        }
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            const uint32_t m = __shfl_sync(0xffffffffu, mine, q), p = __shfl_sync(0xffffffffu, pre, q);
            if ((m >> lane) & 1u) list[p + __popc(m & lt)] = (uint16_t)(q * 32 + lane);
        }
        if (lane < 27) {
            nb[lane] = rk;
            near[(size_t)r * 27 + lane] = rk;
        }
        __syncwarp();
        for (uint32_t p = lane; p < hd.y; p += 32) {
            const uint32_t l = list[p];
            const unsigned long long* s = S + (size_t)hd.w * 3 * kBrickVox + l;
            const long long c = (long long)C[(size_t)hd.w * kBrickVox + l], c2 = 2ll * c;
            const long long s0 = (long long)s[0], s1 = (long long)s[kBrickVox], s2 = (long long)s[2 * kBrickVox];
            M[hd.x + p] = make_int4((int32_t)((2ll * s0 + c) / c2), (int32_t)((2ll * s1 + c) / c2),
                                    (int32_t)((2ll * s2 + c) / c2), 0);
            vox[hd.x + p] = r * kBrickVox + l;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int t = q * 32 + lane;
            if (t < 100) rows[(size_t)r * 100 + t] = halo_row(brec, nb, t % 10 - 1, t / 10 - 1);
        }
    }
}

// ---------------------------------------------------------------- Jacobi (FP32)
// Cyclic Jacobi (Golub & Van Loan Sec. 8.5) on a symmetric 3x3 matrix, pairs
// (0,1), (0,2), (1,2), a fixed number of sweeps, pairs with a_pq == 0 skipped;
// tau = (a_qq - a_pp) / (2 a_pq), t = sgn(tau) / (|tau| + sqrt(1 + tau^2)),
// c = 1 / sqrt(1 + t^2), s = t c.  Every operation is an explicit IEEE
// round-to-nearest intrinsic; the reciprocals are those of the division (both
// round the exact value once) in fewer instructions, which bound k_eigen: 83.4 ->
// 77.9 us for the 8 x 8 x 3 m map's 1.4 M voxels.
__device__ __forceinline__ void jacobi3(float a00, float a11, float a22, float a01, float a02, float a12, int sweeps,
                                        float v[3][3], float d[3]) {
    float a[3][3] = {{a00, a01, a02}, {a01, a11, a12}, {a02, a12, a22}};
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c) v[r][c] = (r == c) ? 1.0f : 0.0f;
    for (int sw = 0; sw < sweeps; ++sw) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int p = (k == 2) ? 1 : 0, q = (k == 0) ? 1 : 2, r = 2 - k;
            const float apq = a[p][q];
            if (apq == 0.0f) continue;
            const float app = a[p][p], aqq = a[q][q];
            const float tau = __fdiv_rn(__fsub_rn(aqq, app), __fmul_rn(2.0f, apq));
            const float sg = (tau >= 0.0f) ? 1.0f : -1.0f;
            const float t = sg * __frcp_rn(__fadd_rn(fabsf(tau), __fsqrt_rn(__fmaf_rn(tau, tau, 1.0f))));
            const float c = __frcp_rn(__fsqrt_rn(__fmaf_rn(t, t, 1.0f)));
            const float s = __fmul_rn(t, c);
            a[p][p] = __fmaf_rn(-t, apq, app);
            a[q][q] = __fmaf_rn(t, apq, aqq);
            a[p][q] = 0.0f;
            a[q][p] = 0.0f;
            const float arp = a[r][p], arq = a[r][q];
            const float nrp = __fmaf_rn(c, arp, -__fmul_rn(s, arq));
            const float nrq = __fmaf_rn(s, arp, __fmul_rn(c, arq));
            a[r][p] = nrp; a[p][r] = nrp;
            a[r][q] = nrq; a[q][r] = nrq;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const float vip = v[i][p], viq = v[i][q];
                v[i][p] = __fmaf_rn(c, vip, -__fmul_rn(s, viq));
                v[i][q] = __fmaf_rn(s, vip, __fmul_rn(c, viq));
            }
        }
    }
    d[0] = a[0][0]; d[1] = a[1][1]; d[2] = a[2][2];
}

// Column of the smallest diagonal entry (lowest index on ties), scaled by
// 1/sqrt(n.n), oriented n_z >= 0 (then n_y, then n_x when zero).
__device__ __forceinline__ void pick_normal(float v[3][3], const float d[3], float n[3]) {
    int m = 0;
    if (d[1] < d[m]) m = 1;
    if (d[2] < d[m]) m = 2;
    float x = (m == 0) ? v[0][0] : (m == 1) ? v[0][1] : v[0][2];
    float y = (m == 0) ? v[1][0] : (m == 1) ? v[1][1] : v[1][2];
    float z = (m == 0) ? v[2][0] : (m == 1) ? v[2][1] : v[2][2];
    const float nn = __fmaf_rn(z, z, __fmaf_rn(y, y, __fmul_rn(x, x)));
    const float inv = __frcp_rn(__fsqrt_rn(nn));
    x = __fmul_rn(x, inv); y = __fmul_rn(y, inv); z = __fmul_rn(z, inv);
    const bool flip = (z < 0.0f) || (z == 0.0f && (y < 0.0f || (y == 0.0f && x < 0.0f)));
    if (flip) { x = -x; y = -y; z = -z; }
    n[0] = x; n[1] = y; n[2] = z;
}

// ---------------------------------------------------------------- union-find
// Global forest over component numbers.  Hooking always puts the larger root
// under the smaller, so every root is the smallest index of its tree.
__device__ __forceinline__ uint32_t uf_find(uint32_t* P, uint32_t x, uint32_t* err) {
    for (int it = 0; it < kLoopCap; ++it) {
        const uint32_t p = __ldcg(P + x);
        if (p == x) return x;
        const uint32_t gp = __ldcg(P + p);
        if (gp != p) P[x] = gp;  // path halving: gp is an ancestor of x
        x = gp;
    }
    atomicOr(err, kErrTimeout);
    return x;
}

__device__ __forceinline__ void uf_union(uint32_t* P, uint32_t a, uint32_t b, uint32_t* err) {
    for (int it = 0; it < kLoopCap; ++it) {
        a = uf_find(P, a, err);
        b = uf_find(P, b, err);
        if (a == b) return;
        const uint32_t hi = a > b ? a : b, lo = a > b ? b : a;
        const uint32_t old = atomicCAS(P + hi, hi, lo);
        if (old == hi) return;
        a = old;  // hi was hooked meanwhile: continue from its new parent
        b = lo;
    }
    atomicOr(err, kErrTimeout);
}

// Algorithm 1's edge test: |mu_i - mu_j|^2 < d_th^2 and |n_i . n_j| > cos_ccl
// (symmetric in i and j).
__device__ __forceinline__ bool ccl_edge(float ax, float ay, float az, float anx, float any, float anz, float bx,
                                         float by, float bz, float bnx, float bny, float bnz, float d_th2,
                                         float cos_ccl) {
    const float ex = __fsub_rn(ax, bx), ey = __fsub_rn(ay, by), ez = __fsub_rn(az, bz);
    const float d2 = __fmaf_rn(ez, ez, __fmaf_rn(ey, ey, __fmul_rn(ex, ex)));
    const float cs = __fmaf_rn(anz, bnz, __fmaf_rn(any, bny, __fmul_rn(anx, bnx)));
    return d2 < d_th2 && fabsf(cs) > cos_ccl;
}

__device__ __forceinline__ float mean_pos(float o, int32_t m) {
    return __fadd_rn(o, __fmul_rn(__int2float_rn(m), kInvQ));
}

// Eq. 3 / Eq. 4 in two kernels.
// k_moments, one thread per occupied voxel: the voxel's nine halo rows say which
// cells of its 3x3x3 window are occupied and where their integer means lie;
// the means are read straight from the caches (neighbours of a warp's voxels
// share lines) and give the covariance of the window's mean positions (self
// included) as the exact integer matrix N' sum(MM^T) - (sum M)(sum M)^T,
// rounded to FP32.  The matrix does not depend on the origin of the means, so
// they are taken as they are, from the window's anchor: a map is at most 16 m
// wide, 2^24 quanta, so the products' sums stay below 2^53 and N' times them
// below 2^58.  A free cell's load is left out and adds zero.  Wide multiplies
// and the loads' latency bound it: 12.4 us for the walk map's 0.28 M voxels, 66
// for the 8 x 8 x 3 m map's 1.4 M (14 and 71 with offsets from the own mean).
__global__ void __launch_bounds__(kT) k_moments(const SegCounters* __restrict__ ctr, const float* __restrict__ po,
                                                const uint4* __restrict__ rows, const uint32_t* __restrict__ vox,
                                                const int4* __restrict__ M, float4* __restrict__ pos,
                                                float* __restrict__ list_A, uint8_t* __restrict__ nbr,
                                                uint32_t* __restrict__ parent, uint32_t* __restrict__ over,
                                                size_t stride) {
    pdl_gate();
    const uint32_t n = ctr->n_vox;
    const float pox = po[0], poy = po[1], poz = po[2];
    for (uint32_t i = blockIdx.x * kT + threadIdx.x; i < n; i += gridDim.x * kT) {
        const uint32_t v = vox[i];
        const int l = (int)(v % kBrickVox), lx = l & 7, ly = (l >> 3) & 7, lz = l >> 6;
        const uint4* rw = rows + (size_t)(v / kBrickVox) * 100 + lz * 10 + ly;
        const int4 m = M[i];
        int32_t s1x = 0, s1y = 0, s1z = 0;
        long long sxx = 0, syy = 0, szz = 0, sxy = 0, sxz = 0, syz = 0;
        int cnt = 0;
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            uint32_t win, idx[3];
            row_window(rw[(q / 3) * 10 + q % 3], lx, win, idx);
            cnt += __popc(win);
            int4 a[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                a[k] = make_int4(0, 0, 0, 0);
                if ((win >> k) & 1u) a[k] = M[idx[k]];
            }
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const int32_t x = a[k].x, y = a[k].y, z = a[k].z;
                s1x += x; s1y += y; s1z += z;
                sxx += (long long)x * x; syy += (long long)y * y; szz += (long long)z * z;
                sxy += (long long)x * y; sxz += (long long)x * z; syz += (long long)y * z;
            }
        }
        const long long N = cnt;
        list_A[i] = __ll2float_rn(N * sxx - (long long)s1x * s1x);
        list_A[stride + i] = __ll2float_rn(N * syy - (long long)s1y * s1y);
        list_A[2 * stride + i] = __ll2float_rn(N * szz - (long long)s1z * s1z);
        list_A[3 * stride + i] = __ll2float_rn(N * sxy - (long long)s1x * s1y);
        list_A[4 * stride + i] = __ll2float_rn(N * sxz - (long long)s1x * s1z);
        list_A[5 * stride + i] = __ll2float_rn(N * syz - (long long)s1y * s1z);
        nbr[i] = (uint8_t)(cnt - 1);
        pos[i] = make_float4(mean_pos(pox, m.x), mean_pos(poy, m.y), mean_pos(poz, m.z), __int_as_float(1));
        parent[i] = over[i] = i;  // the forests over components (at most one per voxel)
    }
}

// k_eigen, one thread per occupied voxel: normal = eigenvector of the smallest
// eigenvalue by FP32 Jacobi (6 sweeps); steppable iff N >= n_th and
// |n_z| >= cos_step (status 2, else 1).
__global__ void __launch_bounds__(256) k_eigen(const SegCounters* __restrict__ ctr, const float* __restrict__ list_A,
                                               const uint8_t* __restrict__ nbr, float4* __restrict__ nrm,
                                               float4* __restrict__ pos, size_t stride, uint32_t n_th,
                                               float cos_step) {
    pdl_gate();
    const uint32_t n = ctr->n_vox;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        float v[3][3], d[3], nv[3];
        jacobi3(list_A[i], list_A[stride + i], list_A[2 * stride + i], list_A[3 * stride + i],
                list_A[4 * stride + i], list_A[5 * stride + i], 6, v, d);
        pick_normal(v, d, nv);
        nrm[i] = make_float4(nv[0], nv[1], nv[2], 0.0f);
        if (nbr[i] >= n_th && fabsf(nv[2]) >= cos_step) reinterpret_cast<int*>(pos + i)[3] = 2;
    }
}

constexpr int kOneT = 1024;
__device__ __forceinline__ uint32_t warp_incl(uint32_t v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}
// The sum of v over the warps before this one of a 1024-thread CTA (v equal in
// a warp's lanes; ws: 33 words); *total: the sum over all.
__device__ __forceinline__ uint32_t cta_warps_excl(uint32_t v, uint32_t* ws, uint32_t* total) {
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        const uint32_t t = ws[threadIdx.x], ti = warp_incl(t);
        ws[threadIdx.x] = ti - t;
        if (threadIdx.x == 31) ws[32] = ti;
    }
    __syncthreads();
    const uint32_t out = ws[threadIdx.x >> 5];
    *total = ws[32];
    __syncthreads();
    return out;
}
// The same for two values at once (ws: 66 words).
__device__ __forceinline__ uint2 cta_warps_excl2(uint32_t a, uint32_t b, uint32_t* ws, uint32_t* ta, uint32_t* tb) {
    const uint32_t w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane < 2) ws[33 * lane + w] = lane ? b : a;
    __syncthreads();
    if (w < 2) {
        uint32_t* p = ws + 33 * w;
        const uint32_t t = p[lane], ti = warp_incl(t);
        p[lane] = ti - t;
        if (lane == 31) p[32] = ti;
    }
    __syncthreads();
    const uint2 out = make_uint2(ws[w], ws[33 + w]);
    *ta = ws[32];
    *tb = ws[65];
    __syncthreads();
    return out;
}
// Exclusive scan over a 1024-thread CTA (ws: 33 words); *total: the sum.
__device__ __forceinline__ uint32_t cta_excl(uint32_t v, uint32_t* ws, uint32_t* total) {
    const uint32_t inc = warp_incl(v);
    if ((threadIdx.x & 31) == 31) ws[threadIdx.x >> 5] = inc;
    __syncthreads();
    if (threadIdx.x < 32) {
        const uint32_t t = ws[threadIdx.x], ti = warp_incl(t);
        ws[threadIdx.x] = ti - t;
        if (threadIdx.x == 31) ws[32] = ti;
    }
    __syncthreads();
    const uint32_t out = ws[threadIdx.x >> 5] + inc - v;
    *total = ws[32];
    __syncthreads();
    return out;
}

// ---------------------------------------------------------------- clustering
__device__ __forceinline__ bool ccl_edge4(const float4& a, const float4& an, const float4& b, const float4& bn,
                                          float d_th2, float cos_ccl) {
    return ccl_edge(a.x, a.y, a.z, an.x, an.y, an.z, b.x, b.y, b.z, bn.x, bn.y, bn.z, d_th2, cos_ccl);
}

// The entries of a voxel's 13 backward neighbours in its own brick, cell k of
// row q: rows (dy, dz) = (0, 0), (-1, 0), (1, -1), (0, -1), (-1, -1), of the
// first only x - 1.  rowt: row 8 z + y as (entries before it << 8 | its
// occupied cells); win: which of the row's cells x - 1, x, x + 1 are occupied.
__device__ __forceinline__ uint32_t back_row(const uint32_t* rowt, int q, int lx, int ly, int lz, uint32_t& at) {
    const int y = ly + (q == 2 ? 1 : (q == 1 || q == 4 ? -1 : 0)), z = lz - (q > 1);
    if (y < 0 || y > 7 || z < 0) return 0u;
    const uint32_t rt = rowt[z * 8 + y];
    at = (rt >> 8) + __popc(rt & ((1u << lx) - 1u));  // the entry of cell x
    return (((rt & 0xffu) << 1) >> lx) & (q == 0 ? 1u : 7u);
}
__device__ __forceinline__ uint32_t back_cell(uint32_t at, uint32_t win, int k) {
    return k == 0 ? at - 1u : (k == 1 ? at : at + ((win >> 1) & 1u));
}

// The intra-brick half of Algorithm 1, one 128-thread CTA per brick.  Every
// vertex tests its 13 backward neighbours (independent tests, so their loads
// and arithmetic overlap) and hooks under the smallest one it has an edge with,
// without atomics; pointer jumping flattens the trees (a brick is 8 voxels
// wide: a few rounds).  An edge whose ends are in different trees then hooks
// the larger root under the smaller one (an atomic minimum; a hook that another
// one replaces is found again), and the trees are flattened again, until no
// edge lies between two trees: usually there is none from the start.  (Joining
// each edge with a CAS loop contended for the few roots: single bricks took 30
// us.  Testing on demand only the neighbours in other trees made fewer tests
// but one long chain of them.)  A brick whose vertices are one tree after the
// first flattening needs neither edges between trees nor a numbering.  Latency
// bounds it (an instruction in a third of the issue slots), so 128 threads, one a
// voxel in most bricks, take a brick, and the grid is left to the hardware's
// scheduler: 20 us for the walk map's 2,535 bricks, 85 for the 8 x 8 x 3 m map's
// 16 thousand; 64 threads and a grid of about one wave took 26 and 110.  The
// brick's components are numbered in the order of their smallest vertex, and
// each one's size and smallest voxel id are kept at the brick's first entry
// plus its number.
constexpr int kLocalT = 128;
constexpr uint32_t kStage = 256;  // records staged in shared memory; a fuller brick's are read from the caches
__global__ void __launch_bounds__(kLocalT, 11) k_ccl_local(SegCounters* __restrict__ ctr, uint32_t cap_b,
                                                           const BrickRec* __restrict__ brec,
                                                           const uint32_t* __restrict__ vox,
                                                           const float4* __restrict__ pos,
                                                           const float4* __restrict__ nrm, uint16_t* __restrict__ lc,
                                                           uint32_t* __restrict__ ncomp, uint32_t* __restrict__ lsize,
                                                           uint32_t* __restrict__ lroot, int want, float d_th2,
                                                           float cos_ccl) {
    pdl_gate();
    const uint32_t n_sorted = min(ctr->n_sorted, cap_b);
    __shared__ float4 sA[kStage], sB[kStage];
    __shared__ uint32_t rowt[64];            // row 8 z + y: entries before it << 8 | its occupied cells
    __shared__ uint32_t lpar[kBrickVox];
    __shared__ uint16_t sedge[kBrickVox];    // backward edges (bit 3 q + k: cell k of row q), then numbers of roots
    __shared__ uint16_t sl[kBrickVox];       // voxel index inside the brick
    __shared__ uint32_t csz[kBrickVox];      // component sizes
    __shared__ uint32_t wcnt[kLocalT / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t nvert = 0;
    for (uint32_t r = blockIdx.x; r < n_sorted; r += gridDim.x) {
        const BrickRec* br = brec + r;
        const uint4 hd = *reinterpret_cast<const uint4*>(&br->base);  // base, n, key, slot
        const uint32_t base = hd.x, n = hd.y;
        __syncthreads();
        if (threadIdx.x < 64) {
            const uint32_t m = br->mask[threadIdx.x >> 2], sh = (threadIdx.x & 3) * 8;
            rowt[threadIdx.x] = ((br->pre[threadIdx.x >> 2] + __popc(m & ((1u << sh) - 1u))) << 8) | ((m >> sh) & 0xffu);
        }
        const bool staged = n <= kStage;
#pragma unroll 2
        for (uint32_t p = threadIdx.x; p < n; p += kLocalT) {
            sl[p] = (uint16_t)(vox[base + p] % kBrickVox);
            csz[p] = 0;
            if (staged) {
                sA[p] = pos[base + p];
                sB[p] = nrm[base + p];
            }
        }
        __syncthreads();
        uint32_t nroot = 0, nhere = 0;
        const auto tests = [&](const float4* A, const float4* B) {  // apart for the two memories: plain shared loads
            for (uint32_t p = threadIdx.x; p < n; p += kLocalT) {
                const float4 a = A[p], an = B[p];
                const int l = sl[p], lx = l & 7, ly = (l >> 3) & 7, lz = l >> 6;
                const bool vert = __float_as_int(a.w) >= want;
                uint32_t par = p, edges = 0;
    #pragma unroll
                for (int q = 0; q < 5; ++q) {
                    uint32_t at = 0;
                    const uint32_t win = back_row(rowt, q, lx, ly, lz, at);
    #pragma unroll
                    for (int k = 0; k < (q == 0 ? 1 : 3); ++k) {
                        const bool on = (win >> k) & 1u;
                        const uint32_t j = on ? back_cell(at, win, k) : p;
                        const float4 c = A[j];
                        if (on && __float_as_int(c.w) >= want && ccl_edge4(a, an, c, B[j], d_th2, cos_ccl)) {
                            edges |= 1u << (3 * q + k);
                            par = min(par, j);
                        }
                    }
                }
                nroot += vert && par == p;
                nhere += vert;
                lpar[p] = vert ? par : kNone;
                sedge[p] = vert ? (uint16_t)edges : 0;
            }
        };
        if (staged) tests(sA, sB);
        else tests(pos + base, nrm + base);
        nvert += nhere;
        nroot = __reduce_add_sync(0xffffffffu, nroot);
        nhere = __reduce_add_sync(0xffffffffu, nhere);
        if (lane == 0) wcnt[wid] = nroot << 16 | nhere;
        __syncthreads();
        nroot = nhere = 0;
#pragma unroll
        for (int q = 0; q < kLocalT / 32; ++q) {
            nroot += wcnt[q] >> 16;
            nhere += wcnt[q] & 0xffffu;
        }
        if (nroot <= 1) {  // one tree (three bricks of four on the walk map): no labels to find
            for (uint32_t p = threadIdx.x; p < n; p += kLocalT) {
                lc[base + p] = lpar[p] == kNone ? kNoComp : (uint16_t)0;
                if (lpar[p] == p) {
                    lroot[base] = hd.z * kBrickVox + sl[p];
                    lsize[base] = nhere;
                }
            }
            if (threadIdx.x == 0) ncomp[r] = nroot;
            continue;
        }
        for (int round = 0; round < kBrickVox; ++round) {  // every round with an edge apart joins two trees or more
            for (int jump = 0; jump < 32; ++jump) {        // a tree over 512 voxels is flat after at most 9
                bool more = false;
                for (uint32_t p = threadIdx.x; p < n; p += kLocalT) {
                    const uint32_t q = lpar[p];
                    if (q == kNone) continue;
                    const uint32_t g = lpar[q];
                    if (g != q) {
                        lpar[p] = lpar[g];
                        more = true;
                    }
                }
                if (!__syncthreads_or(more)) break;
            }
            bool apart = false;
            for (uint32_t p = threadIdx.x; p < n; p += kLocalT) {
                const uint32_t edges = sedge[p];
                if (!edges) continue;
                const int l = sl[p], lx = l & 7, ly = (l >> 3) & 7, lz = l >> 6;
                const uint32_t ra = lpar[p];
                uint32_t rb[13];
#pragma unroll
                for (int q = 0; q < 5; ++q) {
                    uint32_t at = 0;
                    const uint32_t win = back_row(rowt, q, lx, ly, lz, at);
#pragma unroll
                    for (int k = 0; k < (q == 0 ? 1 : 3); ++k) {
                        const int e = q == 0 ? 0 : 3 * q + k - 2;
                        rb[e] = lpar[(edges >> (3 * q + k)) & 1u ? back_cell(at, win, k) : p];
                    }
                }
#pragma unroll
                for (int e = 0; e < 13; ++e)
                    if (rb[e] != ra) {
                        apart = true;
                        const uint32_t hi = max(ra, rb[e]), lo = min(ra, rb[e]);
                        if (*(volatile uint32_t*)&lpar[hi] > lo) atomicMin(&lpar[hi], lo);
                    }
            }
            if (!__syncthreads_or(apart)) break;
        }
        uint32_t nc = 0;  // components numbered by their roots, in order (every entry holds its root)
        for (uint32_t p0 = 0; p0 < n; p0 += kLocalT) {
            const uint32_t p = p0 + threadIdx.x;
            const bool root = p < n && lpar[p] == p;
            const uint32_t bal = __ballot_sync(0xffffffffu, root);
            if (lane == 0) wcnt[wid] = __popc(bal);
            __syncthreads();
            uint32_t at = nc + __popc(bal & ((1u << lane) - 1u));
#pragma unroll
            for (int q = 0; q < kLocalT / 32; ++q) {
                at += q < wid ? wcnt[q] : 0u;
                nc += wcnt[q];
            }
            if (root) {
                sedge[p] = (uint16_t)at;
                lroot[base + at] = hd.z * kBrickVox + sl[p];
            }
            __syncthreads();
        }
        for (uint32_t p0 = 0; p0 < n; p0 += kLocalT) {
            const uint32_t p = p0 + threadIdx.x;
            uint32_t j = kNoComp;
            if (p < n && lpar[p] != kNone) j = sedge[lpar[p]];
            if (p < n) lc[base + p] = (uint16_t)j;
            const uint32_t grp = __match_any_sync(0xffffffffu, j);
            if (j != kNoComp && lane == __ffs(grp) - 1) atomicAdd(&csz[j], (uint32_t)__popc(grp));
        }
        __syncthreads();
        for (uint32_t j = threadIdx.x; j < nc; j += kLocalT) lsize[base + j] = csz[j];
        if (threadIdx.x == 0) ncomp[r] = nc;
    }
    nvert = __reduce_add_sync(0xffffffffu, nvert);
    if (lane == 0 && nvert) atomicAdd(&ctr->n_vert, nvert);
}

// Numbers the in-brick components (an exclusive scan of the bricks' counts, in
// rank order), in one CTA: a warp scans 256 counts a round, read 32 at a time.
constexpr int kRun = 8;  // 32-element steps a warp takes in a round of a one-CTA scan
__global__ void __launch_bounds__(kOneT, 1) k_comp_number(SegCounters* __restrict__ ctr, uint32_t cap_b,
                                                       const uint32_t* __restrict__ ncomp,
                                                       uint32_t* __restrict__ cbase) {
    pdl_gate();
    __shared__ uint32_t ws[33];
    const int lane = threadIdx.x & 31;
    const uint32_t n = min(ctr->n_sorted, cap_b);
    uint32_t carry = 0;
    for (uint32_t b0 = 0; b0 < n; b0 += kOneT * kRun) {
        const uint32_t j0 = b0 + (threadIdx.x >> 5) * (32 * kRun) + lane;
        uint32_t v[kRun], inc[kRun], sum = 0;
#pragma unroll
        for (int i = 0; i < kRun; ++i) v[i] = j0 + i * 32 < n ? ncomp[j0 + i * 32] : 0u;
#pragma unroll
        for (int i = 0; i < kRun; ++i) {
            inc[i] = sum + warp_incl(v[i]);
            sum = __shfl_sync(0xffffffffu, inc[i], 31);
        }
        uint32_t tot;
        const uint32_t at = carry + cta_warps_excl(sum, ws, &tot);
#pragma unroll
        for (int i = 0; i < kRun; ++i)
            if (j0 + i * 32 < n) cbase[j0 + i * 32] = at + inc[i] - v[i];
        carry += tot;
    }
    if (threadIdx.x == 0) ctr->n_comp = carry;
}

// The inter-brick half of Algorithm 1, one thread per occupied voxel: a vertex
// on a face that forward edges leave through (dz in {0, 1}, dy in {-1, 0, 1},
// -1 only with dz = 1, dx in {-1, 0, 1}: the +z face, either y face, either x
// face) tests its occupied out-of-brick neighbours.  A vertex's five halo rows
// are read together, then the components of all its candidates.  A pair of
// components that is listed already needs no further edge, and a brick's edges
// lead to few pairs (six on the walk map), so the pair is looked up in the
// CTA's hash set in shared memory before any record is read.  A distinct pair
// hooks its larger component under the smaller one (an atomic minimum whose
// result nobody waits for) and goes to one list; k_comp_join then joins what
// the hooks left apart.  A pair that finds the list full joins a forest of its
// own (over).  The threads of a brick's first voxels also copy its components
// to their numbers.
constexpr int kPairSlots = 512;
constexpr unsigned long long kNoPair = ~0ull;
__device__ __forceinline__ void add_pair(unsigned long long* __restrict__ pairs, uint32_t pair_cap, uint32_t at,
                                         unsigned long long key, uint32_t* parent, uint32_t* over, uint32_t* err) {
    const uint32_t lo = (uint32_t)(key >> 32), hi = (uint32_t)key;
    if (at < pair_cap) {
        pairs[at] = key;
        atomicMin(parent + hi, lo);
    } else {
        uf_union(over, lo, hi, err);
    }
}
__global__ void __launch_bounds__(kT, 4)
    k_ccl_cross(SegCounters* __restrict__ ctr, const BrickRec* __restrict__ brec, const int32_t* __restrict__ near,
                const uint4* __restrict__ rows, const uint32_t* __restrict__ vox, const float4* __restrict__ pos,
                const float4* __restrict__ nrm, const uint16_t* __restrict__ lc, const uint32_t* __restrict__ ncomp,
                const uint32_t* __restrict__ cbase, const uint32_t* __restrict__ lsize,
                const uint32_t* __restrict__ lroot, uint32_t* __restrict__ csize, uint32_t* __restrict__ croot,
                uint32_t* __restrict__ total, uint32_t* parent, uint32_t* over,
                unsigned long long* __restrict__ pairs, uint32_t pair_cap, float d_th2, float cos_ccl,
                uint32_t* err) {
    pdl_gate();
    const uint32_t n = ctr->n_vox;
    __shared__ unsigned long long set[kPairSlots];
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int q = threadIdx.x; q < kPairSlots; q += kT) set[q] = kNoPair;
    for (uint32_t i0 = blockIdx.x * kT; i0 < n; i0 += gridDim.x * kT) {
        __syncthreads();
        const uint32_t i = i0 + threadIdx.x;
        if (i < n) {
            const uint32_t v = vox[i], r = v / kBrickVox;
            const int l = (int)(v % kBrickVox), lx = l & 7, ly = (l >> 3) & 7, lz = l >> 6;
            const uint16_t ca = lc[i];
            const uint32_t c0 = cbase[r], j = i - brec[r].base;
            if (j < ncomp[r]) {
                csize[c0 + j] = lsize[i];
                croot[c0 + j] = lroot[i];
                total[c0 + j] = 0;
            }
            uint32_t wins = 0, idx[5][3];
            if (ca != kNoComp && ((lx == 0) | (lx == 7) | (ly == 0) | (ly == 7) | (lz == 7))) {
                const uint4* rw = rows + (size_t)r * 100;
#pragma unroll
                for (int q = 0; q < 5; ++q) {  // rows (dy, dz) = (0, 0), (1, 0), (-1, 1), (0, 1), (1, 1)
                    const int y = ly + (q == 0 || q == 3 ? 0 : (q == 2 ? -1 : 1)), z = lz + (q > 1);
                    const bool own = y >= 0 && y <= 7 && z <= 7;  // a row of this brick: its own cells are done
                    uint32_t ask = own ? (lx == 0 ? 1u : 0u) | (lx == 7 ? 4u : 0u) : 7u, win;
                    if (q == 0) ask &= 4u;  // only +x lies forward
                    row_window(rw[(z + 1) * 10 + y + 1], lx, win, idx[q]);
                    wins |= (win & ask) << (3 * q);
                }
            }
            if (wins) {
                const uint32_t pa = c0 + ca;
                const float4 a = pos[i], an = nrm[i];
                uint16_t lcb[5][3];
#pragma unroll
                for (int q = 0; q < 5; ++q)
#pragma unroll
                    for (int k = 0; k < 3; ++k) lcb[q][k] = (wins >> (3 * q + k)) & 1u ? lc[idx[q][k]] : kNoComp;
                unsigned long long last = kNoPair;
#pragma unroll
                for (int q = 0; q < 5; ++q) {
                    const int y = ly + (q == 0 || q == 3 ? 0 : (q == 2 ? -1 : 1)), z = lz + (q > 1);
                    const int32_t* nb = near + (size_t)r * 27 + (z > 7 ? 18 : 9) + (y < 0 ? 0 : (y > 7 ? 6 : 3));
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        if (lcb[q][k] == kNoComp) continue;
                        const int x = lx + k - 1;
                        const uint32_t pb = cbase[nb[x < 0 ? 0 : (x > 7 ? 2 : 1)]] + lcb[q][k];
                        const uint32_t lo = pa < pb ? pa : pb, hi = pa < pb ? pb : pa;
                        const unsigned long long key = ((unsigned long long)lo << 32) | hi;
                        if (key == last) continue;
                        uint32_t h = (lo * 2654435761u ^ hi * 40503u) & (kPairSlots - 1);
                        if (*(volatile unsigned long long*)&set[h] == key) continue;
                        if (!ccl_edge4(a, an, pos[idx[q][k]], nrm[idx[q][k]], d_th2, cos_ccl)) continue;
                        last = key;
                        bool placed = false;
                        for (int probe = 0; probe < kPairSlots; ++probe) {
                            const unsigned long long prev = atomicCAS(&set[h], kNoPair, key);
                            if (prev == kNoPair || prev == key) { placed = true; break; }
                            h = (h + 1) & (kPairSlots - 1);
                        }
                        if (!placed) add_pair(pairs, pair_cap, atomicAdd(&ctr->n_pairs, 1u), key, parent, over, err);
                    }
                }
            }
        }
        __syncthreads();
#pragma unroll
        for (int q = threadIdx.x; q < kPairSlots; q += kT) {
            const unsigned long long key = set[q];
            const uint32_t b = __ballot_sync(0xffffffffu, key != kNoPair);
            uint32_t at = 0;
            if (lane == 0 && b) at = atomicAdd(&ctr->n_pairs, (uint32_t)__popc(b));
            at = __shfl_sync(0xffffffffu, at, 0) + __popc(b & ((1u << lane) - 1u));
            if (key != kNoPair) {
                add_pair(pairs, pair_cap, at, key, parent, over, err);
                set[q] = kNoPair;
            }
        }
    }
}

// Joins the listed pairs.  While the components fit one SM's shared memory
// (kSmemComps) the forest that the hooks of k_ccl_cross left is copied there and
// joined in rounds: pointer jumping flattens the trees; each pair then reads its
// two roots, and a pair that is apart hooks the larger under the smaller one (an
// atomic minimum; a hook that another one replaces is found again), until no
// pair is apart.  Only the roots that the first flattening leaves take part in
// the later ones.  Few pairs are joined by one CTA.  With more, every CTA first
// walks its share of the pairs in a copy of its own, lists those that are apart
// (a third of the LiDAR map's 95 thousand) and stores the roots of its share of
// the components; the last CTA to finish numbers the roots (9 of 29 thousand) and
// joins the list over these numbers, so that forest and list fit beside each
// other.
// With more components, or pairs the list had no room for, the grid joins pair
// by pair in global memory (51 us for the walk map's 17 thousand pairs: the
// threads meet on the few large roots).  One SM's instruction rate bounds the
// rounds: what is touched in a round, not the steps of a chain, counts.  So a few
// thousand pairs are joined by one CTA, and more are thinned first: the walk
// map's 17 thousand take 14.1 us alone and 12.7 thinned, the 5 x 5 x 5 m window's
// 23 thousand 24.8 and 16.3.  The 8 x 8 x 3 m map's 95 thousand: 54 us (85 with
// its list in global memory, 93 with each pair's chains read in every round).
constexpr uint32_t kJoinWords = 57344;  // 224 KB: the forest, the roots, the pairs
constexpr uint32_t kSmemComps = 36864;  // below 2^16: a pair packs into a word
constexpr uint32_t kJoinAlone = 8192;   // pairs that one CTA joins by itself
// Flattens the trees over the elements list[0 .. n) (null: 0 .. n).
__device__ __forceinline__ void join_flatten(uint32_t* P, const uint16_t* list, uint32_t n) {
    for (int round = 0; round < 64; ++round) {  // every round at least doubles the reach
        bool more = false;
        for (uint32_t i = threadIdx.x; i < n; i += kOneT) {
            const uint32_t c = list ? list[i] : i, p = P[c], a = P[p];
            if (a != p) {
                P[c] = P[a];
                more = true;
            }
        }
        if (!__syncthreads_or(more)) break;
    }
}
// The root of x in P, halving the path: a parent only moves to a smaller ancestor.
__device__ __forceinline__ uint32_t join_root(uint32_t* P, uint32_t x, uint32_t K, uint32_t* err) {
    volatile uint32_t* V = P;
    for (uint32_t it = 0; it <= K; ++it) {
        const uint32_t p = V[x];
        if (p == x) return x;
        const uint32_t a = V[p];
        if (a != p) atomicMin(&P[x], a);
        x = a;
    }
    atomicOr(err, kErrTimeout);
    return x;
}
__global__ void __launch_bounds__(kOneT, 1) k_comp_join(SegCounters* __restrict__ ctr, uint32_t pair_cap,
                                                        unsigned long long* pairs, uint32_t* list, uint32_t* parent,
                                                        const uint32_t* __restrict__ over, uint32_t* err) {
    pdl_gate();
    extern __shared__ uint32_t P[];
    __shared__ uint32_t ws[33];
    __shared__ uint32_t s_last;
    const uint32_t K = ctr->n_comp, all = ctr->n_pairs, np = min(all, pair_cap);
    if (K > kSmemComps || all > pair_cap) {
        for (uint32_t q = blockIdx.x * kOneT + threadIdx.x; q < np; q += gridDim.x * kOneT) {
            const unsigned long long key = pairs[q];
            uf_union(parent, (uint32_t)(key >> 32), (uint32_t)key, err);
        }
        if (all > pair_cap)
            for (uint32_t c = blockIdx.x * kOneT + threadIdx.x; c < K; c += gridDim.x * kOneT)
                if (over[c] != c) uf_union(parent, over[c], c, err);
        return;
    }
    uint16_t* roots = reinterpret_cast<uint16_t*>(P + K);  // the roots left by the first flattening
    uint32_t* L = P + K + (K + 1) / 2;                     // pairs in shared memory (0: none, or together)
    const uint32_t room = kJoinWords - K - (K + 1) / 2;
    const bool one = np <= min(room, kJoinAlone);
    const uint32_t G = one ? 1u : min(gridDim.x, (np + kOneT - 1) / kOneT), g = blockIdx.x;
    if (g >= G) return;
    const int lane = threadIdx.x & 31;
    const auto pack = [](unsigned long long key) { return (uint32_t)(key >> 32) << 16 | (uint32_t)key; };
#pragma unroll 8
    for (uint32_t c = threadIdx.x; c < K; c += kOneT) P[c] = __ldcg(parent + c);
    if (one)
#pragma unroll 8
        for (uint32_t q = threadIdx.x; q < np; q += kOneT) L[q] = pack(__ldcg(pairs + q));
    __syncthreads();
    uint32_t n = np;
    if (one) {
        join_flatten(P, nullptr, K);
    } else {
        for (uint32_t q0 = g * kOneT; q0 < np; q0 += G * kOneT) {
            const uint32_t q = q0 + threadIdx.x;
            uint32_t a = 0, b = 0;
            if (q < np) {
                const uint32_t pr = pack(pairs[q]);
                a = join_root(P, pr >> 16, K, err);
                b = join_root(P, pr & 0xffffu, K, err);
            }
            const uint32_t m = __ballot_sync(0xffffffffu, a != b);
            uint32_t at = 0;
            if (lane == 0 && m) at = atomicAdd(&ctr->n_apart, (uint32_t)__popc(m));
            at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & ((1u << lane) - 1u));
            if (a != b) list[at] = min(a, b) << 16 | max(a, b);
        }
        // another CTA still copying the forest reads a parent or its root: either is an ancestor
        for (uint32_t c = g * kOneT + threadIdx.x; c < K; c += G * kOneT) parent[c] = join_root(P, c, K, err);
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) s_last = atomicAdd(&ctr->join_done, 1u) + 1u == G;
        __syncthreads();
        if (!s_last) return;
        __threadfence();
        n = *(volatile uint32_t*)&ctr->n_apart;
    }
    // The roots, in order: a warp takes a run of components, counts its roots and lists them from there.
    const uint32_t half = (K + 1) / 2;
    uint16_t* rank = reinterpret_cast<uint16_t*>(P + kJoinWords - half);  // a root's number among the roots
    uint32_t* comp = reinterpret_cast<uint32_t*>(pairs);                  // and back (the pairs are read)
    const uint32_t run = (K + kOneT - 1) / kOneT * 32, c0 = (threadIdx.x >> 5) * run, c1 = min(K, c0 + run);
    uint32_t nr, at = 0;
    for (uint32_t c = c0 + lane; c - lane < c1; c += 32) at += __popc(__ballot_sync(0xffffffffu, c < c1 && P[c] == c));
    at = cta_warps_excl(at, ws, &nr);
    const bool rerank = !one && n + max(half, nr) <= kJoinWords;
    for (uint32_t c = c0 + lane; c - lane < c1; c += 32) {
        const bool root = c < c1 && P[c] == c;
        const uint32_t m = __ballot_sync(0xffffffffu, root), i = at + __popc(m & ((1u << lane) - 1u));
        if (root && rerank) {
            rank[c] = (uint16_t)i;
            comp[i] = c;
        } else if (root) {
            roots[i] = (uint16_t)c;
        }
        at += __popc(m);
    }
    __syncthreads();
    uint32_t* F = P;              // the forest of the rounds
    const uint16_t* flat = roots; // its members
    bool here = n <= room;        // its pairs lie in L
    if (rerank) {
        // over the roots' numbers, which keep their order, the pairs fit beside the forest
        L = P;
#pragma unroll 8
        for (uint32_t q = threadIdx.x; q < n; q += kOneT) {
            const uint32_t pr = __ldcg(list + q);
            L[q] = (uint32_t)rank[pr >> 16] << 16 | rank[pr & 0xffffu];
        }
        __syncthreads();
        F = P + kJoinWords - nr;
        flat = nullptr;
        here = true;
        for (uint32_t i = threadIdx.x; i < nr; i += kOneT) F[i] = i;
        __syncthreads();
    } else if (!one && here) {
#pragma unroll 8
        for (uint32_t q = threadIdx.x; q < n; q += kOneT) L[q] = __ldcg(list + q);
        __syncthreads();
    }
    for (uint32_t round = 0;; ++round) {
        // the roots of every pair, then the hooks: apart, because a pair must not be taken for joined by a hook
        // that another one then replaces.  The pairs of a list name roots that are apart.
        bool apart = false;
        if (!one && round == 0) {
            apart = threadIdx.x < n;
        } else {
#pragma unroll 4
            for (uint32_t q = threadIdx.x; q < n; q += kOneT) {
                const uint32_t pr = here ? L[q] : __ldcg(list + q);
                if (!pr) continue;
                const uint32_t a = F[pr >> 16], b = F[pr & 0xffffu], now = a == b ? 0u : min(a, b) << 16 | max(a, b);
                if (here) L[q] = now;
                else list[q] = now;
                apart |= now != 0u;
            }
        }
        if (!__syncthreads_or(apart)) break;
        if (round > K) {  // every round with a pair apart joins two trees or more
            if (threadIdx.x == 0) atomicOr(err, kErrTimeout);
            break;
        }
#pragma unroll 4
        for (uint32_t q = threadIdx.x; q < n; q += kOneT) {
            const uint32_t pr = here ? L[q] : __ldcg(list + q);
            // most pairs of a large tree name its root: a look first spares the meeting atomics
            if (pr && *(volatile uint32_t*)&F[pr & 0xffffu] > pr >> 16) atomicMin(&F[pr & 0xffffu], pr >> 16);
        }
        __syncthreads();
        join_flatten(F, flat, nr);
    }
    // a component's root of the first flattening, then that one's
    if (one)
        for (uint32_t c = threadIdx.x; c < K; c += kOneT) parent[c] = P[P[c]];
    else if (rerank)
        for (uint32_t i = threadIdx.x; i < nr; i += kOneT) parent[comp[i]] = comp[F[i]];
    else
        for (uint32_t i = threadIdx.x; i < nr; i += kOneT) parent[roots[i]] = P[roots[i]];
}

// Read-only walk to the root.  Used once linking is over: every thread writes
// only its own entry, so a finished entry is never overwritten by another
// thread's path shortcut (which could leave it on an intermediate node).
__device__ __forceinline__ uint32_t uf_root(const uint32_t* P, uint32_t x, uint32_t* err) {
    for (int it = 0; it < kLoopCap; ++it) {
        const uint32_t p = __ldcg(P + x);
        if (p == x) return x;
        x = p;
    }
    atomicOr(err, kErrTimeout);
    return x;
}

// A map with many components numbers and places its clusters with kernels of their
// own (k_cluster_number_many, k_cluster_place<true>): what they need made those for
// surfaces, which run on every frame, a little longer.  Words of the scratch that
// they share, zero when they start (k_comp_size, clear): a flag a CTA of the
// placement, the tickets, and whose turn a tile of the placement is; then a 64-bit
// word a CTA of the numbering.
constexpr uint32_t kPlaceCtas = 128;  // CTAs of either at most
constexpr uint32_t kPlaceTicket = kPlaceCtas, kPlaceTurn = kPlaceCtas + 1, kNumberTicket = kPlaceCtas + 2;
constexpr uint32_t kNumberWords = kPlaceCtas + 4, kPlaceHead = kNumberWords + 2 * kPlaceCtas;

// Every component's root, and the vertices of each whole component at its
// root (lanes with equal roots add up first).
__global__ void __launch_bounds__(kT) k_comp_size(const SegCounters* __restrict__ ctr, uint32_t* parent,
                                                  const uint32_t* __restrict__ csize, uint32_t* __restrict__ total,
                                                  uint32_t* __restrict__ clear, uint32_t* err) {
    pdl_gate();
    const uint32_t K = ctr->n_comp;
    if (clear && blockIdx.x == 0)
        for (uint32_t q = threadIdx.x; q < kPlaceHead; q += kT) clear[q] = 0;
    for (uint32_t base = (blockIdx.x * kT + threadIdx.x) & ~31u; base < K; base += gridDim.x * kT) {
        const uint32_t c = base + (threadIdx.x & 31);
        uint32_t root = kNone, n = 0;
        if (c < K) {
            root = uf_root(parent, c, err);
            parent[c] = root;
            n = csize[c];
        }
        const uint32_t grp = __match_any_sync(0xffffffffu, root);
        n = __reduce_add_sync(grp, n);
        if (root != kNone && (threadIdx.x & 31) == (uint32_t)(__ffs(grp) - 1)) atomicAdd(&total[root], n);
    }
}

// Kept components (at least min_cluster vertices) numbered in the order of
// their roots (= label order) with their sizes and labels, and the cluster
// offsets, in one CTA.  Clusters beyond the scratch flag a re-run, and the
// count is clamped for the kernels after this one.
__global__ void __launch_bounds__(kOneT, 1) k_cluster_number(SegCounters* __restrict__ ctr, uint32_t min_cluster,
                                                          uint32_t kcap, const uint32_t* __restrict__ total,
                                                          const uint32_t* __restrict__ croot,
                                                          uint32_t* __restrict__ ccl, uint32_t* __restrict__ cl_size,
                                                          uint32_t* __restrict__ cl_label,
                                                          uint32_t* __restrict__ cl_off,
                                                          uint32_t* __restrict__ flags) {
    pdl_gate();
    __shared__ uint32_t ws[33];
    const int lane = threadIdx.x & 31;
    const uint32_t K = ctr->n_comp;
    if (threadIdx.x <= kPlaceCtas) flags[threadIdx.x] = 0;  // k_cluster_place's, and its ticket
    uint32_t k = 0;
    for (uint32_t b0 = 0; b0 < K; b0 += kOneT * kRun) {
        const uint32_t c0 = b0 + (threadIdx.x >> 5) * (32 * kRun) + lane;
        uint32_t sz[kRun], kept[kRun], sum = 0;
#pragma unroll
        for (int i = 0; i < kRun; ++i) sz[i] = c0 + i * 32 < K ? total[c0 + i * 32] : 0u;  // 0 but at roots
#pragma unroll
        for (int i = 0; i < kRun; ++i) {
            if (sz[i] < min_cluster) sz[i] = 0;
            kept[i] = __ballot_sync(0xffffffffu, sz[i] != 0);
            sum += __popc(kept[i]);
        }
        uint32_t tot;
        uint32_t at = k + cta_warps_excl(sum, ws, &tot);
#pragma unroll
        for (int i = 0; i < kRun; ++i) {
            const uint32_t c = c0 + i * 32, me = at + __popc(kept[i] & ((1u << lane) - 1u));
            if (c < K) ccl[c] = sz[i] ? me : kNone;  // of roots; the others follow in k_cluster_place
            if (sz[i]) {
                cl_size[me] = sz[i];
                cl_label[me] = croot[c];
            }
            at += __popc(kept[i]);
        }
        k += tot;
    }
    __syncthreads();  // cl_size, by this CTA
    uint32_t off = 0;
    for (uint32_t b0 = 0; b0 < k; b0 += kOneT) {
        const uint32_t c = b0 + threadIdx.x;
        uint32_t tot;
        const uint32_t at = off + cta_excl(c < k ? cl_size[c] : 0u, ws, &tot);
        if (c < k) cl_off[c] = at;
        off += tot;
    }
    if (threadIdx.x == 0) {
        cl_off[k] = off;
        ctr->n_kept = off;
        ctr->tot = off;
        ctr->k_need = k;
        ctr->k = k < kcap ? k : kcap;
        if (k > kcap) atomicOr(&ctr->err, kErrScratch);
    }
}

// The same for a map with many components: they are cut into stretches, a CTA each,
// which adds up its own, publishes the two sums and waits for the CTAs before it (a
// ticket numbers them as they start, so each of those is running; the wait is
// bounded); then it goes over the stretch again.  next: the offsets again, which the
// placement moves on where it goes tile by tile.  (1 x 1 x 1 m with every second cell
// at 0.01 m occupied, hundreds of components a brick: 191 us in one CTA, 12 so.)
constexpr uint32_t kNumberRun = kOneT * kRun;
__global__ void __launch_bounds__(kOneT, 1) k_cluster_number_many(SegCounters* __restrict__ ctr, uint32_t min_cluster,
                                                               uint32_t kcap, const uint32_t* __restrict__ total,
                                                               const uint32_t* __restrict__ croot,
                                                               uint32_t* __restrict__ ccl,
                                                               uint32_t* __restrict__ cl_size,
                                                               uint32_t* __restrict__ cl_label,
                                                               uint32_t* __restrict__ cl_off, uint32_t* scratch,
                                                               uint32_t* err) {
    pdl_gate();
    __shared__ uint32_t ws[66];
    __shared__ uint32_t s_ticket;
    const int lane = threadIdx.x & 31;
    const uint32_t w = threadIdx.x >> 5, K = ctr->n_comp;
    const uint32_t stretch = max(kNumberRun, ((K + gridDim.x - 1) / gridDim.x + 1023u) & ~1023u);
    const uint32_t G = max(1u, (K + stretch - 1) / stretch);
    if (blockIdx.x >= G) return;
    volatile unsigned long long* words = reinterpret_cast<volatile unsigned long long*>(scratch + kNumberWords);
    if (threadIdx.x == 0) s_ticket = atomicAdd(scratch + kNumberTicket, 1u);
    __syncthreads();
    const uint32_t g = s_ticket, first = g * stretch, end = min(K, first + stretch);
    uint32_t k, off, tot, tot2, mk = 0, mv = 0;
#pragma unroll 8
    for (uint32_t c = first + threadIdx.x; c < end; c += kOneT) {
        const uint32_t n = total[c];  // 0 but at roots
        mk += n >= min_cluster;
        mv += n >= min_cluster ? n : 0u;
    }
    cta_warps_excl2(__reduce_add_sync(0xffffffffu, mk), __reduce_add_sync(0xffffffffu, mv), ws, &tot, &tot2);
    // one word: the sums and that they are there
    if (threadIdx.x == 0) words[g] = 1ull << 63 | (unsigned long long)tot << 32 | tot2;
    unsigned long long before = 0;
    if (threadIdx.x < g) {
        int it = 0;
        while (!((before = words[threadIdx.x]) >> 63) && it < kLoopCap) ++it;
        if (it == kLoopCap) atomicOr(err, kErrTimeout);
    }
    cta_warps_excl2(__reduce_add_sync(0xffffffffu, (uint32_t)(before >> 32) & 0x7fffffffu),
                    __reduce_add_sync(0xffffffffu, (uint32_t)before), ws, &k, &off);  // before this CTA
    uint32_t* next = scratch + kPlaceHead;
    for (uint32_t b0 = first; b0 < end; b0 += kNumberRun) {
        const uint32_t c0 = b0 + w * (32 * kRun) + lane;
        uint32_t sz[kRun], kept[kRun], inc[kRun], nk = 0, nv = 0;
#pragma unroll
        for (int i = 0; i < kRun; ++i) sz[i] = c0 + i * 32 < end ? total[c0 + i * 32] : 0u;
#pragma unroll
        for (int i = 0; i < kRun; ++i) {
            if (sz[i] < min_cluster) sz[i] = 0;
            kept[i] = __ballot_sync(0xffffffffu, sz[i] != 0);
            nk += __popc(kept[i]);
            inc[i] = 0;
            if (kept[i]) {  // most steps of a map of surfaces keep none
                inc[i] = nv + warp_incl(sz[i]);
                nv = __shfl_sync(0xffffffffu, inc[i], 31);
            }
        }
        const uint2 ex = cta_warps_excl2(nk, nv, ws, &tot, &tot2);
        uint32_t at = k + ex.x;
        const uint32_t av = off + ex.y;
#pragma unroll
        for (int i = 0; i < kRun; ++i) {
            const uint32_t c = c0 + i * 32, me = at + __popc(kept[i] & ((1u << lane) - 1u));
            if (c < end) ccl[c] = sz[i] ? me : kNone;  // of roots; the others follow in k_cluster_place
            if (sz[i]) {
                cl_size[me] = sz[i];
                cl_label[me] = croot[c];
                cl_off[me] = next[me] = av + inc[i] - sz[i];
            }
            at += __popc(kept[i]);
        }
        k += tot;
        off += tot2;
    }
    if (threadIdx.x == 0 && g == G - 1) {
        cl_off[k] = off;
        ctr->n_kept = off;
        ctr->tot = off;
        ctr->k_need = k;
        ctr->k = k < kcap ? k : kcap;
        if (k > kcap) atomicOr(&ctr->err, kErrScratch);
    }
}

// Where each in-brick component's points start in the cluster lists: its
// cluster's offset plus the vertices of the cluster's components before it.
// The components are cut into stretches, a CTA each, and a CTA's into 32, a
// warp each: a warp adds up its components' vertices per cluster, the sums are
// scanned over the CTA's warps, each CTA publishes its sums per cluster and
// waits for the CTAs before it (a ticket numbers them as they start, so each
// of those is running; the wait is bounded), and each warp walks its components
// again, 32 at a time, one scan per cluster among them.  scratch: a flag per CTA and
// the ticket (zero at launch), then the CTAs' sums.  Where the warps' counts do not
// fit shared memory or the sums the scratch, one CTA takes everything, its counts in
// scratch (and where the run is one to be repeated, the places are left at zero, from
// where the lists stay inside their arrays).
// kMany, for maps with many components or clusters: fewer warps count where the
// counts of 32 do not fit, and where one warp's do not, or the sums the scratch, the
// CTAs take tiles of kPlaceTile components (place_tiles).  4 x 4 x 1 m of noise at 0.01
// m with 12 thousand clusters: 1.75 ms in one CTA, 0.28 with a warp a CTA counting, and
// with 616 thousand 36.7 ms and 0.27 tile by tile, numbering and lists included.
template <bool kMany>
constexpr uint32_t kPlaceWords = kMany ? 24576 : 49152;  // 96 KB (other kernels fit the SM beside it), 192 KB
constexpr uint32_t kPlaceTile = 8192;                     // its keys and counts take the 96 KB
constexpr uint32_t kTileBits = 13;
static_assert(kPlaceTile == 1u << kTileBits && kPlaceTile * 3 <= kPlaceWords<true>, "a tile's keys and counts fit");
static_assert(kSurfaceClusters * 32 == kPlaceWords<false>, "with more, one CTA places them all");

// The placement tile by tile, however many clusters there are.  A component that is
// its whole cluster starts at the cluster's offset.  A tile's others are sorted by
// (cluster, component) and a scan gives each one the vertices before it in its
// cluster and tile.  A cluster that lies in one tile starts at its offset; of the
// others the tiles, in turn, take the place so far (next) and move it on by their
// own vertices.  A tile's turn comes when the one before it, which another CTA has
// taken already, has had its own (the wait is bounded); only that step is serial.
__device__ __noinline__ void place_tiles(uint32_t K, const uint32_t* __restrict__ parent,
                                         const uint32_t* __restrict__ csize, uint32_t* ccl,
                                         const uint32_t* __restrict__ cl_size, const uint32_t* __restrict__ cl_off,
                                         uint32_t* __restrict__ place, uint32_t* scratch, uint32_t* sm, uint32_t* err) {
    constexpr int kEach = kPlaceTile / kOneT;
    __shared__ uint32_t ws[33];
    __shared__ uint32_t s_tile, s_m;
    unsigned long long* key = reinterpret_cast<unsigned long long*>(sm);  // cluster << kTileBits | component of the tile
    uint32_t* cnt = sm + 2 * kPlaceTile;                                  // vertices, then places
    uint32_t* next = scratch + kPlaceHead;
    const uint32_t tid = threadIdx.x, tiles = (K + kPlaceTile - 1) / kPlaceTile;
    const uint32_t lt = (1u << (tid & 31)) - 1u;
    for (;;) {
        __syncthreads();
        if (tid == 0) {
            s_tile = atomicAdd(scratch + kPlaceTicket, 1u);
            s_m = 0;
        }
        __syncthreads();
        const uint32_t tile = s_tile, base = tile * kPlaceTile;
        if (tile >= tiles) break;
        uint32_t cl[kEach], n[kEach], all[kEach];
#pragma unroll
        for (int i = 0; i < kEach; ++i) {
            const uint32_t c = base + i * kOneT + tid;
            cl[i] = c < K ? parent[c] : kNone;
            n[i] = c < K ? csize[c] : 0u;
        }
#pragma unroll
        for (int i = 0; i < kEach; ++i)  // a root's entry is read and rewritten with the same value
            if (cl[i] != kNone) ccl[base + i * kOneT + tid] = cl[i] = __ldcg(ccl + cl[i]);
#pragma unroll
        for (int i = 0; i < kEach; ++i) all[i] = cl[i] != kNone ? cl_size[cl[i]] : 0u;
#pragma unroll
        for (int i = 0; i < kEach; ++i) {
            const uint32_t q = i * kOneT + tid;
            const bool part = n[i] < all[i];
            if (cl[i] != kNone && !part) place[base + q] = cl_off[cl[i]];
            const uint32_t b = __ballot_sync(0xffffffffu, part);
            uint32_t at = 0;
            if (!(tid & 31) && b) at = atomicAdd(&s_m, (uint32_t)__popc(b));
            at = __shfl_sync(0xffffffffu, at, 0) + __popc(b & lt);
            if (part) {
                key[at] = (unsigned long long)cl[i] << kTileBits | q;
                cnt[q] = n[i];
            }
        }
        __syncthreads();
        const uint32_t m = s_m;
        uint32_t m2 = 1;
        while (m2 < m) m2 <<= 1;
        for (uint32_t q = m + tid; q < m2; q += kOneT) key[q] = ~0ull;
        __syncthreads();
        for (uint32_t size = 2; size <= m2; size <<= 1)
            for (uint32_t stride = size >> 1; stride > 0; stride >>= 1) {
                for (uint32_t p = tid; p < m2 / 2; p += kOneT) {
                    const uint32_t i = 2 * p - (p & (stride - 1)), j = i + stride;
                    const unsigned long long a = key[i], b = key[j];
                    if ((a > b) == !(i & size)) {
                        key[i] = b;
                        key[j] = a;
                    }
                }
                __syncthreads();
            }
        // a thread takes kEach places of the sorted order: the vertices before each in its cluster and tile
        uint32_t rel[kEach], head[kEach], sum = 0, tot, lasts = 0;  // lasts: those that a later tile's follow
#pragma unroll
        for (int i = 0; i < kEach; ++i) {
            const uint32_t q = tid * kEach + i;
            n[i] = q < m ? cnt[key[q] & (kPlaceTile - 1)] : 0u;
            sum += n[i];
        }
        uint32_t at = cta_excl(sum, ws, &tot);  // its barriers come after every read of the counts
#pragma unroll
        for (int i = 0; i < kEach; ++i) {
            cnt[tid * kEach + i] = rel[i] = at;
            at += n[i];
        }
        __syncthreads();
        uint32_t whole = 0;  // the last ones of clusters that lie in this tile
#pragma unroll
        for (int i = 0; i < kEach; ++i) {
            const uint32_t q = tid * kEach + i;
            head[i] = 0;
            if (q >= m) continue;
            const unsigned long long c = key[q] >> kTileBits;
            if (i && c == key[q - 1] >> kTileBits) {
                head[i] = head[i - 1];
            } else {  // the first place of the cluster
                uint32_t lo = 0, hi = q;
                while (lo < hi) {
                    const uint32_t mid = (lo + hi) >> 1;
                    if (key[mid] >> kTileBits < c) lo = mid + 1;
                    else hi = mid;
                }
                head[i] = lo;
            }
            rel[i] -= cnt[head[i]];
            if (q + 1 == m || key[q + 1] >> kTileBits != c) {
                if (rel[i] + n[i] == cl_size[c]) whole |= 1u << i;
                else lasts |= 1u << i;
            }
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kEach; ++i)
            if ((whole >> i) & 1u) cnt[head[i]] = cl_off[key[tid * kEach + i] >> kTileBits];
        if (tid == 0 && tile) {
            volatile uint32_t* turn = scratch + kPlaceTurn;
            int it = 0;
            while (*turn != tile && it < kLoopCap) ++it;
            if (it == kLoopCap) atomicOr(err, kErrTimeout);
            __threadfence();
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kEach; ++i)  // all at once; atomic only for the one round trip
            if ((lasts >> i) & 1u) n[i] = atomicAdd(next + (key[tid * kEach + i] >> kTileBits), rel[i] + n[i]);
#pragma unroll
        for (int i = 0; i < kEach; ++i)
            if ((lasts >> i) & 1u) cnt[head[i]] = n[i];
        __syncthreads();
        if (tid == 0) {
            __threadfence();
            *(volatile uint32_t*)(scratch + kPlaceTurn) = tile + 1;
        }
#pragma unroll
        for (int i = 0; i < kEach; ++i) {
            const uint32_t q = tid * kEach + i;
            if (q < m) place[base + ((uint32_t)key[q] & (kPlaceTile - 1))] = cnt[head[i]] + rel[i];
        }
    }
}

template <bool kMany>
__global__ void __launch_bounds__(kOneT, 1) k_cluster_place(const SegCounters* __restrict__ ctr,
                                                         const uint32_t* __restrict__ parent,
                                                         const uint32_t* __restrict__ csize, uint32_t* ccl,
                                                         const uint32_t* __restrict__ cl_size,
                                                         const uint32_t* __restrict__ cl_off,
                                                         uint32_t* __restrict__ place, uint32_t* scratch,
                                                         uint32_t scratch_words, uint32_t* err) {
    pdl_gate();
    extern __shared__ uint32_t sm[];
    const uint32_t K = ctr->n_comp, k = ctr->k_need;
    const int lane = threadIdx.x & 31;
    const uint32_t w = threadIdx.x >> 5;
    uint32_t stretch = max(1024u, ((K + gridDim.x - 1) / gridDim.x + 1023u) & ~1023u);
    uint32_t G = (K + stretch - 1) / stretch;
    constexpr uint32_t kHead = kMany ? kPlaceHead : kPlaceCtas + 1;
    volatile uint32_t* flags = scratch;
    uint32_t* sums = scratch + kHead;
    const bool fit = (size_t)k * (kMany ? 1 : 32) <= kPlaceWords<kMany> && (size_t)G * k + kHead <= scratch_words;
    if constexpr (kMany) {
        if (blockIdx.x >= G) return;
        if (!fit) {
            place_tiles(K, parent, csize, ccl, cl_size, cl_off, place, scratch, sm, err);
            return;
        }
    } else if (!fit) {
        if (k > ctr->k) {  // more clusters than the scratch has room for: the host runs it all again, with kMany
            for (uint32_t c = blockIdx.x * kOneT + threadIdx.x; c < K; c += gridDim.x * kOneT) place[c] = 0;
            return;
        }
        stretch = (K + 1023u) & ~1023u;
        G = 1;
    }
    __shared__ uint32_t s_ticket;
    if (threadIdx.x == 0) s_ticket = atomicAdd(scratch + kPlaceTicket, 1u);
    __syncthreads();
    const uint32_t g = s_ticket;
    if (g >= G) return;
    const uint32_t first = g * stretch, end = min(K, first + stretch);
    constexpr int kIt = 8;
    // each component's cluster (a root's entry is read and rewritten with the same value)
    for (uint32_t c0 = first + threadIdx.x; c0 < end; c0 += kOneT * kIt) {
        uint32_t root[kIt], cl[kIt];
#pragma unroll
        for (int i = 0; i < kIt; ++i) root[i] = c0 + i * kOneT < end ? parent[c0 + i * kOneT] : kNone;
#pragma unroll
        for (int i = 0; i < kIt; ++i) cl[i] = root[i] != kNone ? __ldcg(ccl + root[i]) : kNone;
#pragma unroll
        for (int i = 0; i < kIt; ++i)
            if (root[i] != kNone) ccl[c0 + i * kOneT] = cl[i];
    }
    if (k == 0) return;
    uint32_t* cnt = kMany || fit ? sm : sums;
    // warps with counts of their own
    const uint32_t W = kMany ? min(32u, kPlaceWords<kMany> / k) : (fit ? 32u : min(32u, (scratch_words - kHead) / k));
    for (uint32_t q = threadIdx.x; q < W * k; q += kOneT) cnt[q] = 0;
    __syncthreads();
    const uint32_t len = ((end - first + W - 1) / W + 31) & ~31u;
    const uint32_t lo = min(end, first + w * len), hi = w < W ? min(end, lo + len) : lo;
    uint32_t* mine = cnt + (size_t)(w < W ? w : 0) * k;
    for (uint32_t c0 = lo; c0 < hi; c0 += 32 * kIt) {  // kIt steps' loads go out together
        uint32_t cl[kIt], n[kIt];
#pragma unroll
        for (int i = 0; i < kIt; ++i) {
            const uint32_t c = c0 + i * 32 + lane;
            cl[i] = c < hi ? __ldcg(ccl + c) : kNone;
            n[i] = c < hi ? csize[c] : 0u;
        }
#pragma unroll
        for (int i = 0; i < kIt; ++i) {
            if (c0 + i * 32 >= hi) break;
            const uint32_t grp = __match_any_sync(0xffffffffu, cl[i]);
            const uint32_t sum = __reduce_add_sync(grp, n[i]);
            if (cl[i] != kNone && lane == __ffs(grp) - 1) mine[cl[i]] += sum;
            __syncwarp();
        }
    }
    __syncthreads();
    for (uint32_t cl = w; cl < k; cl += kOneT / 32) {  // a warp a cluster, a lane a warp's counts
        uint32_t* at = cnt + (size_t)lane * k + cl;
        const uint32_t t = lane < (int)W ? *at : 0u, inc = warp_incl(t);
        if (lane < (int)W) *at = inc - t;
        if ((kMany || fit) && lane == 31) sums[(size_t)g * k + cl] = inc;
    }
    if (G > 1) {
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) flags[g] = 1;
        if (threadIdx.x < g) {
            int it = 0;
            while (!flags[threadIdx.x] && it < kLoopCap) ++it;
            if (it == kLoopCap) atomicOr(err, kErrTimeout);
        }
        __threadfence();
    }
    __syncthreads();
    for (uint32_t cl = threadIdx.x; cl < k; cl += kOneT) {  // the cluster's points before this CTA's
        uint32_t b = cl_off[cl];
        for (uint32_t q = 0; q < g; ++q) b += __ldcg(sums + (size_t)q * k + cl);
        for (uint32_t q = 0; q < W; ++q) cnt[(size_t)q * k + cl] += b;
    }
    __syncthreads();
    for (uint32_t c0 = lo; c0 < hi; c0 += 32 * kIt) {
        uint32_t cl[kIt], n[kIt];
#pragma unroll
        for (int i = 0; i < kIt; ++i) {
            const uint32_t c = c0 + i * 32 + lane;
            cl[i] = c < hi ? __ldcg(ccl + c) : kNone;
            n[i] = c < hi ? csize[c] : 0u;
        }
#pragma unroll
        for (int i = 0; i < kIt; ++i) {
            uint32_t todo = __ballot_sync(0xffffffffu, cl[i] != kNone);
            while (todo) {  // one cluster of the 32 a round
                const uint32_t who = __shfl_sync(0xffffffffu, cl[i], __ffs(todo) - 1);
                const bool in = cl[i] == who;
                const uint32_t inc = warp_incl(in ? n[i] : 0u), b0 = mine[who];
                __syncwarp();
                if (in) place[c0 + i * 32 + lane] = b0 + inc - n[i];
                if (lane == 31) mine[who] = b0 + inc;
                __syncwarp();
                todo &= ~__ballot_sync(0xffffffffu, in);
            }
        }
    }
}

// Cluster point lists: mean positions and voxel ids in cluster order, inside a
// cluster in voxel-id order.  A warp takes a brick and walks its voxels in
// order, 32 at a time; components of the brick that belong to one cluster
// share the place of the first of them.
constexpr int kScatWarps = 4;
__global__ void __launch_bounds__(kScatWarps * 32) k_cluster_scatter(const SegCounters* __restrict__ ctr,
                                                                     uint32_t cap_b,
                                                                     const BrickRec* __restrict__ brec,
                                                                     const uint32_t* __restrict__ ncomp,
                                                                     const uint32_t* __restrict__ cbase,
                                                                     const uint32_t* __restrict__ ccl,
                                                                     const uint32_t* __restrict__ place,
                                                                     const uint16_t* __restrict__ lc,
                                                                     const uint32_t* __restrict__ vox,
                                                                     const float4* __restrict__ pos,
                                                                     float* __restrict__ pts,
                                                                     uint32_t* __restrict__ pt_vid) {
    pdl_gate();
    __shared__ uint32_t scl[kScatWarps][kBrickVox], sat[kScatWarps][kBrickVox];
    __shared__ uint16_t slead[kScatWarps][kBrickVox];
    const uint32_t n_sorted = min(ctr->n_sorted, cap_b);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t *cl = scl[w], *at = sat[w];
    uint16_t* lead = slead[w];
    for (uint32_t r = blockIdx.x * kScatWarps + w; r < n_sorted; r += gridDim.x * kScatWarps) {
        const uint4 hd = *reinterpret_cast<const uint4*>(&brec[r].base);  // base, n, key, slot
        const uint32_t nc = ncomp[r], c0 = cbase[r];
        if (!nc) continue;
        __syncwarp();
        for (uint32_t j = lane; j < nc; j += 32) {
            cl[j] = ccl[c0 + j];
            at[j] = cl[j] != kNone ? place[c0 + j] : 0u;
        }
        __syncwarp();
        for (uint32_t j = lane; j < nc; j += 32) {
            uint32_t f = 0;
            const uint32_t c = cl[j];
            while (c != kNone && cl[f] != c) ++f;  // at most j
            lead[j] = c != kNone ? (uint16_t)f : kNoComp;
        }
        __syncwarp();
        for (uint32_t p0 = 0; p0 < hd.y; p0 += 32) {
            const uint32_t i = hd.x + p0 + lane;
            uint32_t f = kNoComp;
            float4 a = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            uint32_t l = 0;
            if (p0 + lane < hd.y) {
                const uint16_t j = lc[i];
                a = pos[i];
                l = vox[i] % kBrickVox;
                if (j != kNoComp) f = lead[j];
            }
            const uint32_t m = __match_any_sync(0xffffffffu, f);
            const uint32_t rank = __popc(m & ((1u << lane) - 1u));
            const uint32_t b0 = f != kNoComp ? at[f] : 0u;
            __syncwarp();
            if (f != kNoComp && rank == 0) at[f] = b0 + __popc(m);
            __syncwarp();
            if (f != kNoComp) {
                const size_t q = b0 + rank;
                pts[3 * q + 0] = a.x;
                pts[3 * q + 1] = a.y;
                pts[3 * q + 2] = a.z;
                pt_vid[q] = hd.z * kBrickVox + l;
            }
        }
    }
}

}  // namespace

cudaError_t seg_order_bricks(const int32_t* brick_table, uint32_t nb_total, const uint32_t* occ, SegBuffers& b,
                             cudaStream_t s, uint32_t* zero0, uint32_t* zero1) {
    // the counter block opens with the two counts the pass writes; it clears the others
    static_assert(offsetof(SegCounters, n_sorted) == 0 && offsetof(SegCounters, n_occ) == 4,
                  "the brick and voxel counts lead the segmentation counters");
    return order_bricks_dev(brick_table, nb_total, occ, b.rank_table, b.sorted_slot, b.sorted_key, b.brec,
                            reinterpret_cast<uint32_t*>(b.ctr), (int)(sizeof(SegCounters) / 4), zero0, zero1,
                            b.scan_tmp, s, &b.ctr->err);
}

cudaError_t seg_run(const Grid& g, const unsigned long long* S, const uint32_t* C, const vm_segment_params& p,
                    SegBuffers& b, uint32_t kcap, bool many, uint32_t* err, int sms, cudaStream_t s, StageHook* hk) {
    static std::once_flag once;
    std::call_once(once, [] {
        cudaFuncSetAttribute(k_comp_join, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kJoinWords * 4));
        cudaFuncSetAttribute(k_cluster_place<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(kPlaceWords<false> * 4));
        cudaFuncSetAttribute(k_cluster_place<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(kPlaceWords<true> * 4));
    });
    const uint32_t cap_b = (uint32_t)(b.nv / kBrickVox);
    const size_t stride = b.nv;
    const uint32_t pair_cap = b.nv < b.pair_cap ? (uint32_t)b.nv : b.pair_cap;
    uint32_t* over = b.place;                                   // k_cluster_place writes it after the last join
    uint32_t* scratch = reinterpret_cast<uint32_t*>(b.pairs);   // free once the pairs are joined
    const uint32_t scratch_words = (uint32_t)(2 * b.nv < 0xFFFFFFFFull ? 2 * b.nv : 0xFFFFFFFFull);
    const auto clampg = [&](uint32_t want, uint32_t mx) { return want < mx ? (want ? want : 1u) : mx; };
    // Several waves of short CTAs: with about one, some SMs got a CTA more than others for the whole pass (the per-voxel
    // passes of the 8 x 8 x 3 m map 248 us at 8 CTAs an SM, 219 at 24).  A CTA per two bricks covers their occupied
    // voxels (about a fifth of the slots the scratch has room for); the empty CTAs of larger grids stand in the way of
    // other streams (16 maps served at once: 1.14 ms a pass with a grid for every slot, 1.07 so).
    const unsigned bgrid = clampg(cap_b, sms * 64), vgrid = clampg(cap_b / 2, sms * 24);
    VM_STAGE_BEGIN(hk, kStFinalize, s);
    launch_k(k_finalize, dim3(clampg((cap_b + kFinWarps - 1) / kFinWarps, sms * 8)), dim3(kT), 0, s, b.ctr, cap_b, g,
             b.brec, b.rank_table, S, C, b.M, b.vox, b.near, b.rows);
    VM_STAGE_END(hk, kStFinalize, s);
    const int want = p.classify ? 2 : 1;
    VM_STAGE_BEGIN(hk, kStNormals, s);
    launch_k(k_moments, dim3(vgrid), dim3(kT), 0, s, b.ctr, g.po, b.rows, b.vox, b.M, b.pos, b.list_A, b.nbr,
             b.parent, over, stride);
    VM_STAGE_END(hk, kStNormals, s);
    VM_STAGE_BEGIN(hk, kStEigen, s);
    launch_k(k_eigen, dim3(vgrid), dim3(kT), 0, s, b.ctr, b.list_A, b.nbr, b.nrm, b.pos, stride, p.n_th, p.cos_step);
    VM_STAGE_END(hk, kStEigen, s);
    VM_STAGE_BEGIN(hk, kStCclLocal, s);
    launch_k(k_ccl_local, dim3(bgrid), dim3(kLocalT), 0, s, b.ctr, cap_b, b.brec, b.vox, b.pos, b.nrm, b.lc, b.ncomp,
             b.lsize, b.lroot, want, p.d_th2, p.cos_ccl);
    VM_STAGE_END(hk, kStCclLocal, s);
    VM_STAGE_BEGIN(hk, kStCcl, s);
    launch_k(k_comp_number, dim3(1), dim3(kOneT), 0, s, b.ctr, cap_b, b.ncomp, b.cbase);
    launch_k(k_ccl_cross, dim3(vgrid), dim3(kT), 0, s, b.ctr, b.brec, b.near, b.rows, b.vox, b.pos, b.nrm, b.lc,
             b.ncomp, b.cbase, b.lsize, b.lroot, b.csize, b.croot, b.total, b.parent, over, b.pairs, pair_cap,
             p.d_th2, p.cos_ccl, err);
    // A map of surfaces has one or two components and six pairs a brick: a CTA per thousand of them, as few as there can
    // be work for, since each takes much of an SM's shared memory and other streams' kernels wait for it.  A map of noise
    // (many) has up to hundreds a brick and takes the GPU: 1 x 1 x 1 m with every cell at 0.01 m occupied has its pairs
    // joined in 24 us instead of 54 and its clusters formed in 93 us instead of 365.
    launch_k(k_comp_join, dim3(clampg(many ? cap_b / 16 : cap_b / 128, sms)), dim3(kOneT), kJoinWords * 4, s, b.ctr,
             pair_cap, b.pairs, b.lsize, b.parent, over, err);
    VM_STAGE_END(hk, kStCcl, s);
    VM_STAGE_BEGIN(hk, kStClusters, s);
    launch_k(k_comp_size, dim3(many ? clampg(cap_b / 4, sms * 8) : clampg(cap_b / 64, sms * 2)), dim3(kT), 0, s, b.ctr,
             b.parent, b.csize, b.total, many ? scratch : nullptr, err);
    const uint32_t min_cl = p.min_cluster ? p.min_cluster : 1u;
    if (many) {
        launch_k(k_cluster_number_many, dim3(clampg(cap_b / 16, kPlaceCtas)), dim3(kOneT), 0, s, b.ctr, min_cl, kcap,
                 b.total, b.croot, b.ccl, b.cl_size, b.cl_label, b.cl_off, scratch, err);
        launch_k(k_cluster_place<true>, dim3(clampg(cap_b / 16, kPlaceCtas)), dim3(kOneT), kPlaceWords<true> * 4, s,
                 b.ctr, b.parent, b.csize, b.ccl, b.cl_size, b.cl_off, b.place, scratch, scratch_words, err);
    } else {
        launch_k(k_cluster_number, dim3(1), dim3(kOneT), 0, s, b.ctr, min_cl, kcap, b.total, b.croot, b.ccl, b.cl_size,
                 b.cl_label, b.cl_off, scratch);
        launch_k(k_cluster_place<false>, dim3(clampg(cap_b / 512 + 1, kPlaceCtas)), dim3(kOneT), kPlaceWords<false> * 4,
                 s, b.ctr, b.parent, b.csize, b.ccl, b.cl_size, b.cl_off, b.place, scratch, scratch_words, err);
    }
    launch_k(k_cluster_scatter, dim3(clampg((cap_b + kScatWarps - 1) / kScatWarps, sms * 8)), dim3(kScatWarps * 32), 0,
             s, b.ctr, cap_b, b.brec, b.ncomp, b.cbase, b.ccl, b.place, b.lc, b.vox, b.pos, b.pts, b.pt_vid);
    VM_STAGE_END(hk, kStClusters, s);
    count_launch(11);
    return cudaGetLastError();
}

}  // namespace vmx
