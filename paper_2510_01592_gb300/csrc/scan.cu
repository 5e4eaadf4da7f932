// scan.cu -- device-wide exclusive prefix sum, and the ordering of the
// allocated bricks and their occupied voxels by id that every per-voxel array
// of a segmentation follows (Sec. III.C).
#include "vm_internal.cuh"

namespace vmx {
namespace {

constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;  // 2048

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// Block-wide exclusive scan of one value per thread (blockDim.x == kScanThreads).
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t* warp_sums, uint32_t* block_total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t inc = warp_incl_scan(v);
    if (lane == 31) warp_sums[w] = inc;
    __syncthreads();
    if (w == 0) {
        uint32_t s = (lane < kScanThreads / 32) ? warp_sums[lane] : 0u;
        uint32_t si = warp_incl_scan(s);
        if (lane < kScanThreads / 32) warp_sums[lane] = si - s;
        if (lane == kScanThreads / 32 - 1) *block_total = si;
    }
    __syncthreads();
    return inc - v + warp_sums[w];
}

// n_dev (optional): the element count read on the device, clamped to n.
__device__ __forceinline__ size_t dev_count(size_t n, const uint32_t* n_dev) {
    if (!n_dev) return n;
    const size_t d = *n_dev;
    return d < n ? d : n;
}

// Single-pass scan with decoupled look-back (Merrill and Garland, "Single-pass
// parallel prefix scan with decoupled look-back", 2016).  Each CTA takes the
// next tile from a ticket counter (so every earlier tile belongs to a CTA that
// has started), publishes its tile sum, then walks back over earlier tiles'
// published words, 256 at a time, until it meets an inclusive prefix, and
// publishes its own.
// A status word is (epoch << 34 | flag << 32 | value), a 30-bit epoch: words
// of an earlier launch (another epoch) read as not yet published, so no
// clearing pass is needed.  The ticket counter and the epoch share a word, so
// one atomic reads both, and the CTA that draws the last ticket can make it
// ready for the next launch at once.
// The state (that word, 8 bytes unused, then the 64-bit status words) must
// start zeroed once, when its memory is allocated.  Every wait is bounded: a
// wait that runs out sets kErrTimeout in *err and counts the missing prefix
// as 0.
constexpr unsigned long long kFlagAgg = 1ull, kFlagInc = 2ull;
constexpr int kLookbackCap = 1 << 20;

constexpr uint32_t kEpochMask = (1u << 30) - 1u;
__device__ __forceinline__ unsigned long long lb_word(uint32_t epoch, unsigned long long flag, uint32_t v) {
    return ((unsigned long long)(epoch & kEpochMask) << 34) | (flag << 32) | (unsigned long long)v;
}

// The calling thread's ticket and the launch's epoch.
__device__ __forceinline__ uint2 take_tile(uint32_t* state) {
    unsigned long long* word = reinterpret_cast<unsigned long long*>(state);
    const unsigned long long t = atomicAdd(word, 1ull);
    const uint32_t tile = (uint32_t)t, epoch = (uint32_t)(t >> 32);
    if (tile == gridDim.x - 1) *word = (unsigned long long)(epoch + 1u) << 32;
    return make_uint2(tile, epoch);
}

// Publishes the tile's sums, looks back for those of the tiles before it (unless
// skip) and publishes the inclusive ones, for K arrays of nt status words each
// at once, by a CTA of kScanThreads threads.  agg and before: the same in every
// thread.  (A thread looking back a tile at a time took 11.7 us over the 80
// tiles of a walk map's points, the CTA 5.)
template <int K>
__device__ __forceinline__ void cta_look_back(unsigned long long* status, uint32_t nt, uint32_t tile, uint32_t epoch,
                                              const uint32_t (&agg)[K], bool skip, uint32_t (&before)[K],
                                              uint32_t* err) {
    constexpr int kWarps = kScanThreads / 32;
    __shared__ uint32_t part[K][kWarps], stop[K][kWarps];
    const uint32_t tid = threadIdx.x;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        before[k] = 0u;
        if (tid == (uint32_t)k) atomicExch(status + k * nt + tile, lb_word(epoch, tile ? kFlagAgg : kFlagInc, agg[k]));
    }
    if (skip || !tile) return;
    bool done[K] = {};
    for (int64_t top = (int64_t)tile - 1; top >= 0; top -= kScanThreads) {
        const int64_t p = top - tid;
        unsigned long long w[K] = {};
        bool ready[K], all = p < 0;
#pragma unroll
        for (int k = 0; k < K; ++k) ready[k] = p < 0;
        // every earlier tile belongs to a CTA that has started, and publishes before it waits
        for (int it = 0; it < kLookbackCap && !all; ++it) {
            all = true;
#pragma unroll
            for (int k = 0; k < K; ++k) {
                if (ready[k]) continue;
                w[k] = *(volatile unsigned long long*)(status + k * nt + p);
                ready[k] = (uint32_t)(w[k] >> 34) == (epoch & kEpochMask) && ((w[k] >> 32) & 3ull);
                all &= ready[k];
            }
        }
        if (err && !all) atomicOr(err, kErrTimeout);  // never published: counted as 0
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const bool there = ready[k] && p >= 0;
            const uint32_t inc = __ballot_sync(0xffffffffu, there && ((w[k] >> 32) & 3ull) == kFlagInc);
            const uint32_t need = inc ? (inc & (0u - inc)) * 2u - 1u : 0xffffffffu;  // up to the nearest inclusive sum
            const uint32_t sum =
                __reduce_add_sync(0xffffffffu, there && ((need >> (tid & 31)) & 1u) ? (uint32_t)w[k] : 0u);
            if ((tid & 31) == 0) {
                part[k][tid >> 5] = sum;
                stop[k][tid >> 5] = inc;
            }
        }
        __syncthreads();
        bool every = true;
#pragma unroll
        for (int k = 0; k < K; ++k) {
#pragma unroll
            for (int q = 0; q < kWarps; ++q)
                if (!done[k]) {
                    before[k] += part[k][q];
                    done[k] = stop[k][q] != 0u;
                }
            every &= done[k];
        }
        __syncthreads();
        if (every) break;
    }
#pragma unroll
    for (int k = 0; k < K; ++k)
        if (tid == (uint32_t)k) atomicExch(status + k * nt + tile, lb_word(epoch, kFlagInc, before[k] + agg[k]));
}

__global__ void __launch_bounds__(kScanThreads) k_scan_lookback(const uint32_t* in, uint32_t* out, size_t n_cap,
                                                                const uint32_t* __restrict__ n_dev,
                                                                uint32_t* __restrict__ total,
                                                                uint32_t* __restrict__ state, uint32_t* err, int end) {
    pdl_gate();
    __shared__ uint32_t buf[kScanTile];
    __shared__ uint32_t ws[kScanThreads / 32];
    __shared__ uint32_t tot;
    __shared__ uint2 s_tile;
    unsigned long long* status = reinterpret_cast<unsigned long long*>(state + 4);
    const size_t n = dev_count(n_cap, n_dev);
    const uint32_t nt_used = (uint32_t)((n + kScanTile - 1) / kScanTile);
    if (threadIdx.x == 0) s_tile = take_tile(state);
    __syncthreads();
    const uint32_t tile = s_tile.x, epoch = s_tile.y;
    if (tile < nt_used) {
        const size_t base = (size_t)tile * kScanTile;
#pragma unroll
        for (int i = 0; i < kScanItems; ++i) {
            const int t = i * kScanThreads + threadIdx.x;
            const size_t j = base + t;
            buf[t] = (j < n) ? in[j] : 0u;
        }
        __syncthreads();
        uint32_t v[kScanItems];
        uint32_t sum = 0;
#pragma unroll
        for (int i = 0; i < kScanItems; ++i) {
            v[i] = buf[threadIdx.x * kScanItems + i];
            sum += v[i];
        }
        const uint32_t ex_local = block_excl_scan(sum, ws, &tot);
        const uint32_t agg[1] = {tot};
        uint32_t before[1];
        cta_look_back<1>(status, nt_used, tile, epoch, agg, false, before, err);
        if (threadIdx.x == 0 && tile == nt_used - 1) {
            if (total) *total = before[0] + agg[0];
            if (end) out[n] = before[0] + agg[0];  // no tile reads in[n]
        }
        uint32_t ex = ex_local + before[0];
#pragma unroll
        for (int i = 0; i < kScanItems; ++i) {
            buf[threadIdx.x * kScanItems + i] = ex;
            ex += v[i];
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kScanItems; ++i) {
            const int t = i * kScanThreads + threadIdx.x;
            const size_t j = base + t;
            if (j < n) out[j] = buf[t];
        }
    } else if (tile == 0 && threadIdx.x == 0) {  // nothing to scan
        if (total) *total = 0;
        if (end) out[0] = 0;
    }
}

// The allocated bricks in key order and their occupied voxels' places, in one
// pass (a stream compaction with a look-back scan over two sums at once): tile
// t of the brick table counts its allocated entries (slot >= 0) and their
// occupied voxels (from the pool's occupancy bitmap), looks back for the
// bricks and the voxels before the tile, then writes every entry's rank (or
// -1) and, per allocated brick, its slot, key and record at its rank.  The
// last tile writes the two counts to clear[0] and clear[1].  Block 0 also
// clears the words clear[2 .. n_clear) (a counter block that opens with the
// two counts) and zero0 / zero1 (may be null).  A chain of dependent loads
// bounds it, not bytes, so the chain is short: a thread takes one entry and
// keeps its bitmap in registers, and the whole CTA looks back, over 256 earlier
// tiles at a time.  Allocated bricks cluster (a floor fills a whole z layer of
// the table), so small tiles also spread them over the GPU: 5.5 us for the 62
// thousand entries of the 4 x 4 x 2 m map and 14 for the 380 thousand of the
// 8 x 8 x 3 m one; tiles of 1024 with a warp looking back took 11 and 21.7.
constexpr int kOrdTile = kScanThreads;
__global__ void __launch_bounds__(kScanThreads, 6) k_order_bricks(const int32_t* __restrict__ table, uint32_t nb,
                                                               const uint32_t* __restrict__ occ,
                                                               int32_t* __restrict__ rank_table,
                                                               int32_t* __restrict__ sorted_slot,
                                                               int32_t* __restrict__ sorted_key,
                                                               BrickRec* __restrict__ brec,
                                                               uint32_t* __restrict__ clear, int n_clear,
                                                               uint32_t* __restrict__ zero0,
                                                               uint32_t* __restrict__ zero1,
                                                               uint32_t* __restrict__ state, uint32_t* err) {
    pdl_gate();
    __shared__ uint32_t ws[kScanThreads / 32];
    __shared__ uint32_t tot;
    __shared__ uint2 s_tile;
    const uint32_t nt_used = (nb + kOrdTile - 1) / kOrdTile;
    unsigned long long* status = reinterpret_cast<unsigned long long*>(state + 4);  // bricks, then voxels
    if (blockIdx.x == 0) {
        for (int i = 2 + threadIdx.x; i < n_clear; i += kScanThreads) clear[i] = 0u;
        if (threadIdx.x == 0) {
            if (zero0) *zero0 = 0u;
            if (zero1) *zero1 = 0u;
        }
    }
    if (threadIdx.x == 0) s_tile = take_tile(state);
    __syncthreads();
    const uint32_t tile = s_tile.x, epoch = s_tile.y;
    if (tile < nt_used) {
        const uint32_t key = tile * kOrdTile + threadIdx.x;
        const int32_t slot = key < nb ? table[key] : -1;
        uint4 m[4] = {};
        uint32_t n = 0;
        if (slot >= 0) {
#pragma unroll
            for (int q = 0; q < 4; ++q) m[q] = reinterpret_cast<const uint4*>(occ + (size_t)slot * 16)[q];
#pragma unroll
            for (int q = 0; q < 4; ++q) n += __popc(m[q].x) + __popc(m[q].y) + __popc(m[q].z) + __popc(m[q].w);
        } else if (key < nb) {
            rank_table[key] = -1;
        }
        // both sums in one scan: at most 2^17 voxels and 2^8 bricks in a tile
        static_assert(kOrdTile * kBrickVox < (1 << 18), "the voxels of a tile fit below bit 18");
        const uint32_t ex = block_excl_scan(n | (slot >= 0 ? 1u << 18 : 0u), ws, &tot);
        const uint32_t agg[2] = {tot >> 18, tot & 0x3ffffu};
        // an empty tile needs no sums, but the last one counts and every 256th keeps the walks short
        const bool skip = !tot && tile != nt_used - 1 && tile % kScanThreads != 0;
        uint32_t before[2];
        cta_look_back<2>(status, nt_used, tile, epoch, agg, skip, before, err);
        if (tile == nt_used - 1 && threadIdx.x < 2)
            clear[threadIdx.x] = threadIdx.x ? before[1] + agg[1] : before[0] + agg[0];
        if (slot >= 0) {
            const uint32_t rank = before[0] + (ex >> 18);
            BrickRec* r = brec + rank;
            uint32_t run = 0;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                reinterpret_cast<uint4*>(r->mask)[q] = m[q];
                const uint32_t p0 = run, p1 = p0 + __popc(m[q].x), p2 = p1 + __popc(m[q].y), p3 = p2 + __popc(m[q].z);
                run = p3 + __popc(m[q].w);
                reinterpret_cast<uint2*>(r->pre)[q] = make_uint2(p0 | (p1 << 16), p2 | (p3 << 16));
            }
            *reinterpret_cast<uint4*>(&r->base) = make_uint4(before[1] + (ex & 0x3ffffu), run, key, (uint32_t)slot);
            sorted_slot[rank] = slot;
            sorted_key[rank] = (int32_t)key;
            rank_table[key] = (int32_t)rank;
        }
    } else if (tile == 0 && threadIdx.x == 0) {  // an empty table
        clear[0] = 0u;
        clear[1] = 0u;
    }
}

// Small inputs: one 1024-thread CTA scans everything, four items per thread
// per round, carrying the running total across rounds.
constexpr int kSmallThreads = 1024;
constexpr int kSmallItems = 4;
constexpr size_t kSmallMax = 16384;

__global__ void __launch_bounds__(kSmallThreads) k_scan_small(const uint32_t* in, uint32_t* out, size_t n_cap,
                                                              const uint32_t* __restrict__ n_dev, uint32_t* total,
                                                              int end) {
    pdl_gate();
    __shared__ uint32_t ws[kSmallThreads / 32];
    __shared__ uint32_t round_total;
    const size_t n = dev_count(n_cap, n_dev);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t carry = 0;
    for (size_t base = 0; base < n; base += (size_t)kSmallThreads * kSmallItems) {
        const size_t j0 = base + (size_t)threadIdx.x * kSmallItems;
        uint32_t v[kSmallItems], sum = 0;
#pragma unroll
        for (int i = 0; i < kSmallItems; ++i) {
            v[i] = (j0 + i < n) ? in[j0 + i] : 0u;
            sum += v[i];
        }
        const uint32_t inc = warp_incl_scan(sum);
        if (lane == 31) ws[w] = inc;
        __syncthreads();
        if (w == 0) {
            const uint32_t t = ws[lane];
            const uint32_t ti = warp_incl_scan(t);
            ws[lane] = ti - t;
            if (lane == 31) round_total = ti;
        }
        __syncthreads();
        uint32_t ex = carry + ws[w] + (inc - sum);
#pragma unroll
        for (int i = 0; i < kSmallItems; ++i) {
            if (j0 + i < n) out[j0 + i] = ex;
            ex += v[i];
        }
        carry += round_total;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        if (total) *total = carry;
        if (end) out[n] = carry;  // read by no thread: every load is below n
    }
}

}  // namespace

static_assert((size_t)kOrdTile == kOrderTileElems, "order_tmp_words assumes the ordering's tile size");
static_assert((size_t)kScanTile == kScanTileElems, "scan_tmp_words assumes the scan's tile size");

cudaError_t exclusive_scan_dev(const uint32_t* in, uint32_t* out, uint32_t* total, const uint32_t* n_dev, size_t n_cap,
                               uint32_t* tmp, cudaStream_t s, uint32_t* err, bool end) {
    if (n_cap == 0) {
        cudaError_t e = cudaSuccess;
        if (total) e = cudaMemsetAsync(total, 0, sizeof(uint32_t), s);
        if (end && e == cudaSuccess) e = cudaMemsetAsync(out, 0, sizeof(uint32_t), s);
        return e;
    }
    if (n_cap <= kSmallMax) {
        launch_k(k_scan_small, dim3(1), dim3(kSmallThreads), 0, s, in, out, n_cap, n_dev, total, (int)end);
        count_launch(1);
        return cudaGetLastError();
    }
    if (reinterpret_cast<uintptr_t>(tmp) & 7) return cudaErrorInvalidValue;  // 64-bit status words
    const size_t nt = (n_cap + kScanTile - 1) / kScanTile;
    launch_k(k_scan_lookback, dim3((unsigned)nt), dim3(kScanThreads), 0, s, in, out, n_cap, n_dev, total, tmp, err,
             (int)end);
    count_launch(1);
    return cudaGetLastError();
}

cudaError_t order_bricks_dev(const int32_t* table, uint32_t nb, const uint32_t* occ, int32_t* rank_table,
                             int32_t* sorted_slot, int32_t* sorted_key, BrickRec* brec, uint32_t* clear, int n_clear,
                             uint32_t* zero0, uint32_t* zero1, uint32_t* tmp, cudaStream_t s, uint32_t* err) {
    if (reinterpret_cast<uintptr_t>(tmp) & 7) return cudaErrorInvalidValue;  // 64-bit status words
    const size_t nt = ((size_t)nb + kOrdTile - 1) / kOrdTile;
    launch_k(k_order_bricks, dim3((unsigned)(nt ? nt : 1)), dim3(kScanThreads), 0, s, table, nb, occ, rank_table,
             sorted_slot, sorted_key, brec, clear, n_clear, zero0, zero1, tmp, err);
    count_launch(1);
    return cudaGetLastError();
}

}  // namespace vmx
