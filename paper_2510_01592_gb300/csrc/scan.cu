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
// published words until it meets an inclusive prefix, and publishes its own.
// A status word is (epoch << 34 | flag << 32 | value), a 30-bit epoch: words
// of an earlier launch (another epoch) read as not yet published, so no
// clearing pass is needed; the last CTA to finish resets the ticket and
// advances the epoch.
// The state (ticket, done, epoch, then one 64-bit word per tile) must start
// zeroed once, when its memory is allocated.  Every wait is bounded: a wait
// that runs out sets kErrTimeout in *err and counts the missing prefix as 0.
constexpr unsigned long long kFlagAgg = 1ull, kFlagInc = 2ull;
constexpr int kLookbackCap = 1 << 20;

constexpr uint32_t kEpochMask = (1u << 30) - 1u;
__device__ __forceinline__ unsigned long long lb_word(uint32_t epoch, unsigned long long flag, uint32_t v) {
    return ((unsigned long long)(epoch & kEpochMask) << 34) | (flag << 32) | (unsigned long long)v;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_lookback(const uint32_t* in, uint32_t* out, size_t n_cap,
                                                                const uint32_t* __restrict__ n_dev,
                                                                uint32_t* __restrict__ total,
                                                                uint32_t* __restrict__ state, uint32_t* err, int end) {
    pdl_gate();
    __shared__ uint32_t buf[kScanTile];
    __shared__ uint32_t ws[kScanThreads / 32];
    __shared__ uint32_t tot, s_tile, s_prefix;
    unsigned long long* status = reinterpret_cast<unsigned long long*>(state + 4);
    const size_t n = dev_count(n_cap, n_dev);
    const uint32_t nt_used = (uint32_t)((n + kScanTile - 1) / kScanTile);
    const uint32_t epoch = *(volatile uint32_t*)(state + 2);
    if (threadIdx.x == 0) s_tile = atomicAdd(state, 1u);
    __syncthreads();
    const uint32_t tile = s_tile;
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
        if (threadIdx.x == 0) {
            const uint32_t agg = tot;
            uint32_t prefix = 0;
            if (tile == 0) {
                atomicExch(status, lb_word(epoch, kFlagInc, agg));
            } else {
                atomicExch(status + tile, lb_word(epoch, kFlagAgg, agg));
                for (int64_t p = (int64_t)tile - 1; p >= 0; --p) {
                    unsigned long long w = 0;
                    int it = 0;
                    for (; it < kLookbackCap; ++it) {
                        w = *(volatile unsigned long long*)(status + p);
                        if ((uint32_t)(w >> 34) == (epoch & kEpochMask) && ((w >> 32) & 3ull)) break;
                    }
                    if (it == kLookbackCap) {  // the predecessor never published: report, count it as 0
                        if (err) atomicOr(err, kErrTimeout);
                        break;
                    }
                    prefix += (uint32_t)(w & 0xffffffffull);
                    if (((w >> 32) & 3ull) == kFlagInc) break;
                }
                atomicExch(status + tile, lb_word(epoch, kFlagInc, prefix + agg));
            }
            s_prefix = prefix;
            if (tile == nt_used - 1) {
                if (total) *total = prefix + agg;
                if (end) out[n] = prefix + agg;  // no tile reads in[n]
            }
        }
        __syncthreads();
        uint32_t ex = ex_local + s_prefix;
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
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(state + 1, 1u) == gridDim.x - 1) {  // the last CTA: reset for the next launch
            state[0] = 0;
            state[1] = 0;
            state[2] = epoch + 1;
            __threadfence();
        }
    }
}

// Looks back, a warp over 32 earlier tiles at a time, for the sum of the tiles
// before `tile` in one array of status words, and publishes the inclusive sum.
// Every earlier tile belongs to a CTA that has started; the wait is capped.
__device__ __forceinline__ uint32_t warp_look_back(unsigned long long* status, uint32_t tile, uint32_t epoch,
                                                   uint32_t agg, uint32_t* err) {
    const int lane = threadIdx.x & 31;
    uint32_t prefix = 0;
    for (int64_t top = (int64_t)tile - 1; top >= 0; top -= 32) {
        const int64_t p = top - lane;
        unsigned long long w = 0;
        bool ready = p < 0;
        for (int it = 0; it < kLookbackCap; ++it) {
            if (!ready) {
                w = *(volatile unsigned long long*)(status + p);
                ready = (uint32_t)(w >> 34) == (epoch & kEpochMask) && ((w >> 32) & 3ull);
            }
            // the nearest inclusive sum ends the walk: only the tiles up to it have to be there
            const uint32_t inc = __ballot_sync(0xffffffffu, ready && p >= 0 && ((w >> 32) & 3ull) == kFlagInc);
            const uint32_t need = inc ? (inc & (0u - inc)) * 2u - 1u : 0xffffffffu;
            if ((__ballot_sync(0xffffffffu, ready) & need) == need) break;
        }
        const uint32_t inc = __ballot_sync(0xffffffffu, ready && p >= 0 && ((w >> 32) & 3ull) == kFlagInc);
        const uint32_t need = inc ? (inc & (0u - inc)) * 2u - 1u : 0xffffffffu;
        const bool in = (need >> lane) & 1u;
        if (__any_sync(0xffffffffu, in && !ready)) {  // a predecessor never published: report, count it as 0
            if (err && lane == 0) atomicOr(err, kErrTimeout);
        }
        prefix += __reduce_add_sync(0xffffffffu, in && ready && p >= 0 ? (uint32_t)(w & 0xffffffffull) : 0u);
        if (inc) break;
    }
    if (lane == 0) atomicExch(status + tile, lb_word(epoch, kFlagInc, prefix + agg));
    return prefix;
}

// The allocated bricks in key order and their occupied voxels' places, in one
// pass (a stream compaction with the look-back scan above, over two sums at
// once): tile t of the brick table lists its allocated entries (slot >= 0) and
// their occupied voxels (from the pool's occupancy bitmap), looks back for the
// bricks and the voxels before the tile, then writes every entry's rank (or
// -1) and, per allocated brick, its slot, key and record at its rank.  The
// last tile writes the two counts to clear[0] and clear[1].  Block 0 also
// clears the words clear[2 .. n_clear) (a counter block that opens with the
// two counts) and zero0 / zero1 (may be null).  Allocated bricks cluster (a
// floor fills a whole z layer of the table), so tiles are small and a thread
// takes a brick, its whole bitmap in four loads.
constexpr int kOrdItems = 4;
constexpr int kOrdTile = kScanThreads * kOrdItems;
__device__ __forceinline__ void load_bits(const uint32_t* __restrict__ occ, int32_t slot, uint4 (&m)[4]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) m[q] = reinterpret_cast<const uint4*>(occ + (size_t)slot * 16)[q];
}
__global__ void __launch_bounds__(kScanThreads) k_order_bricks(const int32_t* __restrict__ table, uint32_t nb,
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
    __shared__ int32_t buf[kOrdTile];    // the tile's table entries, then its allocated slots
    __shared__ uint16_t lkey[kOrdTile];  // the allocated entries' places in the tile
    __shared__ uint32_t lvox[kOrdTile];  // their occupied voxels, then the voxels before them
    __shared__ uint32_t ws[kScanThreads / 32];
    __shared__ uint32_t tot, s_tile, s_prefix[2];
    const uint32_t nt_used = (nb + kOrdTile - 1) / kOrdTile;
    unsigned long long* status = reinterpret_cast<unsigned long long*>(state + 4);
    if (blockIdx.x == 0) {
        for (int i = 2 + threadIdx.x; i < n_clear; i += kScanThreads) clear[i] = 0u;
        if (threadIdx.x == 0) {
            if (zero0) *zero0 = 0u;
            if (zero1) *zero1 = 0u;
        }
    }
    const uint32_t epoch = *(volatile uint32_t*)(state + 2);
    if (threadIdx.x == 0) s_tile = atomicAdd(state, 1u);
    __syncthreads();
    const uint32_t tile = s_tile;
    if (tile < nt_used) {
        const uint32_t base = tile * kOrdTile;
#pragma unroll
        for (int i = 0; i < kOrdItems; ++i) {
            const uint32_t j = base + i * kScanThreads + threadIdx.x;
            buf[i * kScanThreads + threadIdx.x] = j < nb ? table[j] : -1;
        }
        __syncthreads();
        int32_t v[kOrdItems];
        uint32_t sum = 0;
#pragma unroll
        for (int i = 0; i < kOrdItems; ++i) {
            v[i] = buf[threadIdx.x * kOrdItems + i];
            sum += v[i] >= 0;
            if (v[i] < 0 && base + threadIdx.x * kOrdItems + i < nb)
                rank_table[base + threadIdx.x * kOrdItems + i] = -1;
        }
        uint32_t at = block_excl_scan(sum, ws, &tot);  // its barriers also end the reads of buf
#pragma unroll
        for (int i = 0; i < kOrdItems; ++i)
            if (v[i] >= 0) {
                buf[at] = v[i];
                lkey[at++] = (uint16_t)(threadIdx.x * kOrdItems + i);
            }
        __syncthreads();
        const uint32_t nbr = tot;
        for (uint32_t b = threadIdx.x; b < nbr; b += kScanThreads) {
            uint4 m[4];
            load_bits(occ, buf[b], m);
            uint32_t c = 0;
#pragma unroll
            for (int q = 0; q < 4; ++q) c += __popc(m[q].x) + __popc(m[q].y) + __popc(m[q].z) + __popc(m[q].w);
            lvox[b] = c;
        }
        __syncthreads();
        uint32_t n[kOrdItems], nsum = 0;
#pragma unroll
        for (int i = 0; i < kOrdItems; ++i) {
            const uint32_t b = threadIdx.x * kOrdItems + i;
            n[i] = b < nbr ? lvox[b] : 0u;
            nsum += n[i];
        }
        uint32_t ex = block_excl_scan(nsum, ws, &tot);
#pragma unroll
        for (int i = 0; i < kOrdItems; ++i) {
            const uint32_t b = threadIdx.x * kOrdItems + i;
            if (b < nbr) lvox[b] = ex;
            ex += n[i];
        }
        if (threadIdx.x < 64) {  // warp 0: bricks, warp 1: voxels (its status words lie behind the first's)
            const int which = threadIdx.x >> 5;
            const uint32_t agg = which ? tot : nbr;
            unsigned long long* st = status + (which ? nt_used : 0);
            if ((threadIdx.x & 31) == 0) atomicExch(st + tile, lb_word(epoch, tile ? kFlagAgg : kFlagInc, agg));
            const uint32_t prefix = tile ? warp_look_back(st, tile, epoch, agg, err) : 0u;
            if ((threadIdx.x & 31) == 0) {
                s_prefix[which] = prefix;
                if (tile == nt_used - 1) clear[which] = prefix + agg;
            }
        }
        __syncthreads();
        const uint32_t rank0 = s_prefix[0], vox0 = s_prefix[1];
        for (uint32_t b = threadIdx.x; b < nbr; b += kScanThreads) {
            const int32_t slot = buf[b];
            const uint32_t rank = rank0 + b, key = base + lkey[b];
            uint4 m[4];
            load_bits(occ, slot, m);
            BrickRec* r = brec + rank;
            uint32_t run = 0;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                reinterpret_cast<uint4*>(r->mask)[q] = m[q];
                const uint32_t p0 = run, p1 = p0 + __popc(m[q].x), p2 = p1 + __popc(m[q].y), p3 = p2 + __popc(m[q].z);
                run = p3 + __popc(m[q].w);
                reinterpret_cast<uint2*>(r->pre)[q] = make_uint2(p0 | (p1 << 16), p2 | (p3 << 16));
            }
            *reinterpret_cast<uint4*>(&r->base) = make_uint4(vox0 + lvox[b], run, key, (uint32_t)slot);
            sorted_slot[rank] = slot;
            sorted_key[rank] = (int32_t)key;
            rank_table[key] = (int32_t)rank;
        }
    } else if (tile == 0 && threadIdx.x == 0) {  // an empty table
        clear[0] = 0u;
        clear[1] = 0u;
    }
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(state + 1, 1u) == gridDim.x - 1) {  // the last CTA: reset for the next launch
            state[0] = 0;
            state[1] = 0;
            state[2] = epoch + 1;
            __threadfence();
        }
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
