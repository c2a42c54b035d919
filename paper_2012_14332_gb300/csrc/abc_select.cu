// abc_select.cu -- the k-th smallest of many distances, and the samples at or
// below a distance (paper Sec. 2.2: accept when the distance is at most eps;
// eps chosen as a distance quantile). A distance's bit pattern is its key: the
// patterns of non-negative doubles order like the values.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cuda_runtime.h>

#include "abc_kernels.h"

namespace abcgb {

namespace {

// ---------------------------------------------------------------------------
// The k-th smallest by a bracket from a sample: one pass over the distances.
//
//   pivot    ranks a stratified sample of kPivotSample keys and takes two of
//            them, lo and hi, that the wanted key lies between except with a
//            probability of about 1e-9 (six standard deviations of the sample
//            rank, and eight ranks more);
//   gather   the one pass over all keys: counts those below lo, collects those
//            in [lo, hi] (the candidates) and leaves the rank among them;
//   bin      histograms the candidates in kBins equal bins between the least
//            and the greatest and takes the bin that holds the rank, then
//   finish   collects that bin's keys, a few of them, and selects among them.
// The last block of each step to finish (a ticket, after a memory fence) takes
// the step's decision, and up to kFinish candidates it finishes at once. The
// answer is exact whatever the sample was: a rank outside the bracket, more
// candidates than the buffer holds, a bin that stays too full or counts that do
// not add up leave st->resolved at 0, and the caller runs the radix select.
//
// HBM-bound: the pass is the one read of the distances. The radix select read
// them eight times, its first digits (mostly the exponent, the same few values)
// adding to a few shared-memory counters one after another. At
// 20,000,003 distances and the 1e-4 quantile 430 -> 93 us per call (on the
// device 406 -> 65 us: sample 10, pass 34 at 4.8 TB/s, bins 11, finish 10); at
// the 0.5 quantile 436 -> 140 us; 65,536 distances 70 -> 49 us per call.
// ---------------------------------------------------------------------------
constexpr uint64_t kInfKey = 0x7FF0000000000000ull;
constexpr int kThreads = 256;
constexpr int kPivotLanes = 16;                      // threads that rank one sample key
constexpr int kPivotBlocks = kPivotSample / (kThreads / kPivotLanes);
constexpr int kPerThread = 8;                        // keys a thread loads at once
constexpr int kTile = kThreads * kPerThread;
constexpr int kBins = 2048;
constexpr int kFinish = 4096;                        // keys one block finishes with, in shared memory
static_assert(kFinish >= 2 * kTile, "a tile's candidates fit beside a tile's worth not yet written out");

// position of sample i: one per stratum of n / kPivotSample keys, at an offset
// scrambled from i (a regular grid would alias with ordered inputs)
__device__ __forceinline__ uint64_t pivot_position(uint32_t i, uint64_t n)
{
    const uint64_t begin = i * n / kPivotSample, end = (i + 1ull) * n / kPivotSample;
    const uint32_t h = (i + 1) * 0x9E3779B9u;
    return begin + (uint64_t)(h ^ (h >> 15)) % (end - begin);
}

__global__ void __launch_bounds__(kThreads) pivot_kernel(const double* __restrict__ dist, uint64_t n, uint64_t k,
                                                         int32_t r_lo, int32_t r_hi, SelectState* __restrict__ st)
{
    __shared__ __align__(16) uint64_t s[kPivotSample];
    griddep_wait();      // the distances and the zeroed state are complete
    griddep_release();
    const bool all = n <= kPivotSample;
    for (uint32_t i = threadIdx.x; i < kPivotSample; i += kThreads)
        s[i] = all ? (i < n ? (uint64_t)__double_as_longlong(dist[i]) : ~0ull)
                   : (uint64_t)__double_as_longlong(dist[pivot_position(i, n)]);
    __syncthreads();
    const uint32_t q = (blockIdx.x * kThreads + threadIdx.x) / kPivotLanes, sub = threadIdx.x % kPivotLanes;
    const uint64_t key = s[q];
    int32_t rank = 0;    // keys before this one, ties in sample order
#pragma unroll 8
    for (uint32_t j = 2 * sub; j < kPivotSample; j += 2 * kPivotLanes) {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(&s[j]);
        rank += (v.x < key || (v.x == key && j < q)) + (v.y < key || (v.y == key && j + 1 < q));
    }
#pragma unroll
    for (int off = kPivotLanes / 2; off > 0; off >>= 1) rank += __shfl_xor_sync(0xFFFFFFFFu, rank, off);
    if (sub) return;
    if (all) {
        if (q < n) {
            if (key > kInfKey) atomicAdd(&st->bad, 1ull);
            if ((uint64_t)rank + 1 == k) {
                st->prefix = key;
                st->resolved = 1;
            }
        }
        return;
    }
    if (rank == r_lo) st->lo = key;                  // below rank 0: lo stays 0
    if (rank == r_hi) st->hi = key;
    if (q == 0 && r_hi >= kPivotSample) st->hi = ~0ull;
}

// Inclusive scan of v over the block's threads.
__device__ __forceinline__ uint32_t block_scan(uint32_t v)
{
    __shared__ uint32_t warp_sum[kThreads / 32];
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t u = __shfl_up_sync(0xFFFFFFFFu, v, off);
        if (lane >= (uint32_t)off) v += u;
    }
    if (lane == 31) warp_sum[warp] = v;
    __syncthreads();
#pragma unroll
    for (uint32_t w = 0; w < kThreads / 32; ++w)
        if (w < warp) v += warp_sum[w];
    __syncthreads();
    return v;
}

// The rank-th smallest (1-based) of c keys in shared memory, all in [lo, hi]:
// the range is cut into up to 1024 equal bins and the bin that holds the rank
// becomes the range, until a warp can rank the keys left in it or it is one
// value (64 bits of range lose ten each time). False, and no key, unless each
// range holds as many keys as counted for it and the rank among them: a caller
// then leaves its search unresolved. Called by the whole block, with one answer;
// bins (1024) is shared scratch.
__device__ bool block_select(const uint64_t* keys, uint32_t c, uint64_t lo, uint64_t hi, uint64_t rank, uint32_t* bins,
                             uint64_t* key_out)
{
    __shared__ uint32_t pick_bin, pick_below, pick_count, n_short;
    __shared__ uint64_t short_list[32];
    if (rank < 1 || rank > c || lo > hi) return false;
    uint32_t r = (uint32_t)rank, left = c;
    for (int cut = 0; left > 32; ++cut) {
        if (cut == 7) return false;
        const uint64_t span = hi - lo;
        const int sh = span < 1024 ? 0 : 54 - __clzll((long long)span);   // span >> sh < 1024
        reinterpret_cast<uint4*>(bins)[threadIdx.x] = make_uint4(0, 0, 0, 0);
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < c; i += kThreads)
            if (keys[i] >= lo && keys[i] <= hi) atomicAdd(&bins[(keys[i] - lo) >> sh], 1u);
        __syncthreads();
        const uint4 b4 = reinterpret_cast<const uint4*>(bins)[threadIdx.x];
        const uint32_t sum = b4.x + b4.y + b4.z + b4.w, incl = block_scan(sum);
        uint32_t below = incl - sum;
        if (below < r && r <= incl) {
            const uint32_t h[4] = {b4.x, b4.y, b4.z, b4.w};
            int q = 0;
            while (q < 3 && below + h[q] < r) below += h[q++];
            pick_bin = 4 * threadIdx.x + q;
            pick_below = below;
            pick_count = h[q];
        }
        // with every key of the range counted, r <= left lies in one thread's bins
        if (!__syncthreads_and(threadIdx.x != kThreads - 1 || incl == left)) return false;
        lo += (uint64_t)pick_bin << sh;
        if (sh == 0) {
            *key_out = lo;
            return true;
        }
        hi = lo + ((1ull << sh) - 1);
        r -= pick_below;
        left = pick_count;
        __syncthreads();
    }
    if (threadIdx.x == 0) n_short = 0;
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < c; i += kThreads)
        if (keys[i] >= lo && keys[i] <= hi) {
            const uint32_t at = atomicAdd(&n_short, 1u);
            if (at < 32) short_list[at] = keys[i];
        }
    __syncthreads();
    if (n_short != left) return false;
    // every warp alike: lane's key, and how many of the others come before it
    const uint32_t lane = threadIdx.x & 31u;
    const uint64_t key = lane < left ? short_list[lane] : ~0ull;
    uint32_t before = 0;
    for (uint32_t j = 0; j < left; ++j) {
        const uint64_t v = short_list[j];
        before += v < key || (v == key && j < lane);
    }
    const uint32_t at = __ballot_sync(0xFFFFFFFFu, lane < left && before + 1 == r);
    if (at) *key_out = short_list[__ffs(at) - 1];
    return at != 0;
}

// Whether this block is the last of the grid to reach the ticket (its memory
// operations before it are visible to the last block). Block-uniform.
__device__ __forceinline__ bool last_block(unsigned int* ticket)
{
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    __threadfence();
    return last;
}

// kPerThread keys of the tile that starts at `base`: pairs 2 tid, 2 tid + 1 of
// each quarter, in 16-byte loads issued together where the array is 16-byte
// aligned and the tile whole; ~0 past n.
__device__ __forceinline__ void load_tile(const double* __restrict__ dist, uint64_t n, uint64_t base, bool vec,
                                          uint64_t (&key)[kPerThread])
{
    if (vec && base + kTile <= n) {
        const ulonglong2* p = reinterpret_cast<const ulonglong2*>(dist + base) + threadIdx.x;
#pragma unroll
        for (int q = 0; q < kPerThread / 2; ++q) {
            const ulonglong2 v = __ldg(p + q * kThreads);
            key[2 * q] = v.x;
            key[2 * q + 1] = v.y;
        }
        return;
    }
#pragma unroll
    for (int e = 0; e < kPerThread; ++e) {
        const uint64_t j = base + 2 * ((uint64_t)(e / 2) * kThreads + threadIdx.x) + (e & 1);
        key[e] = j < n ? (uint64_t)__double_as_longlong(__ldg(dist + j)) : ~0ull;
    }
}

__device__ __forceinline__ bool is_vec(const double* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

__global__ void __launch_bounds__(kThreads) gather_kernel(const double* __restrict__ dist, uint64_t n, uint64_t k,
                                                          SelectState* __restrict__ st, uint64_t* __restrict__ cand,
                                                          uint64_t cap)
{
    __shared__ __align__(16) uint64_t buf[kFinish];
    __shared__ __align__(16) uint32_t bins[1024];
    __shared__ uint32_t fill;
    __shared__ unsigned long long slot0, least, most;   // of the block's candidates
    if (threadIdx.x == 0) {
        fill = 0;
        least = ~0ull;
        most = 0;
    }
    const bool vec = is_vec(dist);
    griddep_wait();
    griddep_release();
    const uint64_t lo = __ldcg(&st->lo), hi = __ldcg(&st->hi);
    unsigned long long below = 0, bad = 0;
    const uint64_t step = (uint64_t)gridDim.x * kTile;
    uint64_t next[kPerThread];
    load_tile(dist, n, (uint64_t)blockIdx.x * kTile, vec, next);
    __syncthreads();
    for (uint64_t base = (uint64_t)blockIdx.x * kTile; base < n; base += step) {
        uint64_t key[kPerThread];
#pragma unroll
        for (int q = 0; q < kPerThread; ++q) key[q] = next[q];
        const bool more = base + step < n;
        if (more) load_tile(dist, n, base + step, vec, next);   // in flight while this tile is sorted out
        uint32_t mine = 0;
#pragma unroll
        for (int q = 0; q < kPerThread; ++q) {
            below += key[q] < lo;
            // ~0 is also the padding past n: told apart by the key's position
            if (key[q] > kInfKey) {
                const uint64_t j = base + 2 * ((uint64_t)(q / 2) * kThreads + threadIdx.x) + (q & 1);
                if (j < n) ++bad;
                key[q] = ~0ull;
            } else if (key[q] >= lo && key[q] <= hi) {
                ++mine;
            } else {
                key[q] = ~0ull;
            }
        }
        if (mine) {
            uint32_t at = atomicAdd(&fill, mine);
            unsigned long long a = ~0ull, b = 0;
#pragma unroll
            for (int q = 0; q < kPerThread; ++q)
                if (key[q] != ~0ull) {
                    buf[at++] = key[q];
                    a = min(a, (unsigned long long)key[q]);
                    b = max(b, (unsigned long long)key[q]);
                }
            if (a < least) atomicMin(&least, a);   // a stale read only costs the atomic
            if (b > most) atomicMax(&most, b);
        }
        __syncthreads();
        const uint32_t f = fill;
        __syncthreads();                             // read by all before the next tile adds to it
        if (f > kFinish - kTile || !more) {
            if (threadIdx.x == 0) slot0 = f ? atomicAdd(&st->count, (unsigned long long)f) : 0ull;
            __syncthreads();
            for (uint32_t i = threadIdx.x; i < f; i += kThreads)
                if (slot0 + i < cap) cand[slot0 + i] = buf[i];
            if (threadIdx.x == 0) fill = 0;
            __syncthreads();
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        below += __shfl_xor_sync(0xFFFFFFFFu, below, off);
        bad += __shfl_xor_sync(0xFFFFFFFFu, bad, off);
    }
    if ((threadIdx.x & 31) == 0) {
        if (below) atomicAdd(&st->below, below);
        if (bad) atomicAdd(&st->bad, bad);
    }
    // a block with candidates has a least one, perhaps of key 0 (a distance of
    // exactly 0), which is never ~0
    if (threadIdx.x == 0 && least != ~0ull) {
        atomicMax(&st->not_least, ~least);
        atomicMax(&st->most, most);
    }
    if (!last_block(&st->ticket[0])) return;
    const uint64_t b = __ldcg(&st->below), c = __ldcg(&st->count);
    if (k <= b || k - b > c) return;                 // outside the bracket: unresolved
    if (lo == hi) {
        if (threadIdx.x == 0) {
            st->prefix = lo;
            st->resolved = 1;
        }
    } else if (c <= cap && c <= kFinish) {
        for (uint32_t i = threadIdx.x; i < c; i += kThreads) buf[i] = __ldcg(&cand[i]);
        __syncthreads();
        uint64_t key;
        if (block_select(buf, (uint32_t)c, ~__ldcg(&st->not_least), __ldcg(&st->most), k - b, bins, &key) &&
            threadIdx.x == 0) {
            st->prefix = key;
            st->resolved = 1;
        }
    } else if (c <= cap && threadIdx.x == 0) {
        st->rank = k - b;
        st->stage = 1;
    }
}

__global__ void __launch_bounds__(kThreads) bin_kernel(SelectState* __restrict__ st, const uint64_t* __restrict__ cand,
                                                       uint32_t* __restrict__ bins)
{
    __shared__ uint32_t h[kBins];
    for (int b = threadIdx.x; b < kBins; b += kThreads) h[b] = 0;
    griddep_wait();
    griddep_release();
    __syncthreads();
    if (__ldcg(&st->stage) != 1) return;
    // between the least and the greatest candidate: the bracket's ends may be
    // far outside (0 below the sample's first key)
    const uint64_t lo = ~__ldcg(&st->not_least), span = __ldcg(&st->most) - lo;
    const uint64_t c = __ldcg(&st->count);
    const int sh = span < kBins ? 0 : 53 - __clzll((long long)span);   // span >> sh < kBins
#pragma unroll 4
    for (uint64_t i = (uint64_t)blockIdx.x * kThreads + threadIdx.x; i < c; i += (uint64_t)gridDim.x * kThreads) {
        const uint64_t bin = (__ldcg(&cand[i]) - lo) >> sh;
        if (bin < kBins) atomicAdd(&h[bin], 1u);
    }
    __syncthreads();
    for (int b = threadIdx.x; b < kBins; b += kThreads)
        if (h[b]) atomicAdd(&bins[b], h[b]);
    if (!last_block(&st->ticket[1])) return;
    uint32_t own[kBins / kThreads], sum = 0;
#pragma unroll
    for (int q = 0; q < kBins / kThreads; ++q) {
        own[q] = __ldcg(&bins[threadIdx.x * (kBins / kThreads) + q]);
        sum += own[q];
    }
    const uint32_t incl = block_scan(sum);
    // a candidate outside [least, greatest] was not counted: unresolved
    if (!__syncthreads_and(threadIdx.x != kThreads - 1 || incl == c)) return;
    uint64_t before = incl - sum;
    const uint64_t rank = __ldcg(&st->rank);
    if (!(before < rank && rank <= before + sum)) return;
    int q = 0;
    while (q < kBins / kThreads - 1 && before + own[q] < rank) before += own[q++];
    const uint64_t first = lo + ((uint64_t)(threadIdx.x * (kBins / kThreads) + q) << sh);
    st->rank = rank - before;
    st->lo = first;
    st->hi = first + ((1ull << sh) - 1);
    if (sh == 0) {
        st->prefix = first;
        st->resolved = 1;
        st->stage = 0;
    } else {
        st->stage = own[q] <= kFinish ? 2 : 0;       // a fuller bin: unresolved
    }
}

__global__ void __launch_bounds__(kThreads) finish_kernel(SelectState* __restrict__ st, const uint64_t* __restrict__ cand,
                                                          uint64_t* __restrict__ few)
{
    __shared__ __align__(16) uint64_t buf[kFinish];
    __shared__ __align__(16) uint32_t bins[1024];
    griddep_wait();
    griddep_release();
    if (__ldcg(&st->stage) != 2) return;
    const uint64_t lo = __ldcg(&st->lo), hi = __ldcg(&st->hi), c = __ldcg(&st->count);
#pragma unroll 4
    for (uint64_t i = (uint64_t)blockIdx.x * kThreads + threadIdx.x; i < c; i += (uint64_t)gridDim.x * kThreads) {
        const uint64_t key = __ldcg(&cand[i]);
        if (key >= lo && key <= hi) {
            const uint32_t at = atomicAdd(&st->n_few, 1u);
            if (at < kFinish) few[at] = key;
        }
    }
    if (!last_block(&st->ticket[2])) return;
    const uint32_t m = __ldcg(&st->n_few);
    if (m > kFinish) return;
    for (uint32_t i = threadIdx.x; i < m; i += kThreads) buf[i] = __ldcg(&few[i]);
    __syncthreads();
    uint64_t key;
    if (block_select(buf, m, lo, hi, __ldcg(&st->rank), bins, &key) && threadIdx.x == 0) {
        st->prefix = key;
        st->resolved = 1;
    }
}

// ---------------------------------------------------------------------------
// Radix select of the k-th smallest distance, for the inputs the bracket above
// leaves unresolved: eight passes over the keys, one 8-bit digit per pass from
// the top, one launch per pass. A pass histograms that
// digit among the keys whose higher digits equal the prefix chosen so far;
// the last block of the pass to finish (a ticket counter, after a memory
// fence) picks the digit holding the wanted rank and updates the state in
// device memory, so the passes run back to back with no host round trip. On
// the first pass (mask == 0) hist[256] counts the keys above +infinity's
// pattern: NaN and anything with the sign bit set (negative values and -0),
// which would not order like their values. hist[257] is the ticket counter.
// ---------------------------------------------------------------------------

// One warp: the digit of this pass is the first whose running count reaches
// the rank (k on the first pass); the rank becomes the rank within that
// digit's keys. Lane j holds bins 8j .. 8j + 7 in h (their sum in sum): a
// warp scan of the lanes' sums finds the lane, then that lane walks its eight
// bins and updates the state.
__device__ __forceinline__ void select_digit(const unsigned long long (&h)[8], unsigned long long sum,
                                             SelectState* st, int shift, uint64_t rank)
{
    const int lane = threadIdx.x & 31;
    // inclusive scan of the lanes' sums
    unsigned long long incl = sum;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const unsigned long long v = __shfl_up_sync(0xFFFFFFFFu, incl, off);
        if (lane >= off) incl += v;
    }
    const uint32_t reach = __ballot_sync(0xFFFFFFFFu, incl >= rank);
    // the first lane whose running count reaches the rank (the last lane if
    // none does, which only invalid input allows)
    const int owner = reach ? __ffs(reach) - 1 : 31;
    if (lane == owner) {
        uint64_t below = incl - sum;
        int i = 0;
        for (; i < 7; ++i) {
            if (below + h[i] >= rank) break;
            below += h[i];
        }
        st->rank = rank - below;
        st->prefix |= (uint64_t)(8 * lane + i) << shift;
        st->mask |= (uint64_t)0xFF << shift;
    }
}

__global__ void __launch_bounds__(kThreads) digit_pass_kernel(const double* __restrict__ dist, uint64_t n,
                                                                   SelectState* __restrict__ st, int shift,
                                                                   uint64_t k, unsigned long long* __restrict__ hist)
{
    __shared__ unsigned int h[257];
    __shared__ bool last;
    for (int b = threadIdx.x; b < 257; b += blockDim.x) h[b] = 0;
    // the previous pass (or the kernel that wrote the distances) completes
    // before the state and the keys are read; the next pass may launch now
    griddep_wait();
    griddep_release();
    __syncthreads();
    const uint64_t prefix = st->prefix, prefix_mask = st->mask;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    const bool first = prefix_mask == 0;
    for (uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += stride) {
        const uint64_t key = (uint64_t)__double_as_longlong(dist[j]);
        if ((key & prefix_mask) == prefix) atomicAdd(&h[(key >> shift) & 0xFFu], 1u);
        if (first && key > 0x7FF0000000000000ull) atomicAdd(&h[256], 1u);
    }
    __syncthreads();
    for (int b = threadIdx.x; b < 257; b += blockDim.x)
        if (h[b]) atomicAdd(&hist[b], (unsigned long long)h[b]);
    // the block's counts are in before its ticket is taken
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&hist[257], 1ull) == gridDim.x - 1;
    __syncthreads();
    if (!last || threadIdx.x >= 32) return;
    // the last block: every block's counts are in; read them past L1
    __threadfence();
    const int lane = threadIdx.x;
    unsigned long long hb[8], sum = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        hb[i] = __ldcg(&hist[8 * lane + i]);
        sum += hb[i];
    }
    const uint64_t rank = first ? k : st->rank;
    if (first && lane == 0) st->bad = __ldcg(&hist[256]);
    __syncwarp();
    // the histogram and the ticket counter zeroed for the next pass
#pragma unroll
    for (int i = 0; i < 8; ++i) hist[8 * lane + i] = 0;
    if (lane == 0) {
        hist[256] = 0;
        hist[257] = 0;
    }
    select_digit(hb, sum, st, shift, rank);
}

// ---------------------------------------------------------------------------
// Samples accepted at eps from distances already computed (Sec. 2.2: accept
// when the distance is at most eps): sample j is accepted iff dist[j] <= eps.
// A warp takes 256 consecutive samples at a time, eight a lane in four 16-byte
// loads issued a chunk ahead, reserves the slots of its accepts with one atomicAdd
// and writes index, distance and theta. Every accept is counted; only slots
// below capacity are written. HBM-bound while accepts are few (20,000,003
// distances, 1e-4 of them: 44 us, 3.6 TB/s, as with one load a lane and an
// atomic per 32 samples); with many, the atomics and writes: 0.1 of 4e7
// samples 1068 -> 294 us per call, half of 2e7 686 -> 439 us.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kThreads) select_below_kernel(const __grid_constant__ SelectArgs a)
{
    const uint32_t lane = threadIdx.x & 31u;
    const uint64_t step = (uint64_t)gridDim.x * (kThreads / 32) * 256;
    const bool vec = is_vec(a.dist);
    griddep_wait();   // the distances and the selected key are complete
    const double eps = a.eps_key ? __longlong_as_double((long long)a.eps_key->prefix) : a.eps;
    const auto load = [&](uint64_t base, double (&d)[8]) {
        if (vec && base + 256 <= a.n) {
            const double2* p = reinterpret_cast<const double2*>(a.dist + base) + lane;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const double2 v = __ldg(p + 32 * q);
                d[2 * q] = v.x;
                d[2 * q + 1] = v.y;
            }
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const uint64_t j = base + 64 * (e / 2) + 2 * lane + (e & 1);
                d[e] = j < a.n ? a.dist[j] : __longlong_as_double(-1ll);   // NaN: never accepted
            }
        }
    };
    double next[8];
    uint64_t base = ((uint64_t)blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5)) * 256;
    if (base < a.n) load(base, next);
    for (; base < a.n; base += step) {
        double d[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) d[e] = next[e];
        if (base + step < a.n) load(base + step, next);   // in flight while this chunk is sorted out
        uint32_t take = 0;   // bit e: the lane's e-th sample, base + 64 (e / 2) + 2 lane + e % 2
#pragma unroll
        for (int e = 0; e < 8; ++e) take |= d[e] <= eps ? 1u << e : 0u;
        if (!__any_sync(0xFFFFFFFFu, take)) continue;
        const uint32_t mine = __popc(take);
        uint32_t incl = mine;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, incl, off);
            if (lane >= (uint32_t)off) incl += v;
        }
        unsigned long long slot0 = 0;
        if (lane == 31) slot0 = atomicAdd(a.count, (unsigned long long)incl);
        uint64_t slot = __shfl_sync(0xFFFFFFFFu, slot0, 31) + incl - mine;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            if (!(take >> e & 1u)) continue;
            if (slot < a.capacity) {
                const uint64_t j = base + 64 * (e / 2) + 2 * lane + (e & 1);
                a.idx_out[slot] = a.first_index + j;
                a.dist_out[slot] = d[e];
                if (a.theta_out) {
                    const float4* src = reinterpret_cast<const float4*>(a.theta + 8 * j);
                    float4* to = reinterpret_cast<float4*>(a.theta_out + 8 * slot);
                    to[0] = src[0];
                    to[1] = src[1];
                }
            }
            ++slot;
        }
    }
}

// blocks for n items at `per` a block, at most `per_sm` per SM of the device
cudaError_t blocks_of(uint64_t n, uint64_t per, int per_sm, int* blocks)
{
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const uint64_t want = std::max<uint64_t>(1, (n + per - 1) / per);
    *blocks = (int)std::min<uint64_t>(want, (uint64_t)sms * per_sm);
    return e;
}

}  // namespace

cudaError_t launch_select_below(const SelectArgs& a, cudaStream_t s)
{
    int grid = 0;
    cudaError_t e = blocks_of(a.n, kTile, 4, &grid);
    if (e != cudaSuccess) return e;
    e = launch_overlapped(select_below_kernel, dim3(grid), dim3(kThreads), 0, s, a);
    return e != cudaSuccess ? e : cudaGetLastError();
}

// The ranks [r_lo, r_hi] of the sample that the wanted key lies between.
static void bracket(uint64_t n, uint64_t k, int32_t* r_lo, int32_t* r_hi)
{
    const double q = ((double)k - 0.5) / (double)n, c = q * kPivotSample;
    const double w = 6.0 * std::sqrt(c * (1.0 - q)) + 8.0;
    *r_lo = (int32_t)std::max(-1.0, std::floor(c - w));
    *r_hi = (int32_t)std::min((double)kPivotSample, std::ceil(c + w));
}

uint64_t select_candidates(uint64_t n, uint64_t k)
{
    if (n <= kPivotSample) return 0;
    int32_t r_lo = 0, r_hi = 0;
    bracket(n, k, &r_lo, &r_hi);
    const double share = (double)(r_hi - r_lo + 1) / kPivotSample;
    return std::min<uint64_t>(n, (uint64_t)(2.0 * share * (double)n) + kFinish);
}

cudaError_t launch_kth_bracket(const double* dist, uint64_t n, uint64_t k, SelectWork* w, uint64_t* cand, uint64_t cap,
                               cudaStream_t s)
{
    int32_t r_lo = 0, r_hi = 0;
    bracket(n, k, &r_lo, &r_hi);
    cudaError_t e = launch_overlapped(pivot_kernel, dim3(kPivotBlocks), dim3(kThreads), 0, s, dist, n, k, r_lo, r_hi,
                                      &w->st);
    if (e != cudaSuccess || n <= kPivotSample) return e != cudaSuccess ? e : cudaGetLastError();
    int grid = 0;
    if ((e = blocks_of(n, kTile, 4, &grid)) != cudaSuccess) return e;
    e = launch_overlapped(gather_kernel, dim3(grid), dim3(kThreads), 0, s, dist, n, k, &w->st, cand, cap);
    // half of the buffer is the expected number of candidates: few enough are
    // finished by the gathering kernel's last block
    if (e == cudaSuccess && cap / 2 > kFinish) {
        if ((e = blocks_of(cap / 2, kTile, 1, &grid)) != cudaSuccess) return e;
        e = launch_overlapped(bin_kernel, dim3(grid), dim3(kThreads), 0, s, &w->st, cand, w->bins);
        if (e == cudaSuccess)
            e = launch_overlapped(finish_kernel, dim3(grid), dim3(kThreads), 0, s, &w->st, cand, w->few);
    }
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_kth_radix(const double* dist, uint64_t n, uint64_t k, SelectWork* w, cudaStream_t s)
{
    int grid = 0;
    cudaError_t e = cudaMemsetAsync(w, 0, kSelectZeroBytes, s);
    if (e == cudaSuccess) e = blocks_of(n, kThreads, 6, &grid);
    for (int shift = 56; shift >= 0 && e == cudaSuccess; shift -= 8)
        e = launch_overlapped(digit_pass_kernel, dim3(grid), dim3(kThreads), 0, s, dist, n, &w->st, shift, k, w->hist);
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace abcgb
