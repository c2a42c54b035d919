// abc_staged.cu -- the same per-sample method (paper Sec. 2.1) for calls too
// small to fill the chip with a thread per sample, and the quantile bands of
// trajectories (Sec. 5).
//
// A thread per sample runs T days of a dependent chain, random words included,
// on a chip that is mostly idle when there are a few thousand samples. Only the
// model day depends on the day before; the normals (Philox and Box-Muller, more
// than half of a day's instructions) depend on the sample's index alone. So a
// block here has 32 samples: P warps draw the normals of a stage of P day pairs
// ahead, one pair each, into shared memory, and one warp walks the model
// through them. The arithmetic of a sample is that of a thread
// per sample, instruction for instruction, and so are the results.
// Latency-bound: the model days' chain. On the device, fast arithmetic over 120
// days: 100 trajectories 39 -> 21 us, 8192 102 -> 23 us; exact arithmetic over
// 49 days with early rejection: 10,000 samples 75 -> 47 us.
#include <algorithm>
#include <cstdint>
#include <cuda_runtime.h>

#include "abc_kernels.h"
#include "abc_launch.h"
#include "abc_model.cuh"

namespace abcgb {

namespace {

// Warps that draw: two keep up with a walk that only sums a distance, and leave
// room for more blocks; three share the writing of trajectories (1000 of 90
// days, fast: 12.5 us, 18.6 us with two).
constexpr int kSumProducers = 2;
constexpr int kWriteProducers = 3;
constexpr int staged_threads(int producers) { return 32 * (producers + 1); }

template <int P>
struct Stage {
    float z[P][10][32];   // normals of one day pair per producer: [pair][draw][lane]
};

// Runs the block's 32 samples (lane's sample index i, walked by the last warp
// from state x) through all T days. The sink gets every day's state from the
// walking warp (day), a call after each day pair (pair; false ends the block
// early once no lane wants to go on, if it can stop at all), and a call from
// the producers after each stage (drain, for the stage before).
template <int MODE, int P, typename Sink>
__device__ __forceinline__ void staged_days(const ModelParams& p, uint64_t i, const Theta& t, State x,
                                            Stage<P> (&zs)[2], Sink& sink)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int32_t T = p.T;
    const uint32_t n_pairs = (uint32_t)(T + 1) >> 1, stages = (n_pairs + P - 1) / P;
    const bool walks = warp == P;
    const auto produce = [&](uint32_t st) {
        const uint32_t k = st * P + warp + 1;
        if (k > n_pairs) return;
        float z[10];
        day_pair_normals<MODE>(p, i, k, z);
#pragma unroll
        for (int e = 0; e < 10; ++e) zs[st & 1].z[warp][e][lane] = z[e];
    };
    if (!walks) produce(0);
    __syncthreads();
    for (uint32_t st = 0; st < stages; ++st) {
        bool go = false;
        if (!walks) {
            if (st + 1 < stages) produce(st + 1);
            if (st > 0) sink.drain(st - 1, T);
        } else {
#pragma unroll
            for (int q = 0; q < P; ++q) {
                const uint32_t k = st * P + q + 1;
                if (k > n_pairs) continue;
                float z[10];
#pragma unroll
                for (int e = 0; e < 10; ++e) z[e] = zs[st & 1].z[q][e][lane];
                const int32_t d1 = (int32_t)(2 * k - 1);
                model_day<MODE>(x, t, p.inv_p, z);
                sink.day(d1, 2 * q, x);
                if (d1 < T) {
                    model_day<MODE>(x, t, p.inv_p, z + 5);
                    sink.day(d1 + 1, 2 * q + 1, x);
                }
                go = sink.pair(d1, T, x);
            }
        }
        if (Sink::kStops) {
            if (!__syncthreads_or(go)) return;
        } else {
            __syncthreads();
        }
    }
    if (!walks) sink.drain(stages - 1, T);
}

__device__ __forceinline__ void stage_series(int4* obs_s, const int4* __restrict__ obs, int32_t T)
{
    for (int32_t d = threadIdx.x; d <= T; d += blockDim.x) obs_s[d] = obs[d];
    // read after staged_days' first barrier
}

// distance^2 over all days
struct DistanceSink {
    static constexpr bool kStops = false;
    const int4* obs;
    uint64_t acc = 0;
    __device__ __forceinline__ void day(int32_t d, int, const State& x) { acc = add_day_sq(acc, x, obs[d]); }
    __device__ __forceinline__ bool pair(int32_t, int32_t, const State&) { return true; }
    __device__ __forceinline__ void drain(uint32_t, int32_t) {}
};

template <int MODE>
__global__ void __launch_bounds__(staged_threads(kSumProducers)) staged_distance_kernel(const __grid_constant__ ModelParams p,
                                                                         const __grid_constant__ DistanceArgs a)
{
    extern __shared__ int4 obs_s[];
    __shared__ Stage<kSumProducers> zs[2];
    stage_series(obs_s, a.obs, p.T);
    const uint64_t j = (uint64_t)blockIdx.x * 32 + (threadIdx.x & 31), i = a.first_index + j;
    const bool walks = threadIdx.x >= 32 * kSumProducers;
    float th[8];
    Theta t{};
    State x{};
    if (walks) {
        prior_draw(p, i, th);
        t = make_theta<MODE>(th, p.inv_p);
        x = init_state(t, p.A0, p.R0, p.D0, p.room0);
    }
    DistanceSink sink{obs_s};
    staged_days<MODE, kSumProducers>(p, i, t, x, zs, sink);
    if (!walks || j >= a.n_samples) return;
    a.dist_out[j] = __dsqrt_rn(__ull2double_rn(sink.acc));
    if (a.theta_out) {
        float4* to = reinterpret_cast<float4*>(a.theta_out + 8 * j);
        to[0] = make_float4(th[0], th[1], th[2], th[3]);
        to[1] = make_float4(th[4], th[5], th[6], th[7]);
    }
}

// Rejection with early stopping, as abc_reject_kernel: a lane's sample ends
// when its sum passes the threshold, when its infected have died out too far
// from the series, or after T days; the block ends with its last sample.
template <bool BELOW62>
struct RejectSink {
    static constexpr bool kStops = true;
    const int4* obs;
    uint64_t acc_max, acc;
    uint32_t days;
    int32_t v_bits, m_bits;
    bool active, accept;
    __device__ __forceinline__ void day(int32_t d, int which, const State& x)
    {
        const int4 o = obs[d];
        ((which & 1) ? m_bits : v_bits) = o.w;
        const uint64_t next = BELOW62 ? add_day_sq_below62(acc, x, o) : add_day_sq(acc, x, o);
        acc = active ? next : acc;
    }
    __device__ __forceinline__ bool pair(int32_t d1, int32_t T, const State& x)
    {
        const bool last = d1 + 1 >= T;
        bool over = acc > acc_max;
        if (active && x.I == 0 && !over && !last && (BELOW62 || acc_max < kAccCap))
            over = extinct_over(x, v_bits, m_bits, T - d1 - 1, acc, acc_max);
        if (active) {
            days = (uint32_t)min(d1 + 1, T);
            accept = !over && last;
            active = !(over || last);
        }
        return active;
    }
    __device__ __forceinline__ void drain(uint32_t, int32_t) {}
};

template <int MODE, bool BELOW62>
__global__ void __launch_bounds__(staged_threads(kSumProducers)) staged_reject_kernel(const __grid_constant__ ModelParams p,
                                                                       const __grid_constant__ RejectArgs a)
{
    extern __shared__ int4 obs_s[];
    __shared__ Stage<kSumProducers> zs[2];
    stage_series(obs_s, a.obs, p.T);
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t j = (uint64_t)blockIdx.x * 32 + lane, i = a.first_index + j;
    const bool walks = threadIdx.x >= 32 * kSumProducers;
    float th[8];
    Theta t{};
    State x{};
    if (walks) {
        prior_draw(p, i, th);
        t = make_theta<MODE>(th, p.inv_p);
        x = init_state(t, p.A0, p.R0, p.D0, p.room0);
    }
    // the claim counter stands at or above n_samples afterwards, as when chunks are claimed
    if (threadIdx.x == 0) atomicAdd(a.next, 32ull);
    RejectSink<BELOW62> sink{obs_s, a.acc_max, 0, 0, 0, 0, walks && j < a.n_samples, false};
    staged_days<MODE, kSumProducers>(p, i, t, x, zs, sink);
    if (!walks) return;
    const uint32_t mask = __ballot_sync(0xFFFFFFFFu, sink.accept);
    if (mask) {
        unsigned long long slot0 = 0;
        if (lane == 0) slot0 = atomicAdd(a.count, (unsigned long long)__popc(mask));
        slot0 = __shfl_sync(0xFFFFFFFFu, slot0, 0);
        const uint64_t slot = slot0 + __popc(mask & ((1u << lane) - 1u));
        if (sink.accept && slot < a.capacity) {
            a.idx_out[slot] = i;
            a.dist_out[slot] = __dsqrt_rn(__ull2double_rn(sink.acc));
            float4* to = reinterpret_cast<float4*>(a.theta_out + 8 * slot);
            to[0] = make_float4(th[0], th[1], th[2], th[3]);
            to[1] = make_float4(th[4], th[5], th[6], th[7]);
        }
    }
    unsigned long long days = sink.days;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) days += __shfl_down_sync(0xFFFFFFFFu, days, off);
    if (lane == 0 && a.sim_days) atomicAdd(a.sim_days, days);
}

// Whole trajectories [B][T + 1][6]: the walking warp leaves a stage's states in
// shared memory and the producers write them out during the next stage, a row's
// days as one run of 8-byte words (the rows are 24 (T + 1) bytes apart; a lane
// storing its own six values a day touched 32 sectors with every 4 bytes).
constexpr int kTileDays = 2 * kWriteProducers;   // a stage
struct TrajTile {
    int2 s[32][3 * kTileDays + 1];   // one row's days; the odd stride (in 8 bytes) spreads lanes over the banks
};

struct TrajSink {
    static constexpr bool kStops = false;
    TrajTile* tiles;    // [2]
    int32_t* out;       // the block's first row
    uint32_t rows;
    uint32_t stage;     // of the walking warp
    bool wide;          // rows 8-byte aligned
    __device__ __forceinline__ void day(int32_t, int which, const State& x)
    {
        int2* to = &tiles[stage & 1].s[threadIdx.x & 31][3 * which];
        to[0] = make_int2(x.S, x.I);
        to[1] = make_int2(x.A, x.R);
        to[2] = make_int2(x.D, x.Ru);
    }
    __device__ __forceinline__ bool pair(int32_t d1, int32_t, const State&)
    {
        stage = (uint32_t)(d1 + 1) / kTileDays;   // the next pair's stage
        return true;
    }
    __device__ __forceinline__ void drain(uint32_t st, int32_t T)
    {
        const int32_t d0 = (int32_t)st * kTileDays + 1, days = min(kTileDays, T - d0 + 1);
        if (days == kTileDays)
            copy<3 * kTileDays>(tiles[st & 1], 0, d0, T);
        else
            copy<0>(tiles[st & 1], 3 * (uint32_t)days, d0, T);
    }
    // the stage's first WORDS (0: n) words of every row, days d0 on
    template <uint32_t WORDS>
    __device__ __forceinline__ void copy(const TrajTile& tile, uint32_t n, int32_t d0, int32_t T)
    {
        const uint32_t words = WORDS ? WORDS : n;
        for (uint32_t u = threadIdx.x; u < rows * words; u += 32 * kWriteProducers) {
            const uint32_t r = u / words, c = u - r * words;
            const int2 v = tile.s[r][c];
            int32_t* to = out + (size_t)r * 6 * (T + 1) + 6 * (size_t)d0 + 2 * c;
            if (wide) {
                *reinterpret_cast<int2*>(to) = v;
            } else {
                to[0] = v.x;
                to[1] = v.y;
            }
        }
    }
};

__device__ __forceinline__ void load_theta(const float* __restrict__ src, float th[8])
{
    const float4* s4 = reinterpret_cast<const float4*>(src);
    const float4 l = s4[0], h = s4[1];
    th[0] = l.x; th[1] = l.y; th[2] = l.z; th[3] = l.w;
    th[4] = h.x; th[5] = h.y; th[6] = h.z; th[7] = h.w;
}

template <int MODE>
__global__ void __launch_bounds__(staged_threads(kWriteProducers)) staged_simulate_kernel(const __grid_constant__ ModelParams p,
                                                                         const __grid_constant__ SimulateArgs a)
{
    __shared__ Stage<kWriteProducers> zs[2];
    __shared__ TrajTile tiles[2];
    const uint64_t b0 = (uint64_t)blockIdx.x * 32;
    const uint32_t lane = threadIdx.x & 31, rows = (uint32_t)min(a.B - b0, (uint64_t)32);
    const uint64_t b = b0 + min(lane, rows - 1);   // lanes past the end repeat the last row, unwritten
    const uint64_t i = a.sample_index[b];
    int32_t* out = a.traj_out + (size_t)b0 * 6 * (size_t)(p.T + 1);
    Theta t{};
    State x{};
    if (threadIdx.x >= 32 * kWriteProducers) {
        float th[8];
        load_theta(a.theta + 8 * b, th);
        t = make_theta<MODE>(th, p.inv_p);
        x = init_state(t, p.A0, p.R0, p.D0, p.room0);
        if (lane < rows) {
            int32_t* o = out + (size_t)lane * 6 * (size_t)(p.T + 1);
            o[0] = x.S; o[1] = x.I; o[2] = x.A; o[3] = x.R; o[4] = x.D; o[5] = x.Ru;
        }
    }
    TrajSink sink{tiles, out, rows, 0, (reinterpret_cast<uintptr_t>(a.traj_out) & 7u) == 0};
    staged_days<MODE, kWriteProducers>(p, i, t, x, zs, sink);
}

// The observed compartments as columns [T + 1][3][stride], what the bands read.
struct ColumnSink {
    static constexpr bool kStops = false;
    int32_t* out;       // the lane's entry of day 0, compartment A; NULL past the last row
    size_t stride;
    __device__ __forceinline__ void day(int32_t d, int, const State& x)
    {
        if (!out) return;
        int32_t* to = out + 3 * (size_t)d * stride;
        to[0] = x.A;
        to[stride] = x.R;
        to[2 * stride] = x.D;
    }
    __device__ __forceinline__ bool pair(int32_t, int32_t, const State&) { return true; }
    __device__ __forceinline__ void drain(uint32_t, int32_t) {}
};

template <int MODE>
__global__ void __launch_bounds__(staged_threads(kWriteProducers)) staged_columns_kernel(const __grid_constant__ ModelParams p,
                                                                        const __grid_constant__ ColumnArgs a)
{
    __shared__ Stage<kWriteProducers> zs[2];
    griddep_release();   // the band kernel's blocks may come in and wait
    const uint64_t row = (uint64_t)blockIdx.x * 32 + (threadIdx.x & 31), b = min(row, a.B - 1);
    const uint64_t i = a.sample_index[b];
    Theta t{};
    State x{};
    ColumnSink sink{row < a.B ? a.out + row : nullptr, a.stride};
    if (threadIdx.x >= 32 * kWriteProducers) {
        float th[8];
        load_theta(a.theta + 8 * b, th);
        t = make_theta<MODE>(th, p.inv_p);
        x = init_state(t, p.A0, p.R0, p.D0, p.room0);
        sink.day(0, 0, x);
    }
    staged_days<MODE, kWriteProducers>(p, i, t, x, zs, sink);
}

// ---------------------------------------------------------------------------
// Quantile bands: one block per (day, compartment) column, order statistics
// floor(q (B - 1)) of its B counts. The counts are put in bins equally wide in
// the bits of their float values (so for narrow and for heavy-tailed columns
// alike) between the column's least and greatest, laid out bin by bin in
// shared memory, and each wanted rank is then found inside its bin by a warp
// bisecting the bin's values. A bitonic sort of the column took 91 barriers
// and 4 compare-exchanges a thread between them at B = 8192, and its columns
// were gathered 4 bytes from each trajectory row. 121 days: B = 8192 131 -> 20
// us, B = 100 12 -> 9 us.
// ---------------------------------------------------------------------------
template <int THREADS, int KEYS, int BINS>
__global__ void __launch_bounds__(THREADS) band_kernel(const __grid_constant__ BandArgs a)
{
    static_assert(BINS % THREADS == 0 || THREADS % BINS == 0, "whole bins a thread");
    __shared__ uint32_t v[THREADS * KEYS];
    __shared__ uint32_t start[BINS + 1];       // first position of each bin
    __shared__ uint32_t warp_sum[THREADS / 32];
    __shared__ uint32_t least_s, most_s;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t B = a.B;
    for (int b = threadIdx.x; b < BINS; b += THREADS) start[b] = 0;
    if (threadIdx.x == 0) {
        least_s = 0xFFFFFFFFu;
        most_s = 0;
    }
    griddep_wait();
    const int32_t* __restrict__ col = a.columns + (size_t)blockIdx.x * a.stride;
    int32_t key[KEYS];
    uint32_t bits[KEYS], least = 0xFFFFFFFFu, most = 0;
#pragma unroll
    for (int e = 0; e < KEYS; ++e) {
        const uint32_t b = threadIdx.x + e * THREADS;
        key[e] = b < B ? __ldcg(col + b) : -1;
    }
    __syncthreads();
#pragma unroll
    for (int e = 0; e < KEYS; ++e) {
        bits[e] = __float_as_uint(__int2float_rd(key[e]));   // counts >= 0: rounding down keeps their order
        if (key[e] >= 0) {
            least = min(least, bits[e]);
            most = max(most, bits[e]);
        }
    }
    least = __reduce_min_sync(0xFFFFFFFFu, least);
    most = __reduce_max_sync(0xFFFFFFFFu, most);
    if (lane == 0) {
        atomicMin(&least_s, least);
        atomicMax(&most_s, most);
    }
    __syncthreads();
    const uint32_t lo = least_s, span = most_s - lo;
    constexpr int LOG_BINS = BINS == 2048 ? 11 : 8;
    static_assert(1 << LOG_BINS == BINS, "a power of two");
    const int sh = span < (uint32_t)BINS ? 0 : 32 - LOG_BINS - __clz((int)span);   // span >> sh < BINS
    uint32_t at[KEYS];                          // position inside the bin
#pragma unroll
    for (int e = 0; e < KEYS; ++e)
        if (key[e] >= 0) at[e] = atomicAdd(&start[(bits[e] - lo) >> sh], 1u);
    __syncthreads();
    // exclusive scan of the bins' counts
    constexpr int PER = BINS >= THREADS ? BINS / THREADS : 1;
    uint32_t own[PER], sum = 0;
    const bool has = threadIdx.x * PER < BINS;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        own[q] = has ? start[threadIdx.x * PER + q] : 0;
        sum += own[q];
    }
    uint32_t incl = sum;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t u = __shfl_up_sync(0xFFFFFFFFu, incl, off);
        if (lane >= off) incl += u;
    }
    if (lane == 31) warp_sum[warp] = incl;
    __syncthreads();
    uint32_t first = incl - sum;
    for (int w = 0; w < warp; ++w) first += warp_sum[w];
    if (has) {
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            start[threadIdx.x * PER + q] = first;
            first += own[q];
        }
    }
    if (threadIdx.x == 0) start[BINS] = B;
    __syncthreads();
#pragma unroll
    for (int e = 0; e < KEYS; ++e)
        if (key[e] >= 0) v[start[(bits[e] - lo) >> sh] + at[e]] = (uint32_t)key[e];
    __syncthreads();
    const int32_t T1 = gridDim.x / 3, d = blockIdx.x / 3, c = blockIdx.x % 3;
    for (int32_t k = warp; k < a.n_q; k += THREADS / 32) {
        const uint32_t rank = a.qpos_dev ? a.qpos_dev[k] : a.qpos[k];   // 0-based
        // the bin: the last one that starts at or below the rank
        uint32_t b0 = 0;
#pragma unroll
        for (uint32_t step = BINS / 2; step > 0; step >>= 1)
            if (start[b0 + step] <= rank) b0 += step;
        const uint32_t s0 = start[b0], s1 = start[b0 + 1], want = rank - s0 + 1;
        // bisect the bin's values: the least x with at least `want` of them <= x
        uint32_t x0 = 0xFFFFFFFFu, x1 = 0;
        for (uint32_t q = s0 + lane; q < s1; q += 32) {
            x0 = min(x0, v[q]);
            x1 = max(x1, v[q]);
        }
        x0 = __reduce_min_sync(0xFFFFFFFFu, x0);
        x1 = __reduce_max_sync(0xFFFFFFFFu, x1);
        for (int it = 0; it < 32 && x0 < x1; ++it) {   // the interval halves each time
            const uint32_t mid = x0 + (x1 - x0) / 2;
            uint32_t n = 0;
            for (uint32_t q = s0 + lane; q < s1; q += 32) n += v[q] <= mid ? 1u : 0u;
            n = __reduce_add_sync(0xFFFFFFFFu, n);
            if (n >= want)
                x1 = mid;
            else
                x0 = mid + 1;
        }
        if (lane == 0) a.bands[((size_t)k * T1 + d) * 3 + c] = (float)(int32_t)x0;
    }
}

unsigned blocks_of_32(uint64_t n) { return (unsigned)((n + 31) / 32); }

// The rule between the staged kernels and a thread per sample, in waves of
// resident staged blocks. Once a thread per sample fills the chip, passing the
// normals through shared memory is only more work; rejection gains longest,
// since its blocks end with their last sample, and fast trajectories always
// (the warps that draw also write). Both sides on the device, 90 days:
//   distances   exact 30,000 samples 63 us staged, 65 us plain; 45,000 80 and
//               83; 55,000 92 and 84; fast 20,000 26 and 32; 55,000 45 and 42
//   rejection   exact 65,536 82 and 90; 150,000 143 and 150; 300,000 253 and
//               208; fast 150,000 68 and 74; 300,000 119 and 102
//   trajectories exact 30,000 76 and 84; 45,000 123 and 105; fast 100,003 82
//               and 102; 300,000 230 and 303
constexpr double kDistanceWaves = 1.0, kRejectWaves = 3.0, kExactSimulateWaves = 1.0;

template <typename K>
cudaError_t within_waves(K kernel, size_t smem, int producers, double waves, uint64_t n, bool* fits)
{
    int resident = 0;
    const cudaError_t e = grid_for(kernel, smem, &resident, staged_threads(producers));
    *fits = e == cudaSuccess && (double)n <= waves * 32.0 * resident;
    return e;
}

template <int MODE>
cudaError_t distances_m(const ModelParams& p, const DistanceArgs& a, cudaStream_t s, bool* taken)
{
    const size_t smem = sizeof(int4) * (size_t)(p.T + 1);
    cudaError_t e = within_waves(staged_distance_kernel<MODE>, smem, kSumProducers, kDistanceWaves, a.n_samples, taken);
    if (e != cudaSuccess || !*taken) return e;
    staged_distance_kernel<MODE><<<blocks_of_32(a.n_samples), staged_threads(kSumProducers), smem, s>>>(p, a);
    return cudaGetLastError();
}

template <int MODE, bool BELOW62>
cudaError_t reject_t(const ModelParams& p, const RejectArgs& a, cudaStream_t s, int* blocks_out, bool* taken)
{
    const size_t smem = sizeof(int4) * (size_t)(p.T + 1);
    cudaError_t e = within_waves(staged_reject_kernel<MODE, BELOW62>, smem, kSumProducers, kRejectWaves, a.n_samples, taken);
    if (e != cudaSuccess || !*taken) return e;
    const unsigned blocks = blocks_of_32(a.n_samples);
    if (blocks_out) *blocks_out = (int)blocks;
    staged_reject_kernel<MODE, BELOW62><<<blocks, staged_threads(kSumProducers), smem, s>>>(p, a);
    return cudaGetLastError();
}

template <int MODE>
cudaError_t reject_m(const ModelParams& p, const RejectArgs& a, cudaStream_t s, int* blocks_out, bool* taken)
{
    return a.acc_max < 0x4000000000000000ull ? reject_t<MODE, true>(p, a, s, blocks_out, taken)
                                             : reject_t<MODE, false>(p, a, s, blocks_out, taken);
}

template <int MODE>
cudaError_t simulate_m(const ModelParams& p, const SimulateArgs& a, cudaStream_t s, bool* taken)
{
    *taken = true;
    if (!is_fast(MODE)) {
        cudaError_t e = within_waves(staged_simulate_kernel<MODE>, 0, kWriteProducers, kExactSimulateWaves, a.B, taken);
        if (e != cudaSuccess || !*taken) return e;
    }
    staged_simulate_kernel<MODE><<<blocks_of_32(a.B), staged_threads(kWriteProducers), 0, s>>>(p, a);
    return cudaGetLastError();
}

template <int MODE>
cudaError_t columns_m(const ModelParams& p, const ColumnArgs& a, cudaStream_t s)
{
    staged_columns_kernel<MODE><<<blocks_of_32(a.B), staged_threads(kWriteProducers), 0, s>>>(p, a);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_staged_distances(const ModelParams& p, const DistanceArgs& a, int mode, cudaStream_t s, bool* taken)
{
    return ABC_MODE_DISPATCH(distances_m, mode, p, a, s, taken);
}

cudaError_t launch_staged_reject(const ModelParams& p, const RejectArgs& a, int mode, cudaStream_t s, int* blocks_out,
                                 bool* taken)
{
    return ABC_MODE_DISPATCH(reject_m, mode, p, a, s, blocks_out, taken);
}

cudaError_t launch_staged_simulate(const ModelParams& p, const SimulateArgs& a, int mode, cudaStream_t s, bool* taken)
{
    return ABC_MODE_DISPATCH(simulate_m, mode, p, a, s, taken);
}

cudaError_t launch_columns(const ModelParams& p, const ColumnArgs& a, int mode, cudaStream_t s)
{
    return ABC_MODE_DISPATCH(columns_m, mode, p, a, s);
}

cudaError_t launch_bands(const BandArgs& a, int32_t T, cudaStream_t s)
{
    if (a.B < 1 || a.B > 8192) return cudaErrorInvalidValue;
    const dim3 grid(3 * (unsigned)(T + 1));
    cudaError_t e;
    if (a.B <= 512)
        e = launch_overlapped(band_kernel<128, 4, 256>, grid, dim3(128), 0, s, a);
    else
        e = launch_overlapped(band_kernel<512, 16, 2048>, grid, dim3(512), 0, s, a);
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace abcgb
