// abc_kernels.cu -- sm_103a kernels of ABC rejection sampling (paper Sec. 2.2,
// Sec. 3.1): one simulation per thread, the compartments in registers, the
// observed series in shared memory, the accepted samples compacted with a
// warp ballot and one atomic per warp.
#include <cstdint>
#include <cuda_runtime.h>

#include "abc_kernels.h"
#include "abc_launch.h"
#include "abc_model.cuh"

namespace abcgb {

// Stage the observed series of days 0..T (A, R, D and the extinction terms) into
// shared memory.
__device__ __forceinline__ void stage_observed(int4* obs_s, const int4* __restrict__ obs, int32_t T)
{
    for (int32_t d = threadIdx.x; d <= T; d += blockDim.x) obs_s[d] = obs[d];
    __syncthreads();
}

// ---------------------------------------------------------------------------
// K1: fused rejection with early rejection and lane refill.
//
// The partial sums of the distance^2 only grow, so a sample whose running sum
// exceeds acc_max after some day pair can never be accepted: its lane drops it
// and takes the next sample (the accept set and the accepted distances are
// exactly those of running every sample for all T days). So does the lane of a
// sample whose infected have died out too far from the series (extinct_over). Each warp keeps a
// 64-entry ring of prior draws in shared memory, refilled 32 at a time by the
// whole warp (sample indices claimed with one atomicAdd per 32), so the theta
// draw of a new sample costs one shared-memory read for the lane that needs
// it. The loop advances every active lane by one day pair; all ring
// bookkeeping is warp-uniform. A ring entry holds the sample's parameters as
// the day loop uses them and its initial I0, worked out when the ring is
// refilled (32 samples, one per lane), so handing a sample to an idle lane
// is a few shared-memory reads. Accepted samples are compacted with a ballot
// and one atomicAdd per warp; their theta is re-drawn from the index.
// ---------------------------------------------------------------------------
constexpr int kRing = 64;
// A warp hands new samples to its idle lanes once at least kRefillMinIdle of
// them are idle (all 32 always qualify): the hand-out (ring read, derived
// parameters, initial state) runs on the whole warp, while a lane left idle
// for a day pair costs a 32nd of one. Measured on P = 6e7, T = 100, 2^24
// samples: 3.218 ms per launch at 1 (two pairs per pass), 3.209 at 2 and at 3,
// 3.219 at 4; exact mode's 2^22 samples 2.020 ms at 2, 2.030 at 3, 2.050 at 4.
// Which lane runs a sample, and when, does not change the sample's result.
constexpr uint32_t kRefillMinIdle = 2;

struct WarpRing {
    float4 lo[kRing];     // Theta a0, a, n, beta
    float4 hi[kRing];     // Theta gamma, delta, beta_eta; I0 (int32 bits)
    uint64_t idx[kRing];  // sample index
};

// Ring entry of sample ii: its Theta (kappa folded into I0) and I0.
template <int MODE>
__device__ __forceinline__ void ring_put(WarpRing& ring, uint32_t slot, const ModelParams& p, uint64_t ii,
                                         const float th[8], int32_t A0, int32_t room)
{
    const Theta t = make_theta<MODE>(th, p.inv_p);
    const int32_t I0 = initial_infected(t, A0, room);
    ring.lo[slot] = make_float4(t.a0, t.a, t.n, t.beta);
    ring.hi[slot] = make_float4(t.gamma, t.delta, t.beta_eta, __int_as_float(I0));
    ring.idx[slot] = ii;
}

template <int MODE, bool BELOW62>
__global__ void __launch_bounds__(kBlockThreads) abc_reject_kernel(const __grid_constant__ ModelParams p,
                                                                   const __grid_constant__ RejectArgs a)
{
    extern __shared__ int4 obs_s[];
    stage_observed(obs_s, a.obs, p.T);
    WarpRing* rings = reinterpret_cast<WarpRing*>(obs_s + (p.T + 1));
    const uint32_t lane = threadIdx.x & 31u;
    WarpRing& ring = rings[threadIdx.x >> 5];
    const uint32_t lt_mask = (1u << lane) - 1u;
    const int32_t T = p.T;

    bool active = false;
    uint64_t i = 0, acc = 0;
    // k: the next day pair of the lane's sample (1 with no sample); a sample's
    // simulated days, min(2 (k - 1), T), are counted when its lane takes the next
    uint32_t k = 1, days = 0;
    Theta t{};
    State x;
    uint32_t head = 0, tail = 0;     // ring entries consumed / produced (warp-uniform)
    bool exhausted = false;          // no indices left to claim (warp-uniform)

    while (true) {
        const uint32_t idle = __ballot_sync(0xFFFFFFFFu, !active);
        const uint32_t need = __popc(idle);
        if (need >= kRefillMinIdle) {
            if (tail - head < need && !exhausted) {
                unsigned long long base = 0;
                if (lane == 0) base = atomicAdd(a.next, 32ull);
                base = __shfl_sync(0xFFFFFFFFu, base, 0);
                if (base >= a.n_samples) {
                    exhausted = true;
                } else {
                    const uint64_t left = a.n_samples - base;
                    const uint32_t made = left < 32 ? (uint32_t)left : 32u;
                    if (lane < made) {
                        const uint64_t ii = a.first_index + base + lane;
                        float th[8];
                        prior_draw(p, ii, th);
                        ring_put<MODE>(ring, (tail + lane) & (kRing - 1), p, ii, th, p.A0, p.room0);
                    }
                    tail += made;
                    if (made < 32 || base + 32 >= a.n_samples) exhausted = true;
                    __syncwarp();
                }
            }
            const uint32_t avail = tail - head;
            // every lane idle and nothing left to hand out (the indices are
            // exhausted: a claim would have refilled the ring otherwise); this
            // replaces a second ballot per day pair for the loop's exit
            if (need == 32 && avail == 0) break;
            if (!active) {
                const uint32_t rank = __popc(idle & lt_mask);
                if (rank < avail) {
                    const uint32_t slot = (head + rank) & (kRing - 1);
                    const float4 l = ring.lo[slot], h = ring.hi[slot];
                    i = ring.idx[slot];
                    t.a0 = l.x; t.a = l.y; t.n = l.z; t.beta = l.w;
                    t.gamma = h.x; t.delta = h.y; t.beta_eta = h.z;
                    x = state_from(__float_as_int(h.w), p.A0, p.R0, p.D0, p.room0);
                    days += min(2 * k - 2, (uint32_t)T);
                    acc = 0;
                    k = 1;
                    active = true;
                }
            }
            head += need < avail ? need : avail;
            __syncwarp();
        }

        // fast mode takes three day pairs per pass between hand-outs, cutting
        // the refill and accept checks; per 2^24 samples of P = 6e7, T = 100:
        // 1 pair 3.232 ms, 2 pairs 3.218, 3 pairs 3.209. Exact mode's longer
        // day ran 13 % slower with two pairs.
        bool accept = false;
#pragma unroll
        for (int rep = 0; rep < ((MODE & kFast) ? 3 : 1); ++rep)
        if (active) {
            float z[10];
            day_pair_normals<MODE>(p, i, k, z);
            const int32_t d1 = (int32_t)(2 * k - 1);
            model_day<MODE>(x, t, p.inv_p, z);
            const int4 o1 = obs_s[d1];
            int32_t m_bits = 0;
            acc = BELOW62 ? add_day_sq_below62(acc, x, o1) : add_day_sq(acc, x, o1);
            if (d1 < T) {
                model_day<MODE>(x, t, p.inv_p, z + 5);
                const int4 o2 = obs_s[d1 + 1];
                m_bits = o2.w;
                acc = BELOW62 ? add_day_sq_below62(acc, x, o2) : add_day_sq(acc, x, o2);
            }
            bool over = acc > a.acc_max;
            const bool last = d1 + 1 >= T;
            // a threshold of 2^63 accepts sums that saturate there: nothing is over
            if (x.I == 0 && !over && !last && (BELOW62 || a.acc_max < kAccCap))
                over = extinct_over(x, o1.w, m_bits, T - d1 - 1, acc, a.acc_max);
            accept = !over && last;
            active = !(over || last);
            ++k;
        }
        const uint32_t mask = __ballot_sync(0xFFFFFFFFu, accept);
        if (mask) {
            const uint32_t leader = __ffs(mask) - 1;
            unsigned long long slot0 = 0;
            if (lane == leader) slot0 = atomicAdd(a.count, (unsigned long long)__popc(mask));
            slot0 = __shfl_sync(0xFFFFFFFFu, slot0, leader);
            if (accept) {
                const uint64_t slot = slot0 + __popc(mask & lt_mask);
                if (slot < a.capacity) {
                    float th[8];
                    prior_draw(p, i, th);
                    a.idx_out[slot] = i;
                    a.dist_out[slot] = __dsqrt_rn(__ull2double_rn(acc));
                    float4* to = reinterpret_cast<float4*>(a.theta_out + 8 * slot);
                    to[0] = make_float4(th[0], th[1], th[2], th[3]);
                    to[1] = make_float4(th[4], th[5], th[6], th[7]);
                }
            }
        }
    }
    // simulated model days of this warp (for throughput accounting), the
    // lane's last sample included
    days += min(2 * k - 2, (uint32_t)T);
    unsigned long long d = days;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) d += __shfl_down_sync(0xFFFFFFFFu, d, off);
    if (lane == 0 && a.sim_days) atomicAdd(a.sim_days, d);
}

// ---------------------------------------------------------------------------
// K2: every distance (and optionally every prior draw).
// ---------------------------------------------------------------------------
template <int MODE>
__global__ void __launch_bounds__(kBlockThreads) abc_distance_kernel(const __grid_constant__ ModelParams p,
                                                                     const __grid_constant__ DistanceArgs a)
{
    extern __shared__ int4 obs_s[];
    stage_observed(obs_s, a.obs, p.T);
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; j < a.n_samples; j += stride) {
        const uint64_t i = a.first_index + j;
        float th[8];
        prior_draw(p, i, th);
        const Theta t = make_theta<MODE>(th, p.inv_p);
        const State x0 = init_state(t, p.A0, p.R0, p.D0, p.room0);
        const uint64_t acc = simulate_sample<MODE>(p, i, t, x0, obs_s);
        a.dist_out[j] = __dsqrt_rn(__ull2double_rn(acc));
        if (a.theta_out) {
            float4* to = reinterpret_cast<float4*>(a.theta_out + 8 * j);
            to[0] = make_float4(th[0], th[1], th[2], th[3]);
            to[1] = make_float4(th[4], th[5], th[6], th[7]);
        }
    }
}

// ---------------------------------------------------------------------------
// K3: trajectories of given (theta, sample index) pairs, whole rows
// [T + 1][6] (S, I, A, R, D, Ru), a thread per sample (exact arithmetic only:
// see the rule in abc_staged.cu). A warp keeps kTrajDays
// days of its 32 rows in shared memory and then writes each row's days as one
// run of 8-byte words: a lane storing its own six values a day touched 32
// sectors with every 4 bytes. ALU-bound now: 100,003 rows over 90 days in exact arithmetic
// 442 -> 215 us (218 MB written). Blocks of two warps spread the rows evenly
// over the SMs.
// ---------------------------------------------------------------------------
constexpr int kTrajDays = 8;
constexpr int kTrajThreads = 64;
struct TrajRows {
    int2 s[32][3 * kTrajDays + 1];   // the odd stride (in 8 bytes) spreads lanes over the banks
};

// days d0 .. d0 + days - 1 of the warp's rows to global memory, 8 lanes a row
__device__ __forceinline__ void write_days(const TrajRows& tile, int32_t* out, uint32_t rows, int32_t T, int32_t d0,
                                           int32_t days, bool wide)
{
    const uint32_t lane = threadIdx.x & 31u;
    __syncwarp();
    for (uint32_t r = lane >> 3; r < rows; r += 4) {
        int32_t* to = out + (size_t)r * 6 * (size_t)(T + 1) + 6 * (size_t)d0;
        for (uint32_t c = lane & 7u; c < 3 * (uint32_t)days; c += 8) {
            const int2 v = tile.s[r][c];
            if (wide) {
                *reinterpret_cast<int2*>(to + 2 * c) = v;
            } else {
                to[2 * c] = v.x;
                to[2 * c + 1] = v.y;
            }
        }
    }
    __syncwarp();
}

template <int MODE>
__global__ void __launch_bounds__(kTrajThreads) abc_simulate_kernel(const __grid_constant__ ModelParams p,
                                                                    const __grid_constant__ SimulateArgs a)
{
    __shared__ TrajRows tiles[kTrajThreads / 32];
    const uint32_t lane = threadIdx.x & 31u;
    TrajRows& tile = tiles[threadIdx.x >> 5];
    const bool wide = (reinterpret_cast<uintptr_t>(a.traj_out) & 7u) == 0;
    const int32_t T = p.T;
    const auto put = [&](int32_t slot, const State& x) {
        int2* to = &tile.s[lane][3 * slot];
        to[0] = make_int2(x.S, x.I);
        to[1] = make_int2(x.A, x.R);
        to[2] = make_int2(x.D, x.Ru);
    };
    const uint64_t step = (uint64_t)gridDim.x * kTrajThreads;
    for (uint64_t b0 = (uint64_t)blockIdx.x * kTrajThreads + (threadIdx.x & ~31u); b0 < a.B; b0 += step) {
        const uint32_t rows = (uint32_t)min(a.B - b0, (uint64_t)32);
        const uint64_t b = b0 + min(lane, rows - 1);   // lanes past the end repeat the last row, unwritten
        const uint64_t i = a.sample_index[b];
        int32_t* out = a.traj_out + (size_t)b0 * 6 * (size_t)(T + 1);
        float th[8];
        const float4* ti = reinterpret_cast<const float4*>(a.theta + 8 * b);
        const float4 t0 = ti[0], t1 = ti[1];
        th[0] = t0.x; th[1] = t0.y; th[2] = t0.z; th[3] = t0.w;
        th[4] = t1.x; th[5] = t1.y; th[6] = t1.z; th[7] = t1.w;
        const Theta t = make_theta<MODE>(th, p.inv_p);
        State x = init_state(t, p.A0, p.R0, p.D0, p.room0);
        put(0, x);
        write_days(tile, out, rows, T, 0, 1, wide);
        const uint32_t n_pairs = (uint32_t)(T + 1) >> 1;
        int32_t slot = 0;
        for (uint32_t k = 1; k <= n_pairs; ++k) {
            float z[10];
            day_pair_normals<MODE>(p, i, k, z);
            const int32_t d1 = (int32_t)(2 * k - 1);
            model_day<MODE>(x, t, p.inv_p, z);
            put(slot++, x);
            if (d1 < T) {
                model_day<MODE>(x, t, p.inv_p, z + 5);
                put(slot++, x);
            }
            if (slot == kTrajDays || k == n_pairs) {
                const int32_t last = min(d1 + 1, T);
                write_days(tile, out, rows, T, last - slot + 1, slot, wide);
                slot = 0;
            }
        }
    }
}

// ---------------------------------------------------------------------------
// K4: one day applied to given states.
// ---------------------------------------------------------------------------
template <int MODE>
__global__ void __launch_bounds__(kBlockThreads) abc_step_kernel(const __grid_constant__ ModelParams p,
                                                                 const __grid_constant__ StepArgs a)
{
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t b = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; b < a.B; b += stride) {
        float th[8];
        for (int j = 0; j < 8; ++j) th[j] = a.theta[8 * b + j];
        const Theta t = make_theta<MODE>(th, p.inv_p);
        const int32_t* si = a.state_in + 6 * b;
        State x{si[0], si[1], si[2], si[3], si[4], si[5]};
        const int32_t d = a.day[b];
        float z[10];
        day_pair_normals<MODE>(p, a.sample_index[b], (uint32_t)(d + 1) >> 1, z);
        int32_t n[5];
        model_day<MODE>(x, t, p.inv_p, (d & 1) ? z : z + 5, n);
        int32_t* so = a.state_out + 6 * b;
        so[0] = x.S; so[1] = x.I; so[2] = x.A; so[3] = x.R; so[4] = x.D; so[5] = x.Ru;
        if (a.counts_out)
            for (int k = 0; k < 5; ++k) a.counts_out[5 * b + k] = n[k];
    }
}

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------
static int blocks_for(uint64_t n, int cap, int threads = kBlockThreads)
{
    const uint64_t b = (n + threads - 1) / threads;
    return (int)(b < (uint64_t)cap ? (b > 0 ? b : 1) : (uint64_t)cap);
}

// Threads of a block of the two kernels that stage the series: small blocks
// deal a call of a few waves out evenly (65,536 samples are 256 blocks of 256
// threads: two on some SMs, one on others), unless the series takes so much
// shared memory that small blocks would not fill an SM. Distances over 90 days
// in exact mode: 55,000 samples 103 -> 84 us, 2e6 unchanged.
constexpr int kSmallBlock = 64;
constexpr int32_t kSmallBlockT = 400;
static int series_block_threads(int32_t T) { return T <= kSmallBlockT ? kSmallBlock : kBlockThreads; }

template <int MODE, bool BELOW62>
static cudaError_t launch_reject_t(const ModelParams& p, const RejectArgs& a, cudaStream_t s, int* blocks_out)
{
    const int threads = series_block_threads(p.T), warps = threads / 32;
    const size_t smem = sizeof(int4) * (size_t)(p.T + 1) + sizeof(WarpRing) * warps;
    int grid = 0;
    cudaError_t e = grid_for(abc_reject_kernel<MODE, BELOW62>, smem, &grid, threads);
    if (e != cudaSuccess) return e;
    // persistent: every resident block loops over claimed index chunks
    const uint64_t chunks = (a.n_samples + 31) / 32;
    const uint64_t want = (chunks + warps - 1) / warps;
    if (want < (uint64_t)grid) grid = (int)(want > 0 ? want : 1);
    if (blocks_out) *blocks_out = grid;
    abc_reject_kernel<MODE, BELOW62><<<grid, threads, smem, s>>>(p, a);
    return cudaGetLastError();
}

template <int MODE>
static cudaError_t launch_reject_m(const ModelParams& p, const RejectArgs& a, cudaStream_t s, int* blocks_out)
{
    const bool below62 = a.acc_max < 0x4000000000000000ull;
    return below62 ? launch_reject_t<MODE, true>(p, a, s, blocks_out) : launch_reject_t<MODE, false>(p, a, s, blocks_out);
}

cudaError_t launch_reject(const ModelParams& p, const RejectArgs& a, int mode, cudaStream_t s, int* blocks_out)
{
    bool taken = false;
    const cudaError_t e = launch_staged_reject(p, a, mode, s, blocks_out, &taken);
    if (e != cudaSuccess || taken) return e;
    return ABC_MODE_DISPATCH(launch_reject_m, mode, p, a, s, blocks_out);
}

template <int MODE>
static cudaError_t launch_distances_m(const ModelParams& p, const DistanceArgs& a, cudaStream_t s)
{
    const size_t smem = sizeof(int4) * (size_t)(p.T + 1);
    int grid = 0;
    const int threads = series_block_threads(p.T);
    cudaError_t e = grid_for(abc_distance_kernel<MODE>, smem, &grid, threads);
    if (e != cudaSuccess) return e;
    grid = blocks_for(a.n_samples, grid, threads);
    abc_distance_kernel<MODE><<<grid, threads, smem, s>>>(p, a);
    return cudaGetLastError();
}

cudaError_t launch_distances(const ModelParams& p, const DistanceArgs& a, int mode, cudaStream_t s)
{
    bool taken = false;
    const cudaError_t e = launch_staged_distances(p, a, mode, s, &taken);
    if (e != cudaSuccess || taken) return e;
    return ABC_MODE_DISPATCH(launch_distances_m, mode, p, a, s);
}

template <int MODE>
static cudaError_t launch_simulate_m(const ModelParams& p, const SimulateArgs& a, cudaStream_t s)
{
    int grid = 0;
    cudaError_t e = grid_for(abc_simulate_kernel<MODE>, 0, &grid, kTrajThreads);
    if (e != cudaSuccess) return e;
    grid = blocks_for(a.B, grid, kTrajThreads);
    abc_simulate_kernel<MODE><<<grid, kTrajThreads, 0, s>>>(p, a);
    return cudaGetLastError();
}

cudaError_t launch_simulate(const ModelParams& p, const SimulateArgs& a, int mode, cudaStream_t s)
{
    bool taken = false;
    const cudaError_t e = launch_staged_simulate(p, a, mode, s, &taken);
    if (e != cudaSuccess || taken) return e;
    // fast mode is always staged
    return mode == kExact ? launch_simulate_m<kExact>(p, a, s) : launch_simulate_m<kExact | kLiteral>(p, a, s);
}

template <int MODE>
static cudaError_t launch_step_m(const ModelParams& p, const StepArgs& a, cudaStream_t s)
{
    int grid = 0;
    cudaError_t e = grid_for(abc_step_kernel<MODE>, 0, &grid);
    if (e != cudaSuccess) return e;
    grid = blocks_for(a.B, grid);
    abc_step_kernel<MODE><<<grid, kBlockThreads, 0, s>>>(p, a);
    return cudaGetLastError();
}

cudaError_t launch_step(const ModelParams& p, const StepArgs& a, int mode, cudaStream_t s)
{
    return ABC_MODE_DISPATCH(launch_step_m, mode, p, a, s);
}

}  // namespace abcgb
