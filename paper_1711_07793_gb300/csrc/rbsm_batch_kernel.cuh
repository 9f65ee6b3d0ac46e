// Device side of the batched launch: descriptors, per-warp queues, the
// learned drain and the batch_kernel template.  Its instantiations are
// spread over rbsm_batch_inst_*.cu so that they compile in parallel.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "rbsm.h"
#include "rbsm_device.cuh"
#include "rbsm_mlp.cuh"

namespace rbsm {

struct BatchJobDev {
    const float *x, *y, *z;
    float *sil, *fil;
    uint16_t *codes;
    long long n;
    long long tile_start;        // first work item of the job
    int map;
    int mode;                    // 1, 2, 3
    int vec;                     // all planes 16-byte aligned
    int codes_on;
};

// Passed by value as a __grid_constant__ kernel parameter (about 21 KB,
// inside the 32 KB parameter space), so no descriptor copy to the device
// is needed and the launch can be captured into a CUDA graph as is.
struct BatchArgs {
    MapDev maps[RBSM_BATCH_MAX_MAPS];
    BatchJobDev jobs[RBSM_BATCH_MAX_JOBS];
    int n_jobs;
    int max_dist;
    long long total_tiles;
    unsigned long long *counter;     // n_counters work counters, kCounterStride bytes apart
    int *status;
    const void *mlp;                 // surrogate state block or nullptr
    float tau;                       // guard: largest accepted error estimate
    unsigned long long *stats;       // [0] surrogate answers, [1] fallbacks
    int chunk_tiles;                 // warp tiles per claim of the work counter, 1..kMaxChunkTiles
    int n_counters;                  // kCounters, or 1 in a workspace of kMinWorkspaceBytes
};

// The workspace: kCounters work counters, each in its own kCounterStride
// bytes (the first block also holds the status word and the statistics).
// Atomics on one address, or on one line, go through at about 0.77 a
// nanosecond here, while 6080 warps finish 1.5 tiles in that time, so a
// counter alone forces claims of several tiles.  Claims of one tile keep the
// tiles that are in flight next to each other in memory, which is what the
// DRAM wants: 8 frames of 3840x2160 fragments in one launch took 403 / 381 /
// 375 us at 8 / 4 / 2 tiles per claim of one counter, 669 at 1, and 350 at 1
// tile per claim of 8 counters on lines of their own (4 counters 363 at 2
// tiles, 32 counters 361; 8 counters in one pair of lines 646).
constexpr int kCounterBits = 3, kCounters = 1 << kCounterBits;
constexpr size_t kCounterStride = 512;
constexpr size_t kWorkspaceBytes = kCounters * kCounterStride;
constexpr size_t kMinWorkspaceBytes = 256;       // one counter
constexpr int kMaxChunkTiles = 8;

__device__ __forceinline__ int find_job(const BatchArgs &a, long long tile)
{
    int lo = 0, hi = a.n_jobs - 1;    // last job whose first tile <= tile
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (a.jobs[mid].tile_start <= tile)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ WarpTileIO job_tile(const BatchJobDev &J, int job, long long tile)
{
    WarpTileIO t;
    t.x = J.x; t.y = J.y; t.z = J.z; t.sil = J.sil; t.fil = J.fil; t.codes = J.codes;
    t.first = (tile - J.tile_start) * kWarpTile;
    const long long left = J.n - t.first;
    t.count = left < kWarpTile ? (int)left : kWarpTile;
    t.job = job;
    t.vec = J.vec && t.count == kWarpTile;
    return t;
}

// Job table of a batched launch, for the deferred edge answers.
struct BatchJobs {
    const BatchArgs *a;
    __device__ __forceinline__ JobOut operator()(int j) const
    {
        const BatchJobDev &J = a->jobs[j];
        return JobOut{a->maps[J.map], J.x, J.y, J.z, J.sil, J.fil, J.codes_on ? J.codes : nullptr, J.mode};
    }
};

// Shared memory of the learned variant: the network's biases and weight
// pointers and, per warp, the 32 input rows and 32 outputs of one round of
// edge fragments and the queue of the fragments the network may answer.
template <int kThreads>
struct LearnedSmem {
    mlp::InferWeights w;
    uint16_t feat[kThreads / 32][32 * mlp::kIn];
    float out[kThreads / 32][32 * mlp::kOut];
    EdgeEntry candidate[kThreads / 32][64];     // < 32 left over + one round
    const uint32_t *trust;                      // trusted-pattern bitmap, or nullptr (none in force)
};

// One round of the network over up to 32 candidates (one per lane): each
// lane gathers its fragment's 5x5 features; the fragments whose pattern is
// trusted are packed into input rows and the warp runs the network on as many
// m16 tiles as they fill (0, 1 or 2, on the tensor cores); each of them whose
// error estimate is within the guard takes the estimate, clamped to [0, 1],
// over the exact answer it has.
template <typename Jobs, int kThreads>
__device__ __forceinline__ void network_round(const Jobs &jobs, bool valid, const EdgeEntry &q,
                                              LearnedSmem<kThreads> &ls, int warp, float tau,
                                              unsigned long long *stats)
{
    const unsigned lane = lane_id();
    const unsigned below = (1u << lane) - 1u;
    const int g = lane >> 2, t = lane & 3;
    uint16_t *feat = ls.feat[warp];
    float *yout = ls.out[warp];
    bool trusted = false;
    uint32_t bits = 0;
    float fx = 0.0f, fy = 0.0f, gap = 0.0f;
    if (valid) {
        const JobOut o = jobs((int)(q.bits_job >> 8));
        fragment_features(o.map, __ldg(o.x + q.idx), __ldg(o.y + q.idx), __ldg(o.z + q.idx), bits, fx, fy, gap);
        trusted = mlp::pattern_trusted(ls.trust, bits);
    }
    const unsigned mask = __ballot_sync(0xffffffffu, trusted);
    const int row = __popc(mask & below);
    if (trusted)
        mlp::write_input_row(feat + row * mlp::kIn, bits, fx, fy, gap);
    __syncwarp();
    const int tiles = (__popc(mask) + 15) >> 4;          // m16 tiles with rows in use (0..2)
    for (int mt = 0; mt < tiles; ++mt) {
        uint32_t xa[2][4];
        mlp::load_a(feat, mlp::kIn, mt * 16, 0, lane, xa[0]);
        mlp::load_a(feat, mlp::kIn, mt * 16, 1, lane, xa[1]);
        mlp::HiddenFrags h1, h2;
        uint32_t m1, m2;
        mlp::layer(xa, 2, ls.w.w1t, mlp::kIn, ls.w.b1, lane, h1, m1);
        mlp::layer(h1.a, 4, ls.w.w2t, mlp::kHid, ls.w.b2, lane, h2, m2);
        float y[4];
        mlp::output_layer(h2, ls.w.w3t, ls.w.b3, lane, y);
        if (t == 0) {
            yout[(mt * 16 + g) * 2] = y[0];
            yout[(mt * 16 + g) * 2 + 1] = y[1];
            yout[(mt * 16 + g + 8) * 2] = y[2];
            yout[(mt * 16 + g + 8) * 2 + 1] = y[3];
        }
    }
    __syncwarp();
    bool accepted = false;
    if (trusted) {
        const float v = yout[row * 2], e = yout[row * 2 + 1];
        // the network's own error estimate (a NaN never passes)
        accepted = e <= tau && v == v;
        if (accepted) {
            const JobOut o = jobs((int)(q.bits_job >> 8));
            o.fil[q.idx] = v < 0.0f ? 0.0f : (v > 1.0f ? 1.0f : v);
            if (o.codes) {
                const uint32_t cb = q.bits_job & 0x1fu;
                o.codes[q.idx] = (uint16_t)((cb >> 1) | ((1u - (cb & 1u)) << 4) | (1u << 10));
            }
        }
    }
    const unsigned acc_mask = __ballot_sync(0xffffffffu, accepted);
    if (lane == 0 && acc_mask) {
        const unsigned long long n = (unsigned long long)__popc(acc_mask);
        atomicAdd(&stats[0], n);
        atomicAdd(&stats[1], 0ull - n);                  // they had been counted as fallbacks
    }
    __syncwarp();                                        // rows and outputs read before they are overwritten
}

// Drain rounds of up to 32 queued edge fragments of the learned variant.
// Every fragment gets its exact answer first, in full rounds like the exact
// path's.  The network may only answer FILTER-mode fragments whose walks stop
// inside the 5x5 window, which the walks just told: those go to the warp's
// candidate queue and to the network 32 at a time, and an accepted estimate
// overwrites the exact answer.  So only the fragments that can use them pay
// for the 25 window texels and the products, on full warps.  (The features of
// every edge fragment first, and a second queue of walks for those turned
// down: 128 against 97 us for one 3840x2160 frame, the same answers.)
template <typename Jobs, int kThreads>
__device__ __forceinline__ void drain_queue_learned(const Jobs &jobs, WarpQueue &wq, int &count, int &candidates,
                                                    int max_dist, bool all, LearnedSmem<kThreads> &ls, int warp,
                                                    float tau, unsigned long long *stats)
{
    const unsigned lane = lane_id();
    const unsigned below = (1u << lane) - 1u;
    EdgeEntry *cq = ls.candidate[warp];
    while (count >= 32 || (all && count > 0)) {
        __syncwarp();                      // queue entries and provisional stores are visible
        const int base = count >= 32 ? count - 32 : 0;
        const int k = base + (int)lane;
        bool use_net = false, candidate = false;
        EdgeEntry q{0u, 0u};
        if (k < count) {
            q = wq.q[k];
            const JobOut o = jobs((int)(q.bits_job >> 8));
            use_net = o.mode == 2;
            const int reach = resolve_entry(o, q, max_dist);
            candidate = use_net && (max_dist <= 2 || reach <= 2);
        }
        const unsigned net_mask = __ballot_sync(0xffffffffu, use_net);
        const unsigned mask = __ballot_sync(0xffffffffu, candidate);
        if (candidate)
            cq[candidates + __popc(mask & below)] = q;
        if (lane == 0 && net_mask)
            atomicAdd(&stats[1], (unsigned long long)__popc(net_mask));
        candidates += __popc(mask);
        count = base;
        __syncwarp();                      // candidates written and entries read; exact answers before estimates
        if (candidates >= 32) {
            candidates -= 32;
            network_round<Jobs, kThreads>(jobs, true, cq[candidates + (int)lane], ls, warp, tau, stats);
        }
    }
    if (all && candidates > 0) {
        const EdgeEntry q = cq[min((int)lane, candidates - 1)];
        network_round<Jobs, kThreads>(jobs, (int)lane < candidates, q, ls, warp, tau, stats);
        candidates = 0;
    }
}

template <int kThreads, bool LEARNED>
struct BatchSmem {
    WarpQueue queue[kThreads / 32];
    float4 next[kThreads / 32][3][32];   // each warp's next tile: x, y, z, one float4 per lane and plane
};

template <int kThreads, bool LEARNED>
constexpr size_t batch_smem_bytes()
{
    return sizeof(BatchSmem<kThreads, LEARNED>) + (LEARNED ? sizeof(LearnedSmem<kThreads>) : 0);
}

// Persistent warps take chunks of chunk_tiles warp tiles in job order: the
// first two by their place in the grid, the others from a work counter (a
// CTA's warps share one of the n_counters; counter q hands out every
// n_counters-th chunk), except that with chunks of several tiles the last
// tiles of the launch (two per warp) go out one per claim, so that warps
// finish together.  A claim is issued when the chunk before it starts, and
// its value is read only when the warp gets there, so the atomic's latency
// hides behind a chunk of work.  A warp whose counter has run out goes on
// with the one that has most left.  While a warp works on one tile, the
// asynchronous copies of its next tile's coordinates into the warp's
// shared-memory buffer are in flight: the tile is read out of the buffer
// into registers, the buffer is refilled with the next tile, and the
// registers are classified (the prefetch holds no registers, which makes
// room for 5 CTAs of 256 threads per SM).  The tiles in flight at one time
// are neighbours in the job list, so they share DRAM pages and the L2
// footprint of one region of one map.
//
// UMODE 0: each job's mode and codes flag are read at run time; UMODE
// 2 * mode + codes - 1 (1..6): every job of the launch has that pair, which
// keeps one specialisation of the classification in the loop (the run-time
// dispatch inlines all six and costs registers); UMODE 7..12: the same
// pairs, and no map has a texture (kernels of classify_warp_tile's TEX 0).
template <int kThreads, bool LEARNED, int kMinBlocks, int UMODE>
__global__ void __launch_bounds__(kThreads, kMinBlocks) batch_kernel(const __grid_constant__ BatchArgs a)
{
    constexpr int kPair = UMODE > 6 ? UMODE - 6 : UMODE;
    constexpr int kTex = UMODE > 6 ? 0 : -1;
    constexpr int kFixedMode = (kPair + 1) / 2;
    constexpr bool kFixedCodes = ((kPair + 1) % 2) == 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    auto &bs = *reinterpret_cast<BatchSmem<kThreads, LEARNED> *>(smem_raw);
    auto &ls = *reinterpret_cast<LearnedSmem<kThreads> *>(smem_raw + sizeof(BatchSmem<kThreads, LEARNED>));
    const unsigned lane = lane_id();
    const int warp = threadIdx.x >> 5;
    if (LEARNED) {
        const mlp::State st = mlp::state_of(const_cast<void *>(a.mlp));
        if (threadIdx.x == 0) {
            ls.w.w1t = st.w1t;
            ls.w.w2t = st.w2t;
            ls.w.w3t = st.w3t;
        }
        for (int k = threadIdx.x; k < mlp::kHid; k += kThreads) {
            ls.w.b1[k] = st.master[mlp::kOffB1 + k];
            ls.w.b2[k] = st.master[mlp::kOffB2 + k];
        }
        for (int k = threadIdx.x; k < mlp::kOutPad; k += kThreads)
            ls.w.b3[k] = k < mlp::kOut ? st.master[mlp::kOffB3 + k] : 0.0f;
        if (threadIdx.x == 0)
            ls.trust = *st.trust_on ? st.trust : nullptr;
        __syncthreads();
    }
    WarpQueue &wq = bs.queue[warp];
    const long long total = a.total_tiles;
    const int chunk = a.chunk_tiles;
    const long long warps = (long long)gridDim.x * (kThreads / 32);
    // claims below c1 take `chunk` tiles, later ones a single tile, so the
    // last tiles (about two per warp) are spread one at a time
    const long long tail = 2 * warps;
    const long long c1 = total > tail ? (total - tail) / chunk : 0;
    auto first_tile = [&](long long c) { return c < c1 ? c * chunk : c1 * chunk + (c - c1); };
    // (through a shuffle, as every later claim: the compiler then knows that
    // the tile, its job and their addresses are the same on all lanes)
    const long long c0 = (long long)__shfl_sync(0xffffffffu, blockIdx.x * (kThreads / 32) + (unsigned)warp, 0);
    long long tile = first_tile(c0);
    int csz = c0 < c1 ? chunk : 1;
    if (tile >= total)
        return;
    unsigned counter = blockIdx.x % (unsigned)a.n_counters;
    auto counter_at = [&](unsigned q) { return a.counter + q * (kCounterStride / sizeof(unsigned long long)); };
    auto take = [&]() {
        return 2ull * (unsigned long long)warps + atomicAdd(counter_at(counter), 1ull) * (unsigned)a.n_counters +
               counter;
    };
    unsigned long long claim = (unsigned long long)(warps + c0);    // the next chunk (lane 0's counts)
    int in_chunk = 0;
    int job = find_job(a, tile);
    // tiles [job_lo, job_hi) belong to `job`: the search runs only when a
    // tile falls outside the current job
    long long job_lo = a.jobs[job].tile_start;
    long long job_hi = job + 1 < a.n_jobs ? a.jobs[job + 1].tile_start : total;
    WarpTileIO t = job_tile(a.jobs[job], job, tile);
    float4 (&buf)[3][32] = bs.next[warp];
    stage_tile(t, lane, buf);
    const BatchJobs jobs{&a};
    // the current job's map: in the 48-register variant (5 CTAs per SM) a
    // copy read again only when the job changes, elsewhere read per tile
    // (measured: the copy helps the former by 2.6 % on C5 and slows the
    // 3-CTA variant by 5 % on C4)
    constexpr bool kCopyMap = kMinBlocks >= 5;
    MapDev map = a.maps[a.jobs[job].map];
    int queued = 0;
    int candidates = 0;                        // learned variant: fragments waiting for the network
    for (;;) {
        long long nt;
        if (in_chunk + 1 < csz) {
            nt = tile + 1;
            in_chunk += 1;
        } else {
            if (a.n_counters > 1) {
                const long long claims = c1 + (total - c1 * chunk);
                if (claims > 2 * warps && __shfl_sync(0xffffffffu, claim, 0) >= (unsigned long long)claims) {
                    // this counter has run out: go on with the one that has
                    // most claims left (what a warp leaves, the warps of that
                    // counter's own CTAs take)
                    unsigned left = 0;
                    if (lane < (unsigned)kCounters) {
                        const long long mine = (claims - 2 * warps - (long long)lane + kCounters - 1) >> kCounterBits;
                        const long long n = mine - (long long)*(volatile unsigned long long *)counter_at(lane);
                        left = n > 0 ? ((unsigned)(n < (1 << 24) ? n : (1 << 24)) << 4) | lane : 0u;
                    }
                    left = __reduce_max_sync(0xffffffffu, left);
                    if (left != 0u) {
                        counter = left & 15u;
                        if (lane == 0)
                            claim = take();
                    }
                }
            }
            const long long c = (long long)__shfl_sync(0xffffffffu, claim, 0);
            nt = first_tile(c);
            csz = c < c1 ? chunk : 1;
            in_chunk = 0;
            if (nt < total && lane == 0)
                claim = take();
        }
        const bool more = nt < total;
        int njob = job;
        WarpTileIO tn;
        LaneCoords c;
        fetch_tile<kTex == 0>(t, lane, buf, c);
        if (more) {
            if (nt < job_lo || nt >= job_hi) {
                if (nt < job_lo)
                    njob = find_job(a, nt);
                // mostly a few jobs on (the claims advance through the list)
#pragma unroll 1
                while (njob + 1 < a.n_jobs && a.jobs[njob + 1].tile_start <= nt)
                    ++njob;
                job_lo = a.jobs[njob].tile_start;
                job_hi = njob + 1 < a.n_jobs ? a.jobs[njob + 1].tile_start : total;
                tn = job_tile(a.jobs[njob], njob, nt);
            } else {
                // same job: only the position, the count and the vector flag move
                tn = t;
                tn.first = (nt - job_lo) * kWarpTile;
                const long long left = a.jobs[job].n - tn.first;
                tn.count = left < kWarpTile ? (int)left : kWarpTile;
                tn.vec = a.jobs[job].vec && tn.count == kWarpTile;
            }
            stage_tile(tn, lane, buf);         // next tile's copies fly during this tile
        }
        const BatchJobDev &J = a.jobs[job];
        if (UMODE == 0)
            classify_warp_tile_rt(J.mode, J.codes_on != 0, kCopyMap ? map : a.maps[J.map], t, c, wq, queued);
        else
            classify_warp_tile<kFixedMode ? kFixedMode : 1, kFixedCodes, kTex>(kCopyMap ? map : a.maps[J.map], t, c,
                                                                               wq, queued);
        if (LEARNED)
            drain_queue_learned<BatchJobs, kThreads>(jobs, wq, queued, candidates, a.max_dist, false, ls, warp, a.tau,
                                                     a.stats);
        else
            drain_queue<BatchJobs, kFixedMode>(jobs, wq, queued, a.max_dist, false);
        if (!more)
            break;
        tile = nt;
        if (kCopyMap && njob != job)
            map = a.maps[a.jobs[njob].map];
        job = njob;
        t = tn;
    }
    if (LEARNED)
        drain_queue_learned<BatchJobs, kThreads>(jobs, wq, queued, candidates, a.max_dist, true, ls, warp, a.tau,
                                                 a.stats);
    else
        drain_queue<BatchJobs, kFixedMode>(jobs, wq, queued, a.max_dist, true);
}

using BatchKernelFn = void (*)(BatchArgs);

// Kernel pointers of the instantiations (one function per translation unit).
BatchKernelFn batch_kernel_256_4(bool learned, int umode);
BatchKernelFn batch_kernel_256_3(int umode);
BatchKernelFn batch_kernel_256_5(int umode);
BatchKernelFn batch_kernel_misc(int threads, bool learned);
BatchKernelFn batch_kernel_untextured(bool learned, int umode);      // 7..12; learned: 9, 10

}  // namespace rbsm
