// RPCF: percentage-closer filtering over the RSMSS answer (§5.3 removes the
// skeleton artifacts of the filtered edges with PCF; the paper prints no
// kernel).  A fragment's answer is the mean Listing 5 answer of the k x k
// samples at its texel-space position shifted by whole texels, (u + a,
// v + b), each with the fragment's depth.
//
// The sample is the unit of deferred work: a lane classifies its fragment's
// samples (two texture gathers or five loads each, or all from one block,
// below); off-edge samples add their shadow test at once, edge samples go to
// the warp's queue (fragment and sample index; for k = 3 with the fragment's
// shadow tests, else the drain classifies the sample again) and are walked
// 32 at a time on full warps.  For k > 1 a
// fragment with edge samples keeps its sum in the output plane as a
// fixed-point integer (each sample answer rounded to 2^-F, F = 24 / 22 / 20
// for k = 3 / 5 / 7) below a count of its samples still to come; the adds
// commute, so the result does not depend on their order, and the add that
// takes the count to zero writes the mean in place.  A fragment without
// edge samples writes its mean at once, and one outside the shared block
// (below) walks its own samples, so no second pass is needed.  For k = 1
// there is nothing to add and the answers are stored as floats
// (rsmss_filter's bits, and its kernel on large calls).  Because the answers do not depend on the order of
// the work, the warps of a CTA share its strips as they come free.
#include <cuda_runtime.h>

#include <cstdint>

#include "rbsm.h"
#include "rbsm_device.cuh"
#include "rbsm_host.h"

namespace rbsm {
namespace {

// One CTA of 32 warps per SM for k > 1 (two of 16 warps: 143.8 against 134.5
// us at k = 3, four of 8: 159.7; the larger the CTA, the more strips its
// warps share out; 3840x2160 fragments), and for k = 1, whose kernel fits 48
// registers, two of 20: it gets calls of fewer than 32 tiles of 128 per SM
// (rpcf_entry), where five of 8 and one of 32 come out about as well (320x240 /
// 480x270 / 640x480 / 960x540 fragments, with a texture: 7.2 / 8.3 / 11.2 / 14.1 us with
// two of 20, 7.2 / 7.6 / 11.7 / 14.7 with five of 8, 7.3 / 8.0 / 11.3 / 14.1 with one of
// 32).
template <int K>
constexpr int kRpcfThreads = K == 1 ? 640 : 1024;

// The fixed-point layout of a pending fragment: F fraction bits per sample
// answer, the sum (at most K^2 * 2^F) below bit kCount, and the number of
// samples still to be added at bits kCount..31 (at most K^2):
// k = 3: 9 * 2^24 < 2^28, 9 < 2^4;  k = 5: 25 * 2^22 < 2^27, 25 < 2^5;
// k = 7: 49 * 2^20 < 2^26, 49 < 2^6.  A sample answer is off by at most
// 2^-(F+1), far inside the 1e-5 bar.
template <int K>
struct FixLayout {
    static constexpr int kFrac = K == 3 ? 24 : K == 5 ? 22 : 20;
    static constexpr int kCount = K == 3 ? 28 : K == 5 ? 27 : 26;
    static_assert((unsigned long long)(K * K) << kFrac < (1ull << kCount), "sum overflows into the count");
    static_assert(K * K < (1 << (32 - kCount)), "count overflows");
};
// Edge samples are queued per fragment element: for k <= 3 all of a lane's
// edge samples at once (a warp prefix sum places them), so the queue holds
// < 32 left over + k^2 samples of every lane; for larger k each lane's
// lowest remaining one per round (a ballot each), < 32 + 32.
template <int K>
struct RpcfQueue {
    static constexpr int kCap = K <= 3 ? 32 * K * K + 32 : 64;
    EdgeEntry q[kCap];
};

// A queued sample's number: for k = 3 its bit in the packed 5 x 5 block
// word (row y at bits 5y..5y+4, sample (a, b) at block (a + 2, b + 2)), for
// larger k its index (b + R) * K + (a + R) among the k x k samples.  A k = 3
// entry holds the number in bits 0-4 and the fragment's block word above it.
template <int K>
__device__ __forceinline__ int sample_slot(int q)
{
    return K == 3 ? (q / 3 + 1) * 5 + q % 3 + 1 : q;
}

template <int K>
__device__ __forceinline__ int sample_dx(int slot)
{
    return K == 3 ? slot % 5 - 2 : slot % K - (K - 1) / 2;
}

template <int K>
__device__ __forceinline__ int sample_dy(int slot)
{
    return K == 3 ? slot / 5 - 2 : slot / K - (K - 1) / 2;
}

template <int K>
__device__ __forceinline__ uint32_t to_fix(float v)
{
    return (uint32_t)__float2uint_rn(__fmul_rn(v, (float)(1u << FixLayout<K>::kFrac)));
}

// The mean of k^2 sample answers from their fixed-point sum.
template <int K>
__device__ __forceinline__ float mean_of(uint32_t sum)
{
    return __fdiv_rn(__fmul_rn(__uint2float_rn(sum), 1.0f / (float)(1u << FixLayout<K>::kFrac)), (float)(K * K));
}

// The same for a fragment without edge samples, whose answers are its c lit
// samples: c / k^2.  For k = 3, c * RN(1/9) rounds to RN(c / 9) for every
// c in 0..9 (checked for each c), so a multiply gives the division's bits.
template <int K>
__device__ __forceinline__ float mean_of_lit(uint32_t c)
{
    if (K == 3)
        return __fmul_rn((float)c, 1.0f / 9.0f);
    return __fdiv_rn((float)c, (float)(K * K));
}

// The shared block.  Sample (a, b)'s texel is clamp(floor(u + a)) with u + a
// rounded to float; when every such floor is floor(u) + a (u + a can round
// up to the next integer where it crosses a power of two) and the (K + 2)^2
// block of texels around floor(u), floor(v) lies inside the map (no
// clamping), all K^2 samples' four-neighbourhoods come from that one block:
// 7 texture gathers for k = 3 and ceil((K + 2) / 2)^2 for larger k instead
// of 2 K^2, and one shadow test (Eq. 1) per texel.  Other fragments take the
// per-sample path.
template <int K>
__device__ __forceinline__ bool block_ok(float u, float v, float uhi, float vhi)
{
    constexpr int R = (K - 1) / 2;
    const float fu = floorf(u), fv = floorf(v);
    bool ok = fu >= (float)(R + 1) && fu <= uhi && fv >= (float)(R + 1) && fv <= vhi;    // false for NaN
    // Only the sums can round: for 2 <= u < 2^16 (maps are at most 65536
    // texels wide) and d <= R, u - d is exact (a result at or above the
    // binade of u keeps its spacing, one below it has a finer one), so
    // floor(u - d) is floor(u) - d.
#pragma unroll
    for (int d = 1; d <= R; ++d)
        ok = ok && floorf(__fadd_rn(u, (float)d)) == fu + (float)d && floorf(__fadd_rn(v, (float)d)) == fv + (float)d;
    return ok;
}

// Shadow tests (Eq. 1) as sign bits: the sign of z + np is set where pz > z,
// with np = 0 - pz.  The sum of two floats is negative exactly when pz > z (it
// is never rounded to zero), equal operands give +0 (np is never -0, so a z of
// -0 does too), and a NaN sum (NaN operands, or equal infinities) is the
// canonical one, whose sign is clear, as the comparison is false.  The sums
// run on the FMA pipe and a funnel shift takes two signs at a time, where
// comparisons and selections kept the ALU pipe 70 % busy: 134.5 against 127.3
// us, k = 3, 3840x2160 fragments (k = 5: 291 against 287).
__device__ __forceinline__ uint32_t shadow_bit(float z, float np)
{
    return __float_as_uint(__fadd_rn(z, np)) >> 31;
}

// Bit 0: texel lo is shadowed, bit 1: texel hi.
__device__ __forceinline__ uint32_t shadow_bits2(float lo, float hi, float np)
{
    return __funnelshift_l(__float_as_uint(__fadd_rn(lo, np)), shadow_bit(hi, np), 1);
}

// The block's texels are (floor(u) - R - 1 + x, floor(v) - R - 1 + y).  The
// samples' classification reads the block without its four corners (each
// sample's texel and its four neighbours); bits of the corners may hold
// anything, nothing reads them.  A gather at (X, Y) covers columns X - 1, X
// and rows Y - 1, Y; components x = (lo col, hi row), y = (hi, hi), z = (hi,
// lo), w = (lo, lo).
//
// k = 3: the whole block in one word, bit 5y + x lit: 21 texels, which seven
// gathers cover (rows 0-1 at columns 0-3, rows 3-4 at columns 1-4, and three
// across the middle row).
__device__ __forceinline__ uint32_t block_word3(const MapDev &m, float u, float v, float pz)
{
    const float np = __fsub_rn(0.0f, pz);
    uint32_t s = 0;
    if (m.tex) {
        const float gx = floorf(u) - 1.0f, gy = floorf(v) - 1.0f;
        auto gather = [&](int p, int q) { return tex2Dgather<float4>(m.tex, gx + (float)p, gy + (float)q, 0); };
        float4 g = gather(0, 0);
        s += shadow_bits2(g.w, g.z, np) + (shadow_bits2(g.x, g.y, np) << 5);
        g = gather(2, 0);
        s += (shadow_bits2(g.w, g.z, np) << 2) + (shadow_bits2(g.x, g.y, np) << 7);
        g = gather(1, 3);
        s += (shadow_bits2(g.w, g.z, np) << 16) + (shadow_bits2(g.x, g.y, np) << 21);
        g = gather(3, 3);
        s += (shadow_bits2(g.w, g.z, np) << 18) + (shadow_bits2(g.x, g.y, np) << 23);
        g = gather(0, 2);
        s += (shadow_bits2(g.w, g.z, np) << 10) + (shadow_bit(g.x, np) << 15);
        g = gather(1, 1);
        s += shadow_bit(g.y, np) << 12;
        g = gather(3, 1);
        s += (shadow_bit(g.z, np) << 9) + (shadow_bits2(g.x, g.y, np) << 13);
    } else {
        // plain loads (1279x717 fragments: 61.7 us against 99 us when each
        // lane classified and walked its fragment's samples one by one)
        const float *row = m.depth + (long long)((int)floorf(v) - 2) * m.pitch + ((int)floorf(u) - 2);
#pragma unroll
        for (int y = 0; y < 5; ++y) {
#pragma unroll
            for (int x = 0; x < 5; ++x)
                s |= shadow_bit(__ldg(row + x), np) << (5 * y + x);
            row += m.pitch;
        }
    }
    return ~s & 0x1ffffffu;
}

// Larger k: bit x of rows[y] lit, the whole block by ceil((K + 2) / 2)^2
// gathers.
template <int K>
__device__ __forceinline__ void block_bits(const MapDev &m, float u, float v, float pz, uint32_t (&rows)[K + 2])
{
    constexpr int R = (K - 1) / 2, B = K + 2, G = (B + 1) / 2;
    const float np = __fsub_rn(0.0f, pz);
#pragma unroll
    for (int y = 0; y < B; ++y)
        rows[y] = 0u;
    if (m.tex) {
        const float gx = floorf(u) - (float)R, gy = floorf(v) - (float)R;
#pragma unroll
        for (int n = 0; n < G; ++n) {
#pragma unroll
            for (int c = 0; c < G; ++c) {
                const float4 g = tex2Dgather<float4>(m.tex, gx + (float)(2 * c), gy + (float)(2 * n), 0);
                rows[2 * n] |= shadow_bits2(g.w, g.z, np) << (2 * c);
                if (2 * n + 1 < B)
                    rows[2 * n + 1] |= shadow_bits2(g.x, g.y, np) << (2 * c);
            }
        }
    } else {
        const float *row = m.depth + (long long)((int)floorf(v) - R - 1) * m.pitch + ((int)floorf(u) - R - 1);
#pragma unroll
        for (int y = 0; y < B; ++y) {
#pragma unroll
            for (int x = 0; x < B; ++x)
                rows[y] |= shadow_bit(__ldg(row + x), np) << x;
            row += m.pitch;
        }
    }
#pragma unroll
    for (int y = 0; y < B; ++y)
        rows[y] = ~rows[y];
}

// Persistent warps work on strips of 32 consecutive fragments, one per lane.
// A CTA owns every gridDim.x-th run of kRun strips (its warps' loads stay
// near each other), and its warps take them one at a time from a counter in
// shared memory, so that a strip along a shadow edge, whose samples all walk,
// holds up one warp while the others take the strips after it.
//
// Bound: the texture path's write-back of the block's gathers (7 for k = 3,
// about 16 cycles each for a warp: 92 us of a 3840x2160 frame), then the
// rounds of the longest walks.  A warp used to own a tile of 128 fragments
// (up to 1152 samples, 36 rounds, at k = 3), and the tiles came from a fixed
// partition or one at a time from a global counter; 3840x2160 fragments on
// an 8192^2 map, k = 3 / 5: 179 / 488 us with tiles from the counter, 128.7 /
// 288 us now.
constexpr unsigned kRun = 8;       // 16: 161.7 against 159.7 us, and 48 against 32.4 us for 320x240 fragments

template <int K, int kThreads>
__global__ void __launch_bounds__(kThreads, K == 1 ? 2 : 1)
rpcf_kernel(const MapDev m, const float *__restrict__ x, const float *__restrict__ y,
            const float *__restrict__ z, long long n, float *__restrict__ vis, int max_dist)
{
    constexpr int kWarps = kThreads / 32;
    constexpr int R = (K - 1) / 2;
    __shared__ RpcfQueue<K> wq[kWarps];
    __shared__ unsigned next;                  // strips of this CTA taken
    if (threadIdx.x == 0)
        next = kWarps;
    __syncthreads();
    const unsigned lane = lane_id();
    const unsigned below = (1u << lane) - 1u;
    // the warp's index through a shuffle: the compiler then knows that the
    // strip and what follows from it are the same on all lanes
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
    const long long strips = (n + 31) / 32;
    // strip number k of this CTA
    auto strip_of = [&](unsigned k) {
        return (long long)(k / kRun) * ((long long)gridDim.x * kRun) + (long long)blockIdx.x * kRun + k % kRun;
    };
    long long strip = strip_of((unsigned)warp);
    if (strip >= strips)
        return;
    const float W = (float)m.width, H = (float)m.height;
    // the largest floor(u), floor(v) whose block lies inside the map
    const float uhi = (float)(m.width - R - 2), vhi = (float)(m.height - R - 2);
    uint32_t *acc = reinterpret_cast<uint32_t *>(vis);
    // drain rounds of 32 queued edge samples: walk, answer, add
    auto drain = [&](int &queued, bool all) {
        while (queued >= 32 || (all && queued > 0)) {
            __syncwarp();                  // entries and the fragments' base values are visible
            const int base = queued >= 32 ? queued - 32 : 0;
            const int q = base + (int)lane;
            if (q < queued) {
                const EdgeEntry e = wq[warp].q[q];
                const uint32_t i = e.idx;
                const int sample = K == 3 ? (int)(e.bits_job & 31u) : (int)e.bits_job;
                const float ua = __fadd_rn(__fmul_rn(__ldg(x + i), W), (float)sample_dx<K>(sample));
                const float vb = __fadd_rn(__fmul_rn(__ldg(y + i), H), (float)sample_dy<K>(sample));
                const float pz = __ldg(z + i);
                FragResult r{0.0f, 0.0f, 0};
                uint32_t bits;
                if (K == 3) {
                    // the entry carries the fragment's block word: the
                    // sample's shadow test and its four neighbours' (left,
                    // right one bit away, +y, -y five bits away) are bits of
                    // it, taken with the same depth from the same texels
                    const uint32_t P = e.bits_job >> 5;
                    const uint32_t s0 = (P >> sample) & 1u;
                    bits = s0 | ((((P >> (sample - 1)) & 1u) ^ s0) << 1) | ((((P >> (sample + 1)) & 1u) ^ s0) << 2) |
                           ((((P >> (sample + 5)) & 1u) ^ s0) << 3) | ((((P >> (sample - 5)) & 1u) ^ s0) << 4);
                } else {
                    classify_uv<2, false>(m, ua, vb, pz, r, bits);    // the sample's discontinuity again
                }
                resolve_edge_uv<2>(m, ua, vb, pz, bits, max_dist, r);
                if (K == 1) {
                    vis[i] = r.fil;
                } else {
                    // queued samples come from fragments inside the shared
                    // block (finite coordinates), whose answers are finite
                    constexpr int C = FixLayout<K>::kCount;
                    const uint32_t add = to_fix<K>(r.fil) - (1u << C);    // one sample fewer to come
                    const uint32_t old = atomicAdd(acc + i, add);
                    if ((old >> C) == 1u)                                  // the fragment's last sample
                        vis[i] = mean_of<K>((old + add) & ((1u << C) - 1u));
                }
            }
            __syncwarp();                  // entries read before they are overwritten
            queued = base;
        }
    };
    int queued = 0;
    float xn = 0.0f, yn = 0.0f, zn = 0.0f;         // this lane's fragment of the next strip
    auto load = [&](long long st) {
        const long long f = st * 32 + lane;
        if (f < n) {
            xn = __ldcs(x + f);
            yn = __ldcs(y + f);
            zn = __ldcs(z + f);
        }
    };
    load(strip);
    for (;;) {
        unsigned k = 0;
        if (lane == 0)
            k = atomicAdd(&next, 1u);
        const long long ns = strip_of(__shfl_sync(0xffffffffu, k, 0));
        const bool more = ns < strips;
        const float xe = xn, ye = yn, ze = zn;
        const long long frag = strip * 32 + lane;
        const bool valid = frag < n;
        if (more)
            load(ns);                      // the next strip's loads fly during this one
        const float u = __fmul_rn(xe, W), v = __fmul_rn(ye, H);
        // all samples' texel reads first; off-edge samples add their
        // shadow test to the base value, edge samples set their bit
        uint64_t edges = 0;
        uint32_t base = 0, block = 0;
        float single = 0.0f;
        const bool base_path = K > 1 && valid && block_ok<K>(u, v, uhi, vhi);
        if (base_path) {
            // sample (a, b)'s texel is block (a + R + 1, b + R + 1); it is an
            // edge sample where one of Listing 2's four neighbours differs
            // from it, else it adds its shadow test
            if constexpr (K == 3) {
                // a sample differs from a neighbour one bit (left, right) or
                // five bits (below, above) away, so the four comparisons of
                // Listing 2 cover all nine samples at once
                const uint32_t P = block_word3(m, u, v, ze);
                constexpr uint32_t kSamples = (7u << 6) | (7u << 11) | (7u << 16);   // rows 1-3, columns 1-3
                const uint32_t e = ((P ^ (P >> 1)) | (P ^ (P << 1)) | (P ^ (P >> 5)) | (P ^ (P << 5))) & kSamples;
                edges = e;
                block = P;
                base = (uint32_t)__popc(P & ~e & kSamples) << FixLayout<K>::kFrac;
            } else {
                // a row of samples at once
                uint32_t rows[K + 2];
                block_bits<K>(m, u, v, ze, rows);
                constexpr uint32_t mk = (1u << K) - 1u;
#pragma unroll
                for (int b = 0; b < K; ++b) {
                    const uint32_t c = (rows[b + 1] >> 1) & mk;
                    const uint32_t e = (c ^ (rows[b + 1] & mk)) | (c ^ ((rows[b + 1] >> 2) & mk)) |
                                       (c ^ ((rows[b + 2] >> 1) & mk)) | (c ^ ((rows[b] >> 1) & mk));
                    edges |= (uint64_t)e << (K * b);
                    base += (uint32_t)__popc(c & ~e) << FixLayout<K>::kFrac;
                }
            }
        } else if (K == 1) {
            FragResult r{0.0f, 0.0f, 0};
            uint32_t bits = 0;
            if (valid && classify_uv<2, false>(m, u, v, ze, r, bits))
                edges = 1ull << sample_slot<K>(0);
            single = r.fil;
        } else if (valid) {
            // outside the shared block (the map's border rows and
            // columns, or a non-finite coordinate): the lane walks its
            // own edge samples and writes the mean (rare, so the
            // divergence costs little)
            uint32_t sum = 0;
            bool nan = false;
#pragma unroll 1
            for (int q = 0; q < K * K; ++q) {
                FragResult r{0.0f, 0.0f, 0};
                uint32_t bits = 0;
                const float ua = __fadd_rn(u, (float)(q % K - R)), vb = __fadd_rn(v, (float)(q / K - R));
                if (classify_uv<2, false>(m, ua, vb, ze, r, bits))
                    resolve_edge_uv<2>(m, ua, vb, ze, bits, max_dist, r);
                if (r.fil != r.fil)
                    nan = true;               // a NaN answer (NaN or infinite coordinates)
                else
                    sum += to_fix<K>(r.fil);
            }
            vis[frag] = nan ? __int_as_float(0x7fc00000) : mean_of<K>(sum);
        }
        // the base value is stored before any deferred sample of this
        // fragment can add to it ...
        const uint32_t ne = (uint32_t)__popcll(edges);
        if (valid) {
            if (K == 1)
                vis[frag] = single;
            else if (ne != 0)
                acc[frag] = (ne << FixLayout<K>::kCount) | base;
            else if (base_path)
                vis[frag] = mean_of_lit<K>(base >> FixLayout<K>::kFrac);
        }
        // ... then the edge samples are queued and walked whenever 32
        // are waiting
        if (K <= 3) {
            // all of the lane's edge samples, placed by a prefix sum
            uint32_t incl = ne, total = 0;
            if (__any_sync(0xffffffffu, ne != 0)) {      // about one element in five has none
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const uint32_t t2 = __shfl_up_sync(0xffffffffu, incl, off);
                    if ((int)lane >= off)
                        incl += t2;
                }
                total = __shfl_sync(0xffffffffu, incl, 31);
            }
            if (total != 0u) {
                int pos = queued + (int)(incl - ne);
                uint64_t rest = edges;
                while (rest) {
                    const int q = __ffsll((long long)rest) - 1;
                    rest &= rest - 1;
                    wq[warp].q[pos++] = EdgeEntry{(uint32_t)(frag), K == 3 ? (block << 5) | (uint32_t)q : (uint32_t)q};
                }
                queued += (int)total;
                drain(queued, false);
            }
        } else {
            // each lane's lowest remaining edge sample per round: as many
            // rounds as the most edge samples of any lane's fragment
            uint64_t rest = edges;
            while (__any_sync(0xffffffffu, rest != 0)) {
                const bool has = rest != 0;
                const unsigned mask = __ballot_sync(0xffffffffu, has);
                if (has) {
                    const int q = __ffsll((long long)rest) - 1;
                    rest &= rest - 1;
                    wq[warp].q[queued + __popc(mask & below)] = EdgeEntry{(uint32_t)(frag), (uint32_t)q};
                }
                queued += __popc(mask);
                drain(queued, false);
            }
        }
        if (!more)
            break;
        strip = ns;
    }
    drain(queued, true);
}

template <int K>
int launch_rpcf(const rbsm_map &map, const rbsm_frags &f, float *vis, int max_dist, cudaStream_t stream)
{
    auto kern = rpcf_kernel<K, kRpcfThreads<K>>;
    static KernelSetup setup;
    int occupancy = 0;
    int rc = setup.get(kern, kRpcfThreads<K>, 0, &occupancy);
    if (rc != RBSM_OK)
        return rc;
    const int sms = device_sm_count();
    if (sms <= 0)
        return cuda_fail(cudaErrorNoDevice);
    const long long strips = (f.n + 31) / 32;
    const long long blocks_needed = (strips + kRun - 1) / kRun;
    long long grid = (long long)sms * occupancy;
    if (grid > blocks_needed)
        grid = blocks_needed;
    kern<<<(unsigned)grid, kRpcfThreads<K>, 0, stream>>>(to_dev(map), f.x, f.y, f.z, f.n, vis, max_dist);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return cuda_fail(e);
    return RBSM_OK;
}

}  // namespace
}  // namespace rbsm

namespace rbsm {
namespace {

// ws: the caller's workspace, checked and not used (nullptr: none)
int rpcf_entry(const rbsm_map *map, const rbsm_frags *frags, float *vis, int32_t k, const rbsm_params *params,
               const void *ws, void *stream)
{
    int rc, max_dist;
    if ((rc = check_map(map)) != RBSM_OK) return rc;
    if ((rc = check_frags(frags)) != RBSM_OK) return rc;
    if ((rc = check_params(params, &max_dist)) != RBSM_OK) return rc;
    if (k < 1 || k > RBSM_RPCF_MAX_K || (k & 1) == 0)
        return RBSM_ERR_ARG;
    if (frags->n > 0 && !vis)
        return RBSM_ERR_ARG;
    if ((reinterpret_cast<uintptr_t>(vis) & 3u) != 0)
        return RBSM_ERR_ARG;
    if (frags->n == 0)
        return RBSM_OK;
    // vis holds partial sums while the kernel runs: it must not overlap an input
    if (overlaps_inputs(*map, *frags, vis, (size_t)frags->n * 4u))
        return RBSM_ERR_ARG;
    if (ws && (overlaps_inputs(*map, *frags, ws, 8) ||
               (reinterpret_cast<uintptr_t>(ws) < reinterpret_cast<uintptr_t>(vis) + (uintptr_t)frags->n * 4u &&
                reinterpret_cast<uintptr_t>(vis) < reinterpret_cast<uintptr_t>(ws) + 8u)))
        return RBSM_ERR_ARG;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    // k = 1 is rsmss_filter: with tiles enough for CTAs of 1024 its kernel
    // (3840x2160 / 1277x719 fragments 47.0 / 14.9 against 57.6 / 16.5 us here;
    // 3840x2160 without a texture 66.6 against 75.8); on fewer fragments one
    // strip per warp finishes sooner (320x240 / 640x480 / 960x540 7.2 / 11.2 / 14.1
    // us here, 10.4 / 12.0 / 14.9 with its CTAs of 256)
    if (k == 1 && plain_large(frags->n, device_sm_count()))
        return plain_entry(RBSM_MODE_FILTER, map, frags, vis, nullptr, params, stream);
    switch (k) {
    case 1: return launch_rpcf<1>(*map, *frags, vis, max_dist, s);
    case 3: return launch_rpcf<3>(*map, *frags, vis, max_dist, s);
    case 5: return launch_rpcf<5>(*map, *frags, vis, max_dist, s);
    default: return launch_rpcf<7>(*map, *frags, vis, max_dist, s);
    }
}

}  // namespace
}  // namespace rbsm

extern "C" int rbsm_rpcf(const rbsm_map *map, const rbsm_frags *frags, float *vis, int32_t k,
                         const rbsm_params *params, void *stream)
{
    return rbsm::rpcf_entry(map, frags, vis, k, params, nullptr, stream);
}

extern "C" int rbsm_rpcf_ws(const rbsm_map *map, const rbsm_frags *frags, float *vis, int32_t k,
                            const rbsm_params *params, void *workspace, void *stream)
{
    if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 7u) != 0)
        return RBSM_ERR_ARG;
    return rbsm::rpcf_entry(map, frags, vis, k, params, workspace, stream);
}
