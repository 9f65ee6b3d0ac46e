// Device-side steps of the RBSM per-fragment path for sm_103a.
//
// Per fragment: texel and in-texel offsets (float32, as the paper's GLSL),
// shadow test of the texel and of its four neighbours (Eq. 1, Eq. 2),
// discontinuity directions (Eqs. 3-4).  Fragments off the shadow edge are
// finished there (the plain shadow test, Listing 1).  Edge fragments walk the
// edge (Listing 3), normalise their position (Eq. 5) and take the optimized
// visibility (Listing 4 and/or Listing 5).
//
// Work unit: a warp tile of 128 consecutive fragments (below).  Edge
// fragments of a tile are compacted so that their long, data-dependent walks
// run on adjacent lanes instead of serialising all four fragments of a lane.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace rbsm {

constexpr int kPerThread = 4;

struct MapDev {
    const float *depth;
    int32_t width;
    int32_t height;
    long long pitch;
    cudaTextureObject_t tex;     // 0 = none (plain loads)
};

// Nearest texel with clamp-to-edge addressing; read through the read-only
// (L1-cached) path because neighbouring fragments reuse the same texels.
__device__ __forceinline__ float texel(const MapDev &m, int i, int j)
{
    i = min(max(i, 0), m.width - 1);
    j = min(max(j, 0), m.height - 1);
    return __ldg(m.depth + (long long)j * m.pitch + i);
}

// Eq. 1: 0 (shadowed) when the stored blocker is nearer the light than the
// fragment, 1 otherwise.  No bias.
__device__ __forceinline__ int shadow_test(float pz, float zt)
{
    return pz > zt ? 0 : 1;
}

// Texel and in-texel offset of a texel-space position u along one axis:
// t = clamp(floor(u)), f = u - floor(u) (float32, as the paper's GLSL).
__device__ __forceinline__ void texel_of(float u, int size, int &t, float &f)
{
    float fu = floorf(u);
    f = __fsub_rn(u, fu);
    float c = fminf(fmaxf(fu, 0.0f), (float)(size - 1));
    t = (int)c;
}

// The same from a texture coordinate: u = x * size.
__device__ __forceinline__ void texel_coord(float x, int size, int &t, float &f)
{
    texel_of(__fmul_rn(x, (float)size), size, t, f);
}

// Listing 3, the four walks of an edge fragment.  A texel of a walk continues
// the edge when it keeps the fragment's shadow-test result and shares a
// discontinuity direction with the fragment.  Along x only the +-y
// directions can be shared: the walk's texel has the same result as the
// texel it came from (so no shared direction back along the walk), and the
// fragment has no discontinuity in the walking direction (else the first
// step ends the walk).  Both facts hold with clamp-to-edge addressing too;
// along y the same holds with the axes swapped.  A walk returns +k for an
// end found at step k, -k for a texel that left the edge, -(max_dist+1) when
// all steps continued.
//
// The fragment's own discontinuities settle every walk but two at most.  A
// walk in a direction with a discontinuity ends at its first texel (+1); one
// along an axis without a discontinuity across it leaves the edge there
// (-1).  Of the directions left, a straight edge keeps the two along it, a
// corner one on each axis, a dead end one, and a texel on its own none.  So a
// lane has two walks, A and B, each with its own step and side, and a drain
// round of 32 fragments runs one loop as long as its longest walk, whatever
// axes its lanes walk along (one loop per axis made a round as long as its
// longest x walk and its longest y walk together).
//
// A walk reads its own line and the side line that shares the direction, at
// a fixed offset from it (both side lines where both are in use, a thin
// feature: the second one in a branch that most rounds skip).  A side is only read
// when the fragment has a discontinuity towards it, and at the map border
// the clamped neighbour is the texel itself and shows none, so a side that
// is read exists.  A walk that reaches the border stays on its texel (clamp
// to edge), which continues the edge, for the steps that are left: it finds
// no end, so it is stopped there.  The loads of a step, of both walks, are in
// flight before the first test.  Loads of later steps are not issued ahead
// while most walks are still on: the extra, mostly wasted, requests cost more
// than the latency they hide (two steps per iteration with their loads
// together: 67.2 against 60.7 us on one 3840x2160 frame).  With PAIRS the
// steps after the second, which few walks reach but those take many of, go
// two at a time: silhouette, 1920x1080, 22.1 -> 20.1 us, filtering, 3840x2160,
// 52.5 -> 51.8 in the single-map kernel at 64 registers; the kernels at 48
// spill with it (cascades 369 -> 380 us) and take single steps.
//
// Bound: the latency of the steps and the issue slots of a round's longest
// walk.  rsmss_filter, 3840x2160 fragments on a 4096^2 map, 5 % of them on
// edges: 76.2 us with one loop per axis, 60.7 us with this one (41 us
// without any walk); 64 jobs of cascades in one launch: 504 against 433 us.
// Measured against it, the same answers: the warp taking the open walks of a
// round one pair at a time, 16 steps of each across its lanes (two ballots
// settle a pair): 76 us when at most 8 walks are left open, 97 at 16; and
// texture gathers, two steps each: 63.6 us, and 525 on the cascades.
struct EdgeWalk {
    const float *p;                // the texel reached
    long long step, side;          // to the next texel, and to the side line's texel
    int last;                      // the last step to take; 0 = the walk is done
};

__device__ __forceinline__ EdgeWalk edge_walk(const MapDev &m, const float *p, int i, int j, unsigned d, unsigned d4,
                                              int max_dist)
{
    // directions as the bits of d4: 0 left, 1 right, 2 +y, 3 -y
    const bool vert = d >= 2u, up = d == 1u || d == 2u;
    const long long along = vert ? m.pitch : 1, across = vert ? 1 : m.pitch;
    EdgeWalk w;
    w.p = p;
    w.step = up ? along : -along;
    // sides: the rows j + 1, j - 1 of a walk along x, the columns i + 1, i - 1 of one along y
    w.side = (d4 & (vert ? 2u : 4u)) ? across : -across;
    const int room = vert ? (up ? m.height - 1 - j : j) : (up ? m.width - 1 - i : i);
    w.last = min(room, max_dist);
    return w;
}

// Walk results of the fragment at texel (i, j): rxn, rxp along x towards
// lower and higher columns, ryn, ryp along y towards lower and higher rows.
// Returns the step at which the last of the four ends (max_dist + 1 when one
// does not).
template <bool PAIRS>
__device__ __forceinline__ int edge_walks(const MapDev &m, int i, int j, float pz, bool lit, unsigned d4,
                                           int max_dist, int &rxn, int &rxp, int &ryn, int &ryp)
{
    const unsigned open = (((d4 & 12u) ? 3u : 0u) | ((d4 & 3u) ? 12u : 0u)) & ~d4;
    const unsigned lo = open & (0u - open), hi = open & ~lo;       // walk A's direction, walk B's (or none)
    const bool two = (d4 & 3u) == 3u || (d4 & 12u) == 12u;         // both side lines in use
    const float *p = m.depth + (long long)j * m.pitch + i;
    EdgeWalk A = edge_walk(m, p, i, j, __ffs(lo) - 1, d4, max_dist);
    EdgeWalk B = edge_walk(m, p, i, j, __ffs(hi) - 1, d4, max_dist);
    if (lo == 0u)
        A.last = 0;
    if (hi == 0u)
        B.last = 0;
    int ra = -(max_dist + 1), rb = ra;
    // step k of both walks from the texels and side texels read for it
    auto test = [&](int k, bool a, bool b, float la, float lb, float sa, float sb) {
        // a texel's test differs from the fragment's: the walk's texel (the
        // walk ends), its side texel (the walk continues the edge)
        const bool ea = (pz > la) == lit, eb = (pz > lb) == lit;
        bool ca = (pz > sa) == lit, cb = (pz > sb) == lit;
        if (two) {
            if (a && !ca)
                ca = (pz > __ldg(A.p - A.side)) == lit;
            if (b && !cb)
                cb = (pz > __ldg(B.p - B.side)) == lit;
        }
        if (a && (ea || !ca)) {
            ra = ea ? k : -k;
            A.last = 0;
        }
        if (b && (eb || !cb)) {
            rb = eb ? k : -k;
            B.last = 0;
        }
    };
    int k = 1;
    for (; !PAIRS || k <= 2; ++k) {
        const bool a = k <= A.last, b = k <= B.last;
        if (!a && !b)
            break;
        A.p += A.step;
        B.p += B.step;
        const float la = a ? __ldg(A.p) : 0.0f;
        const float lb = b ? __ldg(B.p) : 0.0f;
        const float sa = a ? __ldg(A.p + A.side) : 0.0f;
        const float sb = b ? __ldg(B.p + B.side) : 0.0f;
        test(k, a, b, la, lb, sa, sb);
    }
    for (; PAIRS && (k <= A.last || k <= B.last); k += 2) {
        const float *pa = A.p + A.step, *pb = B.p + B.step;
        const bool a1 = k <= A.last, b1 = k <= B.last, a2 = k < A.last, b2 = k < B.last;
        const float la1 = a1 ? __ldg(pa) : 0.0f, sa1 = a1 ? __ldg(pa + A.side) : 0.0f;
        const float lb1 = b1 ? __ldg(pb) : 0.0f, sb1 = b1 ? __ldg(pb + B.side) : 0.0f;
        const float la2 = a2 ? __ldg(pa + A.step) : 0.0f, sa2 = a2 ? __ldg(pa + A.step + A.side) : 0.0f;
        const float lb2 = b2 ? __ldg(pb + B.step) : 0.0f, sb2 = b2 ? __ldg(pb + B.step + B.side) : 0.0f;
        A.p = pa;
        B.p = pb;
        test(k, a1, b1, la1, lb1, sa1, sb1);
        A.p += A.step;
        B.p += B.step;
        test(k + 1, k + 1 <= A.last, k + 1 <= B.last, la2, lb2, sa2, sb2);
    }
    rxn = lo == 1u ? ra : (d4 & 1u) ? 1 : -1;
    rxp = lo == 2u ? ra : hi == 2u ? rb : (d4 & 2u) ? 1 : -1;
    ryp = lo == 4u ? ra : hi == 4u ? rb : (d4 & 4u) ? 1 : -1;
    ryn = lo == 8u ? ra : hi == 8u ? rb : (d4 & 8u) ? 1 : -1;
    return max(lo ? abs(ra) : 1, hi ? abs(rb) : 1);
}

// Eq. 5 and the normalisation along one axis: the position of the fragment
// measured from the end that was found, over the length of the aliased edge
// along that axis (|r_neg| + |r_pos| - 1 texels).  With no end found the
// position is 1.  The both-ends position is never read by Listings 4 and 5.
__device__ __forceinline__ float axis_position(int r_neg, int r_pos, float f)
{
    int len = abs(r_neg) + abs(r_pos) - 1;
    if (r_neg > 0 && r_pos <= 0)
        return __fdiv_rn(__fadd_rn((float)(r_neg - 1), f), (float)len);
    if (r_pos > 0 && r_neg <= 0)
        return __fdiv_rn(__fadd_rn((float)(r_pos - 1), __fsub_rn(1.0f, f)), (float)len);
    return 1.0f;
}

// Listing 4 (§4.1).  dx3/dy3: edges on both sides of the axis (d == 0.75);
// ex/ey: ends found along each axis (Eq. 5 code + 1).
__device__ __forceinline__ float silhouette(bool dx3, bool dy3, int ex, int ey, float nx, float ny)
{
    if (dx3 || dy3)
        return 0.0f;                        // short U / O
    if (ex == 2 || ey == 2)
        return 0.0f;                        // long U / O
    if (ex == 0 || ey == 0)
        return 1.0f;                        // I
    return ny < __fsub_rn(1.0f, nx) ? 0.0f : 1.0f;   // L: step(1 - nx, ny)
}

// Listing 5 (§4.2); dz = 1 - s.  The sign factor is +-1, applied as an
// exact negation.
__device__ __forceinline__ float filter(bool dx3, bool dy3, int dz, int ex, int ey, float nx, float ny)
{
    float z = (float)dz;
    float sx = dz ? -nx : nx;
    float sy = dz ? -ny : ny;
    if (dx3 && dy3)
        return z;                           // short O
    if (ex == 2 && ey == 2)
        return z;                           // long O
    if (ex == 2)
        return __fadd_rn(z, sy);            // U open along y
    if (ey == 2)
        return __fadd_rn(z, sx);            // U open along x
    if (ex == 0 || ey == 0)
        return 1.0f - z;                    // I
    float v = __fadd_rn(__fadd_rn(z, sy), sx);   // L: clamp(v, 0, 1)
    v = v < 0.0f ? 0.0f : v;                      // comparisons keep a NaN a NaN
    return v > 1.0f ? 1.0f : v;
}

// Features of the learned surrogate (this project's addition; not in the paper).
// 5x5 shadow-test pattern and nearest blocker depth around texel (i, j)
// (clamp to edge): bit (dy+2)*5 + (dx+2) is set when texel (i+dx, j+dy) is
// lit for depth pz.
__device__ __forceinline__ void window5(const MapDev &m, int i, int j, float pz, uint32_t &bits, float &zmin)
{
    bits = 0;
    zmin = texel(m, i, j);
    int cols[5];
#pragma unroll
    for (int d = 0; d < 5; ++d)
        cols[d] = min(max(i + d - 2, 0), m.width - 1);
#pragma unroll
    for (int dy = 0; dy < 5; ++dy) {
        const float *row = m.depth + (long long)min(max(j + dy - 2, 0), m.height - 1) * m.pitch;
#pragma unroll
        for (int dx = 0; dx < 5; ++dx) {
            const float zt = __ldg(row + cols[dx]);
            bits |= (uint32_t)shadow_test(pz, zt) << (dy * 5 + dx);
            zmin = fminf(zmin, zt);
        }
    }
}

__device__ __forceinline__ void fragment_features(const MapDev &m, float x, float y, float pz, uint32_t &bits,
                                                  float &fx, float &fy, float &gap)
{
    int i, j;
    texel_coord(x, m.width, i, fx);
    texel_coord(y, m.height, j, fy);
    float zmin;
    window5(m, i, j, pz, bits, zmin);
    gap = __fsub_rn(pz, zmin);
}

// Whether the four Listing 3 walks from the fragment's texel stop inside its
// 5x5 window, read from the window's shadow-test pattern (bit (dy+2)*5 +
// (dx+2): texel (i+dx, j+dy) lit).  A walk along x goes on past step k when
// texel (k, 0) has the fragment's test and shares a discontinuity
// direction with the fragment's texel; along a continuing walk only the
// perpendicular directions can be shared (the +-y neighbours of (k, 0)
// against those of (0, 0)).  Steps 1 and 2 read only window texels, so when
// no walk goes on past step 2 (or max_dist <= 2) the exact answer is a
// function of the pattern and the in-texel offsets alone; otherwise it
// depends on texels the window does not hold.
__device__ __forceinline__ bool walks_inside_window(uint32_t pattern, int max_dist)
{
    if (max_dist <= 2)
        return true;
    const uint32_t s0 = (pattern >> 12) & 1u;
    // d[k] = bit k of "texel differs from the fragment's test"
    const uint32_t d = pattern ^ (s0 ? 0x1FFFFFFu : 0u);
    auto diff = [&](int dx, int dy) { return (d >> ((dy + 2) * 5 + (dx + 2))) & 1u; };
    const uint32_t up0 = diff(0, 1), dn0 = diff(0, -1), lf0 = diff(-1, 0), rt0 = diff(1, 0);
    auto goes_on_x = [&](int dx) { return !diff(dx, 0) && ((up0 & diff(dx, 1)) | (dn0 & diff(dx, -1))); };
    auto goes_on_y = [&](int dy) { return !diff(0, dy) && ((lf0 & diff(-1, dy)) | (rt0 & diff(1, dy))); };
    return !(goes_on_x(1) && goes_on_x(2)) && !(goes_on_x(-1) && goes_on_x(-2)) &&
           !(goes_on_y(1) && goes_on_y(2)) && !(goes_on_y(-1) && goes_on_y(-2));
}

// Result of one fragment (reach: the step its longest walk stopped at).
struct FragResult {
    float sil;
    float fil;
    uint16_t code;
    int reach = 0;
};

// Steps 1-2 from the five depths of the texel and its neighbours.
// (The tests stay predicates: a neighbour's discontinuity is its test
// differing from the centre's, and the answer is selected, not converted.)
template <int MODE, bool CODES>
__device__ __forceinline__ bool classify_from(float pz, float zc, float zl, float zr, float zu, float zd,
                                              FragResult &r, uint32_t &bits)
{
    const bool shadowed = pz > zc;             // Eq. 1: s0 = 0
    if (MODE == 1 && !CODES && shadowed) {
        r.sil = 0.0f;
        r.code = 0;
        bits = 0;
        return false;
    }
    const uint32_t dl = (pz > zl) != shadowed;
    const uint32_t dr = (pz > zr) != shadowed;
    const uint32_t du = (pz > zu) != shadowed;
    const uint32_t dd = (pz > zd) != shadowed;
    const uint32_t d4 = dl | (dr << 1) | (du << 2) | (dd << 3);
    bits = (shadowed ? 0u : 1u) | (d4 << 1);
    r.code = (uint16_t)(d4 | (shadowed ? 16u : 0u));
    const float sv = shadowed ? 0.0f : 1.0f;
    r.sil = sv;
    r.fil = sv;
    const bool edge = d4 != 0;
    if (MODE == 1)
        return edge && !shadowed;
    return edge;
}

// The texel of position (u, v) and its four neighbours through the map's
// texture.  Texel coordinates in float (clamp(floor(u)) is an integer-valued
// float, exact below 2^24), then two 2x2 gathers (point sampling, clamp to
// edge, unnormalised coordinates; the footprint of a gather at (u, v) is
// columns u-1, u and rows v-1, v): a at (i, j) columns i-1..i, rows j-1..j; b
// at (i+1, j+1) columns i..i+1, rows j..j+1.  Gather order: x = (lo col, hi
// row), y = (hi, hi), z = (hi, lo), w = (lo, lo), so the texel is a.y, its
// left, right, +y and -y neighbours a.x, b.z, b.x, a.z.
__device__ __forceinline__ void gather_cross(const MapDev &m, float u, float v, float4 &a, float4 &b)
{
    const float ci = fminf(fmaxf(floorf(u), 0.0f), (float)(m.width - 1));
    const float cj = fminf(fmaxf(floorf(v), 0.0f), (float)(m.height - 1));
    a = tex2Dgather<float4>(m.tex, ci, cj, 0);
    b = tex2Dgather<float4>(m.tex, ci + 1.0f, cj + 1.0f, 0);
}

// Steps 1-2 for one fragment: texel, shadow test, four-neighbourhood.
// Returns true when the fragment needs the edge walk for this mode; packs
// s0 and the four directions into `bits` (bit 0 = s0, bits 1-4 = left,
// right, +y, -y).  Clamp-to-edge is applied branch-free: a neighbour
// outside the map is the centre texel itself, so the five loads of a
// fragment (and of the other fragments of the lane) can all be in flight at
// once.
template <int MODE, bool CODES>
__device__ __forceinline__ bool classify_uv(const MapDev &m, float u, float v, float pz,
                                            FragResult &r, uint32_t &bits)
{
    if (m.tex) {
        float4 a, b;
        gather_cross(m, u, v, a, b);
        return classify_from<MODE, CODES>(pz, a.y, a.x, b.z, b.x, a.z, r, bits);
    }
    int i, j;
    float fx, fy;
    texel_of(u, m.width, i, fx);
    texel_of(v, m.height, j, fy);
    const float *c = m.depth + (long long)j * m.pitch + i;
    const float zc = __ldg(c);
    // Listing 1: in silhouette recovery a shadowed fragment stays shadowed and
    // needs no neighbourhood (unless codes are requested).
    if (MODE == 1 && !CODES && pz > zc) {
        r.sil = 0.0f;
        r.code = 0;
        bits = 0;
        return false;
    }
    const long long up = j < m.height - 1 ? m.pitch : 0;
    const long long dn = j > 0 ? m.pitch : 0;
    const int lf = i > 0 ? 1 : 0;
    const int rt = i < m.width - 1 ? 1 : 0;
    return classify_from<MODE, CODES>(pz, zc, __ldg(c - lf), __ldg(c + rt), __ldg(c + up), __ldg(c - dn), r, bits);
}

// Steps 1-2 from a texture coordinate (u = x * W, v = y * H in float32).
template <int MODE, bool CODES>
__device__ __forceinline__ bool classify(const MapDev &m, float x, float y, float pz,
                                         FragResult &r, uint32_t &bits)
{
    return classify_uv<MODE, CODES>(m, __fmul_rn(x, (float)m.width), __fmul_rn(y, (float)m.height), pz, r, bits);
}

// Steps 3-4 for one edge fragment at texel-space position (u, v)
// (recomputes its texel).
template <int MODE, bool PAIRS = false>
__device__ __forceinline__ void resolve_edge_uv(const MapDev &m, float u, float v, float pz,
                                                uint32_t bits, int max_dist, FragResult &r)
{
    int i, j;
    float fx, fy;
    texel_of(u, m.width, i, fx);
    texel_of(v, m.height, j, fy);
    const int s0 = bits & 1;
    const unsigned d4 = (bits >> 1) & 15u;
    // computeFragmentDistanceToSE: the four walks -x, +x, -y, +y
    int rxn, rxp, ryn, ryp;
    r.reach = edge_walks<PAIRS>(m, i, j, pz, s0 != 0, d4, max_dist, rxn, rxp, ryn, ryp);
    int ex = (rxn > 0) + (rxp > 0);
    int ey = (ryn > 0) + (ryp > 0);
    float nx = axis_position(rxn, rxp, fx);
    float ny = axis_position(ryn, ryp, fy);
    const bool dx3 = (d4 & 3u) == 3u, dy3 = (d4 & 12u) == 12u;
    r.code = (uint16_t)(r.code | (ex << 5) | (ey << 7) | (1 << 9));
    if (MODE & 1)
        r.sil = s0 ? silhouette(dx3, dy3, ex, ey, nx, ny) : 0.0f;
    if (MODE & 2)
        r.fil = filter(dx3, dy3, 1 - s0, ex, ey, nx, ny);
}

// Steps 3-4 from a texture coordinate.
template <int MODE, bool PAIRS = false>
__device__ __forceinline__ void resolve_edge(const MapDev &m, float x, float y, float pz,
                                             uint32_t bits, int max_dist, FragResult &r)
{
    resolve_edge_uv<MODE, PAIRS>(m, __fmul_rn(x, (float)m.width), __fmul_rn(y, (float)m.height), pz, bits, max_dist, r);
}

// ------------------------------------------------------------ warp tiles --
//
// A warp owns a tile of kWarpTile = 128 consecutive fragments, 4 per lane.  Warps
// never wait for each other (no CTA barrier).  Per tile a warp classifies its
// fragments, stores every answer at once (edge fragments get a provisional
// value) and appends its edge fragments to its own shared-memory queue.  The
// queue is drained 32 entries at a time, so the walks run with all 32 lanes
// busy, and the drained answers overwrite the provisional ones (still in L2).
// While a warp works on one tile, the copies of its next tile's coordinates
// into the warp's shared-memory buffer are already in flight (cp.async;
// `stage_tile` / `fetch_tile`; the depth-buffer kernel keeps its next tile's
// depths in registers, a quarter of the bytes).

constexpr int kWarpTile = 32 * kPerThread;   // 128 fragments
constexpr int kQueueCap = kWarpTile + 32;    // < 32 left over + one tile

// One deferred edge fragment (8 bytes): which fragment, and what its
// classification found.  The drain reads the fragment's x, y, z again (edge
// fragments are a few percent of the stream, so keeping the queue small and
// the shared memory free for the L1 cache pays more).
struct EdgeEntry {
    uint32_t idx;            // fragment index within the job (fragment sets hold < 2^31)
    uint32_t bits_job;       // s0 | d4 << 1 (5 bits) | job << 8
};

struct WarpQueue {
    EdgeEntry q[kQueueCap];
};

// Coordinates of one warp tile held by a lane (4 fragments).
struct LaneCoords {
    float x[kPerThread], y[kPerThread], z[kPerThread];
};

// Where a warp tile lives: fragments [first, first + count) of a job.
struct WarpTileIO {
    const float *x, *y, *z;
    float *sil, *fil;
    uint16_t *codes;
    long long first;
    int count;               // 1..kWarpTile
    int job;
    bool vec;                // count == kWarpTile and every plane 16-byte aligned
};

// A job as the deferred answers need it: its map, its fragments, its outputs.
struct JobOut {
    MapDev map;
    const float *x, *y, *z;
    float *sil, *fil;
    uint16_t *codes;
    int mode;
};

// Fragment of a warp tile that a lane's element e is: two pairs (8-byte
// accesses) or l, l+32, l+64, l+96 (coalesced 4-byte ones).
__device__ __forceinline__ int tile_slot(bool pairs, unsigned lane, int e)
{
    return pairs ? (e >> 1) * 64 + 2 * (int)lane + (e & 1) : (int)lane + 32 * e;
}

// The coordinates of a tile that is not a vector tile, read directly.
__device__ __forceinline__ void load_tile(const WarpTileIO &t, unsigned lane, LaneCoords &c)
{
#pragma unroll
    for (int e = 0; e < kPerThread; ++e) {
        const int s = tile_slot(false, lane, e);
        const bool ok = s < t.count;
        c.x[e] = ok ? __ldcs(t.x + t.first + s) : 0.0f;
        c.y[e] = ok ? __ldcs(t.y + t.first + s) : 0.0f;
        c.z[e] = ok ? __ldcs(t.z + t.first + s) : 0.0f;
    }
}

// 16-byte asynchronous copy global -> shared (cp.async, cached in L2 only).
__device__ __forceinline__ void copy_async16(void *smem, const void *gmem)
{
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(gmem) : "memory");
}

// Start the copies of a tile's coordinates into the warp's buffer (vector
// tiles; others are loaded directly when they come up).
__device__ __forceinline__ void stage_tile(const WarpTileIO &t, unsigned lane, float4 (&buf)[3][32])
{
    if (t.vec) {
        copy_async16(&buf[0][lane], reinterpret_cast<const float4 *>(t.x + t.first) + lane);
        copy_async16(&buf[1][lane], reinterpret_cast<const float4 *>(t.y + t.first) + lane);
        copy_async16(&buf[2][lane], reinterpret_cast<const float4 *>(t.z + t.first) + lane);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// The staged tile's coordinates in registers (waits for the copies).  A lane
// copied 4 consecutive fragments of each plane and reads two pairs, 2 lane
// and 64 + 2 lane: neighbouring lanes then gather from the same or
// neighbouring texels, which the texture path serves together, and the pairs
// still store 8 bytes at a time.  (8 frames of 3840x2160 in one launch, 64
// cascade jobs, filtering 3840x2160: 350 / 368 / 49.4 us with 4 consecutive
// fragments per lane, 336 / 362 / 47.5 with pairs, 332 / 372 / 47.2 with
// single ones 32 apart.)  The buffer is read by other lanes than the one
// that copied it: a warp barrier after the wait, and another before it is
// refilled.
//
// SINGLES: single fragments 32 apart.  For kernels that read a map without a
// texture: each of a fragment's five loads then covers 32 fragments in a row
// and touches half the lines.  And for the single-map calls, whose answers
// are one plane (filtering 3840x2160 47.7 us with pairs, 47.2 with singles;
// 2560x1440 29.5 and 28.6; silhouette 1920x1080 20.3 and 19.8).  Depth buffers with two answer planes keep the pairs
// (194.7 against 197.9 us for 4 frames).
template <bool SINGLES = false>
__device__ __forceinline__ void fetch_tile(const WarpTileIO &t, unsigned lane, const float4 (&buf)[3][32],
                                           LaneCoords &c)
{
    if (t.vec) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncwarp();
#pragma unroll
        for (int e = 0; SINGLES && e < kPerThread; ++e) {
            c.x[e] = reinterpret_cast<const float *>(buf[0])[lane + 32 * e];
            c.y[e] = reinterpret_cast<const float *>(buf[1])[lane + 32 * e];
            c.z[e] = reinterpret_cast<const float *>(buf[2])[lane + 32 * e];
        }
#pragma unroll
        for (int h = 0; !SINGLES && h < 2; ++h) {
            const float2 vx = reinterpret_cast<const float2 *>(buf[0])[lane + 32 * h];
            const float2 vy = reinterpret_cast<const float2 *>(buf[1])[lane + 32 * h];
            const float2 vz = reinterpret_cast<const float2 *>(buf[2])[lane + 32 * h];
            c.x[2 * h] = vx.x; c.x[2 * h + 1] = vx.y;
            c.y[2 * h] = vy.x; c.y[2 * h + 1] = vy.y;
            c.z[2 * h] = vz.x; c.z[2 * h + 1] = vz.y;
        }
        __syncwarp();
    } else {
        load_tile(t, lane, c);
    }
}

__device__ __forceinline__ unsigned lane_id() { return threadIdx.x & 31u; }

// Walk, normalise and answer one deferred edge fragment; write its answers.
// FIXED_MODE 1..3 when every job of the launch has that mode, 0 to read it
// from the job.
// Returns the step its longest walk stopped at.
template <int FIXED_MODE = 0, bool PAIRS = false>
__device__ __forceinline__ int resolve_entry(const JobOut &o, const EdgeEntry &q, int max_dist)
{
    const uint32_t bits = q.bits_job & 0x1fu;
    const uint32_t d4 = bits >> 1, s0 = bits & 1u;
    FragResult r{0.0f, 0.0f, (uint16_t)(d4 | ((1u - s0) << 4))};
    const float x = __ldg(o.x + q.idx), y = __ldg(o.y + q.idx), z = __ldg(o.z + q.idx);
    switch (FIXED_MODE ? FIXED_MODE : o.mode) {
    case 1: resolve_edge<1, PAIRS>(o.map, x, y, z, bits, max_dist, r); break;
    case 2: resolve_edge<2, PAIRS>(o.map, x, y, z, bits, max_dist, r); break;
    default: resolve_edge<3, PAIRS>(o.map, x, y, z, bits, max_dist, r); break;
    }
    if (o.mode & 1) o.sil[q.idx] = r.sil;
    if (o.mode & 2) o.fil[q.idx] = r.fil;
    if (o.codes) o.codes[q.idx] = r.code;
    return r.reach;
}

// Drain full rounds of 32 queued edge fragments (or everything when
// `all`).  `jobs(job)` returns the JobOut of a job.  The count is uniform
// across the warp.
template <typename Jobs, int FIXED_MODE = 0, bool PAIRS = false>
__device__ __forceinline__ void drain_queue(const Jobs &jobs, WarpQueue &wq, int &count, int max_dist, bool all)
{
    const unsigned lane = lane_id();
    while (count >= 32 || (all && count > 0)) {
        __syncwarp();                      // queue entries and provisional stores are visible
        const int base = count >= 32 ? count - 32 : 0;
        const int k = base + (int)lane;
        if (k < count) {
            const EdgeEntry q = wq.q[k];
            resolve_entry<FIXED_MODE, PAIRS>(jobs((int)(q.bits_job >> 8)), q, max_dist);
        }
        __syncwarp();                      // entries read before they are overwritten
        count = base;
    }
}

// Classify one warp tile whose coordinates the lane holds, store its answers
// (provisional for edge fragments) and queue its edge fragments.  TEX: whether
// the map has a texture, 1 or 0, or -1 to ask the map per tile.  Kernels
// made for one of them hold half the code.  PAIRS: a lane's fragments in a
// vector tile are two pairs, else single ones 32 apart (see fetch_tile).  3840x2160 fragments without a texture: filtering 75.2 us with pairs
// and a kernel for both, 56.4 with TEX 0; silhouette 67.4 and 53.0; depth
// buffers, 4 frames, 313 and 266 (with a texture 195.4 and 193.4, TEX 1).
template <int MODE, bool CODES, int TEX = -1, bool PAIRS = TEX != 0>
__device__ __forceinline__ void classify_warp_tile(const MapDev &m, const WarpTileIO &t, const LaneCoords &c,
                                                   WarpQueue &wq, int &count)
{
    const unsigned lane = lane_id();
    const unsigned below = (1u << lane) - 1u;
    const bool pairs = PAIRS && t.vec;
    FragResult r[kPerThread];
    uint32_t bits[kPerThread];
    bool edge[kPerThread];
    // classify the lane's four fragments first (no warp-wide step in between,
    // so all their texel loads are issued back to back) ...
    if (TEX < 0 ? m.tex != 0 : TEX != 0) {
        // one branch for the four fragments' eight gathers: tested per
        // fragment, the texture handle put a branch between one fragment's
        // gathers and the next one's (depth buffers, 4 frames of 3840x2160
        // pixels: 241 against 219 us; planes, 8 frames in one launch: 369
        // against 349 us).  Bound: a gather's four components take the
        // texture path about 16 cycles to write back for a warp, 26 us of a
        // 3840x2160 frame; fetching the right and upper neighbours one by one
        // instead (two point fetches, or two loads, for the second gather)
        // was slower: 458 and 494 us for the 8 frames.
        // A partial tile's lanes past its end hold zeros and are masked after.
        const float W = (float)m.width, H = (float)m.height;
        float4 a[kPerThread], b[kPerThread];
#pragma unroll
        for (int e = 0; e < kPerThread; ++e)
            gather_cross(m, __fmul_rn(c.x[e], W), __fmul_rn(c.y[e], H), a[e], b[e]);
#pragma unroll
        for (int e = 0; e < kPerThread; ++e)
            edge[e] = classify_from<MODE, CODES>(c.z[e], a[e].y, a[e].x, b[e].z, b[e].x, a[e].z, r[e], bits[e]);
        if (!t.vec) {
#pragma unroll
            for (int e = 0; e < kPerThread; ++e)
                edge[e] = edge[e] && tile_slot(false, lane, e) < t.count;
        }
    } else if (TEX == 0) {
        // the four fragments' own texels first, then their neighbours, so
        // that no fragment's loads wait for another's.  In silhouette recovery
        // a shadowed fragment needs no neighbours, and its lane loads none: a view
        // whose fragments run across the map's rows touches a line of its own
        // with every load (2828x2828 fragments on a 4096^2 map, rows of
        // fragments along its columns: all shadowed 42.7 us, half 151, lit 142;
        // with the neighbours loaded in any case 116, 185 and 141; a 1920x1080
        // view of a scene 21.5 and 20.9; one fragment after the other 61 us for
        // 8 M lit fragments in order, where this takes 38).  A partial tile's
        // lanes past its end hold zeros and are masked after.
        const float *p[kPerThread];
        float zc[kPerThread];
        int i[kPerThread], j[kPerThread];
#pragma unroll
        for (int e = 0; e < kPerThread; ++e) {
            float f;
            texel_of(__fmul_rn(c.x[e], (float)m.width), m.width, i[e], f);
            texel_of(__fmul_rn(c.y[e], (float)m.height), m.height, j[e], f);
            p[e] = m.depth + (long long)j[e] * m.pitch + i[e];
            zc[e] = __ldg(p[e]);
        }
        float4 nb[kPerThread];
#pragma unroll
        for (int e = 0; e < kPerThread; ++e) {
            nb[e] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (MODE == 1 && !CODES && c.z[e] > zc[e])
                continue;                      // classify_from asks for no neighbour
            nb[e].x = __ldg(p[e] - (i[e] > 0 ? 1 : 0));
            nb[e].y = __ldg(p[e] + (i[e] < m.width - 1 ? 1 : 0));
            nb[e].z = __ldg(p[e] + (j[e] < m.height - 1 ? m.pitch : 0));
            nb[e].w = __ldg(p[e] - (j[e] > 0 ? m.pitch : 0));
        }
#pragma unroll
        for (int e = 0; e < kPerThread; ++e) {
            edge[e] = classify_from<MODE, CODES>(c.z[e], zc[e], nb[e].x, nb[e].y, nb[e].z, nb[e].w, r[e], bits[e]);
            if (!t.vec)
                edge[e] = edge[e] && tile_slot(false, lane, e) < t.count;
        }
    } else if (t.vec) {
#pragma unroll
        for (int e = 0; e < kPerThread; ++e)
            edge[e] = classify<MODE, CODES>(m, c.x[e], c.y[e], c.z[e], r[e], bits[e]);
    } else {
#pragma unroll
        for (int e = 0; e < kPerThread; ++e) {
            r[e] = FragResult{0.0f, 0.0f, 0};
            bits[e] = 0;
            edge[e] = false;
            if ((int)lane + 32 * e < t.count)
                edge[e] = classify<MODE, CODES>(m, c.x[e], c.y[e], c.z[e], r[e], bits[e]);
        }
    }
    // ... then queue the edge fragments, one ballot per element
#pragma unroll
    for (int e = 0; e < kPerThread; ++e) {
        const int s = tile_slot(pairs, lane, e);
        const unsigned mask = __ballot_sync(0xffffffffu, edge[e]);
        if (edge[e]) {
            wq.q[count + __popc(mask & below)] =
                EdgeEntry{(uint32_t)(t.first + s), bits[e] | ((uint32_t)t.job << 8)};
        }
        count += __popc(mask);
    }
    if (pairs) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const long long g = t.first + tile_slot(true, lane, 2 * h);
            if (MODE & 1)
                __stcg(reinterpret_cast<float2 *>(t.sil + g), make_float2(r[2 * h].sil, r[2 * h + 1].sil));
            if (MODE & 2)
                __stcg(reinterpret_cast<float2 *>(t.fil + g), make_float2(r[2 * h].fil, r[2 * h + 1].fil));
            if (CODES)
                __stcg(reinterpret_cast<unsigned *>(t.codes + g),
                       (uint32_t)r[2 * h].code | ((uint32_t)r[2 * h + 1].code << 16));
        }
    } else {
#pragma unroll
        for (int e = 0; e < kPerThread; ++e) {
            const int s = tile_slot(false, lane, e);
            if (s >= t.count)
                continue;
            const long long g = t.first + s;
            if (MODE & 1) t.sil[g] = r[e].sil;
            if (MODE & 2) t.fil[g] = r[e].fil;
            if (CODES) t.codes[g] = r[e].code;
        }
    }
}

// Dispatch on the runtime mode / codes pair of a job.
__device__ __forceinline__ void classify_warp_tile_rt(int mode, bool codes, const MapDev &m, const WarpTileIO &t,
                                                      const LaneCoords &c, WarpQueue &wq, int &count)
{
    switch (mode * 2 + (codes ? 1 : 0)) {
    case 2: classify_warp_tile<1, false>(m, t, c, wq, count); break;
    case 3: classify_warp_tile<1, true>(m, t, c, wq, count); break;
    case 4: classify_warp_tile<2, false>(m, t, c, wq, count); break;
    case 5: classify_warp_tile<2, true>(m, t, c, wq, count); break;
    case 6: classify_warp_tile<3, false>(m, t, c, wq, count); break;
    default: classify_warp_tile<3, true>(m, t, c, wq, count); break;
    }
}

}  // namespace rbsm
