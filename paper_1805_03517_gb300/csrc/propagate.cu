// propagate.cu -- per-level refinement of the matches (FlowFields++, arXiv 1805.03517, Sec. 3.1): coarse-to-fine
// hand-over and propagation towards the four quadrants with random search.
//
// Schedule of one iteration t at one level (the same schedule the oracle runs): for each quadrant direction
// d = 0..3 (neighbours left+top, right+top, left+bottom, right+bottom), two half-sweeps over the pixels with
// (x + y) even, then odd.  A pixel of the active colour tries neighbour 1 (horizontal), neighbour 2 (vertical)
// and, for d >= 1, its current flow plus a hashed random offset in [-R, R]^2 (skipped if zero); a candidate
// is taken iff its cost (WHT SAD or Census Hamming distance) is strictly lower; targets outside the level are
// rejected.  Neighbours always have the other colour, so every half-sweep is a fully parallel map.
//
// Temporal blocking: one CTA owns a tile of a level and runs n_iter whole iterations (8 half-sweeps each) in
// shared memory before writing the tile back, reading the level state from one buffer and writing another.
// It loads the tile plus a halo of 4 * n_iter pixels and, before half-sweep j, recomputes every pixel whose
// value the remaining half-sweeps need: the region grows backwards from the tile by one pixel on the two
// upstream sides of each later half-sweep.  Recomputed halo pixels use exactly the inputs of the CTA that owns
// them, so every tile's output equals the global schedule bit for bit.
//
// The work of a tile has three variants.  The direct one gives every pixel of a half-sweep a thread, which scores the
// pixel's candidates.  The resident one gives every pixel of the region its own thread for the whole launch; tiles small
// enough take it (prop_resident).  The listed one skips the candidates that are known not to be cheaper and gives threads
// only to the pixels left; dataflow launches of enough pixels to keep the GPU busy take it (prop_listed).
#include <climits>
#include <cstddef>

#include "ff_internal.h"

namespace ff {

// first index violation of a debug-bounds build (see idx_ok): code, index, limit
static __device__ int g_bounds[4];

cudaError_t bounds_take_propagate(int rec[3]) {
    int h[4] = {0, 0, 0, 0};
    cudaError_t e = cudaMemcpyFromSymbol(h, g_bounds, sizeof h);
    if (e == cudaSuccess && h[0] != 0) {
        const int z[4] = {0, 0, 0, 0};
        e = cudaMemcpyToSymbol(g_bounds, z, sizeof z);
    }
    rec[0] = h[0], rec[1] = h[1], rec[2] = h[2];
    return e;
}

// Bounds codes of this file's checks.
enum : int { kBoundsOwn = 1, kBoundsCand1, kBoundsCand2, kBoundsRandom, kBoundsSmemOwn, kBoundsSmemN1,
             kBoundsSmemN2, kBoundsTileRead, kBoundsTileSmem, kBoundsTileWrite, kBoundsParent, kBoundsHandoverDesc,
             kBoundsBlockRead, kBoundsBlockSmem, kBoundsBlockWrite, kBoundsRingN1, kBoundsRingN2 };

__device__ __forceinline__ int flow_x(uint32_t f) { return (int)(int16_t)(f & 0xffffu); }
__device__ __forceinline__ int flow_y(uint32_t f) { return ((int)f) >> 16; }
__device__ __forceinline__ uint32_t pack_flow(int dx, int dy) { return (uint32_t)(dx & 0xffff) | ((uint32_t)dy << 16); }
__device__ __forceinline__ bool in_level(int x, int y, int w, int h) {
    return (unsigned)x < (unsigned)w && (unsigned)y < (unsigned)h;
}

// Eight 32-bit words (one 32-B sector of a descriptor) with one 256-bit read-only load.
__device__ __forceinline__ void load_words8(const char* p, uint32_t (&d)[8]) {
    asm("ld.global.nc.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
        : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3]), "=r"(d[4]), "=r"(d[5]), "=r"(d[6]), "=r"(d[7])
        : "l"(p));
}

// The two matching costs (Sec. 3.1), as policies of the hand-over and propagation kernels: 32-B sectors per
// descriptor, load of one sector, and the sector's share of the distance.  Every share is non-negative, so the sum
// over the first sectors bounds the distance from below.
//
// SAD of the 48 WHT coefficients, one colour channel per sector.  The feature maps store every coefficient in
// offset binary (C ^ 0x8000, i.e. C + 32768 as uint16, which preserves order), so per half max - min is |a - b| in
// [0, 32640] and a plain 32-bit subtraction of the packed max/min never borrows across halves.  Two packed
// differences add without carrying (2 * 32640 < 65536); __dp2a_lo then adds both 16-bit halves into the int32 sum.
// The 64 products of the 8x8 transform are orthogonal, so a channel's difference of two patches (each |difference|
// <= 255) has a Euclidean norm of at most 64 * 255 and its 16 coefficients an absolute sum of at most 4 * 64 * 255:
// a distance is at most 3 * 65280 = 195,840 < 2^18.
struct CostSad {
    static constexpr int kSectors = 3;
    __device__ __forceinline__ static void load(const void* __restrict__ f, int idx, int k, uint32_t (&d)[8]) {
        load_words8(reinterpret_cast<const char*>(f) + (size_t)idx * kDescBytes + 32 * k, d);
    }
    __device__ __forceinline__ static int dist(const uint32_t (&a)[8], const uint32_t (&b)[8], int s0) {
        unsigned s = (unsigned)s0;
#pragma unroll
        for (int k = 0; k < 8; k += 2) {
            uint32_t d0 = __vmaxu2(a[k], b[k]) - __vminu2(a[k], b[k]);
            uint32_t d1 = __vmaxu2(a[k + 1], b[k + 1]) - __vminu2(a[k + 1], b[k + 1]);
            s = __dp2a_lo(d0 + d1, 0x0101u, s);
        }
        return (int)s;
    }
};

// Hamming distance of the three 48-bit Census patterns (one sector per pixel; its words 6 and 7 are zero).
struct CostCensus {
    static constexpr int kSectors = 1;
    __device__ __forceinline__ static void load(const void* __restrict__ f, int idx, int, uint32_t (&d)[8]) {
        load_words8(reinterpret_cast<const char*>(f) + (size_t)idx * kCensusBytes, d);
    }
    __device__ __forceinline__ static int dist(const uint32_t (&a)[8], const uint32_t (&b)[8], int s) {
#pragma unroll
        for (int k = 0; k < 6; k++) s += __popc(a[k] ^ b[k]);
        return s;
    }
};

// One sector of descriptor idx; a debug-bounds build checks the index against the map's n descriptors (zeros if
// outside).
template <class C>
__device__ __forceinline__ void load_chk(const void* __restrict__ f, int idx, int n, int code, int k, uint32_t (&d)[8]) {
    if (idx_ok(g_bounds, code, idx, n)) {
        C::load(f, idx, k, d);
    } else {
#pragma unroll
        for (int i = 0; i < 8; i++) d[i] = 0;
    }
}

// A whole descriptor.
template <class C>
__device__ __forceinline__ void load_all(const void* __restrict__ f, int idx, int n, int code,
                                         uint32_t (&d)[C::kSectors][8]) {
#pragma unroll
    for (int k = 0; k < C::kSectors; k++) load_chk<C>(f, idx, n, code, k, d[k]);
}
template <class C>
__device__ __forceinline__ int dist_all(const uint32_t (&a)[C::kSectors][8], const uint32_t (&b)[C::kSectors][8]) {
    int s = 0;
#pragma unroll
    for (int k = 0; k < C::kSectors; k++) s = C::dist(a[k], b[k], s);
    return s;
}

// Cost of the descriptor at (x, y) of fa against (tx, ty) of fb (both inside the w x h level).
template <class C>
__device__ __forceinline__ int cost_at(const void* __restrict__ fa, const void* __restrict__ fb, int w, int h, int x,
                                       int y, int tx, int ty) {
    uint32_t a[C::kSectors][8], b[C::kSectors][8];
    load_all<C>(fa, feat_index(x, y, w), w * h, kBoundsHandoverDesc, a);
    load_all<C>(fb, feat_index(tx, ty, w), w * h, kBoundsHandoverDesc, b);
    return dist_all<C>(a, b);
}

// ---------------------------------------------------------------------------------------------------------
// hand-over: flow = 2 x parent flow (parent = (min(x/2, pw-1), min(y/2, ph-1))) or the given flow; cost of it.

template <class C>
__global__ __launch_bounds__(256) void k_handover(const HandoverProblem* __restrict__ probs, int n_probs,
                                                  int64_t total) {
    grid_dependency_sync();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        int lo = 0, hi = n_probs - 1;
        while (lo < hi) {  // last problem with pix_base <= i
            int mid = (lo + hi + 1) >> 1;
            if (probs[mid].pix_base <= i) lo = mid; else hi = mid - 1;
        }
        const HandoverProblem& P = probs[lo];
        int p = (int)(i - P.pix_base);
        const int u = p % P.w, v = p / P.w;
        const bool grid = P.g > 1;
        const int g = grid ? P.g : 1, lw = grid ? P.lw : P.w, lh = grid ? P.lh : P.h;
        const int x = g * u, y = g * v;  // level coordinates
        uint32_t f;
        if (P.parent && P.same_level) {  // from the grid of stride 2g: the same flow, its target clamped
            const int pi = min(v >> 1, P.ph - 1) * P.pw + min(u >> 1, P.pw - 1);
            uint32_t pf = idx_ok(g_bounds, kBoundsParent, pi, P.pw * P.ph) ? P.parent[pi] : 0u;
            f = pack_flow(min(max(x + flow_x(pf), 0), lw - 1) - x, min(max(y + flow_y(pf), 0), lh - 1) - y);
        } else if (P.parent) {  // from the level above: twice the parent pixel's flow
            int px = min(x >> 1, P.pw - 1), py = min(y >> 1, P.ph - 1);
            uint32_t pf = idx_ok(g_bounds, kBoundsParent, py * P.pw + px, P.pw * P.ph) ? P.parent[py * P.pw + px] : 0u;
            f = pack_flow(2 * flow_x(pf), 2 * flow_y(pf));
        } else {
            f = P.flow_in[p];
        }
        int tx = x + flow_x(f), ty = y + flow_y(f);
        int c = INT_MAX;  // unreachable for valid inputs: a handed-over flow always lands inside the level
        if (in_level(tx, ty, lw, lh)) c = cost_at<C>(P.fa, P.fb, lw, lh, x, y, tx, ty);
        P.flow_out[p] = f;
        P.cost_out[p] = c;
    }
}

void launch_handover(const HandoverProblem* probs_dev, int n_probs, int64_t total_pix, int cost, cudaStream_t st) {
    int64_t blocks = (total_pix + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    if (blocks < 1) blocks = 1;
    if (cost == FF_COST_CENSUS)
        launch_k(k_handover<CostCensus>, dim3((int)blocks), dim3(256), 0, st, probs_dev, n_probs, total_pix);
    else
        launch_k(k_handover<CostSad>, dim3((int)blocks), dim3(256), 0, st, probs_dev, n_probs, total_pix);
}

// ---------------------------------------------------------------------------------------------------------
// propagation + random search

// Extra pixels (left, up, right, down) recomputed before half-sweep j = 2*d + colour of the last fused
// iteration; earlier iterations add kHaloPerIter on every side per remaining iteration.
__constant__ int8_t c_grow[8][4] = {{3, 3, 4, 4}, {2, 2, 4, 4}, {2, 1, 3, 4}, {2, 0, 2, 4},
                                    {1, 0, 2, 3}, {0, 0, 2, 2}, {0, 0, 1, 1}, {0, 0, 0, 0}};

size_t prop_smem_bytes(int tw, int th, int n_iter) {
    int H = kHaloPerIter * n_iter;
    return (size_t)(tw + 2 * H) * (th + 2 * H) * 8;
}

// The key of iteration t's random offsets, and of level pixel (X, Y) in it.
__device__ __forceinline__ uint32_t iter_key(const PropProblem& P, int t) {
    return mix32(P.seed ^ mix32((uint32_t)P.dir * 65536u + (uint32_t)P.level * 256u + (uint32_t)t));
}
__device__ __forceinline__ uint32_t pixel_key(uint32_t k1, int X, int Y) {
    return mix32(k1 ^ ((uint32_t)Y * 65536u + (uint32_t)X));
}

// The variants of a tile's work: one pixel of a half-sweep at a time per thread, every pixel of the region by its own
// thread, and lists of the pixels with something to try.
enum Variant { kDirect, kResident, kListed };

// Where a tile task reads the state of its region and writes its interior, and which iterations it runs.
struct TileIO {
    const uint32_t* flow_in;
    const int32_t* cost_in;
    uint32_t* flow_out;
    int32_t* cost_out;
    int t0, n_iter;
};

// ---- direct variant

// Geometry of the tile a CTA is working on (all coordinates are level coordinates).
struct TileGeom {
    int x0, y0, x1, y1;      // tile interior
    int lx0, ly0, RW, RH;    // loaded region (tile + halo, clipped to the level)
};

// Regions of the half-sweeps of one iteration, in shared memory: x0, y0, x1, y1 in level coordinates, and
// ceil(2^32 / slots per row), by which the index of a pixel of the active colour is divided.
struct SweepRegions {
    int4 r[8];
    uint32_t inv[8];
    // Thread j sets that of half-sweep j (colour j&1 of direction j>>1) with `rem` halo pixels still to be consumed.
    __device__ __forceinline__ void set(const TileGeom& G, int w, int h, int rem) {
        const int j = threadIdx.x;
        if (j >= 8) return;
        r[j] = make_int4(max(G.x0 - c_grow[j][0] - rem, 0), max(G.y0 - c_grow[j][1] - rem, 0),
                         min(G.x1 + c_grow[j][2] + rem, w), min(G.y1 + c_grow[j][3] + rem, h));
        inv[j] = 0xffffffffu / (uint32_t)((r[j].z - r[j].x + 1) >> 1) + 1u;  // (unused for one slot per row)
    }
};

// Per-launch constants of the pixel updates, read from the problem once per tile.
struct SweepConst {
    const void* fa;
    const void* fb;
    int g, lw, lh;       // grid stride and level size: grid pixel (x, y) is level pixel (g*x, g*y)
    int R;               // random-search radius
    uint32_t span, inv;  // 2R + 1 and floor(2^32 / span)
    // hash % span - R; the quotient is at most one too small
    __device__ __forceinline__ int offset(uint32_t hash) const {
        const uint32_t m = hash - __umulhi(hash, inv) * span;
        return (int)(m >= span ? m - span : m) - R;
    }
};
__device__ __forceinline__ SweepConst sweep_const(const PropProblem& P, bool grid) {
    const uint32_t span = 2u * P.rs_radius + 1u;
    // (2^32 and 2^32 - 1 have the same quotient, except for span 1, where every offset is 0 anyway)
    return {P.fa, P.fb, grid ? P.g : 1, grid ? P.lw : P.w, grid ? P.lh : P.h, P.rs_radius, span, 0xffffffffu / span};
}

// The candidates of one pixel (x, y) of a grid in a half-sweep of direction d: neighbour 1 (horizontal, flow f1, valid
// if v1), neighbour 2 (vertical, f2, v2) and, for d >= 1, the hashed random offset around the flow after them.  cur / c
// hold the pixel's flow and cost and are updated; false if there was nothing to try (they are unchanged).  One thread
// per pixel holds the whole descriptors.  (Four threads per pixel, one sector each, were slower at every level: 51
// instead of 38 us already for the 32x24 level of the 128x96 pair.)
template <class C>
__device__ __forceinline__ bool update_direct(const SweepConst& K, int x, int y, int d, uint32_t k1, bool v1, uint32_t f1,
                                              bool v2, uint32_t f2, uint32_t& cur, int& c) {
    // flows and targets are in level pixels
    const int g = K.g, lw = K.lw, lh = K.lh;
    const int n_d = lw * lh;  // descriptors of the level
    // a candidate equal to the current flow (or to an already tried one) cannot be strictly cheaper
    const int X = g * x, Y = g * y;  // level coordinates
    const bool e1 = v1 && f1 != cur && in_level(X + flow_x(f1), Y + flow_y(f1), lw, lh);
    const bool e2 = v2 && f2 != cur && !(v1 && f2 == f1) && in_level(X + flow_x(f2), Y + flow_y(f2), lw, lh);
    if (!(e1 || e2 || d >= 1)) return false;
    // issue every independent load (own descriptor, neighbour candidates) before compute, the hash among them
    uint32_t a[C::kSectors][8], b1[C::kSectors][8], b2[C::kSectors][8];
    load_all<C>(K.fa, feat_index(X, Y, lw), n_d, kBoundsOwn, a);
    if (e1) load_all<C>(K.fb, feat_index(X + flow_x(f1), Y + flow_y(f1), lw), n_d, kBoundsCand1, b1);
    if (e2) load_all<C>(K.fb, feat_index(X + flow_x(f2), Y + flow_y(f2), lw), n_d, kBoundsCand2, b2);
    int ox = 0, oy = 0;
    if (d >= 1) {
        const uint32_t k2 = pixel_key(k1, X, Y);
        ox = K.offset(mix32(k2 ^ (uint32_t)(2 * d)));
        oy = K.offset(mix32(k2 ^ (uint32_t)(2 * d + 1)));
    }
    if (e1) {
        const int s1 = dist_all<C>(a, b1);
        if (s1 < c) { cur = f1; c = s1; }
    }
    if (e2) {
        const int s2 = dist_all<C>(a, b2);
        if (s2 < c) { cur = f2; c = s2; }
    }
    if (ox != 0 || oy != 0) {
        const int fx = flow_x(cur) + ox, fy = flow_y(cur) + oy;
        if (in_level(X + fx, Y + fy, lw, lh)) {
            load_all<C>(K.fb, feat_index(X + fx, Y + fy, lw), n_d, kBoundsRandom, b1);
            const int s3 = dist_all<C>(a, b1);
            if (s3 < c) { cur = pack_flow(fx, fy); c = s3; }
        }
    }
    return true;
}

// One half-sweep of a tile's region (direct variant).
template <class C>
__device__ __forceinline__ void halfsweep_direct(const SweepConst& K, const TileGeom& G, int w, int h, const int4 r,
                                                 uint32_t inv, uint32_t* sflow, int32_t* scost, int j, uint32_t k1) {
    const int d = j >> 1, colour = j & 1;
    const int HW = (r.z - r.x + 1) >> 1, total = HW * (r.w - r.y);
    for (int i = threadIdx.x; i < total; i += blockDim.x) {
        const int row = HW > 1 ? (int)__umulhi((uint32_t)i, inv) : i;  // i, HW < 2^15: i / HW
        const int y = r.y + row, x = r.x + 2 * (i - row * HW) + ((r.x + y + colour) & 1);
        if (x >= r.z) continue;
        const int sidx = (y - G.ly0) * G.RW + (x - G.lx0);
        const int n_s = G.RW * G.RH;  // shared-memory entries
        if (!idx_ok(g_bounds, kBoundsSmemOwn, sidx, n_s)) continue;
        uint32_t cur = sflow[sidx];
        int c = scost[sidx];
        const int n1x = x + ((d & 1) ? 1 : -1);
        const int n2y = y + ((d & 2) ? 1 : -1);
        const bool v1 = (unsigned)n1x < (unsigned)w;
        const bool v2 = (unsigned)n2y < (unsigned)h;
        const uint32_t f1 = v1 && idx_ok(g_bounds, kBoundsSmemN1, sidx + (n1x - x), n_s) ? sflow[sidx + (n1x - x)] : 0u;
        const uint32_t f2 =
            v2 && idx_ok(g_bounds, kBoundsSmemN2, sidx + (n2y - y) * G.RW, n_s) ? sflow[sidx + (n2y - y) * G.RW] : 0u;
        if (!update_direct<C>(K, x, y, d, k1, v1, f1, v2, f2, cur, c)) continue;
        sflow[sidx] = cur;
        scost[sidx] = c;
    }
}

// ---- resident variant: a region of at most one pixel per thread
//
// A small level is a chain of half-sweeps, and a half-sweep one of a thread's instructions and gathers: of a warp's time
// at level 4 of the 1242x375 pair, 42 % is issuing, 41 % waiting for gathers, and a half-sweep takes about a
// microsecond whether the region has 60 or 170 pixels of its colour.  So every pixel of the region has a thread that
// keeps its flow, cost and own descriptor in registers for all iterations of the launch (half the threads have the
// pixels of one colour, half those of the other), which leaves three things off the chain.  A neighbour is tried only
// if its flow is not the one tried last on that side (a candidate that was not cheaper never becomes so).  The random
// candidate around the present flow, known before the half-sweep, is scored during the half-sweep of the other colour,
// when the thread has nothing else to do; only a pixel that takes a neighbour's flow scores another one after it.  And
// there is no index arithmetic.  Pass times (6 iterations, us) of the best tiles with / without, by pixels: WHT-SAD 96
// 34 / 50, 1.5 k 54 / 58, 3.7 k 50 / 61, 10 k 68 / 78, 16 k 67 / 77, 25 k 82 / 94, 38 k 88 / 94, 42 k 102 / 98; Census
// 33 / 43, 42 / 48, 45 / 50, 52 / 52, 57 / 53, 60 / 70, 72 / 74, 85 / 74 (with two CTAs per SM; with the third 54 at 16 k).
// (A pair of pixels per thread, one of each colour and no thread idle, nor anything scored ahead: 90 instead of 61 at 3.7 k,
// spills included.)

// Cost of the flow (fx, fy) of level pixel (X, Y) with descriptor a, INT_MAX if its target is outside the level.
// (The arrays of predicated loads are zeroed, here and below: left uninitialised, they stay live around the loops and
// the kernel spills.)
template <class C>
__device__ __forceinline__ int score(const SweepConst& K, int X, int Y, const uint32_t (&a)[C::kSectors][8], int fx, int fy) {
    if (!in_level(X + fx, Y + fy, K.lw, K.lh)) return INT_MAX;
    uint32_t b[C::kSectors][8] = {};
    load_all<C>(K.fb, feat_index(X + fx, Y + fy, K.lw), K.lw * K.lh, kBoundsRandom, b);
    return dist_all<C>(a, b);
}

// One tile of one problem, as propagate_tile_direct, whose geometry and regions it takes.  The flows are in shared
// memory by colour: pixel (rx, ry) of the region has slot ry * ceil(RW / 2) + rx / 2 of its colour.
template <class C, bool DF>
__device__ __forceinline__ void propagate_tile_resident(const SweepConst& K, const TileGeom& G, const PropProblem& P,
                                                        uint32_t* smem, const TileIO& io, SweepRegions* s_regions) {
    const int w = P.w, h = P.h, n_iter = io.n_iter;
    const int HW = (G.RW + 1) >> 1, n_slots = HW * G.RH, half = (int)blockDim.x >> 1;
    const int colour = (int)threadIdx.x >= half, slot = (int)threadIdx.x - colour * half;
    const int row = slot / HW, y = G.ly0 + row;
    const int odd = (G.lx0 + y + colour) & 1;  // the pixel's column in the region is odd
    const int x = G.lx0 + 2 * (slot - row * HW) + odd;
    const bool mine = row < G.RH && x < G.lx0 + G.RW;
    const int X = K.g * x, Y = K.g * y, lw = K.lw, lh = K.lh, n_d = lw * lh;
    uint32_t* const own = smem + colour * n_slots + slot;
    const uint32_t* const other = smem + (colour ^ 1) * n_slots + slot;
    const size_t g = (size_t)y * w + x;
    const bool ok = mine && idx_ok(g_bounds, kBoundsTileRead, (long long)g, (long long)w * h) &&
                    (!FF_DEBUG_BOUNDS || idx_ok(g_bounds, kBoundsTileSmem, 2 * n_slots - 1, dyn_smem_bytes() / 4));
    uint32_t a[C::kSectors][8];
    load_all<C>(K.fa, ok ? feat_index(X, Y, lw) : 0, n_d, kBoundsOwn, a);
    uint32_t cur = !ok ? 0u : DF ? __ldcg(io.flow_in + g) : io.flow_in[g];
    int c = !ok ? 0 : DF ? __ldcg(io.cost_in + g) : io.cost_in[g];
    uint32_t left = cur, right = cur, up = cur, down = cur;  // the flow last tried from each side
    if (ok) *own = cur;
    __syncthreads();
    int ahead = INT_MAX, ox = 0, oy = 0;  // the next random candidate: its cost around the present flow, its offset
#pragma unroll 1
    for (int it = 0; it < n_iter; it++) {
        const uint32_t k2 = pixel_key(iter_key(P, io.t0 + it), X, Y);
        const SweepRegions& S = s_regions[it & 1];
        if (it + 1 < n_iter) s_regions[(it + 1) & 1].set(G, w, h, kHaloPerIter * (n_iter - 2 - it));
#pragma unroll 1
        for (int j = 0; j < 8; j++) {
            const int d = j >> 1;
            if ((j & 1) == colour) {
                const int4 r = S.r[j];
                if (ok && x >= r.x && x < r.z && y >= r.y && y < r.w) {
                    const int dx = (d & 1) ? 1 : -1, dy = (d & 2) ? 1 : -1;
                    // the horizontal neighbour has the pixel's slot, or the next one on its side
                    const int s1 = odd == (d & 1) ? dx : 0, s2 = dy * HW;
                    const bool v1 = (unsigned)(x + dx) < (unsigned)w && idx_ok(g_bounds, kBoundsSmemN1, slot + s1, n_slots);
                    const bool v2 = (unsigned)(y + dy) < (unsigned)h && idx_ok(g_bounds, kBoundsSmemN2, slot + s2, n_slots);
                    const uint32_t f1 = v1 ? other[s1] : cur, f2 = v2 ? other[s2] : cur;
                    const uint32_t l1 = (d & 1) ? right : left, l2 = (d & 2) ? down : up;
                    if (d & 1) right = f1; else left = f1;
                    if (d & 2) down = f2; else up = f2;
                    const uint32_t cur0 = cur;
                    const bool e1 = f1 != l1 && f1 != cur && in_level(X + flow_x(f1), Y + flow_y(f1), lw, lh);
                    const bool e2 = f2 != l2 && f2 != cur && f2 != f1 && in_level(X + flow_x(f2), Y + flow_y(f2), lw, lh);
                    if (e1 || e2) {
                        uint32_t b1[C::kSectors][8] = {}, b2[C::kSectors][8] = {};
                        if (e1) load_all<C>(K.fb, feat_index(X + flow_x(f1), Y + flow_y(f1), lw), n_d, kBoundsCand1, b1);
                        if (e2) load_all<C>(K.fb, feat_index(X + flow_x(f2), Y + flow_y(f2), lw), n_d, kBoundsCand2, b2);
                        if (e1) {
                            const int s = dist_all<C>(a, b1);
                            if (s < c) { cur = f1; c = s; }
                        }
                        if (e2) {
                            const int s = dist_all<C>(a, b2);
                            if (s < c) { cur = f2; c = s; }
                        }
                    }
                    if (d >= 1 && (ox != 0 || oy != 0)) {
                        const int fx = flow_x(cur) + ox, fy = flow_y(cur) + oy;
                        const int s = cur == cur0 ? ahead : score<C>(K, X, Y, a, fx, fy);
                        if (s < c) { cur = pack_flow(fx, fy); c = s; }
                    }
                    if (cur != cur0) *own = cur;
                }
            } else if (j >= 1 && j < 7) {  // the pixel's next half-sweep is j + 1, with a random candidate
                const int4 r = S.r[j + 1];
                if (ok && x >= r.x && x < r.z && y >= r.y && y < r.w) {
                    const int dn = (j + 1) >> 1;
                    ox = K.offset(mix32(k2 ^ (uint32_t)(2 * dn)));
                    oy = K.offset(mix32(k2 ^ (uint32_t)(2 * dn + 1)));
                    ahead = score<C>(K, X, Y, a, flow_x(cur) + ox, flow_y(cur) + oy);
                }
            }
            __syncthreads();
        }
    }
    if (!ok || x < G.x0 || x >= G.x1 || y < G.y0 || y >= G.y1) return;
    if (!idx_ok(g_bounds, kBoundsTileWrite, (long long)g, (long long)w * h)) return;
    io.flow_out[g] = cur;
    io.cost_out[g] = c;
}

// One tile of one problem: load the tile and its halo, run n_iter iterations in shared memory (RES: with the resident
// variant), write the tile.
// With DF, a dataflow task, the state was written by other CTAs of the running launch and is therefore read from L2.
template <class C, bool DF, bool RES>
__device__ __forceinline__ void propagate_tile_direct(const PropProblem& P, int tile, const PropLaunch& L,
                                                      uint32_t* smem, const TileIO& io) {
    __shared__ SweepRegions s_regions[2];  // of iterations it and it + 1
    const int w = P.w, h = P.h;
    const int n_iter = io.n_iter;
    TileGeom G;
    G.x0 = (tile % P.tiles_x) * L.tw;
    G.y0 = (tile / P.tiles_x) * L.th;
    G.x1 = min(G.x0 + L.tw, w);
    G.y1 = min(G.y0 + L.th, h);
    const int H = kHaloPerIter * n_iter;
    G.lx0 = max(G.x0 - H, 0);
    G.ly0 = max(G.y0 - H, 0);
    G.RW = min(G.x1 + H, w) - G.lx0;
    G.RH = min(G.y1 + H, h) - G.ly0;
    uint32_t* sflow = smem;
    int32_t* scost = reinterpret_cast<int32_t*>(smem + G.RW * G.RH);
    const SweepConst K = sweep_const(P, L.grid != 0);
    s_regions[0].set(G, w, h, kHaloPerIter * (n_iter - 1));
    if constexpr (RES) {
        propagate_tile_resident<C, DF>(K, G, P, smem, io, s_regions);
    } else {
        for (int i = threadIdx.x; i < G.RW * G.RH; i += blockDim.x) {
            int r = i / G.RW, c = i - r * G.RW;
            size_t g = (size_t)(G.ly0 + r) * w + G.lx0 + c;
            // flow and cost of the region (2 words per pixel) must fit the launch's dynamic shared memory
            const bool ok = idx_ok(g_bounds, kBoundsTileRead, (long long)g, (long long)w * h) &&
                            (!FF_DEBUG_BOUNDS ||
                             idx_ok(g_bounds, kBoundsTileSmem, 2 * G.RW * G.RH - 1, dyn_smem_bytes() / 4));
            sflow[i] = !ok ? 0u : DF ? __ldcg(io.flow_in + g) : io.flow_in[g];
            scost[i] = !ok ? 0 : DF ? __ldcg(io.cost_in + g) : io.cost_in[g];
        }
        __syncthreads();
        for (int it = 0; it < n_iter; it++) {
            const uint32_t k1 = iter_key(P, io.t0 + it);
            const SweepRegions& S = s_regions[it & 1];
            if (it + 1 < n_iter) s_regions[(it + 1) & 1].set(G, w, h, kHaloPerIter * (n_iter - 2 - it));
            for (int j = 0; j < 8; j++) {
                halfsweep_direct<C>(K, G, w, h, S.r[j], S.inv[j], sflow, scost, j, k1);
                __syncthreads();
            }
        }
        const int TW = G.x1 - G.x0;
        for (int i = threadIdx.x; i < TW * (G.y1 - G.y0); i += blockDim.x) {
            int r = i / TW, c = i - r * TW;
            int sidx = (G.y0 + r - G.ly0) * G.RW + (G.x0 + c - G.lx0);
            size_t g = (size_t)(G.y0 + r) * w + G.x0 + c;
            if (!idx_ok(g_bounds, kBoundsTileWrite, (long long)g, (long long)w * h) ||
                !idx_ok(g_bounds, kBoundsTileSmem, sidx, G.RW * G.RH))
                continue;
            io.flow_out[g] = sflow[sidx];
            io.cost_out[g] = scost[sidx];
        }
    }
}

// ---- listed variant (dataflow form)
//
// What bounds the direct variant at level 0 of the 1242x375 pair is gathers and instructions alike: 28.9 M sectors
// and 59 M instructions per iteration, most of them for candidates that are known not to be cheaper, at 44 % of the
// issue slots.  This variant loads 13 M sectors per iteration and runs 32 instead of 16 warps per SM: level 0 in 531
// instead of 663 us (all six iterations), of the 1920x1080 pair in 1674 instead of 2760.

// What a pixel still has to try, one byte per pixel in shared memory.  Costs only fall and
// a candidate's cost is fixed, so a candidate that was not cheaper than a pixel's flow never becomes so: a
// neighbour's flow needs a trial only if it changed since the pixel last tried that neighbour, and a random candidate
// that the screening found not cheaper needs none while the pixel keeps its flow.  On the 1242x375 pair this leaves,
// per pixel and iteration of level 0, 2.0, 1.3, 0.6, 0.4, 0.3 and 0.25 neighbour trials in iterations 0..5 instead of
// 2.3 to 3.0; results are the same bit for bit.
//   bits 0..3  the left, right, upper, lower neighbour's flow has changed since its last trial
//   bits 4..6  the random candidate of direction 1, 2, 3 has to be scored
constexpr uint32_t kTodoAll = 0x7f7f7f7fu;
__device__ __forceinline__ uint32_t todo_bits(int d) {  // those of direction d
    return (1u << (d & 1)) | (4u << (d >> 1)) | (d ? 8u << d : 0u);
}

// The state word between the tasks of a pass (in the cost buffers):
//   bits 31..14  cost of the flow (at most 195,840, see CostSad; Census 144)
//   bits 13..11  the random candidates of the next iteration that have to be scored (screen)
//   bits 3..0    1 + the half-sweep of the iteration that last changed the flow, 0: none did
// In shared memory the flags are in the todo bytes.
// (Other words than these are read here after a wait that expired; every use of their bits stays in range.)
constexpr int kCostShift = 14, kFlagShift = 11;
constexpr uint32_t kStampMask = 15u, kCostMax = (1u << (32 - kCostShift)) - 1;
__device__ __forceinline__ uint32_t pack_state(int cost) { return min((uint32_t)cost, kCostMax) << kCostShift; }
// Constants of a problem, in shared memory.
struct alignas(16) Sweep {
    const void* fa;
    const void* fb;
    int g, lw, lh, half;  // grid stride and level size: grid pixel (x, y) is level pixel (g*x, g*y); (lw + 1) / 2
    uint32_t span, inv;   // 2R + 1 (R: random-search radius) and floor(2^32 / span)
    int R, pad;
    __device__ __forceinline__ void set(const PropProblem& P, bool grid) {
        fa = P.fa;
        fb = P.fb;
        g = grid ? P.g : 1;
        lw = grid ? P.lw : P.w;
        lh = grid ? P.lh : P.h;
        half = (lw + 1) >> 1;
        R = P.rs_radius;
        span = 2u * P.rs_radius + 1u;
        inv = 0xffffffffu / span;  // (2^32 has the same quotient, except for span 1, where every offset is 0 anyway)
    }
};

// Reads of CTA-wide constants in shared memory by address.  Every pixel takes a fresh copy of the address the compiler
// cannot see through, so the constants are read where they are used (four at a time, a broadcast) and hold no
// registers across the pixels.
__device__ __forceinline__ uint32_t fresh(uint32_t a) {
    asm volatile("" : "+r"(a));
    return a;
}
__device__ __forceinline__ int4 lds_int4(uint32_t a) {
    int4 v;
    asm("ld.shared.v4.s32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
    return v;
}
struct SweepRef {
    uint32_t a;  // address of a Sweep
    __device__ __forceinline__ const void* ptr(uint32_t offset) const {
        uint64_t v;
        asm("ld.shared.u64 %0, [%1];" : "=l"(v) : "r"(a + offset));
        return reinterpret_cast<const void*>(v);
    }
    __device__ __forceinline__ const void* fa() const { return ptr(offsetof(Sweep, fa)); }
    __device__ __forceinline__ const void* fb() const { return ptr(offsetof(Sweep, fb)); }
    __device__ __forceinline__ int4 level() const { return lds_int4(a + (uint32_t)offsetof(Sweep, g)); }  // g, lw, lh, half
    __device__ __forceinline__ int g() const { return level().x; }
    // Descriptor of level pixel (X, Y) in the colour-split rows (feat_index).
    __device__ __forceinline__ int index(int X, int Y) const {
        const int4 L = level();
        return Y * L.y + (X >> 1) + ((X & 1) ? L.w : 0);
    }
    __device__ __forceinline__ bool inside(int X, int Y) const {
        const int4 L = level();
        return in_level(X, Y, L.y, L.z);
    }
    __device__ __forceinline__ int n_desc() const {  // of the level (debug-bounds checks)
        return FF_DEBUG_BOUNDS ? level().y * level().z : 0;
    }
    // hash % span - R; the quotient is at most one too small
    __device__ __forceinline__ static int offset(uint32_t hash, const int4& r) {
        const uint32_t span = (uint32_t)r.x, m = hash - __umulhi(hash, (uint32_t)r.y) * span;
        return (int)(m >= span ? m - span : m) - r.z;
    }
    // The random offset of direction d for the pixel key k2.
    __device__ __forceinline__ void random_offset(uint32_t k2, int d, int& ox, int& oy) const {
        const int4 r = lds_int4(a + (uint32_t)offsetof(Sweep, span));  // span, inv, R
        ox = offset(mix32(k2 ^ (uint32_t)(2 * d)), r);
        oy = offset(mix32(k2 ^ (uint32_t)(2 * d + 1)), r);
    }
};

// The candidates of one pixel (x, y) of a grid in a half-sweep of direction d, one thread per pixel: neighbour 1
// (horizontal, flow f1, to be tried if t1), neighbour 2 (vertical, f2, t2) and, for d >= 1, the hashed random
// offset around the flow after them.  The random candidate is scored if `rnd`, or if a neighbour was taken (else it
// is known not to be cheaper).  cur / c hold the pixel's flow and cost and are updated.
// Each candidate's three sectors are loaded together and one candidate after the other, so that a late half-sweep,
// where a pixel has one candidate to try, waits for one gather (level 0 of the 1242x375 pair: 541 us; both neighbours
// side by side, sector by sector, and the random candidate until its partial distance settles it: 565).
template <class C>
__device__ __forceinline__ void update_pixel(const SweepRef K, int x, int y, int d, uint32_t k1, bool t1, uint32_t f1,
                                             bool t2, uint32_t f2, bool rnd, uint32_t& cur, int& c) {
    const int g = K.g(), X = g * x, Y = g * y;  // level coordinates, in which flows and targets are
    const int n_d = K.n_desc();
    // a candidate equal to the current flow (or to an already tried one) cannot be strictly cheaper
    const bool e1 = t1 && f1 != cur && K.inside(X + flow_x(f1), Y + flow_y(f1));
    const bool e2 = t2 && f2 != cur && !(t1 && f2 == f1) && K.inside(X + flow_x(f2), Y + flow_y(f2));
    const uint32_t cur0 = cur;
    uint32_t a[C::kSectors][8];
    load_all<C>(K.fa(), K.index(X, Y), n_d, kBoundsOwn, a);
    if (e1 || e2) {
        const uint32_t f = e1 ? f1 : f2;
        uint32_t b[C::kSectors][8];
        load_all<C>(K.fb(), K.index(X + flow_x(f), Y + flow_y(f)), n_d, kBoundsCand1, b);
        const int s1 = dist_all<C>(a, b);
        if (s1 < c) { cur = f; c = s1; }
    }
    if (e1 && e2) {
        uint32_t b[C::kSectors][8];
        load_all<C>(K.fb(), K.index(X + flow_x(f2), Y + flow_y(f2)), n_d, kBoundsCand2, b);
        const int s2 = dist_all<C>(a, b);
        if (s2 < c) { cur = f2; c = s2; }
    }
    if (d >= 1 && (rnd || cur != cur0)) {
        int ox, oy;
        K.random_offset(pixel_key(k1, X, Y), d, ox, oy);
        const int fx = flow_x(cur) + ox, fy = flow_y(cur) + oy;
        if ((ox != 0 || oy != 0) && K.inside(X + fx, Y + fy)) {
            uint32_t b[C::kSectors][8];
            load_all<C>(K.fb(), K.index(X + fx, Y + fy), n_d, kBoundsRandom, b);
            const int s3 = dist_all<C>(a, b);
            if (s3 < c) { cur = pack_flow(fx, fy); c = s3; }
        }
    }
}

// Shared memory of a CTA of the tile and dataflow forms: the head, then for the region (tile + halo, clipped to the
// grid) flow words and state words, row by row, todo bytes and the list.  A row has 2^(slots + 1) pixels (the region's
// width rounded up to a power of two, so that places are shifts and masks).  The todo bytes and the list index the
// pixels of a colour: slot b = (ry + 1) << slots | rx >> 1 for region pixel (rx, ry).  The todo bytes have a row of
// padding above and below the region, so that a pixel's neighbours always have a byte (a mark that runs over the side
// of a row falls on another pixel of the region and only costs it a needless trial).  The layout is one launch's.
struct alignas(16) TileShared {
    Sweep K;
    int lx0, ly0, w, h;    // first pixel of the region, size of the grid
    int x0, y0, x1, y1;    // tile interior
    int RW, RH;            // region
    int4 rect[8];          // region of half-sweep j relative to the loaded region: x0, y0, x1, y1
    int n_list[8];         // its list entries
    TileIO io;
};
constexpr int kHeadWords = 96;
static_assert(sizeof(TileShared) <= 4 * kHeadWords, "head of the shared memory");
constexpr int kMaxSlots = 1 << 13;  // slots a list entry can index

struct TileLayout {
    int slots, rows;  // log2 of the slots of a row; rows of the region
    __host__ __device__ int n_pixels() const { return (2 * rows) << slots; }
    __host__ __device__ int n_slots() const { return (rows + 2) << slots; }  // with the padding
    __host__ __device__ int o_state() const { return kHeadWords + n_pixels(); }
    __host__ __device__ int o_todo() const { return o_state() + n_pixels(); }
    __host__ __device__ int todo_words() const { return n_slots() >> 2; }  // per colour
    __host__ __device__ int o_list() const { return o_todo() + 2 * todo_words(); }
    __host__ size_t bytes() const { return 4 * (size_t)o_list() + 2 * (size_t)n_slots(); }
};
TileLayout tile_layout(int tw, int th) {
    TileLayout T{2, th + 2 * kHaloPerIter};
    while ((2 << T.slots) < tw + 2 * kHaloPerIter) T.slots++;
    return T;
}
size_t prop_launch_smem(int tw, int th, int n_iter, bool listed) {
    return listed ? tile_layout(tw, th).bytes() : prop_smem_bytes(tw, th, n_iter);
}
void prop_fit_tile(int& tw, int& th) {
    for (;;) {
        const TileLayout T = tile_layout(tw, th);
        if (T.bytes() <= kMaxTileSmem && T.n_slots() <= kMaxSlots) return;
        int& longer = th >= tw ? th : tw;
        longer -= (longer + 7) / 8;
    }
}

// The line between the variants, from both timed in their best tiles (all iterations of a pass, WHT-SAD, T = 6, us,
// direct / listed): 167 k pixels 160 / 199, 232 k 235 / 250, 259 k 248 / 248, 346 k 297 / 293, 614 k 360 / 299, 932 k
// 663 / 531, 1.04 M 708 / 527, 4.1 M 2760 / 1674, 5.6 M 3794 / 2800; Census 232 k 147 / 156, 614 k 266 / 217, 4.1 M 1649 /
// 1050.  Below it a half-sweep's chain of dependent loads bounds a pass, not the amount of work, and the direct
// variant's chain is the shorter one.  What does not suit the listed variant keeps the direct one: the tile form (one
// 640x480 direction 795 us listed, 639 direct: a launch per iteration leaves the screening's tail exposed), 128 threads
// (level 0 of the 1242x375 pair in 48x24 tiles: 900 us listed, 663 direct), and regions that leave over a quarter of
// their power-of-two rows empty (64x32 tiles, 72 wide: 688, 669 direct).
// In the first iteration nothing is known yet, so a pass of one iteration has only the lists' cost (level 0 of the 1920x1080
// pair 764 us, 612 direct).  One of two gains from 1.2 M pixels on under Census (4.1 M 541 us, 594 direct in its best
// tiles); under WHT-SAD it depends on the frames (1.26 M, shifted textures, 213, 272 direct; 2.07 M, an animation, 672,
// 629), so it stays direct.
// With fewer tiles than its CTAs (1024 threads per SM) a part of them idles, which the direct variant's half as many do
// not, until enough iterations are skipped (466 k pixels in 198 tiles of 56x40, us, listed / direct: 434 / 274 with three
// iterations, 716 / 539 with six, even with twelve).  Rows of 128 slots gain from more iterations on (1920x1080 direction
// in 120x24 tiles 1164 / 925 with three).
int64_t prop_listed_pixels(int T, int cost) {
    return T >= 3 ? 300000 : T == 2 && cost == FF_COST_CENSUS ? 1200000 : INT64_MAX;
}
bool prop_listed(int64_t pass_pixels, int64_t pass_tiles, int tw, int threads, int T, int cost, bool dataflow, int n_sms) {
    const int RW = tw + 2 * kHaloPerIter;
    int pitch = 8;
    while (pitch < RW) pitch *= 2;
    return dataflow && pass_pixels >= prop_listed_pixels(T, cost) && threads >= 256 && 4 * RW >= 3 * pitch &&
           (T >= 10 || pass_tiles * threads >= (int64_t)n_sms * 1024) && (T >= 6 || pitch <= 64);
}

// The resident variant takes every tile it can (regions of at most one pixel per thread): in the same tiles it was not
// slower in any of 4,320 passes of 1.2 k to 4.1 M pixels, both costs, 1, 3 and 6 iterations, 128 to 512 threads (8x8
// pixels and 256 threads: 57 instead of 73 us at level 4 of the 1242x375 pair, 72 instead of 80 at level 3).
bool prop_resident(int tw, int th, int n_iter, int threads) {
    const int H = kHaloPerIter * n_iter;
    return 2 * ((tw + 2 * H + 1) / 2) * (th + 2 * H) <= threads;
}

extern __shared__ __align__(16) uint32_t g_smem[];
__device__ __forceinline__ TileShared& tile_shared() { return *reinterpret_cast<TileShared*>(g_smem); }
__device__ __forceinline__ SweepRef tile_sweep() { return {fresh(smem_u32(g_smem)) + (uint32_t)offsetof(TileShared, K)}; }
__device__ __forceinline__ int4 tile_origin() { return lds_int4(fresh(smem_u32(g_smem)) + (uint32_t)offsetof(TileShared, lx0)); }

// The flow of the pixel of slot b changed: the neighbours (of the other colour, whose todo bytes these are) that look
// at it and are in `who` (bit 0 the pixel to the right, 1 left, 2 below, 3 above) have it to try.  Of the pixels left
// and right of it, one has the same slot.
__device__ __forceinline__ void mark_neighbours(uint32_t* todo, int b, int slots, int rx, uint32_t who) {
    const bool odd = rx & 1;
    const int sh = 8 * (b & 3);
    uint32_t* at = todo + (b >> 2);
    if (who & 4u) atomicOr(at + (1 << slots >> 2), 4u << sh);
    if (who & 8u) atomicOr(at - (1 << slots >> 2), 8u << sh);
    if (who & (odd ? 2u : 1u)) atomicOr(at, (odd ? 2u : 1u) << sh);
    const int side = odd ? b + 1 : b - 1;
    if (who & (odd ? 1u : 2u)) atomicOr(todo + (side >> 2), (odd ? 1u : 2u) << (8 * (side & 3)));
}

// Screening of the random candidates of the next iteration, at the end of an iteration (k1: the next one's key): for
// every pixel of the tile, the candidates of directions 1..3 around its present flow are scored side by
// side, sector by sector, each until its partial distance reaches the pixel's cost.  A candidate that reaches it is
// not cheaper, and stays so while the pixel keeps its flow; the others (a few per cent) are flagged in the state word
// and scored again in their half-sweep, as are those of pixels whose flow has changed by then.  So the own descriptor is loaded
// once per iteration instead of once per direction, candidates of matched pixels are mostly dropped after one of their
// three sectors, three gathers are in flight per thread, the half-sweeps are left with few pixels, and a tile screens
// its own pixels only: the flags of its halo come with the state its neighbours wrote.
// What bounds it is L1 (a quarter to a third of a pass at level 0).  So both colours go row by row, not one colour
// after the other: a 128-byte line holds parts of two pixels' descriptors, and the second finds it in L1 (level 0 of
// the 1920x1080 pair 1700 us, 1770 colour by colour; of the 1242x375 pair 538, 543).  Within a row the columns of even
// x come first; plain rows (1708, 538) and warps of 16x2, 8x4 and 4x8 pixels (1725, 1700, 1710; 540, 538, 540) are no
// faster.
template <class C, int THREADS>
__device__ __forceinline__ void screen(const TileLayout T, const int4 r, uint32_t k1) {
    const int tid = (int)fresh(threadIdx.x);
    const int W = r.z - r.x, total = W * (r.w - r.y);
    const uint32_t inv = 0xffffffffu / (uint32_t)W + 1u;  // ceil(2^32 / W): i / W = umulhi(i, inv) for i < 2^15
#pragma unroll 1
    for (int i = tid; i < total; i += THREADS) {
        const int4 O = tile_origin();
        const SweepRef K = tile_sweep();
        const int row = W > 1 ? (int)__umulhi((uint32_t)i, inv) : i, k = i - row * W;
        const int odd = (O.x + r.x) & 1, n_even = (W + 1 - odd) >> 1;  // columns of even x, then those of odd x
        const int ry = r.y + row, rx = r.x + (k < n_even ? 2 * k + odd : 2 * (k - n_even) + 1 - odd);
        const int sidx = (ry << (T.slots + 1)) + rx;
        if (!idx_ok(g_bounds, kBoundsSmemOwn, sidx, T.n_pixels())) continue;
        const uint32_t cur = g_smem[kHeadWords + sidx];
        const int c = (int)(g_smem[T.o_state() + sidx] >> kCostShift);
        const int g = K.g(), X = g * (O.x + rx), Y = g * (O.y + ry), n_d = K.n_desc();
        uint32_t live = 0;
        int idx[3], s[3];
        {
            const int cx = X + flow_x(cur), cy = Y + flow_y(cur);
            const uint32_t k2 = pixel_key(k1, X, Y);
#pragma unroll
            for (int q = 0; q < 3; q++) {
                int ox, oy;
                K.random_offset(k2, q + 1, ox, oy);
                if ((ox != 0 || oy != 0) && K.inside(cx + ox, cy + oy)) live |= 1u << q;
                idx[q] = K.index(cx + ox, cy + oy);
                s[q] = 0;
            }
        }
        const int own = K.index(X, Y);
#pragma unroll
        for (int k = 0; k < C::kSectors; k++) {
            if (!live) break;
            uint32_t a[8], b[3][8] = {};
            load_chk<C>(K.fa(), own, n_d, kBoundsOwn, k, a);
#pragma unroll
            for (int q = 0; q < 3; q++)
                if (live >> q & 1u) load_chk<C>(K.fb(), idx[q], n_d, kBoundsRandom, k, b[q]);
#pragma unroll
            for (int q = 0; q < 3; q++)
                if (live >> q & 1u) {
                    s[q] = C::dist(a, b[q], s[q]);
                    if (s[q] >= c) live &= ~(1u << q);
                }
        }
        if (live) g_smem[T.o_state() + sidx] |= live << kFlagShift;
    }
}

// One half-sweep of a tile's region.  The CTA collects the pixels of the region's rows whose
// todo bytes hold something to try in this direction in a list (four pixels per thread and read, placed by ballots and
// one counter), and updates them from the list, one per thread: a half-sweep with few such pixels costs few gathers
// and few instructions.  A list entry is the slot and three bits, what to try: neighbour 1, neighbour 2, random.
template <class C, int THREADS>
__device__ __forceinline__ void halfsweep(const TileLayout T, int j, uint32_t k1) {
    const int tid = (int)fresh(threadIdx.x);
    const int d = j >> 1, colour = j & 1;
    uint32_t* const mine = g_smem + T.o_todo() + colour * T.todo_words();
    uint16_t* const list = reinterpret_cast<uint16_t*>(g_smem + T.o_list());
    {
        const int4 r = tile_shared().rect[j];
        const uint32_t bits = todo_bits(d) * 0x01010101u;
        const int lane = tid & 31, w1 = (r.w + 1) << T.slots >> 2;
#pragma unroll 1
        for (int base = ((r.y + 1) << T.slots >> 2) + (tid & ~31); base < w1; base += THREADS) {
            const int i = base + lane;
            uint32_t v = 0;
            if (i < w1) {
                v = mine[i];
                if (v & bits) mine[i] = v & ~bits;  // (a neighbour tried now needs no trial until it changes again)
                v &= bits;
            }
            if (!__any_sync(0xffffffffu, v != 0)) continue;
            uint32_t nz = (v + kTodoAll) & 0x80808080u;  // bit 7 of every byte with something to try
            const unsigned cnt = __popc(nz), below = (1u << lane) - 1u;
            const unsigned c0 = __ballot_sync(0xffffffffu, cnt & 1u), c1 = __ballot_sync(0xffffffffu, cnt & 2u),
                           c2 = __ballot_sync(0xffffffffu, cnt & 4u);
            int pos = 0;
            if (lane == 0) pos = atomicAdd(&tile_shared().n_list[j], __popc(c0) + 2 * __popc(c1) + 4 * __popc(c2));
            pos = __shfl_sync(0xffffffffu, pos, 0) + __popc(c0 & below) + 2 * __popc(c1 & below) + 4 * __popc(c2 & below);
#pragma unroll 1
            while (nz) {
                const int s = __ffs((int)nz) - 8;  // first bit of the byte
                const uint32_t t = v >> s;
                list[pos++] = (uint16_t)((uint32_t)(4 * i + (s >> 3)) | (t & 3u ? 0x2000u : 0u) | (t & 12u ? 0x4000u : 0u) |
                                         (t & 0x70u ? 0x8000u : 0u));
                nz &= nz - 1;
            }
        }
    }
    __syncthreads();
    const int n = tile_shared().n_list[j];
    if (n == 0) return;  // (uniform)
#pragma unroll 1
    for (int i = tid; i < n; i += THREADS) {
        const uint32_t e = list[i];
        const int4 O = tile_origin();
        const int b = (int)(e & 0x1fffu), ry = (b >> T.slots) - 1;
        const int rx = 2 * (b & ((1 << T.slots) - 1)) + ((O.x + O.y + ry + colour) & 1);
        const int sidx = (ry << (T.slots + 1)) + rx;
        const int4 r = lds_int4(fresh(smem_u32(&tile_shared().rect[j])));
        if (rx < r.x || rx >= r.z || !idx_ok(g_bounds, kBoundsSmemOwn, sidx, T.n_pixels())) continue;
        const int x = O.x + rx, y = O.y + ry;
        uint32_t cur = g_smem[kHeadWords + sidx];
        const uint32_t cur0 = cur;
        int c = (int)(g_smem[T.o_state() + sidx] >> kCostShift);
        const int n1 = sidx + ((d & 1) ? 1 : -1), n2 = sidx + ((d & 2) ? 2 << T.slots : -(2 << T.slots));
        const bool t1 = (e & 0x2000u) && (unsigned)(x + ((d & 1) ? 1 : -1)) < (unsigned)O.z &&
                        idx_ok(g_bounds, kBoundsSmemN1, n1, T.n_pixels());
        const bool t2 = (e & 0x4000u) && (unsigned)(y + ((d & 2) ? 1 : -1)) < (unsigned)O.w &&
                        idx_ok(g_bounds, kBoundsSmemN2, n2, T.n_pixels());
        const uint32_t f1 = t1 ? g_smem[kHeadWords + n1] : 0u, f2 = t2 ? g_smem[kHeadWords + n2] : 0u;
        update_pixel<C>(tile_sweep(), x, y, d, k1, t1, f1, t2, f2, (e & 0x8000u) != 0, cur, c);
        if (cur != cur0) {
            g_smem[kHeadWords + sidx] = cur;
            g_smem[T.o_state() + sidx] = (uint32_t)c << kCostShift | (uint32_t)(j + 1);
            mark_neighbours(g_smem + T.o_todo() + (colour ^ 1) * T.todo_words(), b, T.slots, rx, 15u);
            if (d < 3) atomicOr(mine + (b >> 2), ((0x70u << d) & 0x70u) << (8 * (b & 3)));  // random candidates to come
        }
    }
    __syncthreads();
}

// Regions of the half-sweeps, without list entries yet (threads 0..7).
__device__ __forceinline__ void set_regions() {
    const int j = threadIdx.x;
    TileShared& S = tile_shared();
    if (j < 8) {
        S.rect[j] = make_int4(max(S.x0 - c_grow[j][0], 0) - S.lx0, max(S.y0 - c_grow[j][1], 0) - S.ly0,
                              min(S.x1 + c_grow[j][2], S.w) - S.lx0, min(S.y1 + c_grow[j][3], S.h) - S.ly0);
        S.n_list[j] = 0;
    }
}

// One tile of one problem: load the tile and its halo, run iteration io.t0 in shared memory, write the tile.  The state
// was written by other CTAs of the running launch and is therefore read from L2.  Between the tasks of a pass the cost
// buffers hold state words; a pass starts from plain costs and its last iteration leaves plain costs.  The head of the shared memory is set (tile_setup).
// With a counter, the CTA's next task is taken while this one is written, into *s_next.
template <class C, int THREADS>
__device__ __forceinline__ void propagate_tile_listed(const PropProblem& P, const TileLayout T, int* counter, int* s_next) {
    TileShared& S = tile_shared();
    {
        uint32_t* todo = g_smem + T.o_todo();
        const int RW = S.RW, n_s = RW * S.RH, n_todo = 2 * T.todo_words();
        const bool first = S.io.t0 == 0;  // of the pass: everything is still to be tried
#pragma unroll 1
        for (int i = threadIdx.x; i < n_todo; i += THREADS)  // (nothing for the slots past the region's width)
            todo[i] = first && 8 * (i & ((1 << T.slots >> 2) - 1)) < RW ? kTodoAll : 0u;
        set_regions();
        if (!first) __syncthreads();
        const uint32_t inv = 0xffffffffu / (uint32_t)RW + 1u;
#pragma unroll 1
        for (int i = threadIdx.x; i < n_s; i += THREADS) {
            const int r = RW > 1 ? (int)__umulhi((uint32_t)i, inv) : i, c = i - r * RW;
            const size_t g = (size_t)(S.ly0 + r) * S.w + S.lx0 + c;
            // the region must fit the launch's dynamic shared memory
            const bool ok = idx_ok(g_bounds, kBoundsTileRead, (long long)g, (long long)S.w * S.h) &&
                            (!FF_DEBUG_BOUNDS || (idx_ok(g_bounds, kBoundsTileSmem, RW - 1, 2 << T.slots) &&
                                                  idx_ok(g_bounds, kBoundsTileSmem, S.RH - 1, T.rows) &&
                                                  idx_ok(g_bounds, kBoundsTileSmem, 4 * T.o_list() + 2 * T.n_slots() - 1,
                                                         dyn_smem_bytes())));
            uint32_t f = 0, st = 0;
            if (ok) {
                f = __ldcg(S.io.flow_in + g);
                st = (uint32_t)__ldcg(S.io.cost_in + g);
            }
            const int sidx = (r << (T.slots + 1)) + c;
            g_smem[kHeadWords + sidx] = f;
            g_smem[T.o_state() + sidx] = first ? pack_state((int)st) : st >> kCostShift << kCostShift;
            if (!first && (st & ((1u << kCostShift) - 1))) {
                const uint32_t live = st >> kFlagShift & 7u, stamp = st & kStampMask;
                const uint32_t who = still_concerned(stamp);
                const int colour = (S.lx0 + c + S.ly0 + r) & 1, b = ((r + 1) << T.slots) + (c >> 1);
                if (live) atomicOr(todo + colour * T.todo_words() + (b >> 2), live << (8 * (b & 3) + 4));
                if (who) mark_neighbours(todo + (colour ^ 1) * T.todo_words(), b, T.slots, c, who);
            }
        }
        __syncthreads();
    }
    const int t = S.io.t0;
    const bool plain = t + 1 == P.T;
    const uint32_t k1 = iter_key(P, t);
#pragma unroll 1
    for (int j = 0; j < 8; j++) halfsweep<C, THREADS>(T, j, k1);
    if (!plain) {
        const uint32_t kn = iter_key(P, t + 1);
        screen<C, THREADS>(T, S.rect[7], kn);  // of the tile
    }
    __syncthreads();
    int next = 0;
    if (counter && threadIdx.x == 0) next = atomicAdd(counter, 1);
    const int TW = S.x1 - S.x0, n_out = TW * (S.y1 - S.y0);
    const uint32_t inv = 0xffffffffu / (uint32_t)TW + 1u;
#pragma unroll 1
    for (int i = threadIdx.x; i < n_out; i += THREADS) {
        const int r = TW > 1 ? (int)__umulhi((uint32_t)i, inv) : i, c = i - r * TW;
        const int sidx = ((S.y0 + r - S.ly0) << (T.slots + 1)) + (S.x0 + c - S.lx0);
        const size_t g = (size_t)(S.y0 + r) * S.w + S.x0 + c;
        if (!idx_ok(g_bounds, kBoundsTileWrite, (long long)g, (long long)S.w * S.h) ||
            !idx_ok(g_bounds, kBoundsTileSmem, sidx, T.n_pixels()))
            continue;
        S.io.flow_out[g] = g_smem[kHeadWords + sidx];
        const uint32_t st = g_smem[T.o_state() + sidx];
        S.io.cost_out[g] = (int32_t)(plain ? st >> kCostShift : st);
    }
    if (counter && threadIdx.x == 0) *s_next = next;
}

// Problem and geometry of the CTA's next tile, by one thread.
__device__ __forceinline__ void tile_setup(const PropProblem& P, int tile, const PropLaunch& L) {
    TileShared& S = tile_shared();
    S.K.set(P, L.grid != 0);
    S.w = P.w;
    S.h = P.h;
    S.x0 = (tile % P.tiles_x) * L.tw;
    S.y0 = (tile / P.tiles_x) * L.th;
    S.x1 = min(S.x0 + L.tw, P.w);
    S.y1 = min(S.y0 + L.th, P.h);
    S.lx0 = max(S.x0 - kHaloPerIter, 0);
    S.ly0 = max(S.y0 - kHaloPerIter, 0);
    S.RW = min(S.x1 + kHaloPerIter, P.w) - S.lx0;
    S.RH = min(S.y1 + kHaloPerIter, P.h) - S.ly0;
}

// Persistent launch: each CTA takes tiles from the launch's queue until it is empty, so the last wave has no idle tail.
// CTA b starts with entry b; the others are taken with an atomic counter (zeroed before the launch), and a launch with a
// CTA per tile takes none.  At small levels a launch is a chain of memory round trips, of which this leaves out two (level
// 4 of the 1242x375 pair 64 -> 61 us, level 3 79 -> 77; the three launches of the 32x24 level of the 128x96 pair 61 -> 58).
// A CTA takes its next tile when it has finished the one before: taken at that one's start, the launch's last tiles are
// held by CTAs that are still busy while others idle (a 128x96 pair in 8x8 tiles of three iterations 298 instead of 268
// us, a 1242x375 direction without allocation 1001 instead of 953, 1920x1080 in 32x32 tiles under Census 2985, 2960).
// queue[i] = (problem index, tile index in problem).
// Instantiated for 128, 256 and 512 threads, per cost, direct and resident.
// The Census kernels are held to the registers of three CTAs of 256 threads per SM (direct 78, resident 71; unbounded 92
// and 85, two CTAs).  Direct: a 1920x1080 pair in 32x32 tiles 2.96 instead of 3.63 ms, a 1024x436 direction without
// allocation 510 instead of 630 us.  Resident: 27.9 k pixels in 8x8 tiles (448 of them, on 304 CTAs two rounds) 57 us
// instead of 90.
template <int THREADS, class C, bool RES>
__global__ __launch_bounds__(THREADS, (C::kSectors > 1 ? 512 : 768) / THREADS) void k_propagate(
    const PropProblem* __restrict__ probs, const int2* __restrict__ queue, int n_tiles, int* __restrict__ counter,
    PropLaunch L) {
    grid_dependency_sync();
    __shared__ int s_next;
    const int G = (int)gridDim.x;
    for (int q = (int)blockIdx.x; q < n_tiles; q = s_next) {
        const int2 e = queue[q];
        const PropProblem& P = probs[e.x];
        const TileIO io = {P.flow_in, P.cost_in, P.flow_out, P.cost_out, P.t0, P.n_iter};
        propagate_tile_direct<C, false, RES>(P, e.y, L, g_smem, io);
        if (G >= n_tiles) return;
        if (threadIdx.x == 0) s_next = G + atomicAdd(counter, 1);
        __syncthreads();
    }
}

// Dataflow form: every iteration of a level in one persistent launch.  Task q is iteration t = q / n_tiles of
// queue entry q % n_tiles (tasks are taken in that order); it starts once the 3x3 tiles around its tile, itself
// included, have finished iteration t - 1, so no launch boundary separates the iterations and a CTA that
// finishes early goes on with the next iteration's tiles.  A task of iteration t reads its region (the tile and
// a halo of one iteration, kHaloPerIter <= tile size, so inside those nine tiles) from the buffer iteration t - 1
// wrote and writes its tile to the next: flow_alt for even t, flow_in for odd t, flow_out for the last (a buffer
// the host keeps apart from the one the iteration before wrote).  A tile overwrites a buffer its neighbours read
// one iteration earlier only after they finished that iteration, by the same rule.  Progress is published with
// a release after the tile's stores and read with an acquire; the region is then read from L2.  A task waits
// only for tasks taken before it by running CTAs, so there is no deadlock whatever the residency; every wait is
// bounded (wait_limit polls; on expiry kErrDataflow goes to the error word and the CTA stops waiting).
// The round trips between two tasks overlap where they may: a warp that neither takes tasks nor polls publishes the
// finished one, and the listed variant takes its next task while it writes the present one (which waits for nothing any
// more, so the argument above holds): level 0 of the 1242x375 pair 538 -> 531 us, of the 1920x1080 pair 1700 -> 1674
// (with Census 290 -> 294).  A task taken at the start of the one before is held too long (682, 1855), and in the
// direct variant, with a tile or two per CTA and iteration, even one taken that late is (level 2: 109 -> 113).
// Affine variant (L.affine): no queue counter; CTA b owns entries b, b + G, ... of every iteration (G CTAs, at
// most the resident ones) and runs them iteration by iteration, keeping its tiles' descriptors in its L1.  Its
// waits are for iteration t - 1 of tiles other CTAs own, which wait only for earlier iterations, so every CTA
// makes progress once the grid is resident (with the grid sized to the resident CTAs, it is).
__device__ __forceinline__ int ld_acquire_gpu(const int* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release_gpu(int* p, int v) {
    asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// CTAs per SM: the listed variant is held to the registers of 1024 threads, the others to those of 512, under Census of
// 640, so that five CTAs of 128 threads reside (direct 86 registers, unbounded 102 and four CTAs: level 0 of a 1920x1080
// pair in 32x32 tiles 1628 instead of 1919 us).
template <int THREADS, class C, Variant V>
__global__ __launch_bounds__(THREADS, (V == kListed ? 1024 : C::kSectors > 1 ? 512 : 640) / THREADS) void k_propagate_df(
    const PropProblem* __restrict__ probs, const int2* __restrict__ queue, int n_tiles, int* __restrict__ counter,
    PropLaunch L, TileLayout LT) {
    grid_dependency_sync();
    __shared__ int s_next;
    const int T = L.dataflow, n_tasks = n_tiles * T;
    bool failed = false;  // a wait of this CTA expired: stop waiting (CTA-uniform)
    // affine: CTA b owns queue entries b, b + G, b + 2G, ... (G CTAs) for every iteration and runs them
    // iteration by iteration, so a tile's region stays in the same SM's L1 from one iteration to the next
    const int G = (int)gridDim.x, per_iter = (n_tiles - (int)blockIdx.x + G - 1) / G;  // entries this CTA owns
    for (int k = 0;; k++) {
        int q;
        if (L.affine) {
            if (k >= per_iter * T) return;
            const int ti = k / per_iter;
            q = ti * n_tiles + (int)blockIdx.x + (k - ti * per_iter) * G;
        } else {
            if (V != kListed || k == 0) {
                if (threadIdx.x == 0) s_next = atomicAdd(counter, 1);
                __syncthreads();
            }
            q = s_next;
            if (q >= n_tasks) return;
        }
        const int t = q / n_tiles;
        const int2 e = queue[q - t * n_tiles];
        const PropProblem& P = probs[e.x];
        const bool src_alt = t > 0 && ((t - 1) & 1) == 0;  // iteration t - 1 wrote flow_alt iff t - 1 is even
        const bool dst_alt = (t & 1) == 0;
        const TileIO io = {src_alt ? P.flow_alt : P.flow_in, src_alt ? P.cost_alt : P.cost_in,
                           t == T - 1 ? P.flow_out : dst_alt ? P.flow_alt : P.flow_in,
                           t == T - 1 ? P.cost_out : dst_alt ? P.cost_alt : P.cost_in, P.t0 + t, 1};
        if constexpr (V == kListed)
            if (threadIdx.x == 32) tile_setup(P, e.y, L), tile_shared().io = io;
        bool ok = true;
        if (t > 0 && !failed && threadIdx.x < 9) {  // one waiting thread per tile of the 3x3 neighbourhood
            const int tiles_y = (P.h + L.th - 1) / L.th;
            const int nx = e.y % P.tiles_x + (int)threadIdx.x % 3 - 1, ny = e.y / P.tiles_x + (int)threadIdx.x / 3 - 1;
            if (nx >= 0 && nx < P.tiles_x && ny >= 0 && ny < tiles_y) {
                const int* f = P.progress + ny * P.tiles_x + nx;
                ok = false;
                for (uint32_t i = 0; i < L.wait_limit && !ok; i++) {
                    ok = ld_acquire_gpu(f) >= t;
                    if (!ok && i > 64) __nanosleep(128);
                }
                if (!ok) atomicCAS(L.err, 0, kErrDataflow);
            }
        }
        failed = __syncthreads_or(!ok) != 0 || failed;
        if constexpr (V == kListed)
            propagate_tile_listed<C, THREADS>(P, LT, L.affine ? nullptr : counter, &s_next);
        else
            propagate_tile_direct<C, true, V == kResident>(P, e.y, L, g_smem, io);
        __syncthreads();  // every store of the tile is issued
        if (threadIdx.x == 64 && !L.withhold) {
            __threadfence();
            st_release_gpu(P.progress + e.y, t + 1);
        }
    }
}

// ---------------------------------------------------------------------------------------------------------
// Cluster form: one cluster of n CTAs per problem runs every iteration of the launch over the whole grid, with no
// halo recomputation.  CTA r owns block r of the partition cluster_partition() gives and keeps the block's flow
// and cost in shared memory, with a one-pixel ring of the neighbouring blocks' edge flows.  After computing an
// edge pixel of the active colour, a CTA stores its flow straight into the ring of each CTA beside that edge
// (st.async into the neighbour's shared memory, completing 4 bytes on the neighbour's mbarrier of that
// half-sweep), and before the next half-sweep reads its ring it waits on its own mbarrier for the edges it
// receives.  The waits are CTA-scope: a cluster-wide barrier per half-sweep, an acquire at cluster scope, also
// emptied the L1 that the next half-sweep's gathers reuse (8 % L1 hits instead of 83 % at level 4 of the
// 1242x375 pair).  A half-sweep reads exactly the state the previous one left, so the schedule is the tile
// form's, evaluated once per pixel.  Every wait is bounded (wait_limit polls); one that expires records
// kErrClusterEdges in the error word and the CTA stops waiting (the launch runs to its end; ff_sync then fails).
// An alternative for small levels of a few problems, where the tile form's halo is most of the work; the
// autotuner weighs the two forms per level.

__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ int cluster_rank() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return (int)r;
}
__device__ __forceinline__ int cluster_ctas() {
    uint32_t n;
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(n));
    return (int)n;
}
// Address, in the cluster's shared-memory window, of `p` (this CTA's shared memory) in CTA `rank`.
__device__ __forceinline__ uint32_t cluster_addr(const void* p, int rank) {
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
    return a;
}
// 4-byte store into another CTA's shared memory that completes 4 bytes on the mbarrier `bar` (cluster window).
__device__ __forceinline__ void st_async_u32(uint32_t addr, uint32_t v, uint32_t bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(addr), "r"(v),
                 "r"(bar)
                 : "memory");
}
// Number of v in [a, b) with (k + v) of colour c ((k + v) & 1 == c).
__device__ __forceinline__ int colour_count(int k, int a, int b, int c) {
    const int first = a + ((c - k - a) & 1);
    return first < b ? (b - 1 - first) / 2 + 1 : 0;
}

template <int THREADS, class C>
__global__ __launch_bounds__(THREADS, 1) void k_propagate_cl(const PropProblem* __restrict__ probs, PropLaunch L) {
    grid_dependency_sync();
    uint32_t* smem = g_smem;
    const int n = cluster_ctas(), r = cluster_rank();
    const PropProblem& P = probs[blockIdx.x / n];
    const int w = P.w, h = P.h;
    int bx = 1, by = 1;
    cluster_partition(w, h, n, bx, by);  // the host launches only problems that have a partition
    const int bi = r % bx, bj = r / bx;
    const int x0 = bi * w / bx, x1 = (bi + 1) * w / bx, y0 = bj * h / by, y1 = (bj + 1) * h / by;
    const int bw = x1 - x0, bh = y1 - y0, nb = bw * bh;
    const int mw = (w + bx - 1) / bx, mh = (h + by - 1) / by;
    uint64_t* mbar = reinterpret_cast<uint64_t*>(smem);  // [2]: the edges received in even / odd half-sweeps
    uint32_t* ring_l = smem + 4;                         // [mh] flows of column x0 - 1
    uint32_t* ring_r = ring_l + mh;                      // [mh] column x1
    uint32_t* ring_u = ring_r + mh;                      // [mw] row y0 - 1
    uint32_t* ring_d = ring_u + mw;                      // [mw] row y1
    uint32_t* sflow = ring_d + mw;                       // [mw * mh] the block, row-major with width bw
    int32_t* scost = reinterpret_cast<int32_t*>(sflow + mw * mh);
    const bool has_l = bi > 0, has_r = bi + 1 < bx, has_u = bj > 0, has_d = bj + 1 < by;
    // an edge pixel's flow goes to the opposite ring of the CTA beside it, completing on that CTA's mbarrier
    const uint32_t to_l = has_l ? cluster_addr(ring_r, r - 1) : 0u, mb_l = has_l ? cluster_addr(mbar, r - 1) : 0u;
    const uint32_t to_r = has_r ? cluster_addr(ring_l, r + 1) : 0u, mb_r = has_r ? cluster_addr(mbar, r + 1) : 0u;
    const uint32_t to_u = has_u ? cluster_addr(ring_d, r - bx) : 0u, mb_u = has_u ? cluster_addr(mbar, r - bx) : 0u;
    const uint32_t to_d = has_d ? cluster_addr(ring_u, r + bx) : 0u, mb_d = has_d ? cluster_addr(mbar, r + bx) : 0u;
    // bytes received per half-sweep of colour c: the neighbours' edge pixels of that colour next to this block
    uint32_t rx_bytes[2];
#pragma unroll
    for (int c = 0; c < 2; c++)
        rx_bytes[c] = 4u * (uint32_t)((has_l ? colour_count(x0 - 1, y0, y1, c) : 0) +
                                      (has_r ? colour_count(x1, y0, y1, c) : 0) +
                                      (has_u ? colour_count(y0 - 1, x0, x1, c) : 0) +
                                      (has_d ? colour_count(y1, x0, x1, c) : 0));
    const bool fits = !FF_DEBUG_BOUNDS ||
                      idx_ok(g_bounds, kBoundsBlockSmem, (long long)cluster_smem_bytes(w, h, bx, by) - 1,
                             dyn_smem_bytes());
    const int J = 8 * P.n_iter;
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&mbar[0]), 1);
        mbar_init(smem_u32(&mbar[1]), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        // half-sweeps 0 and 1: the first phase of each mbarrier (a colour with no edges to receive never waits)
        if (rx_bytes[0] != 0) mbar_expect_tx(smem_u32(&mbar[0]), rx_bytes[0]);
        if (J > 1 && rx_bytes[1] != 0) mbar_expect_tx(smem_u32(&mbar[1]), rx_bytes[1]);
    }
    // the block and the ring from the launch's input state
    const long long n_in = (long long)w * h;
    for (int i = threadIdx.x; i < nb; i += THREADS) {
        const long long gi = (long long)(y0 + i / bw) * w + x0 + i % bw;
        const bool ok = fits && idx_ok(g_bounds, kBoundsBlockRead, gi, n_in);
        sflow[i] = ok ? P.flow_in[gi] : 0u;
        scost[i] = ok ? P.cost_in[gi] : 0;
    }
    for (int i = threadIdx.x; i < bh; i += THREADS) {
        const long long left = (long long)(y0 + i) * w + x0 - 1, right = (long long)(y0 + i) * w + x1;
        if (has_l && fits && idx_ok(g_bounds, kBoundsBlockRead, left, n_in)) ring_l[i] = P.flow_in[left];
        if (has_r && fits && idx_ok(g_bounds, kBoundsBlockRead, right, n_in)) ring_r[i] = P.flow_in[right];
    }
    for (int i = threadIdx.x; i < bw; i += THREADS) {
        const long long up = (long long)(y0 - 1) * w + x0 + i, down = (long long)y1 * w + x0 + i;
        if (has_u && fits && idx_ok(g_bounds, kBoundsBlockRead, up, n_in)) ring_u[i] = P.flow_in[up];
        if (has_d && fits && idx_ok(g_bounds, kBoundsBlockRead, down, n_in)) ring_d[i] = P.flow_in[down];
    }
    cluster_sync_all();  // every CTA of the cluster running, its block loaded and its mbarriers armed
    const int HW = (bw + 1) >> 1, total = HW * bh;
    const SweepConst K = sweep_const(P, L.grid != 0);
    bool failed = false;  // a wait expired: stop waiting (CTA-uniform)
    uint32_t k1 = 0;
    for (int j = 0; j < J; j++) {
        if ((j & 7) == 0) {
            const uint32_t t = (uint32_t)(P.t0 + (j >> 3));
            k1 = mix32(P.seed ^ mix32((uint32_t)P.dir * 65536u + (uint32_t)P.level * 256u + t));
        }
        const int d = (j & 7) >> 1, colour = j & 1;
        const uint32_t slot = 8u * (uint32_t)(j & 1);  // byte offset of this half-sweep's mbarrier
        for (int i = threadIdx.x; i < total; i += THREADS) {
            const int row = i / HW, slot_x = i - row * HW;
            const int y = y0 + row;
            const int x = x0 + 2 * slot_x + ((x0 + y + colour) & 1);
            if (x >= x1 || !fits) continue;
            const int sidx = row * bw + (x - x0);
            uint32_t cur = sflow[sidx];
            int c = scost[sidx];
            const int n1x = x + ((d & 1) ? 1 : -1);
            const int n2y = y + ((d & 2) ? 1 : -1);
            const bool v1 = (unsigned)n1x < (unsigned)w;
            const bool v2 = (unsigned)n2y < (unsigned)h;
            uint32_t f1 = 0u, f2 = 0u;
            if (v1) {
                if (n1x < x0)
                    f1 = idx_ok(g_bounds, kBoundsRingN1, row, mh) ? ring_l[row] : 0u;
                else if (n1x >= x1)
                    f1 = idx_ok(g_bounds, kBoundsRingN1, row, mh) ? ring_r[row] : 0u;
                else
                    f1 = sflow[sidx + (n1x - x)];
            }
            if (v2) {
                if (n2y < y0)
                    f2 = idx_ok(g_bounds, kBoundsRingN2, x - x0, mw) ? ring_u[x - x0] : 0u;
                else if (n2y >= y1)
                    f2 = idx_ok(g_bounds, kBoundsRingN2, x - x0, mw) ? ring_d[x - x0] : 0u;
                else
                    f2 = sflow[sidx + (n2y - y) * bw];
            }
            if (update_direct<C>(K, x, y, d, k1, v1, f1, v2, f2, cur, c)) {
                sflow[sidx] = cur;
                scost[sidx] = c;
            }
            if (!L.withhold) {  // every edge pixel of the colour is sent, changed or not (fixed byte counts)
                if (has_l && x == x0) st_async_u32(to_l + 4u * row, cur, mb_l + slot);
                if (has_r && x == x1 - 1) st_async_u32(to_r + 4u * row, cur, mb_r + slot);
                if (has_u && y == y0) st_async_u32(to_u + 4u * (x - x0), cur, mb_u + slot);
                if (has_d && y == y1 - 1) st_async_u32(to_d + 4u * (x - x0), cur, mb_d + slot);
            }
        }
        // the neighbours' edges of this colour, read by the next half-sweep
        const bool rx = rx_bytes[j & 1] != 0;
        // (this wait is on the critical path of every half-sweep: spin for the first 4096 polls, then sleep)
        const bool ok =
            failed || !rx || mbar_wait(smem_u32(&mbar[j & 1]), (uint32_t)(j >> 1) & 1u, L.wait_limit, 4096);
        if (!ok) atomicCAS(L.err, 0, kErrClusterEdges);
        // the same mbarrier's next phase, half-sweep j + 2, armed before this CTA sends any edge of half-sweep
        // j + 1 (which the neighbours' sends of j + 2 wait for); as it expects bytes, it cannot complete before
        // every thread here has seen this phase complete, for the same reason
        if (threadIdx.x == 0 && rx && ok && !failed && j + 2 < J)
            mbar_expect_tx(smem_u32(&mbar[j & 1]), rx_bytes[j & 1]);
        failed = __syncthreads_or(!ok) != 0 || failed;
    }
    for (int i = threadIdx.x; i < nb; i += THREADS) {
        const long long gi = (long long)(y0 + i / bw) * w + x0 + i % bw;
        if (!fits || !idx_ok(g_bounds, kBoundsBlockWrite, gi, n_in)) continue;
        P.flow_out[gi] = sflow[i];
        P.cost_out[gi] = scost[i];
    }
    cluster_sync_all();  // no CTA leaves while edge stores of its neighbours may still target its shared memory
}

using PropKernel = void (*)(const PropProblem*, const int2*, int, int*, PropLaunch);
using PropClusterKernel = void (*)(const PropProblem*, PropLaunch);

using PropDataflowKernel = void (*)(const PropProblem*, const int2*, int, int*, PropLaunch, TileLayout);

template <class C, bool RES>
PropKernel prop_kernel_t(int threads) {
    return threads == 128   ? k_propagate<128, C, RES>
           : threads == 512 ? k_propagate<512, C, RES>
                            : k_propagate<256, C, RES>;
}
PropKernel prop_kernel(int threads, int cost, bool resident) {
    if (resident)
        return cost == FF_COST_CENSUS ? prop_kernel_t<CostCensus, true>(threads) : prop_kernel_t<CostSad, true>(threads);
    return cost == FF_COST_CENSUS ? prop_kernel_t<CostCensus, false>(threads) : prop_kernel_t<CostSad, false>(threads);
}

// The listed variant is instantiated for 256 and 512 threads (prop_listed), the others for 128 too.
template <class C, Variant V>
PropDataflowKernel prop_df_kernel_t(int threads) {
    if constexpr (V != kListed)
        if (threads == 128) return k_propagate_df<128, C, V>;
    return threads == 512 ? k_propagate_df<512, C, V> : k_propagate_df<256, C, V>;
}
template <Variant V>
PropDataflowKernel prop_df_kernel_v(int threads, int cost) {
    return cost == FF_COST_CENSUS ? prop_df_kernel_t<CostCensus, V>(threads) : prop_df_kernel_t<CostSad, V>(threads);
}
PropDataflowKernel prop_df_kernel(int threads, int cost, Variant v) {
    return v == kListed     ? prop_df_kernel_v<kListed>(threads, cost)
           : v == kResident ? prop_df_kernel_v<kResident>(threads, cost)
                            : prop_df_kernel_v<kDirect>(threads, cost);
}

// The cluster form is instantiated for 256 and 512 threads, per cost.
PropClusterKernel prop_cl_kernel(int threads, int cost) {
    if (cost == FF_COST_CENSUS) return threads == 512 ? k_propagate_cl<512, CostCensus> : k_propagate_cl<256, CostCensus>;
    return threads == 512 ? k_propagate_cl<512, CostSad> : k_propagate_cl<256, CostSad>;
}

cudaLaunchConfig_t cluster_config(int n_ctas, int cluster, int threads, size_t smem, cudaStream_t st,
                                  cudaLaunchAttribute (&attr)[2]) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(n_ctas);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = FF_PDL;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cfg;
}

cudaError_t init_kernel_attributes() {
    cudaFuncAttributes fa;
    cudaError_t e0 = cudaFuncGetAttributes(&fa, k_handover<CostSad>);
    if (e0 == cudaSuccess) e0 = cudaFuncGetAttributes(&fa, k_handover<CostCensus>);
    if (e0 != cudaSuccess) return e0;
    for (int cost : {FF_COST_WHT_SAD, FF_COST_CENSUS}) {
        for (int t : {128, 256, 512}) {
            const void* ks[5] = {reinterpret_cast<const void*>(prop_kernel(t, cost, false)),
                                 reinterpret_cast<const void*>(prop_kernel(t, cost, true)),
                                 reinterpret_cast<const void*>(prop_df_kernel(t, cost, kDirect)),
                                 reinterpret_cast<const void*>(prop_df_kernel(t, cost, kResident)),
                                 reinterpret_cast<const void*>(prop_df_kernel(t, cost, kListed))};
            for (int v = 0; v < 5; v++) {
                cudaError_t e = cudaFuncSetAttribute(ks[v], cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                     (int)(v == 4 ? kMaxTileSmem : kMaxPropSmem));
                if (e != cudaSuccess) return e;
            }
        }
        for (int t : {256, 512}) {
            PropClusterKernel k = prop_cl_kernel(t, cost);
            cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxPropSmem);
            if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
            if (e != cudaSuccess) return e;
        }
    }
    return cudaSuccess;
}

bool prop_threads_ok(int threads) { return threads == 128 || threads == 256 || threads == 512; }

int prop_blocks_per_sm(int tw, int th, int n_iter, int threads, int cost, bool dataflow, bool listed) {
    const Variant v = listed ? kListed : prop_resident(tw, th, n_iter, threads) ? kResident : kDirect;
    const void* k = dataflow ? reinterpret_cast<const void*>(prop_df_kernel(threads, cost, v))
                             : reinterpret_cast<const void*>(prop_kernel(threads, cost, v == kResident));
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, threads, prop_launch_smem(tw, th, n_iter, listed)) !=
        cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    return n > 0 ? n : 1;
}

int prop_cluster_capacity(int cluster, int threads, int cost, size_t smem) {
    if (cluster < 1 || cluster > kMaxCluster || (threads != 256 && threads != 512) || smem > kMaxPropSmem) return 0;
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = cluster_config(cluster, cluster, threads, smem, nullptr, attr);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, prop_cl_kernel(threads, cost), &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

void launch_propagate(const PropProblem* probs_dev, const int2* queue_dev, int n_tiles, int* counter_dev, int grid,
                      const PropLaunch& L, cudaStream_t st) {
    if (L.cluster > 0) {
        cudaLaunchAttribute attr[2];
        cudaLaunchConfig_t cfg = cluster_config(grid, L.cluster, L.threads, (size_t)L.cl_smem, st, attr);
        cudaLaunchKernelEx(&cfg, prop_cl_kernel(L.threads, L.cost), probs_dev, L);
        return;
    }
    const size_t smem = prop_launch_smem(L.tw, L.th, L.max_iter, L.listed != 0);
    const bool resident = prop_resident(L.tw, L.th, L.dataflow > 0 ? 1 : L.max_iter, L.threads);
    const Variant v = L.listed ? kListed : resident ? kResident : kDirect;
    if (L.dataflow > 0)
        launch_k(prop_df_kernel(L.threads, L.cost, v), dim3(grid), dim3(L.threads), smem, st, probs_dev, queue_dev, n_tiles,
                 counter_dev, L, tile_layout(L.tw, L.th));
    else
        launch_k(prop_kernel(L.threads, L.cost, resident), dim3(grid), dim3(L.threads), smem, st, probs_dev, queue_dev,
                 n_tiles, counter_dev, L);
}

}  // namespace ff
