// Pruned exact nearest-neighbour search (Eq. 1, Eq. 2): the points of both clouds of a frame
// are put in the order of a space-filling curve, every 8 consecutive points get a bounding box,
// and a query only evaluates the boxes that its best distance so far does not exclude.
//
// Exactness. The reported distance is the float32 direct form d = fma(dz, dz, fma(dy, dy,
// dx dx)), dx = fl(a - b), and ties go to the lowest index, as in the other engines. The lower
// bound of a box is the same expression on e = max(fl(lo - a), fl(a - hi), 0) per coordinate.
// Rounding is monotone, so for every b in [lo, hi] e <= |fl(a - b)|, and the bound is at most
// the float32 distance of every point of the box; a box is left out only if its bound is above
// the query's current minimum, so no point that attains the minimum (or ties with it) is missed,
// whatever the input. The same holds for a box of queries against a box of points.
//
// k_tree_prep: one cluster of CTAs per (frame, side) samples the sim points (or reads the given
// ones), computes curve keys, sorts by them and writes points and boxes. k_tree_search: one warp
// per 32 consecutive queries of the sorted order.
#include <cooperative_groups.h>

#include <cfloat>

#include <algorithm>

#include "dc_sampling.cuh"

namespace cg = cooperative_groups;

namespace dc {

namespace {

constexpr int PREP_THREADS = 512;
constexpr int PREP_WARPS = PREP_THREADS / 32;
constexpr int KEY_AXIS_BITS = 8;                    // curve cells per axis: 256
constexpr int KEY_BITS = 3 * KEY_AXIS_BITS;
// counting-sort cells: 2^10 to 2^15, their 16-bit counters packed in pairs (or, for more than
// 65 535 points, 2^14 cells with 32-bit counters), in 64 KB of shared memory at most
constexpr int CELL_BITS_MIN = 10, CELL_BITS_PACKED = 15, CELL_BITS_WIDE = 14;
constexpr int CELL_BYTES = 64 * 1024;
// a counting-sort cell of more points than this keeps them in arrival order (ranks are unique
// within 256 consecutive positions, and the ranking window reaches that far to both sides)
constexpr int REFINE_MAX = 256;
constexpr int REFINE_RING = 4 * PREP_THREADS;       // entries of the ranking window's ring
constexpr int REFINE_BYTES = REFINE_RING * 4;
constexpr float PAD_COORD = 1e18f;                  // padding point of the last block of 8

// ---------------------------------------------------------------------------------------
// curve keys
// ---------------------------------------------------------------------------------------
// Hilbert index as a state machine over octants (C. Hamilton, A. Rau-Chaplin, "Compact Hilbert
// indices", 2008): a state is the entry corner e and direction d of a cell; octant b of it has
// the digit w, and its own state follows. Two levels per table look-up: entry
// [state << 6 | octant << 3 | octant] = next state << 6 | digit << 3 | digit. Along the Hilbert
// curve runs of points are compact: in Morton order, whose runs jump, a query tile evaluates 20
// to 45% more boxes.
struct alignas(16) HilbertTable {
    unsigned short v[24 * 64];
    static constexpr unsigned rotr(unsigned x, int k) { return ((x >> (k % 3)) | (x << (3 - k % 3))) & 7u; }
    static constexpr unsigned rotl(unsigned x, int k) { return ((x << (k % 3)) | (x >> (3 - k % 3))) & 7u; }
    static constexpr int trailing_ones(unsigned x) {
        int c = 0;
        while (x & 1u) {
            ++c;
            x >>= 1;
        }
        return c;
    }
    static constexpr void step(unsigned& e, int& d, unsigned b, unsigned& w) {
        const unsigned g = rotr(b ^ e, d + 1);
        w = g ^ (g >> 1) ^ (g >> 2);  // inverse Gray code
        const unsigned i = w == 0 ? 0 : 2 * ((w - 1) / 2);
        e ^= rotl(i ^ (i >> 1), d + 1);
        const int dw = w == 0 ? 0 : trailing_ones(w % 2 == 0 ? w - 1 : w) % 3;
        d = (d + dw + 1) % 3;
    }
    constexpr HilbertTable() : v() {
        for (int st = 0; st < 24; ++st)
            for (unsigned o = 0; o < 64; ++o) {
                unsigned e = st / 3, w1 = 0, w2 = 0;
                int d = st % 3;
                step(e, d, o >> 3, w1);
                step(e, d, o & 7u, w2);
                v[st * 64 + o] = (unsigned short)(((e * 3 + d) << 6) | (w1 << 3) | w2);
            }
    }
};
__device__ const HilbertTable c_hilbert{};

__device__ __forceinline__ unsigned spread3(unsigned x) {  // bit j of 8 to bit 3 j
    x = (x | (x << 8)) & 0x00F00Fu;
    x = (x | (x << 4)) & 0x0C30C3u;
    return (x | (x << 2)) & 0x249249u;
}

__device__ __forceinline__ unsigned hilbert_key(const unsigned short* t, unsigned x, unsigned y,
                                                unsigned z) {
    static_assert(KEY_AXIS_BITS == 8, "spread3 and the octants below take 8 bits per axis");
    const unsigned m = spread3(x) | (spread3(y) << 1) | (spread3(z) << 2);
    unsigned st = 0, k = 0;
#pragma unroll
    for (int j = KEY_BITS - 6; j >= 0; j -= 6) {
        const unsigned v = t[st | ((m >> j) & 63u)];
        st = v & ~63u;
        k = (k << 6) | (v & 63u);
    }
    return k;
}

// lower corner and cells per unit length of a frame's key grid (cubic cells)
struct KeyBox {
    float x, y, z, inv;
};

// cell of a point: x | y << 8 | z << 16
__device__ __forceinline__ unsigned grid_cell(const KeyBox& b, float x, float y, float z) {
    constexpr float TOP = (float)((1 << KEY_AXIS_BITS) - 1);
    // points outside the grid (and NaN) take the nearest cell: keys only order the points
    const unsigned ix = (unsigned)fminf(fmaxf((x - b.x) * b.inv, 0.0f), TOP);
    const unsigned iy = (unsigned)fminf(fmaxf((y - b.y) * b.inv, 0.0f), TOP);
    const unsigned iz = (unsigned)fminf(fmaxf((z - b.z) * b.inv, 0.0f), TOP);
    return ix | iy << KEY_AXIS_BITS | iz << (2 * KEY_AXIS_BITS);
}

__device__ __forceinline__ unsigned point_key(const unsigned short* t, const KeyBox& b, float x, float y,
                                              float z) {
    constexpr unsigned MASK = (1u << KEY_AXIS_BITS) - 1;
    const unsigned c = grid_cell(b, x, y, z);
    return hilbert_key(t, c & MASK, (c >> KEY_AXIS_BITS) & MASK, c >> (2 * KEY_AXIS_BITS));
}

__device__ __forceinline__ float max3(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// The key grid of a frame, from 128 points of each side: per axis, the medians of the lows and
// of the highs of 32 groups of 8 points, widened by 15% of their distance (the median low of 8
// uniform values is at 8% of their range). A few far outliers, which would squeeze the cloud
// into a few cells of their box, do not move the medians. Both sides of a frame compute the same
// grid from the same points, so that a query's key finds a block near it on the other side. Where
// the sides are unlike (apart, or of very different sizes: their own medians differ by over eight
// times the extent of the common box, which is then near that of their intersection), that grid may
// put a whole side into a few cells, unsorted, and nothing could be pruned there: a side whose sample
// lies in clearly fewer of its coarse cells than of those of the grid of its own medians takes the
// latter (and its starting bounds are loose then: from the extent itself on, one side of half the
// other's size took 204 instead of 146 us). 8 frames of 10 000 points a side, 10 extents apart:
// 1390 -> 190 us; one side 1000 times smaller: 880 -> 200 us. Called by the whole block; box_sample
// reads the points, so that other work can be put between their loads and key_box; s_p is scratch.
constexpr int BOX_THREADS = 256;
static_assert(PREP_WARPS >= 12, "a warp per median");
struct BoxSample {
    float p[3];
};
__device__ __forceinline__ BoxSample box_sample(const float* __restrict__ P, int np,
                                                const float* __restrict__ Y, int ny) {
    BoxSample b{{0.f, 0.f, 0.f}};
    constexpr int HALF = BOX_THREADS / 2;
    if (threadIdx.x < BOX_THREADS) {
        const bool first = threadIdx.x < HALF;
        const int n = first ? np : ny, t = first ? threadIdx.x : threadIdx.x - HALF;
        const float* q = (first ? P : Y) + 3LL * (int)((long long)t * n / HALF);
        b.p[0] = q[0], b.p[1] = q[1], b.p[2] = q[2];
    }
    return b;
}
// the grid over the box of lows med[0..2] and negated highs med[3..5]
__device__ __forceinline__ KeyBox grid_of(const float* med) {
    float lo[3], ext = 0.0f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float a = med[k], h = -med[3 + k];
        const float d = fmaxf(h - a, 0.0f);
        lo[k] = fabsf(a) <= COORD_MAX ? a - 0.15f * d : 0.0f;
        ext = fmaxf(ext, 1.3f * d);
    }
    KeyBox r{lo[0], lo[1], lo[2], 0.0f};
    r.inv = ext > 1e-30f && ext < 1e30f ? (float)(1 << KEY_AXIS_BITS) / ext : 0.0f;
    return r;
}

// The grid of a side unlike the other (see key_box). Called by the whole block; out of line, so that
// the preparation keeps its registers.
__device__ __noinline__ KeyBox unlike_grid(BoxSample b, int side, KeyBox both, KeyBox own,
                                                unsigned* s_cell) {
    // points of the side's sample in the coarse cell (of 8 per axis) of one before them, in either
    // grid: at random in space about 15 of 128, on a surface 70, on a line 120
    constexpr unsigned COARSE = 0xE0E0E0u;
    constexpr int CLEARLY = 32;
    static_assert(KEY_AXIS_BITS == 8, "top three bits of each axis");
    constexpr int HALF = BOX_THREADS / 2;
    const int t = (int)threadIdx.x - side * HALF;
    const bool mine = t >= 0 && t < HALF;
    if (mine) {
        s_cell[t] = grid_cell(both, b.p[0], b.p[1], b.p[2]) & COARSE;
        s_cell[HALF + t] = grid_cell(own, b.p[0], b.p[1], b.p[2]) & COARSE;
    }
    __syncthreads();
    bool met[2] = {false, false};
    if (mine)
        for (int j = 0; j < t; ++j) {
            met[0] |= s_cell[j] == s_cell[t];
            met[1] |= s_cell[HALF + j] == s_cell[HALF + t];
        }
    const int in_both = __syncthreads_count(met[0]), in_own = __syncthreads_count(met[1]);
    return in_own + CLEARLY <= in_both ? own : both;
}

__device__ KeyBox key_box(const BoxSample& b, int side, float (*s_p)[BOX_THREADS]) {
    __shared__ float s_low[6][32];  // lows, then negated highs, of every group
    __shared__ float s_med[3][6];   // medians: of both sides' groups, of each side's
    __shared__ float s_off[6];      // how far the sides' differ
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid < BOX_THREADS) {
        float v[6];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const bool ok = coord_ok(b.p[k]);
            s_p[k][tid] = b.p[k];
            v[k] = ok ? b.p[k] : INFINITY;
            v[3 + k] = ok ? -b.p[k] : INFINITY;
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1)
#pragma unroll
            for (int k = 0; k < 6; ++k) v[k] = fminf(v[k], __shfl_xor_sync(0xffffffffu, v[k], o));
        if ((lane & 7) == 0)
#pragma unroll
            for (int k = 0; k < 6; ++k) s_low[k][tid >> 3] = v[k];
    }
    __syncthreads();
    if (warp < 6) {  // the median: the value of rank 16 (ties by lane)
        const float v = s_low[warp][lane];
        int rank = 0;
#pragma unroll
        for (int j = 0; j < 32; ++j) {
            const float u = __shfl_sync(0xffffffffu, v, j);
            rank += u < v || (u == v && j < lane) ? 1 : 0;
        }
        if (rank == 16) s_med[0][warp] = v;
    } else if (warp < 12) {
        // of a side's 16 groups: rank 8. Here a group is every 16th point of the sample, so that it
        // spans the cloud also where neighbours follow each other (the rows of a mesh).
        const int k = warp - 6 < 3 ? warp - 6 : warp - 9;
        const float sign = warp - 6 < 3 ? 1.0f : -1.0f;
        float v = INFINITY;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float p = s_p[k][(lane >> 4) * (BOX_THREADS / 2) + 16 * j + (lane & 15)];
            if (coord_ok(p)) v = fminf(v, sign * p);
        }
        int rank = 0;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const float u = __shfl_sync(0xffffffffu, v, (lane & 16) + j);
            rank += u < v || (u == v && j < (lane & 15)) ? 1 : 0;
        }
        const unsigned who = __ballot_sync(0xffffffffu, rank == 8);  // a lane of each half
        const float a = __shfl_sync(0xffffffffu, v, __ffs(who) - 1);
        const float c = __shfl_sync(0xffffffffu, v, 31 - __clz(who));
        if (lane == 0) {
            s_med[1][warp - 6] = a;
            s_med[2][warp - 6] = c;
            s_off[warp - 6] = fabsf(a - c);
        }
    }
    __syncthreads();
    const KeyBox both = grid_of(s_med[0]);
    // inv: cells per 1.3 times the extent; an infinite or undefined difference is above any limit
    const float off = fmaxf(max3(s_off[0], s_off[1], s_off[2]), max3(s_off[3], s_off[4], s_off[5]));
    constexpr float LIMIT = 8.0f * (float)(1 << KEY_AXIS_BITS) / 1.3f;
    if (both.inv > 0.0f && off * both.inv <= LIMIT) return both;
    return unlike_grid(b, side, both, grid_of(s_med[1 + side]), reinterpret_cast<unsigned*>(s_p));
}

// ---------------------------------------------------------------------------------------
// preparation
// ---------------------------------------------------------------------------------------
// Inclusive prefix sums of the face areas in cdf[F] (shared or global), bit for bit those of
// the area kernels: 1024 segments of ceil(F / 1024) faces, two per thread, summed with two-float
// compensation and scanned in the same order. Called by the whole block.
__device__ void tree_scan_cdf(float* cdf, int F, int* err) {
    __shared__ FF s_w[32];
    static_assert(CDF_THREADS == 1024 && PREP_THREADS == 512, "two segments per thread");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int per = (F + CDF_THREADS - 1) / CDF_THREADS;
    FF v[2] = {{0.0f, 0.0f}, {0.0f, 0.0f}};
    const int fa = min(F, tid * per), fb = min(F, (tid + PREP_THREADS) * per);
    for (int j = 0; j < per; ++j) {
        if (fa + j < F) v[0] = ff_add1(v[0], cdf[fa + j]);
        if (fb + j < F) v[1] = ff_add1(v[1], cdf[fb + j]);
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        FF u[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            u[h].hi = __shfl_up_sync(0xffffffffu, v[h].hi, o);
            u[h].lo = __shfl_up_sync(0xffffffffu, v[h].lo, o);
            if (lane >= o) v[h] = ff_add(u[h], v[h]);
        }
    }
    if (lane == 31) {
        s_w[warp] = v[0];
        s_w[warp + PREP_WARPS] = v[1];
    }
    __syncthreads();
    if (warp == 0) {
        FF t = s_w[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            FF u = {__shfl_up_sync(0xffffffffu, t.hi, o), __shfl_up_sync(0xffffffffu, t.lo, o)};
            if (lane >= o) t = ff_add(u, t);
        }
        s_w[lane] = t;
    }
    __syncthreads();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int f0 = min(F, (tid + h * PREP_THREADS) * per), f1 = min(F, f0 + per);
        FF ex = {__shfl_up_sync(0xffffffffu, v[h].hi, 1), __shfl_up_sync(0xffffffffu, v[h].lo, 1)};
        if (lane == 0) ex = {0.0f, 0.0f};
        const int sw = warp + h * PREP_WARPS;
        FF run = sw > 0 ? ff_add(s_w[sw - 1], ex) : ex;
        for (int f = f0; f < f1; ++f) {
            run = ff_add1(run, cdf[f]);
            cdf[f] = run.hi;
        }
        if (f1 == F && f0 < f1) {
            const float A = run.hi;
            if (!(A > 0.0f) || !isfinite(A)) set_status(err, DC_EDEGENERATE);
        }
    }
    __syncthreads();
}

// Area weights of two faces and their corners q[9] (zeros, and weight 0, for a face with an index
// out of range; bad is set for it and for coordinates out of range); the loads of both overlap.
__device__ __forceinline__ void face_record2(const float* __restrict__ verts,
                                             const int* __restrict__ faces,
                                             const uint8_t* __restrict__ mask, int V,
                                             const int (&f)[2], float (&q)[2][9], float (&A)[2],
                                             bool& bad) {
    int v[2][3];
    bool in[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
#pragma unroll
        for (int c = 0; c < 3; ++c) v[h][c] = __ldg(faces + 3 * f[h] + c);
        in[h] = (unsigned)v[h][0] < (unsigned)V && (unsigned)v[h][1] < (unsigned)V &&
                (unsigned)v[h][2] < (unsigned)V;
        bad |= !in[h];
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int k = 0; k < 3; ++k)
                q[h][3 * c + k] = in[h] ? __ldg(verts + 3LL * v[h][c] + k) : 0.0f;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        A[h] = corner_area(q[h], bad);
        if (mask && mask[f[h]] == 0) A[h] = 0.0f;
    }
}

// Counting-sort cells of n points: 2^bits of them
__device__ __forceinline__ int cell_bits(int n, int most) {
    int b = CELL_BITS_MIN;
    while (b < most && (1 << b) < n) ++b;
    return b;
}

// counter of cell c: 16 bits of word c / 2 (packed), or word c
__device__ __forceinline__ int cell_add(int* h, bool packed, int c) {
    if (!packed) return atomicAdd(h + c, 1);
    const int sh = 16 * (c & 1);
    return (int)(((unsigned)atomicAdd(h + (c >> 1), 1 << sh) >> sh) & 0xffffu);
}
__device__ __forceinline__ int cell_get(const int* h, bool packed, int c) {
    if (!packed) return h[c];
    return (int)(((unsigned)h[c >> 1] >> (16 * (c & 1))) & 0xffffu);
}

// Prepares every (frame, side): one cluster of S CTAs each, CTA r takes the r-th slice of the
// side's points. Unit u is side u / n_frames of frame u % n_frames.
//   1. sim side: face areas and corner records (each CTA a share; the areas go into every CTA's
//      shared memory), their scan, and the slice's points from their draws; target side: the
//      points as given
//   2. curve keys; histogram of their top bits (cells) in shared memory
//   3. scan over cells and slices (through distributed shared memory), scatter of the points'
//      keys and indices
//   4. each point's rank within its cell by its whole key; the sorted points as blocks of 8
//      (x[8] y[8] z[8] index[8], one 128-byte line)
//   5. bounding boxes of 8, 64 and 512 consecutive points
// Bound by latency: chains of dependent gathers (face pick, corners) and one block-wide meeting
// per phase. 40 frames of 10 000 points against as many: 62 us at 37% of the load pipe, its warps
// waiting 4.7 cycles per instruction for memory and 3.6 at barriers. One kernel for all phases
// keeps the counters and the draws' points on chip; clusters of 3 instead of 2 for those 80 sides
// (240 CTAs instead of 160) 210 -> 198 us per call. 64 uneven trajectories, 1.14e8 points:
// 6.1 ms with 1024 threads and gathers from global memory, 5.0 ms with face records and two
// points per step, 4.5 ms with the ring below, 4.6 ms with the boxes' lowest indices and the check of the
// key grid.
template <int S>
__global__ void __launch_bounds__(PREP_THREADS, 2)
    k_tree_prep(UniformArgs a, Ws w, int uniform, int n_frames, int rows, int cdf_shared) {
    __shared__ __align__(16) unsigned short s_tab[24 * 64];
    constexpr int TAB_WORDS = (24 * 32 + PREP_THREADS - 1) / PREP_THREADS;
    static_assert(sizeof(s_tab) >= 3 * BOX_THREADS * sizeof(float), "key_box's scratch");
    unsigned tab[TAB_WORDS];
#pragma unroll
    for (int h = 0; h < TAB_WORDS; ++h)
        tab[h] = threadIdx.x + h * PREP_THREADS < 24 * 32
                     ? reinterpret_cast<const unsigned*>(c_hilbert.v)[threadIdx.x + h * PREP_THREADS]
                     : 0u;
    pdl_wait();
    cg::cluster_group cl = cg::this_cluster();
    auto meet = [&]() {
        if (S > 1)
            cl.sync();
        else
            __syncthreads();
    };
    auto remote = [&](auto* p, int q) {
        if (S > 1)
            return cl.map_shared_rank(p, q);
        else
            return p;
    };
    const int r = S > 1 ? (int)cl.block_rank() : 0;
    extern __shared__ __align__(16) int s_dyn[];
    __shared__ int s_err;
    __shared__ int s_wtot[32];
    __shared__ int s_total;
    __shared__ FrameDesc s_fr;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int unit = blockIdx.x / S;
    const int side = unit >= n_frames ? 1 : 0, k = side ? unit - n_frames : unit;

    if (tid == 0) {
        s_err = DC_OK;
        s_fr = uniform ? uniform_frame(a, w, k) : w.frames[k];
        if (side == 0 && r == 0) {
            if (uniform) w.frames[k] = s_fr;
            if (k == 0) {
                WsHeader* h = w.hdr;
                h->status = DC_OK;
                if (uniform) {
                    h->n_frames = a.T;
                    h->n_units = 0;
                    h->total_sub = 0;
                    h->total_rows = a.T * s_fr.Npad;
                    h->total_cols = a.T * s_fr.Mpad;
                    h->sum_f = a.T * a.F;
                    h->mode = a.mode;
                    h->planned = 0;
                    h->any_grad = a.grad != nullptr;
                    h->max_v = a.V;
                    h->slices = a.slices;
                    h->warps = a.warps;
                    h->engine = a.engine;
                    h->tc_units = 0;
                    h->tc_total = 0;
                }
                h->tc_fallback = 0;
                h->tc_next = 0;
                h->tree_n = 0;
                h->tree_wide = 0;
            }
        }
    }
    __syncthreads();
    const FrameDesc& fr = s_fr;
    const int n = side ? fr.M : fr.N;
    const int npad = side ? fr.Mpad : fr.Npad;
    const int base = side ? fr.col0 : fr.row0;  // offset in the side's padded rows
    const long long gbase = side ? (long long)rows + base : base;
    // the steps of the search (TREE_STEP queries each) find their frame here
    for (int s = r * PREP_THREADS + tid; s < npad / TREE_STEP; s += S * PREP_THREADS)
        w.step_frame[gbase / TREE_STEP + s] = k;
    const bool grad = side == 0 && fr.grad && fr.verts;  // its accumulators start from zero
    if (grad)
        for (int v = r * PREP_THREADS + tid; v < fr.V; v += S * PREP_THREADS)
            w.grad4[fr.v0 + v] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (fr.skip) {  // the same for the whole cluster
        if (tid == 0 && r == 0) w.tree_err[2 * k + side] = DC_OK;
        pdl_trigger();
        return;
    }

    const bool packed = n <= 65535;
    const int cb = cell_bits(n, packed ? CELL_BITS_PACKED : CELL_BITS_WIDE);
    const int words = packed ? 1 << (cb - 1) : 1 << cb, low = KEY_BITS - cb;
    // the shared memory holds the CDF until the points are sampled, then the cells' counters and
    // the refinement's buffers
    int* const hist = s_dyn;
    float* const cdf = cdf_shared ? reinterpret_cast<float*>(s_dyn) : w.cdf + fr.cdf0;
    const BoxSample sample =
        box_sample(fr.pts ? fr.pts : fr.verts, fr.pts ? fr.N : fr.V, fr.tgt, fr.M);
    const bool sampled = side == 0 && !fr.pts;
    float4* const rec = w.frec + 3LL * fr.cdf0;  // the frame's face records
    bool bad = false;
    if (sampled) {
        if (S > 1) cl.sync();  // every CTA of the cluster runs: its shared memory may be written
        const int fa = (int)((long long)fr.F * r / S), fb = (int)((long long)fr.F * (r + 1) / S);
        for (int fs = fa + tid; fs < fb; fs += 2 * PREP_THREADS) {
            const int ff[2] = {fs, min(fs + PREP_THREADS, fb - 1)};  // the last may be done twice
            float q[2][9], A[2];
            face_record2(fr.verts, fr.faces, fr.mask, fr.V, ff, q, A, bad);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int f = ff[h];
                rec[3 * f] = make_float4(q[h][0], q[h][1], q[h][2], q[h][3]);
                rec[3 * f + 1] = make_float4(q[h][4], q[h][5], q[h][6], q[h][7]);
                rec[3 * f + 2] = make_float4(q[h][8], 0.f, 0.f, 0.f);
                if (cdf_shared) {
#pragma unroll
                    for (int c = 0; c < S; ++c) remote(cdf, c)[f] = A[h];
                } else {
                    cdf[f] = A[h];
                }
            }
        }
        if (bad) set_status(&s_err, DC_EINVAL);
    }
    // the Hilbert table's memory is key_box's scratch first: 3 KB more would cost two CTAs on meshes of
    // 19 600 faces (78 KB of areas each) the step from 92 to 60 KB of L1, 430 -> 490 us for 100 frames
    // (key_box has met since it last read the scratch)
    const KeyBox box = key_box(sample, side, reinterpret_cast<float(*)[BOX_THREADS]>(s_tab));
#pragma unroll
    for (int h = 0; h < TAB_WORDS; ++h)
        if (tid + h * PREP_THREADS < 24 * 32)
            reinterpret_cast<unsigned*>(s_tab)[tid + h * PREP_THREADS] = tab[h];
    if (!sampled) __syncthreads();  // (the areas' meeting follows otherwise)
    if (sampled) {
        meet();  // all areas are in place
        // a CDF too large for shared memory lives in the frame's global slot, scanned by CTA 0
        if (cdf_shared || r == 0) tree_scan_cdf(cdf, fr.F, &s_err);
        if (!cdf_shared) meet();
    }

    // ---- points and keys: two points per thread and step, so that their chains of dependent
    // loads overlap ----
    const int i0 = (int)((long long)n * r / S), i1 = (int)((long long)n * (r + 1) / S);
    float4* const xs = side ? w.y + base : w.x + base;
    bad = false;
    for (int ib = i0 + tid; ib < i1; ib += 2 * PREP_THREADS) {
        const int ii[2] = {ib, min(ib + PREP_THREADS, i1 - 1)};  // the last may be done twice
        float v[2][3];
        const float* src = sampled ? fr.draws : (side ? fr.tgt : fr.pts);
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int c = 0; c < 3; ++c) v[h][c] = src[3LL * ii[h] + c];
        float4 x[2];
        int4 q[2];
        if (sampled) {
            int f[2];
            pick_face2(cdf, fr.F, v[0][0], v[1][0], f[0], f[1]);
            float4 ra[2], rb[2];
            float rc[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                ra[h] = rec[3 * f[h]];
                rb[h] = rec[3 * f[h] + 1];
                rc[h] = rec[3 * f[h] + 2].x;
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
#pragma unroll
                for (int c = 0; c < 3; ++c) bad |= !(v[h][c] >= 0.0f && v[h][c] <= 1.0f);
                float w0, w1, w2;
                bary_weights(v[h][1], v[h][2], w0, w1, w2);
                x[h] = make_float4(bary_point(w0, w1, w2, ra[h].x, ra[h].w, rb[h].z),
                                   bary_point(w0, w1, w2, ra[h].y, rb[h].x, rb[h].w),
                                   bary_point(w0, w1, w2, ra[h].z, rb[h].y, rc[h]), 0.0f);
                q[h] = make_int4(f[h], __float_as_int(w0), __float_as_int(w1), __float_as_int(w2));
            }
        } else {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
#pragma unroll
                for (int c = 0; c < 3; ++c) bad |= !coord_ok(v[h][c]);
                x[h] = make_float4(v[h][0], v[h][1], v[h][2], 0.0f);
                q[h] = make_int4(-1, 0, 0, 0);
            }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            xs[ii[h]] = x[h];
            if (!side) w.fw[base + ii[h]] = q[h];
            if (grad) w.tgx[base + ii[h]] = make_float4(0.f, 0.f, 0.f, 0.f);
            w.tkey[gbase + ii[h]] = point_key(s_tab, box, x[h].x, x[h].y, x[h].z);
        }
    }
    if (bad) set_status(&s_err, DC_EINVAL);

    // ---- histogram of the cells ----
    __syncthreads();  // the CDF is not needed any more
    for (int c = tid; c < words; c += PREP_THREADS) hist[c] = 0;
    __syncthreads();
    constexpr int U = 4;  // keys in flight per thread
    for (int ib = i0 + tid; ib < i1; ib += U * PREP_THREADS) {
        unsigned key[U];
#pragma unroll
        for (int h = 0; h < U; ++h) {
            const int i = ib + h * PREP_THREADS;
            key[h] = i < i1 ? w.tkey[gbase + i] : 0u;
        }
#pragma unroll
        for (int h = 0; h < U; ++h)
            if (ib + h * PREP_THREADS < i1) (void)cell_add(hist, packed, (int)(key[h] >> low));
    }
    meet();  // every slice's histogram is complete
    // the first error of the side ends up in CTA 0's word
    if (S > 1 && tid == 0 && r > 0 && s_err != DC_OK) atomicCAS(remote(&s_err, 0), DC_OK, s_err);

    // ---- starts of every (cell, slice): CTA r scans its share of the words over all slices ----
    {
        const int first = words / 32 * r / S, end = words / 32 * (r + 1) / S;  // chunks of 32
        const int cw = (end - first + PREP_WARPS - 1) / PREP_WARPS;
        const int ch0 = min(end, first + warp * cw), ch1 = min(end, ch0 + cw);
        auto word_sum = [&](int v) { return packed ? (v & 0xffff) + (int)((unsigned)v >> 16) : v; };
        int tot = 0;
        for (int ch = ch0; ch < ch1; ++ch) {
            const int c = 32 * ch + lane;
#pragma unroll
            for (int s = 0; s < S; ++s) tot += word_sum(remote(hist, s)[c]);
        }
        tot = __reduce_add_sync(0xffffffffu, tot);
        if (lane == 0) s_wtot[warp] = tot;
        __syncthreads();
        if (warp == 0) {
            int v = lane < PREP_WARPS ? s_wtot[lane] : 0;
            const int self = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v += u;
            }
            s_wtot[lane] = v - self;
            if (lane == 31) s_total = v;
        }
        meet();
        int run = s_wtot[warp];
#pragma unroll
        for (int s = 0; s < S; ++s)
            if (s < r) run += *remote(&s_total, s);
        for (int ch = ch0; ch < ch1; ++ch) {
            const int c = 32 * ch + lane;
            int cnt[S], sum = 0;
#pragma unroll
            for (int s = 0; s < S; ++s) {
                cnt[s] = remote(hist, s)[c];
                sum += word_sum(cnt[s]);
            }
            int v = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v += u;
            }
            int start = run + v - sum;
            run += __shfl_sync(0xffffffffu, v, 31);
            if (packed) {  // the even cell's slices, then the odd cell's
                int even[S];
#pragma unroll
                for (int s = 0; s < S; ++s) {
                    even[s] = start;
                    start += cnt[s] & 0xffff;
                }
#pragma unroll
                for (int s = 0; s < S; ++s) {
                    remote(hist, s)[c] = even[s] | (start << 16);
                    start += (int)((unsigned)cnt[s] >> 16);
                }
            } else {
#pragma unroll
                for (int s = 0; s < S; ++s) {
                    remote(hist, s)[c] = start;
                    start += cnt[s];
                }
            }
        }
    }
    meet();

    // ---- index << 32 | key << 8, in cell order, in one store (stores to 32 lines take the load
    // pipe 32 cycles whatever their width) ----
    u64* const ord = w.tord + gbase;
    for (int ib = i0 + tid; ib < i1; ib += U * PREP_THREADS) {
        unsigned key[U];
#pragma unroll
        for (int h = 0; h < U; ++h) {
            const int i = ib + h * PREP_THREADS;
            key[h] = i < i1 ? w.tkey[gbase + i] : 0u;
        }
#pragma unroll
        for (int h = 0; h < U; ++h) {
            const int i = ib + h * PREP_THREADS;
            if (i < i1) {
                const int pos = cell_add(hist, packed, (int)(key[h] >> low));
                ord[pos] = ((u64)(unsigned)i << 32) | (key[h] << 8);
            }
        }
    }
    meet();

    // ---- rank within the cell, and the sorted points. The counters now hold the cells' ends, the
    // last slice's the ends over all slices. CTA r takes the r-th slice of the positions, one
    // chunk of PREP_THREADS at a time; the keys of the chunks before and after stay in a ring in
    // shared memory, so that a thread ranks its point among its cell's without waiting for
    // memory, and the next chunk is in flight meanwhile. ----
    {
        const int p0 = (int)((long long)n * r / S), p1 = (int)((long long)n * (r + 1) / S);
        if (S > 1 && r != S - 1 && p0 < p1) {
            // the ends of the cells that the slice meets
            const int* last = remote(hist, S - 1);
            const int ca = (int)((unsigned)ord[p0] >> (8 + low)) - 1;
            const int cz = (int)((unsigned)ord[p1 - 1] >> (8 + low));
            const int sh = packed ? 1 : 0;
            for (int c = (max(ca, 0) >> sh) + tid; c <= cz >> sh; c += PREP_THREADS)
                hist[c] = last[c];
        }
        unsigned* const ring = reinterpret_cast<unsigned*>(s_dyn) + CELL_BYTES / 4;
        float* pts = w.tpts + 4 * gbase;
        const int chunks = div_up(p1 - p0, PREP_THREADS);
        auto fetch = [&](int c) {
            const int p = p0 + c * PREP_THREADS + tid;
            return p >= 0 && p < n ? ord[p] : ~0ull;
        };
        // keys with the position's low bits: all different among 256 consecutive positions
        auto keep = [&](int c, u64 v) {
            const int p = p0 + c * PREP_THREADS + tid;
            ring[p & (REFINE_RING - 1)] = v == ~0ull ? ~0u : ((unsigned)v | (unsigned)(p & 255));
        };
        u64 cur = fetch(0), next = fetch(1), after = fetch(2);
        keep(-1, fetch(-1));
        keep(0, cur);
        keep(1, next);
        for (int ch = 0; ch < chunks; ++ch) {
            __syncthreads();  // chunks ch - 1, ch and ch + 1 are in the ring
            const int p = p0 + ch * PREP_THREADS + tid;
            const bool on = p < p1;
            const unsigned key = (unsigned)cur >> 8, o = (unsigned)cur | (unsigned)(p & 255);
            const int i = (int)(cur >> 32);
            keep(ch + 2, after);  // the slot of chunk ch - 2
            cur = next;
            next = after;
            after = fetch(ch + 3);
            if (!on) continue;
            const float4 v = xs[i];
            const float x = v.x, y = v.y, z = v.z;
            const int cell = (int)(key >> low);
            const int e = cell_get(hist, packed, cell);
            const int s = cell > 0 ? cell_get(hist, packed, cell - 1) : 0;
            int pos = p;
            if (e - s <= REFINE_MAX) {
                // from a multiple of 4 on: the entries before s are of lower cells, those from e
                // on of higher ones
                pos = s & ~3;
                for (int q = pos; q < e; q += 8) {
                    const uint4 k0 = *reinterpret_cast<const uint4*>(ring + (q & (REFINE_RING - 1)));
                    const uint4 k1 =
                        *reinterpret_cast<const uint4*>(ring + ((q + 4) & (REFINE_RING - 1)));
                    pos += (k0.x < o) + (k0.y < o) + (k0.z < o) + (k0.w < o) + (k1.x < o) +
                           (k1.y < o) + (k1.z < o) + (k1.w < o);
                }
            }
            float* b = pts + 32LL * (pos >> 3) + (pos & 7);
            b[0] = x;
            b[8] = y;
            b[16] = z;
            b[24] = __int_as_float(i);
            w.tkey[gbase + pos] = key;  // from here on in sorted order
            if ((pos & 7) == 0) w.tkb[gbase / 8 + (pos >> 3)] = key;
        }
        if (r == S - 1 && tid < 8 && (n & 7) != 0 && tid >= (n & 7)) {
            float* b = pts + 32LL * (n >> 3) + tid;  // padding points of the last block
            b[0] = b[8] = b[16] = PAD_COORD;
            b[24] = __int_as_float(0x7fffffff);
        }
    }
    meet();
    if (tid == 0 && r == 0) w.tree_err[2 * k + side] = s_err;

    // ---- boxes: a warp per 512 points, a lane per 8 of them, twice. The w lane of the lower
    // corner of a box of 64 or 512 holds the lowest index in it: a box at exactly a query's minimum
    // can only matter with a lower index than the one found. ----
    const int nb = (n + 7) / 8, nb2 = (n + 511) / 512;
    float4* box0 = w.tbox + 2 * (gbase / 8);
    float4* box1 = w.tbox1 + 2 * (gbase / 64);
    float4* box2 = w.tbox2 + 2 * (gbase / TREE_STEP);
    for (int b2 = r * PREP_WARPS + warp; b2 < nb2; b2 += S * PREP_WARPS) {
        float l2[3] = {INFINITY, INFINITY, INFINITY}, h2[3] = {-INFINITY, -INFINITY, -INFINITY};
        int first2 = 0x7fffffff;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int b = 64 * b2 + 32 * h + lane;
            float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
            int first = 0x7fffffff;
            if (b < nb) {
                const float4* q = reinterpret_cast<const float4*>(w.tpts + 4 * gbase) + 8LL * b;
                const int m = min(8, n - 8 * b);
                const int4 ia = *reinterpret_cast<const int4*>(q + 6);
                const int4 ib = *reinterpret_cast<const int4*>(q + 7);
                first = min(min(min(ia.x, ia.y), min(ia.z, ia.w)),
                            min(min(ib.x, ib.y), min(ib.z, ib.w)));
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const float4 u = q[2 * c], v = q[2 * c + 1];
                    const float t[8] = {u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (j < m) {
                            lo[c] = fminf(lo[c], t[j]);
                            hi[c] = fmaxf(hi[c], t[j]);
                        }
                }
            }
            if (b < (nb + 7) / 8 * 8) {  // empty boxes up to a whole box of 64
                box0[2 * b] = make_float4(lo[0], lo[1], lo[2], 0.f);
                box0[2 * b + 1] = make_float4(hi[0], hi[1], hi[2], 0.f);
            }
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) {
                first = min(first, __shfl_xor_sync(0xffffffffu, first, o));
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    lo[c] = fminf(lo[c], __shfl_xor_sync(0xffffffffu, lo[c], o));
                    hi[c] = fmaxf(hi[c], __shfl_xor_sync(0xffffffffu, hi[c], o));
                }
            }
            first2 = min(first2, first);
            if ((lane & 7) == 0 && b < nb) {
                box1[2 * (b >> 3)] = make_float4(lo[0], lo[1], lo[2], __int_as_float(first));
                box1[2 * (b >> 3) + 1] = make_float4(hi[0], hi[1], hi[2], 0.f);
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                l2[c] = fminf(l2[c], lo[c]);
                h2[c] = fmaxf(h2[c], hi[c]);
            }
        }
#pragma unroll
        for (int o = 16; o > 4; o >>= 1)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                l2[c] = fminf(l2[c], __shfl_xor_sync(0xffffffffu, l2[c], o));
                h2[c] = fmaxf(h2[c], __shfl_xor_sync(0xffffffffu, h2[c], o));
            }
        first2 = __reduce_min_sync(0xffffffffu, first2);
        if (lane == 0) {
            box2[2 * b2] = make_float4(l2[0], l2[1], l2[2], __int_as_float(first2));
            box2[2 * b2 + 1] = make_float4(h2[0], h2[1], h2[2], 0.f);
        }
    }
    pdl_trigger();
}

// ---------------------------------------------------------------------------------------
// search
// ---------------------------------------------------------------------------------------
// One query per thread. CTAs of one warp free their slots as soon as it is done, and the block-wide
// values are known to be the same in all lanes: 4.7% faster than two warps on 64 uneven trajectories
// (18.0 against 18.9 ms), four warps 5.1% slower.
constexpr int SEARCH_THREADS = 32;
constexpr int SEARCH_CTAS = 32;  // per SM: 64 registers (28 CTAs: 18.5 against 18.0 ms)
// A query whose starting bound is 2^5 times (as squared distance) that of the tile's others
constexpr int OUTLIER_LOG2 = 5;
// A tile whose box meets more boxes than this is searched query by query (or walked as a whole, see
// walk_tile): 512-point boxes per 32 of them, 64-point boxes in all.
constexpr int WIDE_BOX2 = 16;
constexpr int WIDE_BOX1 = 40;
// Tiles that are wide or have this many outliers are rare in ordinary clouds. Beyond one in
// FEW_WIDE of all tiles (and FEW_WIDE in all) each is looked at for walking as a whole.
constexpr int MANY_OUTLIERS = 8;
constexpr int FEW_WIDE = 16;
// Boxes of 64 points on their way to a warp: their eight boxes of 8 and their points are copied
// to shared memory while the ones before are searched.
constexpr int STAGES = 2;  // a power of two
struct TreeStage {
    float4 pts[64];  // eight blocks of x[8] y[8] z[8] index[8]
    float4 box[16];  // (lo, hi) of the eight blocks
};
struct TreeWarp {
    TreeStage stage[STAGES];
    int hit[WIDE_BOX1 + 32];  // the boxes of 64 that the tile meets
};

__device__ __forceinline__ void copy16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// the other side's points and boxes
struct TreeCols {
    const float4* pts;   // 8 float4 per block of 8 points: x, y, z, index
    const float4* box0;  // (lo, hi) of 8 points
    const float4* box1;  // of 64
    const float4* box2;  // of 512
    int nb, nb1, nb2;
};

// minimum and maximum over the warp
__device__ __forceinline__ float warp_min(float v) {
    float r;
    asm("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ float warp_max(float v) {
    float r;
    asm("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}

// lower bound of the float32 distances between the boxes [alo, ahi] and [lo, hi]
__device__ __forceinline__ float box_bound(float3 alo, float3 ahi, float4 lo, float4 hi) {
    const float ex = max3(__fsub_rn(lo.x, ahi.x), __fsub_rn(alo.x, hi.x), 0.0f);
    const float ey = max3(__fsub_rn(lo.y, ahi.y), __fsub_rn(alo.y, hi.y), 0.0f);
    const float ez = max3(__fsub_rn(lo.z, ahi.z), __fsub_rn(alo.z, hi.z), 0.0f);
    return __fmaf_rn(ez, ez, __fmaf_rn(ey, ey, __fmul_rn(ex, ex)));
}

__device__ __forceinline__ float2 lohalf(float4 v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hihalf(float4 v) { return make_float2(v.z, v.w); }

// squared distances of two points (negated query coordinates nx, ny, nz, each twice): the
// difference with the query rounds the same in either direction
__device__ __forceinline__ float2 dist2x2(float2 px, float2 py, float2 pz, float2 nx, float2 ny,
                                          float2 nz) {
    const float2 dx = __fadd2_rn(px, nx), dy = __fadd2_rn(py, ny), dz = __fadd2_rn(pz, nz);
    return __ffma2_rn(dz, dz, __ffma2_rn(dy, dy, __fmul2_rn(dx, dx)));
}

// this lane's query against the 8 points of block b (the same block for the whole warp, or one
// of its own per lane): the distances
__device__ __forceinline__ void block_dist(const float4* __restrict__ P, float2 nx, float2 ny,
                                           float2 nz, float2 (&d)[4]) {
    const float4 xa = __ldg(P), xb = __ldg(P + 1), ya = __ldg(P + 2), yb = __ldg(P + 3),
                 za = __ldg(P + 4), zb = __ldg(P + 5);
    d[0] = dist2x2(lohalf(xa), lohalf(ya), lohalf(za), nx, ny, nz);
    d[1] = dist2x2(hihalf(xa), hihalf(ya), hihalf(za), nx, ny, nz);
    d[2] = dist2x2(lohalf(xb), lohalf(yb), lohalf(zb), nx, ny, nz);
    d[3] = dist2x2(hihalf(xb), hihalf(yb), hihalf(zb), nx, ny, nz);
}

__device__ __forceinline__ float block_min(const float2 (&d)[4]) {
    return min3(min3(min3(fminf(d[0].x, d[0].y), d[1].x, d[1].y), d[2].x, d[2].y), d[3].x,
                d[3].y);
}

// the j-th set bit of m for the lanes' groups of eight (lane >> 3 = j), -1 beyond the last; up
// to four bits are taken off m
__device__ __forceinline__ int take4(unsigned& m, int group) {
    const int b0 = __ffs(m) - 1;
    m &= m - 1;
    const int b1 = __ffs(m) - 1;
    m &= m - 1;
    const int b2 = __ffs(m) - 1;
    m &= m - 1;
    const int b3 = __ffs(m) - 1;
    m &= m - 1;
    return group == 0 ? b0 : (group == 1 ? b1 : (group == 2 ? b2 : b3));
}

// the columns of side `side` of frame fr
__device__ __forceinline__ TreeCols tree_cols(const Ws& w, const FrameDesc* fr, int side, int rows) {
    const int nc = side ? fr->N : fr->M;
    const long long c = side ? fr->row0 : (long long)rows + fr->col0;
    TreeCols C;
    C.pts = reinterpret_cast<const float4*>(w.tpts) + c;
    C.box0 = w.tbox + 2 * (c / 8);
    C.box1 = w.tbox1 + 2 * (c / 64);
    C.box2 = w.tbox2 + 2 * (c / TREE_STEP);
    C.nb = (nc + 7) / 8;
    C.nb1 = (nc + 63) / 64;
    C.nb2 = (nc + 511) / 512;
    return C;
}

// A tile that meets most boxes, a lane per query (`own`: its bound). First better bounds: every
// query's distances to the points of the box of 64 nearest to it in the box of 512 nearest to it.
// If the queries then still need, each by itself, DENSE_SHARE of the boxes of 8 on average (up to
// 64 of them are tested; at exactly the bound lie ties, which do not count), as where all points are
// about equally far away or a cloud has too many scales to be sorted, nothing can be pruned, and the
// tile is walked to the end (done): every box is tested for all of it, a block that any query needs
// is evaluated by all, its points loaded once for the warp. Where all tiles are like that this is
// brute force, and a warp per query took up to seven times as long (8 frames of 10 000 points around
// a sphere's centre against as many on it: 4650 us, now 920). At 0.14 of the boxes (clouds side by
// side) a warp per query is still faster, 230 against 370 us.
struct TileWalk {
    float md;  // the minimum (the bound, if not done), its lowest index and place
    int nn, at;
    bool done;
};
constexpr float DENSE_SHARE = 0.25f;
__device__ __noinline__ TileWalk walk_tile(TreeCols C, const float* qb, float own, bool valid) {
    const float3 q = make_float3(__ldg(qb), __ldg(qb + 8), __ldg(qb + 16));
    const float2 nx = make_float2(-q.x, -q.x), ny = make_float2(-q.y, -q.y),
                 nz = make_float2(-q.z, -q.z);
    auto bound = [&](const float4* box, int i) {
        return box_bound(q, q, __ldg(box + 2 * i), __ldg(box + 2 * i + 1));
    };
    // this lane's nearest of the boxes [a, b), the first among equals
    auto nearest = [&](const float4* box, int a, int b) {
        float l = INFINITY;
        int at = a;
        for (int k = a; k < b; ++k) {
            const float t = bound(box, k);
            if (t < l) l = t, at = k;
        }
        return at;
    };
    const int b2 = nearest(C.box2, 0, C.nb2);
    const int b1 = nearest(C.box1, 8 * b2, min(8 * b2 + 8, C.nb1));
    for (int b = 8 * b1; b < min(8 * b1 + 8, C.nb); ++b) {
        float2 d[4];
        block_dist(C.pts + 8LL * b, nx, ny, nz, d);
        own = fminf(own, block_min(d));
    }
    __syncwarp();
    const int step = (C.nb + 63) / 64;
    int need = 0, boxes = 0;
    for (int b = 0; b < C.nb; b += step, ++boxes) need += bound(C.box0, b) < own ? 1 : 0;
    const int all = __reduce_add_sync(0xffffffffu, valid ? need : 0);
    const int queries = __popc(__ballot_sync(0xffffffffu, valid));
    TileWalk r{own, 0x7fffffff, 0, (float)all > DENSE_SHARE * (float)(boxes * queries)};
    if (!r.done) return r;
    if (!valid) r.md = -1.0f;  // needs nothing
    auto meets = [&](const float4* box, int i) {
        return __any_sync(0xffffffffu, bound(box, i) <= r.md);
    };
    for (int i2 = 0; i2 < C.nb2; ++i2) {
        if (!meets(C.box2, i2)) continue;
        for (int i1 = 8 * i2; i1 < min(8 * i2 + 8, C.nb1); ++i1) {
            if (!meets(C.box1, i1)) continue;
#pragma unroll 2
            for (int b = 8 * i1; b < min(8 * i1 + 8, C.nb); ++b) {
                float2 d[4];
                block_dist(C.pts + 8LL * b, nx, ny, nz, d);
                if (block_min(d) > r.md) continue;
                const float* id = reinterpret_cast<const float*>(C.pts + 8LL * b) + 24;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const float v = j & 1 ? d[j >> 1].y : d[j >> 1].x;
                    if (!(v <= r.md)) continue;  // (NaN: no distance)
                    const int i = __float_as_int(__ldg(id + j));
                    if (v < r.md || i < r.nn) r.md = v, r.nn = i, r.at = 8 * b + j;
                }
            }
        }
    }
    return r;
}

// Every warp takes 32 consecutive queries of one side of one frame in sorted order, so they lie
// close together and mostly need the same boxes.
//   - Starting bounds: the block at each query's own key among the other side's keys.
//   - The queries walk the boxes together: 32 boxes of 512 points per step against the box of the
//     queries, then the hits' boxes of 64, then per hit its boxes of 8 against the box of each
//     quad's queries. A box of 8 is evaluated when any quad needs it.
//   - Register tile: the four lanes of a quad hold the same four queries, and lane t evaluates
//     points 2 t and 2 t + 1 of a block (packed float32 operations). With one query per lane every lane loaded all of a block (96 bytes), and the
//     32 x 96 bytes through the load pipe took longer than the arithmetic (78% of the pipe's
//     wavefronts at 54% issue).
//   - Only each lane's minimum and its block are tracked; indices are found there at the end.
//   - Queries that would widen the walk of the others (outliers: a bound far above theirs), all
//     queries of a tile that meets too many boxes, and queries that met their minimum in two
//     blocks (exact ties, whose lowest index must win) are queued for k_tree_single; tiles that
//     nothing prunes are walked as a whole by walk_tile.
// Bound by instruction issue and the load pipe: 2650 instructions per tile, of which about 20
// blocks of 8 evaluated (50 each) and 9 boxes of 64 staged are most; 70% of issue slots, 60% of
// the load pipe's wavefronts, 2.4 cycles per instruction waiting for memory. 40 frames of 10 000
// points against as many: 90 us, where evaluating every pair takes 630 us (tensor-core filter)
// or 943 us (direct form). 64 uneven trajectories: 10.9 ms (one query per lane 11.5 ms and
// 3.8 ms in k_tree_single, without the gradient's sums), the tensor-core filter 158 ms.
__global__ void __launch_bounds__(SEARCH_THREADS, SEARCH_CTAS)
    k_tree_search(Ws w, int rows, int bidir) {
    pdl_wait();
    __shared__ TreeWarp s_warp[SEARCH_THREADS / 32];
    const int lane = threadIdx.x & 31, t = lane & 3, g = lane >> 2;
    const int gt = blockIdx.x * SEARCH_THREADS + (threadIdx.x & ~31);  // the tile's first query
    const int side = gt >= rows ? 1 : 0;
    const int k = w.step_frame[gt / TREE_STEP];
    const FrameDesc* fr = w.frames + k;
    const int pos0 = gt - (side ? rows + fr->col0 : fr->row0);
    if (pos0 == 0 && lane == 0 && side == 0) {
        // errors of the preparation (both sides; in Eq. 2 the targets are no queries)
        const int e0 = w.tree_err[2 * k], e1 = w.tree_err[2 * k + 1];
        if (e0 != DC_OK) set_status(&w.hdr->status, e0);
        if (e1 != DC_OK) set_status(&w.hdr->status, e1);
    }
    if (fr->skip) return;
    const int n = side ? fr->M : fr->N;
    if (pos0 >= n) return;

    const TreeCols C = tree_cols(w, fr, side, rows);
    // the quad's queries, negated and each twice (beyond the last query: its block again)
    float2 nx[4], ny[4], nz[4];
    {
        const int blk = min((pos0 >> 3) + (g >> 1), (n - 1) >> 3);
        const float4* P = reinterpret_cast<const float4*>(w.tpts) + (gt - pos0) + 8LL * blk + (g & 1);
        const float4 x = __ldg(P), y = __ldg(P + 2), z = __ldg(P + 4);
        nx[0] = make_float2(-x.x, -x.x), nx[1] = make_float2(-x.y, -x.y);
        nx[2] = make_float2(-x.z, -x.z), nx[3] = make_float2(-x.w, -x.w);
        ny[0] = make_float2(-y.x, -y.x), ny[1] = make_float2(-y.y, -y.y);
        ny[2] = make_float2(-y.z, -y.z), ny[3] = make_float2(-y.w, -y.w);
        nz[0] = make_float2(-z.x, -z.x), nz[1] = make_float2(-z.y, -z.y);
        nz[2] = make_float2(-z.z, -z.z), nz[3] = make_float2(-z.w, -z.w);
    }
    // lane l's own query is query l of the tile
    const bool valid = pos0 + lane < n;
    float own;  // its bound
    bool act;
    const int own_pos = min(pos0 + lane, n - 1);
    const float* const qb = w.tpts + 4LL * (gt - pos0) + 32LL * (own_pos >> 3) + (own_pos & 7);
    {
        const float qx = __ldg(qb), qy = __ldg(qb + 8), qz = __ldg(qb + 16);
        // Starting bound: the last block whose first key is not above the query's own. The warp
        // narrows the tile's first key down to 32 blocks, 32 probes per step; each query then
        // looks among these (their keys lie close together; beyond the last one it takes that).
        const unsigned* kc = w.tkb + (side ? fr->row0 : (long long)rows + fr->col0) / 8;
        const unsigned key = __ldg(w.tkey + (gt - pos0) + own_pos);
        const unsigned key0 = __shfl_sync(0xffffffffu, key, 0);
        int lo = 0;
        for (int len = C.nb; len > 32;) {
            const int step = (len + 31) / 32, b = lo + lane * step;
            const bool le = lane * step < len && __ldg(kc + min(b, C.nb - 1)) <= key0;
            const int c = __popc(__ballot_sync(0xffffffffu, le));
            const int skip = max(c - 1, 0) * step;
            lo += skip;
            len = min(step, len - skip);
        }
        {
            const unsigned kb = lo + lane < C.nb ? __ldg(kc + lo + lane) : 0xffffffffu;
            int p = 0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                if (__shfl_sync(0xffffffffu, kb, p + o) <= key) p += o;
            lo += p;
        }
        float2 d[4];
        block_dist(C.pts + 8LL * lo, make_float2(-qx, -qx), make_float2(-qy, -qy),
                   make_float2(-qz, -qz), d);
        const float m = block_min(d);
        own = m <= FLT_MAX ? m : FLT_MAX;  // NaN: no bound (empty boxes, at infinity, stay out)
        // outliers: a bound 2^OUTLIER_LOG2 or more above the others' (mean of the exponents)
        const int e = (int)(__float_as_uint(own) >> 23), count = min(32, n - pos0);
        const int sum = __reduce_add_sync(0xffffffffu, valid ? e : 0);
        act = valid && (e * count <= sum + OUTLIER_LOG2 * count || own == FLT_MAX);
    }
    // per query of the quad: the bound (-1: not searched here), the same in all four lanes; this
    // lane's minimum, the blocks it was met in (box of 64 << 6 | first block << 3 | second block);
    // and whether some query's minimum was met in other blocks too
    float bound[4], best[4];
    int bblk[4];
    bool tie = false;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        bound[j] = __shfl_sync(0xffffffffu, act ? own : -1.0f, (lane & ~3) + j);
        best[j] = INFINITY;
        bblk[j] = -1;
    }
    // the box of the quad's queries and their largest bound, and the tile's
    float3 slo = make_float3(INFINITY, INFINITY, INFINITY);
    float3 shi = make_float3(-INFINITY, -INFINITY, -INFINITY);
#pragma unroll
    for (int j = 0; j < 4; ++j)
        if (bound[j] >= 0.0f) {
            slo.x = fminf(slo.x, -nx[j].x), shi.x = fmaxf(shi.x, -nx[j].x);
            slo.y = fminf(slo.y, -ny[j].x), shi.y = fmaxf(shi.y, -ny[j].x);
            slo.z = fminf(slo.z, -nz[j].x), shi.z = fmaxf(shi.z, -nz[j].x);
        }
    float sR = fmaxf(max3(bound[0], bound[1], bound[2]), bound[3]);
    const float3 qlo = make_float3(warp_min(slo.x), warp_min(slo.y), warp_min(slo.z));
    const float3 qhi = make_float3(warp_max(shi.x), warp_max(shi.y), warp_max(shi.z));
    const float R = fmaxf(warp_max(sR), 0.0f);
    // one block of 8, or two at once (their minimum is folded once)
    auto eval = [&](const float4* blk, int code) {
        const float2* P = reinterpret_cast<const float2*>(blk) + t;
        const float2 px = P[0], py = P[4], pz = P[8];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float2 d = dist2x2(px, py, pz, nx[j], ny[j], nz[j]);
            const float m = fminf(d.x, d.y);
            tie |= m == best[j];
            bblk[j] = m < best[j] ? code : bblk[j];
            best[j] = fminf(best[j], m);
        }
    };
    auto eval2 = [&](const float4* ba, const float4* bb, int code) {
        const float2* P = reinterpret_cast<const float2*>(ba) + t;
        const float2* Q = reinterpret_cast<const float2*>(bb) + t;
        const float2 px = P[0], py = P[4], pz = P[8], qx = Q[0], qy = Q[4], qz = Q[8];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float2 d = dist2x2(px, py, pz, nx[j], ny[j], nz[j]);
            const float2 f = dist2x2(qx, qy, qz, nx[j], ny[j], nz[j]);
            const float m = min3(fminf(d.x, d.y), f.x, f.y);
            tie |= m == best[j];
            bblk[j] = m < best[j] ? code : bblk[j];
            best[j] = fminf(best[j], m);
        }
    };

    // the boxes of 64 that the tile meets
    TreeWarp& sw = s_warp[threadIdx.x >> 5];
    int hits = 0;
    bool wide = false;
    {
        const int grp = lane >> 3, sub = lane & 7;
        for (int s = 0; s < C.nb2 && !wide; s += 32) {
            const int i2 = s + lane, c2 = min(i2, C.nb2 - 1);
            const float l2 = box_bound(qlo, qhi, __ldg(C.box2 + 2 * c2), __ldg(C.box2 + 2 * c2 + 1));
            unsigned m2 = __ballot_sync(0xffffffffu, (l2 <= R) & (i2 < C.nb2));
            wide = __popc(m2) > WIDE_BOX2;
            while (m2 && !wide) {
                const int t2 = take4(m2, grp);
                const int i1 = (s + t2) * 8 + sub, c1 = min(max(i1, 0), C.nb1 - 1);
                const float l1 =
                    box_bound(qlo, qhi, __ldg(C.box1 + 2 * c1), __ldg(C.box1 + 2 * c1 + 1));
                const bool hit = (l1 <= R) & (t2 >= 0) & (i1 < C.nb1);
                const unsigned m1 = __ballot_sync(0xffffffffu, hit);
                if (hit) sw.hit[hits + __popc(m1 & ((1u << lane) - 1u))] = i1;
                hits += __popc(m1);
                wide = hits > WIDE_BOX1;
            }
        }
        __syncwarp();
    }
    bool done = false;  // by walk_tile, its indices and places in sw.hit (free then)
    if (wide || __popc(__ballot_sync(0xffffffffu, valid && !act)) >= MANY_OUTLIERS) {
        int met = 0;
        if (lane == 0) met = atomicAdd(&w.hdr->tree_wide, 1);
        met = __shfl_sync(0xffffffffu, met, 0);
        if (met >= max(FEW_WIDE, (int)gridDim.x / FEW_WIDE)) {
            const TileWalk r = walk_tile(C, qb, own, valid);
            own = r.md;
            done = r.done;
            if (done) sw.hit[lane] = r.nn, sw.hit[32 + lane] = r.at;
        }
    }
    // their blocks
    if (!wide && !done) {
        auto stage = [&](int h) {
            if (h < hits) {
                TreeStage& st = sw.stage[h & (STAGES - 1)];
                const int b1 = sw.hit[h];
                const float4* P = C.pts + 64LL * b1;
                copy16(&st.pts[lane], P + lane);
                copy16(&st.pts[lane + 32], P + lane + 32);
                if (lane < 16) copy16(&st.box[lane], C.box0 + 16 * b1 + lane);
            }
            copy_commit();  // (an empty group keeps the count)
        };
#pragma unroll
        for (int h = 0; h < STAGES - 1; ++h) stage(h);
        for (int h = 0; h < hits; ++h) {
            copy_wait<STAGES - 2>();
            __syncwarp();  // the stage has landed for every lane, and the one before is done with
            stage(h + STAGES - 1);
            const TreeStage& st = sw.stage[h & (STAGES - 1)];
            const int b1 = sw.hit[h];
            // each box of 8 against the queries of each quad: lane t tests boxes t and t + 4
            const float l0 = box_bound(slo, shi, st.box[2 * t], st.box[2 * t + 1]);
            const float l1 = box_bound(slo, shi, st.box[2 * t + 8], st.box[2 * t + 9]);
            unsigned m = __reduce_or_sync(
                0xffffffffu, (l0 <= sR ? 1u << t : 0u) | (l1 <= sR ? 16u << t : 0u));
            if (!m) continue;
            do {
                const int c = __ffs(m) - 1;
                m &= m - 1;
                if (m) {
                    const int d = __ffs(m) - 1;
                    m &= m - 1;
                    eval2(st.pts + 8 * c, st.pts + 8 * d, (b1 << 6) | (c << 3) | d);
                } else {
                    eval(st.pts + 8 * c, (b1 << 6) | (c << 3) | c);
                }
            } while (m);
            const bool better = best[0] < bound[0] || best[1] < bound[1] || best[2] < bound[2] ||
                                best[3] < bound[3];
            if (__any_sync(0xffffffffu, better)) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    float v = best[j];
                    v = fminf(v, __shfl_xor_sync(0xffffffffu, v, 1));
                    v = fminf(v, __shfl_xor_sync(0xffffffffu, v, 2));
                    bound[j] = fminf(bound[j], v);
                }
                sR = fmaxf(max3(bound[0], bound[1], bound[2]), bound[3]);
            }
        }
    }

    // The indices: the lowest one attaining the query's minimum among the quad's lanes, and its
    // place in the sorted order; lane t keeps those of the quad's t-th query, its own.
    float md = own;
    int nn = 0x7fffffff, at = 0;
    const unsigned tied = __ballot_sync(0xffffffffu, tie) >> (lane & ~3);
    const bool alone = valid && !done && (wide || !act || (tied & 0xfu) != 0);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float v = best[j];
        v = fminf(v, __shfl_xor_sync(0xffffffffu, v, 1));
        v = fminf(v, __shfl_xor_sync(0xffffffffu, v, 2));
        int i = 0x7fffffff, p = 0;
        if (bblk[j] >= 0 && best[j] == v) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int b = 8 * (bblk[j] >> 6) + ((h ? bblk[j] : bblk[j] >> 3) & 7);
                const float2* P = reinterpret_cast<const float2*>(C.pts + 8LL * b) + t;
                const float2 d = dist2x2(__ldg(P), __ldg(P + 4), __ldg(P + 8), nx[j], ny[j], nz[j]);
                const float2 id = __ldg(P + 12);
                const int ix = __float_as_int(id.x), iy = __float_as_int(id.y);
                if (d.x == v && ix < i) i = ix, p = 8 * b + 2 * t;
                if (d.y == v && iy < i) i = iy, p = 8 * b + 2 * t + 1;
            }
        }
        const int mine = i;
        i = min(i, __shfl_xor_sync(0xffffffffu, i, 1));
        i = min(i, __shfl_xor_sync(0xffffffffu, i, 2));
        // indices are distinct: one lane holds the minimum
        const unsigned holds = __ballot_sync(0xffffffffu, mine == i) >> (lane & ~3);
        p = __shfl_sync(0xffffffffu, p, (lane & ~3) + ((__ffs(holds) - 1) & 3));
        if (t == j) {
            nn = i;
            at = p;
            md = fminf(md, v);
        }
    }
    if (done) nn = sw.hit[lane], at = sw.hit[32 + lane];  // (own is the minimum)
    // the pair's gradient, added to the sim point's (the query's own, or its neighbour's for a
    // target query), 16 bytes at once
    const float gs = grad_scale(fr, side, bidir);
    if (gs != 0.0f && valid && !alone && nn != 0x7fffffff) {
        const float* A = w.tpts + 4LL * (gt - pos0) + 32LL * ((pos0 + lane) >> 3) + ((pos0 + lane) & 7);
        const float* B = reinterpret_cast<const float*>(C.pts) + 32LL * (at >> 3) + (at & 7);
        const float sg = side ? -gs : gs;  // sim point - target, whichever is the query
        red_add4(w.tgx + fr->row0 + (side ? at : pos0 + lane),
                 __fmul_rn(sg, __fsub_rn(__ldg(A), __ldg(B))),
                 __fmul_rn(sg, __fsub_rn(__ldg(A + 8), __ldg(B + 8))),
                 __fmul_rn(sg, __fsub_rn(__ldg(A + 16), __ldg(B + 16))));
    }
    if (valid) {
        // this lane's query's index; the slot of a queued query carries its bound
        const int pos = pos0 + lane;
        const int qi = __float_as_int(__ldg(w.tpts + 4LL * (gt - pos0) + 32LL * (pos >> 3) + 24 + (pos & 7)));
        u64* out_p = side ? w.pba + fr->col0 : w.pab + fr->row0;
        out_p[qi] = alone || nn != 0x7fffffff ? ((u64)__float_as_uint(md) << 32) | (unsigned)nn : EMPTY;
    }
    const unsigned am = __ballot_sync(0xffffffffu, alone);
    if (am) {
        int at = 0;
        if (lane == 0) at = atomicAdd(&w.hdr->tree_n, __popc(am));
        at = __shfl_sync(0xffffffffu, at, 0);
        if (alone) w.tqueue[at + __popc(am & ((1u << lane) - 1u))] = gt + lane;
    }
    pdl_trigger();
}

// The queued queries, one warp each: the same walk with the query's own box (a point), every
// lane one point of four blocks of 8. Bound by latency (three levels of dependent loads, 12.6
// cycles per instruction), so 64 warps per SM at 32 registers, although that spills: with 42 or
// 51 registers (48 and 40 warps) the 100-frame call of 32 768 points takes 1770 and 1784 us
// instead of 1755. 64 uneven trajectories 1.24 ms, 40 frames of 10 000 points 31 us.
constexpr int SINGLE_THREADS = 128;
__global__ void __launch_bounds__(SINGLE_THREADS, 16) k_tree_single(Ws w, int rows, int bidir) {
    pdl_wait();
    const int lane = threadIdx.x & 31, grp = lane >> 3, sub = lane & 7;
    const int count = w.hdr->tree_n;
    const int step = gridDim.x * (SINGLE_THREADS / 32);
    for (int e = (int)(blockIdx.x * SINGLE_THREADS + threadIdx.x) / 32; e < count; e += step) {
        const int g = w.tqueue[e];
        const int side = g >= rows ? 1 : 0;
        const FrameDesc* fr = w.frames + w.step_frame[g / TREE_STEP];
        const TreeCols C = tree_cols(w, fr, side, rows);
        const int base = side ? rows + fr->col0 : fr->row0, pos = g - base;
        const float* qb = w.tpts + 4LL * base + 32LL * (pos >> 3) + (pos & 7);
        const float3 q = make_float3(__ldg(qb), __ldg(qb + 8), __ldg(qb + 16));
        u64* slot = (side ? w.pba + fr->col0 : w.pab + fr->row0) + __float_as_int(__ldg(qb + 24));
        float R = __uint_as_float((unsigned)(*slot >> 32));  // the bound so far
        unsigned md = 0x7f800000u, mi = 0x7fffffffu;  // this lane's minimum and its index
        int mb = 0;                                    // and its block
        // The lanes whose box (of 512 or 64; bound l, lowest index `first`) matters. Exact ties: one
        // whose bound is R itself matters only with a lower index than the lowest one found at R.
        // (Where points coincide, all boxes tie: 8 frames of 10 000 coincident points took 4970 us
        // without this, 270 us with it.)
        auto matter = [&](float l, float first) {
            unsigned m = __ballot_sync(0xffffffffu, l <= R);
            if (__any_sync(0xffffffffu, l == R)) {
                const unsigned found =
                    __reduce_min_sync(0xffffffffu, __uint_as_float(md) == R ? mi : 0x7fffffffu);
                m = __ballot_sync(0xffffffffu, l < R || (l == R && __float_as_uint(first) < found));
            }
            return m;
        };
        // this lane's point of block b
        auto point = [&](int b) {
            const float* P = reinterpret_cast<const float*>(C.pts + 8LL * b) + sub;
            const float dx = __fsub_rn(q.x, __ldg(P)), dy = __fsub_rn(q.y, __ldg(P + 8)),
                        dz = __fsub_rn(q.z, __ldg(P + 16));
            const unsigned i = __float_as_uint(__ldg(P + 24));
            const unsigned db =
                __float_as_uint(__fmaf_rn(dz, dz, __fmaf_rn(dy, dy, __fmul_rn(dx, dx))));
            if (db < md || (db == md && i < mi)) md = db, mi = i, mb = b;
        };
        for (int s = 0; s < C.nb2; s += 32) {
            const int i2 = s + lane;
            float lb = INFINITY, first = 0.f;
            if (i2 < C.nb2) {
                const float4 lo = __ldg(C.box2 + 2 * i2);
                first = lo.w;
                lb = box_bound(q, q, lo, __ldg(C.box2 + 2 * i2 + 1));
            }
            unsigned m2 = matter(lb, first);
            if (s == 0 && __popc(m2) > 2) {
                // a loose bound: the points of the nearest box of 64 in the nearest box of 512
                const unsigned near2 = __reduce_min_sync(0xffffffffu, __float_as_uint(lb));
                const int n2 = __ffs(__ballot_sync(0xffffffffu, __float_as_uint(lb) == near2)) - 1;
                const int i1 = 8 * n2 + sub;
                float l1 = INFINITY;
                if (i1 < C.nb1)
                    l1 = box_bound(q, q, __ldg(C.box1 + 2 * i1), __ldg(C.box1 + 2 * i1 + 1));
                const unsigned near1 = __reduce_min_sync(0xffffffffu, __float_as_uint(l1));
                const int n1 =
                    8 * n2 + ((__ffs(__ballot_sync(0xffffffffu, __float_as_uint(l1) == near1)) - 1) & 7);
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    if (8 * n1 + 4 * h + grp < C.nb) point(8 * n1 + 4 * h + grp);
                R = fminf(R, __uint_as_float(__reduce_min_sync(0xffffffffu, md)));
                m2 = matter(lb, first);
            }
            while (m2) {
                const int t2 = take4(m2, grp);
                const int i1 = (s + t2) * 8 + sub;
                float l1 = INFINITY, first1 = 0.f;
                if (t2 >= 0 && i1 < C.nb1) {
                    const float4 lo = __ldg(C.box1 + 2 * i1);
                    first1 = lo.w;
                    l1 = box_bound(q, q, lo, __ldg(C.box1 + 2 * i1 + 1));
                }
                unsigned m1 = matter(l1, first1);
                while (m1) {
                    const int t1 = take4(m1, grp);
                    const int i0 = __shfl_sync(0xffffffffu, i1, t1 & 31) * 8 + sub;
                    bool hit = false;
                    if (t1 >= 0 && i0 < C.nb)
                        hit = box_bound(q, q, __ldg(C.box0 + 2 * i0), __ldg(C.box0 + 2 * i0 + 1)) <= R;
                    unsigned m0 = __ballot_sync(0xffffffffu, hit);
                    while (m0) {
                        const int t0 = take4(m0, grp);
                        const int b = __shfl_sync(0xffffffffu, i0, t0 & 31);
                        if (t0 >= 0) point(b);
                    }
                    R = fminf(R, __uint_as_float(__reduce_min_sync(0xffffffffu, md)));
                }
            }
        }
        const unsigned dm = __reduce_min_sync(0xffffffffu, md);
        const unsigned im = __reduce_min_sync(0xffffffffu, md == dm ? mi : 0x7fffffffu);
        if (lane == 0) *slot = im == 0x7fffffffu ? EMPTY : ((u64)dm << 32) | im;
        const float gs = grad_scale(fr, side, bidir);
        const unsigned who = __ballot_sync(0xffffffffu, md == dm && mi == im);
        if (gs != 0.0f && im != 0x7fffffffu && lane == __ffs(who) - 1) {
            const float* P = reinterpret_cast<const float*>(C.pts + 8LL * mb) + sub;
            const float sg = side ? -gs : gs;
            red_add4(w.tgx + fr->row0 + (side ? 8 * mb + sub : pos),
                     __fmul_rn(sg, __fsub_rn(q.x, __ldg(P))),
                     __fmul_rn(sg, __fsub_rn(q.y, __ldg(P + 8))),
                     __fmul_rn(sg, __fsub_rn(q.z, __ldg(P + 16))));
        }
    }
    pdl_trigger();
}

// ---------------------------------------------------------------------------------------
// losses and vertex gradients
// ---------------------------------------------------------------------------------------
constexpr int OUT_THREADS = 256;

// Blocks [0, loss_blocks): the loss partials of OUT_THREADS / lanes (frame, slice)s each, and the
// neighbours where the caller wants them, from the (distance, index) records, coalesced. `lanes`
// threads sum a slice in the order of the general epilogue (a thread per row, every lanes-th row;
// then a tree over the threads), so the losses are bit for bit those of the other engines.
// The other blocks: TREE_STEP sim points in sorted order each, their gradient spread over their
// face's vertices with the barycentric weights (Eq. 4), 16 bytes per vertex. In sorted order
// neighbouring points share faces and vertices, so the face look-ups hit L1; against one atomic
// per coordinate and (point, target) pair the points' sums save half the scatter, and vectors
// two thirds of the rest (64 uneven trajectories: 3.8 ms as one epilogue, 1.4 ms here). Bound by
// the latency of its gathers and the L2's atomics (40 frames of 10 000 points: 21 us, of 20 MB).
__global__ void __launch_bounds__(OUT_THREADS) k_tree_out(Ws w, int n_frames, int slices, int lanes,
                                                          int loss_blocks, int steps, int bidir) {
    pdl_entry();
    const int tid = threadIdx.x;
    if ((int)blockIdx.x >= loss_blocks) {
        // two steps per block, so that two chains of dependent loads overlap
        const FrameDesc* fr[2];
        float4 g[2];
        int4 q[2];
        int i[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int step = 2 * (blockIdx.x - loss_blocks) + h;
            fr[h] = w.frames + w.step_frame[min(step, steps - 1)];
            const int at = step * TREE_STEP + tid, p = at - fr[h]->row0;
            q[h].x = -1;
            i[h] = -1;
            if (step < steps && !fr[h]->skip && fr[h]->grad && fr[h]->verts && p < fr[h]->N) {
                g[h] = w.tgx[at];
                i[h] = __float_as_int(
                    __ldg(w.tpts + 4LL * fr[h]->row0 + 32LL * (p >> 3) + 24 + (p & 7)));
            }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if (i[h] >= 0) q[h] = __ldg(w.fw + fr[h]->row0 + i[h]);
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if (q[h].x >= 0) scatter_face(w, fr[h], q[h], g[h]);
        return;
    }
    __shared__ float s_red[2][OUT_THREADS / 8];
    const int ks = blockIdx.x * (OUT_THREADS / lanes) + tid / lanes, t = tid & (lanes - 1);
    const bool on = ks < n_frames * slices;
    const int k = on ? ks / slices : 0, sl = on ? ks - k * slices : 0;
    const FrameDesc* fr = w.frames + k;
    const bool live = on && !fr->skip;
#pragma unroll 1
    for (int side = 0; side < (bidir ? 2 : 1); ++side) {
        const int n = side ? fr->M : fr->N, nc = side ? fr->N : fr->M;
        const u64* rec = side ? w.pba + fr->col0 : w.pab + fr->row0;
        int* nn = side ? fr->nn_ba : fr->nn_ab;
        const int a = (int)((long long)n * sl / slices), b = (int)((long long)n * (sl + 1) / slices);
        float s = 0.f, c = 0.f;
        bool bad = false;
        if (live) {
#pragma unroll 4
            for (int i = a + t; i < b; i += lanes) {
                const u64 p = __ldg(rec + i);
                const unsigned j = (unsigned)p;
                if (p != EMPTY) {  // compensated sum
                    const float y = __fsub_rn(__uint_as_float((unsigned)(p >> 32)), c);
                    const float u = __fadd_rn(s, y);
                    c = __fsub_rn(__fsub_rn(u, s), y);
                    s = u;
                }
                bad |= p == EMPTY || j >= (unsigned)nc;
                if (nn) nn[i] = p == EMPTY ? -1 : (int)j;
            }
        }
        if (bad) set_status(&w.hdr->status, DC_EDEVICE);
        // eight threads at a time, then over their sums
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) s = __fadd_rn(s, __shfl_down_sync(0xffffffffu, s, o, 8));
        if ((tid & 7) == 0) s_red[side][tid >> 3] = s;
    }
    __syncthreads();
    // one thread per side of each slice; the tree of a warp over lanes / 8 values, zeros beyond
    const int sides = tid & 1, q = tid >> 1, at = blockIdx.x * (OUT_THREADS / lanes) + q;
    if (q < OUT_THREADS / lanes && at < n_frames * slices) {
        float v[OUT_THREADS / 8];
#pragma unroll
        for (int i = 0; i < OUT_THREADS / 8; ++i)
            v[i] = i < lanes / 8 && (sides == 0 || bidir) ? s_red[sides][q * (lanes / 8) + i] : 0.f;
#pragma unroll
        for (int o = OUT_THREADS / 16; o > 0; o >>= 1)
#pragma unroll
            for (int i = 0; i < o; ++i) v[i] = __fadd_rn(v[i], v[i + o]);
        w.part[2 * at + sides] = v[0];
    }
}

int g_prep_smem[64];  // per device: dynamic shared memory the preparation may use
int g_sms[64];        // and SMs

}  // namespace

cudaError_t launch_tree(const UniformArgs* a, const Ws& w, int n_frames, int max_f, int max_n,
                        int rows, int cols, int mode, cudaStream_t s) {
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) dev = 0;
    constexpr int STATIC = 7 * 1024;  // room for the static shared memory
    if (g_prep_smem[dev] == 0) {
        int optin = 0, sms = 0;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        g_sms[dev] = sms > 0 ? sms : 1;
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
        optin = (optin > 0 ? optin : 99 * 1024) - STATIC;
        for (auto f : {k_tree_prep<1>, k_tree_prep<2>, k_tree_prep<3>, k_tree_prep<4>,
                       k_tree_prep<6>, k_tree_prep<8>}) {
            cudaError_t e =
                cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
            if (e) return e;
        }
        g_prep_smem[dev] = optin;
    }
    // Few frames: a cluster of up to 8 CTAs per (frame, side), as many as are resident at once
    // (two per SM), each with at least one point per thread.
    int S = 1;
    for (int q : {2, 3, 4, 6, 8})
        if (n_frames * q <= g_sms[dev] && max_n >= q * PREP_THREADS) S = q;
    // the CDF, later the cells and the refinement's buffers: two CTAs per SM up to 27 000 faces
    size_t smem = CELL_BYTES + REFINE_BYTES;
    const bool cdf_shared = 4 * (size_t)max_f <= (size_t)g_prep_smem[dev];
    if (cdf_shared) smem = std::max(smem, 4 * (size_t)max_f);

    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(2 * n_frames * S);
    cfg.blockDim = dim3(PREP_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = S;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = S > 1 ? 2 : 1;
    const UniformArgs none{};
    auto kernel = S == 8   ? k_tree_prep<8>
                  : S == 6 ? k_tree_prep<6>
                  : S == 4 ? k_tree_prep<4>
                  : S == 3 ? k_tree_prep<3>
                  : S == 2 ? k_tree_prep<2>
                           : k_tree_prep<1>;
    cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, a ? *a : none, w, (int)(a != nullptr),
                                       n_frames, rows, (int)cdf_shared);
    count_launch();
    if (e) return e;
    prof_before(s);
    const int total = rows + (mode == DC_BIDIR_MEAN ? cols : 0);
    const int bidir = mode == DC_BIDIR_MEAN;
    e = launch_pdl(k_tree_search, total / SEARCH_THREADS, SEARCH_THREADS, 0, s, w, rows, bidir);
    count_launch();
    if (!e) {
        e = launch_pdl(k_tree_single, std::min(16 * g_sms[dev], total / SINGLE_THREADS), SINGLE_THREADS, 0,
                       s, w, rows, bidir);
        count_launch();
    }
    prof_after(s);
    return e ? e : cudaGetLastError();
}

// After launch_tree: loss partials, neighbours, gradients, then the frame losses and their total.
// max_v: largest V of the frames with a gradient (0: no gradient).
cudaError_t launch_tree_out(const Ws& w, int n_frames, int slices, int lanes, int max_v, int rows,
                            int mode, float* total, cudaStream_t s) {
    const int bidir = mode == DC_BIDIR_MEAN;
    const int loss_blocks = div_up(n_frames * slices, OUT_THREADS / lanes);
    const int steps = rows / TREE_STEP;
    cudaError_t e = launch_pdl(k_tree_out, loss_blocks + (max_v > 0 ? div_up(steps, 2) : 0),
                               OUT_THREADS, 0, s, w, n_frames, slices, lanes, loss_blocks, steps,
                               bidir);
    count_launch();
    if (!e && max_v > 0) e = launch_grad_out(w, n_frames, max_v, s);
    return e ? e : launch_frame_loss(w, n_frames, slices, bidir, total, s);
}

}  // namespace dc
