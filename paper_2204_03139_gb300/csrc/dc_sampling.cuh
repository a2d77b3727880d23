// Device code of the sampling step (Sec. III-B, Eq. 3) shared by the staging kernels and the
// pruned search's preparation: frame records of uniform trajectories, face areas, the
// compensated prefix sum, the face pick and the barycentric point.
#pragma once

#include "dc_async.cuh"
#include "dc_internal.cuh"

namespace dc {
namespace {

__device__ __forceinline__ bool coord_ok(float v) { return fabsf(v) <= COORD_MAX; }

// Frame k's weight w_t in the total and the multiplier of its gradient. The forward uses w_t
// for both. The recomputing backward gets the objective's derivatives: g_t = dJ/dL_t =
// w_t dJ/dL_total + dJ/dL_t(direct), and 0 for a frame of weight 0, whose forward L_t is the
// constant 0.
__device__ __forceinline__ void frame_scales(const UniformArgs& a, int k, float& w, float& gs) {
    w = a.weight ? a.weight[k] : 1.0f;
    if (a.bwd) {
        const float gt = a.gtotal ? a.gtotal[0] : 0.0f;
        const float gf = a.gframes ? a.gframes[k] : 0.0f;
        gs = w == 0.0f ? 0.0f : __fadd_rn(__fmul_rn(w, gt), gf);
    } else {
        gs = w;
    }
}

// The record of frame k of a uniform trajectory (unit0 left at 0).
__device__ __forceinline__ FrameDesc uniform_frame(const UniformArgs& a, const Ws& w, int k) {
    const int Npad = round_up(a.N, ROW_PAD), Mpad = round_up(a.M, COL_PAD);
    FrameDesc f;
    f.verts = a.verts ? a.verts + 3LL * k * a.V : nullptr;
    f.faces = a.faces;
    f.mask = a.mask;
    f.draws = a.draws ? a.draws + 3LL * k * a.N : nullptr;
    f.pts = a.pts ? a.pts + 3LL * k * a.N : nullptr;
    f.tgt = a.tgt ? a.tgt + 3LL * k * a.M : nullptr;
    f.loss = a.loss ? a.loss + k : w.loss + k;
    // the pruned search needs no neighbour buffers of its own
    const bool tree = a.engine == ENGINE_TREE;
    f.nn_ab = a.nn_ab ? a.nn_ab + (long long)k * a.N
                      : (tree ? nullptr : w.nnab + (long long)k * Npad);
    f.nn_ba = a.nn_ba ? a.nn_ba + (long long)k * a.M
                      : (tree ? nullptr : w.nnba + (long long)k * Mpad);
    f.grad = a.grad ? a.grad + 3LL * k * a.V : nullptr;
    f.out_pts = a.out_pts ? a.out_pts + 3LL * k * a.N : nullptr;
    f.out_face = a.out_face ? a.out_face + (long long)k * a.N : nullptr;
    f.out_bary = a.out_bary ? a.out_bary + 3LL * k * a.N : nullptr;
    f.V = a.V;
    f.F = a.F;
    f.N = a.N;
    f.M = a.M;
    f.Npad = Npad;
    f.Mpad = Mpad;
    frame_scales(a, k, f.weight, f.gscale);
    f.skip = f.weight == 0.0f || f.gscale == 0.0f;
    f.row0 = k * Npad;
    f.col0 = k * Mpad;
    f.cdf0 = k * a.F;
    f.v0 = k * a.V;
    f.unit0 = 0;
    return f;
}

// ---------------------------------------------------------------------------------------
// area CDF: two-float (compensated) prefix sum of the float32 face areas, so that the
// stored C_f is the float32 rounding of the exact prefix sum of those areas
// ---------------------------------------------------------------------------------------
struct FF {
    float hi, lo;
};

__device__ __forceinline__ FF ff_norm(float s, float e) {
    float h = __fadd_rn(s, e);
    return {h, __fsub_rn(e, __fsub_rn(h, s))};
}

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

__device__ __forceinline__ FF ff_add(FF a, FF b) {
    float s, e;
    two_sum(a.hi, b.hi, s, e);
    return ff_norm(s, __fadd_rn(e, __fadd_rn(a.lo, b.lo)));
}

__device__ __forceinline__ FF ff_add1(FF a, float b) {
    float s, e;
    two_sum(a.hi, b, s, e);
    return ff_norm(s, __fadd_rn(e, a.lo));
}

// area 1/2 |(p1 - p0) x (p2 - p0)| of the triangle with corners q[9]; flags bad coordinates
__device__ __forceinline__ float corner_area(const float (&q)[9], bool& bad) {
#pragma unroll
    for (int k = 0; k < 9; ++k) bad |= !coord_ok(q[k]);
    // explicit roundings: both passes of the scan must see bit-identical areas
    const float e1x = __fsub_rn(q[3], q[0]), e1y = __fsub_rn(q[4], q[1]),
                e1z = __fsub_rn(q[5], q[2]);
    const float e2x = __fsub_rn(q[6], q[0]), e2y = __fsub_rn(q[7], q[1]),
                e2z = __fsub_rn(q[8], q[2]);
    const float cx = __fsub_rn(__fmul_rn(e1y, e2z), __fmul_rn(e1z, e2y));
    const float cy = __fsub_rn(__fmul_rn(e1z, e2x), __fmul_rn(e1x, e2z));
    const float cz = __fsub_rn(__fmul_rn(e1x, e2y), __fmul_rn(e1y, e2x));
    const float n2 = __fmaf_rn(cz, cz, __fmaf_rn(cy, cy, __fmul_rn(cx, cx)));
    return __fmul_rn(0.5f, __fsqrt_rn(n2));
}

// area of face f = 1/2 |(p1 - p0) x (p2 - p0)|; flags bad indices / coordinates
__device__ __forceinline__ float face_area(const float* __restrict__ verts,
                                           const int* __restrict__ faces, int V, int f,
                                           bool& bad_idx, bool& bad_val) {
    const int i0 = faces[3 * f], i1 = faces[3 * f + 1], i2 = faces[3 * f + 2];
    if ((unsigned)i0 >= (unsigned)V || (unsigned)i1 >= (unsigned)V ||
        (unsigned)i2 >= (unsigned)V) {
        bad_idx = true;
        return 0.0f;
    }
    const float* p0 = verts + 3LL * i0;
    const float* p1 = verts + 3LL * i1;
    const float* p2 = verts + 3LL * i2;
    const float q[9] = {p0[0], p0[1], p0[2], p1[0], p1[1], p1[2], p2[0], p2[1], p2[2]};
    return corner_area(q, bad_val);
}

// The area weight of face f: its area, or 0 for a face outside the sampled subset
// (Sec. IV-F). The face is still checked, so that bad indices are reported either way.
__device__ __forceinline__ float face_weight(const float* __restrict__ verts,
                                             const int* __restrict__ faces,
                                             const uint8_t* __restrict__ mask, int V, int f,
                                             bool& bad_idx, bool& bad_val) {
    const float a = face_area(verts, faces, V, f, bad_idx, bad_val);
    return (mask && mask[f] == 0) ? 0.0f : a;
}

constexpr int CDF_THREADS = 1024;

// What the area step needs to know about one frame.
struct AreaFrame {
    const float* verts;   // [V][3]
    const int* faces;     // [F][3]
    const uint8_t* mask;  // [F] nullable
    float* grad;          // [V][3] nullable: zeroed here for the epilogue's accumulation
    float* cdf;           // [F] out
    int F, V;
    bool skip;            // weight 0: only the gradient (zero) is written
};

// Face pick by inverse CDF: the first face with C_f > r_f A
__device__ __forceinline__ int pick_face(const float* cdf, int F, float rf) {
    const float t = __fmul_rn(rf, cdf[F - 1]);
    int lo = 0, hi = F;  // first f with cdf[f] > t
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (cdf[mid] > t)
            hi = mid;
        else
            lo = mid + 1;
    }
    return min(lo, F - 1);
}

// pick_face of two draws at once: their binary searches' dependent loads overlap
__device__ __forceinline__ void pick_face2(const float* cdf, int F, float ra, float rb, int& fa,
                                           int& fb) {
    const float A = cdf[F - 1];
    const float ta = __fmul_rn(ra, A), tb = __fmul_rn(rb, A);
    int la = 0, lb = 0;  // first f with cdf[f] > t, by halving steps over [l, l + len)
    for (int len = F; len > 0;) {
        const int half = len >> 1;
        const bool ga = cdf[min(la + half, F - 1)] <= ta && la + half < F;
        const bool gb = cdf[min(lb + half, F - 1)] <= tb && lb + half < F;
        la = ga ? la + half + 1 : la;
        lb = gb ? lb + half + 1 : lb;
        len = half;
    }
    fa = min(la, F - 1);
    fb = min(lb, F - 1);
}

// barycentric weights of the draw (r1, r2), and the point's coordinate with corners a, b, c
__device__ __forceinline__ void bary_weights(float r1, float r2, float& w0, float& w1, float& w2) {
    const float s = __fsqrt_rn(r1);
    w0 = __fsub_rn(1.0f, s);
    w1 = __fmul_rn(s, __fsub_rn(1.0f, r2));
    w2 = __fmul_rn(s, r2);
}
__device__ __forceinline__ float bary_point(float w0, float w1, float w2, float a, float b,
                                            float c) {
    return __fmaf_rn(w2, c, __fmaf_rn(w1, b, __fmul_rn(w0, a)));
}

// The point of the draw (r_f, r1, r2): x = point, q = (face, w0, w1, w2 bits). False, with x = 0
// and no face, when the face has a vertex index out of range.
__device__ __forceinline__ bool pick_point(const float* cdf, int F, int V,
                                           const float* __restrict__ verts,
                                           const int* __restrict__ faces, float rf, float r1,
                                           float r2, float4& x, int4& q) {
    const int f = pick_face(cdf, F, rf);
    const int i0 = faces[3 * f], i1 = faces[3 * f + 1], i2 = faces[3 * f + 2];
    if ((unsigned)i0 >= (unsigned)V || (unsigned)i1 >= (unsigned)V ||
        (unsigned)i2 >= (unsigned)V) {
        x = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        return false;
    }
    const float* p0 = verts + 3LL * i0;
    const float* p1 = verts + 3LL * i1;
    const float* p2 = verts + 3LL * i2;
    float w0, w1, w2;
    bary_weights(r1, r2, w0, w1, w2);
    x.x = bary_point(w0, w1, w2, p0[0], p1[0], p2[0]);
    x.y = bary_point(w0, w1, w2, p0[1], p1[1], p2[1]);
    x.z = bary_point(w0, w1, w2, p0[2], p1[2], p2[2]);
    q = make_int4(f, __float_as_int(w0), __float_as_int(w1), __float_as_int(w2));
    return true;
}

// ---- gradient accumulators of 16 bytes ----
__device__ __forceinline__ void red_add4(float4* p, float x, float y, float z) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(x), "f"(y), "f"(z),
                 "f"(0.0f)
                 : "memory");
}

// Multiplier of (point - neighbour) in dL/dpoint for the queries of a side: 2 g / N (sim points)
// or 2 g / M (targets) in Eq. 1, 2 g in Eq. 2 (the derivative of the squared distance); 0 when
// the frame has no gradient.
__device__ __forceinline__ float grad_scale(const FrameDesc* fr, int side, int bidir) {
    if (!fr->grad || !fr->verts) return 0.0f;
    const float g = __fmul_rn(2.0f, fr->gscale);
    return bidir ? __fdiv_rn(g, (float)(side ? fr->M : fr->N)) : g;
}


// a sim point's gradient g to the vertices of its face (q: face, weights) of frame fr
__device__ __forceinline__ void scatter_face(const Ws& w, const FrameDesc* fr, int4 q, float4 g) {
    const float wt[3] = {__int_as_float(q.y), __int_as_float(q.z), __int_as_float(q.w)};
    const int* f = fr->faces + 3LL * q.x;
    int v[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) v[k] = __ldg(f + k);
#pragma unroll
    for (int k = 0; k < 3; ++k)
        if ((unsigned)v[k] < (unsigned)fr->V)
            red_add4(w.grad4 + fr->v0 + v[k], __fmul_rn(wt[k], g.x), __fmul_rn(wt[k], g.y),
                     __fmul_rn(wt[k], g.z));
}

}  // namespace
}  // namespace dc
