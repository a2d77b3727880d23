// The recomputing backward (dc_loss_traj_bwd): the vertex gradient of given neighbours, with the
// sampled points recomputed from the draws.
//
// Every pair (sim point, target) contributes c (x - y) to its sim point's gradient (derivative of
// Eq. 1 / 2), and a sim point's gradient goes to its face's vertices with the barycentric weights
// (Eq. 4). The pairs are summed per sim point first, so each point is scattered once however many
// targets chose it, and both sums use 16-byte vector atomics: a target costs one of them and a sim
// point three, instead of nine scalar atomics each. Bound by the L2's random accesses (the
// neighbour gathers and the atomics). 100 frames of 32 768 points against as many targets: the
// general staging and epilogue, which this replaces, took 138 + 404 us; the rows here 145, the
// columns 42, the scatter 63 and the copy out 9 us.
#include <algorithm>

#include "dc_sampling.cuh"

namespace dc {

namespace {

constexpr int ROW_THREADS = 512;
constexpr int COL_THREADS = 256;
constexpr int OUT_THREADS = 256;

// Rows of a (frame, slice): the sampled points and face records, and c (x - y) of each point and
// its neighbour as the start of its sum. Two points per thread and step, so that their chains of
// dependent loads overlap. The frame's CDF in shared memory (cdf_shared) or where it is.
__global__ void __launch_bounds__(ROW_THREADS) k_bwd_rows(Ws w, int slices, int bidir,
                                                          int cdf_shared) {
    pdl_entry();
    extern __shared__ float s_cdf[];
    const int k = blockIdx.x / slices, sl = blockIdx.x - k * slices, tid = threadIdx.x;
    const FrameDesc* fr = w.frames + k;
    if (sl == 0 && tid == 0 && w.frame_err[k] != DC_OK) set_status(&w.hdr->status, w.frame_err[k]);
    if (fr->skip) return;
    const int F = fr->F, V = fr->V, N = fr->N, M = fr->M;
    for (int v = sl * ROW_THREADS + tid; v < V; v += slices * ROW_THREADS)
        w.grad4[fr->v0 + v] = make_float4(0.f, 0.f, 0.f, 0.f);
    const float* cdf = w.cdf + fr->cdf0;
    if (cdf_shared) {
        for (int f = tid; f < F; f += ROW_THREADS) s_cdf[f] = cdf[f];
        __syncthreads();
        cdf = s_cdf;
    }
    const float c = grad_scale(fr, 0, bidir);
    const int a = (int)((long long)N * sl / slices), b = (int)((long long)N * (sl + 1) / slices);
    bool bad = false;
    for (int ib = a + tid; ib < b; ib += 2 * ROW_THREADS) {
        const int ii[2] = {ib, min(ib + ROW_THREADS, b - 1)};  // the last may be done twice
        float d[2][3], y[2][3];
        int nn[2], f[2], v[2][3];
        bool in[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
#pragma unroll
            for (int m = 0; m < 3; ++m) d[h][m] = fr->draws[3LL * ii[h] + m];
            nn[h] = fr->nn_ab[ii[h]];
            if ((unsigned)nn[h] >= (unsigned)M) {
                bad = true;
                nn[h] = -1;
            }
        }
        pick_face2(cdf, F, d[0][0], d[1][0], f[0], f[1]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
#pragma unroll
            for (int m = 0; m < 3; ++m) {
                v[h][m] = __ldg(fr->faces + 3 * f[h] + m);
                y[h][m] = nn[h] >= 0 ? __ldg(fr->tgt + 3LL * nn[h] + m) : 0.0f;
                bad |= !(d[h][m] >= 0.0f && d[h][m] <= 1.0f);
            }
            in[h] = (unsigned)v[h][0] < (unsigned)V && (unsigned)v[h][1] < (unsigned)V &&
                    (unsigned)v[h][2] < (unsigned)V;
            bad |= !in[h];
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float p[3][3];
#pragma unroll
            for (int m = 0; m < 3; ++m)
#pragma unroll
                for (int q = 0; q < 3; ++q)
                    p[m][q] = in[h] ? __ldg(fr->verts + 3LL * v[h][m] + q) : 0.0f;
            float w0, w1, w2;
            bary_weights(d[h][1], d[h][2], w0, w1, w2);
            const float4 x = make_float4(bary_point(w0, w1, w2, p[0][0], p[1][0], p[2][0]),
                                         bary_point(w0, w1, w2, p[0][1], p[1][1], p[2][1]),
                                         bary_point(w0, w1, w2, p[0][2], p[1][2], p[2][2]), 0.0f);
            const int i = fr->row0 + ii[h];
            w.x[i] = x;
            w.fw[i] = make_int4(in[h] ? f[h] : -1, __float_as_int(w0), __float_as_int(w1),
                                __float_as_int(w2));
            const float s = nn[h] >= 0 ? c : 0.0f;
            w.tgx[i] = make_float4(__fmul_rn(s, __fsub_rn(x.x, y[h][0])),
                                   __fmul_rn(s, __fsub_rn(x.y, y[h][1])),
                                   __fmul_rn(s, __fsub_rn(x.z, y[h][2])), 0.0f);
        }
    }
    if (bad) set_status(&w.hdr->status, DC_EINVAL);
}

// Targets (blockIdx.y: frame): their coordinates are checked, and in Eq. 1 c (x - y) is added to
// their neighbour's sum.
__global__ void __launch_bounds__(COL_THREADS) k_bwd_cols(Ws w, int bidir) {
    pdl_entry();
    const FrameDesc* fr = w.frames + blockIdx.y;
    const int j = blockIdx.x * COL_THREADS + threadIdx.x;
    if (fr->skip || j >= fr->M) return;
    const float* t = fr->tgt + 3LL * j;
    const float y[3] = {t[0], t[1], t[2]};
    bool bad = !coord_ok(y[0]) || !coord_ok(y[1]) || !coord_ok(y[2]);
    if (bidir) {
        const int i = fr->nn_ba[j];
        if ((unsigned)i < (unsigned)fr->N) {
            const float4 x = w.x[fr->row0 + i];
            const float c = grad_scale(fr, 1, bidir);
            red_add4(w.tgx + fr->row0 + i, __fmul_rn(c, __fsub_rn(x.x, y[0])),
                     __fmul_rn(c, __fsub_rn(x.y, y[1])), __fmul_rn(c, __fsub_rn(x.z, y[2])));
        } else {
            bad = true;
        }
    }
    if (bad) set_status(&w.hdr->status, DC_EINVAL);
}

// sim points (blockIdx.y: frame): their sums to their faces' vertices
__global__ void __launch_bounds__(COL_THREADS) k_bwd_scatter(Ws w) {
    pdl_entry();
    const FrameDesc* fr = w.frames + blockIdx.y;
    const int i = blockIdx.x * COL_THREADS + threadIdx.x;
    if (fr->skip || i >= fr->N) return;
    const float4 g = w.tgx[fr->row0 + i];
    const int4 q = w.fw[fr->row0 + i];
    if (q.x < 0) return;
    scatter_face(w, fr, q, g);
}

// vertex gradients from their 16-byte accumulators to the caller's [V][3] (0 for skipped frames)
__global__ void __launch_bounds__(OUT_THREADS) k_grad_out(Ws w) {
    pdl_entry();
    const FrameDesc* fr = w.frames + blockIdx.x;
    if (!fr->grad || !fr->verts) return;
    for (int v = blockIdx.y * OUT_THREADS + threadIdx.x; v < fr->V; v += gridDim.y * OUT_THREADS) {
        const float4 g = fr->skip ? make_float4(0.f, 0.f, 0.f, 0.f) : __ldg(w.grad4 + fr->v0 + v);
        fr->grad[3LL * v] = g.x;
        fr->grad[3LL * v + 1] = g.y;
        fr->grad[3LL * v + 2] = g.z;
    }
}

int g_rows_smem[64];  // per device: dynamic shared memory of k_bwd_rows

}  // namespace

cudaError_t launch_grad_out(const Ws& w, int n_frames, int max_v, cudaStream_t s) {
    cudaError_t e = launch_pdl(k_grad_out, dim3(n_frames, std::min(64, div_up(max_v, 4 * OUT_THREADS))),
                               OUT_THREADS, 0, s, w);
    count_launch();
    return e;
}

cudaError_t launch_backward(const UniformArgs& a, const Ws& w, cudaStream_t s) {
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) dev = 0;
    if (g_rows_smem[dev] == 0) {
        int optin = 0;
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
        if (optin <= 0) optin = 48 * 1024;
        cudaError_t e = cudaFuncSetAttribute(k_bwd_rows, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             optin);
        if (e) return e;
        g_rows_smem[dev] = optin;
    }
    const int bidir = a.mode == DC_BIDIR_MEAN;
    cudaError_t e = launch_build_area(a, w, s);
    if (e) return e;
    const size_t need = (size_t)a.F * sizeof(float);
    const int shared = need <= (size_t)g_rows_smem[dev];
    e = launch_pdl(k_bwd_rows, a.T * a.slices, ROW_THREADS, shared ? need : 0, s, w, a.slices, bidir,
                   shared);
    count_launch();
    if (e) return e;
    e = launch_pdl(k_bwd_cols, dim3(div_up(a.M, COL_THREADS), a.T), COL_THREADS, 0, s, w, bidir);
    count_launch();
    if (e) return e;
    e = launch_pdl(k_bwd_scatter, dim3(div_up(a.N, COL_THREADS), a.T), COL_THREADS, 0, s, w);
    count_launch();
    return e ? e : launch_grad_out(w, a.T, a.V, s);
}

}  // namespace dc
