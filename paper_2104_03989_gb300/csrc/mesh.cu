// Mesh operations (Sec. 5.1): smooth vertex normals and tangents from positions
// and UVs, recomputed every step, with their adjoint; the uniform Laplacian
// regularizer of Eq. 4.
//
// Both run one thread per vertex and gather over a vertex -> face (or one-ring)
// CSR table, so results do not depend on atomic ordering.
#include "mesh.cuh"

namespace adms {

__global__ void k_frame_fwd(FrameArgs a) {
    int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v < a.V) frame_vertex(a, v);
}

// the normalisation of vertex c's normal (k = 0) or tangent (k = 1) sum as the
// forward left it: the unit vector and the signed inverse length
__device__ __forceinline__ Nrm3 stored_nrm3(const FrameArgs& a, int c, int k) {
    float4 y = k == 0 ? a.vnrm[c] : a.vtan[c];
    float2 iv = a.inv[c];
    float s = k == 0 ? iv.x : iv.y;
    Nrm3 r;
    r.y = f3(y.x, y.y, y.z);
    r.inv = fabsf(s);
    r.big = s > 0.f;
    return r;
}

// dL/d(normal sum) of vertex c: the adjoint of its normalisation (k_frame_bwd1's tmp_n)
__device__ __forceinline__ float3 sum_grad(const FrameArgs& a, int c, int k) {
    const double* g = (k == 0 ? a.g_nrm : a.g_tan) + 3 * c;
    return nrm3_bwd(stored_nrm3(a, c, k), f3((float)g[0], (float)g[1], (float)g[2]));
}

// phase 1: gradients w.r.t. the unnormalised sums
__global__ void k_frame_bwd1(FrameArgs a) {
    int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= a.V) return;
    float3 n, t;
    vertex_sums(a, v, n, t);
    float3 gn = nrm3_bwd(nrm3(n), f3((float)a.g_nrm[3 * v], (float)a.g_nrm[3 * v + 1], (float)a.g_nrm[3 * v + 2]));
    float3 gt = nrm3_bwd(nrm3(t), f3((float)a.g_tan[3 * v], (float)a.g_tan[3 * v + 1], (float)a.g_tan[3 * v + 2]));
    a.tmp_n[v] = make_float4(gn.x, gn.y, gn.z, 0.f);
    a.tmp_t[v] = make_float4(gt.x, gt.y, gt.z, 0.f);
}

// g_pos[v] += the pixel stage's float64 position gradient + g (the frame adjoint);
// the float64 accumulator is zeroed for the next backward
__device__ __forceinline__ void fold_position_grad(const FrameArgs& a, int v, float3 g) {
    double* acc = a.g_pos_acc + 3 * v;
    double g0 = acc[0] + (double)g.x, g1 = acc[1] + (double)g.y, g2 = acc[2] + (double)g.z;
    if (a.status && !(isfinite(g0) && isfinite(g1) && isfinite(g2))) atomicExch(a.status, (int)ADMS_ERR_NONFINITE);
    a.g_pos[3 * v] += (float)g0;
    a.g_pos[3 * v + 1] += (float)g1;
    a.g_pos[3 * v + 2] += (float)g2;
    acc[0] = 0.0;
    acc[1] = 0.0;
    acc[2] = 0.0;
}

// phase 2: each vertex gathers its share of every incident face's adjoint
__global__ void k_frame_bwd2(FrameArgs a) {
    int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= a.V) return;
    float3 g = zero3();
    int lo = a.vf_off[v], hi = a.vf_off[v + 1];
    for (int j0 = lo; j0 < hi; j0 += ADMS_GATHER) {
        FaceFrame ff[ADMS_GATHER];
        float3 Gfn[ADMS_GATHER], Gft[ADMS_GATHER];
#pragma unroll
        for (int q = 0; q < ADMS_GATHER; ++q) {
            ff[q] = face_frame(a, a.vf_face[min(j0 + q, hi - 1)]);
            Gfn[q] = f3(a.tmp_n[ff[q].idx[0]]) + f3(a.tmp_n[ff[q].idx[1]]) + f3(a.tmp_n[ff[q].idx[2]]);
            Gft[q] = f3(a.tmp_t[ff[q].idx[0]]) + f3(a.tmp_t[ff[q].idx[1]]) + f3(a.tmp_t[ff[q].idx[2]]);
        }
#pragma unroll
        for (int q = 0; q < ADMS_GATHER; ++q) {
            if (j0 + q >= hi) continue;
            float3 ge1 = cross3(ff[q].e2, Gfn[q]), ge2 = cross3(Gfn[q], ff[q].e1);
            if (ff[q].sgn != 0) {
                float3 gtv = (float)ff[q].sgn * nrm3_bwd(nrm3(ff[q].tv), Gft[q]);
                ge1 += ff[q].d2y * gtv;
                ge2 -= ff[q].d1y * gtv;
            }
            if (ff[q].idx[0] == v) g -= ge1 + ge2;
            if (ff[q].idx[1] == v) g += ge1;
            if (ff[q].idx[2] == v) g += ge2;
        }
    }
    fold_position_grad(a, v, g);
}

// k_frame_bwd1 and k_frame_bwd2 in one launch, after a frame_forward that kept the
// normalisations (a.inv): eight threads per vertex, slot s taking the vertex's
// incident faces s, s + 8, ... and forming their corners' normalisation adjoints
// itself; the slots' sums are combined by shuffles in a fixed order
#define ADMS_FRAME_SLOTS 8
template <int N>
__global__ void __launch_bounds__(128) k_frame_bwd_fused(const __grid_constant__ Pack<FrameArgs, N> P) {
    const FrameArgs& a = P.a[N == 1 ? 0 : blockIdx.y];
    int gid = blockIdx.x * blockDim.x + threadIdx.x;
    int v = gid / ADMS_FRAME_SLOTS, slot = gid % ADMS_FRAME_SLOTS;
    bool valid = v < a.V;
    float3 g = zero3();
    if (valid) {
        int lo = a.vf_off[v], hi = a.vf_off[v + 1];
        for (int j = lo + slot; j < hi; j += ADMS_FRAME_SLOTS) {
            FaceFrame ff = face_frame(a, a.vf_face[j]);
            float3 Gfn = sum_grad(a, ff.idx[0], 0) + sum_grad(a, ff.idx[1], 0) + sum_grad(a, ff.idx[2], 0);
            float3 ge1 = cross3(ff.e2, Gfn), ge2 = cross3(Gfn, ff.e1);
            if (ff.sgn != 0) {
                float3 Gft = sum_grad(a, ff.idx[0], 1) + sum_grad(a, ff.idx[1], 1) + sum_grad(a, ff.idx[2], 1);
                float3 gtv = (float)ff.sgn * nrm3_bwd(nrm3(ff.tv), Gft);
                ge1 += ff.d2y * gtv;
                ge2 -= ff.d1y * gtv;
            }
            if (ff.idx[0] == v) g -= ge1 + ge2;
            if (ff.idx[1] == v) g += ge1;
            if (ff.idx[2] == v) g += ge2;
        }
    }
    // the eight slots of a vertex are consecutive lanes of one warp
#pragma unroll
    for (int o = ADMS_FRAME_SLOTS / 2; o > 0; o >>= 1) {
        g.x += __shfl_down_sync(0xffffffffu, g.x, o, ADMS_FRAME_SLOTS);
        g.y += __shfl_down_sync(0xffffffffu, g.y, o, ADMS_FRAME_SLOTS);
        g.z += __shfl_down_sync(0xffffffffu, g.z, o, ADMS_FRAME_SLOTS);
    }
    if (valid && slot == 0) fold_position_grad(a, v, g);
}

cudaError_t frame_forward(const FrameArgs& a, cudaStream_t st) {
    k_frame_fwd<<<(a.V + 127) / 128, 128, 0, st>>>(a);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t frame_backward(const FrameArgs* as, int n, cudaStream_t st) {
    return launch_packed(as, n, 128, st, k_frame_bwd_fused<1>, k_frame_bwd_fused<ADMS_BATCH_JOBS>,
                         [](const FrameArgs& a) { return (a.V * ADMS_FRAME_SLOTS + 127) / 128; });
}

cudaError_t frame_backward(const FrameArgs& a, cudaStream_t st) {
    if (a.inv) return frame_backward(&a, 1, st);
    k_frame_bwd1<<<(a.V + 127) / 128, 128, 0, st>>>(a);
    k_frame_bwd2<<<(a.V + 127) / 128, 128, 0, st>>>(a);
    count_launches(2);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ Laplacian (Eq. 4)
__global__ void k_lap_fwd(LapArgs a) {
    __shared__ double red[4];
    lap_vertex(a, blockIdx.x * blockDim.x + threadIdx.x, red);
}

cudaError_t laplacian_forward(const LapArgs& a, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(&a.st->lap_sum, 0, sizeof(double), st);
    if (e) return e;
    k_lap_fwd<<<(a.V + 127) / 128, 128, 0, st>>>(a);
    count_launches(1);
    return cudaGetLastError();
}

__global__ void k_lap_value(LapArgs a, float* out) { *out = (float)(a.st->lap_sum / (double)a.V); }

// g = scale * dL_delta/dpos, written (not accumulated) into a.g_pos
__global__ void k_lap_grad_out(LapArgs a, float scale) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= a.V) return;
    float s = 2.f * scale / (float)a.V;
    float3 g = f3(a.delta[3 * k], a.delta[3 * k + 1], a.delta[3 * k + 2]);
    ring_adjoint(a, k, g);
    a.g_pos[3 * k] = s * g.x;
    a.g_pos[3 * k + 1] = s * g.y;
    a.g_pos[3 * k + 2] = s * g.z;
}

cudaError_t laplacian_value(const LapArgs& a, float* out, cudaStream_t st) {
    k_lap_value<<<1, 1, 0, st>>>(a, out);
    count_launches(1);
    return cudaGetLastError();
}

// g_pos += lambda_t dL_delta/dpos
__global__ void k_lap_add(LapArgs a) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= a.V || a.st->status) return;
    float scale = 2.f * a.st->lam / (float)a.V;
    float3 g = f3(a.delta[3 * k], a.delta[3 * k + 1], a.delta[3 * k + 2]);
    ring_adjoint(a, k, g);
    a.g_pos[3 * k] += scale * g.x;
    a.g_pos[3 * k + 1] += scale * g.y;
    a.g_pos[3 * k + 2] += scale * g.z;
}

cudaError_t laplacian_add(const LapArgs& a, cudaStream_t st) {
    k_lap_add<<<(a.V + 127) / 128, 128, 0, st>>>(a);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t laplacian_gradient(const LapArgs& a, float scale, cudaStream_t st) {
    k_lap_grad_out<<<(a.V + 127) / 128, 128, 0, st>>>(a, scale);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace adms
