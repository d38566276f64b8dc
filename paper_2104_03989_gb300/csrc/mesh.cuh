// Device code of the mesh operations (Sec. 5.1): the vertex frame and the uniform
// Laplacian of Eq. 4, per vertex, gathered over a vertex -> face (or one-ring) CSR table,
// so that results do not depend on atomic ordering. The kernels that run them are in
// mesh.cu, raster.cu (beside the tile lists) and optim.cu (with the positions' Adam).
#pragma once

#include "kernels.cuh"

namespace adms {

struct FaceFrame {
    float3 e1, e2, fn, tv;
    float d1y, d2y;
    int sgn;
    int idx[3];
};

__device__ __forceinline__ FaceFrame face_frame(const FrameArgs& a, int f) {
    FaceFrame r;
    int i0 = a.tri[3 * f], i1 = a.tri[3 * f + 1], i2 = a.tri[3 * f + 2];
    r.idx[0] = i0;
    r.idx[1] = i1;
    r.idx[2] = i2;
    float3 p0 = f3(a.pos[3 * i0], a.pos[3 * i0 + 1], a.pos[3 * i0 + 2]);
    float3 p1 = f3(a.pos[3 * i1], a.pos[3 * i1 + 1], a.pos[3 * i1 + 2]);
    float3 p2 = f3(a.pos[3 * i2], a.pos[3 * i2 + 1], a.pos[3 * i2 + 2]);
    float2 u0 = a.uv[a.tri_uv[3 * f]], u1 = a.uv[a.tri_uv[3 * f + 1]], u2 = a.uv[a.tri_uv[3 * f + 2]];
    r.e1 = p1 - p0;
    r.e2 = p2 - p0;
    r.fn = cross3(r.e1, r.e2);
    float d1x = u1.x - u0.x, d2x = u2.x - u0.x;
    r.d1y = u1.y - u0.y;
    r.d2y = u2.y - u0.y;
    float det = d1x * r.d2y - d2x * r.d1y;
    r.sgn = det > 0.f ? 1 : (det < 0.f ? -1 : 0);
    r.tv = r.d2y * r.e1 - r.d1y * r.e2;
    return r;
}

// The gathers over a vertex's faces (or one-ring) run in batches of ADMS_GATHER:
// the batch's loads are issued together (the last entry repeated past the end)
// and summed in list order, so each sum keeps the order of a plain loop while the
// dependent loads of a vertex take ceil(valence / ADMS_GATHER) round trips
// instead of one per face.
#define ADMS_GATHER 4

// unnormalised vertex normal (sum of face normals) and tangent (sum of signed unit face tangents)
__device__ __forceinline__ void vertex_sums(const FrameArgs& a, int v, float3& n, float3& t) {
    n = zero3();
    t = zero3();
    int lo = a.vf_off[v], hi = a.vf_off[v + 1];
    for (int j0 = lo; j0 < hi; j0 += ADMS_GATHER) {
        FaceFrame ff[ADMS_GATHER];
#pragma unroll
        for (int q = 0; q < ADMS_GATHER; ++q) ff[q] = face_frame(a, a.vf_face[min(j0 + q, hi - 1)]);
#pragma unroll
        for (int q = 0; q < ADMS_GATHER; ++q) {
            if (j0 + q < hi) {
                n += ff[q].fn;
                if (ff[q].sgn != 0) t += (float)ff[q].sgn * nrm3(ff[q].tv).y;
            }
        }
    }
}

// smooth normal, tangent and their inverse lengths of vertex v
__device__ __forceinline__ void frame_vertex(const FrameArgs& a, int v) {
    float3 n, t;
    vertex_sums(a, v, n, t);
    Nrm3 nn = nrm3(n), tn = nrm3(t);
    a.vpos[v] = make_float4(a.pos[3 * v], a.pos[3 * v + 1], a.pos[3 * v + 2], 0.f);
    a.vnrm[v] = make_float4(nn.y.x, nn.y.y, nn.y.z, 0.f);
    a.vtan[v] = make_float4(tn.y.x, tn.y.y, tn.y.z, 0.f);
    if (a.inv) a.inv[v] = make_float2(nn.big ? nn.inv : -nn.inv, tn.big ? tn.inv : -tn.inv);
}

// delta_i of vertex i (none past the last); the block's sum of |delta|^2 is added to
// st->lap_sum (every thread of the block calls it; red: a double per warp)
__device__ __forceinline__ void lap_vertex(const LapArgs& a, int i, double* red) {
    double s = 0.0;
    if (i < a.V) {
        int lo = a.ring_off[i], hi = a.ring_off[i + 1];
        float3 m = zero3();
        for (int j0 = lo; j0 < hi; j0 += ADMS_GATHER) {
            float3 pk[ADMS_GATHER];
#pragma unroll
            for (int q = 0; q < ADMS_GATHER; ++q) {
                int k = a.ring[min(j0 + q, hi - 1)];
                pk[q] = f3(a.pos[3 * k], a.pos[3 * k + 1], a.pos[3 * k + 2]);
            }
#pragma unroll
            for (int q = 0; q < ADMS_GATHER; ++q)
                if (j0 + q < hi) m += pk[q];
        }
        float inv = hi > lo ? 1.f / (float)(hi - lo) : 0.f;
        float3 d = f3(a.pos[3 * i], a.pos[3 * i + 1], a.pos[3 * i + 2]) - inv * m;
        if (a.delta_ref) d -= f3(a.delta_ref[3 * i], a.delta_ref[3 * i + 1], a.delta_ref[3 * i + 2]);
        a.delta[3 * i] = d.x;
        a.delta[3 * i + 1] = d.y;
        a.delta[3 * i + 2] = d.z;
        s = (double)dot3(d, d);
    }
    s = warp_sum_d(s);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double sum = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) sum += red[w];
        atomicAdd(&a.st->lap_sum, sum);
    }
}

// g -= sum over the one-ring i of vertex k of delta_i / |ring(i)| (the adjoint of
// the one-ring means, gathered per vertex)
__device__ __forceinline__ void ring_adjoint(const LapArgs& a, int k, float3& g) {
    int lo = a.ring_off[k], hi = a.ring_off[k + 1];
    for (int j0 = lo; j0 < hi; j0 += ADMS_GATHER) {
        float inv[ADMS_GATHER];
        float3 d[ADMS_GATHER];
#pragma unroll
        for (int q = 0; q < ADMS_GATHER; ++q) {
            int i = a.ring[min(j0 + q, hi - 1)];
            inv[q] = 1.f / (float)(a.ring_off[i + 1] - a.ring_off[i]);
            d[q] = f3(a.delta[3 * i], a.delta[3 * i + 1], a.delta[3 * i + 2]);
        }
#pragma unroll
        for (int q = 0; q < ADMS_GATHER; ++q)
            if (j0 + q < hi) g -= inv[q] * d[q];
    }
}

}  // namespace adms
