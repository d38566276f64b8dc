// Per-pixel deferred shading, silhouette antialiasing, image loss and the fused
// backward (Sec. 5.2 renderer, Sec. 5.3 objective).
//
// No G-buffer is stored: every per-pixel kernel recomputes the perspective-
// correct barycentrics and the interpolated attributes from the visibility
// key (triangle id) and the per-view vertex data.
//
// Precision: screen positions arrive as float-float pairs computed in float64
// per vertex, so offsets from the pixel centre keep float32 relative
// precision; attributes are interpolated as corner-0 value + weighted corner
// differences, which keeps texel coordinates of large textures accurate and
// lets the barycentric adjoint use (a_j - a) without cancellation. Vertex
// gradients are accumulated in float64.
#include "pixel.cuh"

namespace adms {

// ------------------------------------------------------------------ single-job kernels (16x16 tiles)
// the listed pixels of one job (A.refine[0] of them), grid-stride
__global__ void __launch_bounds__(64) k_shade_refine(ShadeArgs A) {
    int n = A.refine[0];
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        shade_refine_px(A, A.refine[1 + i]);
}

// A 16x16 tile of pixels is shaded by 256 / THREADS blocks, each a band of 16 x (THREADS / 16)
// rows. COLS: columns of a warp, 8 (a warp takes 8x4 pixels) or 16 (16x2). The forward's compact
// warps meet fewer triangles and texels: 94.2 -> 92.3 us (8 views of 512x512 of a dense mesh), 836
// -> 822 (peeled layers, two passes). The backward keeps rows: 8x4 gave 1% there, opaque, and lost
// 1.5% on peeled layers, and the other order of its atomics flips Adam's first step at texels
// whose gradients cancel.
template <int THREADS, int COLS>
__device__ __forceinline__ void band_pixel(int W, int& px, int& py) {
    constexpr int PARTS = 256 / THREADS, ACROSS = ADMS_TILE / COLS, ROWS = 32 / COLS;
    int tiles_x = (W + ADMS_TILE - 1) / ADMS_TILE;
    int tile = blockIdx.x / PARTS, part = blockIdx.x % PARTS;
    int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    px = (tile % tiles_x) * ADMS_TILE + COLS * (warp % ACROSS) + lane % COLS;
    py = (tile / tiles_x) * ADMS_TILE + part * (ADMS_TILE / PARTS) + ROWS * (warp / ACROSS) + lane / COLS;
}

// Block shapes (threads per block x resident blocks per SM, i.e. the register cap 65536 /
// (threads x blocks)), measured per kernel. SHARE (maps of one size, decided by the host per
// launch) is a template argument: one kernel holding both forms cost the maps of different
// sizes 3% (895 -> 920 us for the two passes over 16 views of 1024x1024). Equal maps, 8 views
// of 512x512: 8 blocks 74.5 us, 6: 80.0, 10: 77.9, 12: 77.4; different ones, 16 views of
// 1024x1024: 8 blocks 894 us, 6: 964, 10: 883, 12: 832, but with the refinement inline (small
// grids) 8 is ahead (69.0 against 70.3 us at 5 of 333x501). AA + loss: 16 blocks; 12 are
// ahead where few warps enter the pair loop (5 of 333x501: 32.4 against 34.4 us) and behind where
// many do (600k leaf quads 69.8 against 66.2, peeled layers 961 against 912).
#define ADMS_FWD_THREADS 128
constexpr int fwd_blocks(bool inline_refine, int share) { return share != 1 && !inline_refine ? 12 : 8; }
#define ADMS_AA_THREADS 128
#define ADMS_AA_BLOCKS 16
template <bool INLINE, int SHARE>
__global__ void __launch_bounds__(ADMS_FWD_THREADS, fwd_blocks(INLINE, SHARE)) k_shade_fwd(ShadeArgs A) {
    int px, py;
    band_pixel<ADMS_FWD_THREADS, 8>(A.W, px, py);
    // blockIdx.z: the layer of a depth-peeled job (the layers' shading is independent; a launch
    // and a refinement pass per layer left eight tails and eight nearly empty passes, 15 us each)
    shade_fwd_px<INLINE, SHARE>(A, blockIdx.y, px, py, (size_t)blockIdx.z * ((size_t)A.B * A.H * A.W));
}

// FINISH: the last block finishes the call's loss (a launch of its own otherwise)
template <bool PEEL, bool FINISH, bool GIVEN = false>
__global__ void __launch_bounds__(ADMS_AA_THREADS, ADMS_AA_BLOCKS) k_aa_loss(ShadeArgs A, JobState* fin, float* out) {
    __shared__ float red[ADMS_AA_THREADS / 16];
    int bx = (A.W + 31) / 32;  // a warp takes 32 columns of one row
    LossSum sum;
    aa_pixel<PEEL, GIVEN>(A, blockIdx.y, (blockIdx.x % bx) * 32 + (threadIdx.x & 31),
                   (blockIdx.x / bx) * (ADMS_AA_THREADS / 32) + (threadIdx.x >> 5), sum);
    add_block_loss(A, sum, red);
    if (FINISH && threadIdx.x == 0 && last_block(fin, TICKET_LOSS, gridDim.x * gridDim.y)) finish_job_loss(fin, out);
}

// resident blocks per SM of the fused backward (register cap 65536 / (threads x this))
// (the plain-method step: 256 threads x 3 blocks 0.174 ms; 128 x 5: 0.175; 128 x 6:
// 0.171; 128 x 7: 0.171)
#ifndef ADMS_BWD_BLOCKS
#define ADMS_BWD_BLOCKS 6
#endif
#ifndef ADMS_BWD_THREADS
#define ADMS_BWD_THREADS 128  // 256: a block per 16x16 tile; 128: two blocks of 16x8 pixels
#endif
template <bool PEEL>
__global__ void __launch_bounds__(ADMS_BWD_THREADS, ADMS_BWD_BLOCKS) k_shade_bwd(ShadeArgs A) {
    __shared__ float rows[(ADMS_BWD_THREADS / 32) * 32 * ADMS_VROW];
    int px, py;
    band_pixel<ADMS_BWD_THREADS, 16>(A.W, px, py);
    shade_bwd_px<PEEL>(A, blockIdx.y, px, py, rows + (threadIdx.x >> 5) * 32 * ADMS_VROW);
}

// MSAA forward: a block takes a 32x32-sample region (four samples per thread), its
// (pixel, triangle) groups are compacted into a shared-memory list and each group is
// shaded by one thread; every sample copies its group's colour. (A 16x16 region holds
// only ~70 groups at 2x2 MSAA, which left most of a block's warps waiting while three
// shaded.)
#define ADMS_MSAA_REGION 32
__global__ void __launch_bounds__(256, 4) k_shade_fwd_msaa(ShadeArgs A) {
    constexpr int R = ADMS_MSAA_REGION, N = R * R, PER = N / 256;
    __shared__ int tri[N];
    __shared__ short list[N];
    __shared__ float4 col[N];
    __shared__ int count;
    int rx = (A.W + R - 1) / R;
    int b = blockIdx.y, tid = threadIdx.x;
    int x0 = (blockIdx.x % rx) * R, y0 = (blockIdx.x / rx) * R;
    if (tid == 0) count = 0;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        int t = tid + 256 * k, px = x0 + (t % R), py = y0 + (t / R);
        bool inside = px < A.W && py < A.H;
        tri[t] = inside ? key_tri(A.keys[((size_t)b * A.H + py) * A.W + px]) : -1;
    }
    __syncthreads();
    int lead[PER];
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        int t = tid + 256 * k;
        lead[k] = group_leader(A.msaa, x0, y0, R, x0 + (t % R), y0 + (t / R), tri[t], tri);
        if (lead[k] == t) list[atomicAdd(&count, 1)] = (short)t;
    }
    __syncthreads();
    int n = count;
    for (int i = tid; i < n; i += 256) {
        int t = list[i];
        int sx = x0 + (t % R), sy = y0 + (t / R);
        col[t] = shade_covered(A, b, sx, sy, tri[t], ((size_t)b * A.H + sy) * A.W + sx);
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        int t = tid + 256 * k, px = x0 + (t % R), py = y0 + (t / R);
        if (px < A.W && py < A.H)
            A.pre[((size_t)b * A.H + py) * A.W + px] = lead[k] >= 0 ? col[lead[k]] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

// MSAA backward over a 32x32-sample region (four samples per thread): the AA
// adjoint runs per sample; the shading adjoint of a (pixel, triangle) group is
// linear in its colour gradient and its samples share the shading, so the group's
// leader takes the sum of its samples' gradients (in a fixed order) and the
// compacted leaders run the adjoint once per group
__global__ void __launch_bounds__(256, 3) k_shade_bwd_msaa(ShadeArgs A) {
    constexpr int R = ADMS_MSAA_REGION, N = R * R, PER = N / 256;
    __shared__ int tri[N];
    __shared__ float3 gsum[N];
    __shared__ short list[N];
    __shared__ int count;
    __shared__ float rows[8 * 32 * ADMS_VROW];
    int rx = (A.W + R - 1) / R;
    int b = blockIdx.y, tid = threadIdx.x;
    int x0 = (blockIdx.x % rx) * R, y0 = (blockIdx.x / rx) * R;
    if (tid == 0) count = 0;
    for (int k = 0; k < PER; ++k) {
        int t = tid + 256 * k, px = x0 + (t % R), py = y0 + (t / R);
        int f = -1;
        float3 gc = zero3();
        if (px < A.W && py < A.H) {
            size_t pix = ((size_t)b * A.H + py) * A.W + px;
            unsigned long long kp = A.keys[pix];
            f = key_tri(kp);
            gc = aa_adjoint<false>(A, b, px, py, pix, kp);
        }
        tri[t] = f;
        gsum[t] = gc;
    }
    __syncthreads();
    // leaders sum their groups (registers first: other leaders still read gsum)
    float3 g[PER];
    bool leader[PER];
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        int t = tid + 256 * k, px = x0 + (t % R), py = y0 + (t / R);
        int f = tri[t];
        g[k] = zero3();
        leader[k] = false;
        if (f < 0) continue;
        int sm = A.msaa, ox = (px / sm) * sm, oy = (py / sm) * sm;
        int first = -1;
        for (int y = max(oy, y0); y < min(oy + sm, y0 + R); ++y)
            for (int x = max(ox, x0); x < min(ox + sm, x0 + R); ++x) {
                int u = (y - y0) * R + (x - x0);
                if (tri[u] != f) continue;
                if (first < 0) first = u;
                g[k] += gsum[u];
            }
        leader[k] = first == t;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        int t = tid + 256 * k;
        if (leader[k] && (g[k].x != 0.f || g[k].y != 0.f || g[k].z != 0.f)) {
            gsum[t] = g[k];
            list[atomicAdd(&count, 1)] = (short)t;
        }
    }
    __syncthreads();
    int n = count;
    // warp-uniform trips: the vertex scatter is warp-collective
    for (int base = tid & ~31; base < n; base += 256) {
        int i = base + (tid & 31);
        int fl = -1;
        float* wrows = rows + (tid >> 5) * 32 * ADMS_VROW;
        if (i < n) {
            int t = list[i];
            fl = tri[t];
            shading_adjoint<false>(A, b, x0 + (t % R), y0 + (t / R), fl, gsum[t], 0.f, wrows + (tid & 31) * ADMS_VROW);
        }
        scatter_vertex_rows(A, fl, wrows);
    }
}

// ------------------------------------------------------------------ persistent batched kernels
// One launch covers (job, view, tile) work items of up to 64 jobs with
// different meshes, textures, view counts and resolutions. Block k takes items
// k, k + gridDim.x, ... (equal tiles of tw x (256 / tw) pixels, so a static
// stride balances them without a shared counter). The jobs' arguments are
// kernel parameters: read-only, no copy per block, and no aliasing with the
// stores and atomics of the pixel code.
// refinement lists of a batch (see k_shade_refine): reset before the shading
// launch, then one grid-stride pass per job (blockIdx.y)
__global__ void k_refine_reset(const ShadeBatch P, int n) {
    int k = threadIdx.x;
    if (k < n && P.a[k].refine) P.a[k].refine[0] = 0;
}
__global__ void __launch_bounds__(256) k_refine_batch(const ShadeBatch P) {
    const ShadeArgs& A = P.a[blockIdx.y];
    if (!A.refine) return;
    int n = A.refine[0];
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        shade_refine_px(A, A.refine[1 + i]);
}

// Two blocks of 128 threads take a tile, as in the single-job kernels: shorter tails and finer
// register rounding (eight uneven jobs: backward 498 -> 484 us, shading 206 -> 190, AA + loss 143
// -> 135 against blocks of 256). The grid and the tuned blocks per SM stay in tiles. Shading at 10
// blocks per SM: 190 us, at the single-job kernel's 8: 208.
constexpr int batch_blocks(int kind) { return kind == 2 ? ADMS_BWD_BLOCKS : kind == 1 ? ADMS_AA_BLOCKS : 10; }
template <int KIND>
__global__ void __launch_bounds__(128, batch_blocks(KIND))
    k_pixels_batch(const ShadeBatch P, const WorkItem* __restrict__ items, int n, int tw, int job0) {
    __shared__ float red[8];
    __shared__ float rows[KIND == 2 ? 4 * 32 * ADMS_VROW : 1];
    for (int it = blockIdx.x; it < 2 * n; it += gridDim.x) {
        WorkItem w = items[it >> 1];
        const ShadeArgs& A = P.a[w.job - job0];
        int t = (int)threadIdx.x + 128 * (it & 1);
        int px = w.x0 + t % tw, py = w.y0 + t / tw;
        if (KIND == 0) shade_fwd_px(A, w.view, px, py);
        else if (KIND == 1) {
            LossSum sum;
            aa_pixel<false>(A, w.view, px, py, sum);
            add_block_loss(A, sum, red);
        }
        else shade_bwd_px(A, w.view, px, py, rows + (threadIdx.x >> 5) * 32 * ADMS_VROW);
    }
}

// ------------------------------------------------------------------ supersample resolve
// Was bound by its instructions (54.6 M a launch at 2x2 samples of 8 views of 512x512: 64-bit
// divisions for the pixel, loops of unknown length, six tone maps on a black background): a view
// per grid row, the usual 2x2 (SS) unrolled, black on black skipped as in the AA + loss.
// AA and resolve of two passes: 296 -> 264 us.
template <int SS>  // samples a side, 0: r.S
__global__ void __launch_bounds__(256) k_resolve(ResolveArgs r) {
    __shared__ float red[16];
    const int S = SS ? SS : r.S;
    unsigned rem = blockIdx.x * blockDim.x + threadIdx.x;
    int b = blockIdx.y;
    LossSum sum;
    if (rem < (unsigned)(r.H * r.W)) {
        int py = rem / (unsigned)r.W, px = rem - py * r.W;
        size_t pix = (size_t)b * r.H * r.W + rem;
        int SW = S * r.W;
        size_t base = ((size_t)b * S * r.H + (size_t)py * S) * SW + (size_t)px * S;
        float3 c = zero3();
        float mask[SS ? SS * SS : 1];
#pragma unroll
        for (int sy = 0; sy < S; ++sy)
#pragma unroll
            for (int sx = 0; sx < S; ++sx) {
                float4 a = r.acol[base + (size_t)sy * SW + sx];
                c += f3of(a);
                if (SS) mask[sy * SS + sx] = a.w;
            }
        float inv = 1.f / (float)(S * S);
        c = inv * c;
        if (r.out_img) {
            r.out_img[pix * 3] = c.x;
            r.out_img[pix * 3 + 1] = c.y;
            r.out_img[pix * 3 + 2] = c.z;
        }
        if (r.ref) {
            const float* y = r.ref + pix * 3;
            float y0 = y[0], y1 = y[1], y2 = y[2];
            float g0 = 0.f, g1 = 0.f, g2 = 0.f;
            if (c.x != 0.f || c.y != 0.f || c.z != 0.f || y0 != 0.f || y1 != 0.f || y2 != 0.f) {
                float l0 = loss_term(r.loss_kind, c.x, y0, &g0), l1 = loss_term(r.loss_kind, c.y, y1, &g1),
                      l2 = loss_term(r.loss_kind, c.z, y2, &g2);
                sum.add(l0, l1, l2);
            }
            float k = r.loss_scale * inv;  // each sample carries 1 / s^2 of its pixel
#pragma unroll
            for (int sy = 0; sy < S; ++sy)
#pragma unroll
                for (int sx = 0; sx < S; ++sx) {
                    size_t q = base + (size_t)sy * SW + sx;
                    r.gprime[q] = make_float4(g0 * k, g1 * k, g2 * k, SS ? mask[sy * SS + sx] : r.acol[q].w);
                }
        }
    }
    if (!r.loss_acc) return;
    double s = sum.block(red);
    if (threadIdx.x == 0 && s != 0.0) atomicAdd(r.loss_acc, s * (double)r.loss_scale);
}

cudaError_t resolve_loss(const ResolveArgs& r, cudaStream_t st) {
    dim3 grid((unsigned)(((long long)r.H * r.W + 255) / 256), r.B);
    auto k = r.S == 2 ? k_resolve<2> : k_resolve<0>;
    k<<<grid, 256, 0, st>>>(r);
    count_launches(1);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ launchers
static dim3 pix_grid(const ShadeArgs& a) {
    int tx = (a.W + ADMS_TILE - 1) / ADMS_TILE, ty = (a.H + ADMS_TILE - 1) / ADMS_TILE;
    return dim3(tx * ty, a.B);
}
// the grid of band_pixel<threads>: 256 / threads blocks per tile
static dim3 band_grid(const ShadeArgs& a, int threads) {
    dim3 g = pix_grid(a);
    g.x *= 256 / threads;
    return g;
}

// grids of up to this many samples refine their bright pixels in the shading
// kernel itself (no list, no second launch)
#ifndef ADMS_INLINE_REFINE_PX
#define ADMS_INLINE_REFINE_PX (1 << 20)
#endif

cudaError_t shade_forward(const ShadeArgs& a, cudaStream_t st, int layers) {
    bool inline_refine = a.msaa <= 1 && (size_t)a.B * a.H * a.W <= ADMS_INLINE_REFINE_PX;
    bool list = a.refine && !inline_refine;
    if (list) {
        cudaError_t e = cudaMemsetAsync(a.refine, 0, sizeof(int), st);
        if (e) return e;
    }
    int share = share_of(a);
    if (a.msaa > 1) {
        int R = ADMS_MSAA_REGION;
        k_shade_fwd_msaa<<<dim3(((a.W + R - 1) / R) * ((a.H + R - 1) / R), a.B), 256, 0, st>>>(a);
    } else {
        auto k = inline_refine
                     ? (share == 1 ? k_shade_fwd<true, 1> : share == 2 ? k_shade_fwd<true, 2> : k_shade_fwd<true, 0>)
                     : (share == 1 ? k_shade_fwd<false, 1> : share == 2 ? k_shade_fwd<false, 2> : k_shade_fwd<false, 0>);
        dim3 grid = band_grid(a, ADMS_FWD_THREADS);
        grid.z = layers;
        k<<<grid, ADMS_FWD_THREADS, 0, st>>>(a);
    }
    count_launches(1);
    if (list) {
        // a few thousand pixels, a long dependent chain each: small blocks spread them over every
        // SM (128 blocks of 256 filled 30 SMs; the displaced mesh's shading 837 -> 822 us)
        k_shade_refine<<<608, 64, 0, st>>>(a);
        count_launches(1);
    }
    return cudaGetLastError();
}
// up to this many blocks (one view of 512x512), where a pass is bound by the host's launches;
// at 16384 blocks the counter costs what the launch does (49.4 us against 45.0 + 5.1)
#define ADMS_FINISH_BLOCKS 2048
cudaError_t aa_loss_forward(const ShadeArgs& a, cudaStream_t st, JobState* finish, float* out, bool* finished) {
    int rows = ADMS_AA_THREADS / 32;
    dim3 grid(((a.W + 31) / 32) * ((a.H + rows - 1) / rows), a.B);
    bool fin = finish && !a.peel && a.loss_acc && (long long)grid.x * grid.y <= ADMS_FINISH_BLOCKS;
    if (finished) *finished = fin;
    auto k = a.peel ? k_aa_loss<true, false> : fin ? k_aa_loss<false, true> : k_aa_loss<false, false>;
    k<<<grid, ADMS_AA_THREADS, 0, st>>>(a, finish, out);
    count_launches(1);
    return cudaGetLastError();
}
cudaError_t aa_loss_given(const ShadeArgs& a, cudaStream_t st) {
    int rows = ADMS_AA_THREADS / 32;
    dim3 grid(((a.W + 31) / 32) * ((a.H + rows - 1) / rows), a.B);
    k_aa_loss<false, false, true><<<grid, ADMS_AA_THREADS, 0, st>>>(a, nullptr, nullptr);
    count_launches(1);
    return cudaGetLastError();
}
cudaError_t shade_backward(const ShadeArgs& a, cudaStream_t st) {
    if (a.msaa > 1) {
        int R = ADMS_MSAA_REGION;
        k_shade_bwd_msaa<<<dim3(((a.W + R - 1) / R) * ((a.H + R - 1) / R), a.B), 256, 0, st>>>(a);
    } else {
        auto k = a.peel ? k_shade_bwd<true> : k_shade_bwd<false>;
        k<<<band_grid(a, ADMS_BWD_THREADS), ADMS_BWD_THREADS, 0, st>>>(a);
    }
    count_launches(1);
    return cudaGetLastError();
}

// in tiles (256 pixels, two blocks of the pixel kernels) per SM, as pixels_batched's blocks are
int batched_occupancy(int kind) {
    if (kind == 3) return raster_batch_occupancy();
    int n = 0;
    cudaError_t e = kind == 0   ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_pixels_batch<0>, 128, 0)
                    : kind == 1 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_pixels_batch<1>, 128, 0)
                                : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_pixels_batch<2>, 128, 0);
    return e == cudaSuccess && n > 1 ? n / 2 : 1;
}

cudaError_t pixels_batched(int kind, const ShadeArgs* args, const int* item_off, int n_jobs, const WorkItem* items,
                           int tw, int blocks, cudaStream_t st) {
    ShadeBatch P;
    for (int j0 = 0; j0 < n_jobs; j0 += ADMS_BATCH_JOBS) {
        int j1 = std::min(n_jobs, j0 + ADMS_BATCH_JOBS);
        int s0 = item_off[j0], n = item_off[j1] - s0;
        if (n <= 0) continue;
        memcpy(P.a, args + j0, sizeof(ShadeArgs) * (j1 - j0));
        int g = 2 * std::min(blocks, n);
        if (kind == 0) {
            k_refine_reset<<<1, ADMS_BATCH_JOBS, 0, st>>>(P, j1 - j0);
            k_pixels_batch<0><<<g, 128, 0, st>>>(P, items + s0, n, tw, j0);
            k_refine_batch<<<dim3(64, j1 - j0), 256, 0, st>>>(P);
            count_launches(2);
        }
        else if (kind == 1) k_pixels_batch<1><<<g, 128, 0, st>>>(P, items + s0, n, tw, j0);
        else k_pixels_batch<2><<<g, 128, 0, st>>>(P, items + s0, n, tw, j0);
        count_launches(1);
        cudaError_t e = cudaGetLastError();
        if (e) return e;
    }
    return cudaSuccess;
}

}  // namespace adms
