// Vertex transform, triangle setup, binning and tiled fixed-point rasterization
// with a packed depth|triangle-id z-buffer (Sec. 5.2: rasterization primitive).
//
// The visibility arithmetic is fixed bit for bit so that the keys are exact:
//   clip_r = ((M[r][0] x + M[r][1] y) + M[r][2] z) + M[r][3]   (float32, each op RN, no FMA)
//   sx = (clip.x / clip.w)(W/2) + W/2, sy = H/2 - (clip.y / clip.w)(H/2), X = rint(256 sx)
//   E_ab(S) = (X_b - X_a)(S_y - Y_a) - (Y_b - Y_a)(S_x - X_a) in int64 at S = (256 i + 128, 256 j + 128)
//   covered: every edge of the positively wound triangle has E > 0, or E = 0 on a top/left edge
//   d = (z0 + b1 (z1 - z0)) + b2 (z2 - z0), b1 = (float)E_20 / (float)A, b2 = (float)E_01 / (float)A
//   key = (float_bits(d) << 32) | triangle id, minimum per pixel.
#include "mesh.cuh"

namespace adms {

// m0 x + m1 y + m2 z + m3 (float inputs, double-float result)
__device__ __forceinline__ DF df_row(const float* m, float x, float y, float z) {
    DF p0 = df_two_prod(m[0], x), p1 = df_two_prod(m[1], y), p2 = df_two_prod(m[2], z);
    DF s = df_two_sum(p0.hi, p1.hi);
    float t = __fadd_rn(s.lo, __fadd_rn(p0.lo, p1.lo));
    DF u = df_two_sum(s.hi, p2.hi);
    t = __fadd_rn(t, __fadd_rn(u.lo, p2.lo));
    DF v = df_two_sum(u.hi, m[3]);
    t = __fadd_rn(t, v.lo);
    return df_fast_two_sum(v.hi, t);
}
// a / b
__device__ __forceinline__ DF df_div(DF a, DF b) {
    float q1 = __fdiv_rn(a.hi, b.hi);
    DF p = df_two_prod(q1, b.hi);
    // r = a - q1 b, the leading terms cancel exactly up to p.lo
    float r = __fsub_rn(__fadd_rn(__fsub_rn(__fsub_rn(a.hi, p.hi), p.lo), a.lo), __fmul_rn(q1, b.lo));
    return df_fast_two_sum(q1, __fdiv_rn(r, b.hi));
}
// c0 + s q (float c0, s; double-float q)
__device__ __forceinline__ DF df_affine(float c0, float s, DF q) {
    DF p = df_two_prod(q.hi, s);
    float e = __fmaf_rn(q.lo, s, p.lo);
    DF u = df_two_sum(c0, p.hi);
    return df_fast_two_sum(u.hi, __fadd_rn(u.lo, e));
}

// ---------------------------------------------------------------- transform
// vertex i (view-major) of a job
__device__ __forceinline__ void transform_vertex(const float* __restrict__ pos, int V,
                                                 const adms_view* __restrict__ views, int W, int H,
                                                 float4* __restrict__ clip, VtxS* __restrict__ vs,
                                                 float4* __restrict__ scr, int i) {
    int b = i / V, v = i - b * V;
    const float* M = views[b].mvp;
    float x = pos[3 * v], y = pos[3 * v + 1], z = pos[3 * v + 2];
    {
        // shading-side screen position to ~48 bits as a (hi, lo) float pair:
        // sx = (W/2) (cx / cw) + W/2, sy = H/2 - (H/2) (cy / cw) in double-float
        // arithmetic (float64 runs at a small fraction of the float32 rate here)
        DF cx = df_row(M, x, y, z), cy = df_row(M + 4, x, y, z), cw = df_row(M + 12, x, y, z);
        float hW = 0.5f * (float)W, hH = 0.5f * (float)H;
        DF sx = df_affine(hW, hW, df_div(cx, cw));
        DF sy = df_affine(hH, -hH, df_div(cy, cw));
        scr[i] = make_float4(sx.hi, sx.lo, sy.hi, sy.lo);
    }
    float c[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        float s = __fadd_rn(__fmul_rn(M[4 * r], x), __fmul_rn(M[4 * r + 1], y));
        s = __fadd_rn(s, __fmul_rn(M[4 * r + 2], z));
        c[r] = __fadd_rn(s, M[4 * r + 3]);
    }
    clip[i] = make_float4(c[0], c[1], c[2], c[3]);
    VtxS o;
    o.X = 0;
    o.Y = 0;
    o.z = 0.f;
    o.ok = 0;
    if (c[3] > 1e-6f) {
        float hW = 0.5f * (float)W, hH = 0.5f * (float)H;
        float sx = __fadd_rn(__fmul_rn(__fdiv_rn(c[0], c[3]), hW), hW);
        float sy = __fsub_rn(hH, __fmul_rn(__fdiv_rn(c[1], c[3]), hH));
        float fx = __fmul_rn(sx, 256.f), fy = __fmul_rn(sy, 256.f);
        if (fabsf(fx) <= 134217728.f && fabsf(fy) <= 134217728.f) {
            o.X = __float2int_rn(fx);
            o.Y = __float2int_rn(fy);
            o.z = __fadd_rn(__fmul_rn(__fdiv_rn(c[2], c[3]), 0.5f), 0.5f);
            o.ok = 1;
        }
    }
    vs[i] = o;
}

// A single job's views in pageable host memory come with the launch: the vertices are
// transformed from the parameters and block 0 writes them to the job's buffer for the kernels
// that follow (a pageable copy costs the host 9 us).
struct ViewSet {
    adms_view v[ADMS_PARAM_VIEWS];
    int n;
};
// The first launch of a raster pass: the first nb_vert blocks of a job transform its vertices,
// the rest set its keys to empty and clear the tile counts and whatever else of 4-byte words
// the pass needs at zero (four memset launches before).
#define ADMS_BEGIN_CLEARS (ADMS_PREP_CLEARS + 3)
struct BeginArgs {
    const float* pos;
    const adms_view* views;
    float4* clip;
    VtxS* vs;
    float4* scr;
    unsigned long long* keys;
    long long n_keys;
    ClearSeg z[ADMS_BEGIN_CLEARS];
    int V, B, W, H, nb_vert, nb_fill;
};
template <int N>
__device__ __forceinline__ void begin_body(const Pack<BeginArgs, N>& P, const ViewSet* vs) {
    const BeginArgs& A = P.a[N == 1 ? 0 : blockIdx.y];
    int blk = blockIdx.x;
    if (vs && blk == 0) {
        int* to = reinterpret_cast<int*>(const_cast<adms_view*>(A.views));
        const int* from = reinterpret_cast<const int*>(vs->v);
        for (int i = threadIdx.x; i < vs->n * (int)(sizeof(adms_view) / 4); i += 256) to[i] = from[i];
    }
    if (blk < A.nb_vert) {
        int i = blk * 256 + threadIdx.x;
        if (i < A.B * A.V) transform_vertex(A.pos, A.V, vs ? vs->v : A.views, A.W, A.H, A.clip, A.vs, A.scr, i);
        return;
    }
    blk -= A.nb_vert;
    if (blk >= A.nb_fill) return;
    long long t = (long long)blk * 256 + threadIdx.x, step = (long long)A.nb_fill * 256;
    if (reinterpret_cast<uintptr_t>(A.keys) & 15) {
        for (long long i = t; i < A.n_keys; i += step) A.keys[i] = ADMS_EMPTY_KEY;
    } else {
        ulonglong2 e = make_ulonglong2(ADMS_EMPTY_KEY, ADMS_EMPTY_KEY);
        for (long long i = t; i < A.n_keys / 2; i += step) reinterpret_cast<ulonglong2*>(A.keys)[i] = e;
        if (t == 0 && (A.n_keys & 1)) A.keys[A.n_keys - 1] = ADMS_EMPTY_KEY;
    }
#pragma unroll
    for (int k = 0; k < ADMS_BEGIN_CLEARS; ++k)
        for (long long i = t; i < A.z[k].n; i += step) A.z[k].p[i] = 0;
}
template <int N>
__global__ void __launch_bounds__(256) k_begin(const __grid_constant__ Pack<BeginArgs, N> P) {
    begin_body(P, nullptr);
}
__global__ void __launch_bounds__(256) k_begin_views(const __grid_constant__ Pack<BeginArgs, 1> P,
                                                     const __grid_constant__ ViewSet vs) {
    begin_body(P, &vs);
}

// ---------------------------------------------------------------- tile-list allocation
// Each tile's list segment [off, off + count) in the list buffer: a warp scans its 32
// tiles' counts by shuffles and reserves their segments together with one 64-bit
// atomicAdd on *total (zeroed by k_begin), so the segments lie in no particular
// order, as the entries inside a segment already do (the raster's per-pixel minimum
// does not depend on either). Offsets saturate at INT_MAX (the list-capacity check
// catches an overflow); *total ends exact. Many small blocks rather than one large
// scan block: a 1024-thread block does not fit on an SM beside a resident
// streamed-Adam block, which a pipelined step runs at the same time.
struct AllocArgs {
    const int* count;
    int n;
    int* off;
    unsigned long long* total;
};
template <int N>
__global__ void __launch_bounds__(256) k_list_alloc(const __grid_constant__ Pack<AllocArgs, N> P) {
    const AllocArgs& A = P.a[N == 1 ? 0 : blockIdx.y];
    const int n = A.n;
    int i = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
    long long c = i < n ? A.count[i] : 0;
    long long x = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    unsigned long long base = 0;
    if (lane == 31 && x > 0) base = atomicAdd(A.total, (unsigned long long)x);
    base = __shfl_sync(0xffffffffu, base, 31);
    if (i < n) A.off[i] = (int)min((long long)base + x - c, (long long)0x7fffffff);
}

// ---------------------------------------------------------------- edge functions
// Oriented edge functions of a triangle (s E_k, s the sign of its snapped area; edge 0 =
// 1->2, 1 = 2->0, 2 = 0->1): a_k = -s dy, b_k = s dx, value a_k (Sx - Xa) + b_k (Sy - Ya),
// covered where value >= thr_k for every k.
//
// "Near" triangles (snapped extents of at most ADMS_NEAR = 96 pixels a side) are evaluated
// in int32: at any sample within 16 pixels of the box |Sx - Xa|, |Sy - Ya| <= 112 * 256 =
// 28672 and |a|, |b| <= 24576, so |value| <= 2 * 28672 * 24576 < 2^31, and the area fits
// too; the values, and with them the keys, are those of the int64 form. It saves the wide
// multiplies, and above all the int64 -> float conversions of the depth: those run on the
// FP64 pipe at 1/64 rate (the tile raster held it 50% busy). Larger triangles keep int64.
#define ADMS_NEAR (96 * 256)

template <typename T>
struct Edges {
    T a[3], b[3], area;  // area: absolute
    int x[3], y[3];      // a point of each edge
    int thr[3];
    int sg;
    __device__ __forceinline__ T at(int k, int Sx, int Sy) const {
        return a[k] * (T)(Sx - x[k]) + b[k] * (T)(Sy - y[k]);
    }
};

template <typename T>
__device__ __forceinline__ Edges<T> make_edges(const int X[3], const int Y[3]) {
    Edges<T> e;
    T A = (T)(X[1] - X[0]) * (T)(Y[2] - Y[0]) - (T)(Y[1] - Y[0]) * (T)(X[2] - X[0]);
    e.sg = A > 0 ? 1 : -1;
    e.area = A > 0 ? A : -A;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        int i = (k + 1) % 3, j = (k + 2) % 3;
        int odx = e.sg * (X[j] - X[i]), ody = e.sg * (Y[j] - Y[i]);
        e.a[k] = (T)-ody;
        e.b[k] = (T)odx;
        e.x[k] = X[i];
        e.y[k] = Y[i];
        e.thr[k] = ((ody < 0) || (ody == 0 && odx > 0)) ? 0 : 1;
    }
    return e;
}

// Calls f(tile index) for the 16x16 tiles of the box in which the triangle may cover a
// sample: a tile goes when some edge function is below its threshold at the tile's sample
// where it is largest. The setup's counts and the fill's entries come from the same loop.
// (A box of one tile is taken as it is.) On billboards of ~60 pixels a third of the boxes'
// tiles go; their entries, records and tests with them.
template <typename T, typename F>
__device__ __forceinline__ void for_tiles(const Edges<T>& e, const TriBin& tb, int tiles_x, F&& f) {
    int tx0 = tb.bx0 / ADMS_TILE, tx1 = tb.bx1 / ADMS_TILE, ty0 = tb.by0 / ADMS_TILE, ty1 = tb.by1 / ADMS_TILE;
    if (tx0 == tx1 && ty0 == ty1) {
        f(ty0 * tiles_x + tx0);
        return;
    }
    constexpr int step = 256 * ADMS_TILE, last = 256 * (ADMS_TILE - 1);
    T row[3];
#pragma unroll
    for (int k = 0; k < 3; ++k)
        row[k] = e.at(k, step * tx0 + 128 + (e.a[k] > 0 ? last : 0), step * ty0 + 128 + (e.b[k] > 0 ? last : 0)) -
                 e.thr[k];
    for (int ty = ty0; ty <= ty1; ++ty) {
        T v[3] = {row[0], row[1], row[2]};
        for (int tx = tx0; tx <= tx1; ++tx) {
            if ((v[0] | v[1] | v[2]) >= 0) f(ty * tiles_x + tx);
#pragma unroll
            for (int k = 0; k < 3; ++k) v[k] += e.a[k] * (T)step;
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) row[k] += e.b[k] * (T)step;
    }
}

// Whether the lanes that walk their boxes together may all do so in int32. The 64-bit form finds the
// same tiles for near triangles too, and a warp of both kinds walks once instead of once per kind:
// 80 triangles in one view of 512x512 61.6 -> 48.8 us for the lists and 11.4 -> 8.5 for the setup,
// loss and gradients of 288 at 1024x1024 232 -> 209. (Without the edge tests: 43.8 and 4.3, but
// 7.5 us of raster instead of 6.2.)
__device__ __forceinline__ bool all_near(bool near) { return __all_sync(__activemask(), near); }

// depth key from the oriented edge values e1, e2 (b1 = s E_20 / A = e1 / |A|: the sign
// cancels exactly), or ADMS_EMPTY_KEY outside the depth range
__device__ __forceinline__ unsigned long long depth_key(float e1, float e2, float area, float z0, float dz1, float dz2,
                                                        int id) {
    float b1 = __fdiv_rn(e1, area), b2 = __fdiv_rn(e2, area);
    float d = __fadd_rn(__fadd_rn(z0, __fmul_rn(b1, dz1)), __fmul_rn(b2, dz2));
    if (!(d >= 0.f && d <= 1.f)) return ADMS_EMPTY_KEY;
    if (d == 0.f) d = 0.f;
    return ((unsigned long long)__float_as_uint(d) << 32) | (unsigned)id;
}

// A lower bound on the keys of a triangle with vertex depths z0, z1, z2 (its high word):
// the interpolated depth d = z0 + b1 (z1 - z0) + b2 (z2 - z0) (b1, b2 >= 0, b1 + b2 <= 1,
// each operation rounded once) is at least min z less a few units of rounding of
// the largest |z| (1e-6 x max(1, |z|) covers them with room), and a key needs d >= 0.
__device__ __forceinline__ unsigned key_floor(float z0, float z1, float z2) {
    float zmn = fminf(z0, fminf(z1, z2));
    float zmx = fmaxf(fabsf(z0), fmaxf(fabsf(z1), fabsf(z2)));
    return __float_as_uint(fmaxf(zmn - 1e-6f * fmaxf(1.f, zmx), 0.f));
}

// A near triangle as the per-sample loops read it, at sample offsets (x, y) from an origin:
//   p = (E0', A0, B0, C), q = (E1', A1, B1, -), r = (|area|, z0, dz1, dz2)
// E_k' = value - thr_k at the origin, A, B the steps per pixel, C the sum of the three E'
// (the edge functions add up to |area| everywhere): covered where e0, e1 and C - e0 - e1
// are all non-negative.
__device__ __forceinline__ int near_third(int c, int e0, int e1) {  // c - e0 - e1 (fits; the partial sum may wrap)
    return (int)((unsigned)c - (unsigned)e0 - (unsigned)e1);
}
__device__ __forceinline__ void near_pack(const Edges<int>& e, int Sx, int Sy, int4& p, int4& q) {
    int E0 = e.at(0, Sx, Sy) - e.thr[0], E1 = e.at(1, Sx, Sy) - e.thr[1];
    p = make_int4(E0, 256 * e.a[0], 256 * e.b[0], e.area - e.thr[0] - e.thr[1] - e.thr[2]);
    q = make_int4(E1, 256 * e.a[1], 256 * e.b[1], 0);
}

// ---------------------------------------------------------------- setup, small triangles, tile counts
// One thread per (view, triangle). Near triangles whose pixel box holds at most small_px
// samples are rasterized here directly, one 64-bit atomicMin per covered sample (the
// minimum does not depend on the order); the others get a record and are counted into the
// tiles they may touch.
//
// The direct raster flattens the warp's triangles: their packed edge functions go to shared
// memory, their sample counts are scanned, and the lanes take the boxes' samples 32 at a
// time whatever triangle they belong to. The triangle of a lane is the number of boxes that
// begin at or before its sample, from one mask of the beginnings in the batch (__reduce_or
// and a population count), so that every lane of every batch but the last has a sample. (A
// thread per triangle of up to 16 samples and the whole warp per larger one left half of
// the lanes idle and moved 30 words a triangle by shuffles: 3.41 -> 1.63 ms for 600k leaf
// quads under 8 views of 512x512, 0.40 -> 0.20 ms for 62k displaced triangles under 16 of
// 1024x1024, 12.4 -> 6.6 us for 5000 triangles under 8 of 512x512.)
//
// ZF (in.zfilter): the stored key is read before the depth is computed, for dense clouds (a
// foliage canopy puts ~160 fragments on each sample). zlo is a lower bound on every key of
// the triangle, so above the stored key the sample is done; else the key goes in only if it
// is below the stored one. The stored key only ever decreases, so a read that lags behind
// other threads' updates can only let an unneeded atomicMin through. Without it (closed
// surfaces, about two fragments per sample) the read would only add a round trip.
//
// From ADMS_ROUNDS_MIN triangles x views on, a single filtered job goes in four rounds of an eighth,
// an eighth, a quarter and a half of the triangles, between them a pass over the tiles' stored
// depths, by which the later rounds drop what is hidden. One pass against rounds, whole renders in
// us (leaves of half-side 0.015 - 0.03, 120 fragments on a sample at 2^22 under 8 views of 512x512):
//   triangles x views     2^18         2^20         2^21         2^22         2^23          2^24
//   8 of 512x512       222 : 429    386 : 461    593 : 545    992 : 738   1795 : 1132   3374 : 1874
//   4 of 1024x1024     512 : 746   1198 : 1259  2075 : 1831  3817 : 2675  7183 : 3912  14110 : 6120
//   4 of 256x256        93 : 161    168 : 203    260 : 272    459 : 409    838 : 682    1591 : 1225
// The line is where every size of image gains. (Leaves so small that five fragments land on a sample,
// which is not what the filter is for, lose 11% at 2^22 and 4% at 2^24.) Jobs of a batched call take
// one pass: their launches are shared, and a candidate is far smaller than a reference.
#define ADMS_ROUNDS_MIN (1 << 22)
// resident blocks per SM: 4 (5: 1% faster on the displaced mesh, 3% slower on 11k billboards),
// 5 with the key read, whose latency the extra warps hide (the canopy's preparation 1.15 ->
// 1.06 ms; 6: 1.07, 3: 1.29)
constexpr int setup_blocks(bool zf) { return zf ? 5 : 4; }
struct DirectTri {  // 80 bytes: 16-byte reads of consecutive slots touch distinct banks
    int4 p, q, r;
    int id;
    unsigned inv_w;      // 2^32 / box width, rounded up (0: width 1)
    long long origin;    // key index of the box's first sample
    int start, width;    // first of its samples among the warp's
    unsigned zlo;
    int thr;             // thr_1 | thr_2 << 1
};
struct SetupArgs {
    const int* tri;
    const VtxS* vs;
    TriRec* rec;
    TriBin* bin;
    int8_t* asign;
    int* tile_count;
    unsigned long long* keys;
    int F, V, B, W, H, tiles_x, tiles_y, small_px, zfilter;
    // a round of a dense cloud (ZF): the triangles of groups c0 .. c0 + cw - 1 of every eight
    // groups of eight, per_view threads per view; hiz: per tile the largest stored depth after
    // the rounds before (null: none)
    int c0, cw, per_view;
    const unsigned* hiz;
};

// Whether every sample of the box shows something nearer than zlo: hiz[tile] is the largest
// depth word stored in the tile some time ago, and stored keys only decrease.
__device__ __forceinline__ bool box_hidden(const SetupArgs& A, int b, int bx0, int bx1, int by0, int by1,
                                           unsigned zlo) {
    const unsigned* h = A.hiz + (size_t)b * A.tiles_x * A.tiles_y;
    for (int ty = by0 / ADMS_TILE; ty <= by1 / ADMS_TILE; ++ty)
        for (int tx = bx0 / ADMS_TILE; tx <= bx1 / ADMS_TILE; ++tx)
            if (zlo <= h[ty * A.tiles_x + tx]) return false;
    return true;
}
// the largest depth word of each 16x16 tile's stored keys (all ones where a sample is empty),
// a warp per tile
__global__ void __launch_bounds__(256) k_tile_depth(const unsigned long long* __restrict__ keys, int n_tiles, int tiles_x,
                                                    int tiles_y, int W, int H, unsigned* __restrict__ hiz) {
    int t = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (t >= n_tiles) return;
    int per_view = tiles_x * tiles_y, b = t / per_view, r = t % per_view;
    int x = (r % tiles_x) * ADMS_TILE + (lane & 15), y0 = (r / tiles_x) * ADMS_TILE + (lane >> 4);
    unsigned m = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        int y = y0 + 2 * k;
        if (x < W && y < H) m = max(m, (unsigned)(__ldcg(keys + ((size_t)b * H + y) * W + x) >> 32));
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0) hiz[t] = m;
}
// ZF: compiled with the key read; taken where the job asks for it
template <bool ZF, int N>
__global__ void __launch_bounds__(256, setup_blocks(ZF)) k_setup(const __grid_constant__ Pack<SetupArgs, N> P) {
    __shared__ DirectTri slots[8][32];
    const SetupArgs& A = P.a[N == 1 ? 0 : blockIdx.y];
    const int* __restrict__ tri = A.tri;
    const VtxS* __restrict__ vs = A.vs;
    unsigned long long* __restrict__ keys = A.keys;
    const int F = A.F, V = A.V, B = A.B, W = A.W, H = A.H, tiles_x = A.tiles_x, tiles_y = A.tiles_y;
    const bool zf = ZF && (N == 1 || A.zfilter);
    const unsigned full = 0xffffffffu;
    const int per_view = ZF && N == 1 ? A.per_view : F;
    if ((long long)blockIdx.x * blockDim.x >= (long long)B * per_view) return;
    int i = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
    int npx = 0;  // samples of this lane's direct triangle
    DirectTri t;
    int b = i / per_view, f = i - b * per_view;
    if (ZF && N == 1) f = 8 * ((f / (8 * A.cw)) * 8 + A.c0 + (f / 8) % A.cw) + (f & 7);
    if (b < B && f < F) {
        i = b * F + f;
        const VtxS* vb = vs + (size_t)b * V;
        VtxS v0 = vb[tri[3 * f]], v1 = vb[tri[3 * f + 1]], v2 = vb[tri[3 * f + 2]];
        TriBin tb;
        tb.bx0 = tb.by0 = 1;
        tb.bx1 = tb.by1 = 0;
        int8_t sgn = 0;
        if (v0.ok && v1.ok && v2.ok) {
            int X[3] = {v0.X, v1.X, v2.X}, Y[3] = {v0.Y, v1.Y, v2.Y};
            long long area = (long long)(X[1] - X[0]) * (Y[2] - Y[0]) - (long long)(Y[1] - Y[0]) * (X[2] - X[0]);
            if (area != 0) {
                sgn = area > 0 ? 1 : -1;
                int minX = min(X[0], min(X[1], X[2])), maxX = max(X[0], max(X[1], X[2]));
                int minY = min(Y[0], min(Y[1], Y[2])), maxY = max(Y[0], max(Y[1], Y[2]));
                // samples at 256 i + 128; |X| <= 2^27, so the shifts round down without overflow
                int ilo = max((minX + 127) >> 8, 0), ihi = min((maxX - 128) >> 8, W - 1);
                int jlo = max((minY + 127) >> 8, 0), jhi = min((maxY - 128) >> 8, H - 1);
                if (ilo <= ihi && jlo <= jhi) {
                    bool near = maxX - minX <= ADMS_NEAR && maxY - minY <= ADMS_NEAR;
                    float dz1 = __fsub_rn(v1.z, v0.z), dz2 = __fsub_rn(v2.z, v0.z);
                    int w = ihi - ilo + 1, n = w * (jhi - jlo + 1);  // at most 2^28
                    unsigned zlo = zf ? key_floor(v0.z, v1.z, v2.z) : 0u;
                    if (ZF && N == 1 && A.hiz && box_hidden(A, b, ilo, ihi, jlo, jhi, zlo)) {
                        // nothing of it can be seen: no record, no samples
                    } else if (near && n <= A.small_px) {
                        npx = n;
                        Edges<int> e = make_edges<int>(X, Y);
                        near_pack(e, 256 * ilo + 128, 256 * jlo + 128, t.p, t.q);
                        t.r = make_int4(__float_as_int(__int2float_rn(e.area)), __float_as_int(v0.z),
                                        __float_as_int(dz1), __float_as_int(dz2));
                        t.id = f;
                        t.inv_w = w > 1 ? 0xffffffffu / (unsigned)w + 1u : 0u;
                        t.origin = ((long long)b * H + jlo) * W + ilo;
                        t.width = w;
                        t.zlo = zlo;
                        t.thr = e.thr[1] | (e.thr[2] << 1);
                    } else {
                        tb.bx0 = (short)ilo;
                        tb.bx1 = (short)ihi;
                        tb.by0 = (short)jlo;
                        tb.by1 = (short)jhi;
                        TriRec r;
                        r.X[0] = X[0], r.X[1] = X[1], r.X[2] = X[2];
                        r.Y[0] = Y[0], r.Y[1] = Y[1], r.Y[2] = Y[2];
                        r.z0 = v0.z;
                        r.dz1 = dz1;
                        r.dz2 = dz2;
                        r.near = near;
                        r.box = tb;
                        A.rec[i] = r;
                        int* tc = A.tile_count + (size_t)b * tiles_x * tiles_y;
                        auto count = [&](int k) { atomicAdd(tc + k, 1); };
                        if (all_near(near)) for_tiles(make_edges<int>(X, Y), tb, tiles_x, count);
                        else for_tiles(make_edges<long long>(X, Y), tb, tiles_x, count);
                    }
                }
            }
        }
        A.asign[i] = sgn;
        A.bin[i] = tb;
    }
    unsigned direct = __ballot_sync(full, npx > 0);
    if (!direct) return;
    int upto = npx;  // inclusive scan of the sample counts
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(full, upto, o);
        if (lane >= o) upto += y;
    }
    int total = __shfl_sync(full, upto, 31);
    t.start = upto - npx;
    DirectTri* ws = slots[threadIdx.x >> 5];
    if (npx > 0) ws[__popc(direct & ((1u << lane) - 1u))] = t;
    __syncwarp();
    int before = 0;  // boxes that begin before the batch
    for (int base = 0; base < total; base += 32) {
        int at = t.start - base;
        unsigned begins = __reduce_or_sync(full, npx > 0 && at >= 0 && at < 32 ? 1u << at : 0u);
        const DirectTri& d = ws[before + __popc(begins & (full >> (31 - lane))) - 1];
        before += __popc(begins);
        if (base + lane >= total) break;
        int k = base + lane - d.start, w = d.width;
        int y = w > 1 ? (int)__umulhi((unsigned)k, d.inv_w) : k, x = k - y * w;
        int4 p = d.p, q = d.q;
        int e0 = p.x + p.y * x + p.z * y, e1 = q.x + q.y * x + q.z * y, e2 = near_third(p.w, e0, e1);
        if ((e0 | e1 | e2) < 0) continue;
        unsigned long long* a = keys + d.origin + (long long)y * W + x;
        unsigned long long cur = ADMS_EMPTY_KEY;
        if (zf) {
            cur = __ldcg(a);
            if (d.zlo > (unsigned)(cur >> 32)) continue;
        }
        int4 r = d.r;
        unsigned long long key =
            depth_key(__int2float_rn(e1 + (d.thr & 1)), __int2float_rn(e2 + (d.thr >> 1)), __int_as_float(r.x),
                      __int_as_float(r.y), __int_as_float(r.z), __int_as_float(r.w), d.id);
        if (zf ? key < cur : key != ADMS_EMPTY_KEY) atomicMin(a, key);
    }
}

// ---------------------------------------------------------------- tile lists
// The entries of the tile lists: list[0 .. capacity), then the second half of the records'
// allocation (a record takes 48 of the 96 bytes per triangle and view that its buffer
// holds), so that a list of 20 entries per triangle fits where 8 did.
struct TileLists {
    const int* list;
    const int* ext;
    long long capacity, total;
    __device__ __forceinline__ int get(long long p) const { return p < capacity ? list[p] : ext[p - capacity]; }
    __device__ __forceinline__ void set(long long p, int v) const {
        if (p < total) const_cast<int*>(p < capacity ? list + p : ext + (p - capacity))[0] = v;
    }
};

// Per (view, triangle), after the scan of the tile counts: the triangle's
// silhouette-edge mask, then its entries in the tile lists. Bit e of
// silmask[b][f] is set when edge e of triangle f is a silhouette edge in view b:
// no neighbour across it, or a neighbour whose snapped area has another sign.
//
// FRAME: the launch also forms the vertex frame and the Laplacian where they are due (new
// positions), in its first blocks: both need only the positions and take about as long as the
// lists, so that neither costs a launch, a second stream or a join before the shading.
struct FillArgs {
    const TriRec* rec;
    const TriBin* bin;
    const int* tile_off;
    int* tile_cursor;
    TileLists lists;
    const int* adj;
    const int8_t* asign;
    uint8_t* silmask;
    int F, B, tiles_x, tiles_y;
    int nb_frame, nb_lap, nb_fill;
    FrameArgs f;
    LapArgs l;
};
// 6 blocks per SM without the frames: most threads of a large mesh only look their box up
template <bool FRAME, int N>
__global__ void __launch_bounds__(256, FRAME ? 5 : 6) k_bin_fill(const __grid_constant__ Pack<FillArgs, N> P) {
    const FillArgs& A = P.a[N == 1 ? 0 : blockIdx.y];
    int blk = blockIdx.x;
    if (FRAME) {
        __shared__ double red[8];
        if (blk < A.nb_frame) {
            int v = blk * 256 + threadIdx.x;
            if (v < A.f.V) frame_vertex(A.f, v);
            return;
        }
        blk -= A.nb_frame;
        if (blk < A.nb_lap) {
            lap_vertex(A.l, blk * 256 + threadIdx.x, red);
            return;
        }
        blk -= A.nb_lap;
    }
    int i = blk * 256 + threadIdx.x;
    if (i >= A.B * A.F) return;
    int b = i / A.F, f = i - b * A.F;
    {
        const int8_t* sg = A.asign + (size_t)b * A.F;
        int sf = sg[f];
        uint8_t msk = 0;
        if (sf != 0) {
#pragma unroll
            for (int e = 0; e < 3; ++e) {
                int nb = A.adj[3 * f + e];
                if (nb < 0 || sg[nb] != sf) msk |= (uint8_t)(1u << e);
            }
        }
        A.silmask[i] = msk;
    }
    TriBin tb = A.bin[i];
    if (tb.bx0 > tb.bx1) return;
    size_t tbase = (size_t)b * A.tiles_x * A.tiles_y;
    TriRec r = A.rec[i];
    auto fill = [&](int k) {
        A.lists.set((long long)A.tile_off[tbase + k] + atomicAdd(A.tile_cursor + tbase + k, 1), f);
    };
    if (all_near(r.near)) for_tiles(make_edges<int>(r.X, r.Y), tb, A.tiles_x, fill);
    else for_tiles(make_edges<long long>(r.X, r.Y), tb, A.tiles_x, fill);
}

// ---------------------------------------------------------------- tiled raster
// One block per (view, 16x16 tile), one pixel per thread, a warp per 8x4 pixels. The tile's
// triangles are staged through shared memory in chunks of 256: a thread takes one record,
// forms its edge functions at the tile and the mask of the 8x4 blocks that it may cover
// (box, and for near triangles the edges); the masks become one word per block and staging
// warp by ballots, and each warp walks the set bits of its block. The minimum does not
// depend on the order. Issue-bound (66%), with the FP64 pipe half busy on int64 -> float
// conversions and 17 of 32 lanes active in 16x2 strips, at 69.9 us for 8 views of 512x512 of
// 5000 triangles before; 47.5 us now (58% issue, 22 lanes, 28.6 M against 50.4 M warp
// instructions). The k-buffer form on 11k billboards with 8 layers: 6.06 ms (its tile lists
// had overflowed) -> 0.41 ms, 0.24 with the classes below.
//
// Each pixel starts from the key left by the small-triangle pass. A tile whose list did
// not fit scans every binned triangle of its view instead.
// BUCKETS > 1 (the k-buffer): the walk takes each staging warp's triangles front to back in
// four classes of their depth floor, and a lane whose buffer is full of nearer fragments passes
// a triangle over by the floor alone. Of 70 fragments a sample of 11k billboards, in list order
// about 25 entered a buffer of 8 and every one was divided out (313 M warp instructions a launch,
// 77% issue): two passes over 8 views of 512x512 817 -> 470 us. The keys do not depend on the order.
template <int BUCKETS>
struct TileSmem {
    int4 p[256], q[256], r[256];  // near_pack at the tile's first sample; q.w: flags
    int4 s[256];                  // large triangles; .w: the depth floor (BUCKETS > 1)
    int id[256];
    unsigned mask[BUCKETS][8][8];  // [class][8x4 block][staging warp]
};
template <int KB>
constexpr int depth_buckets = KB > 1 ? 4 : 1;
#define ADMS_LARGE 8  // q.w: bits 0-2 thresholds, bit 3 large

// minimum key / the KB smallest keys in kb[0] < kb[1] < ... (the keys of one sample are
// distinct, each triangle giving at most one): a fragment sinks into place and the largest
// falls out
template <int KB>
struct KeySink {
    unsigned long long kb[KB];
    __device__ __forceinline__ void take(unsigned long long key) {
        if (key >= kb[KB - 1]) return;
#pragma unroll
        for (int i = 0; i < KB; ++i) {
            unsigned long long lo = key < kb[i] ? key : kb[i];
            key = key < kb[i] ? kb[i] : key;
            kb[i] = lo;
        }
    }
};

// per-view arrays of one raster launch
struct TileArgs {
    const TriRec* rec;
    const TriBin* bin;
    int F, W, H, tiles_x, tiles_y;
    const int* tile_off;
    const int* tile_count;
    TileLists lists;
    unsigned long long* overflow_ctr;
};

// the pixel of a thread in its tile
__device__ __forceinline__ int tile_x(int tid) { return ((tid >> 5) & 1) * 8 + (tid & 7); }
__device__ __forceinline__ int tile_y(int tid) { return (tid >> 6) * 4 + ((tid >> 3) & 3); }

template <int KB>
__device__ __forceinline__ void raster_tile_walk(const TileArgs& A, int b, int tile, long long off, int cnt,
                                                 TileSmem<depth_buckets<KB>>& sm, KeySink<KB>& sink) {
    constexpr int BUCKETS = depth_buckets<KB>;
    int tx = tile % A.tiles_x, ty = tile / A.tiles_x;
    int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int lx = tile_x(tid), ly = tile_y(tid);
    const TriRec* rb = A.rec + (size_t)b * A.F;
    const TriBin* bb = A.bin + (size_t)b * A.F;
    bool overflow = cnt > 0 && off + cnt > A.lists.total;
    int n = overflow ? A.F : cnt;
    if (overflow && tid == 0) atomicAdd(A.overflow_ctr, 1ull);
    int ox = tx * ADMS_TILE, oy = ty * ADMS_TILE;
    int S0x = 256 * ox + 128, S0y = 256 * oy + 128;
    for (int c0 = 0; c0 < n; c0 += 256) {
        int m = min(256, n - c0);
        __syncthreads();
        unsigned mask = 0, zlo = 0;
        if (tid < m) {
            int f = overflow ? c0 + tid : A.lists.get(off + c0 + tid);
            TriBin tb = overflow ? bb[f] : rb[f].box;
            // the box in the tile's pixels; empty boxes (not binned) and other tiles' fall out
            int x0 = max(tb.bx0 - ox, 0), x1 = min(tb.bx1 - ox, ADMS_TILE - 1);
            int y0 = max(tb.by0 - oy, 0), y1 = min(tb.by1 - oy, ADMS_TILE - 1);
            if (x0 <= x1 && y0 <= y1) {
                TriRec t = rb[f];
                unsigned cols = (x0 < 8 ? 1u : 0u) | (x1 >= 8 ? 2u : 0u);
                for (int w = y0 >> 2; w <= (y1 >> 2); ++w) mask |= cols << (2 * w);
                float area;
                if (t.near) {
                    Edges<int> e = make_edges<int>(t.X, t.Y);
                    int4 p, q;
                    near_pack(e, S0x, S0y, p, q);
                    q.w = e.thr[0] | (e.thr[1] << 1) | (e.thr[2] << 2);
                    area = __int2float_rn(e.area);
                    sm.p[tid] = p;
                    sm.q[tid] = q;
                    // the blocks where every edge function reaches its threshold at its largest sample
                    int ax[3] = {p.y, q.y, -(p.y + q.y)}, by[3] = {p.z, q.z, -(p.z + q.z)};
                    int v[3] = {p.x, q.x, near_third(p.w, p.x, q.x)};
#pragma unroll
                    for (int k = 0; k < 3; ++k) v[k] += max(7 * ax[k], 0) + max(3 * by[k], 0);
#pragma unroll
                    for (int w = 0; w < 8; ++w) {
                        int x = 8 * (w & 1), y = 4 * (w >> 1);
                        int e0 = v[0] + ax[0] * x + by[0] * y, e1 = v[1] + ax[1] * x + by[1] * y,
                            e2 = v[2] + ax[2] * x + by[2] * y;
                        if ((e0 | e1 | e2) < 0) mask &= ~(1u << w);
                    }
                } else {
                    Edges<long long> e = make_edges<long long>(t.X, t.Y);
                    long long E[3];
#pragma unroll
                    for (int k = 0; k < 3; ++k) E[k] = e.at(k, S0x, S0y);
                    area = __ll2float_rn(e.area);
                    sm.p[tid] = make_int4((int)E[0], (int)(E[0] >> 32), (int)E[1], (int)(E[1] >> 32));
                    sm.q[tid] = make_int4((int)E[2], (int)(E[2] >> 32), (int)e.a[0],
                                          ADMS_LARGE | e.thr[0] | (e.thr[1] << 1) | (e.thr[2] << 2));
                    sm.s[tid] = make_int4((int)e.b[0], (int)e.a[1], (int)e.b[1], 0);
                }
                sm.r[tid] = make_int4(__float_as_int(area), __float_as_int(t.z0), __float_as_int(t.dz1),
                                      __float_as_int(t.dz2));
                sm.id[tid] = f;
                if (BUCKETS > 1) {
                    zlo = key_floor(t.z0, t.z0 + t.dz1, t.z0 + t.dz2);
                    sm.s[tid].w = (int)zlo;
                }
            }
        }
        int bucket = 0;
        if (BUCKETS > 1) {
            unsigned near = __reduce_min_sync(0xffffffffu, mask ? zlo : 0xffffffffu);
            unsigned far = __reduce_max_sync(0xffffffffu, mask ? zlo : 0u);
            unsigned step = (far - near) / BUCKETS + 1;  // (no triangle in the warp: no bit is set below)
            bucket = (zlo >= near + step) + (zlo >= near + 2 * step) + (zlo >= near + 3 * step);
        }
#pragma unroll
        for (int k = 0; k < 8 * BUCKETS; ++k) {
            unsigned mw = __ballot_sync(0xffffffffu, (mask >> (k & 7)) & (bucket == k >> 3 ? 1u : 0u));
            if (lane == k) sm.mask[k >> 3][k & 7][warp] = mw;
        }
        __syncthreads();
        for (int k = 0; k < BUCKETS; ++k) {
            for (int g = 0; g < m; g += 32) {
                for (unsigned mm = sm.mask[k][warp][g >> 5]; mm; mm &= mm - 1) {
                    int j = g + __ffs(mm) - 1;
                    if (BUCKETS > 1 && (unsigned)sm.s[j].w > (unsigned)(sink.kb[KB - 1] >> 32)) continue;
                    int4 p = sm.p[j], q = sm.q[j];
                    float f1, f2;
                    if (!(q.w & ADMS_LARGE)) {
                        int e0 = p.x + p.y * lx + p.z * ly, e1 = q.x + q.y * lx + q.z * ly,
                            e2 = near_third(p.w, e0, e1);
                        if ((e0 | e1 | e2) < 0) continue;
                        f1 = __int2float_rn(e1 + ((q.w >> 1) & 1));
                        f2 = __int2float_rn(e2 + (q.w >> 2));
                    } else {
                        int4 s = sm.s[j];
                        long long E0 = ((long long)p.y << 32) | (unsigned)p.x, E1 = ((long long)p.w << 32) | (unsigned)p.z;
                        long long E2 = ((long long)q.y << 32) | (unsigned)q.x;
                        int dx = 256 * lx, dy = 256 * ly;
                        long long e0 = E0 + (long long)q.z * dx + (long long)s.x * dy;
                        long long e1 = E1 + (long long)s.y * dx + (long long)s.z * dy;
                        // a_2 = -(a_0 + a_1): the edges of a closed triangle
                        long long e2 = E2 - ((long long)q.z + s.y) * dx - ((long long)s.x + s.z) * dy;
                        if (e0 < (q.w & 1) || e1 < ((q.w >> 1) & 1) || e2 < ((q.w >> 2) & 1)) continue;
                        f1 = __ll2float_rn(e1);
                        f2 = __ll2float_rn(e2);
                    }
                    int4 r = sm.r[j];
                    sink.take(depth_key(f1, f2, __int_as_float(r.x), __int_as_float(r.y), __int_as_float(r.z),
                                        __int_as_float(r.w), sm.id[j]));
                }
            }
        }
    }
}

// one 16x16 tile of one view: the minimum key per pixel
__device__ __forceinline__ void raster_tile_body(const TileArgs& A, unsigned long long* __restrict__ keys, int b,
                                                 int tile, TileSmem<1>& sm) {
    size_t t = (size_t)b * A.tiles_x * A.tiles_y + tile;
    int cnt = A.tile_count[t];
    if (cnt == 0) return;  // no binned triangle: the small-triangle pass left the final keys
    long long off = A.tile_off[t];
    int px = (tile % A.tiles_x) * ADMS_TILE + tile_x(threadIdx.x), py = (tile / A.tiles_x) * ADMS_TILE + tile_y(threadIdx.x);
    bool inside = px < A.W && py < A.H;
    size_t pix = ((size_t)b * A.H + py) * A.W + px;
    KeySink<1> sink;
    sink.kb[0] = inside ? keys[pix] : ADMS_EMPTY_KEY;
    raster_tile_walk<1>(A, b, tile, off, cnt, sm, sink);
    if (inside) keys[pix] = sink.kb[0];
}

__global__ void __launch_bounds__(256) k_raster(const TileArgs A, unsigned long long* __restrict__ keys) {
    __shared__ TileSmem<1> sm;
    raster_tile_body(A, keys, blockIdx.y, blockIdx.x, sm);
}

// the same for a mostly empty grid: block k takes tiles k, k + gridDim.x, ... of all views, up
// to 32, reads their counts together and skips the empty ones
__global__ void __launch_bounds__(256) k_raster_sparse(const TileArgs A, unsigned long long* __restrict__ keys,
                                                       int n_tiles) {
    __shared__ TileSmem<1> sm;
    long long t = blockIdx.x + (long long)(threadIdx.x & 31) * gridDim.x;
    unsigned live = __ballot_sync(0xffffffffu, t < n_tiles && A.tile_count[t] > 0);
    int per_view = A.tiles_x * A.tiles_y;
    for (; live; live &= live - 1) {
        int k = blockIdx.x + (__ffs(live) - 1) * gridDim.x;
        raster_tile_body(A, keys, k / per_view, k % per_view, sm);
    }
}

// Depth peeling in one pass (Sec. 5.2): per sample the L nearest fragments,
// front to back, which are exactly the layers that L peeling passes with a
// two-sided test on the packed depth|id key would find (the keys of a sample are
// distinct). The walk of k_raster with a KB-entry k-buffer per thread in registers
// (KB >= L); every triangle must be binned (no small-triangle pass). keys holds
// L slices of [B][H][W].
template <int KB>
__global__ void __launch_bounds__(256) k_raster_kbuf(const TileArgs A, unsigned long long* __restrict__ keys, int L,
                                                     int B) {
    __shared__ TileSmem<depth_buckets<KB>> sm;
    int b = blockIdx.y, tile = blockIdx.x;
    int px = (tile % A.tiles_x) * ADMS_TILE + tile_x(threadIdx.x), py = (tile / A.tiles_x) * ADMS_TILE + tile_y(threadIdx.x);
    KeySink<KB> sink;
#pragma unroll
    for (int i = 0; i < KB; ++i) sink.kb[i] = ADMS_EMPTY_KEY;
    size_t t = (size_t)b * A.tiles_x * A.tiles_y + tile;
    raster_tile_walk<KB>(A, b, tile, A.tile_off[t], A.tile_count[t], sm, sink);
    if (px >= A.W || py >= A.H) return;
    size_t pix = ((size_t)b * A.H + py) * A.W + px, layer = (size_t)B * A.H * A.W;
#pragma unroll
    for (int i = 0; i < KB; ++i)
        if (i < L) keys[pix + (size_t)i * layer] = sink.kb[i];
}

static TileLists tile_lists(const TriRec* rec, const int* list, long long capacity, long long records) {
    return TileLists{list, reinterpret_cast<const int*>(rec + records), capacity, tile_list_room(capacity, records)};
}

struct RasterBatch {
    TileArgs a[ADMS_BATCH_JOBS];
    unsigned long long* keys[ADMS_BATCH_JOBS];
};
// persistent: block k takes items k, k + gridDim.x, ... (the items are equal
// 16x16 tiles, so a static stride balances them without a shared counter); the
// jobs' arguments are kernel parameters (up to ADMS_BATCH_JOBS per launch)
__global__ void __launch_bounds__(256) k_raster_batch(const __grid_constant__ RasterBatch P,
                                                      const WorkItem* __restrict__ items, int n, int job0) {
    __shared__ TileSmem<1> sm;
    for (int it = blockIdx.x; it < n; it += gridDim.x) {
        WorkItem w = items[it];
        const TileArgs& A = P.a[w.job - job0];
        int tile = (w.y0 / ADMS_TILE) * A.tiles_x + w.x0 / ADMS_TILE;
        raster_tile_body(A, P.keys[w.job - job0], w.view, tile, sm);
    }
}

int raster_batch_occupancy() {
    int n = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_raster_batch, 256, 0);
    return e == cudaSuccess && n > 0 ? n : 1;
}

cudaError_t raster_tiles_batched(const RasterJob* args, const int* item_off, int n_jobs, const WorkItem* items,
                                 int blocks, cudaStream_t st) {
    RasterBatch P;
    for (int j0 = 0; j0 < n_jobs; j0 += ADMS_BATCH_JOBS) {
        int j1 = std::min(n_jobs, j0 + ADMS_BATCH_JOBS);
        int s0 = item_off[j0], n = item_off[j1] - s0;
        if (n <= 0) continue;
        for (int j = j0; j < j1; ++j) {
            const RasterJob& r = args[j];
            P.a[j - j0] = TileArgs{r.rec, r.bin, r.F, r.W, r.H, r.tiles_x, r.tiles_y, r.tile_off, r.tile_count,
                                   tile_lists(r.rec, r.list, r.capacity, r.records), r.overflow_ctr};
            P.keys[j - j0] = r.keys;
        }
        k_raster_batch<<<std::min(blocks, n), 256, 0, st>>>(P, items + s0, n, j0);
        count_launches(1);
        cudaError_t e = cudaGetLastError();
        if (e) return e;
    }
    return cudaSuccess;
}

// ---------------------------------------------------------------- host launchers
cudaError_t raster_prepare(const PrepJob* jobs, int n, cudaStream_t st) {
    // a single job's arguments stay on the stack: the per-stage and no-allocation calls allocate
    // nothing, and have nobody to catch what a failed allocation throws
    struct Args {
        BeginArgs begin{};
        SetupArgs setup{};
        AllocArgs alloc{};
        FillArgs fill{};
    } one;
    std::vector<BeginArgs> begins(n > 1 ? n : 0);
    std::vector<SetupArgs> setups(n > 1 ? n : 0);
    std::vector<AllocArgs> allocs(n > 1 ? n : 0);
    std::vector<FillArgs> fills(n > 1 ? n : 0);
    BeginArgs* begin = n > 1 ? begins.data() : &one.begin;
    SetupArgs* setup = n > 1 ? setups.data() : &one.setup;
    AllocArgs* alloc = n > 1 ? allocs.data() : &one.alloc;
    FillArgs* fill = n > 1 ? fills.data() : &one.fill;
    bool zf = false, frame = false;
    for (int k = 0; k < n; ++k) {
        const RasterIn& in = jobs[k].in;
        RasterScratch& s = *jobs[k].s;
        int tiles_x = (in.W + ADMS_TILE - 1) / ADMS_TILE, tiles_y = (in.H + ADMS_TILE - 1) / ADMS_TILE;
        int ntiles = in.B * tiles_x * tiles_y;
        BeginArgs& g = begin[k];
        g.pos = in.pos;
        g.views = in.views;
        g.clip = s.clip;
        g.vs = s.vs;
        g.scr = s.scr;
        g.V = in.V;
        g.B = in.B;
        g.W = in.W;
        g.H = in.H;
        g.keys = in.keys;
        g.n_keys = in.keys && in.small_px > 0 ? (long long)in.B * in.H * in.W : 0;
        int z = 0;
        long long words = 0;
        auto clear = [&](void* p, size_t bytes) {
            g.z[z++] = ClearSeg{static_cast<int*>(p), (long long)(bytes / 4)};
            words += (long long)(bytes / 4);
        };
        clear(s.tile_count, sizeof(int) * (size_t)ntiles);
        clear(s.tile_cursor, sizeof(int) * (size_t)ntiles);
        if (s.total_pairs) clear(s.total_pairs, sizeof(long long));
        for (int c = 0; c < jobs[k].n_clear; ++c) clear(jobs[k].clear[c], jobs[k].clear_bytes[c]);
        g.nb_vert = (in.B * in.V + 255) / 256;
        // 16 stores of 16 bytes per thread for the keys, 16 of 4 for the rest
        g.nb_fill = (int)std::max<long long>(1, std::max(g.n_keys / 2, words) / (256 * 16));
        setup[k] = SetupArgs{in.tri, s.vs, s.rec, s.bin, s.asign, s.tile_count, in.keys, in.F, in.V, in.B, in.W, in.H,
                             tiles_x, tiles_y, in.small_px, in.zfilter && in.small_px > ADMS_SMALL_PX, 0, 8, in.F, nullptr};
        zf = zf || setup[k].zfilter;
        alloc[k] = AllocArgs{s.tile_count, ntiles, s.tile_off, reinterpret_cast<unsigned long long*>(s.total_pairs)};
        FillArgs& f = fill[k];
        f.rec = s.rec;
        f.bin = s.bin;
        f.tile_off = s.tile_off;
        f.tile_cursor = s.tile_cursor;
        f.lists = tile_lists(s.rec, s.list, s.list_capacity, (long long)in.B * in.F);
        f.adj = in.adj;
        f.asign = s.asign;
        f.silmask = s.silmask;
        f.F = in.F;
        f.B = in.B;
        f.tiles_x = tiles_x;
        f.tiles_y = tiles_y;
        f.nb_fill = (in.B * in.F + 255) / 256;
        if (jobs[k].frame) {
            f.f = jobs[k].f;
            f.nb_frame = (f.f.V + 255) / 256;
        }
        if (jobs[k].lap) {
            f.l = jobs[k].l;
            f.nb_lap = (f.l.V + 255) / 256;
        }
        frame = frame || f.nb_frame || f.nb_lap;
    }
    constexpr int M = ADMS_BATCH_JOBS;
    cudaError_t e = cudaSuccess;
    if (n == 1 && jobs[0].host_views) {
        Pack<BeginArgs, 1> p;
        p.a[0] = begin[0];
        ViewSet vs;
        vs.n = jobs[0].in.B;
        if (vs.n > ADMS_PARAM_VIEWS) return cudaErrorInvalidValue;
        memcpy(vs.v, jobs[0].host_views, sizeof(adms_view) * vs.n);
        k_begin_views<<<begin[0].nb_vert + begin[0].nb_fill, 256, 0, st>>>(p, vs);
        count_launches(1);
        e = cudaGetLastError();
    } else {
        e = launch_packed(begin, n, 256, st, k_begin<1>, k_begin<M>,
                          [](const BeginArgs& a) { return a.nb_vert + a.nb_fill; });
    }
    auto tri_blocks = [](const SetupArgs& a) { return (a.B * a.F + 255) / 256; };
    if (!e && zf && n == 1 && (long long)setup[0].B * setup[0].F >= ADMS_ROUNDS_MIN) {
        // tile_off holds the tiles' depths until the list allocation writes it
        SetupArgs a = setup[0];
        int nt = a.B * a.tiles_x * a.tiles_y;
        unsigned* hiz = reinterpret_cast<unsigned*>(jobs[0].s->tile_off);
        const int first[5] = {0, 1, 2, 4, 8};
        for (int r = 0; r < 4 && !e; ++r) {
            a.c0 = first[r];
            a.cw = first[r + 1] - first[r];
            a.per_view = (a.F + 63) / 64 * 8 * a.cw;
            a.hiz = r ? hiz : nullptr;
            e = launch_packed(&a, 1, 256, st, k_setup<true, 1>, k_setup<true, M>,
                              [](const SetupArgs& q) { return (int)(((long long)q.B * q.per_view + 255) / 256); });
            if (e || r == 3) break;
            k_tile_depth<<<(nt + 7) / 8, 256, 0, st>>>(a.keys, nt, a.tiles_x, a.tiles_y, a.W, a.H, hiz);
            count_launches(1);
            e = cudaGetLastError();
        }
    } else if (!e) {
        e = zf ? launch_packed(setup, n, 256, st, k_setup<true, 1>, k_setup<true, M>, tri_blocks)
               : launch_packed(setup, n, 256, st, k_setup<false, 1>, k_setup<false, M>, tri_blocks);
    }
    if (!e)
        e = launch_packed(alloc, n, 256, st, k_list_alloc<1>, k_list_alloc<M>,
                          [](const AllocArgs& a) { return (a.n + 255) / 256; });
    auto fill_blocks = [](const FillArgs& a) { return a.nb_frame + a.nb_lap + a.nb_fill; };
    if (!e)
        e = frame ? launch_packed(fill, n, 256, st, k_bin_fill<true, 1>, k_bin_fill<true, M>, fill_blocks)
                  : launch_packed(fill, n, 256, st, k_bin_fill<false, 1>, k_bin_fill<false, M>, fill_blocks);
    return e;
}

cudaError_t raster_prepare(const RasterIn& in, RasterScratch& s, cudaStream_t st) {
    PrepJob j;
    j.in = in;
    j.s = &s;
    return raster_prepare(&j, 1, st);
}

#define ADMS_RASTER_GRID 2048
static TileArgs tile_args(const RasterIn& in, const RasterScratch& s) {
    return TileArgs{s.rec, s.bin, in.F, in.W, in.H, (in.W + ADMS_TILE - 1) / ADMS_TILE,
                    (in.H + ADMS_TILE - 1) / ADMS_TILE, s.tile_off, s.tile_count,
                    tile_lists(s.rec, s.list, s.list_capacity, (long long)in.B * in.F), s.overflow_ctr};
}

cudaError_t raster_tiles(const RasterIn& in, RasterScratch& s, cudaStream_t st) {
    TileArgs a = tile_args(in, s);
    // A job that rasterizes most of its triangles directly has mostly empty tiles: a grid of
    // ADMS_RASTER_GRID blocks looks them over (16 views of 1024x1024 of a displaced mesh, two
    // passes: 83 -> 16 us; 600k leaf quads 65 -> 36). Where the tiles hold work the hardware's
    // block scheduling balances better (plain mesh, a block per tile 41.2 us, two tiles 45.4,
    // four 48.0).
    int n = a.tiles_x * a.tiles_y * in.B;
    int per = in.small_px > ADMS_SMALL_PX ? std::min(n / ADMS_RASTER_GRID, 32) : 1;
    if (per > 1) k_raster_sparse<<<(n + per - 1) / per, 256, 0, st>>>(a, in.keys, n);
    else k_raster<<<dim3(a.tiles_x * a.tiles_y, in.B), 256, 0, st>>>(a, in.keys);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t raster_tiles_peeled(const RasterIn& in, RasterScratch& s, int L, cudaStream_t st) {
    if (L < 1 || L > 16) return cudaErrorInvalidValue;
    TileArgs a = tile_args(in, s);
    dim3 grid(a.tiles_x * a.tiles_y, in.B);
#define ADMS_KBUF_LAUNCH(KB) k_raster_kbuf<KB><<<grid, 256, 0, st>>>(a, in.keys, L, in.B)
    if (L <= 2) ADMS_KBUF_LAUNCH(2);
    else if (L <= 4) ADMS_KBUF_LAUNCH(4);
    else if (L <= 8) ADMS_KBUF_LAUNCH(8);
    else ADMS_KBUF_LAUNCH(16);
#undef ADMS_KBUF_LAUNCH
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t raster_views(const RasterIn& in, RasterScratch& s, cudaStream_t st) {
    cudaError_t e = raster_prepare(in, s, st);
    if (e) return e;
    return raster_tiles(in, s, st);
}

}  // namespace adms
