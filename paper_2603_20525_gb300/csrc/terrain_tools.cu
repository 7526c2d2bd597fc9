// terrain_tools.cu - terrain preprocessing for the planner (arxiv 2603.20525):
//
//   * Level of detail (Sec. V-B).  Each model gets its own Gaussian-smoothed
//     copy of the heightmap (0.3 m standard deviation for the SRB model, the
//     length scale of a wheel; 1.5 m for the planar model, that of the
//     chassis).  The two-dimensional Gaussian is a product of one-dimensional
//     ones, so it runs as a row pass and a column pass, each through a
//     shared-memory tile with its halo; the map is extended by its nearest
//     border node and the kernel is cut at four standard deviations.
//   * Costmap of the distance constraints (Sec. IV-C, IV-D).  At every node
//     the signed distance to each obstacle or path-boundary perimeter is turned
//     into the normalised quadratic soft-constraint cost rate and summed over
//     the perimeters, so that the rollout only interpolates it.  Four nodes per
//     thread; each 32 x 32 tile streams the edges of the perimeters that can
//     cost anything in it through shared memory in chunks.
#include <cuda_runtime.h>
#include <math_constants.h>

#include <stdint.h>

#include "fastmath.cuh"
#include "terrain_tools.cuh"

namespace atp {

namespace {

constexpr int kRowThreads = 256;  // row-pass CTA
// Outputs per thread: 4 row outputs (of two rows) below this radius and 8 from
// it on, where the wider window loads fewer values per output; 8 column
// outputs (of two columns), in CTAs of 64 columns below it and of 32 columns
// and twice the rows from it on, whose halo is then the smaller part of the
// tile.  16 column outputs gained nothing (84 registers).  2048^2 nodes, both
// passes: 31.2 -> 26.4 us at 12 cells, 73.9 -> 61.5 us at 60, 197 -> 162 us at
// 200 against one row or column per thread without the packing.
constexpr int kLodWideMinR = 16;

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

// Normalised weights w[k], k = 0..2r, of exp(-(k - r)^2 / (2 s^2)), each twice
// for the packed FMAs, made by every CTA the same way: the terms, then their
// sum in a fixed order (per thread a strided run, then a fixed shuffle tree
// and a fixed pass over the warps), so every CTA holds the same bits.  Needs
// blockDim.x * blockDim.y a multiple of 32 and at most 1024 threads.
__device__ void gauss_weights_cta(float2 *w, int r, float inv2s2)
{
    __shared__ float s_part[32];
    __shared__ float s_total;
    const int n = 2 * r + 1;
    const int t = threadIdx.y * blockDim.x + threadIdx.x;
    const int nt = blockDim.x * blockDim.y;
    float part = 0.f;
    for (int k = t; k < n; k += nt) {
        const float d = (float)(k - r);
        const float e = expf(-(d * d) * inv2s2);
        w[k].x = e;
        part += e;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    if ((t & 31) == 0) s_part[t >> 5] = part;
    __syncthreads();
    if (t == 0) {
        float z = 0.f;
        for (int i = 0; i < nt / 32; ++i) z += s_part[i];
        s_total = z;
    }
    __syncthreads();
    const float z = s_total;
    for (int k = t; k < n; k += nt) {
        const float v = w[k].x / z;
        w[k] = make_float2(v, v);
    }
    __syncthreads();
}

// The same weights for 2r + 1 <= 32, made by the CTA's first warp alone: one
// term per lane and the lanes' sum through the same shuffle tree, every lane
// dividing by lane 0's total.  The CTA-wide form adds only the other warps'
// zero sums to that total, so the bits are the same.  The other warps go
// straight on to their tile loads, and the caller's next barrier publishes
// the weights.
__device__ __forceinline__ void gauss_weights_warp(float2 *w, int r, float inv2s2)
{
    const int t = threadIdx.y * blockDim.x + threadIdx.x;
    if (t >= 32) return;
    const int n = 2 * r + 1;
    float e = 0.f;
    if (t < n) {
        const float d = (float)(t - r);
        e = expf(-(d * d) * inv2s2);
    }
    float z = e;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
    z = __shfl_sync(0xffffffffu, z, 0);
    if (t < n) w[t] = make_float2(e / z, e / z);
}

// The weights of a pass: the first warp alone for the narrow windows (r below
// kLodWideMinR, so 2r + 1 <= 31), the whole CTA otherwise.
static_assert(2 * (kLodWideMinR - 1) + 1 <= 32, "the narrow windows' weights fit one warp");
template <bool NARROW>
__device__ __forceinline__ void gauss_weights(float2 *w, int r, float inv2s2)
{
    if (NARROW)
        gauss_weights_warp(w, r, inv2s2);
    else
        gauss_weights_cta(w, r, inv2s2);
}

// acc[q] = sum over taps k = first .. last-1, in order, of w[k] v(k + q),
// two outputs packed in each float2, from a window of OUT + 4 positions that
// four loads refill every four taps.  The window's slots rotate through an
// unrolled run of groups, so nothing moves.  load(x) gives positions x .. x + 3
// (x a multiple of 4).
template <int OUT, class Load>
__device__ __forceinline__ void convolve(const float2 *w, int first, int last, float2 (&acc)[OUT], const Load &load)
{
    constexpr int kWin = OUT + 4, kRun = OUT == 8 ? 6 : kWin / 4;
    float2 v[kWin];
#pragma unroll
    for (int q = 0; q < OUT; ++q) acc[q] = make_float2(0.f, 0.f);
#pragma unroll
    for (int x = 0; x < kWin; x += 4) load(x, v[x], v[x + 1], v[x + 2], v[x + 3]);
    const int groups = (last + 3) / 4;
    for (int g0 = 0; g0 < groups; g0 += kRun) {
#pragma unroll
        for (int u = 0; u < kRun; ++u) {
            const int g = g0 + u;
            if (g < groups) {
                const bool whole = 4 * g >= first && 4 * g + 4 <= last;
                const float4 wa = ((const float4 *)w)[2 * g], wb = ((const float4 *)w)[2 * g + 1];
                const float2 wg[4] = {make_float2(wa.x, wa.y), make_float2(wa.z, wa.w), make_float2(wb.x, wb.y),
                                      make_float2(wb.z, wb.w)};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    if (whole || (4 * g + e >= first && 4 * g + e < last)) {
                        const float2 wk = wg[e];
#pragma unroll
                        for (int q = 0; q < OUT; ++q) acc[q] = fma2(wk, v[(4 * u + e + q) % kWin], acc[q]);
                    }
                }
                constexpr int kNext = kWin;
                load(4 * g + kNext, v[(4 * u) % kWin], v[(4 * u + 1) % kWin], v[(4 * u + 2) % kWin],
                     v[(4 * u + 3) % kWin]);
            }
        }
    }
}

// out[j][i] = sum_k w[k] in[j][clamp(i + k - r)], each sum over k in order, for
// two rows: the tile holds their values side by side, so that one packed FMA
// serves both (the passes are bound by instruction issue, not by the FMA
// pipe).  Thread t makes outputs OUT t .. OUT t + OUT - 1 of the CTA's 256 OUT.
// VEC: rows are 16-byte aligned, the tile starts at a multiple of four columns
// (`shift` columns before the first tap) and is filled by 16-byte loads.  Every
// OUT positions of the tile are padded by two, so that a warp's 16-byte loads
// fall on distinct banks.
template <int OUT, bool VEC>
__global__ void __launch_bounds__(kRowThreads) lod_rows_kernel(LodParams p)
{
    constexpr int kRowTile = kRowThreads * OUT;
    const auto at = [](int x) { return x / OUT * (OUT + 2) + x % OUT; };
    extern __shared__ __align__(16) float2 sm2[];
    const int n = 2 * p.r + 1;
    const int shift = VEC ? (4 - (p.r & 3)) & 3 : 0;
    float2 *w = sm2;                                        // shift + n, padded to 8
    float2 *tile = sm2 + ((n + 11) & ~7);                   // kRowTile + 2r + 16
    gauss_weights<OUT == 4>(w + shift, p.r, p.inv2s2);
    const int j = 2 * blockIdx.y, j1 = min(j + 1, p.ny - 1);
    const int i0 = blockIdx.x * kRowTile, s0 = i0 - p.r - shift;
    const float *row0 = p.in + (size_t)j * p.nx, *row1 = p.in + (size_t)j1 * p.nx;
    const int n_tile = kRowTile + 2 * p.r + 16;
    if (VEC) {
        for (int t = threadIdx.x; t < n_tile / 4; t += kRowThreads) {
            const int x = s0 + 4 * t;
            float4 a, b;
            if (x >= 0 && x + 3 < p.nx) {
                a = __ldg((const float4 *)(row0 + x));
                b = __ldg((const float4 *)(row1 + x));
            } else {
                const int x0 = clampi(x, 0, p.nx - 1), x1 = clampi(x + 1, 0, p.nx - 1);
                const int x2 = clampi(x + 2, 0, p.nx - 1), x3 = clampi(x + 3, 0, p.nx - 1);
                a = make_float4(__ldg(row0 + x0), __ldg(row0 + x1), __ldg(row0 + x2), __ldg(row0 + x3));
                b = make_float4(__ldg(row1 + x0), __ldg(row1 + x1), __ldg(row1 + x2), __ldg(row1 + x3));
            }
            float4 *t4 = (float4 *)(tile + at(4 * t));
            t4[0] = make_float4(a.x, b.x, a.y, b.y);
            t4[1] = make_float4(a.z, b.z, a.w, b.w);
        }
        for (int t = (n_tile & ~3) + threadIdx.x; t < n_tile; t += kRowThreads) {
            const int x = clampi(s0 + t, 0, p.nx - 1);
            tile[at(t)] = make_float2(__ldg(row0 + x), __ldg(row1 + x));
        }
    } else {
        for (int t = threadIdx.x; t < n_tile; t += kRowThreads) {
            const int x = clampi(s0 + t, 0, p.nx - 1);
            tile[at(t)] = make_float2(__ldg(row0 + x), __ldg(row1 + x));
        }
    }
    __syncthreads();
    const int ib = i0 + OUT * threadIdx.x;
    if (ib >= p.nx) return;
    const float2 *mine = tile + (OUT + 2) * threadIdx.x;
    float2 acc[OUT];
    convolve<OUT>(w, shift, shift + n, acc, [&](int x, float2 &a, float2 &b, float2 &c, float2 &d) {
        const float4 *t4 = (const float4 *)(mine + at(x));
        const float4 u = t4[0], v = t4[1];
        a = make_float2(u.x, u.y);
        b = make_float2(u.z, u.w);
        c = make_float2(v.x, v.y);
        d = make_float2(v.z, v.w);
    });
    float *o0 = p.out + (size_t)j * p.nx + ib, *o1 = p.out + (size_t)j1 * p.nx + ib;
    if (VEC) {                                              // nx is a multiple of 4, so whole float4
#pragma unroll
        for (int q = 0; q < OUT; q += 4) {
            if (ib + q < p.nx) {
                *(float4 *)(o0 + q) = make_float4(acc[q].x, acc[q + 1].x, acc[q + 2].x, acc[q + 3].x);
                if (j1 > j) *(float4 *)(o1 + q) = make_float4(acc[q].y, acc[q + 1].y, acc[q + 2].y, acc[q + 3].y);
            }
        }
    } else {
#pragma unroll
        for (int q = 0; q < OUT; ++q) {
            if (ib + q < p.nx) {
                o0[q] = acc[q].x;
                if (j1 > j) o1[q] = acc[q].y;
            }
        }
    }
}

// out[j][i] = sum_k w[k] in[clamp(j + k - r)][i], each sum over k in order; a
// CTA of CX x 256/CX threads covers 2 CX columns and 256/CX OUT rows, thread
// (x, y) rows OUT y .. OUT y + OUT - 1 of columns 2x and 2x + 1, packed.  VEC:
// the map's column pairs are 8-byte aligned.
template <int OUT, int CX, bool VEC, bool NARROW>
__global__ void __launch_bounds__(256) lod_cols_kernel(LodParams p)
{
    constexpr int kColTile = 256 / CX * OUT;
    extern __shared__ __align__(16) float2 sm2[];
    const int n = 2 * p.r + 1;
    float2 *w = sm2;                                        // n, padded to a multiple of 32
    float2 *tile = sm2 + ((n + 31) & ~31);                  // [kColTile + 2r + 8][CX]
    gauss_weights<NARROW>(w, p.r, p.inv2s2);
    const int i = blockIdx.x * (2 * CX) + 2 * threadIdx.x;
    const int j0 = blockIdx.y * kColTile;
    const int ia = min(i, p.nx - 1), ib = min(i + 1, p.nx - 1);
    const int n_rows = kColTile + 2 * p.r + 8;
    for (int t = threadIdx.y; t < n_rows; t += 256 / CX) {
        const float *row = p.in + (size_t)clampi(j0 - p.r + t, 0, p.ny - 1) * p.nx;
        tile[t * CX + threadIdx.x] = VEC ? __ldg((const float2 *)(row + min(i, p.nx - 2)))
                                         : make_float2(__ldg(row + ia), __ldg(row + ib));
    }
    __syncthreads();
    const int jb = OUT * threadIdx.y;        // first of this thread's rows in the tile
    if (i >= p.nx || j0 + jb >= p.ny) return;
    const float2 *col = tile + jb * CX + threadIdx.x;
    float2 acc[OUT];
    convolve<OUT>(w, 0, n, acc, [&](int x, float2 &a, float2 &b, float2 &c, float2 &d) {
        a = col[x * CX];
        b = col[x * CX + CX];
        c = col[x * CX + 2 * CX];
        d = col[x * CX + 3 * CX];
    });
#pragma unroll
    for (int q = 0; q < OUT; ++q) {
        const int j = j0 + jb + q;
        if (j >= p.ny) break;
        float *o = p.out + (size_t)j * p.nx + i;
        if (VEC) {
            *(float2 *)o = acc[q];
        } else {
            o[0] = acc[q].x;
            if (i + 1 < p.nx) o[1] = acc[q].y;
        }
    }
}

size_t rows_smem(int r, int out)
{
    return sizeof(float2) * (size_t)(((2 * r + 1 + 11) & ~7) + (kRowThreads * out + 2 * r + 16 + out) / out * (out + 2));
}
size_t cols_smem(int r, int out, int cx)
{
    return sizeof(float2) * (size_t)(((2 * r + 1 + 31) & ~31) + (256 / cx * out + 2 * r + 8) * cx);
}

template <int ROW_OUT, bool VEC>
cudaError_t lod_rows(const LodParams &p, cudaStream_t stream)
{
    const size_t smem = rows_smem(p.r, ROW_OUT);
    const cudaError_t e = cudaFuncSetAttribute(lod_rows_kernel<ROW_OUT, VEC>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)rows_smem(kLodMaxRadius, ROW_OUT));
    if (e != cudaSuccess) return e;
    const int tile = kRowThreads * ROW_OUT;
    const dim3 grid((unsigned)((p.nx + tile - 1) / tile), (unsigned)((p.ny + 1) / 2));
    lod_rows_kernel<ROW_OUT, VEC><<<grid, kRowThreads, smem, stream>>>(p);
    return cudaGetLastError();
}

template <int OUT, int CX, bool VEC, bool NARROW>
cudaError_t lod_cols(const LodParams &p, cudaStream_t stream)
{
    constexpr size_t kMaxSmem = 226 * 1024;       // less the static arrays
    const size_t smem = cols_smem(p.r, OUT, CX);
    const cudaError_t e = cudaFuncSetAttribute(lod_cols_kernel<OUT, CX, VEC, NARROW>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem);
    if (e != cudaSuccess) return e;
    const int rows = 256 / CX * OUT;
    const dim3 grid((unsigned)((p.nx + 2 * CX - 1) / (2 * CX)), (unsigned)((p.ny + rows - 1) / rows));
    lod_cols_kernel<OUT, CX, VEC, NARROW><<<grid, dim3(CX, 256 / CX), smem, stream>>>(p);
    return cudaGetLastError();
}

template <bool VEC>
cudaError_t lod_cols_by_radius(const LodParams &p, cudaStream_t stream)
{
    if (p.r < kLodWideMinR) return lod_cols<8, 32, VEC, true>(p, stream);
    return lod_cols<8, 16, VEC, false>(p, stream);
}

}  // namespace

cudaError_t launch_lod_smooth(const float *in, float *tmp, float *out, int nx, int ny, int r,
                              float inv2s2, cudaStream_t stream)
{
    if (r < 0 || r > kLodMaxRadius) return cudaErrorInvalidValue;
    LodParams p;
    p.nx = nx;
    p.ny = ny;
    p.r = r;
    p.inv2s2 = inv2s2;
    p.in = in;
    p.out = tmp;
    const bool vec_rows = nx % 4 == 0 && ((uintptr_t)in | (uintptr_t)tmp) % 16 == 0;
    cudaError_t e;
    if (r < kLodWideMinR)
        e = vec_rows ? lod_rows<4, true>(p, stream) : lod_rows<4, false>(p, stream);
    else
        e = vec_rows ? lod_rows<8, true>(p, stream) : lod_rows<8, false>(p, stream);
    if (e != cudaSuccess) return e;
    p.in = tmp;
    p.out = out;
    const bool vec_cols = nx % 2 == 0 && ((uintptr_t)tmp | (uintptr_t)out) % 8 == 0;
    return vec_cols ? lod_cols_by_radius<true>(p, stream) : lod_cols_by_radius<false>(p, stream);
}

// ---------------------------------------------------------------------------
// Costmap.  Coordinates are taken relative to the terrain origin (in FP64 once
// per vertex and node, then FP32), so that the FP32 distance arithmetic works
// on metres from the map corner rather than on large world coordinates.

namespace {

constexpr int kTile = 32;         // nodes per side of a CTA's tile
constexpr int kRows = 4;          // nodes per thread, 8 rows apart
constexpr int kChunk = 256;       // edges staged per pass, one per thread
// the tile's perimeter scan takes one thread of the 32 x 8 CTA per perimeter
static_assert(kCostmapMaxPolys <= 256, "one costmap thread per perimeter");

// Edge v of perimeter q in the costmap's coordinates: metres from the map
// corner, FP64 once per vertex, then FP32.
__device__ __forceinline__ CostmapEdge make_edge(const CostmapParams &p, int v, int q)
{
    const int u = v + 1 < p.start[q + 1] ? v + 1 : p.start[q];
    const float ax = (float)(p.xy[2 * v] - p.x0), ay = (float)(p.xy[2 * v + 1] - p.y0);
    const float bx = (float)(p.xy[2 * u] - p.x0), by = (float)(p.xy[2 * u + 1] - p.y0);
    const float ex = bx - ax, ey = by - ay;
    const float l2 = fmaf(ex, ex, ey * ey);
    CostmapEdge e;
    e.a = make_float4(ax, ay, ex, ey);
    e.b = make_float4(bx, by, l2, __int_as_float(q));
    return e;
}

// Whether nothing can be said of where an edge costs anything: a vertex at
// infinity, a NaN, or coordinates so large that the rounding of the distance
// and of the inside test (a few parts in 2^24 of them) is no longer small
// against `reach`.  Its perimeter is never left out of a tile.  Edges on the
// map pass: `reach` is at least 1e-5 of its side.
__device__ __forceinline__ bool unbounded(float4 a, float4 b, float reach)
{
    return !((fabsf(a.x) + fabsf(a.y)) + (fabsf(b.x) + fabsf(b.y)) < 524288.f * reach);
}

// One warp per perimeter: its edges, where they are kept, and its bounding box
// grown by `reach` (the whole plane where an edge is unbounded).
__global__ void __launch_bounds__(32) costmap_edges_kernel(const __grid_constant__ CostmapParams p, float reach)
{
    const int q = blockIdx.x, v0 = p.start[q], v1 = p.start[q + 1];
    float x0 = CUDART_INF_F, y0 = CUDART_INF_F, x1 = -CUDART_INF_F, y1 = -CUDART_INF_F;
    bool whole = false;
    for (int v = v0 + (int)threadIdx.x; v < v1; v += 32) {
        const CostmapEdge e = make_edge(p, v, q);
        if (p.edge) p.edge[v] = e;
        whole = whole || unbounded(e.a, e.b, reach);
        x0 = fminf(x0, e.a.x);
        y0 = fminf(y0, e.a.y);
        x1 = fmaxf(x1, e.a.x);
        y1 = fmaxf(y1, e.a.y);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        x0 = fminf(x0, __shfl_xor_sync(0xffffffffu, x0, o));
        y0 = fminf(y0, __shfl_xor_sync(0xffffffffu, y0, o));
        x1 = fmaxf(x1, __shfl_xor_sync(0xffffffffu, x1, o));
        y1 = fmaxf(y1, __shfl_xor_sync(0xffffffffu, y1, o));
    }
    whole = __any_sync(0xffffffffu, whole);
    if (threadIdx.x == 0)
        p.box[q] = whole ? make_float4(-CUDART_INF_F, -CUDART_INF_F, CUDART_INF_F, CUDART_INF_F)
                         : make_float4(x0 - reach, y0 - reach, x1 + reach, y1 + reach);
}

// off[k] <= v < off[k + 1]
__device__ __forceinline__ int perimeter_of(int v, const int *off, int n)
{
    int lo = 0, hi = n;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (off[mid] <= v) lo = mid;
        else hi = mid;
    }
    return lo;
}

// Even-odd rule with a ray towards +x, for the edge from (a.x, a.y) along
// (a.z, a.w) to (b.x, b.y).
__device__ __forceinline__ bool crosses(float4 a, float4 b, float px, float py)
{
    if ((a.y > py) == (b.y > py)) return false;
    return px < fmaf((py - a.y) / (b.y - a.y), a.z, a.x);
}

// A CTA of 32 x 8 threads makes a tile of 32 x 32 nodes, four per thread.  It
// first finds the perimeters that can cost anything in the tile: without the
// signed distances, an obstacle whose grown box misses the tile adds exactly
// nothing, and neither does a path boundary that holds the tile with every edge
// farther than `reach` (the edges are tested by all threads at once).  The
// edges of the others go through shared memory, in their order.
__global__ void __launch_bounds__(256) costmap_kernel(const __grid_constant__ CostmapParams p, float reach)
{
    __shared__ float4 s_a[kChunk], s_b[kChunk];
    __shared__ int s_id[kCostmapMaxPolys];        // the tile's perimeters, in order
    __shared__ int s_off[kCostmapMaxPolys + 1];   // prefix of their vertex counts
    __shared__ int s_near[kCostmapMaxPolys];      // path boundaries: 2 for a near edge, bit 0 inside
    __shared__ int s_wn[8], s_wv[8];
    __shared__ float s_x[kTile], s_y[kTile];
    const int t = threadIdx.y * 32 + threadIdx.x;
    const bool all = p.sdist != nullptr;
    // node coordinates, FP64 once per row and column of the tile
    if (t < kTile) s_x[t] = (float)((double)(blockIdx.x * kTile + t) * p.cell);
    else if (t < 2 * kTile) s_y[t - kTile] = (float)((double)(blockIdx.y * kTile + t - kTile) * p.cell);
    if (t < p.n_poly) s_near[t] = 0;
    __syncthreads();
    const float tx0 = s_x[0], tx1 = s_x[kTile - 1], ty0 = s_y[0], ty1 = s_y[kTile - 1];
    if (!all && p.n_path > 0) {
        const float mx = s_x[kTile / 2], my = s_y[kTile / 2];
        for (int v = t; v < p.n_vert; v += 256) {
            int q;
            float4 a, b;
            if (p.edge) {
                b = __ldg(&p.edge[v].b);
                q = __float_as_int(b.w);
                if (p.kind[q] != 1) continue;
                a = __ldg(&p.edge[v].a);
            } else {
                q = perimeter_of(v, p.start, p.n_poly);
                if (p.kind[q] != 1) continue;
                const CostmapEdge e = make_edge(p, v, q);
                a = e.a;
                b = e.b;
            }
            const bool near = unbounded(a, b, reach) ||
                              !(fmaxf(a.x, b.x) + reach < tx0 || fminf(a.x, b.x) - reach > tx1 ||
                                fmaxf(a.y, b.y) + reach < ty0 || fminf(a.y, b.y) - reach > ty1);
            if (near) atomicOr(&s_near[q], 2);
            if (crosses(a, b, mx, my)) atomicXor(&s_near[q], 1);
        }
        __syncthreads();
    }
    // the perimeters that count here, in their order, by a block-wide scan
    // over one thread per perimeter
    bool keep = false;
    int nv = 0;
    if (t < p.n_poly) {
        keep = true;
        if (!all) {
            if (p.kind[t] == 0) {
                const float4 b = p.box[t];
                keep = !(b.z < tx0 || b.x > tx1 || b.w < ty0 || b.y > ty1);
            } else {
                keep = s_near[t] != 1;
            }
        }
        nv = keep ? p.start[t + 1] - p.start[t] : 0;
    }
    const int lane = t & 31, wid = t >> 5;
    const unsigned bal = __ballot_sync(0xffffffffu, keep);
    int inc = nv;                                  // inclusive scan of vertex counts
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += u;
    }
    if (lane == 31) {
        s_wn[wid] = __popc(bal);
        s_wv[wid] = inc;
    }
    __syncthreads();
    int bn = 0, bv = 0, n_keep = 0, n_vert = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        if (w < wid) {
            bn += s_wn[w];
            bv += s_wv[w];
        }
        n_keep += s_wn[w];
        n_vert += s_wv[w];
    }
    if (keep) {
        const int k = bn + __popc(bal & ((1u << lane) - 1u));
        s_id[k] = t;
        s_off[k] = bv + inc - nv;
    }
    if (t == 0) s_off[n_keep] = n_vert;
    const float px = s_x[threadIdx.x];
    float py[kRows], c[kRows], smin[kRows], d2[kRows];
    bool inside[kRows];
#pragma unroll
    for (int m = 0; m < kRows; ++m) {
        py[m] = s_y[threadIdx.y + 8 * m];
        c[m] = 0.f;
        smin[m] = d2[m] = CUDART_INF_F;
        inside[m] = false;
    }
    int cur = -1;
    // the signed distance of the polygon just finished and its cost
    const auto finish = [&](int q) {
        const bool path = p.kind[q] != 0;
#pragma unroll
        for (int m = 0; m < kRows; ++m) {
            const float d = sqrtf(d2[m]);
            const float s = inside[m] != path ? -d : d;
            const float v = 1.f - s * p.inv_eps;
            if (v > 0.f) c[m] = fmaf(p.sigma * v, v, c[m]);
            smin[m] = fminf(smin[m], s);
            d2[m] = CUDART_INF_F;
            inside[m] = false;
        }
    };
    for (int c0 = 0; c0 < n_vert; c0 += kChunk) {
        __syncthreads();
        const int vc = c0 + t;
        if (vc < n_vert) {
            const int lo = perimeter_of(vc, s_off, n_keep);
            const int v = p.start[s_id[lo]] + (vc - s_off[lo]);
            if (p.edge) {
                s_a[t] = __ldg(&p.edge[v].a);
                s_b[t] = __ldg(&p.edge[v].b);
            } else {
                const CostmapEdge e = make_edge(p, v, s_id[lo]);
                s_a[t] = e.a;
                s_b[t] = e.b;
            }
        }
        __syncthreads();
        const int m_e = min(kChunk, n_vert - c0);
        for (int e = 0; e < m_e; ++e) {
            const float4 a = s_a[e], b = s_b[e];
            const int q = __float_as_int(b.w);
            if (q != cur) {
                if (cur >= 0) finish(cur);
                cur = q;
            }
            const float rx = px - a.x;
#pragma unroll
            for (int m = 0; m < kRows; ++m) {
                // distance to the segment
                const float ry = py[m] - a.y;
                float u = b.z > 0.f ? fmaf(rx, a.z, ry * a.w) / b.z : 0.f;
                u = fminf(fmaxf(u, 0.f), 1.f);
                const float dx = px - fmaf(u, a.z, a.x), dy = py[m] - fmaf(u, a.w, a.y);
                d2[m] = fminf(d2[m], fmaf(dx, dx, dy * dy));
                inside[m] = inside[m] != crosses(a, b, px, py[m]);
            }
        }
    }
    if (cur >= 0) finish(cur);
    const int i = blockIdx.x * kTile + threadIdx.x;
    if (i >= p.nx) return;
#pragma unroll
    for (int m = 0; m < kRows; ++m) {
        const int j = blockIdx.y * kTile + threadIdx.y + 8 * m;
        if (j >= p.ny) return;
        const size_t o = (size_t)j * p.nx + i;
        p.cost[o] = c[m];
        if (all) p.sdist[o] = smin[m];
    }
}

}  // namespace

cudaError_t launch_costmap(const CostmapParams &p, float reach, cudaStream_t stream)
{
    if (p.n_poly < 1 || p.n_poly > kCostmapMaxPolys) return cudaErrorInvalidValue;
    costmap_edges_kernel<<<(unsigned)p.n_poly, 32, 0, stream>>>(p, reach);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)((p.nx + kTile - 1) / kTile), (unsigned)((p.ny + kTile - 1) / kTile));
    costmap_kernel<<<grid, dim3(32, 8), 0, stream>>>(p, reach);
    return cudaGetLastError();
}

}  // namespace atp
