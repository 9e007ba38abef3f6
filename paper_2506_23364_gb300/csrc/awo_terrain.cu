// awo_terrain.cu -- DEM decode, normals/steepness and release-cell selection.
//
// These are streaming passes over the W x H grid (HBM-bound).  Each kernel is
// a grid-stride loop sized in multiples of the SM count, moving 16-byte
// vectors when its buffers are aligned (a general path covers ragged sizes
// and offsets).  Arithmetic uses explicit round-to-nearest intrinsics so no
// multiply-add is ever fused.
#include <math.h>
#include <stdio.h>

#include <mutex>
#include <vector>

#include "awo_internal.cuh"
#include "awo_particle.cuh"  // rcp_sqrt_rn

namespace awo {

int sm_count()
{
    static std::mutex mu;
    static std::vector<int> cache;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 1;
    std::lock_guard<std::mutex> lock(mu);
    if ((int)cache.size() <= dev) cache.resize(dev + 1, 0);
    if (cache[dev] == 0) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) n = 1;
        cache[dev] = n;
    }
    return cache[dev];
}

// ---------------------------------------------------------------------------
// a0. decode: h = (float)q * scale
// ---------------------------------------------------------------------------
// Four heights per thread (8-byte load, float4 store) when both buffers allow
// it, then a scalar tail.
// A thread issues the loads of DECODE_UNROLL groups of four heights (each
// coalesced across the grid) before their stores, so that enough bytes are
// in flight per SM to keep HBM busy.
constexpr int DECODE_UNROLL = 4;

__global__ void k_decode_u16(const uint16_t* __restrict__ q, int64_t n, float scale, float* __restrict__ h, bool vec4)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t n4 = vec4 ? n / 4 : 0;
    for (int64_t k0 = tid; k0 < n4; k0 += DECODE_UNROLL * stride) {
        uint2 w[DECODE_UNROLL];
#pragma unroll
        for (int u = 0; u < DECODE_UNROLL; ++u) {
            const int64_t k = k0 + u * stride;
            w[u] = k < n4 ? __ldg(reinterpret_cast<const uint2*>(q) + k) : make_uint2(0u, 0u);
        }
#pragma unroll
        for (int u = 0; u < DECODE_UNROLL; ++u) {
            const int64_t k = k0 + u * stride;
            if (k < n4)
                reinterpret_cast<float4*>(h)[k] = make_float4(__fmul_rn(__uint2float_rn(w[u].x & 0xffffu), scale),
                                                              __fmul_rn(__uint2float_rn(w[u].x >> 16), scale),
                                                              __fmul_rn(__uint2float_rn(w[u].y & 0xffffu), scale),
                                                              __fmul_rn(__uint2float_rn(w[u].y >> 16), scale));
        }
    }
    for (int64_t i = 4 * n4 + tid; i < n; i += stride) h[i] = __fmul_rn(__uint2float_rn((unsigned)q[i]), scale);
}

// ---------------------------------------------------------------------------
// a1. normals + tan^2 + optional slope in degrees.  One thread per run of 4
// cells of a row (no 64-bit division: a 32-bit item index splits into row and
// run).  When rows are 16-byte aligned (W % 4 == 0 and aligned buffers) the
// run's heights, the rows above and below and the outputs move as float4;
// the two horizontal neighbours outside the run are scalar loads (L1 hits)
// (k_normals_tiles).  Otherwise each thread takes single cells, side by side
// in a warp, with the same arithmetic (k_normals_cells).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void normal_of(float gx, float gy, float& nx, float& ny, float& nz, float& t2)
{
    t2 = __fadd_rn(__fmul_rn(gx, gx), __fmul_rn(gy, gy));
    const float inv = rcp_sqrt_rn(__fadd_rn(t2, 1.0f));  // = __frcp_rn(__fsqrt_rn(.)) bit for bit, one branch
    nx = __fmul_rn(-gx, inv);
    ny = __fmul_rn(-gy, inv);
    nz = inv;
}

__device__ __forceinline__ float slope_deg_of(float t2) { return atanf(sqrtf(t2)) * 57.295779513082320876f; }

// Heights for the normals: FP32 metres, or (FROM_U16) uint16 words decoded
// exactly as k_decode_u16 does, h = (float)q * scale.
template <bool FROM_U16>
struct HeightSrc {
    const void* p;
    float scale;
    __device__ __forceinline__ float at(int64_t i) const
    {
        if (FROM_U16) return __fmul_rn(__uint2float_rn((unsigned)__ldg(static_cast<const uint16_t*>(p) + i)), scale);
        return __ldg(static_cast<const float*>(p) + i);
    }
    // four consecutive heights from i (16-byte aligned floats / 8-byte aligned words)
    __device__ __forceinline__ float4 at4(int64_t i) const
    {
        if (FROM_U16) {
            const uint2 w = __ldg(reinterpret_cast<const uint2*>(static_cast<const uint16_t*>(p) + i));
            return make_float4(__fmul_rn(__uint2float_rn(w.x & 0xffffu), scale),
                               __fmul_rn(__uint2float_rn(w.x >> 16), scale),
                               __fmul_rn(__uint2float_rn(w.y & 0xffffu), scale),
                               __fmul_rn(__uint2float_rn(w.y >> 16), scale));
        }
        return __ldg(reinterpret_cast<const float4*>(static_cast<const float*>(p) + i));
    }
};

// The buffers and constants of one normals pass.  h_out (FROM_U16): the
// decoded heights, each written by the thread of its run, so a0 and a1 take
// one pass: awo_decode_u16 followed by awo_normals, without re-reading h.
template <bool FROM_U16>
struct NormalsArgs {
    HeightSrc<FROM_U16> h;
    int W, H;
    float cs;
    float* nrm;        // three planes, or null
    float* tan2;       // or null
    float* slope_deg;  // or null
    float* h_out;
};

// Divisions of the finite differences by cs and 2 cs: div_rn_by_rcp, = __fdiv_rn.
struct SpanDiv {
    float den1, den2, rden1, rden2;
};

__device__ __forceinline__ SpanDiv span_div(float cs)
{
    const float cs2 = __fmul_rn(cs, 2.0f);
    return SpanDiv{cs, cs2, __frcp_rn(cs), __frcp_rn(cs2)};
}

// The run of 4 cells at (x0, y), rows 16-byte aligned: reads, computes and
// writes; returns the four tan^2.  The range tests of the eight divisions
// and four reciprocal roots (see div_rn_by_rcp, rcp_sqrt_mid) are one: a
// difference's magnitude lies in [2^-60, 2^60] or is zero (which, less one,
// lies above every bound), a root's argument t2 + 1 is at least 1 or NaN.  A run
// outside takes the general form cell by cell.  With a test and a branch for
// each, the pass was bound by issue (8192^2 from uint16 with slope: 319 us).
template <bool FROM_U16>
__device__ __forceinline__ float4 normals_run(const NormalsArgs<FROM_U16>& a, const SpanDiv& d, int y, int x0)
{
    const int W = a.W, H = a.H;
    const int64_t plane = (int64_t)W * H;
    const int yl = y > 0 ? y - 1 : 0, yr = y < H - 1 ? y + 1 : H - 1;
    const int64_t row = (int64_t)y * W;
    const float4 c = a.h.at4(row + x0);
    const float4 up = a.h.at4((int64_t)yl * W + x0);
    const float4 dn = a.h.at4((int64_t)yr * W + x0);
    const float left = x0 > 0 ? a.h.at(row + x0 - 1) : c.x;
    const float right = x0 + 4 < W ? a.h.at(row + x0 + 4) : c.w;
    if (FROM_U16) *reinterpret_cast<float4*>(a.h_out + row + x0) = c;
    // differences and their spans: cells of the run's ends may be one-sided
    // (or W == 1: not with W % 4 == 0); a single row has gy = 0
    const float dx[4] = {__fsub_rn(c.y, left), __fsub_rn(c.z, c.x), __fsub_rn(c.w, c.y), __fsub_rn(right, c.z)};
    const float dy[4] = {__fsub_rn(dn.x, up.x), __fsub_rn(dn.y, up.y), __fsub_rn(dn.z, up.z), __fsub_rn(dn.w, up.w)};
    const bool one_l = x0 == 0, one_r = x0 + 4 >= W, one_y = yr - yl != 2;
    const float dny = one_y ? d.den1 : d.den2, rdy = one_y ? d.rden1 : d.rden2;
    float nx[4], ny[4], nz[4], t2[4];
    uint32_t least = 0xffffffffu, most = 0u;
    float top = 0.0f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const bool one = k == 0 ? one_l : (k == 3 ? one_r : false);
        const float den = one ? d.den1 : d.den2, rden = one ? d.rden1 : d.rden2;
        const uint32_t bx = __float_as_uint(dx[k]) & 0x7fffffffu, by = __float_as_uint(dy[k]) & 0x7fffffffu;
        least = min(least, min(bx - 1u, by - 1u));
        most = max(most, max(bx, by));
        const float gx = with_sign(div_rn_mid(dx[k], den, rden), dx[k]);
        const float gy = with_sign(div_rn_mid(dy[k], dny, rdy), dy[k]);
        t2[k] = __fadd_rn(__fmul_rn(gx, gx), __fmul_rn(gy, gy));
        const float x = __fadd_rn(t2[k], 1.0f);
        top = fmaxf(top, x);  // a NaN comes from a difference that is one, too
        nz[k] = rcp_sqrt_mid(x);
        nx[k] = __fmul_rn(-gx, nz[k]);
        ny[k] = __fmul_rn(-gy, nz[k]);
    }
    const bool fast = least >= DIV_LOW - 1u && most <= DIV_HIGH && top <= 0x1p100f && d.den1 >= 0x1p-60f &&
                      d.den2 <= 0x1p60f;
    if (!fast) {
#pragma unroll 1
        for (int k = 0; k < 4; ++k) {
            const bool one = k == 0 ? one_l : (k == 3 ? one_r : false);
            const float gx = div_rn_by_rcp<true>(k == 0 ? dx[0] : (k == 1 ? dx[1] : (k == 2 ? dx[2] : dx[3])),
                                                 one ? d.den1 : d.den2, one ? d.rden1 : d.rden2);
            const float gy = yr > yl ? div_rn_by_rcp<true>(k == 0 ? dy[0] : (k == 1 ? dy[1] : (k == 2 ? dy[2] : dy[3])),
                                                           dny, rdy)
                                     : 0.0f;
            float ox, oy, oz, ot;
            normal_of(gx, gy, ox, oy, oz, ot);
#pragma unroll
            for (int m = 0; m < 4; ++m)
                if (m == k) nx[m] = ox, ny[m] = oy, nz[m] = oz, t2[m] = ot;
        }
    }
    if (a.nrm) {
        *reinterpret_cast<float4*>(a.nrm + row + x0) = make_float4(nx[0], nx[1], nx[2], nx[3]);
        *reinterpret_cast<float4*>(a.nrm + plane + row + x0) = make_float4(ny[0], ny[1], ny[2], ny[3]);
        *reinterpret_cast<float4*>(a.nrm + 2 * plane + row + x0) = make_float4(nz[0], nz[1], nz[2], nz[3]);
    }
    const float4 t = make_float4(t2[0], t2[1], t2[2], t2[3]);
    if (a.tan2) *reinterpret_cast<float4*>(a.tan2 + row + x0) = t;
    if (a.slope_deg)
        *reinterpret_cast<float4*>(a.slope_deg + row + x0) =
            make_float4(slope_deg_of(t.x), slope_deg_of(t.y), slope_deg_of(t.z), slope_deg_of(t.w));
    return t;
}

// ---------------------------------------------------------------------------
// b. release selection, deterministic and ordered.
//   1. mask + per-tile count   (tile = RT_THREADS * RT_CELLS cells)
//   2. exclusive scan of the tile counts (one block; large grids only)
//   3. scatter of the selected indices in increasing order
// ---------------------------------------------------------------------------
constexpr int RT_THREADS = 256;
constexpr int RT_CELLS = 16;
constexpr int RT_TILE = RT_THREADS * RT_CELLS;

__device__ __forceinline__ int block_exclusive_scan(int v, int* total)
{
    __shared__ int warp_sums[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) warp_sums[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int nw = blockDim.x >> 5;
        int s = lane < nw ? warp_sums[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int t = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += t;
        }
        warp_sums[lane] = s;  // inclusive over warps
    }
    __syncthreads();
    int base = warp > 0 ? warp_sums[warp - 1] : 0;
    *total = warp_sums[(blockDim.x >> 5) - 1];
    __syncthreads();
    return base + incl - v;
}

// Sum of v over the block of THREADS, in thread 0 (call once per kernel: one barrier).
template <int THREADS = RT_THREADS>
__device__ __forceinline__ uint32_t block_total(int v)
{
    __shared__ int warp_total[THREADS / 32];
    const int t = __reduce_add_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) warp_total[threadIdx.x >> 5] = t;
    __syncthreads();
    int total = 0;
    if (threadIdx.x == 0) {
#pragma unroll
        for (int w = 0; w < THREADS / 32; ++w) total += warp_total[w];
    }
    return (uint32_t)total;
}

// Selection bits of the RT_CELLS consecutive cells from `base` (bit k: cell
// base + k is in [t_lo, t_hi]; cells past n are not).  Full, 16-byte-aligned
// runs load as four float4.
__device__ __forceinline__ uint32_t select_bits(const float* __restrict__ tan2, int64_t base, int64_t n, float t_lo,
                                                float t_hi)
{
    uint32_t bits = 0u;
    if (base + RT_CELLS <= n && (((uintptr_t)(tan2 + base)) & 15u) == 0) {
        const float4* p = reinterpret_cast<const float4*>(tan2 + base);
#pragma unroll
        for (int q = 0; q < RT_CELLS / 4; ++q) {
            const float4 t = __ldg(p + q);
            bits |= ((t_lo <= t.x && t.x <= t_hi) ? 1u : 0u) << (4 * q);
            bits |= ((t_lo <= t.y && t.y <= t_hi) ? 1u : 0u) << (4 * q + 1);
            bits |= ((t_lo <= t.z && t.z <= t_hi) ? 1u : 0u) << (4 * q + 2);
            bits |= ((t_lo <= t.w && t.w <= t_hi) ? 1u : 0u) << (4 * q + 3);
        }
    } else {
#pragma unroll
        for (int k = 0; k < RT_CELLS; ++k) {
            if (base + k < n) {
                const float t = __ldg(tan2 + base + k);
                if (t_lo <= t && t <= t_hi) bits |= 1u << k;
            }
        }
    }
    return bits;
}

// Bits of the non-zero bytes among the RT_CELLS mask bytes from `base`.
__device__ __forceinline__ uint32_t mask_bits(const uint8_t* __restrict__ mask, int64_t base, int64_t n)
{
    uint32_t bits = 0u;
    if (base + RT_CELLS <= n && (((uintptr_t)(mask + base)) & 15u) == 0) {
        const uint4 m = __ldg(reinterpret_cast<const uint4*>(mask + base));
        const uint32_t w[4] = {m.x, m.y, m.z, m.w};
#pragma unroll
        for (int q = 0; q < RT_CELLS / 4; ++q) {
            // bit 7 of every non-zero byte, then the four bits side by side (bit 8 b + 7 moves to 28 + b; the
            // product's other terms are distinct bits below 28)
            const uint32_t set = (w[q] | ((w[q] & 0x7f7f7f7fu) + 0x7f7f7f7fu)) & 0x80808080u;
            bits |= ((set * 0x00204081u) >> 28) << (4 * q);
        }
    } else {
#pragma unroll
        for (int k = 0; k < RT_CELLS; ++k)
            if (base + k < n && __ldg(mask + base + k) != 0) bits |= 1u << k;
    }
    return bits;
}

// The low four bits as 0/1 bytes (bit b to bit 8 b: the product's terms are distinct bits).
__device__ __forceinline__ uint32_t bytes_of(uint32_t bits)
{
    return ((bits & 15u) * 0x00204081u) & 0x01010101u;
}

// Writes the selection bits as 0/1 bytes (one uint4 when full and aligned).
__device__ __forceinline__ void store_mask(uint8_t* __restrict__ mask, int64_t base, int64_t n, uint32_t bits)
{
    uint32_t packed[RT_CELLS / 4];
#pragma unroll
    for (int q = 0; q < RT_CELLS / 4; ++q) packed[q] = bytes_of(bits >> (4 * q));
    if (base + RT_CELLS <= n && (((uintptr_t)(mask + base)) & 15u) == 0) {
        *reinterpret_cast<uint4*>(mask + base) = make_uint4(packed[0], packed[1], packed[2], packed[3]);
    } else {
        for (int k = 0; k < RT_CELLS; ++k)
            if (base + k < n) mask[base + k] = (uint8_t)((bits >> k) & 1u);
    }
}

// Where a block's selected indices go.  SUM: the counts of the tiles before
// its first are added up by the block itself (tile_base holds the tile
// counts, at most SUM_TILES_MAX, and the last block writes the number
// selected); else tile_base holds the scan's offsets.  On grids of up to 4096
// tiles (2^24 cells) the sum costs less than the scan's launch: a block
// reads at most 16 KB of counts from the L2 (with the single clearing launch
// of awo_simulate: 2048^2 workflow 996 -> 982 us, parabola 131 -> 120 us).
constexpr int SUM_TILES_MAX = 4096;

template <bool SUM>
__device__ __forceinline__ uint32_t scatter_base(const uint32_t* __restrict__ tile_base, uint32_t first_tile)
{
    if (!SUM) return tile_base[first_tile];
    __shared__ uint32_t part[RT_THREADS / 32];
    uint32_t s = 0u;
    for (uint32_t t = threadIdx.x; t < first_tile; t += RT_THREADS) s += __ldg(tile_base + t);
    s = __reduce_add_sync(0xffffffffu, s);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
    __syncthreads();
    s = 0u;
#pragma unroll
    for (int w = 0; w < RT_THREADS / 32; ++w) s += part[w];
    return s;
}

__global__ void __launch_bounds__(RT_THREADS) k_release_mask(const float* __restrict__ tan2, int64_t n, float t_lo,
                                                             float t_hi, uint8_t* __restrict__ mask,
                                                             uint32_t* __restrict__ tile_count)
{
    const int64_t base = (int64_t)blockIdx.x * RT_TILE + (int64_t)threadIdx.x * RT_CELLS;
    const uint32_t bits = select_bits(tan2, base, n, t_lo, t_hi);
    if (mask) store_mask(mask, base, n, bits);
    const uint32_t total = block_total(__popc(bits));
    if (threadIdx.x == 0) tile_count[blockIdx.x] = total;
}

// Aligned rows (a run of 4 cells is 4 consecutive indices): a block makes the
// normals of one release tile, and (tile_count not null) tests each tan^2
// while it is in registers and writes the mask and the tile's count -- a1 and
// the first release pass in one: tan^2 is not read back (4 of the 32 bytes
// that the two passes move per cell) and a launch is saved.  Bound by HBM:
// 8192^2 from uint16 with slope, normals and release 408 -> 313 us (86% of the
// measured copy bandwidth).  A block per tile rather than a persistent
// grid-stride loop, whose blocks all reached the same rows' end together.
template <bool FROM_U16>
__global__ void __launch_bounds__(RT_THREADS) k_normals_tiles(const __grid_constant__ NormalsArgs<FROM_U16> a,
                                                                float t_lo, float t_hi, uint8_t* __restrict__ mask,
                                                                uint32_t* __restrict__ tile_count)
{
    const uint32_t runs = (uint32_t)a.W >> 2, items = runs * (uint32_t)a.H;
    const SpanDiv d = span_div(a.cs);
    const uint32_t first = blockIdx.x * (uint32_t)(RT_TILE / 4);
    const uint32_t y_first = first / runs, x_first = first - y_first * runs;  // in runs
    int count = 0;
#pragma unroll 1
    for (uint32_t k = threadIdx.x; k < RT_TILE / 4; k += RT_THREADS) {
        if (first + k >= items) break;
        uint32_t y = y_first, x = x_first + k;
        if (x >= runs) {
            const uint32_t rows = x / runs;
            y += rows;
            x -= rows * runs;
        }
        const float4 t = normals_run<FROM_U16>(a, d, (int)y, (int)(4u * x));
        if (!tile_count) continue;
        const uint32_t sel = ((t_lo <= t.x && t.x <= t_hi) ? 1u : 0u) | ((t_lo <= t.y && t.y <= t_hi) ? 0x100u : 0u) |
                             ((t_lo <= t.z && t.z <= t_hi) ? 0x10000u : 0u) |
                             ((t_lo <= t.w && t.w <= t_hi) ? 0x1000000u : 0u);
        if (mask) *reinterpret_cast<uint32_t*>(mask + 4 * (size_t)(first + k)) = sel;
        count += __popc(sel);
    }
    if (tile_count) {
        const uint32_t total = block_total(count);
        if (threadIdx.x == 0) tile_count[blockIdx.x] = total;
    }
}

// The same for any width and alignment: single cells, a warp's side by side,
// so that every load and store is coalesced whatever the rows' alignment
// (four consecutive cells a thread, one after the other, touched each sector
// four times and took 3325 x 4197 with the release pass 238 -> 94 us, 4.0
// times the aligned pass's time a cell before and 1.6 now).  512 threads: 256 or 1024 took
// 626 x 422 19.1 -> 20-22 us.  A block takes `span` cells: a release tile when
// it counts one.
constexpr int NC_THREADS = 512;

template <bool FROM_U16>
__global__ void __launch_bounds__(NC_THREADS) k_normals_cells(const __grid_constant__ NormalsArgs<FROM_U16> a,
                                                                uint32_t span, float t_lo, float t_hi,
                                                                uint8_t* __restrict__ mask,
                                                                uint32_t* __restrict__ tile_count)
{
    const uint32_t W = (uint32_t)a.W, H = (uint32_t)a.H, n = W * H;  // below 2^31
    const SpanDiv d = span_div(a.cs);
    const bool spans = d.den1 >= 0x1p-60f && d.den2 <= 0x1p60f;
    const uint32_t first = blockIdx.x * span;
    const uint32_t y_first = first / W, x_first = first - y_first * W;
    int count = 0;
#pragma unroll 2
    for (uint32_t k = threadIdx.x; k < span; k += NC_THREADS) {
        const uint32_t i = first + k;
        if (i >= n) break;
        uint32_t y = y_first, x = x_first + k;
        if (x >= W) {
            const uint32_t rows = x / W;
            y += rows;
            x -= rows * W;
        }
        const uint32_t xl = x > 0u ? i - 1u : i, xr = x + 1u < W ? i + 1u : i;
        const uint32_t yl = y > 0u ? i - W : i, yr = y + 1u < H ? i + W : i;
        const float dx = __fsub_rn(a.h.at(xr), a.h.at(xl)), dy = __fsub_rn(a.h.at(yr), a.h.at(yl));
        if (FROM_U16) a.h_out[i] = a.h.at(i);
        const bool two_x = xr - xl == 2u, two_y = yr - yl == 2u * W;
        const float denx = two_x ? d.den2 : d.den1, rdx = two_x ? d.rden2 : d.rden1;
        const float deny = two_y ? d.den2 : d.den1, rdy = two_y ? d.rden2 : d.rden1;
        // one range test for both divisions and the root, as in normals_run
        const uint32_t bx = __float_as_uint(dx) & 0x7fffffffu, by = __float_as_uint(dy) & 0x7fffffffu;
        const float gx = with_sign(div_rn_mid(dx, denx, rdx), dx), gy = with_sign(div_rn_mid(dy, deny, rdy), dy);
        float t2 = __fadd_rn(__fmul_rn(gx, gx), __fmul_rn(gy, gy));
        const float top = __fadd_rn(t2, 1.0f);
        float nz = rcp_sqrt_mid(top);
        float nx = __fmul_rn(-gx, nz), ny = __fmul_rn(-gy, nz);
        if (!(min(bx - 1u, by - 1u) >= DIV_LOW - 1u && max(bx, by) <= DIV_HIGH && top <= 0x1p100f && spans)) {
            const float ex = xr > xl ? div_rn_by_rcp<true>(dx, denx, rdx) : 0.0f;
            const float ey = yr > yl ? div_rn_by_rcp<true>(dy, deny, rdy) : 0.0f;
            normal_of(ex, ey, nx, ny, nz, t2);
        }
        if (a.nrm) {
            a.nrm[i] = nx;
            a.nrm[(size_t)n + i] = ny;
            a.nrm[2 * (size_t)n + i] = nz;
        }
        if (a.tan2) a.tan2[i] = t2;
        if (a.slope_deg) a.slope_deg[i] = slope_deg_of(t2);
        if (tile_count) {
            const uint32_t sel = t_lo <= t2 && t2 <= t_hi ? 1u : 0u;
            if (mask) mask[i] = (uint8_t)sel;
            count += (int)sel;
        }
    }
    if (tile_count) {
        const uint32_t total = block_total<NC_THREADS>(count);
        if (threadIdx.x == 0) tile_count[blockIdx.x] = total;
    }
}

// Exclusive scan of tile counts in one block of 1024 threads; also writes the
// total to *d_n.  Each thread scans a contiguous run of tiles.  Up to 16 tiles
// per thread (grids up to 2^26 cells) the run is held in registers and read
// and written as uint4 when the buffers allow, so the scan costs one round
// trip to memory; larger grids read their runs twice (measured on GB300, the
// three release passes at 8192^2: 0.106 -> 0.096 ms).
__global__ void __launch_bounds__(1024) k_release_scan(const uint32_t* __restrict__ tile_count, int n_tiles,
                                                       uint32_t* __restrict__ tile_offset, uint32_t* __restrict__ d_n)
{
    const int per = (n_tiles + blockDim.x - 1) / blockDim.x;
    const int lo = threadIdx.x * per;
    const int hi = min(lo + per, n_tiles);
    int total;
    if (per <= 16) {
        uint32_t c[16];
        const bool vec = (per & 3) == 0 && (((uintptr_t)tile_count) & 15u) == 0 && (((uintptr_t)tile_offset) & 15u) == 0 &&
                         hi - lo == per;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (vec && 4 * q < per) {
                const uint4 v = __ldg(reinterpret_cast<const uint4*>(tile_count + lo) + q);
                c[4 * q] = v.x, c[4 * q + 1] = v.y, c[4 * q + 2] = v.z, c[4 * q + 3] = v.w;
            } else {
#pragma unroll
                for (int k = 4 * q; k < 4 * q + 4; ++k) c[k] = lo + k < hi ? __ldg(tile_count + lo + k) : 0u;
            }
        }
        int s = 0;
#pragma unroll
        for (int k = 0; k < 16; ++k) s += (int)c[k];
        uint32_t run = (uint32_t)block_exclusive_scan(s, &total);
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const uint32_t here = run;
            run += c[k];
            c[k] = here;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (vec && 4 * q < per) {
                reinterpret_cast<uint4*>(tile_offset + lo)[q] = make_uint4(c[4 * q], c[4 * q + 1], c[4 * q + 2],
                                                                           c[4 * q + 3]);
            } else {
#pragma unroll
                for (int k = 4 * q; k < 4 * q + 4; ++k)
                    if (lo + k < hi) tile_offset[lo + k] = c[k];
            }
        }
    } else {
        // more than 16 tiles a thread (release textures): two passes over the
        // thread's range, 16-byte loads unrolled so that several are in flight
        const bool vec = (per & 3) == 0 && (((uintptr_t)tile_count) & 15u) == 0 &&
                         (((uintptr_t)tile_offset) & 15u) == 0 && hi - lo == per;
        const uint4* src = reinterpret_cast<const uint4*>(tile_count + lo);
        uint32_t s = 0u;
        if (vec) {
#pragma unroll 2
            for (int q = 0; q < per / 4; ++q) {
                const uint4 v = __ldg(src + q);
                s += v.x + v.y + v.z + v.w;
            }
        } else {
            for (int t = lo; t < hi; ++t) s += tile_count[t];
        }
        uint32_t run = (uint32_t)block_exclusive_scan((int)s, &total);
        if (vec) {
            uint4* dst = reinterpret_cast<uint4*>(tile_offset + lo);
#pragma unroll 2
            for (int q = 0; q < per / 4; ++q) {
                const uint4 v = __ldg(src + q);
                uint4 o;
                o.x = run;
                o.y = o.x + v.x;
                o.z = o.y + v.y;
                o.w = o.z + v.z;
                run = o.w + v.w;
                dst[q] = o;
            }
        } else {
            for (int t = lo; t < hi; ++t) {
                tile_offset[t] = run;
                run += tile_count[t];
            }
        }
    }
    if (threadIdx.x == 0) *d_n = (uint32_t)total;
}

// Ordered scatter of the selected indices of a tile.
template <bool SUM>
__global__ void __launch_bounds__(RT_THREADS) k_release_scatter(const float* __restrict__ tan2, int64_t n, float t_lo,
                                                                float t_hi, const uint32_t* __restrict__ tile_base,
                                                                uint32_t* __restrict__ cells, uint32_t* __restrict__ d_n)
{
    const int64_t base = (int64_t)blockIdx.x * RT_TILE + (int64_t)threadIdx.x * RT_CELLS;
    uint32_t bits = select_bits(tan2, base, n, t_lo, t_hi);
    const uint32_t before = scatter_base<SUM>(tile_base, blockIdx.x);
    int total;
    uint32_t off = (uint32_t)block_exclusive_scan(__popc(bits), &total) + before;
    if (SUM && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *d_n = before + (uint32_t)total;
    while (bits) {
        const int k = __ffs(bits) - 1;
        bits &= bits - 1;
        cells[off++] = (uint32_t)(base + k);
    }
}

// Release cells given by a mask -- a caller's (known release areas, Sec. 5.2:
// "known release points encoded in a pre-computed texture") or the one the
// first release pass wrote: per-tile counts and ordered scatter of the cells
// whose mask byte is non-zero.
__global__ void __launch_bounds__(RT_THREADS) k_mask_count(const uint8_t* __restrict__ mask, int64_t n,
                                                           uint32_t* __restrict__ tile_count)
{
    const int64_t base = (int64_t)blockIdx.x * RT_TILE + (int64_t)threadIdx.x * RT_CELLS;
    const uint32_t total = block_total(__popc(mask_bits(mask, base, n)));
    if (threadIdx.x == 0) tile_count[blockIdx.x] = total;
}

// The scatter pass takes SC_RUNS consecutive runs per thread, so a block
// covers SC_RUNS release tiles and starts at the offset of the first: four
// mask loads in flight per thread and a quarter of the blocks and block scans
// (measured on GB300, the three release passes at 8192^2: 0.111 -> 0.106 ms).
// Each thread writes its own indices, a few to a sector.  Collecting a block's
// in shared memory to write them side by side took 2% longer over the whole
// terrain of a 4096^2 DEM at 2x, a loop of the warp over its lanes with
// indices (coalesced too) 6%: nearly every lane has some.  21 us for 67 M
// texels, 64% of the issue slots, 12 us at the copy rate.
constexpr int SC_RUNS = 4;
constexpr int SC_TILE = RT_TILE * SC_RUNS;

template <bool SUM>
__global__ void __launch_bounds__(RT_THREADS) k_mask_scatter(const uint8_t* __restrict__ mask, int64_t n,
                                                             const uint32_t* __restrict__ tile_base,
                                                             uint32_t* __restrict__ cells, uint32_t* __restrict__ d_n)
{
    const int64_t base = (int64_t)blockIdx.x * SC_TILE + (int64_t)threadIdx.x * (RT_CELLS * SC_RUNS);
    uint32_t bits[SC_RUNS];
    int count = 0;
#pragma unroll
    for (int r = 0; r < SC_RUNS; ++r) {
        bits[r] = mask_bits(mask, base + r * RT_CELLS, n);
        count += __popc(bits[r]);
    }
    const uint32_t before = scatter_base<SUM>(tile_base, blockIdx.x * SC_RUNS);
    int total;
    uint32_t off = (uint32_t)block_exclusive_scan(count, &total) + before;
    if (SUM && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *d_n = before + (uint32_t)total;
    uint32_t* out = cells + off;
    const uint32_t b0 = (uint32_t)base;
#pragma unroll
    for (int half = 0; half < 2; ++half) {
        uint32_t b = bits[2 * half] | bits[2 * half + 1] << 16;
        while (b) {
            *out++ = b0 + 32u * half + (uint32_t)(__ffs(b) - 1);
            b &= b - 1u;
        }
    }
}

// Release points on a texture at 2^r times the DEM resolution
// (awo_release_texture): per tile of RT_TILE texels, the mask and its count.
// A texel's steepness is the bilinear interpolation of tan^2 at its centre,
// with the footprint rule and FP32 weights of the particles' height sampling.
__device__ __forceinline__ float texel_centre(uint32_t a, float scale, float n_m1)
{
    const float c = __fsub_rn(__fmul_rn(__fadd_rn(__uint2float_rn(a), 0.5f), scale), 0.5f);
    return fminf(fmaxf(c, 0.0f), n_m1);
}

// A run of RT_CELLS texels of a texture at 2^R times the DEM resolution
// (R >= 0) whose first texel index a along the row is a multiple of 2^R (every
// run of the kernel below: runs start at multiples of RT_CELLS and rows have
// W 2^R texels).  Texel a + k is centred at u = A + (2k + 1 - 2^R) / 2^(R+1)
// with A = a / 2^R, so its footprint column is A + delta(k) and its weight
// frac(k), both fixed for the run -- exactly what texel_centre and the floor
// give when no clamping occurs.
template <int R>
struct TexRun {
    static constexpr int S = 1 << R;
    __host__ __device__ static constexpr int num(int k) { return 2 * k + 1 - S; }
    __host__ __device__ static constexpr int fdiv(int x, int d) { return x >= 0 ? x / d : -((-x + d - 1) / d); }
    __host__ __device__ static constexpr int delta(int k) { return fdiv(num(k), 2 * S); }
    __host__ __device__ static constexpr float frac(int k) { return (float)(num(k) - delta(k) * 2 * S) / (float)(2 * S); }
    __host__ __device__ static constexpr float one_minus_frac(int k) { return 1.0f - frac(k); }  // exact: frac has <= 4 bits
    static constexpr int DMIN = delta(0), DMAX = delta(RT_CELLS - 1);
    static constexpr int NC = DMAX - DMIN + 2;  // footprint columns the run reads
};

// Selection bits of a run in one texture row, away from both row ends: the
// two tan^2 rows under it are loaded once (NC values each) and every texel
// interpolates with compile-time weights.  Same arithmetic as the general
// path, texel by texel.  VEC: tan2 + row + A is 16-byte aligned (tan2
// aligned, W and A multiples of 4), so the aligned groups of four among the
// NC columns are read as float4 -- a quarter of the load instructions, which
// bound this pass through the L1 otherwise.
template <int R, bool VEC>
__device__ __forceinline__ uint32_t texel_run_bits(const float* __restrict__ tan2, int row, int dj, int A, float oy,
                                                   float fy, float t_lo, float t_hi)
{
    using T = TexRun<R>;
    float top[T::NC], bot[T::NC];
    const float* p = tan2 + row + A;
#pragma unroll
    for (int i = T::DMIN; i <= T::DMAX + 1; ++i) {
        const int g = i & ~3;  // start of i's aligned group of four (relative to A)
        const bool whole = VEC && g >= T::DMIN && g + 3 <= T::DMAX + 1;
        if (whole && i == g) {
            const float4 qt = __ldg(reinterpret_cast<const float4*>(p + i));
            const float4 qb = __ldg(reinterpret_cast<const float4*>(p + dj + i));
            top[i - T::DMIN] = qt.x, top[i - T::DMIN + 1] = qt.y, top[i - T::DMIN + 2] = qt.z,
                          top[i - T::DMIN + 3] = qt.w;
            bot[i - T::DMIN] = qb.x, bot[i - T::DMIN + 1] = qb.y, bot[i - T::DMIN + 2] = qb.z,
                          bot[i - T::DMIN + 3] = qb.w;
        } else if (!whole) {
            top[i - T::DMIN] = __ldg(p + i);
            bot[i - T::DMIN] = __ldg(p + dj + i);
        }
    }
    uint32_t bits = 0u;
#pragma unroll
    for (int k = 0; k < RT_CELLS; ++k) {
        const int c = T::delta(k) - T::DMIN;
        const float fx = T::frac(k), ox = T::one_minus_frac(k);
        const float tp = __fadd_rn(__fmul_rn(top[c], ox), __fmul_rn(top[c + 1], fx));
        const float bt = __fadd_rn(__fmul_rn(bot[c], ox), __fmul_rn(bot[c + 1], fx));
        const float Tk = __fadd_rn(__fmul_rn(tp, oy), __fmul_rn(bt, fy));
        bits |= ((t_lo <= Tk && Tk <= t_hi) ? 1u : 0u) << k;
    }
    return bits;
}

// Runs in one row away from the row ends take texel_run_bits; the rest the
// general per-texel path.
// VEC as in texel_run_bits (host-checked alignment of tan2 and W; R <= 2).
template <int R, bool VEC>
__global__ void __launch_bounds__(RT_THREADS) k_release_texture_mask(const float* __restrict__ tan2, int W, int H,
                                                                     uint32_t Wr, int64_t n, float scale,
                                                                     float t_lo, float t_hi,
                                                                     uint8_t* __restrict__ mask,
                                                                     uint32_t* __restrict__ tile_count)
{
    // the texture has fewer than 2^31 texels: 32-bit indices throughout
    const uint32_t tile = blockIdx.x;
    const uint32_t base = tile * (uint32_t)RT_TILE + threadIdx.x * (uint32_t)RT_CELLS;
    const uint32_t n32 = (uint32_t)n;
    const float wm1 = __int2float_rn(W - 1), hm1 = __int2float_rn(H - 1);
    uint32_t b = 0u, a = 0u;
    if (base < n32) {
        b = base / Wr;
        a = base - b * Wr;
    }
    // row terms, recomputed when the run wraps to the next texture row
    float v = texel_centre(b, scale, hm1);
    int j0 = __float2int_rd(v);
    float fy = __fsub_rn(v, __int2float_rn(j0)), oy = __fsub_rn(1.0f, fy);
    int row = j0 * W, dj = j0 + 1 < H ? W : 0;
    uint32_t bits = 0u;
    bool done = false;
    if (base + RT_CELLS <= n32 && a + RT_CELLS <= Wr) {
        const int A = (int)(a >> R);
        if (A + TexRun<R>::DMIN >= 0 && A + TexRun<R>::DMAX + 1 <= W - 2) {
            bits = texel_run_bits<R, VEC>(tan2, row, dj, A, oy, fy, t_lo, t_hi);
            done = true;
        }
    }
    if (!done) {
        // footprint of the previous texel: on a finer texture 2^r consecutive
        // texels share one, so its four values are loaded once
        int o_prev = -1;
        float t00 = 0.0f, t10 = 0.0f, t01 = 0.0f, t11 = 0.0f;
#pragma unroll
        for (int k = 0; k < RT_CELLS; ++k) {
            if (base + k < n32) {
                const float u = texel_centre(a, scale, wm1);
                const int i0 = __float2int_rd(u);
                const float fx = __fsub_rn(u, __int2float_rn(i0));
                const int o = row + i0;
                if (o != o_prev) {
                    const int di = i0 + 1 < W ? 1 : 0;
                    t00 = __ldg(tan2 + o);
                    t10 = __ldg(tan2 + o + di);
                    t01 = __ldg(tan2 + o + dj);
                    t11 = __ldg(tan2 + o + dj + di);
                    o_prev = o;
                }
                const float ox = __fsub_rn(1.0f, fx);
                const float top = __fadd_rn(__fmul_rn(t00, ox), __fmul_rn(t10, fx));
                const float bot = __fadd_rn(__fmul_rn(t01, ox), __fmul_rn(t11, fx));
                const float T = __fadd_rn(__fmul_rn(top, oy), __fmul_rn(bot, fy));
                bits |= ((t_lo <= T && T <= t_hi) ? 1u : 0u) << k;
                if (++a == Wr) {
                    a = 0u;
                    ++b;
                    v = texel_centre(b, scale, hm1);
                    j0 = __float2int_rd(v);
                    fy = __fsub_rn(v, __int2float_rn(j0));
                    oy = __fsub_rn(1.0f, fy);
                    row = j0 * W;
                    dj = j0 + 1 < H ? W : 0;
                }
            }
        }
    }
    store_mask(mask, base, n, bits);
    const uint32_t total = block_total(__popc(bits));
    if (threadIdx.x == 0) tile_count[tile] = total;
}

// Coarser textures (R < 0), any width: single texels, a warp's side by side,
// with the footprint of its centre.  (A run of 16 texels a thread, whose
// footprints share nothing here, was a chain of 16 loads: terrain of 2112 x
// 1344 at 1/2 40.3 -> 27.5 us, of 3001 x 2999 at 1/4, normals included, 158 ->
// 69 us.  On finer textures the runs' shared loads win: 3325 x 4197 at 2x 189
// against 263 us.)
__global__ void __launch_bounds__(NC_THREADS) k_release_texture_texels(const float* __restrict__ tan2, int W, int H,
                                                                         uint32_t Wr, uint32_t n, float scale,
                                                                         float t_lo, float t_hi,
                                                                         uint8_t* __restrict__ mask,
                                                                         uint32_t* __restrict__ tile_count)
{
    const float wm1 = __int2float_rn(W - 1), hm1 = __int2float_rn(H - 1);
    const uint32_t first = blockIdx.x * (uint32_t)RT_TILE;
    const uint32_t b_first = first / Wr, a_first = first - b_first * Wr;
    int count = 0;
#pragma unroll 4
    for (uint32_t k = threadIdx.x; k < (uint32_t)RT_TILE; k += NC_THREADS) {
        if (first + k >= n) break;
        uint32_t b = b_first, a = a_first + k;
        if (a >= Wr) {
            const uint32_t rows = a / Wr;
            b += rows;
            a -= rows * Wr;
        }
        const float u = texel_centre(a, scale, wm1), v = texel_centre(b, scale, hm1);
        const int i0 = __float2int_rd(u), j0 = __float2int_rd(v);
        const float fx = __fsub_rn(u, __int2float_rn(i0)), fy = __fsub_rn(v, __int2float_rn(j0));
        const float ox = __fsub_rn(1.0f, fx), oy = __fsub_rn(1.0f, fy);
        const int o = j0 * W + i0, di = i0 + 1 < W ? 1 : 0, dj = j0 + 1 < H ? W : 0;
        const float t00 = __ldg(tan2 + o), t10 = __ldg(tan2 + o + di);
        const float t01 = __ldg(tan2 + o + dj), t11 = __ldg(tan2 + o + dj + di);
        const float top = __fadd_rn(__fmul_rn(t00, ox), __fmul_rn(t10, fx));
        const float bot = __fadd_rn(__fmul_rn(t01, ox), __fmul_rn(t11, fx));
        const float T = __fadd_rn(__fmul_rn(top, oy), __fmul_rn(bot, fy));
        const uint32_t sel = t_lo <= T && T <= t_hi ? 1u : 0u;
        mask[first + k] = (uint8_t)sel;
        count += (int)sel;
    }
    const uint32_t total = block_total<NC_THREADS>(count);
    if (threadIdx.x == 0) tile_count[blockIdx.x] = total;
}

// Rows that share their tan^2 rows (R = 1, 2): texture rows b = 2^R j + 2^(R-1)
// ... 2^R j + 2^(R-1) + 2^R - 1 all have their centres between DEM rows j and
// j + 1, so their texels at one column interpolate the same two horizontal
// interpolations, with their own vertical weights.  A block takes one tile
// column (RT_TILE texels of a row; rows are whole tiles) of the rows of group
// blockIdx.y, each thread a run of RT_CELLS texels in every row: the tan^2
// values and the horizontal interpolations are computed once for the group,
// the vertical combination per row (the same operations, in the same order, as
// k_release_texture_mask).  Group 0 holds the 2^(R-1) rows above the first of
// those and group H the 2^(R-1) below the last: their centres clamp to the
// DEM's first and last row.  The runs at a row's ends are not texel by texel
// but differ only in the weights of their 2^(R-1) clamped texels and in the
// columns of their outer loads (one slow lane in every block had the other
// warps wait at its barrier, 7.6 warps an issue), and the texels are selected
// as bytes of the mask's words: 46 -> 36 us for the mask of a 4096^2 DEM at
// 2x, 89 -> 71 us for the whole terrain of a 2048^2 one at 4x.  Issue slots
// bound it (16 warp instructions per 32 texels before; HBM would take 20 us).
// (The edge rows in launches of their own and a block scan where only its
// total is wanted: 61 us.)
template <int R, bool VEC>
__global__ void __launch_bounds__(RT_THREADS) k_release_texture_rows(const float* __restrict__ tan2, int W, int H,
                                                                     uint32_t Wr, int64_t n, float scale,
                                                                     float t_lo, float t_hi,
                                                                     uint8_t* __restrict__ mask,
                                                                     uint32_t* __restrict__ tile_count)
{
    using T = TexRun<R>;
    constexpr int ROWS = 1 << R, HALF = ROWS / 2;
    const uint32_t tiles_per_row = Wr / (uint32_t)RT_TILE;
    const int group = (int)blockIdx.y;
    const bool edge = group == 0 || group == H;
    const int j = group == 0 ? 0 : group - 1;  // DEM row under the group
    const int dj = j + 1 < H ? W : 0;          // to the row below, clamped
    const uint32_t b0 = group == 0 ? 0u : (uint32_t)j * ROWS + HALF;  // first texture row of the group
    const uint32_t a = blockIdx.x * (uint32_t)RT_TILE + threadIdx.x * (uint32_t)RT_CELLS;
    const float hm1 = __int2float_rn(H - 1);
    float oy[ROWS], fy[ROWS];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        const float v = texel_centre(b0 + r, scale, hm1);  // in [j, j + 1) (rows of the group)
        fy[r] = __fsub_rn(v, __int2float_rn(j));
        oy[r] = __fsub_rn(1.0f, fy[r]);
    }
    const int row = j * W;
    uint32_t sel[ROWS][RT_CELLS / 4];  // the run's mask bytes
#pragma unroll
    for (int r = 0; r < ROWS; ++r)
#pragma unroll
        for (int q = 0; q < RT_CELLS / 4; ++q) sel[r][q] = 0u;
    const int A = (int)(a >> R);
    const bool first = A == 0, last = A + T::DMAX + 1 == W;  // the runs at the row's ends
    float top[T::NC], bot[T::NC];
    const float* p = tan2 + row + A;
#pragma unroll
    for (int i = T::DMIN; i <= T::DMAX + 1; ++i) {
        const int g = i & ~3;
        const bool whole = VEC && g >= 0 && g + 3 <= T::DMAX;
        if (whole && i == g) {
            const float4 qt = __ldg(reinterpret_cast<const float4*>(p + i));
            const float4 qb = __ldg(reinterpret_cast<const float4*>(p + dj + i));
            top[i - T::DMIN] = qt.x, top[i - T::DMIN + 1] = qt.y, top[i - T::DMIN + 2] = qt.z,
                          top[i - T::DMIN + 3] = qt.w;
            bot[i - T::DMIN] = qb.x, bot[i - T::DMIN + 1] = qb.y, bot[i - T::DMIN + 2] = qb.z,
                          bot[i - T::DMIN + 3] = qb.w;
        } else if (!whole) {
            const int c = min(max(i, -A), W - 1 - A);  // inside the row
            top[i - T::DMIN] = __ldg(p + c);
            bot[i - T::DMIN] = __ldg(p + dj + c);
        }
    }
#pragma unroll
    for (int k = 0; k < RT_CELLS; ++k) {
        const int c = T::delta(k) - T::DMIN;
        float fx = T::frac(k), ox = T::one_minus_frac(k);
        float tl = top[c], tr = top[c + 1], bl = bot[c], br = bot[c + 1];
        if (k < HALF && first) {  // centre clamped to column 0: weights 1 and 0 of columns 0 and 1
            fx = 0.0f, ox = 1.0f;
            tl = top[c + 1], tr = top[c + 2], bl = bot[c + 1], br = bot[c + 2];
        }
        if (k >= RT_CELLS - HALF && last) {  // clamped to column W - 1: weights 1 and 0 of that column
            fx = 0.0f, ox = 1.0f;
            tr = tl, br = bl;
        }
        const float tp = __fadd_rn(__fmul_rn(tl, ox), __fmul_rn(tr, fx));
        const float bt = __fadd_rn(__fmul_rn(bl, ox), __fmul_rn(br, fx));
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            const float Tk = __fadd_rn(__fmul_rn(tp, oy[r]), __fmul_rn(bt, fy[r]));
            if (t_lo <= Tk && Tk <= t_hi) sel[r][k / 4] |= 1u << (8 * (k % 4));
        }
    }
    const bool aligned = ((uintptr_t)mask & 15u) == 0;  // and so every run: rows are whole tiles
    __shared__ int s_count[ROWS][RT_THREADS / 32];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        if (!edge || r < HALF) {
            uint8_t* m = mask + (size_t)(b0 + r) * Wr + a;
            if (aligned) {
                *reinterpret_cast<uint4*>(m) = make_uint4(sel[r][0], sel[r][1], sel[r][2], sel[r][3]);
            } else {
#pragma unroll
                for (int k = 0; k < RT_CELLS; ++k) m[k] = (uint8_t)(sel[r][k / 4] >> (8 * (k % 4)));
            }
        }
        const uint32_t bytes = sel[r][0] + sel[r][1] + sel[r][2] + sel[r][3];  // at most 4 each
        const int c = __reduce_add_sync(0xffffffffu, (int)((bytes * 0x01010101u) >> 24));
        if ((threadIdx.x & 31) == 0) s_count[r][threadIdx.x >> 5] = c;
    }
    __syncthreads();
    if (threadIdx.x < (edge ? HALF : ROWS)) {
        int total = 0;
#pragma unroll
        for (int w = 0; w < RT_THREADS / 32; ++w) total += s_count[threadIdx.x][w];
        tile_count[(b0 + threadIdx.x) * tiles_per_row + blockIdx.x] = (uint32_t)total;
    }
}

static float tan2_of_degrees(double deg)
{
    double t = tan(deg * (3.14159265358979323846 / 180.0));
    return (float)(t * t);
}

}  // namespace awo

using namespace awo;

extern "C" const char* awo_status_string(awo_status s)
{
    switch (s) {
        case AWO_OK: return "ok";
        case AWO_EINVAL: return "invalid argument";
        case AWO_ENOMEM: return "workspace too small";
        case AWO_ECUDA: return "CUDA error";
        case AWO_ETIMEOUT: return "bounded device wait timed out";
        case AWO_EOVERFLOW: return "32-bit count overflow";
        case AWO_ECANCELLED: return "cancelled";
    }
    return "unknown status";
}

extern "C" int32_t awo_version(void) { return 10300; }

extern "C" awo_status awo_decode_u16(const uint16_t* d_q, awo_grid g, float scale, float* d_h, void* stream)
{
    if (!d_q || !d_h || !grid_ok(g) || !(scale > 0.0f) || !(scale < 3.0e38f)) return AWO_EINVAL;
    const int64_t n = cells_of(g);
    const bool vec4 = (((uintptr_t)d_q) & 7u) == 0 && (((uintptr_t)d_h) & 15u) == 0;
    k_decode_u16<<<stream_blocks(vec4 ? n / 4 + 1 : n, 256), 256, 0, as_stream(stream)>>>(d_q, n, scale, d_h, vec4);
    return launch_status();
}

// Rows and buffers of a pass over runs of four cells are aligned for it.
static bool runs_aligned(awo_grid g, const void* heights, size_t heights_align, const void* a, const void* b,
                         const void* c, const void* d, const void* mask)
{
    const uintptr_t p = (uintptr_t)a | (uintptr_t)b | (uintptr_t)c | (uintptr_t)d;
    return (g.width % 4) == 0 && ((uintptr_t)heights & (heights_align - 1)) == 0 && (p & 15u) == 0 &&
           ((uintptr_t)mask & 3u) == 0;
}

template <bool FROM_U16>
static awo_status launch_normals(const NormalsArgs<FROM_U16>& a, awo_grid g, bool aligned, cudaStream_t s)
{
    const int64_t n = cells_of(g);
    if (aligned)
        k_normals_tiles<FROM_U16><<<(unsigned)((n + RT_TILE - 1) / RT_TILE), RT_THREADS, 0, s>>>(a, 0.0f, 0.0f, nullptr,
                                                                                                 nullptr);
    else {
        // a quarter of a tile a block while whole tiles would leave SMs with few blocks (501 x 151: parabola
        // workflow 125.7 -> 122.2 us; 3001 x 2999 the other way round 75.2 -> 69.2 us)
        const int64_t span = n >= (int64_t)sm_count() * 4 * RT_TILE ? RT_TILE : RT_TILE / 4;
        k_normals_cells<FROM_U16><<<(unsigned)((n + span - 1) / span), NC_THREADS, 0, s>>>(a, (uint32_t)span, 0.0f,
                                                                                          0.0f, nullptr, nullptr);
    }
    return launch_status();
}

extern "C" awo_status awo_normals(const float* d_h, awo_grid g, float* d_normal, float* d_tan2,
                                  float* d_slope_deg, void* stream)
{
    if (!d_h || !grid_ok(g)) return AWO_EINVAL;
    if (!d_normal && !d_tan2 && !d_slope_deg) return AWO_OK;
    return launch_normals(NormalsArgs<false>{{d_h, 1.0f}, g.width, g.height, g.cell_size, d_normal, d_tan2, d_slope_deg,
                                             nullptr},
                          g, runs_aligned(g, d_h, 16, d_normal, d_tan2, d_slope_deg, nullptr, nullptr), as_stream(stream));
}

extern "C" awo_status awo_normals_u16(const uint16_t* d_q, awo_grid g, float scale, float* d_h, float* d_normal,
                                      float* d_tan2, float* d_slope_deg, void* stream)
{
    if (!d_q || !d_h || !grid_ok(g) || !(scale > 0.0f) || !(scale < 3.0e38f)) return AWO_EINVAL;
    if (!d_normal && !d_tan2 && !d_slope_deg) return awo_decode_u16(d_q, g, scale, d_h, stream);
    return launch_normals(
        NormalsArgs<true>{{d_q, scale}, g.width, g.height, g.cell_size, d_normal, d_tan2, d_slope_deg, d_h}, g,
        runs_aligned(g, d_q, 8, d_normal, d_tan2, d_slope_deg, d_h, nullptr), as_stream(stream));
}

// The release passes after the tile counts: their offsets (a scan of its own
// above SUM_TILES_MAX tiles) and the ordered scatter from the mask (1 byte per
// cell instead of 4) or, without one, from tan^2.
static void scan_and_scatter(const float* d_tan2, const uint8_t* d_mask, int64_t n, int tiles, float t_lo, float t_hi,
                             const uint32_t* tile_count, uint32_t* tile_offset, uint32_t* d_cells, uint32_t* d_n,
                             cudaStream_t s)
{
    const bool sum = tiles <= SUM_TILES_MAX;
    if (!sum) k_release_scan<<<1, 1024, 0, s>>>(tile_count, tiles, tile_offset, d_n);
    const uint32_t* base = sum ? tile_count : tile_offset;
    if (d_mask) {
        auto kern = sum ? k_mask_scatter<true> : k_mask_scatter<false>;
        kern<<<(tiles + SC_RUNS - 1) / SC_RUNS, RT_THREADS, 0, s>>>(d_mask, n, base, d_cells, d_n);
    } else {
        auto kern = sum ? k_release_scatter<true> : k_release_scatter<false>;
        kern<<<tiles, RT_THREADS, 0, s>>>(d_tan2, n, t_lo, t_hi, base, d_cells, d_n);
    }
}

extern "C" size_t awo_release_workspace_bytes(awo_grid g)
{
    if (!grid_ok(g)) return 0;
    int64_t tiles = (cells_of(g) + RT_TILE - 1) / RT_TILE;
    return (size_t)(2 * tiles * sizeof(uint32_t) + 256);
}

// The checks of awo_release on its arguments (the heights' are made by the caller).
static awo_status release_args(const float* d_tan2, awo_grid g, double lo, double hi, const uint32_t* d_cells,
                               const uint32_t* d_n, const void* d_ws, size_t ws_bytes)
{
    if (!d_tan2 || !d_cells || !d_n || !d_ws || !grid_ok(g)) return AWO_EINVAL;
    if (!(lo >= 0.0) || !(hi < 90.0) || lo > hi) return AWO_EINVAL;
    if ((((uintptr_t)d_ws) & 15u) != 0) return AWO_EINVAL;
    return ws_bytes < awo_release_workspace_bytes(g) ? AWO_ENOMEM : AWO_OK;
}

extern "C" awo_status awo_release(const float* d_tan2, awo_grid g, double slope_lo_deg, double slope_hi_deg,
                                  uint8_t* d_mask, uint32_t* d_cells, uint32_t* d_n, void* d_ws, size_t ws_bytes,
                                  void* stream)
{
    const awo_status st = release_args(d_tan2, g, slope_lo_deg, slope_hi_deg, d_cells, d_n, d_ws, ws_bytes);
    if (st != AWO_OK) return st;
    const int64_t n = cells_of(g);
    const int tiles = (int)((n + RT_TILE - 1) / RT_TILE);
    uint32_t* tile_count = static_cast<uint32_t*>(d_ws);
    uint32_t* tile_offset = tile_count + tiles;
    const float t_lo = tan2_of_degrees(slope_lo_deg), t_hi = tan2_of_degrees(slope_hi_deg);
    cudaStream_t s = as_stream(stream);
    k_release_mask<<<tiles, RT_THREADS, 0, s>>>(d_tan2, n, t_lo, t_hi, d_mask, tile_count);
    scan_and_scatter(d_tan2, d_mask, n, tiles, t_lo, t_hi, tile_count, tile_offset, d_cells, d_n, s);
    return launch_status();
}

// a0 + a1 + b, with the release mask and counts taken in the normals' pass.
template <bool FROM_U16>
static awo_status normals_release(const NormalsArgs<FROM_U16>& a, awo_grid g, bool aligned, double lo, double hi,
                                  uint8_t* d_mask, uint32_t* d_cells, uint32_t* d_n, void* d_ws, cudaStream_t s)
{
    const int64_t n = cells_of(g);
    const int tiles = (int)((n + RT_TILE - 1) / RT_TILE);
    uint32_t* tile_count = static_cast<uint32_t*>(d_ws);
    const float t_lo = tan2_of_degrees(lo), t_hi = tan2_of_degrees(hi);
    if (aligned)
        k_normals_tiles<FROM_U16><<<tiles, RT_THREADS, 0, s>>>(a, t_lo, t_hi, d_mask, tile_count);
    else
        k_normals_cells<FROM_U16><<<tiles, NC_THREADS, 0, s>>>(a, (uint32_t)RT_TILE, t_lo, t_hi, d_mask, tile_count);
    scan_and_scatter(a.tan2, d_mask, n, tiles, t_lo, t_hi, tile_count, tile_count + tiles, d_cells, d_n, s);
    return launch_status();
}

extern "C" awo_status awo_normals_release(const float* d_h, awo_grid g, float* d_normal, float* d_tan2,
                                          float* d_slope_deg, double slope_lo_deg, double slope_hi_deg,
                                          uint8_t* d_mask, uint32_t* d_cells, uint32_t* d_n, void* d_ws,
                                          size_t ws_bytes, void* stream)
{
    if (!d_h) return AWO_EINVAL;
    const awo_status st = release_args(d_tan2, g, slope_lo_deg, slope_hi_deg, d_cells, d_n, d_ws, ws_bytes);
    if (st != AWO_OK) return st;
    return normals_release(
        NormalsArgs<false>{{d_h, 1.0f}, g.width, g.height, g.cell_size, d_normal, d_tan2, d_slope_deg, nullptr}, g,
        runs_aligned(g, d_h, 16, d_normal, d_tan2, d_slope_deg, nullptr, d_mask), slope_lo_deg, slope_hi_deg, d_mask,
        d_cells, d_n, d_ws, as_stream(stream));
}

extern "C" awo_status awo_normals_u16_release(const uint16_t* d_q, awo_grid g, float scale, float* d_h, float* d_normal,
                                              float* d_tan2, float* d_slope_deg, double slope_lo_deg,
                                              double slope_hi_deg, uint8_t* d_mask, uint32_t* d_cells, uint32_t* d_n,
                                              void* d_ws, size_t ws_bytes, void* stream)
{
    if (!d_q || !d_h || !(scale > 0.0f) || !(scale < 3.0e38f)) return AWO_EINVAL;
    const awo_status st = release_args(d_tan2, g, slope_lo_deg, slope_hi_deg, d_cells, d_n, d_ws, ws_bytes);
    if (st != AWO_OK) return st;
    return normals_release(
        NormalsArgs<true>{{d_q, scale}, g.width, g.height, g.cell_size, d_normal, d_tan2, d_slope_deg, d_h}, g,
        runs_aligned(g, d_q, 8, d_normal, d_tan2, d_slope_deg, d_h, d_mask), slope_lo_deg, slope_hi_deg, d_mask,
        d_cells, d_n, d_ws, as_stream(stream));
}

// ---------------------------------------------------------------------------
// Release selection with a scratch array inside the library, for callers that
// cannot pass a workspace (see awo_release_noalloc in awo.h).  The array holds
// the tile counts and tile offsets of the three passes for grids up to
// AWO_RELEASE_NOALLOC_MAX_CELLS cells.
// ---------------------------------------------------------------------------
namespace awo {

constexpr int NOALLOC_MAX_TILES = (int)(AWO_RELEASE_NOALLOC_MAX_CELLS / RT_TILE);
static __device__ __align__(256) uint32_t g_release_scratch[2 * NOALLOC_MAX_TILES];

// Device address of g_release_scratch for the current device.  In host code
// the symbol name is only a host-side stand-in, so the address is looked up
// once per device with cudaGetSymbolAddress while that device is current.
static awo_status noalloc_scratch(uint32_t** out)
{
    static std::mutex mu;
    static std::vector<uint32_t*> addr;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return AWO_ECUDA;
    std::lock_guard<std::mutex> lock(mu);
    if ((int)addr.size() <= dev) addr.resize(dev + 1, nullptr);
    if (addr[dev] == nullptr) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_release_scratch) != cudaSuccess || p == nullptr) {
            cudaGetLastError();
            return AWO_ECUDA;
        }
        addr[dev] = static_cast<uint32_t*>(p);
    }
    *out = addr[dev];
    return AWO_OK;
}

}  // namespace awo

extern "C" awo_status awo_release_noalloc(const float* d_tan2, awo_grid g, double slope_lo_deg, double slope_hi_deg,
                                          uint8_t* d_mask, uint32_t* d_cells, uint32_t* d_n, void* stream)
{
    if (!d_tan2 || !d_cells || !d_n || !grid_ok(g)) return AWO_EINVAL;
    if (!(slope_lo_deg >= 0.0) || !(slope_hi_deg < 90.0) || slope_lo_deg > slope_hi_deg) return AWO_EINVAL;
    const int64_t n = cells_of(g);
    if (n > AWO_RELEASE_NOALLOC_MAX_CELLS) return AWO_ENOMEM;
    uint32_t* scratch = nullptr;
    awo_status st = noalloc_scratch(&scratch);
    if (st != AWO_OK) return st;
    const int tiles = (int)((n + RT_TILE - 1) / RT_TILE);
    uint32_t* tile_count = scratch;
    uint32_t* tile_offset = scratch + NOALLOC_MAX_TILES;
    const float t_lo = tan2_of_degrees(slope_lo_deg), t_hi = tan2_of_degrees(slope_hi_deg);
    cudaStream_t s = as_stream(stream);
    k_release_mask<<<tiles, RT_THREADS, 0, s>>>(d_tan2, n, t_lo, t_hi, d_mask, tile_count);
    scan_and_scatter(d_tan2, d_mask, n, tiles, t_lo, t_hi, tile_count, tile_offset, d_cells, d_n, s);
    return launch_status();
}

extern "C" awo_status awo_release_from_mask(const uint8_t* d_mask, awo_grid g, uint32_t* d_cells, uint32_t* d_n,
                                            void* d_ws, size_t ws_bytes, void* stream)
{
    if (!d_mask || !d_cells || !d_n || !d_ws || !grid_ok(g)) return AWO_EINVAL;
    if ((((uintptr_t)d_ws) & 15u) != 0) return AWO_EINVAL;
    if (ws_bytes < awo_release_workspace_bytes(g)) return AWO_ENOMEM;
    const int64_t n = cells_of(g);
    const int tiles = (int)((n + RT_TILE - 1) / RT_TILE);
    uint32_t* tile_count = static_cast<uint32_t*>(d_ws);
    uint32_t* tile_offset = tile_count + tiles;
    cudaStream_t s = as_stream(stream);
    k_mask_count<<<tiles, RT_THREADS, 0, s>>>(d_mask, n, tile_count);
    scan_and_scatter(nullptr, d_mask, n, tiles, 0.0f, 0.0f, tile_count, tile_offset, d_cells, d_n, s);
    return launch_status();
}

// ---------------------------------------------------------------------------
// b''. Release points on a texture of chosen resolution: mask and tile counts
// in one pass, then the scan and the ordered scatter of the mask's texels.
// ---------------------------------------------------------------------------
extern "C" awo_status awo_release_texture_dims(awo_grid g, int32_t release_log2, int32_t* width, int32_t* height)
{
    int64_t wr, hr;
    if (!width || !height || !release_texture_dims(g, release_log2, &wr, &hr)) return AWO_EINVAL;
    *width = (int32_t)wr;
    *height = (int32_t)hr;
    return AWO_OK;
}

extern "C" size_t awo_release_texture_workspace_bytes(awo_grid g, int32_t release_log2)
{
    int64_t wr, hr;
    if (!release_texture_dims(g, release_log2, &wr, &hr)) return 0;
    const int64_t tiles = (wr * hr + RT_TILE - 1) / RT_TILE;
    return (size_t)(2 * tiles * sizeof(uint32_t) + 256);
}

extern "C" awo_status awo_release_texture(const float* d_tan2, awo_grid g, int32_t release_log2, double slope_lo_deg,
                                          double slope_hi_deg, uint8_t* d_mask, uint32_t* d_texels, uint32_t* d_n,
                                          void* d_ws, size_t ws_bytes, void* stream)
{
    int64_t wr, hr;
    if (!d_tan2 || !d_mask || !d_texels || !d_n || !d_ws || !release_texture_dims(g, release_log2, &wr, &hr))
        return AWO_EINVAL;
    if (!(slope_lo_deg >= 0.0) || !(slope_hi_deg < 90.0) || slope_lo_deg > slope_hi_deg) return AWO_EINVAL;
    if ((((uintptr_t)d_ws) & 15u) != 0) return AWO_EINVAL;
    if (ws_bytes < awo_release_texture_workspace_bytes(g, release_log2)) return AWO_ENOMEM;
    const int64_t n = wr * hr;
    const int tiles = (int)((n + RT_TILE - 1) / RT_TILE);
    uint32_t* tile_count = static_cast<uint32_t*>(d_ws);
    uint32_t* tile_offset = tile_count + tiles;
    const float t_lo = tan2_of_degrees(slope_lo_deg), t_hi = tan2_of_degrees(slope_hi_deg);
    const float scale = ldexpf(1.0f, -release_log2);
    cudaStream_t s = as_stream(stream);
    // float4 reads of tan2 rows: base 16-byte aligned and W a multiple of 4,
    // so that every row and every run start (a multiple of 16 / 2^r cells) is
    const bool vec = (((uintptr_t)d_tan2) & 15u) == 0 && (g.width & 3) == 0;
    if ((release_log2 == 1 || release_log2 == 2) && g.height >= 2 && g.height < 65535 && wr % RT_TILE == 0) {
        // rows are whole tiles: one launch of row groups that share their tan^2 rows
        const dim3 grid((unsigned)(wr / RT_TILE), (unsigned)g.height + 1u);  // at most 65535 groups
        if (release_log2 == 1) {
            if (vec)
                k_release_texture_rows<1, true><<<grid, RT_THREADS, 0, s>>>(d_tan2, g.width, g.height, (uint32_t)wr,
                                                                           n, scale, t_lo, t_hi, d_mask, tile_count);
            else
                k_release_texture_rows<1, false><<<grid, RT_THREADS, 0, s>>>(d_tan2, g.width, g.height, (uint32_t)wr,
                                                                            n, scale, t_lo, t_hi, d_mask, tile_count);
        } else {
            if (vec)
                k_release_texture_rows<2, true><<<grid, RT_THREADS, 0, s>>>(d_tan2, g.width, g.height, (uint32_t)wr,
                                                                           n, scale, t_lo, t_hi, d_mask, tile_count);
            else
                k_release_texture_rows<2, false><<<grid, RT_THREADS, 0, s>>>(d_tan2, g.width, g.height, (uint32_t)wr,
                                                                            n, scale, t_lo, t_hi, d_mask, tile_count);
        }
    } else if (release_log2 < 0) {
        k_release_texture_texels<<<tiles, NC_THREADS, 0, s>>>(d_tan2, g.width, g.height, (uint32_t)wr, (uint32_t)n, scale,
                                                              t_lo, t_hi, d_mask, tile_count);
    } else {
        auto kern = release_log2 == 0   ? (vec ? k_release_texture_mask<0, true> : k_release_texture_mask<0, false>)
                    : release_log2 == 1 ? (vec ? k_release_texture_mask<1, true> : k_release_texture_mask<1, false>)
                    : release_log2 == 2 ? (vec ? k_release_texture_mask<2, true> : k_release_texture_mask<2, false>)
                                        : k_release_texture_mask<3, false>;
        kern<<<tiles, RT_THREADS, 0, s>>>(d_tan2, g.width, g.height, (uint32_t)wr, n, scale, t_lo, t_hi, d_mask,
                                          tile_count);
    }
    scan_and_scatter(nullptr, d_mask, n, tiles, 0.0f, 0.0f, tile_count, tile_offset, d_texels, d_n, s);
    return launch_status();
}
