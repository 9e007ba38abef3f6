// awo_overlay.cu -- velocity indicator and overlay mipmap (Sec. 3, Fig. 4).
//
// Both are streaming passes.  Six levels of the mipmap come from one kernel:
// a block reduces its 64 x 64 tile of level 0 to level 1 and then, in shared
// memory, to each further level (counts summed in 64 bits and saturated,
// velocities by max), so level 0 is read once and every level written once;
// deeper levels come from the sixth in the same way.  The
// workflow's call also makes the velocity from the maximum energy inside the
// same pass (awo_finalize_lod).
#include <string.h>

#include "awo_internal.cuh"

namespace awo {

// vel = sqrt((2 g) maxe); float4 loads and stores when both rasters are
// 16-byte aligned, then a scalar tail.  A thread issues the loads of
// STREAM_UNROLL float4 (each coalesced across the grid) before their stores,
// so that enough bytes are in flight per SM to keep HBM busy.
constexpr int STREAM_UNROLL = 4;

__global__ void k_finalize(const float* __restrict__ maxe, int64_t n, float g2, float* __restrict__ vel, bool vec4)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t n4 = vec4 ? n / 4 : 0;
    for (int64_t q = tid; q < n4; q += STREAM_UNROLL * stride) {
        float4 m[STREAM_UNROLL];
#pragma unroll
        for (int u = 0; u < STREAM_UNROLL; ++u) {
            const int64_t k = q + u * stride;
            m[u] = k < n4 ? __ldg(reinterpret_cast<const float4*>(maxe) + k) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int u = 0; u < STREAM_UNROLL; ++u) {
            const int64_t k = q + u * stride;
            if (k < n4)
                reinterpret_cast<float4*>(vel)[k] =
                    make_float4(__fsqrt_rn(__fmul_rn(g2, m[u].x)), __fsqrt_rn(__fmul_rn(g2, m[u].y)),
                                __fsqrt_rn(__fmul_rn(g2, m[u].z)), __fsqrt_rn(__fmul_rn(g2, m[u].w)));
        }
    }
    for (int64_t i = 4 * n4 + tid; i < n; i += stride) vel[i] = __fsqrt_rn(__fmul_rn(g2, maxe[i]));
}

// Levels 1 .. 1 + LOD_FUSED - 1 of the mipmap in one pass over level 0.  A
// block owns a 32 x 32 tile of level 1 (a 64 x 64 tile of level 0) and all
// its descendants: 16 x 16 of level 2, ... 1 x 1 of level 6, since the tiles
// of every level nest.  Level 1 is reduced from level 0 in global memory,
// each further level from the previous one in shared memory; every texel is
// the saturating count sum and the velocity maximum of its existing children
// (children past a level's edge are ignored).  One read of
// level 0 and one write of each level, instead of a read and a write per
// level with a launch each.  FROM_MAXE: level 0's velocity is not read but
// made from the maximum energy as it is needed, vel = sqrt((2 g) maxe), and
// written (awo_finalize fused in): each level-0 cell is the child of exactly
// one level-1 texel, so each is computed and written once.
// Bound by HBM: 8192^2, velocity and a full chain 187 -> 166 us (984 MB, 88% of
// the copy rate) with 16-byte loads, two level-1 texels a thread and row, where
// rows are whole groups of four; 8-byte ones for other even rows.  Odd rows take
// single cells, whose loads do not wait for one another: 5003 x 4099, 8 levels,
// 68.4 -> 55.3 us (with a branch before each load the one texel a thread of the
// second launch took 4.8 us; a kernel of its own, one texel a thread, 2.3).
constexpr int LOD_TILE = 32;   // level-1 tile side
constexpr int LOD_FUSED = 6;   // levels a block can finish: 32, 16, 8, 4, 2, 1

struct LodArgs {
    const uint32_t* c0;
    const float* v0;  // level-0 velocity, or the maximum energy when FROM_MAXE
    float* vel0;      // FROM_MAXE: level-0 velocity out (may alias v0)
    float g2;         // FROM_MAXE: 2 g
    int w[LOD_FUSED + 1], h[LOD_FUSED + 1];  // level sizes 0 .. LOD_FUSED
    uint32_t* c[LOD_FUSED];                  // outputs of levels 1 .. LOD_FUSED
    float* v[LOD_FUSED];
    int n_out;                               // levels written, 1 .. LOD_FUSED
    bool vec2;                               // level-0 child pairs as uint2 / float2
    bool vec4;                               // two of them as uint4 / float4, their results as uint2 / float2
};

template <bool FROM_MAXE>
__device__ __forceinline__ float2 lod_vel0_pair(const LodArgs& a, uint32_t i)
{
    const float2 x = __ldg(reinterpret_cast<const float2*>(a.v0 + i));
    if (!FROM_MAXE) return x;
    const float2 v = make_float2(__fsqrt_rn(__fmul_rn(a.g2, x.x)), __fsqrt_rn(__fmul_rn(a.g2, x.y)));
    *reinterpret_cast<float2*>(a.vel0 + i) = v;
    return v;
}

template <bool FROM_MAXE>
__device__ __forceinline__ float4 lod_vel0_four(const LodArgs& a, uint32_t i)
{
    const float4 x = __ldg(reinterpret_cast<const float4*>(a.v0 + i));
    if (!FROM_MAXE) return x;
    const float4 v = make_float4(__fsqrt_rn(__fmul_rn(a.g2, x.x)), __fsqrt_rn(__fmul_rn(a.g2, x.y)),
                                 __fsqrt_rn(__fmul_rn(a.g2, x.z)), __fsqrt_rn(__fmul_rn(a.g2, x.w)));
    *reinterpret_cast<float4*>(a.vel0 + i) = v;
    return v;
}

__device__ __forceinline__ uint32_t saturated(unsigned long long sum)
{
    return sum > 0xFFFFFFFFull ? 0xFFFFFFFFu : (uint32_t)sum;
}

template <bool FROM_MAXE>
__global__ void __launch_bounds__(256) k_lod_fused(const __grid_constant__ LodArgs a)
{
    __shared__ uint32_t sc[2][LOD_TILE][LOD_TILE + 1];
    __shared__ float sv[2][LOD_TILE][LOD_TILE + 1];
    const int tid = threadIdx.x, tx = tid & 31, ty = tid >> 5;
    const int bx = blockIdx.x, by = blockIdx.y;
    // level 1 from level 0
    if (a.vec4) {  // two texels a thread and row: w0 a multiple of 4, so both exist or neither
        const int w0 = a.w[0], h0 = a.h[0], w1 = a.w[1], h1 = a.h[1];
        const int x = 2 * (tid & 15), X = bx * LOD_TILE + x;
#pragma unroll
        for (int k = 0; k < LOD_TILE / 16; ++k) {
            const int y = (tid >> 4) + 16 * k, Y = by * LOD_TILE + y;
            if (X < w1 && Y < h1) {
                const uint32_t r0 = (uint32_t)(2 * Y) * (uint32_t)w0 + (uint32_t)(2 * X);
                const uint4 c_0 = __ldg(reinterpret_cast<const uint4*>(a.c0 + r0));
                const float4 v_0 = lod_vel0_four<FROM_MAXE>(a, r0);
                unsigned long long sl = (unsigned long long)c_0.x + c_0.y, sr = (unsigned long long)c_0.z + c_0.w;
                float ml = fmaxf(v_0.x, v_0.y), mr = fmaxf(v_0.z, v_0.w);
                if (2 * Y + 1 < h0) {
                    const uint32_t r1 = r0 + (uint32_t)w0;
                    const uint4 c_1 = __ldg(reinterpret_cast<const uint4*>(a.c0 + r1));
                    const float4 v_1 = lod_vel0_four<FROM_MAXE>(a, r1);
                    sl += (unsigned long long)c_1.x + c_1.y;
                    sr += (unsigned long long)c_1.z + c_1.w;
                    ml = fmaxf(ml, fmaxf(v_1.x, v_1.y));
                    mr = fmaxf(mr, fmaxf(v_1.z, v_1.w));
                }
                const uint2 c = make_uint2(saturated(sl), saturated(sr));
                const uint32_t o = (uint32_t)Y * (uint32_t)w1 + (uint32_t)X;  // even: w1 and X are
                *reinterpret_cast<uint2*>(a.c[0] + o) = c;
                *reinterpret_cast<float2*>(a.v[0] + o) = make_float2(ml, mr);
                sc[0][y][x] = c.x;
                sc[0][y][x + 1] = c.y;
                sv[0][y][x] = ml;
                sv[0][y][x + 1] = mr;
            }
        }
    } else {  // four texels per thread, rows ty, ty + 8, ...
        const int w0 = a.w[0], h0 = a.h[0], w1 = a.w[1], h1 = a.h[1];
        const int X = bx * LOD_TILE + tx;
#pragma unroll
        for (int k = 0; k < LOD_TILE / 8; ++k) {
            const int y = ty + 8 * k, Y = by * LOD_TILE + y;
            if (X < w1 && Y < h1) {
                const int sx = 2 * X, sy = 2 * Y;
                const bool hx = sx + 1 < w0, hy = sy + 1 < h0;
                const uint32_t r0 = (uint32_t)sy * (uint32_t)w0 + (uint32_t)sx, r1 = r0 + (uint32_t)w0;
                unsigned long long sum;
                float m;
                if (a.vec2) {  // w0 even: both columns exist and the pair is 8-byte aligned
                    const uint2 c_0 = __ldg(reinterpret_cast<const uint2*>(a.c0 + r0));
                    const float2 v_0 = lod_vel0_pair<FROM_MAXE>(a, r0);
                    sum = (unsigned long long)c_0.x + c_0.y;
                    m = fmaxf(v_0.x, v_0.y);
                    if (hy) {
                        const uint2 c_1 = __ldg(reinterpret_cast<const uint2*>(a.c0 + r1));
                        const float2 v_1 = lod_vel0_pair<FROM_MAXE>(a, r1);
                        sum += (unsigned long long)c_1.x + c_1.y;
                        m = fmaxf(m, fmaxf(v_1.x, v_1.y));
                    }
                } else {
                    // a child past the edge is the one before it again (the same maximum, not added), so that
                    // no load waits for a branch
                    const uint32_t i01 = r0 + (hx ? 1u : 0u), i10 = hy ? r1 : r0, i11 = i10 + (hx ? 1u : 0u);
                    const uint32_t c00 = __ldg(a.c0 + r0), c01 = __ldg(a.c0 + i01), c10 = __ldg(a.c0 + i10),
                                   c11 = __ldg(a.c0 + i11);
                    float v00 = __ldg(a.v0 + r0), v01 = __ldg(a.v0 + i01), v10 = __ldg(a.v0 + i10),
                          v11 = __ldg(a.v0 + i11);
                    if (FROM_MAXE) {
                        v00 = __fsqrt_rn(__fmul_rn(a.g2, v00));
                        v01 = __fsqrt_rn(__fmul_rn(a.g2, v01));
                        v10 = __fsqrt_rn(__fmul_rn(a.g2, v10));
                        v11 = __fsqrt_rn(__fmul_rn(a.g2, v11));
                        a.vel0[r0] = v00;
                        if (hx) a.vel0[i01] = v01;
                        if (hy) a.vel0[i10] = v10;
                        if (hx && hy) a.vel0[i11] = v11;
                    }
                    sum = (unsigned long long)c00 + (hx ? c01 : 0u) + (hy ? c10 : 0u);
                    sum += hx && hy ? c11 : 0u;
                    m = fmaxf(fmaxf(v00, v01), fmaxf(v10, v11));
                }
                const uint32_t c = saturated(sum);
                const uint32_t o = (uint32_t)Y * (uint32_t)w1 + (uint32_t)X;
                a.c[0][o] = c;
                a.v[0][o] = m;
                sc[0][y][tx] = c;
                sv[0][y][tx] = m;
            }
        }
    }
    // levels 2 .. n_out from the previous level in shared memory
    int t = LOD_TILE, src = 0;
    for (int l = 2; l <= a.n_out; ++l) {
        __syncthreads();
        const int t2 = t >> 1;
        if (tid < t2 * t2) {
            const int x = tid % t2, y = tid / t2;
            const int X = bx * t2 + x, Y = by * t2 + y;
            if (X < a.w[l] && Y < a.h[l]) {
                const int wp = a.w[l - 1], hp = a.h[l - 1];
                const bool hx = 2 * X + 1 < wp, hy = 2 * Y + 1 < hp;
                unsigned long long sum = sc[src][2 * y][2 * x];
                float m = sv[src][2 * y][2 * x];
                if (hx) {
                    sum += sc[src][2 * y][2 * x + 1];
                    m = fmaxf(m, sv[src][2 * y][2 * x + 1]);
                }
                if (hy) {
                    sum += sc[src][2 * y + 1][2 * x];
                    m = fmaxf(m, sv[src][2 * y + 1][2 * x]);
                    if (hx) {
                        sum += sc[src][2 * y + 1][2 * x + 1];
                        m = fmaxf(m, sv[src][2 * y + 1][2 * x + 1]);
                    }
                }
                const uint32_t c = saturated(sum);
                const uint32_t o = (uint32_t)Y * (uint32_t)a.w[l] + (uint32_t)X;
                a.c[l - 1][o] = c;
                a.v[l - 1][o] = m;
                sc[src ^ 1][y][x] = c;
                sv[src ^ 1][y][x] = m;
            }
        }
        src ^= 1;
        t = t2;
    }
}

}  // namespace awo

using namespace awo;

extern "C" awo_status awo_finalize(const float* d_maxe, awo_grid g, float gravity, float* d_vel, void* stream)
{
    if (!d_maxe || !d_vel || !grid_ok(g) || !(gravity > 0.0f) || !(gravity < 1.0e38f)) return AWO_EINVAL;
    const int64_t n = cells_of(g);
    const bool vec4 = ((((uintptr_t)d_maxe) | ((uintptr_t)d_vel)) & 15u) == 0;
    k_finalize<<<stream_blocks(vec4 ? n / 4 + 1 : n, 256), 256, 0, as_stream(stream)>>>(d_maxe, n, 2.0f * gravity,
                                                                                        d_vel, vec4);
    return launch_status();
}

// Levels 1 .. levels-1 from level 0 = (d_count, v0): a fused launch for every
// LOD_FUSED levels, each from the last level of the one before (a launch for
// each level past the sixth took 2.6-3.2 us a level, 20 us of the 375 us of a
// full 8192^2 chain and its colouring).  from_maxe: v0 is the maximum energy
// and level 0's velocity is written to d_vel (g2 = 2 g).
static awo_status lod_levels(const uint32_t* d_count, const float* v0, bool from_maxe, float g2, float* d_vel,
                             awo_grid g, int32_t levels, uint32_t* const* d_count_lv, float* const* d_vel_lv,
                             cudaStream_t s)
{
    int w = g.width, h = g.height;
    for (int done = 0; done + 1 < levels; done += LOD_FUSED, from_maxe = false) {
        LodArgs a;
        memset(&a, 0, sizeof(a));
        a.c0 = done ? d_count_lv[done - 1] : d_count;
        a.v0 = done ? d_vel_lv[done - 1] : v0;
        a.vel0 = d_vel;
        a.g2 = g2;
        a.n_out = levels - 1 - done < LOD_FUSED ? levels - 1 - done : LOD_FUSED;
        a.w[0] = w;
        a.h[0] = h;
        for (int k = 1; k <= a.n_out; ++k) {
            a.w[k] = (a.w[k - 1] + 1) / 2;
            a.h[k] = (a.h[k - 1] + 1) / 2;
            a.c[k - 1] = d_count_lv[done + k - 1];
            a.v[k - 1] = d_vel_lv[done + k - 1];
        }
        a.vec2 = w % 2 == 0 &&
                 ((((uintptr_t)a.c0) | ((uintptr_t)a.v0) | (from_maxe ? (uintptr_t)d_vel : (uintptr_t)0)) & 7u) == 0;
        a.vec4 = w % 4 == 0 &&
                 ((((uintptr_t)a.c0) | ((uintptr_t)a.v0) | (from_maxe ? (uintptr_t)d_vel : (uintptr_t)0)) & 15u) == 0 &&
                 ((((uintptr_t)a.c[0]) | ((uintptr_t)a.v[0])) & 7u) == 0;
        const dim3 grid((unsigned)((a.w[1] + LOD_TILE - 1) / LOD_TILE), (unsigned)((a.h[1] + LOD_TILE - 1) / LOD_TILE));
        if (from_maxe)
            k_lod_fused<true><<<grid, 256, 0, s>>>(a);
        else
            k_lod_fused<false><<<grid, 256, 0, s>>>(a);
        const awo_status st = launch_status();
        if (st != AWO_OK) return st;
        w = a.w[a.n_out];
        h = a.h[a.n_out];
    }
    return AWO_OK;
}

extern "C" awo_status awo_overlay_lod(const uint32_t* d_count, const float* d_vel, awo_grid g, int32_t levels,
                                      uint32_t* const* d_count_lv, float* const* d_vel_lv, void* stream)
{
    if (!d_count || !d_vel || !grid_ok(g) || levels < 1 || levels > 16) return AWO_EINVAL;
    if (levels > 1 && (!d_count_lv || !d_vel_lv)) return AWO_EINVAL;
    for (int l = 0; l + 1 < levels; ++l)
        if (!d_count_lv[l] || !d_vel_lv[l]) return AWO_EINVAL;
    if (levels == 1) return AWO_OK;
    return lod_levels(d_count, d_vel, false, 0.0f, nullptr, g, levels, d_count_lv, d_vel_lv, as_stream(stream));
}

extern "C" awo_status awo_finalize_lod(const float* d_maxe, const uint32_t* d_count, awo_grid g, float gravity,
                                       int32_t levels, float* d_vel, uint32_t* const* d_count_lv,
                                       float* const* d_vel_lv, void* stream)
{
    if (!d_maxe || !d_count || !d_vel || !grid_ok(g) || levels < 1 || levels > 16) return AWO_EINVAL;
    if (!(gravity > 0.0f) || !(gravity < 1.0e38f)) return AWO_EINVAL;
    if (levels > 1 && (!d_count_lv || !d_vel_lv)) return AWO_EINVAL;
    for (int l = 0; l + 1 < levels; ++l)
        if (!d_count_lv[l] || !d_vel_lv[l]) return AWO_EINVAL;
    if (levels == 1) return awo_finalize(d_maxe, g, gravity, d_vel, stream);
    return lod_levels(d_count, d_maxe, true, 2.0f * gravity, d_vel, g, levels, d_count_lv, d_vel_lv,
                      as_stream(stream));
}
