// awo_simulate.cu -- Monte-Carlo avalanche trajectories (Sec. 5.2).
//
// Design (GB300):
//  * Persistent kernel, one lane per particle.  The particles are numbered
//    cell-major (start record, then particle j); a warp takes a chunk of
//    consecutive particles at a time from a global counter (one atomic per
//    chunk) and walks it with a warp-uniform cursor (one integer division per
//    chunk, none per particle).  The chunk size (32 .. 1024 particles) follows
//    from the particle count and the grid, so that a release list of a few
//    cells is still spread over many warps.  The start records are in a
//    processing order that spreads consecutive blocks of release cells over
//    the grid (order_slot): the lanes of a warp work on neighbouring cells,
//    while the warps of the GPU work all over the grid and its memory
//    partitions.
//  * 32 particles start together and make their first two moves ("fresh"
//    pair); the survivors then run beside survivors of earlier starts, and
//    lanes whose particle ends take over a waiting one from the warp's pool in
//    shared memory (awo_particle.cuh, run_particles).
//  * A particle starts from the 16-byte start record of its release cell
//    (position, height, first move vector before its random part), written by
//    a prologue kernel that also records the release visits of all N
//    particles of the cell with one reduction.  Each loop iteration is two
//    moves and their visits from one Philox block (moves n and n + 1 take
//    words 0-1 and 2-3 of block n >> 1; live lanes are always at an even n
//    there) -- direction from the gradient kept in registers, step, footprint
//    and energy at the new position, record -- written without data-dependent
//    branches.
//  * Visits go to the rasters as fire-and-forget reductions (RED.ADD on the
//    count, RED.MAX on the bits of the non-negative energy, the latter only if
//    it can raise the maximum, where looking pays: check_pays).  Merging the
//    lanes of a warp that hit the same cell (__match_any_sync, at the first
//    move, at both moves of a fresh pair or at every move) was slower wherever
//    the look is taken (8192^2 18.2 against 17.6 ms, at every move 19.6).
//  * On grids of at least 2^19 cells the 2x2 footprint of a move is one
//    texture gather through a texture object that views the DEM's words
//    (clamp addressing is the footprint clamp; indices and weights are still
//    computed here), in place of four loads, their addresses and clamps.
//  * Arithmetic is FP32 with explicit round-to-nearest intrinsics: no fused
//    multiply-add that changes a rounding, IEEE sqrt and reciprocal, so every
//    particle follows the formulas of awo.h bit for bit.
//  * What bounds it: issue on the 8192^2 workload (82% of issue slots; 145-150
//    warp instructions per move of a warp, from 222), the visits' traffic to
//    the L2 and the footprint gathers' latency on the long-trajectory ones
//    (2048^2: 73% of issue slots, L2 62%, from 67% and 72%).  Measured and not
//    kept: the paired arithmetic of a move in packed FP32 (fma.rn.f32x2, its
//    products kept separately rounded by an addend of -0 that the compiler
//    cannot see): 17.1 against 17.2 ms; 40 registers for 12 blocks an SM: 17.4.
#include <math.h>
#include <string.h>

#include <mutex>

#include "awo_particle.cuh"

namespace awo {

constexpr int SIM_THREADS = 128, SIM_THREADS_MAX = 256;
constexpr uint32_t SIM_CHUNK_MAX = 1024;  // particles per global fetch, at most
// fetches a warp makes on an even split, at least: chunks of neighbouring
// cells carry similar work, so few large chunks leave some warps with much
// more of it (2048^2 workload: 4 -> 16 chunks a warp, 1.80 -> 1.72 ms)
constexpr uint32_t SIM_CHUNKS_PER_WARP = 16;

__device__ __forceinline__ uint32_t release_count(const SimArgs& a)
{
    uint32_t n = a.n_cells_max;
    if (a.n_cells_dev) n = min(n, *a.n_cells_dev);
    return n;
}

// Start of a call: the work counter and the statistics zeroed, and n words of
// both rasters (CLEAR_OUTPUTS; 0 otherwise) -- one launch where three memsets
// took three (2 us each between the kernels of a small call; at 8192^2 as fast
// as the memsets).
__global__ void __launch_bounds__(256) k_sim_clear(uint32_t* __restrict__ count, uint32_t* __restrict__ maxe, int64_t n,
                                                   SimWorkspace* ws, bool vec4)
{
    asm volatile("griddepcontrol.launch_dependents;");
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t n4 = vec4 ? n / 4 : 0;
    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
    for (int64_t q = tid; q < n4; q += stride) {
        reinterpret_cast<uint4*>(count)[q] = zero;
        reinterpret_cast<uint4*>(maxe)[q] = zero;
    }
    for (int64_t i = 4 * n4 + tid; i < n; i += stride) count[i] = maxe[i] = 0u;
    if (tid < 6) ws->stats.n[tid] = 0ull;
    if (tid == 6) ws->work.next_item = 0ull;
}

// End of a call: request blockIdx.x's statistics to the caller's array, byte
// by byte (of any alignment).  The kernels count in the workspace, so that the
// array holds the last call's statistics until this one's are complete.
__global__ void __launch_bounds__(64) k_sim_publish(const StatsCounters* from, unsigned char* stats)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");  // the particle kernel
    const unsigned i = threadIdx.x;
    if (i < sizeof(awo_sim_stats))
        stats[(size_t)blockIdx.x * sizeof(awo_sim_stats) + i] =
            reinterpret_cast<const unsigned char*>(from[blockIdx.x].n)[i];
}

awo_status publish_stats(const StatsCounters* from, awo_sim_stats* d_stats, int n, bool early, cudaStream_t s)
{
    return launch_kernel(k_sim_publish, (unsigned)n, 64u, 0, -1, early, s, from,
                         reinterpret_cast<unsigned char*>(d_stats)) == cudaSuccess
               ? launch_status()
               : AWO_ECUDA;
}

// Prologue: per release-list entry, the start record (at its slot in the
// processing order of awo_particle.cuh) and the release visit of all N particles (count +=
// N; their energy is 0, so the maximum is unchanged).  Grid-stride over the
// entries, whose number may be on the device.
// TEXELS: the entries are texels of the release texture.  It also counts the
// particles of entries outside the grid (rejected) and, when max_steps = 0
// (every particle capped at its release visit; the particle kernel is not
// launched), the particles and caps.
template <bool TEXELS>
__global__ void __launch_bounds__(256) k_sim_starts(const __grid_constant__ SimArgs a)
{
    const uint32_t n_cells = release_count(a);
    const uint32_t B = order_block(a.N);
    const uint32_t nb = n_cells / B;
    __shared__ uint32_t s_sinv;
    if (threadIdx.x == 0) s_sinv = order_stride_inverse(nb);
    asm volatile("griddepcontrol.launch_dependents;");
    asm volatile("griddepcontrol.wait;" ::: "memory");  // k_sim_clear
    __syncthreads();
    const uint32_t Sinv = s_sinv;
    // the slot of the thread's entries, advanced per grid stride G (a
    // multiple of B: B <= 32 divides the block size) instead of one 64-bit
    // modulo per entry: entry ci + G is in block ci / B + G / B, same offset
    const uint32_t G = gridDim.x * blockDim.x;
    const uint32_t ci0 = blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned long long step = nb ? ((unsigned long long)(G / B) * Sinv) % nb : 0ull;
    unsigned long long sb = nb ? ((unsigned long long)(ci0 / B) * Sinv) % nb : 0ull;
    unsigned long long good = 0ull, bad = 0ull;
    for (uint32_t ci = ci0; ci < n_cells; ci += G) {
        const uint32_t slot = ci < nb * B ? (uint32_t)sb * B + (ci & (B - 1u)) : ci;  // = order_slot(ci)
        sb += step;
        if (sb >= nb) sb -= nb;
        const uint32_t entry = __ldg(a.cells + ci);
        bool ok;
        if (TEXELS) {
            TexelStart st = texel_start(a.h, a.W, a.H, a.tg, entry);
            first_vector(st, a.P, a.oneP);
            ok = st.t != ~0u;
            if (ok) atomicAdd(a.count + st.vcell, a.N);
            static_cast<TexelStart*>(a.starts)[slot] = st;
        } else {
            CellStart st = cell_start(a.h, a.W, a.H, a.n_grid, entry);
            first_vector(st, a.P, a.oneP);
            ok = st.xy != ~0u;
            if (ok) atomicAdd(a.count + entry, a.N);
            static_cast<CellStart*>(a.starts)[slot] = st;
        }
        good += ok ? 1ull : 0ull;
        bad += ok ? 0ull : 1ull;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        good += __shfl_xor_sync(0xffffffffu, good, o);
        bad += __shfl_xor_sync(0xffffffffu, bad, o);
    }
    if ((threadIdx.x & 31) == 0) {
        if (bad) atomicAdd(&a.stats[5], bad * a.N);
        if (good && a.max_steps == 0u) {
            atomicAdd(&a.stats[1], good * a.N);
            atomicAdd(&a.stats[3], good * a.N);
        }
    }
}

// The particle kernel, in two instances per kind of record and footprint:
// with and without the look at a cell's maximum (CHECK).  Which one runs
// depends on the release count, which the host does not know, so both are
// launched and one of them ends at once (as one kernel that holds both loops,
// or with the choice as a predicate, the 8192^2 workload took 2% more).
//
// Every launch lets the next one start as soon as its blocks are resident
// (programmatic dependent launch), so the blocks of a batch's next launch
// fill the SMs as this one's warps run out of particles.  The last block of a
// launch does nothing but wait for the launch before it, so that a launch is
// complete only when all before it are, and what follows on the stream is
// ordered after every one.  (The same wait at the end of a working block cost
// 8 registers and 5% on the 8192^2 workload.)
template <bool TEXELS, bool TEX, bool PLAIN, bool CHECK>
__global__ void __launch_bounds__(SIM_THREADS_MAX) k_simulate(const __grid_constant__ SimArgs a)
{
    extern __shared__ uint32_t s_pool[];  // POOL_WORDS per warp
    asm volatile("griddepcontrol.launch_dependents;");
    const uint32_t blocks = gridDim.x - 1u;
    if (blockIdx.x == blocks) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        return;
    }
    const unsigned long long total = (unsigned long long)release_count(a) * a.N;
    const bool check = a.check ? *a.check != 0u : check_pays(total, a.look_min, a.n_grid);
    const uint32_t warp = threadIdx.x >> 5;
    // a few particles: one warp a block, so that they spread over the SMs
    // (parabola, 6144 particles: 149 -> 135 us)
    if (check == CHECK && total > 32ull * blocks * warp) {
        // particles of entries inside the grid (the prologue has counted the others)
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            const unsigned long long run = total - a.stats[5];
            a.stats[1] = run;
            atomicAdd(&a.stats[4], run);
        }
        // particles a warp takes per fetch: a multiple of 32 in [32,
        // SIM_CHUNK_MAX], about total / (warps * SIM_CHUNKS_PER_WARP)
        const unsigned long long even = total / ((unsigned long long)blocks * (blockDim.x >> 5) * SIM_CHUNKS_PER_WARP);
        uint32_t chunk = even > SIM_CHUNK_MAX ? SIM_CHUNK_MAX : max((uint32_t)even & ~31u, a.least_chunk);
        if (a.group) chunk = a.group;
        run_particles<TEXELS, TEX ? 1 : 0, CHECK, PLAIN>(a, total, chunk, a.min_idle, a.next_item, a.stats,
                                                  s_pool + warp * POOL_WORDS);
    }
}

template <bool TEXELS, bool TEX, bool PLAIN>
static awo_status launch_both(const SimArgs& a, int threads, bool after_particles, bool look, cudaStream_t s)
{
    const awo_status st = launch_persistent<k_simulate<TEXELS, TEX, PLAIN, true>>(a, threads, after_particles, s);
    return st != AWO_OK || look ? st : launch_persistent<k_simulate<TEXELS, TEX, PLAIN, false>>(a, threads, true, s);
}

awo_status launch_particles(const SimArgs& a, int threads, bool after_particles, bool look, cudaStream_t s)
{
    const bool plain = a.s == 1.0f && a.kD == 0.0f;
    auto launch = a.tg.texels ? (a.tex ? (plain ? launch_both<true, true, true> : launch_both<true, true, false>)
                                       : (plain ? launch_both<true, false, true> : launch_both<true, false, false>))
                              : (a.tex ? (plain ? launch_both<false, true, true> : launch_both<false, true, false>)
                                       : (plain ? launch_both<false, false, true> : launch_both<false, false, false>));
    return launch(a, threads, after_particles, look, s);
}

void sim_constants(SimArgs& a, const float* d_h, awo_grid g, const awo_sim_params* p, uint32_t* d_count, float* d_maxe,
                   cudaStream_t s)
{
    memset(&a, 0, sizeof(a));
    // each one FP32 rounding in the documented order
    const float D = p->step_scale * g.cell_size;
    a.h = d_h;
    a.count = d_count;
    a.maxe = d_maxe;
    a.W = g.width;
    a.H = g.height;
    a.n_grid = (uint32_t)cells_of(g);
    a.Wm1 = (float)(g.width - 1);
    a.Hm1 = (float)(g.height - 1);
    a.P = p->persistence;
    a.oneP = 1.0f - p->persistence;
    a.R = p->randomness;
    a.R23 = scaled_randomness(p->randomness);
    a.s = p->step_scale;
    a.kD = p->drag_k * D;
    a.muD = p->mu * D;
    a.N = p->traj_per_cell;
    a.max_steps = p->max_steps;
    a.keys = philox_keys(p->seed);
    int64_t wr = 0, hr = 0;
    release_texture_dims(g, p->release_log2, &wr, &hr);  // checked by sim_params_ok
    a.tg.Wr = (uint32_t)wr;
    a.tg.n_tex = (uint32_t)(wr * hr);
    a.tg.scale = ldexpf(1.0f, -p->release_log2);
    a.tg.texels = p->release_log2 != 0 ? 1u : 0u;
    a.tex = dem_texture(d_h, g, s);
    a.min_idle = 1u;
    a.least_chunk = 32u;
    a.look_min = look_paths(p->step_scale);
}

// Texture views of DEM buffers for the gathers of k_simulate: a texture
// object is a descriptor of (address, width, height, row pitch) -- no copy;
// the words are viewed as 32-bit unsigned texels, returned bit for bit --
// created on the first call with a buffer and kept for the life of the
// process (at most DEM_VIEWS_MAX of grids from DEM_VIEW_LARGE_CELLS and as
// many of smaller ones, so that these, which gain less, never take a large
// one's place; further buffers take the load path), so that a graph that
// captured a launch keeps a valid view.  A view needs the row pitch and the base
// address aligned to the device's texture pitch and texture alignments and a
// grid within the 2D pitch-linear texture limits;
// otherwise (or if creation fails) the kernel gathers with loads.  While the
// launch stream is being captured into a graph no view is created (an
// existing one is used, else the loads), so a capture never sees a call it
// might refuse.  Grids
// under DEM_VIEW_MIN_CELLS take the loads too: measured on GB300 (whole
// workflow, texture gathers against loads, many / few particles), 768^2 1012
// against 1085 / 250 against 252 us, 512^2 603 / 604, 165 / 165, 256^2 871 / 892
// and 380 / 372, 81 / 77 (a DEM that small stays in L1, where the loads' latency
// is shorter); 8192^2 5.5% less time.
constexpr int DEM_VIEWS_MAX = 256;
constexpr int64_t DEM_VIEW_MIN_CELLS = int64_t(1) << 19, DEM_VIEW_LARGE_CELLS = int64_t(1) << 20;

struct DemView {
    const float* h;
    int W, H, dev;
    cudaTextureObject_t tex;
};

cudaTextureObject_t dem_texture(const float* d_h, awo_grid g, cudaStream_t s)
{
    if (cells_of(g) < DEM_VIEW_MIN_CELLS) return 0;
    static std::mutex mu;
    static DemView tables[2][DEM_VIEWS_MAX];
    static int used[2] = {0, 0};
    const int large = cells_of(g) >= DEM_VIEW_LARGE_CELLS ? 1 : 0;
    DemView* views = tables[large];
    int& n_views = used[large];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    std::lock_guard<std::mutex> lock(mu);
    for (int i = 0; i < n_views; ++i)
        if (views[i].h == d_h && views[i].W == g.width && views[i].H == g.height && views[i].dev == dev)
            return views[i].tex;
    if (n_views == DEM_VIEWS_MAX) return 0;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) {
        cudaGetLastError();
        return 0;
    }
    int pitch_align = 0, base_align = 0, max_w = 0, max_h = 0;
    if (cudaDeviceGetAttribute(&pitch_align, cudaDevAttrTexturePitchAlignment, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&base_align, cudaDevAttrTextureAlignment, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&max_w, cudaDevAttrMaxTexture2DLinearWidth, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&max_h, cudaDevAttrMaxTexture2DLinearHeight, dev) != cudaSuccess || pitch_align <= 0 ||
        base_align <= 0)
        return 0;
    const size_t pitch = (size_t)g.width * sizeof(float);
    if ((pitch % (size_t)pitch_align) != 0 || ((uintptr_t)d_h % (uintptr_t)base_align) != 0 || g.width > max_w ||
        g.height > max_h)
        return 0;
    cudaResourceDesc rd;
    memset(&rd, 0, sizeof(rd));
    rd.resType = cudaResourceTypePitch2D;
    rd.res.pitch2D.devPtr = const_cast<float*>(d_h);
    rd.res.pitch2D.desc = cudaCreateChannelDesc<unsigned int>();  // raw words: no subnormal flush
    rd.res.pitch2D.width = (size_t)g.width;
    rd.res.pitch2D.height = (size_t)g.height;
    rd.res.pitch2D.pitchInBytes = pitch;
    cudaTextureDesc td;
    memset(&td, 0, sizeof(td));
    td.addressMode[0] = cudaAddressModeClamp;
    td.addressMode[1] = cudaAddressModeClamp;
    td.filterMode = cudaFilterModePoint;
    td.readMode = cudaReadModeElementType;
    td.normalizedCoords = 0;
    cudaTextureObject_t t = 0;
    if (cudaCreateTextureObject(&t, &rd, &td, nullptr) != cudaSuccess) {
        cudaGetLastError();  // a failed creation is not a launch error
        return 0;
    }
    views[n_views++] = DemView{d_h, g.width, g.height, dev, t};
    return t;
}

}  // namespace awo

using namespace awo;

static size_t starts_offset() { return (sizeof(SimWorkspace) + 255) / 256 * 256; }

// Events of awo_simulate_time_kernel for the next awo_simulate of this thread.
static thread_local cudaEvent_t t_kernel_events[2] = {nullptr, nullptr};

extern "C" awo_status awo_simulate_time_kernel(void* ev_start, void* ev_stop)
{
    if ((ev_start == nullptr) != (ev_stop == nullptr)) return AWO_EINVAL;
    t_kernel_events[0] = static_cast<cudaEvent_t>(ev_start);
    t_kernel_events[1] = static_cast<cudaEvent_t>(ev_stop);
    return AWO_OK;
}

extern "C" awo_status awo_dem_gather_path(const float* d_h, awo_grid g, void* stream, int32_t* texture)
{
    if (!d_h || !texture || !grid_ok(g)) return AWO_EINVAL;
    *texture = dem_texture(d_h, g, as_stream(stream)) != 0 ? 1 : 0;
    return AWO_OK;
}

extern "C" size_t awo_simulate_workspace_bytes(uint32_t n_cells_max)
{
    return starts_offset() + (size_t)n_cells_max * sizeof(TexelStart);
}

extern "C" awo_status awo_simulate(const float* d_h, awo_grid g, const uint32_t* d_cells, const uint32_t* d_n_cells,
                                   uint32_t n_cells_max, const awo_sim_params* p, uint32_t* d_count, float* d_maxe,
                                   awo_sim_stats* d_stats, void* d_ws, size_t ws_bytes, void* stream)
{
    const cudaEvent_t ev_start = t_kernel_events[0], ev_stop = t_kernel_events[1];  // consumed by this call
    t_kernel_events[0] = t_kernel_events[1] = nullptr;
    if (!d_h || !d_count || !d_maxe || !d_ws || !grid_ok(g)) return AWO_EINVAL;
    if (n_cells_max > 0 && !d_cells) return AWO_EINVAL;
    if (!sim_params_ok(p, g)) return AWO_EINVAL;
    if ((((uintptr_t)d_ws) & 15u) != 0 || (((uintptr_t)d_count) & 3u) != 0 || (((uintptr_t)d_maxe) & 3u) != 0)
        return AWO_EINVAL;
    if (ws_bytes < awo_simulate_workspace_bytes(n_cells_max)) return AWO_ENOMEM;
    cudaStream_t s = as_stream(stream);
    SimWorkspace* ws = static_cast<SimWorkspace*>(d_ws);

    SimArgs a;
    sim_constants(a, d_h, g, p, d_count, d_maxe, s);
    a.cells = d_cells;
    a.n_cells_dev = d_n_cells;
    a.n_cells_max = n_cells_max;
    a.next_item = &ws->work.next_item;
    a.stats = ws->stats.n;
    a.starts = static_cast<char*>(d_ws) + starts_offset();

    const int64_t n_clear = (p->flags & AWO_SIM_CLEAR_OUTPUTS) ? cells_of(g) : 0;
    const bool vec4 = ((((uintptr_t)d_count) | ((uintptr_t)d_maxe)) & 15u) == 0;
    k_sim_clear<<<stream_blocks(vec4 ? n_clear / 4 : n_clear, 256), 256, 0, s>>>(
        d_count, reinterpret_cast<uint32_t*>(d_maxe), n_clear, ws, vec4);
    awo_status st = launch_status();
    if (st != AWO_OK) return st;

    const bool work = a.N > 0 && n_cells_max > 0;
    if (work) {
        const unsigned pro_blocks = stream_blocks((int64_t)n_cells_max, 256);
        if (launch_kernel(a.tg.texels ? k_sim_starts<true> : k_sim_starts<false>, pro_blocks, 256, 0, -1, true, s, a) !=
            cudaSuccess)
            return AWO_ECUDA;
    }
    if (ev_start && cudaEventRecord(ev_start, s) != cudaSuccess) return AWO_ECUDA;
    if (work && a.max_steps != 0u) {  // else every particle is capped at its release visit
        st = launch_particles(a, SIM_THREADS, false, false, s);
        if (st != AWO_OK) return st;
    }
    if (ev_stop && cudaEventRecord(ev_stop, s) != cudaSuccess) return AWO_ECUDA;
    if (d_stats) return publish_stats(&ws->stats, d_stats, 1, ev_stop == nullptr, s);
    return AWO_OK;
}
