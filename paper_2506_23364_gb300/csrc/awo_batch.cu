// awo_batch.cu -- many avalanche-overlay requests in one call.
//
// Requests are each a DEM, a release list, parameters and rasters.  The
// request table travels in the kernels' parameter blocks, so a call needs no
// host-to-device copy and can be captured in a CUDA graph.  Kernels:
//   k_batch_prepare  one block: release counts (possibly on the device), the
//                    prefix sums of cells and of units of work, zeroed
//                    counters;
//   k_batch_starts   per release cell of every request: its start record (in
//                    the processing order of awo_particle.cuh) and
//                    the release visits of its particles;
//   k_simulate       for a request with many particles, a launch of its own
//                    (awo_simulate.cu), allowed to start while the one before
//                    it still runs its last particles;
//   k_batch_simulate for all others together, persistent: a warp takes a unit,
//                    which names a request, and runs that request's particles
//                    (run_particles, the loop of awo_simulate) until none is
//                    left to take.
// Every request's rasters equal those of awo_simulate on that request alone:
// the particles take the same steps.
#include <math.h>

#include <algorithm>
#include <cstddef>
#include <cstring>
#include <vector>

#include "awo_particle.cuh"

namespace awo {

// What the prologue needs of a request.
struct BatchReq {
    const float* h;
    uint32_t* count;
    int W, H;
    float P, oneP, s;
    uint32_t max_steps;
    const uint32_t* cells;
    const uint32_t* n_cells_dev;
    uint32_t n_cells_max, n_grid, N;
    uint32_t starts_off;  // its first 32-byte start-record slot
    uint32_t id;          // its index in the caller's array
    uint32_t own_launch;  // OwnLaunch
    TexelGeom tg;
};

// Requests that share an instance of the particle kernel: records of texels
// or cells, footprints by texture or by loads.
constexpr int BATCH_KINDS = 2;

// Requests are in launch order (BatchArgs.r) but for the statistics, which are
// in the caller's.
struct BatchHeader {
    WorkCounter work[AWO_BATCH_MAX];
    StatsCounters stats[AWO_BATCH_MAX];
    unsigned long long n_part[AWO_BATCH_MAX];  // particles of each request for k_batch_simulate
    uint32_t cell_prefix[AWO_BATCH_MAX + 1];   // start records before each request
    uint32_t unit_prefix[AWO_BATCH_MAX + 1];   // units of work before each request
    uint32_t n_cells[AWO_BATCH_MAX];
    uint32_t own_cells[AWO_BATCH_MAX];   // n_cells of the requests with a launch of their own, else 0
    uint32_t order_sinv[AWO_BATCH_MAX];  // processing order of each request's entries
    uint32_t next_unit[BATCH_KINDS];     // units taken, by launch
    uint32_t chunk;                      // particles a warp takes per fetch, at most
    uint32_t check;                      // check_pays of the whole batch
};
constexpr size_t BATCH_HEADER_BYTES = ((sizeof(BatchHeader) + 255) / 256) * 256;

static_assert(sizeof(awo_sim_request) == 112, "awo_sim_request layout (C ABI)");
static_assert(offsetof(awo_sim_request, params) == 48, "awo_sim_request layout (C ABI)");
static_assert(sizeof(awo_tuning) == 16, "awo_tuning layout (C ABI)");

struct BatchArgs {
    BatchReq r[AWO_BATCH_MAX];
    uint32_t n_req;
    uint32_t sim_warps;           // warps of k_batch_simulate's launch
    unsigned long long look_min;  // look_paths of whole-cell steps
    BatchHeader* hdr;
    TexelStart* starts;  // one 32-byte slot per release-list entry (CellStarts fill the first half of a request's)
};
static_assert(sizeof(BatchArgs) <= 32764, "the request table must fit the kernel parameter block");

// A request of the particle kernel (names read by AWO_MOVE_WORDS and run_particles, as in SimArgs).
struct BatchSimReq {
    const float* h;
    uint32_t* count;
    float* maxe;
    int W, H;
    float Wm1, Hm1, P, oneP, R, s, R23, kD, muD;
    uint32_t max_steps;
    KeysTable keys;
    uint32_t N, id;
    void* starts;
    cudaTextureObject_t tex;
};

struct BatchSimArgs {
    BatchSimReq r[AWO_BATCH_MAX];
    uint32_t first, n;   // the launch's requests
    uint32_t kind;       // its work counter
    uint32_t group;      // particles a warp takes per fetch, 0: chosen by the kernel
    uint32_t min_idle;   // idle lanes a refill needs: 1, or 32 (lock-step batches)
    BatchHeader* hdr;
};
static_assert(sizeof(BatchSimArgs) <= 32764, "the request table must fit the kernel parameter block");

// How the particles of a batch are shared out.  A unit of work stands for one
// warp on one request: the warp that takes it runs the request's particles
// until none is left to take.  The batch has UNITS_PER_WARP units for each
// warp of the launch, split over the requests by their particles, so that
// some requests are always at work while another one's last particles run
// out.  But warps wait for their requests' constants when an SM works on many
// requests (the stall on indexed constant loads is 1.3 warps an issue with the
// shares below, 20.8 without a least share), so a request gets at least one in
// REQUESTS_IN_FLIGHT of the warps (or one for every 32 of its particles).  A
// warp that finds no unit left joins a request that has more particles
// waiting than its own warps take next.  Measured (ms; 128 regions of 256^2 with
// 64 particles per release cell / 128 of 512^2 with 16 / 32 of 1024^2 with 32), 2
// units a warp and a share of 1 in 8: 2.76 / 2.81 / 3.87; 1 in 32 3.45 / 3.29 / 4.19;
// no least share 4.14 / 3.99 / 4.19, with 1 unit a warp 4.95 / 4.77 / 6.45; all warps
// on each request in turn 3.89 / 4.57 / 4.12.
constexpr uint32_t UNITS_PER_WARP = 2, REQUESTS_IN_FLIGHT = 8;
constexpr uint32_t CHUNKS_PER_WARP = 32;  // fetches a warp makes on an even split (16: 12 of 1280^2 5.80 -> 5.95 ms)

// Requests with a launch of k_simulate each: their constants are then at
// fixed places of the parameter block, which runs up to 167 G moves/s where
// k_batch_simulate, issue-bound, ends at 140; but a launch leaves the GPU
// partly idle at its end, and costs the host 4 us.  Only the instance with the
// look is launched, so they need a batch for which looking pays: a second
// launch's 1500 blocks, which end at once, had to trickle through the few
// slots that the first one's last particles left free.  Their warps take
// OWN_CHUNK particles a fetch or more: with 32, fetches at the one counter
// held them back.  12 of 1280^2, 5.7 M particles each: 5.74 ms together, 7.66
// with two launches each, 5.67 with one, 5.27 with one and 128 a fetch (96 5.29,
// 256 5.38); 4 of 2048^2, 23 M each, 7.4 together, 6.03 so; 16 of 1024^2, 2.9 M
// each, 3.52 together, 3.33 with launches of their own, 4.4 M each 5.27 and 4.59;
// 12 of 512^2..2048^2 7.35 (8.47 all together, 7.75 with two launches each).
// The number of particles is known on the device alone, so the host launches
// for every request that can have LARGE_PARTICLES at the share of release
// cells that steep terrain has (1 in 22), and the launch ends at once when
// there are fewer (32 of 2048^2 with few release cells: 2.38 -> 2.47 ms).  A
// request that is alone of its kind has its own launch, too.
constexpr unsigned long long LARGE_PARTICLES = 3000000ull, LARGE_MOST = 22ull * LARGE_PARTICLES;
constexpr uint32_t OWN_CHUNK = 128;
enum OwnLaunch : uint32_t { OWN_NEVER, OWN_IF_LARGE, OWN_ALWAYS };

// Index r with prefix[r] <= g < prefix[r+1] (prefix has n + 1 entries).
template <typename T>
__device__ __forceinline__ int find_request(const T* prefix, int n, T g)
{
    int lo = 0, hi = n;  // invariant: prefix[lo] <= g < prefix[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (prefix[mid] <= g)
            lo = mid;
        else
            hi = mid;
    }
    return lo;
}

// Sum over the lanes of a warp up to this one.
template <typename T>
__device__ __forceinline__ T warp_inclusive(T v)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const T t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// One thread per request.
__global__ void __launch_bounds__(AWO_BATCH_MAX) k_batch_prepare(const __grid_constant__ BatchArgs a)
{
    constexpr int WARPS = AWO_BATCH_MAX / 32;
    __shared__ unsigned long long s_total[WARPS], s_grid[WARPS];
    __shared__ double s_paths[WARPS];
    __shared__ uint32_t s_cells[WARPS], s_units[WARPS];
    const int t = threadIdx.x, warp = t >> 5;
    const bool last_lane = (t & 31) == 31;
    const bool mine = t < (int)a.n_req;
    uint32_t nc = 0u;
    unsigned long long np = 0ull, grid = 0ull;
    double paths = 0.0;  // particles over their steps, as in look_paths
    if (mine) {
        const BatchReq& q = a.r[t];
        nc = q.n_cells_max;
        if (q.n_cells_dev) nc = min(nc, *q.n_cells_dev);
        if (q.N == 0u) nc = 0u;  // no particles, no release visits
        a.hdr->n_cells[t] = nc;
        a.hdr->order_sinv[t] = order_stride_inverse(nc / order_block(q.N));
        // particles for the particle kernel: none for a request with max_steps = 0
        // (every particle capped at its release visit, counted by k_batch_starts)
        np = q.max_steps != 0u ? (unsigned long long)nc * q.N : 0ull;
        grid = q.n_grid;
        paths = (double)np / q.s;
        a.hdr->work[t] = WorkCounter{};
        a.hdr->stats[t] = StatsCounters{};
    }
    const unsigned long long np_up = warp_inclusive(np), grid_up = warp_inclusive(grid);
    const double paths_up = warp_inclusive(paths);
    if (last_lane) s_total[warp] = np_up, s_grid[warp] = grid_up, s_paths[warp] = paths_up;
    __syncthreads();
    unsigned long long total = 0ull;
#pragma unroll
    for (int w = 0; w < WARPS; ++w) total += s_total[w];
    unsigned long long grids = 0ull;
    double sum_paths = 0.0;
#pragma unroll
    for (int w = 0; w < WARPS; ++w) grids += s_grid[w], sum_paths += s_paths[w];
    const bool check = sum_paths >= (double)a.look_min || total >= 7ull * grids;  // as check_pays
    const bool own = mine && (a.r[t].own_launch == OWN_ALWAYS ||
                              (a.r[t].own_launch == OWN_IF_LARGE && check && np >= LARGE_PARTICLES));
    // FP32 is enough to share out the work (a 64-bit division costs more than the rest of this kernel)
    const float warps = (float)a.sim_warps, unit = fmaxf((float)total / (warps * UNITS_PER_WARP), 32.0f);
    const float least = fminf((float)np / 32.0f, warps / REQUESTS_IN_FLIGHT);
    const uint32_t units = own ? 0u : (uint32_t)ceilf(fminf(fmaxf((float)np / unit, least), warps));
    uint32_t cells1 = warp_inclusive(nc), units1 = warp_inclusive(units);
    if (last_lane) s_cells[warp] = cells1, s_units[warp] = units1;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < WARPS; ++w)
        if (w < warp) cells1 += s_cells[w], units1 += s_units[w];
    if (t < BATCH_KINDS) a.hdr->next_unit[t] = 0u;
    a.hdr->n_part[t] = own ? 0ull : np;
    a.hdr->own_cells[t] = own ? nc : 0u;
    a.hdr->cell_prefix[t + 1] = cells1;
    a.hdr->unit_prefix[t + 1] = units1;
    if (t == 0) {
        a.hdr->cell_prefix[0] = a.hdr->unit_prefix[0] = 0u;
        a.hdr->chunk = max((uint32_t)fminf((float)total / (warps * CHUNKS_PER_WARP), 1024.0f) & ~31u, 32u);
        a.hdr->check = check ? 1u : 0u;
    }
}

__global__ void __launch_bounds__(256) k_batch_starts(const __grid_constant__ BatchArgs a)
{
    __shared__ uint32_t s_cp[AWO_BATCH_MAX + 1];
    const int n = (int)a.n_req;
    for (int i = threadIdx.x; i <= n; i += blockDim.x) s_cp[i] = a.hdr->cell_prefix[i];
    __syncthreads();
    const uint32_t total = s_cp[n];
    for (uint32_t g = blockIdx.x * blockDim.x + threadIdx.x; g < total; g += gridDim.x * blockDim.x) {
        const int r = find_request<uint32_t>(s_cp, n, g);
        const BatchReq& q = a.r[r];
        const uint32_t ci = g - s_cp[r];
        const uint32_t entry = __ldg(q.cells + ci);
        const uint32_t B = order_block(q.N);
        const uint32_t slot = order_slot(ci, B, (s_cp[r + 1] - s_cp[r]) / B, a.hdr->order_sinv[r]);
        bool ok;
        if (q.tg.texels) {
            TexelStart st = texel_start(q.h, q.W, q.H, q.tg, entry);
            first_vector(st, q.P, q.oneP);
            ok = st.t != ~0u;
            if (ok) atomicAdd(q.count + st.vcell, q.N);
            a.starts[q.starts_off + slot] = st;
        } else {
            CellStart st = cell_start(q.h, q.W, q.H, q.n_grid, entry);
            first_vector(st, q.P, q.oneP);
            ok = st.xy != ~0u;
            if (ok) atomicAdd(q.count + entry, q.N);
            reinterpret_cast<CellStart*>(a.starts + q.starts_off)[slot] = st;
        }
        // particles of entries outside the grid are rejected; with max_steps = 0
        // every particle is capped at its release visit (no particle kernel work)
        unsigned long long* st6 = a.hdr->stats[q.id].n;
        if (!ok) atomicAdd(st6 + 5, (unsigned long long)q.N);
        if (ok && q.max_steps == 0u) {
            atomicAdd(st6 + 1, (unsigned long long)q.N);
            atomicAdd(st6 + 3, (unsigned long long)q.N);
        }
    }
}

// One launch per kind of request and instance (with and without the look: one
// of the two ends at once, as in k_simulate).  Persistent; the last block
// orders the launch after the one before it (see k_simulate).
//
// A request's constants are read where they are used, by constant loads
// indexed with the request (11% of the instructions): held in a lane's
// registers they took 62-92 of them.  64 registers, 8 blocks an SM: 48 (and 16
// bytes spilled) gave 2% more on large requests and took 5-8% longer on small
// ones, which are bound by latency.  128 regions of 64^2 1.44 -> 0.85 ms against a
// launch for each, of 512^2 with 16 particles per release cell 5.43 -> 2.85, 32 of
// 1024^2 with 32 6.05 -> 3.84.
template <bool TEXELS, bool PLAIN, bool CHECK>
__global__ void __launch_bounds__(256, 4) k_batch_simulate(const __grid_constant__ BatchSimArgs a)
{
    extern __shared__ uint32_t s_pool[];  // POOL_WORDS per warp
    asm volatile("griddepcontrol.launch_dependents;");
    if (blockIdx.x == gridDim.x - 1u) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        return;
    }
    if ((a.hdr->check != 0u) != CHECK) return;
    const uint32_t lane = threadIdx.x & 31u;
    uint32_t* pool = s_pool + (threadIdx.x >> 5) * POOL_WORDS;
    const uint32_t* prefix = a.hdr->unit_prefix + a.first;
    bool units_left = true;
    while (true) {
        uint32_t g = 0u, i = 0u;
        if (units_left) {
            if (lane == 0u) g = atomicAdd(&a.hdr->next_unit[a.kind], 1u);
            g = prefix[0] + __shfl_sync(0xffffffffu, g, 0);
            units_left = g < prefix[a.n];
        }
        if (units_left) {
            // the request of unit g: as many come before it as end at or below g
#pragma unroll
            for (uint32_t k = 0u; k < AWO_BATCH_MAX; k += 32u)
                i += (uint32_t)__popc(__ballot_sync(0xffffffffu, k + lane < a.n && prefix[k + lane + 1u] <= g));
        } else {
            // no unit left: the first request with more particles waiting than its own warps take next
            i = a.n;
            for (uint32_t k = 0u; k < a.n && i == a.n; k += 32u) {
                const uint32_t j = min(k + lane, a.n - 1u), c = a.first + j;
                const unsigned which =
                    __ballot_sync(0xffffffffu, __ldcg(&a.hdr->work[c].next_item) + 32ull * (prefix[j + 1u] - prefix[j]) <
                                                   a.hdr->n_part[c]);
                if (which) i = min(k + (uint32_t)__ffs(which) - 1u, a.n - 1u);
            }
            if (i == a.n) break;
        }
        const uint32_t r = a.first + i;
        const BatchSimReq& q = a.r[r];
        const unsigned long long total = a.hdr->n_part[r];
        unsigned long long* stats = a.hdr->stats[q.id].n;
        const uint32_t unit0 = prefix[i], units = prefix[i + 1] - unit0;
        if (units_left && g == unit0 && lane == 0u) {
            // particles of entries inside the grid (the prologue has counted the others)
            const unsigned long long run = total - stats[5];
            stats[1] = run;
            atomicAdd(&stats[4], run);
        }
        // particles a warp takes per fetch: the batch's, or one warp's share where that is less
        const unsigned long long share = total / units;
        uint32_t chunk = share < a.hdr->chunk ? max((uint32_t)share & ~31u, 32u) : a.hdr->chunk;
        if (a.group) chunk = a.group;
        if (q.tex)
            run_particles<TEXELS, 1, CHECK, PLAIN>(q, total, chunk, a.min_idle, &a.hdr->work[r].next_item, stats, pool);
        else
            run_particles<TEXELS, 0, CHECK, PLAIN>(q, total, chunk, a.min_idle, &a.hdr->work[r].next_item, stats, pool);
        __syncwarp();  // the pool is empty; its words before the next request's
    }
}

template <bool TEXELS, bool PLAIN>
static awo_status launch_kind(const BatchSimArgs& a, int threads, bool early, cudaStream_t s)
{
    const awo_status st = launch_persistent<k_batch_simulate<TEXELS, PLAIN, true>>(a, threads, early, s);
    return st != AWO_OK ? st : launch_persistent<k_batch_simulate<TEXELS, PLAIN, false>>(a, threads, true, s);
}

static bool tuning_ok(const awo_tuning* t)
{
    if (!t) return true;
    if (t->threads_per_block != 0 && t->threads_per_block != 64 && t->threads_per_block != 128 &&
        t->threads_per_block != 256)
        return false;
    if (t->group_particles != 0 && (t->group_particles < 32 || t->group_particles > 65536)) return false;
    if (t->refill != AWO_REFILL_LANE && t->refill != AWO_REFILL_WARP) return false;
    return true;
}

static bool requests_ok(const awo_sim_request* reqs, int32_t n_req, uint64_t* total_cells)
{
    if (!reqs || n_req < 1 || n_req > AWO_BATCH_MAX) return false;
    uint64_t tot = 0;
    for (int i = 0; i < n_req; ++i) {
        const awo_sim_request& q = reqs[i];
        if (!q.d_h || !q.d_count || !q.d_maxe || !grid_ok(q.grid)) return false;
        if (q.n_cells_max > 0 && !q.d_cells) return false;
        if (!sim_params_ok(&q.params, q.grid)) return false;
        if ((((uintptr_t)q.d_count) & 3u) != 0 || (((uintptr_t)q.d_maxe) & 3u) != 0) return false;
        tot += q.n_cells_max;
    }
    if (tot >= ((uint64_t)1 << 31)) return false;
    *total_cells = tot;
    return true;
}

}  // namespace awo

using namespace awo;

extern "C" size_t awo_simulate_batched_workspace_bytes(const awo_sim_request* reqs, int32_t n_req)
{
    uint64_t tot = 0;
    if (!requests_ok(reqs, n_req, &tot)) return 0;
    return BATCH_HEADER_BYTES + (size_t)tot * sizeof(TexelStart);
}

extern "C" awo_status awo_simulate_batched(const awo_sim_request* reqs, int32_t n_req, const awo_tuning* tuning,
                                           awo_sim_stats* d_stats, void* d_ws, size_t ws_bytes, void* stream)
{
    uint64_t total = 0;
    if (!requests_ok(reqs, n_req, &total) || !tuning_ok(tuning) || !d_ws) return AWO_EINVAL;
    if ((((uintptr_t)d_ws) & 15u) != 0) return AWO_EINVAL;
    if (ws_bytes < BATCH_HEADER_BYTES + (size_t)total * sizeof(TexelStart)) return AWO_ENOMEM;
    const int threads = (tuning && tuning->threads_per_block) ? tuning->threads_per_block : 128;
    cudaStream_t s = as_stream(stream);

    BatchArgs a;
    memset(&a, 0, sizeof(a));
    a.n_req = (uint32_t)n_req;
    a.look_min = look_paths(1.0f);
    a.hdr = static_cast<BatchHeader*>(d_ws);
    a.starts = reinterpret_cast<TexelStart*>(static_cast<char*>(d_ws) + BATCH_HEADER_BYTES);
    // the requests by kind, each kind's in the caller's order
    BatchSimArgs b;
    memset(&b, 0, sizeof(b));
    b.hdr = a.hdr;
    b.group = tuning ? (uint32_t)tuning->group_particles : 0u;
    b.min_idle = tuning && tuning->refill == AWO_REFILL_WARP ? 32u : 1u;
    bool plain = true;
    uint32_t kind_first[BATCH_KINDS + 1] = {0}, off = 0, at = 0;
    SimArgs own[AWO_BATCH_MAX];
    for (int kind = 0; kind < BATCH_KINDS; ++kind) {
        kind_first[kind] = at;
        for (int i = 0; i < n_req; ++i) {
            if ((reqs[i].params.release_log2 != 0) != (kind == 1)) continue;
            const awo_sim_request& q = reqs[i];
            SimArgs& c = own[at];
            sim_constants(c, q.d_h, q.grid, &q.params, q.d_count, q.d_maxe, s);
            BatchSimReq& d = b.r[at];
            d.h = c.h;
            d.count = c.count;
            d.maxe = c.maxe;
            d.W = c.W;
            d.H = c.H;
            d.Wm1 = c.Wm1;
            d.Hm1 = c.Hm1;
            d.P = c.P;
            d.oneP = c.oneP;
            d.R = c.R;
            d.s = c.s;
            d.R23 = c.R23;
            d.kD = c.kD;
            d.muD = c.muD;
            d.max_steps = c.max_steps;
            d.keys = c.keys;
            d.N = c.N;
            d.id = (uint32_t)i;
            d.starts = a.starts + off;
            d.tex = c.tex;
            plain = plain && c.s == 1.0f && c.kD == 0.0f;
            BatchReq& e = a.r[at];
            e.h = c.h;
            e.count = c.count;
            e.W = c.W;
            e.H = c.H;
            e.P = c.P;
            e.oneP = c.oneP;
            e.s = c.s;
            e.max_steps = c.max_steps;
            e.cells = q.d_cells;
            e.n_cells_dev = q.d_n_cells;
            e.n_cells_max = q.n_cells_max;
            e.n_grid = c.n_grid;
            e.N = c.N;
            e.starts_off = off;
            e.id = (uint32_t)i;
            e.own_launch = (unsigned long long)q.n_cells_max * c.N >= LARGE_MOST ? OWN_IF_LARGE : OWN_NEVER;
            e.tg = c.tg;
            off += q.n_cells_max;
            ++at;
            if (q.params.flags & AWO_SIM_CLEAR_OUTPUTS) {
                const size_t bytes = (size_t)cells_of(q.grid) * sizeof(uint32_t);
                if (cudaMemsetAsync(q.d_count, 0, bytes, s) != cudaSuccess) return AWO_ECUDA;
                if (cudaMemsetAsync(q.d_maxe, 0, bytes, s) != cudaSuccess) return AWO_ECUDA;
            }
        }
    }
    kind_first[BATCH_KINDS] = at;
    for (int kind = 0; kind < BATCH_KINDS; ++kind)
        if (kind_first[kind + 1] == kind_first[kind] + 1u) a.r[kind_first[kind]].own_launch = OWN_ALWAYS;
    a.sim_warps = particle_blocks<k_batch_simulate<false, false, true>>(threads) * (unsigned)(threads / 32);
    k_batch_prepare<<<1, AWO_BATCH_MAX, 0, s>>>(a);
    if (total > 0) k_batch_starts<<<stream_blocks((int64_t)total, 256), 256, 0, s>>>(a);
    awo_status st = launch_status();
    bool after_particles = false;
    for (int r = 0; r < n_req && st == AWO_OK; ++r) {
        SimArgs& c = own[r];
        if (a.r[r].own_launch == OWN_NEVER || c.N == 0u || c.max_steps == 0u || a.r[r].n_cells_max == 0u) continue;
        c.n_cells_dev = a.hdr->own_cells + r;
        c.n_cells_max = a.r[r].n_cells_max;
        c.next_item = &a.hdr->work[r].next_item;
        c.stats = a.hdr->stats[a.r[r].id].n;
        c.starts = a.starts + a.r[r].starts_off;
        c.group = b.group;
        c.min_idle = b.min_idle;
        c.check = &a.hdr->check;
        c.least_chunk = a.r[r].own_launch == OWN_IF_LARGE ? OWN_CHUNK : 32u;
        st = launch_particles(c, threads, after_particles, a.r[r].own_launch == OWN_IF_LARGE, s);
        after_particles = true;
    }
    for (int kind = 0; kind < BATCH_KINDS && st == AWO_OK && total > 0; ++kind) {
        b.first = kind_first[kind];
        b.n = kind_first[kind + 1] - b.first;
        b.kind = (uint32_t)kind;
        if (b.n == 0u) continue;
        if (b.n == 1u && a.r[b.first].own_launch == OWN_ALWAYS) continue;
        auto launch = kind == 0 ? (plain ? launch_kind<false, true> : launch_kind<false, false>)
                                : (plain ? launch_kind<true, true> : launch_kind<true, false>);
        st = launch(b, threads, after_particles, s);
        after_particles = true;
    }
    if (st != AWO_OK) return st;
    if (d_stats) return publish_stats(a.hdr->stats, d_stats, n_req, after_particles, s);
    return AWO_OK;
}

extern "C" awo_status awo_tune_batched(const awo_sim_request* reqs, int32_t n_req, void* d_ws, size_t ws_bytes,
                                       void* stream, awo_tuning* best, float* best_ms)
{
    uint64_t total = 0;
    if (!requests_ok(reqs, n_req, &total) || !best) return AWO_EINVAL;
    std::vector<awo_sim_request> rq(reqs, reqs + n_req);
    for (auto& q : rq) q.params.flags |= AWO_SIM_CLEAR_OUTPUTS;
    cudaStream_t s = as_stream(stream);
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess) return AWO_ECUDA;
    if (cudaEventCreate(&e1) != cudaSuccess) {
        cudaEventDestroy(e0);
        return AWO_ECUDA;
    }
    const int threads[] = {64, 128, 256};
    const int groups[] = {0, 256, 1024, 4096};  // 0: chosen from the particle count
    const int refills[] = {AWO_REFILL_LANE, AWO_REFILL_WARP};
    float best_t = 3.0e38f;
    awo_tuning best_cfg = {128, 0, AWO_REFILL_LANE, 0};
    awo_status result = AWO_OK;
    for (int rf : refills)
        for (int th : threads)
            for (int gp : groups) {
                awo_tuning t = {th, gp, rf, 0};
                float t_min = 3.0e38f;
                for (int rep = 0; rep < 2 && result == AWO_OK; ++rep) {
                    if (cudaEventRecord(e0, s) != cudaSuccess) result = AWO_ECUDA;
                    if (result == AWO_OK)
                        result = awo_simulate_batched(rq.data(), n_req, &t, nullptr, d_ws, ws_bytes, stream);
                    if (result == AWO_OK && cudaEventRecord(e1, s) != cudaSuccess) result = AWO_ECUDA;
                    if (result == AWO_OK && cudaEventSynchronize(e1) != cudaSuccess) result = AWO_ECUDA;
                    float ms = 0.f;
                    if (result == AWO_OK && cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) result = AWO_ECUDA;
                    if (result == AWO_OK) t_min = std::min(t_min, ms);
                }
                if (result != AWO_OK) break;
                if (t_min < best_t) {
                    best_t = t_min;
                    best_cfg = t;
                }
            }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (result != AWO_OK) return result;
    *best = best_cfg;
    if (best_ms) *best_ms = best_t;
    return AWO_OK;
}
