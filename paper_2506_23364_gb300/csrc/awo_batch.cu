// awo_batch.cu -- many avalanche-overlay requests in one call.
//
// Requests are each a DEM, a release list, parameters and rasters.  The
// request table travels in the kernels' parameter blocks, so a call needs no
// host-to-device copy and can be captured in a CUDA graph.  Kernels:
//   k_batch_prepare  one block: release counts (possibly on the device), the
//                    prefix sums of cells, zeroed counters;
//   k_batch_starts   per release cell of every request: its start record (in
//                    the processing order of awo_particle.cuh) and
//                    the release visits of its particles;
//   k_simulate       one launch per request (awo_simulate.cu), each allowed to
//                    start while the one before it still runs its last
//                    particles, so that the requests run as one stream of
//                    work without a tail between them.  A request's
//                    constants are then at fixed places of the parameter
//                    block: one persistent kernel over all requests kept them
//                    in registers (62 of them, 90 with the pool: 5 blocks an
//                    SM), and read by request index they cost 21 of 189 warp
//                    instructions per move.  12 regions 512^2..2048^2, the
//                    particle part: 9.71 ms as one kernel, 8.23 ms so.
// Every request's rasters equal those of awo_simulate on that request alone:
// it is the same kernel.
#include <math.h>

#include <algorithm>
#include <cstddef>
#include <cstring>
#include <mutex>
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
    TexelGeom tg;
};

struct BatchHeader {
    SimWorkspace ws[AWO_BATCH_MAX];           // each request's work counter (and statistics)
    uint32_t cell_prefix[AWO_BATCH_MAX + 1];  // start records before each request
    uint32_t n_cells[AWO_BATCH_MAX];
    uint32_t check;                           // check_pays of the whole batch
    uint32_t order_sinv[AWO_BATCH_MAX];       // processing order of each request's entries
};
constexpr size_t BATCH_HEADER_BYTES = ((sizeof(BatchHeader) + 255) / 256) * 256;

static_assert(sizeof(awo_sim_request) == 112, "awo_sim_request layout (C ABI)");
static_assert(offsetof(awo_sim_request, params) == 48, "awo_sim_request layout (C ABI)");
static_assert(sizeof(awo_tuning) == 16, "awo_tuning layout (C ABI)");

struct BatchArgs {
    BatchReq r[AWO_BATCH_MAX];
    uint32_t n_req;
    unsigned long long look_min;  // look_paths of whole-cell steps
    BatchHeader* hdr;
    unsigned long long* stats;  // 6 per request, stats_step words apart
    uint32_t stats_step;
    TexelStart* starts;  // one 32-byte slot per release-list entry (CellStarts fill the first half of a request's)
};
static_assert(sizeof(BatchArgs) <= 32764, "the request table must fit the kernel parameter block");

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

__global__ void __launch_bounds__(AWO_BATCH_MAX) k_batch_prepare(const __grid_constant__ BatchArgs a)
{
    __shared__ uint32_t s_nc[AWO_BATCH_MAX];
    __shared__ unsigned long long s_np[AWO_BATCH_MAX];
    const int t = threadIdx.x;
    uint32_t nc = 0u;
    if (t < (int)a.n_req) {
        const BatchReq& q = a.r[t];
        nc = q.n_cells_max;
        if (q.n_cells_dev) nc = min(nc, *q.n_cells_dev);
        if (q.N == 0u) nc = 0u;  // no particles, no release visits
        a.hdr->n_cells[t] = nc;
        a.hdr->order_sinv[t] = order_stride_inverse(nc / order_block(q.N));
    }
    s_nc[t] = nc;
    // particles for the particle kernel: none for a request with max_steps = 0
    // (every particle capped at its release visit, counted by k_batch_starts)
    s_np[t] = (t < (int)a.n_req && a.r[t].max_steps != 0u) ? (unsigned long long)nc * a.r[t].N : 0ull;
    if (t < (int)a.n_req) {
        a.hdr->ws[t] = SimWorkspace{};
        for (int i = 0; i < 6; ++i) a.stats[(size_t)t * a.stats_step + i] = 0ull;
    }
    __syncthreads();
    if (t == 0) {
        unsigned long long total = 0ull, grid = 0ull;
        double paths = 0.0;  // particles over their steps, as in look_paths
        uint32_t cs = 0u;
        for (int r = 0; r < (int)a.n_req; ++r) {
            a.hdr->cell_prefix[r] = cs;
            cs += s_nc[r];
            total += s_np[r];
            paths += (double)s_np[r] / a.r[r].s;
            grid += a.r[r].n_grid;
        }
        a.hdr->cell_prefix[a.n_req] = cs;
        a.hdr->check = paths >= (double)a.look_min || total >= 7ull * grid ? 1u : 0u;  // as check_pays
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
        unsigned long long* st6 = a.stats + (size_t)r * a.stats_step;
        if (!ok) atomicAdd(st6 + 5, (unsigned long long)q.N);
        if (ok && q.max_steps == 0u) {
            atomicAdd(st6 + 1, (unsigned long long)q.N);
            atomicAdd(st6 + 3, (unsigned long long)q.N);
        }
    }
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
    const uint32_t group = tuning ? (uint32_t)tuning->group_particles : 0u;
    const int refill = tuning ? tuning->refill : AWO_REFILL_LANE;
    cudaStream_t s = as_stream(stream);

    BatchArgs a;
    memset(&a, 0, sizeof(a));
    a.n_req = (uint32_t)n_req;
    a.look_min = look_paths(1.0f);
    a.hdr = static_cast<BatchHeader*>(d_ws);
    a.starts = reinterpret_cast<TexelStart*>(static_cast<char*>(d_ws) + BATCH_HEADER_BYTES);
    // the kernels count into the caller's statistics where they can
    const bool direct = d_stats && (((uintptr_t)d_stats) & 7u) == 0;
    a.stats = direct ? reinterpret_cast<unsigned long long*>(d_stats) : a.hdr->ws[0].stats;
    a.stats_step = (uint32_t)((direct ? sizeof(awo_sim_stats) : sizeof(SimWorkspace)) / sizeof(unsigned long long));
    SimArgs sim[AWO_BATCH_MAX];  // (no allocation that could throw)
    uint32_t off = 0;
    for (int i = 0; i < n_req; ++i) {
        const awo_sim_request& q = reqs[i];
        SimArgs& c = sim[i];
        sim_constants(c, q.d_h, q.grid, &q.params, q.d_count, q.d_maxe, s);
        c.n_cells_dev = a.hdr->n_cells + i;
        c.n_cells_max = q.n_cells_max;
        c.next_item = &a.hdr->ws[i].next_item;
        c.stats = a.stats + (size_t)i * a.stats_step;
        c.starts = a.starts + off;
        c.group = group;
        c.min_idle = refill == AWO_REFILL_WARP ? 32u : 1u;
        c.check = &a.hdr->check;
        BatchReq& b = a.r[i];
        b.h = q.d_h;
        b.count = q.d_count;
        b.W = c.W;
        b.H = c.H;
        b.P = c.P;
        b.oneP = c.oneP;
        b.s = c.s;
        b.max_steps = c.max_steps;
        b.cells = q.d_cells;
        b.n_cells_dev = q.d_n_cells;
        b.n_cells_max = q.n_cells_max;
        b.n_grid = c.n_grid;
        b.N = c.N;
        b.starts_off = off;
        b.tg = c.tg;
        off += q.n_cells_max;
        if (q.params.flags & AWO_SIM_CLEAR_OUTPUTS) {
            const size_t bytes = (size_t)cells_of(q.grid) * sizeof(uint32_t);
            if (cudaMemsetAsync(q.d_count, 0, bytes, s) != cudaSuccess) return AWO_ECUDA;
            if (cudaMemsetAsync(q.d_maxe, 0, bytes, s) != cudaSuccess) return AWO_ECUDA;
        }
    }
    k_batch_prepare<<<1, AWO_BATCH_MAX, 0, s>>>(a);
    if (total > 0) k_batch_starts<<<stream_blocks((int64_t)total, 256), 256, 0, s>>>(a);
    awo_status st = launch_status();
    bool after_particles = false;
    for (int i = 0; i < n_req && st == AWO_OK; ++i) {
        if (sim[i].N == 0u || sim[i].n_cells_max == 0u || sim[i].max_steps == 0u) continue;  // counted by the prologue
        st = launch_particles(sim[i], threads, after_particles, s);
        after_particles = true;
    }
    if (st != AWO_OK) return st;
    if (d_stats && !direct &&
        cudaMemcpy2DAsync(d_stats, sizeof(awo_sim_stats), a.hdr->ws[0].stats, sizeof(SimWorkspace), sizeof(awo_sim_stats),
                          (size_t)n_req, cudaMemcpyDeviceToDevice, s) != cudaSuccess)
        return AWO_ECUDA;
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
