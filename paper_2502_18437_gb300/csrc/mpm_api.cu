// C ABI of the MLS-MPM library (include/mpm.h): context lifecycle, factory
// calls, substep scheduling with CUDA-graph replay, blocking state readback.
//
// Object model after Sec. V-A of arXiv 2502.18437: mpm_substep is the
// asynchronous Scene::advance (everything is enqueued on the context's
// stream), mpm_read_state the blocking Scene::fetchResults.
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <thread>

#include "mpm_ctx.cuh"

using namespace mpm;

namespace mpm {

int status_from_cuda(cudaError_t e)
{
    if (e == cudaSuccess) return MPM_OK;
    if (e == cudaErrorMemoryAllocation) return MPM_ERR_OUT_OF_MEMORY;
    return MPM_ERR_CUDA;
}

#define MPM_CK(call)                                      \
    do {                                                  \
        cudaError_t e_ = (call);                          \
        if (e_ != cudaSuccess) return status_from_cuda(e_); \
    } while (0)

static int timeout_ms(const mpm_ctx* c) { return c->cfg.timeout_ms > 0 ? c->cfg.timeout_ms : 10000; }

// Wait for all work enqueued on the context's stream, polling an event with a
// bound instead of blocking inside the driver; after kSpinUs with pauses (each takes
// some 70 us, as long as a small scene's whole readback).
constexpr int kSpinUs = 20000;

int wait_stream(mpm_ctx* c)
{
    MPM_CK(cudaEventRecord(c->ev, c->stream));
    const auto t0 = std::chrono::steady_clock::now();
    for (;;) {
        cudaError_t e = cudaEventQuery(c->ev);
        if (e == cudaSuccess) return MPM_OK;
        if (e != cudaErrorNotReady) return status_from_cuda(e);
        const auto us = std::chrono::duration_cast<std::chrono::microseconds>(std::chrono::steady_clock::now() - t0).count();
        if (us / 1000 > timeout_ms(c)) return MPM_ERR_TIMEOUT;
        if (us < kSpinUs) std::this_thread::yield();
        else std::this_thread::sleep_for(std::chrono::microseconds(20));
    }
}

// (rounded up so that states stored one after another keep their planes aligned)
size_t state_bytes(int cap) { return ((size_t)cap * kStateFloats * sizeof(float) + 255) & ~(size_t)255; }

PState state_view(float* base, int cap)
{
    PState s;
    s.q = reinterpret_cast<float4*>(base);
    s.mu = base + 4 * (size_t)kPlanes * cap;
    s.lam = s.mu + cap;
    return s;
}

int ensure_stage(mpm_ctx* c, size_t bytes)
{
    if (bytes <= c->stage_bytes) return MPM_OK;
    if (c->d_stage) {
        MPM_CK(cudaStreamSynchronize(c->stream));
        cudaFree(c->d_stage);
        c->d_stage = nullptr;
        c->stage_bytes = 0;
    }
    MPM_CK(cudaMalloc(&c->d_stage, bytes));
    c->stage_bytes = bytes;
    return MPM_OK;
}

static int ensure_pinned(mpm_ctx* c, size_t bytes)
{
    if (bytes <= c->pinned_bytes) return MPM_OK;
    if (c->h_pinned) {
        MPM_CK(cudaStreamSynchronize(c->stream));
        cudaFreeHost(c->h_pinned);
        c->h_pinned = nullptr;
        c->pinned_bytes = 0;
    }
    MPM_CK(cudaMallocHost(&c->h_pinned, bytes));
    c->pinned_bytes = bytes;
    return MPM_OK;
}

static bool is_pinned_host(const void* p)
{
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeHost;
}

// Device address of page-locked, mapped host memory (kernels read or write it
// directly over the host link), or null for any other pointer.
static void* mapped_host(const void* p)
{
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    return at.type == cudaMemoryTypeHost ? at.devicePointer : nullptr;
}

int upload_scenes(mpm_ctx* c)
{
    if (!c->scenes_dirty) return MPM_OK;
    MPM_CK(cudaMemcpyAsync(c->d_scenes, c->h_scenes.data(), sizeof(SceneDev) * c->n_scenes, cudaMemcpyHostToDevice,
                           c->stream));
    c->scenes_dirty = false;
    return MPM_OK;
}

void clear_graphs(mpm_ctx* c)
{
    for (auto& kv : c->graphs) cudaGraphExecDestroy(kv.second);
    c->graphs.clear();
}

// G2P CTA size of a launch over np particles: the set value, or by default 256
// threads below 512k particles and 128 above.  Both hold 24 warps of 80 registers on an
// SM; what decides is that the 128-thread shape leaves L1 the shared memory it does not
// need (prepare_kernels).  A substep with 128 and with 256 threads: 4M particles 400 and
// 415 us, 1M 121.0 and 119.6, 262k 42.3 and 41.5, 131k 32.4 and 33.1, 16k 19.1 and 19.2;
// with a sphere in the scene 4M 419 and 421, 1M 134.4 and 132.1, 262k 46.8 and 46.5, 131k
// 36.3 and 36.7, 16k 22.1 and 24.9.  The standard-MPM and PB-MPM G2P variants exist at
// 128 threads only.
static int g2p_threads_for(const mpm_ctx* c, int np)
{
    if (c->cfg.solver != MPM_SOLVER_MLS) return 128;
    if (c->g2p_threads) return c->g2p_threads;
    return np < (1 << 19) ? 256 : 128;
}

// Slots that each P2G warp stages: a warp's share of half the set pass, or by default 32 where
// that gives every warp that fits on the chip one chunk at most and 64 above (a pass of 32
// lanes takes 64 slots' runs as well as 32 slots': at 131k particles, 1.1 chunks of 32 a warp,
// a substep of the standard MPM takes 44.9 us with 32 and 41.1 with 64).
int p2g_slots_for(const mpm_ctx* c, int np)
{
    if (c->p2g_chunk) return c->p2g_chunk / (2 * kP2GThreads / 32);
    return (long long)np < 32ll * c->num_sms * 24 ? 32 : 64;
}

static int cap_occ(const mpm_ctx* c, int occ)
{
    if (occ < 1) occ = 1;
    if (c->ctas_per_sm > 0 && c->ctas_per_sm < occ) occ = c->ctas_per_sm;
    return occ;
}

StepArgs step_args(mpm_ctx* c, float dt, int s0, int s1, const PState& in, const PState& out)
{
    StepArgs a{};
    a.r.s0 = s0;
    a.r.s1 = s1;
    a.r.bb0 = c->brick_base[s0];
    a.r.nbr = c->brick_base[s1] - c->brick_base[s0];
    a.r.t0 = c->tile_base[s0];
    a.r.nt = c->tile_base[s1] - c->tile_base[s0];
    a.r.p0 = c->h_scenes[s0].p_begin;
    int pend = s1 < c->n_scenes ? c->h_scenes[s1].p_begin : c->total_particles;
    a.r.np = pend - a.r.p0;
    a.sb = c->sb;
    a.scenes = c->d_scenes;
    a.rigids = c->d_rigids;
    a.pose = c->d_pose;
    a.impulse = c->d_impulse;
    a.t_scene = c->d_time;
    a.epoch = c->d_epoch;
    a.brick_epoch = c->brick_epoch;
    a.err = c->d_err;
    a.G = c->G;
    a.V = c->V;
    a.in = in;
    a.out = out;
    a.cap = c->cap;
    a.dt = dt;
    for (int i = 0; i < 3; ++i) a.gravity[i] = c->cfg.gravity[i];
    a.bound = c->cfg.bound;
    a.floor_sticky = c->cfg.floor_sticky;
    a.model = c->cfg.model;
    a.plasticity = c->cfg.plasticity;
    a.yield_stress = c->cfg.yield_stress;
    // the occupancy queries are host calls: ask once per variant and context
    const int g2p_threads = g2p_threads_for(c, a.r.np);
    const int ti = g2p_threads == 128 ? 0 : g2p_threads == 512 ? 2 : 1;
    int& og = c->occ_g2p[c->g2p_regs64 ? 1 : 0][ti];
    if (!og) og = std::max(1, occupancy_g2p(g2p_threads, c->g2p_regs64));
    a.g2p_ctas = c->num_sms * cap_occ(c, og);
    a.p2g_slots = p2g_slots_for(c, a.r.np);
    int& op = c->occ_p2g[a.p2g_slots / 16 - 1];
    if (!op) op = std::max(1, occupancy_p2g(a.p2g_slots));
    if (!c->occ_grid) c->occ_grid = std::max(1, occupancy_grid());
    if (!c->occ_grid_plain) c->occ_grid_plain = std::max(1, occupancy_grid_plain());
    if (!c->occ_fused) c->occ_fused = std::max(1, occupancy_g2p2g());
    a.g2p_regs64 = c->g2p_regs64;
    a.p2g_ctas = c->num_sms * cap_occ(c, op);
    a.grid_ctas = c->num_sms * c->occ_grid;
    a.grid_plain_ctas = c->num_sms * c->occ_grid_plain;
    a.fused_ctas = c->num_sms * cap_occ(c, c->occ_fused);
    a.g2p_threads = g2p_threads;
    a.solver = c->cfg.solver;
    a.pb_beta = c->cfg.pb_beta;
    a.any_rigid = 0;
    a.rigid_ext = 0;
    a.any_solid = 0;
    for (int sc = s0; sc < s1; ++sc) {
        if (c->h_scenes[sc].n_rigid > 0) a.any_rigid = 1;
        for (int k = 0; k < kMaxRigids; ++k) {
            const int ty = c->rigid_type[(size_t)sc * kMaxRigids + k];
            if (ty == MPM_ARC || ty == MPM_MESH_SLICER) a.rigid_ext = 1;
            if (ty == MPM_SPHERE || ty == MPM_BOX) a.any_solid = 1;
        }
    }
    return a;
}

// One substep of every scene.  Unfused (default): sort, P2G, grid update, G2P.
// Fused (MPM_OPT_FUSED): sort, P2G only when G does not already hold this state's P2G
// (need_p2g), grid update, then the fused G2P + P2G, which leaves the next
// substep's P2G in G.
int enqueue_substep(mpm_ctx* c, float dt, const PState& in, const PState& out, bool need_p2g)
{
    const int groups = c->launch_mode == 1 ? c->n_scenes : 1;
    for (int g = 0; g < groups; ++g) {
        const int s0 = c->launch_mode == 1 ? g : 0;
        const int s1 = c->launch_mode == 1 ? g + 1 : c->n_scenes;
        StepArgs a = step_args(c, dt, s0, s1, in, out);
        a.tau_valid = c->tau_valid;
        cudaEvent_t* ev = nullptr;
        if (c->phase_timing) {
            if (c->phase_used + 5 > c->phase_events.size()) {
                for (int k = 0; k < 5 * 64; ++k) {
                    cudaEvent_t e;
                    MPM_CK(cudaEventCreate(&e));
                    c->phase_events.push_back(e);
                }
            }
            ev = &c->phase_events[c->phase_used];
            c->phase_used += 5;
        }
        if (ev) MPM_CK(cudaEventRecord(ev[0], c->stream));
        MPM_CK(launch_sort(a, c->stream));
        if (ev) MPM_CK(cudaEventRecord(ev[1], c->stream));
        if (a.solver == MPM_SOLVER_PB) {
            // PB-MPM: cycles of constraint + P2G, grid update and G2P of v and C at
            // fixed positions (the sort above serves them all); gravity in the first
            // cycle only; the last cycle's G2P integrates x and F and ends the substep
            const int cycles = c->cfg.pb_iterations > 0 ? c->cfg.pb_iterations : 10;
            for (int k = 0; k < cycles; ++k) {
                StepArgs b = a;
                if (k > 0) {
                    for (int d = 0; d < 3; ++d) b.gravity[d] = 0.f;
                }
                MPM_CK(launch_p2g(b, c->stream));
                MPM_CK(launch_grid(b, c->stream, false));
                if (k + 1 < cycles) MPM_CK(launch_g2p_vc(b, c->stream));
                else {
                    if (ev) MPM_CK(cudaEventRecord(ev[2], c->stream));
                    if (ev) MPM_CK(cudaEventRecord(ev[3], c->stream));
                    MPM_CK(launch_g2p(b, c->stream));
                }
            }
            if (ev) MPM_CK(cudaEventRecord(ev[4], c->stream));
            continue;
        }
        if (!c->fused || need_p2g) MPM_CK(launch_p2g(a, c->stream));
        if (ev) MPM_CK(cudaEventRecord(ev[2], c->stream));
        MPM_CK(launch_grid(a, c->stream, c->fused != 0));
        if (ev) MPM_CK(cudaEventRecord(ev[3], c->stream));
        if (c->fused) MPM_CK(launch_g2p2g(a, c->stream));
        else MPM_CK(launch_g2p(a, c->stream));
        if (ev) MPM_CK(cudaEventRecord(ev[4], c->stream));
    }
    // the unfused G2P stores the new stress; the fused kernel keeps it in registers;
    // PB-MPM stores none
    c->tau_valid = !c->fused && c->cfg.solver != MPM_SOLVER_PB;
    return MPM_OK;
}

// The state or dt changed: G's pending scatter no longer applies.
int invalidate_pending(mpm_ctx* c)
{
    c->g_pending = false;
    c->tau_valid = false;
    return MPM_OK;
}

cudaError_t reset_histogram(mpm_ctx* c) { return launch_reset_histogram(c->sb, c->total_bricks, c->total_tiles, c->total_particles, c->stream); }

int ensure_keys(mpm_ctx* c)
{
    if (c->keys_valid) return MPM_OK;
    MPM_CK(reset_histogram(c));
    StepArgs a = step_args(c, 0.f, 0, c->n_scenes, c->st[c->cur], c->st[c->cur ^ 1]);
    MPM_CK(launch_prepare(a, c->st[c->cur], c->stream));
    c->keys_valid = true;
    return MPM_OK;
}

}  // namespace mpm

// ===================================================================== ABI

extern "C" const char* mpm_status_string(int s)
{
    switch (s) {
    case MPM_OK: return "ok";
    case MPM_ERR_INVALID_ARGUMENT: return "invalid argument";
    case MPM_ERR_OUT_OF_MEMORY: return "out of memory";
    case MPM_ERR_CUDA: return "CUDA runtime error";
    case MPM_ERR_OUT_OF_DOMAIN: return "a particle left its scene's grid";
    case MPM_ERR_NONFINITE: return "a particle value became non-finite";
    case MPM_ERR_INVERTED: return "inverted element (det F <= 0) where the law needs ln J";
    case MPM_ERR_CAPACITY: return "particle capacity exceeded";
    case MPM_ERR_TIMEOUT: return "bounded wait timed out";
    case MPM_ERR_STATE: return "call out of order";
    case MPM_ERR_INTERNAL: return "device-side consistency check failed";
    default: return "unknown status";
    }
}

static void free_ctx(mpm_ctx* c)
{
    if (!c) return;
    cudaStreamSynchronize(c->stream);
    mpm_tape_free(c);
    clear_graphs(c);
    cudaFree(c->arena);
    cudaFree(c->d_stage);
    if (c->h_pinned) cudaFreeHost(c->h_pinned);
    if (c->ev) cudaEventDestroy(c->ev);
    for (cudaEvent_t e : c->phase_events) cudaEventDestroy(e);
    if (c->own_stream) cudaStreamDestroy(c->stream);
    delete c;
}

extern "C" int mpm_destroy(mpm_ctx* c);

extern "C" int mpm_create(const mpm_config* cfg, void* stream, mpm_ctx** out)
{
    if (!cfg || !out) return MPM_ERR_INVALID_ARGUMENT;
    *out = nullptr;
    if (cfg->n_scenes < 1 || cfg->max_particles < 0 || cfg->max_particles > (int64_t)1 << 30) return MPM_ERR_INVALID_ARGUMENT;
    if (cfg->model != MPM_FIXED_COROTATED && cfg->model != MPM_NEO_HOOKEAN) return MPM_ERR_INVALID_ARGUMENT;
    if (cfg->plasticity != MPM_PLASTIC_NONE && cfg->plasticity != MPM_PLASTIC_VON_MISES) return MPM_ERR_INVALID_ARGUMENT;
    if (cfg->bound < 0) return MPM_ERR_INVALID_ARGUMENT;
    if (cfg->solver < MPM_SOLVER_MLS || cfg->solver > MPM_SOLVER_PB) return MPM_ERR_INVALID_ARGUMENT;
    if (cfg->solver == MPM_SOLVER_PB &&
        (cfg->pb_iterations < 0 || cfg->pb_iterations > 1000 || !(cfg->pb_beta >= 0.f && cfg->pb_beta <= 1.f) ||
         cfg->plasticity != MPM_PLASTIC_NONE))
        return MPM_ERR_INVALID_ARGUMENT;
    mpm_ctx* c = new mpm_ctx();
    c->cfg = *cfg;
    c->cfg.scene_grid_n = nullptr;
    c->stream = static_cast<cudaStream_t>(stream);
    c->n_scenes = cfg->n_scenes;
    c->scene_n.resize(c->n_scenes);
    c->brick_base.resize(c->n_scenes + 1);
    long long bricks = 0;
    for (int s = 0; s < c->n_scenes; ++s) {
        const int n = cfg->scene_grid_n ? cfg->scene_grid_n[s] : cfg->grid_n;
        if (n < 8 || n > 1024 || n % 4 != 0 || 2 * cfg->bound >= n) { delete c; return MPM_ERR_INVALID_ARGUMENT; }
        c->scene_n[s] = n;
        c->brick_base[s] = (int)bricks;
        bricks += (long long)(n / 4) * (n / 4) * (n / 4);
    }
    if (bricks * 64 >= ((long long)1 << 31)) { delete c; return MPM_ERR_INVALID_ARGUMENT; }
    c->brick_base[c->n_scenes] = (int)bricks;
    c->total_bricks = (int)bricks;
    // scan tiles: 2^shift bricks of one scene, at least 64; wider tiles keep
    // the number of tiles (whose counts every scan CTA adds up) near 2048 or less
    {
        int shift = kMinTileShift;
        auto tiles = [&](int sh) {
            long long t = 0;
            for (int s = 0; s < c->n_scenes; ++s)
                t += ((long long)(c->brick_base[s + 1] - c->brick_base[s]) + (1 << sh) - 1) >> sh;
            return t;
        };
        while (shift < 24 && tiles(shift) > 2048) ++shift;
        c->sb.tile_shift = shift;
        c->tile_base.resize(c->n_scenes + 1);
        int t = 0;
        for (int s = 0; s < c->n_scenes; ++s) {
            c->tile_base[s] = t;
            t += (c->brick_base[s + 1] - c->brick_base[s] + (1 << shift) - 1) >> shift;
        }
        c->tile_base[c->n_scenes] = t;
        c->total_tiles = t;
    }
    c->cap = (int)std::max<int64_t>(cfg->max_particles, 1);
    c->h_scenes.resize(c->n_scenes);
    for (int s = 0; s < c->n_scenes; ++s) {
        SceneDev& d = c->h_scenes[s];
        memset(&d, 0, sizeof d);
        d.n = c->scene_n[s];
        d.nb = d.n / 4;
        d.brick_base = c->brick_base[s];
        d.tile_base = c->tile_base[s];
        d.nb_log2 = -1;
        for (int k = 0; k < 31; ++k)
            if ((1 << k) == d.nb) d.nb_log2 = k;
    }
    c->h_rigids.assign((size_t)c->n_scenes * kMaxRigids, RigidDev{});
    c->rigid_type.assign((size_t)c->n_scenes * kMaxRigids, MPM_RIGID_NONE);
    for (auto& r : c->h_rigids) r.type = MPM_RIGID_NONE;

    cudaError_t e = cudaGetDevice(&c->device);
    if (e == cudaSuccess && !c->stream) {
        // graphs cannot be captured on the legacy default stream: use a private one
        e = cudaStreamCreateWithFlags(&c->stream, cudaStreamNonBlocking);
        c->own_stream = e == cudaSuccess;
    }
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&c->num_sms, cudaDevAttrMultiProcessorCount, c->device);
    if (e == cudaSuccess) e = prepare_kernels();
    const size_t nbk = (size_t)c->total_bricks;
    // one allocation for all buffers; those that start from zero come first
    struct Part { void** p; size_t bytes; };
    std::vector<Part> parts;
    auto alloc = [&](void** p, size_t bytes) { parts.push_back({p, (bytes + 255) & ~(size_t)255}); };
    alloc((void**)&c->sb.cnt, sizeof(int) * nbk);
    alloc((void**)&c->sb.ccnt, sizeof(int) * nbk * 64);
    alloc((void**)&c->sb.counters, sizeof(int) * CTR_COUNT);
    alloc((void**)&c->sb.tile_n, sizeof(int) * c->total_tiles);
    alloc((void**)&c->G, sizeof(float4) * nbk * 64);
    alloc((void**)&c->V, sizeof(float4) * nbk * 64);
    alloc((void**)&c->d_impulse, sizeof(double) * c->n_scenes * kMaxRigids * 6);
    alloc((void**)&c->d_err, sizeof(unsigned) * c->n_scenes);
    alloc((void**)&c->d_time, sizeof(double) * c->n_scenes);
    alloc((void**)&c->d_epoch, sizeof(int) * c->n_scenes);
    const size_t n_zero = parts.size();
    for (int i = 0; i < 2; ++i) alloc((void**)&c->state_mem[i], state_bytes(c->cap));
    alloc((void**)&c->sb.key, sizeof(int) * c->cap);
    alloc((void**)&c->sb.rank, sizeof(int) * c->cap);
    alloc((void**)&c->sb.perm, sizeof(int) * c->cap);
    alloc((void**)&c->sb.act_brick, sizeof(int) * nbk);
    alloc((void**)&c->sb.act_start, sizeof(int) * nbk);
    alloc((void**)&c->sb.act_count, sizeof(int) * nbk);
    alloc((void**)&c->sb.act_scene, sizeof(int) * nbk);
    alloc((void**)&c->sb.nact_brick, sizeof(int) * nbk);
    alloc((void**)&c->sb.nact_scene, sizeof(int) * nbk);
    c->sb.list_size = c->total_bricks;
    alloc((void**)&c->brick_epoch, sizeof(int) * nbk);
    alloc((void**)&c->d_scenes, sizeof(SceneDev) * c->n_scenes);
    alloc((void**)&c->d_rigids, sizeof(RigidDev) * c->n_scenes * kMaxRigids);
    alloc((void**)&c->d_inv, sizeof(int) * c->cap);
    alloc((void**)&c->d_pose, sizeof(RigidPose) * c->n_scenes * kMaxRigids);
    size_t zero = 0, total = 0;
    for (size_t i = 0; i < parts.size(); ++i) {
        total += parts[i].bytes;
        if (i < n_zero) zero += parts[i].bytes;
    }
    if (e == cudaSuccess) e = cudaMalloc(&c->arena, total);
    if (e == cudaSuccess) {
        char* at = static_cast<char*>(c->arena);
        for (const Part& q : parts) {
            *q.p = at;
            at += q.bytes;
        }
    }
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&c->ev, cudaEventDisableTiming);
    if (e == cudaSuccess) {
        for (int i = 0; i < 2; ++i) c->st[i] = state_view(c->state_mem[i], c->cap);
        cudaMemsetAsync(c->arena, 0, zero, c->stream);
        cudaMemsetAsync(c->brick_epoch, 0xff, sizeof(int) * nbk, c->stream);
        e = cudaMemcpyAsync(c->d_rigids, c->h_rigids.data(), sizeof(RigidDev) * c->h_rigids.size(),
                            cudaMemcpyHostToDevice, c->stream);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) {
        free_ctx(c);
        return status_from_cuda(e);
    }
    *out = c;
    return MPM_OK;
}

extern "C" int mpm_destroy(mpm_ctx* c)
{
    free_ctx(c);
    return MPM_OK;
}

extern "C" int mpm_get_option(mpm_ctx* c, int option, int64_t* value)
{
    if (!c || !value) return MPM_ERR_INVALID_ARGUMENT;
    switch (option) {
    case MPM_OPT_USE_GRAPHS: *value = c->use_graphs; break;
    case MPM_OPT_LAUNCH_MODE: *value = c->launch_mode; break;
    case MPM_OPT_P2G_THREADS: *value = kP2GThreads; break;
    case MPM_OPT_G2P_THREADS: *value = g2p_threads_for(c, c->total_particles); break;
    case MPM_OPT_CTAS_PER_SM: *value = c->ctas_per_sm; break;
    case MPM_OPT_GRAPH_CHUNK: *value = c->graph_chunk; break;
    case MPM_OPT_PHASE_TIMING: *value = c->phase_timing; break;
    case MPM_OPT_P2G_CHUNK: *value = p2g_slots_for(c, c->total_particles) * (2 * kP2GThreads / 32); break;
    case MPM_OPT_FUSED: *value = c->fused; break;
    case MPM_OPT_G2P_REGS64: *value = c->g2p_regs64; break;
    default: return MPM_ERR_INVALID_ARGUMENT;
    }
    return MPM_OK;
}

extern "C" int mpm_set_option(mpm_ctx* c, int option, int64_t value)
{
    if (!c) return MPM_ERR_INVALID_ARGUMENT;
    switch (option) {
    case MPM_OPT_USE_GRAPHS: c->use_graphs = value != 0; break;
    case MPM_OPT_LAUNCH_MODE:
        if (value != 0 && value != 1) return MPM_ERR_INVALID_ARGUMENT;
        c->launch_mode = (int)value;
        break;
    case MPM_OPT_P2G_THREADS:
        if (value != kP2GThreads) return MPM_ERR_INVALID_ARGUMENT;
        break;
    case MPM_OPT_P2G_CHUNK:
        if (value != 2 * kP2GThreads && value != 3 * kP2GThreads && value != 4 * kP2GThreads)
            return MPM_ERR_INVALID_ARGUMENT;
        c->p2g_chunk = (int)value;
        break;
    case MPM_OPT_G2P_THREADS:
        if (value != 0 && value != 128 && value != 256 && value != 512) return MPM_ERR_INVALID_ARGUMENT;
        c->g2p_threads = (int)value;
        break;
    case MPM_OPT_CTAS_PER_SM:
        if (value < 0 || value > 32) return MPM_ERR_INVALID_ARGUMENT;
        c->ctas_per_sm = (int)value;
        break;
    case MPM_OPT_GRAPH_CHUNK:
        if (value < 1 || value > 64) return MPM_ERR_INVALID_ARGUMENT;
        c->graph_chunk = (int)value;
        break;
    case MPM_OPT_PHASE_TIMING: c->phase_timing = value != 0; break;
    case MPM_OPT_G2P_REGS64: c->g2p_regs64 = value != 0; break;
    case MPM_OPT_FUSED:
        if (value != 0 && c->cfg.solver != MPM_SOLVER_MLS) return MPM_ERR_INVALID_ARGUMENT;
        c->fused = value != 0;
        invalidate_pending(c);
        break;
    default: return MPM_ERR_INVALID_ARGUMENT;
    }
    clear_graphs(c);
    return MPM_OK;
}

extern "C" int mpm_scene_count(mpm_ctx* c, int scene, int64_t* count)
{
    if (!c || !count || scene < 0 || scene >= c->n_scenes) return MPM_ERR_INVALID_ARGUMENT;
    *count = c->h_scenes[scene].p_count;
    return MPM_OK;
}

// Copy a caller buffer of `bytes` to device memory (returns a device pointer).
static int stage_input(mpm_ctx* c, const void* src, size_t bytes, int mem, size_t stage_off, const void** dev)
{
    if (!src) { *dev = nullptr; return MPM_OK; }
    if (mem == MPM_MEM_DEVICE) { *dev = src; return MPM_OK; }
    char* dst = static_cast<char*>(c->d_stage) + stage_off;
    MPM_CK(cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, c->stream));
    *dev = dst;
    return MPM_OK;
}

static size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

extern "C" int mpm_add_particles(mpm_ctx* c, int scene, int64_t n, const float* x, const float* v, const float* E,
                                 const float* nu, float E0, float nu0, float rho, float V0, int mem,
                                 int64_t* first_id_out)
{
    if (!c || scene < 0 || scene >= c->n_scenes || n < 0 || (n > 0 && !x)) return MPM_ERR_INVALID_ARGUMENT;
    if (mem != MPM_MEM_HOST && mem != MPM_MEM_DEVICE) return MPM_ERR_INVALID_ARGUMENT;
    if (!(rho > 0.f) || !(V0 > 0.f)) return MPM_ERR_INVALID_ARGUMENT;
    if (!E && !(E0 >= 0.f)) return MPM_ERR_INVALID_ARGUMENT;
    if (!nu && !(nu0 > -1.f && nu0 < 0.5f)) return MPM_ERR_INVALID_ARGUMENT;
    if ((int64_t)c->total_particles + n > c->cap) return MPM_ERR_CAPACITY;
    SceneDev& sc = c->h_scenes[scene];
    const float m_p = rho * V0;
    if (sc.p_count > 0 && (sc.m_p != m_p || sc.V0 != V0)) return MPM_ERR_INVALID_ARGUMENT;
    if (first_id_out) *first_id_out = sc.p_count;
    if (n == 0) return MPM_OK;
    if (c->recording) return MPM_ERR_STATE;

    const size_t bx = align256(sizeof(float) * 3 * n), bs = align256(sizeof(float) * n);
    int st = ensure_stage(c, 2 * bx + 2 * bs);
    if (st) return st;
    const void *dx = nullptr, *dv = nullptr, *dE = nullptr, *dnu = nullptr;
    if ((st = stage_input(c, x, sizeof(float) * 3 * n, mem, 0, &dx))) return st;
    if ((st = stage_input(c, v, sizeof(float) * 3 * n, mem, bx, &dv))) return st;
    if ((st = stage_input(c, E, sizeof(float) * n, mem, 2 * bx, &dE))) return st;
    if ((st = stage_input(c, nu, sizeof(float) * n, mem, 2 * bx + bs, &dnu))) return st;

    // material: uniform unless the scene ever sees per-particle values or a second (E0, nu0)
    const float mu0 = E0 / (2.f * (1.f + nu0)), lam0 = E0 * nu0 / ((1.f + nu0) * (1.f - 2.f * nu0));
    bool pp = E || nu || (sc.p_count > 0 && (sc.mu != mu0 || sc.lam != lam0));
    const int p_at = sc.p_begin + sc.p_count;
    const int tail = c->total_particles - p_at;
    PState cur = c->st[c->cur];
    if (tail > 0) {
        // make room: copy into the spare buffer with the later scenes shifted by n
        PState nxt = c->st[c->cur ^ 1];
        struct Part { const char* src; char* dst; size_t item; };
        std::vector<Part> parts;
        for (int k = 0; k < kPlanes; ++k)
            parts.push_back({reinterpret_cast<const char*>(cur.q + (size_t)k * c->cap),
                             reinterpret_cast<char*>(nxt.q + (size_t)k * c->cap), sizeof(float4)});
        parts.push_back({reinterpret_cast<const char*>(cur.mu), reinterpret_cast<char*>(nxt.mu), sizeof(float)});
        parts.push_back({reinterpret_cast<const char*>(cur.lam), reinterpret_cast<char*>(nxt.lam), sizeof(float)});
        for (const Part& q : parts) {
            if (p_at > 0) MPM_CK(cudaMemcpyAsync(q.dst, q.src, q.item * p_at, cudaMemcpyDeviceToDevice, c->stream));
            MPM_CK(cudaMemcpyAsync(q.dst + q.item * (p_at + n), q.src + q.item * p_at, q.item * tail,
                                   cudaMemcpyDeviceToDevice, c->stream));
        }
        c->cur ^= 1;
        cur = nxt;
    }
    MPM_CK(launch_init_particles(cur, c->cap, p_at, (int)n, sc.p_count, static_cast<const float*>(dx),
                                 static_cast<const float*>(dv), static_cast<const float*>(dE),
                                 static_cast<const float*>(dnu), E0, nu0, c->stream));
    if (pp && !sc.pp_mat && sc.p_count > 0) {
        // per-particle arrays of the existing particles were not carried: refill them
        std::vector<float> mu(sc.p_count, sc.mu), lam(sc.p_count, sc.lam);
        MPM_CK(cudaMemcpyAsync(cur.mu + sc.p_begin, mu.data(), sizeof(float) * sc.p_count, cudaMemcpyHostToDevice, c->stream));
        MPM_CK(cudaMemcpyAsync(cur.lam + sc.p_begin, lam.data(), sizeof(float) * sc.p_count, cudaMemcpyHostToDevice, c->stream));
    }
    if (sc.p_count == 0) {
        sc.m_p = m_p;
        sc.V0 = V0;
        sc.mu = mu0;
        sc.lam = lam0;
    }
    sc.pp_mat = sc.pp_mat || pp;
    sc.p_count += (int)n;
    for (int s = scene + 1; s < c->n_scenes; ++s) c->h_scenes[s].p_begin += (int)n;
    c->total_particles += (int)n;
    c->scenes_dirty = true;
    c->keys_valid = false;
    invalidate_pending(c);
    clear_graphs(c);
    st = upload_scenes(c);
    if (st) return st;
    if (mem == MPM_MEM_HOST) {
        // the caller may reuse its buffers once we return (pageable copies are staged by
        // the runtime; wait for the stream so pinned sources are consumed too)
        st = wait_stream(c);
        if (st) return st;
    }
    return MPM_OK;
}

extern "C" int mpm_set_rigid(mpm_ctx* c, int scene, int rigid_id, const mpm_rigid* r)
{
    if (!c || !r || scene < 0 || scene >= c->n_scenes || rigid_id < 0 || rigid_id >= kMaxRigids) return MPM_ERR_INVALID_ARGUMENT;
    const int slot = scene * kMaxRigids + rigid_id;
    RigidDev d{};
    if (r->type == MPM_RIGID_NONE) {
        d.type = MPM_RIGID_NONE;
    } else {
        if (r->type < MPM_SPHERE || r->type > MPM_MESH_SLICER) return MPM_ERR_INVALID_ARGUMENT;
        if (r->type == MPM_SEGMENTS && (r->n_points < 2 || r->n_points > MPM_MAX_SEGMENT_POINTS)) return MPM_ERR_INVALID_ARGUMENT;
        if (r->type == MPM_ARC && !(r->half[0] > 0.f && r->half[2] > 0.f && r->half[2] <= 6.2831855f))
            return MPM_ERR_INVALID_ARGUMENT;
        if (r->type == MPM_MESH_SLICER) {
            if (r->n_points < 3 || r->n_points > MPM_MAX_SEGMENT_POINTS || r->n_triangles < 1 ||
                r->n_triangles > MPM_MAX_MESH_TRIANGLES || r->n_spine < 0 || r->n_spine == 1 ||
                r->n_spine > MPM_MAX_SPINE_POINTS)
                return MPM_ERR_INVALID_ARGUMENT;
            for (int k = 0; k < 3 * r->n_triangles; ++k) {
                const int v = (&r->triangles[0][0])[k];
                if (v < 0 || v >= r->n_points) return MPM_ERR_INVALID_ARGUMENT;
            }
            for (int k = 0; k < r->n_spine; ++k)
                if (r->spine[k] < 0 || r->spine[k] >= r->n_points) return MPM_ERR_INVALID_ARGUMENT;
        }
        const double qn = std::sqrt((double)r->quat[0] * r->quat[0] + (double)r->quat[1] * r->quat[1] +
                                    (double)r->quat[2] * r->quat[2] + (double)r->quat[3] * r->quat[3]);
        if (!(qn > 0.0)) return MPM_ERR_INVALID_ARGUMENT;
        d.type = r->type;
        d.n_pts = (r->type == MPM_SEGMENTS || r->type == MPM_MESH_SLICER) ? r->n_points : 0;
        if (r->type == MPM_MESH_SLICER) {
            d.n_tris = r->n_triangles;
            d.n_spine = r->n_spine;
            for (int k = 0; k < 3 * d.n_tris; ++k) d.shape.tris[k] = (unsigned char)(&r->triangles[0][0])[k];
            for (int k = 0; k < d.n_spine; ++k) d.shape.spine[k] = (unsigned char)r->spine[k];
        }
        for (int i = 0; i < 3; ++i) {
            d.c0[i] = r->center[i];
            d.vel[i] = r->vel[i];
            d.omega[i] = r->omega[i];
            d.half[i] = r->half[i];
        }
        for (int i = 0; i < 4; ++i) d.q0[i] = (float)(r->quat[i] / qn);
        d.mu_k = r->mu_k;
        d.c_d = r->c_d;
        d.margin = r->margin;
        d.radius = r->radius;
        d.thickness = r->thickness;
        d.spine_radius = r->spine_radius;
        d.t_set = c->h_time;
        for (int k = 0; k < 3 * d.n_pts; ++k) d.shape.pts[k] = (&r->points[0][0])[k];
        // (widened by far more than the distances' rounding, relative to the shape and its reach;
        // without end where a point is not finite)
        // (fmax leaves a NaN out: a comparison with it touches nothing, but the other reach still does)
        const float reach = std::fmax(r->type == MPM_SEGMENTS ? r->radius : std::fmax(0.5f * r->thickness, r->spine_radius), 0.f) +
                            std::fmax(r->margin, 0.f);
        for (int i = 0; i < 3 && d.n_pts > 0; ++i) {
            float lo = d.shape.pts[i], hi = lo, big = std::fabs(lo), sum = lo;
            for (int k = 1; k < d.n_pts; ++k) {
                lo = std::min(lo, d.shape.pts[3 * k + i]);
                hi = std::max(hi, d.shape.pts[3 * k + i]);
                sum += d.shape.pts[3 * k + i];
                big = std::max(big, std::fabs(d.shape.pts[3 * k + i]));
            }
            const float wide = std::isfinite(sum) ? reach + 1e-5f * (reach + big) + 1e-30f : INFINITY;
            if (!std::isfinite(sum)) lo = hi = 0.f;
            d.lo[i] = lo - wide;
            d.hi[i] = hi + wide;
        }
    }
    // refused before anything changes: poses belong to a moment, not to a graph
    cudaStreamCaptureStatus capturing;
    MPM_CK(cudaStreamIsCapturing(c->stream, &capturing));
    if (capturing != cudaStreamCaptureStatusNone) return MPM_ERR_CUDA;
    c->h_rigids[slot] = d;
    if (c->rigid_type[slot] != d.type) clear_graphs(c);  // captured launches carry the kinds of rigids
    c->rigid_type[slot] = d.type;
    int nr = 0;
    for (int k = 0; k < kMaxRigids; ++k)
        if (c->rigid_type[scene * kMaxRigids + k] != MPM_RIGID_NONE) nr = k + 1;
    if (c->h_scenes[scene].n_rigid != nr) {
        c->h_scenes[scene].n_rigid = nr;
        c->scenes_dirty = true;
        clear_graphs(c);  // captured substeps carry whether any scene has a rigid
    }
    // the description travels in the launch's arguments: nothing to wait for
    MPM_CK(launch_set_rigid(d, c->d_rigids + slot, c->stream));
    return upload_scenes(c);
}

static uint32_t float_bits(float f)
{
    uint32_t u;
    memcpy(&u, &f, 4);
    return u;
}

extern "C" int mpm_substep(mpm_ctx* c, float dt, int n_substeps)
{
    if (!c || !(dt > 0.f) || !std::isfinite(dt) || n_substeps < 0) return MPM_ERR_INVALID_ARGUMENT;
    if (n_substeps == 0) return MPM_OK;
    int st = upload_scenes(c);
    if (st) return st;
    if ((st = ensure_keys(c))) return st;
    if (c->recording) {
        for (int k = 0; k < n_substeps; ++k)
            if ((st = mpm_tape_record_substep(c, dt))) return st;
        return MPM_OK;
    }
    int left = n_substeps;
    const bool pending = c->fused && c->g_pending && c->g_dt == dt;
    // One direct substep first where the captured graphs' assumptions do not hold
    // yet: the fused kernel needs this state's P2G already in G, and the captured
    // P2G reads the stress that the previous G2P stored.
    const bool direct_first = c->fused ? !pending : (!c->tau_valid || c->g_dirty);
    if (direct_first) {
        // a fresh P2G: clear whatever scatter G still holds, then one direct substep
        if (c->g_dirty) MPM_CK(cudaMemsetAsync(c->G, 0, sizeof(float4) * (size_t)c->total_bricks * 64, c->stream));
        if ((st = enqueue_substep(c, dt, c->st[c->cur], c->st[c->cur ^ 1], true))) return st;
        c->cur ^= 1;
        c->h_time += (double)dt;
        --left;
    }
    c->g_pending = c->fused != 0;
    c->g_dirty = c->fused != 0;
    c->g_dt = dt;
    if (!c->use_graphs || c->phase_timing) {
        for (int k = 0; k < left; ++k) {
            if ((st = enqueue_substep(c, dt, c->st[c->cur], c->st[c->cur ^ 1], false))) return st;
            c->cur ^= 1;
            c->h_time += (double)dt;
        }
        return MPM_OK;
    }
    while (left > 0) {
        const int L = left < c->graph_chunk ? left : c->graph_chunk;
        auto key = std::make_tuple(float_bits(dt), L, c->cur);
        auto it = c->graphs.find(key);
        if (it == c->graphs.end()) {
            cudaGraph_t g;
            MPM_CK(cudaStreamBeginCapture(c->stream, cudaStreamCaptureModeThreadLocal));
            int cur = c->cur;
            int err = MPM_OK;
            for (int k = 0; k < L && !err; ++k) {
                err = enqueue_substep(c, dt, c->st[cur], c->st[cur ^ 1], false);
                cur ^= 1;
            }
            cudaError_t ce = cudaStreamEndCapture(c->stream, &g);
            if (err) return err;
            MPM_CK(ce);
            cudaGraphExec_t ex;
            ce = cudaGraphInstantiate(&ex, g, 0);
            cudaGraphDestroy(g);
            MPM_CK(ce);
            it = c->graphs.emplace(key, ex).first;
        }
        MPM_CK(cudaGraphLaunch(it->second, c->stream));
        if (L & 1) c->cur ^= 1;
        for (int k = 0; k < L; ++k) c->h_time += (double)dt;
        left -= L;
    }
    return MPM_OK;
}

static int error_status(unsigned bits)
{
    // a non-finite value is reported first: its NaN position also fails the domain test
    if (bits & MPM_EBIT_NONFINITE) return MPM_ERR_NONFINITE;
    if (bits & MPM_EBIT_OUT_OF_DOMAIN) return MPM_ERR_OUT_OF_DOMAIN;
    if (bits & MPM_EBIT_INVERTED) return MPM_ERR_INVERTED;
    if (bits & MPM_EBIT_TIMEOUT) return MPM_ERR_TIMEOUT;
    if (bits & MPM_EBIT_INTERNAL) return MPM_ERR_INTERNAL;
    return MPM_OK;
}

extern "C" int mpm_get_error(mpm_ctx* c, int scene, uint32_t* bits)
{
    if (!c || !bits || scene < 0 || scene >= c->n_scenes) return MPM_ERR_INVALID_ARGUMENT;
    int st = ensure_pinned(c, 64);
    if (st) return st;
    MPM_CK(cudaMemcpyAsync(c->h_pinned, c->d_err + scene, sizeof(unsigned), cudaMemcpyDeviceToHost, c->stream));
    if ((st = wait_stream(c))) return st;
    *bits = *static_cast<unsigned*>(c->h_pinned);
    return MPM_OK;
}

static const int kFieldComps[6] = {3, 3, 9, 9, 1, 0};

extern "C" int mpm_read_state(mpm_ctx* c, int scene, uint32_t fields, void* const* dst, int mem)
{
    if (!c || !dst || scene < 0 || scene >= c->n_scenes || (fields & ~63u) || !fields) return MPM_ERR_INVALID_ARGUMENT;
    if (mem != MPM_MEM_HOST && mem != MPM_MEM_DEVICE) return MPM_ERR_INVALID_ARGUMENT;
    const SceneDev& sc = c->h_scenes[scene];
    const int np = sc.p_count;
    int nf = 0;
    for (int f = 0; f < 6; ++f)
        if (fields & (1u << f)) {
            if (!dst[nf]) return MPM_ERR_INVALID_ARGUMENT;
            ++nf;
        }
    int st;
    const PState cur = c->st[c->cur];
    // device staging for host reads that are not pinned; pinned host arrays of x, v, C and F
    // are written by the kernel itself
    bool mapped = mem == MPM_MEM_HOST && !(fields & ~15u);
    void* at[6] = {};  // where the kernels write each field
    for (int f = 0, k = 0; f < 6; ++f)
        if (fields & (1u << f)) {
            at[f] = mapped ? mapped_host(dst[k]) : dst[k];
            mapped = mapped && at[f];
            ++k;
        }
    const bool staged = mem == MPM_MEM_HOST && !mapped;
    size_t bytes[6] = {}, stage_need = 0, pin_need = 64;
    for (int f = 0, k = 0; f < 6; ++f) {
        if (!(fields & (1u << f))) continue;
        bytes[f] = f == 5 ? sizeof(double) * kMaxRigids * 6 : sizeof(float) * kFieldComps[f] * (size_t)np;
        if (staged) {
            stage_need += align256(bytes[f]);
            if (!is_pinned_host(dst[k])) pin_need += align256(bytes[f]);
        }
        ++k;
    }
    if ((st = ensure_stage(c, stage_need))) return st;
    if ((st = ensure_pinned(c, pin_need))) return st;
    if (staged) {
        size_t off = 0;
        for (int f = 0; f < 6; ++f)
            if (fields & (1u << f)) {
                at[f] = static_cast<char*>(c->d_stage) + off;
                off += align256(bytes[f]);
            }
    }
    if (fields & 15u) {
        Fields h{};
        for (int f = 0; f < 4; ++f) h.f[f] = static_cast<float*>(at[f]);
        MPM_CK(launch_fields(cur, c->st[c->cur ^ 1], c->cap, sc.p_begin, np, c->d_inv, h, true, mapped, c->stream));
    }
    if (fields & MPM_FIELD_ORDER) MPM_CK(launch_order(cur, sc.p_begin, np, static_cast<int*>(at[4]), c->stream));
    if (fields & MPM_FIELD_IMPULSE) {
        double* imp = c->d_impulse + (size_t)scene * kMaxRigids * 6;
        MPM_CK(cudaMemcpyAsync(at[5], imp, bytes[5], cudaMemcpyDeviceToDevice, c->stream));
        MPM_CK(cudaMemsetAsync(imp, 0, bytes[5], c->stream));
    }
    size_t poff = 64;
    struct Pending { void* dst; size_t poff, bytes; };
    std::vector<Pending> pend;
    for (int f = 0, k = 0; staged && f < 6; ++f) {
        if (!(fields & (1u << f))) continue;
        void* out = dst[k++];
        if (!bytes[f]) continue;
        if (is_pinned_host(out)) {
            MPM_CK(cudaMemcpyAsync(out, at[f], bytes[f], cudaMemcpyDeviceToHost, c->stream));
        } else {
            MPM_CK(cudaMemcpyAsync(static_cast<char*>(c->h_pinned) + poff, at[f], bytes[f], cudaMemcpyDeviceToHost, c->stream));
            pend.push_back({out, poff, bytes[f]});
            poff += align256(bytes[f]);
        }
    }
    MPM_CK(cudaMemcpyAsync(c->h_pinned, c->d_err + scene, sizeof(unsigned), cudaMemcpyDeviceToHost, c->stream));
    if ((st = wait_stream(c))) return st;
    for (auto& p : pend) memcpy(p.dst, static_cast<char*>(c->h_pinned) + p.poff, p.bytes);
    return error_status(*static_cast<unsigned*>(c->h_pinned));
}

extern "C" int mpm_write_state(mpm_ctx* c, int scene, uint32_t fields, const void* const* src, int mem)
{
    if (!c || !src || scene < 0 || scene >= c->n_scenes || !fields || (fields & ~15u)) return MPM_ERR_INVALID_ARGUMENT;
    if (mem != MPM_MEM_HOST && mem != MPM_MEM_DEVICE) return MPM_ERR_INVALID_ARGUMENT;
    if (c->recording) return MPM_ERR_STATE;
    const SceneDev& sc = c->h_scenes[scene];
    const int np = sc.p_count;
    size_t need = 0;
    for (int f = 0, k = 0; f < 4; ++f)
        if (fields & (1u << f)) {
            if (!src[k++]) return MPM_ERR_INVALID_ARGUMENT;
            need += align256(sizeof(float) * kFieldComps[f] * (size_t)np);
        }
    int st = MPM_OK;
    const PState cur = c->st[c->cur];
    Fields h{};
    bool mapped = mem == MPM_MEM_HOST;  // pinned host arrays are read by the kernel itself
    for (int f = 0, k = 0; f < 4; ++f)
        if (fields & (1u << f)) {
            h.f[f] = static_cast<float*>(mapped ? mapped_host(src[k]) : const_cast<void*>(src[k]));
            mapped = mapped && h.f[f];
            ++k;
        }
    if (mem == MPM_MEM_HOST && !mapped) {
        if ((st = ensure_stage(c, need))) return st;
        size_t off = 0;
        for (int f = 0, k = 0; f < 4; ++f) {
            if (!(fields & (1u << f))) continue;
            const size_t bytes = sizeof(float) * kFieldComps[f] * (size_t)np;
            const void* d = nullptr;
            if ((st = stage_input(c, src[k++], bytes, mem, off, &d))) return st;
            off += align256(bytes);
            h.f[f] = static_cast<float*>(const_cast<void*>(d));
        }
    }
    MPM_CK(launch_fields(cur, c->st[c->cur ^ 1], c->cap, sc.p_begin, np, c->d_inv, h, false, mapped, c->stream));
    // new positions need new brick keys; any new field changes the pending P2G
    if (fields & MPM_FIELD_X) c->keys_valid = false;
    invalidate_pending(c);
    if (mem == MPM_MEM_HOST) return wait_stream(c);
    return MPM_OK;
}

extern "C" int mpm_read_grid(mpm_ctx* c, int scene, float* dst, int mem)
{
    if (!c || !dst || scene < 0 || scene >= c->n_scenes) return MPM_ERR_INVALID_ARGUMENT;
    if (mem != MPM_MEM_HOST && mem != MPM_MEM_DEVICE) return MPM_ERR_INVALID_ARGUMENT;
    const int n = c->scene_n[scene];
    const size_t bytes = sizeof(float) * 4 * (size_t)n * n * n;
    int st;
    float* out = dst;
    if (mem == MPM_MEM_HOST) {
        if ((st = ensure_stage(c, bytes))) return st;
        out = static_cast<float*>(c->d_stage);
    }
    MPM_CK(cudaMemsetAsync(out, 0, bytes, c->stream));
    MPM_CK(launch_read_grid(c->V, c->brick_epoch, c->d_epoch, c->d_scenes, scene, n, c->brick_base[scene], out, c->stream));
    const bool direct = mem == MPM_MEM_HOST && is_pinned_host(dst);
    if (mem == MPM_MEM_HOST && !direct && (st = ensure_pinned(c, bytes))) return st;
    if (mem == MPM_MEM_HOST)
        MPM_CK(cudaMemcpyAsync(direct ? (void*)dst : c->h_pinned, out, bytes, cudaMemcpyDeviceToHost, c->stream));
    if ((st = wait_stream(c))) return st;
    if (mem == MPM_MEM_HOST && !direct) memcpy(dst, c->h_pinned, bytes);
    return MPM_OK;
}

extern "C" int mpm_autotune(mpm_ctx* c, float dt, int trial_substeps, float* best_ms_out)
{
    if (!c || !(dt > 0.f) || trial_substeps < 1 || trial_substeps > 1000) return MPM_ERR_INVALID_ARGUMENT;
    if (c->recording) return MPM_ERR_STATE;
    int st = upload_scenes(c);
    if (st) return st;
    if ((st = ensure_keys(c))) return st;
    // snapshot everything a substep changes
    const size_t sbytes = state_bytes(c->cap);
    const size_t nbk = (size_t)c->total_bricks;
    const size_t total = sbytes + 2 * sizeof(int) * c->cap + sizeof(int) * nbk * 66 + sizeof(int) * c->total_tiles +
                         (sizeof(double) + sizeof(int) + sizeof(unsigned) + sizeof(double) * kMaxRigids * 6) * c->n_scenes;
    char* snap = nullptr;
    MPM_CK(cudaMalloc(&snap, total));
    struct Item { void* live; size_t bytes; };
    const int cur0 = c->cur;
    Item items[] = {{c->state_mem[cur0], sbytes}, {c->sb.key, sizeof(int) * c->cap}, {c->sb.rank, sizeof(int) * c->cap},
                    {c->sb.cnt, sizeof(int) * nbk}, {c->sb.ccnt, sizeof(int) * nbk * 64},
                    {c->sb.tile_n, sizeof(int) * c->total_tiles},
                    {c->brick_epoch, sizeof(int) * nbk},
                    {c->d_time, sizeof(double) * c->n_scenes}, {c->d_epoch, sizeof(int) * c->n_scenes},
                    {c->d_err, sizeof(unsigned) * c->n_scenes},
                    {c->d_impulse, sizeof(double) * kMaxRigids * 6 * c->n_scenes}};
    auto copy_all = [&](bool save) -> cudaError_t {
        size_t off = 0;
        for (auto& it : items) {
            cudaError_t e = save ? cudaMemcpyAsync(snap + off, it.live, it.bytes, cudaMemcpyDeviceToDevice, c->stream)
                                 : cudaMemcpyAsync(it.live, snap + off, it.bytes, cudaMemcpyDeviceToDevice, c->stream);
            if (e != cudaSuccess) return e;
            off += it.bytes;
        }
        return cudaSuccess;
    };
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaError_t ce = copy_all(true);
    if (ce == cudaSuccess) ce = cudaEventCreate(&e0);
    if (ce == cudaSuccess) ce = cudaEventCreate(&e1);
    int best[4] = {c->p2g_chunk, c->g2p_threads, c->ctas_per_sm, c->g2p_regs64};
    float best_ms = 3.4e38f;
    const int chunks[3] = {2 * kP2GThreads, 3 * kP2GThreads, 4 * kP2GThreads};
    const int threads[3] = {128, 256, 512};
    const int ctas[2] = {0, 2};
    const int T = trial_substeps + (trial_substeps & 1);
    const bool tau_valid0 = c->tau_valid;
    const bool graphs = c->use_graphs && !c->phase_timing;
    for (int a = 0; a < 3 && ce == cudaSuccess && st == MPM_OK; ++a)
        for (int b = 0; b < 3 && ce == cudaSuccess && st == MPM_OK; ++b)
            for (int r64 = 0; r64 < 2 && ce == cudaSuccess && st == MPM_OK; ++r64)
            for (int k = 0; k < 2 && ce == cudaSuccess && st == MPM_OK; ++k) {
                c->p2g_chunk = chunks[a];
                c->g2p_threads = threads[b];
                c->g2p_regs64 = r64;
                c->ctas_per_sm = ctas[k];
                c->tau_valid = tau_valid0;  // the restored state's stored stress
                // one untimed warm-up substep from a clean accumulator, then the timed trial:
                // graph replays (an even number of substeps, so that the replayed graph
                // reads the buffer it was captured for) when graphs are on, else direct launches
                ce = cudaMemsetAsync(c->G, 0, sizeof(float4) * nbk * 64, c->stream);
                if (ce == cudaSuccess) st = enqueue_substep(c, dt, c->st[c->cur], c->st[c->cur ^ 1], true);
                c->cur ^= 1;
                if (graphs) {
                    cudaGraph_t g = nullptr;
                    cudaGraphExec_t ex = nullptr;
                    if (!st && ce == cudaSuccess) ce = cudaStreamBeginCapture(c->stream, cudaStreamCaptureModeThreadLocal);
                    if (!st && ce == cudaSuccess) {
                        int cur = c->cur;
                        for (int s = 0; s < T && !st; ++s) {
                            st = enqueue_substep(c, dt, c->st[cur], c->st[cur ^ 1], false);
                            cur ^= 1;
                        }
                        const cudaError_t ce2 = cudaStreamEndCapture(c->stream, &g);
                        if (ce == cudaSuccess) ce = ce2;
                    }
                    if (!st && ce == cudaSuccess) ce = cudaGraphInstantiate(&ex, g, 0);
                    if (g) cudaGraphDestroy(g);
                    if (!st && ce == cudaSuccess) ce = cudaGraphLaunch(ex, c->stream);
                    if (!st && ce == cudaSuccess) ce = cudaEventRecord(e0, c->stream);
                    if (!st && ce == cudaSuccess) ce = cudaGraphLaunch(ex, c->stream);
                    if (!st && ce == cudaSuccess) ce = cudaEventRecord(e1, c->stream);
                    if (!st && ce == cudaSuccess) st = wait_stream(c);
                    if (ex) cudaGraphExecDestroy(ex);
                } else {
                    if (!st && ce == cudaSuccess) ce = cudaEventRecord(e0, c->stream);
                    for (int s = 0; s < T && !st && ce == cudaSuccess; ++s) {
                        st = enqueue_substep(c, dt, c->st[c->cur], c->st[c->cur ^ 1], false);
                        c->cur ^= 1;
                    }
                    if (!st && ce == cudaSuccess) ce = cudaEventRecord(e1, c->stream);
                    if (!st && ce == cudaSuccess) st = wait_stream(c);
                }
                float ms = 0.f;
                if (!st && ce == cudaSuccess) ce = cudaEventElapsedTime(&ms, e0, e1);
                ms /= T;
                if (!st && ce == cudaSuccess && ms < best_ms) {
                    best_ms = ms;
                    best[0] = chunks[a];
                    best[1] = threads[b];
                    best[2] = ctas[k];
                    best[3] = r64;
                }
                c->cur = cur0;
                if (ce == cudaSuccess) ce = copy_all(false);
            }
    if (ce == cudaSuccess && st == MPM_OK) st = wait_stream(c);
    c->cur = cur0;
    // the trials left scatters in G that do not belong to the restored state
    c->g_pending = false;
    c->g_dirty = true;
    c->tau_valid = tau_valid0;
    c->p2g_chunk = best[0];
    c->g2p_threads = best[1];
    c->g2p_regs64 = best[3];
    c->ctas_per_sm = best[2];
    clear_graphs(c);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    cudaFree(snap);
    if (ce != cudaSuccess) return status_from_cuda(ce);
    if (st) return st;
    if (best_ms_out) *best_ms_out = best_ms;
    return MPM_OK;
}

extern "C" int mpm_phase_stats(mpm_ctx* c, double* ms, int64_t* n_substeps, int64_t* active, int reset)
{
    if (!c) return MPM_ERR_INVALID_ARGUMENT;
    int st = ensure_pinned(c, 64);
    if (st) return st;
    MPM_CK(cudaMemcpyAsync(c->h_pinned, c->sb.counters, sizeof(int) * 2, cudaMemcpyDeviceToHost, c->stream));
    if ((st = wait_stream(c))) return st;
    double sum[4] = {0, 0, 0, 0};
    for (size_t k = 0; k + 5 <= c->phase_used; k += 5)
        for (int p = 0; p < 4; ++p) {
            float t = 0.f;
            MPM_CK(cudaEventElapsedTime(&t, c->phase_events[k + p], c->phase_events[k + p + 1]));
            sum[p] += t;
        }
    if (ms)
        for (int p = 0; p < 4; ++p) ms[p] = sum[p];
    if (n_substeps) *n_substeps = (int64_t)(c->phase_used / 5);
    if (active) {
        active[0] = static_cast<int*>(c->h_pinned)[0];
        active[1] = static_cast<int*>(c->h_pinned)[1];
    }
    if (reset) c->phase_used = 0;
    return MPM_OK;
}
