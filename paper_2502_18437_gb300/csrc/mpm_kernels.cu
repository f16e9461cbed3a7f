// Forward substep kernels of the MLS-MPM transfer loop (arXiv 2502.18437,
// Algorithm 1) for GB300 (sm_103a):
//   k_scan     brick histogram -> particle offsets, active particle-brick and
//              node-brick lists (tile counts kept by the key producers: no
//              inter-CTA waits, empty tiles skipped)
//   k_scatter  counting-sort scatter: permutation sorted slot -> particle, by brick
//              and cell
//   k_p2g      P2G (Eq. 1, Eq. 8; standard MPM Eq. 2, 3): runs of particles of one
//              cell summed in registers, added to HBM with vector atomics
//   k_grid     grid update (Eq. 3), rigid contact (Sec. IV, Eq. 11, Eq. 12),
//              domain walls (k_grid_plain where no scene has a rigid)
//   k_grid_clear  reset of the P2G accumulator where no G2P does it
//   k_g2p      G2P (Eq. 4, Eq. 9, Eq. 10), one thread per slot with its stencil
//              through L1, plasticity, next brick key + rank, reset of the accumulator
#include <cstdint>
#include <cstdio>

#include "mpm_transfer.cuh"

namespace mpm {

// ----------------------------------------------------------------- scan
//
// A scan tile is 2^tile_shift consecutive bricks of one scene (tiles never
// straddle scenes).  The key producers (G2P, k_prepare) count the particles of
// every brick and every tile as they go, so each CTA of the scan (one per tile of
// the range) knows the first slot of its bricks from the tile counts before it,
// without waiting for another CTA.  The list of node bricks (the grid update's and the
// reset's) needs no order, that of particle bricks (the fused kernel's; the others only
// ask whether it is empty) only the big bricks first, so that the fused kernel's CTAs
// end on small ones: each CTA appends its own to them with one atomic per list.  A node brick is active when it or one of its 7
// lower neighbours (-1 in any subset of the axes) holds particles, since a
// particle's 3-node stencil reaches at most 2 nodes beyond its base cell, i.e.
// into the next brick: the scan looks the 8 counts up.  (Before, the first warp of
// G2P to reach a brick marked 8 flags with one exchange after the other: 17 us of
// G2P's 81 on a 1M block.)  A tile that no particle can reach returns at once.

// Sum of v over the CTA's threads before this one (excl) and over all (total).
__device__ __forceinline__ void block_scan(int v, int* s_warp, int& excl, int& total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int t = __shfl_up_sync(kFull, incl, d);
        if (lane >= d) incl += t;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    int before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < kScanThreads / 32; ++w) {
        const int t = s_warp[w];
        if (w < warp) before += t;
        all += t;
    }
    __syncthreads();
    excl = before + incl - v;
    total = all;
}

__global__ void __launch_bounds__(kScanThreads) k_scan(StepArgs a)
{
    chain_wait();
    __shared__ int s_warp[kScanThreads / 32];
    __shared__ int s_sum[3][kScanThreads / 32];
    __shared__ int s_base[3], s_total[3];
    __shared__ int s_brick[kScanThreads], s_start[kScanThreads];  // the chunk's particle bricks
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const SortBufs& sb = a.sb;
    const int tile = a.r.t0 + blockIdx.x;
    if (blockIdx.x == 0 && tid == 0) sb.counters[CTR_WORK_G2P] = 0;
    // scene of the tile
    int s = a.r.s0;
    if (a.r.s1 - a.r.s0 > 1) {
        int hi = a.r.s1 - 1;
        while (s < hi) {
            const int mid = (s + hi + 1) >> 1;
            if (a.scenes[mid].tile_base <= tile) s = mid;
            else hi = mid - 1;
        }
    }
    const SceneDev& sc = a.scenes[s];
    if (a.any_rigid && tile == sc.tile_base && tid < sc.n_rigid) {
        // the rigids' poses at the scene's clock, for the grid update
        RigidPose& P = a.pose[s * kMaxRigids + tid];
        rigid_pose_at(a.rigids[s * kMaxRigids + tid], a.t_scene[s], P.c, P.R);
    }
    const int nb = sc.nb, bricks = nb * nb * nb;
    const int l0 = (tile - sc.tile_base) << sb.tile_shift, l1 = min(l0 + (1 << sb.tile_shift), bricks);
    // particles of the tiles before this one, of the whole range, and of the tiles
    // whose particles can activate a node brick here
    const int near0 = sc.tile_base + (max(l0 - nb * nb - nb - 1, 0) >> sb.tile_shift);
    int pre = 0, all = 0, near = 0;
    for (int t = a.r.t0 + tid; t < a.r.t0 + a.r.nt; t += kScanThreads) {
        const int c = __ldcg(&sb.tile_n[t]);
        all += c;
        if (t < tile) pre += c;
        if (t >= near0 && t <= tile) near |= c;
    }
    pre = __reduce_add_sync(kFull, pre);
    all = __reduce_add_sync(kFull, all);
    near = __reduce_or_sync(kFull, near);
    if (lane == 0) {
        s_sum[0][warp] = pre;
        s_sum[1][warp] = all;
        s_sum[2][warp] = near;
    }
    __syncthreads();
    pre = all = near = 0;
#pragma unroll
    for (int w = 0; w < kScanThreads / 32; ++w) {
        pre += s_sum[0][w];
        all += s_sum[1][w];
        near |= s_sum[2][w];
    }
    if (all != a.r.np) {
        // histogram and particle count disagree: empty lists skip this substep's work
        if (blockIdx.x == 0 && tid == 0) atomicOr(&a.err[a.r.s0], MPM_EBIT_INTERNAL);
        return;
    }
    if (near == 0) return;
    const unsigned lt = (1u << lane) - 1u;
    int start0 = a.r.p0 + pre;
    for (int chunk = l0; chunk < l1; chunk += kScanThreads) {
        const int lb = chunk + tid, b = sc.brick_base + lb;
        int c = 0;
        bool node = false;
        if (lb < l1) {
            const int* cnt = sb.cnt + b;
            int bx, by, bz;
            brick_coords(nb, sc.nb_log2, lb, bx, by, bz);
            int n[8];
#pragma unroll
            for (int o = 0; o < 8; ++o) {
                const int dx = o >> 2, dy = (o >> 1) & 1, dz = o & 1;
                n[o] = bx >= dx && by >= dy && bz >= dz ? __ldcg(cnt - (dx * nb + dy) * nb - dz) : 0;
            }
            c = n[0];
#pragma unroll
            for (int o = 0; o < 8; ++o) node = node || n[o] > 0;
        }
        int before, total;
        block_scan(c, s_warp, before, total);
        // places in the lists
        const unsigned big = __ballot_sync(kFull, c >= kBigBrick), small = __ballot_sync(kFull, c > 0 && c < kBigBrick),
                       nodes = __ballot_sync(kFull, node);
        if (lane == 0) {
            s_sum[0][warp] = __popc(big);
            s_sum[1][warp] = __popc(small);
            s_sum[2][warp] = __popc(nodes);
        }
        __syncthreads();
        if (tid < 3) {
            int t = 0;
#pragma unroll
            for (int w = 0; w < kScanThreads / 32; ++w) {
                const int k = s_sum[tid][w];
                s_sum[tid][w] = t;
                t += k;
            }
            s_base[tid] = t ? atomicAdd(&sb.counters[CTR_N_BIG + tid], t) : 0;
            s_total[tid] = t;
        }
        __syncthreads();
        if (c > 0) {
            const int e = c >= kBigBrick
                              ? s_base[0] + s_sum[0][warp] + __popc(big & lt)
                              : sb.list_size - 1 - (s_base[1] + s_sum[1][warp] + __popc(small & lt));
            const int start = start0 + before;
            const int at = s_sum[0][warp] + s_sum[1][warp] + __popc((big | small) & lt);
            s_brick[at] = b;
            s_start[at] = start;
            sb.act_brick[e] = b;
            sb.act_start[e] = start;
            sb.act_count[e] = c;
            sb.act_scene[e] = s;
        }
        if (node) {
            const int e = s_base[2] + s_sum[2][warp] + __popc(nodes & lt);
            sb.nact_brick[e] = b;
            sb.nact_scene[e] = s;
        }
        start0 += total;
        __syncthreads();
        // a warp per brick: its cells' counts become their first slots
        const int n_act = s_total[0] + s_total[1];
#pragma unroll 4
        for (int i = warp; i < n_act; i += kScanThreads / 32) {
            int2* cells = reinterpret_cast<int2*>(sb.ccnt + (size_t)s_brick[i] * 64) + lane;
            const int2 k = *cells;
            int incl = k.x + k.y;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int t = __shfl_up_sync(kFull, incl, d);
                if (lane >= d) incl += t;
            }
            const int even = s_start[i] + incl - k.x - k.y;
            *cells = make_int2(even, even + k.x);
        }
        __syncthreads();  // the shared lists are rewritten by the next chunk
    }
}

__global__ void k_reset_histogram(SortBufs sb, int bricks, int tiles)
{
    chain_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < bricks && sb.cnt[i]) {
        // only bricks with particles have counts in their cells
        sb.cnt[i] = 0;
        for (int k = 0; k < 16; ++k) reinterpret_cast<int4*>(sb.ccnt + (size_t)i * 64)[k] = make_int4(0, 0, 0, 0);
    }
    if (i < tiles) sb.tile_n[i] = 0;
    if (i >= CTR_N_BIG && i <= CTR_N_NACT) sb.counters[i] = 0;
}

// Counting-sort scatter: a particle's slot is its cell's first slot plus its rank.  Also
// clears the range's tile counts for the next substep (the scan has read them).
// Each thread takes kScatterPer particles, 256 apart, with their loads issued
// together (a 1M-particle range in one wave of CTAs).
// (The cells' first slots come from the scan, a warp a brick: 1M particles 5.4 us.  Taken
// here, by each warp for its particles' bricks, 10.5 us, and 89 us for particles in no order.)
__global__ void __launch_bounds__(256) k_scatter(StepArgs a)
{
    chain_wait();
    const int g0 = blockIdx.x * (256 * kScatterPer) + threadIdx.x;
    int key[kScatterPer], rank[kScatterPer], dst[kScatterPer];
#pragma unroll
    for (int u = 0; u < kScatterPer; ++u) {
        const int g = g0 + u * 256;
        key[u] = -1;
        rank[u] = 0;
        if (g < a.r.np) {
            key[u] = a.sb.key[a.r.p0 + g];
            rank[u] = a.sb.rank[a.r.p0 + g];
        }
    }
#pragma unroll
    for (int u = 0; u < kScatterPer; ++u) {
        const int brick = key[u] >> 6;
        dst[u] = (key[u] >= 0 && brick >= a.r.bb0 && brick < a.r.bb0 + a.r.nbr) ? a.sb.ccnt[key[u]] + rank[u] : -1;
    }
#pragma unroll
    for (int u = 0; u < kScatterPer; ++u) {
        const int g = g0 + u * 256;
        if (g < a.r.np) {
            if (dst[u] >= a.r.p0 && dst[u] < a.r.p0 + a.r.np) a.sb.perm[dst[u]] = a.r.p0 + g;
            else atomicOr(&a.err[a.r.s0], MPM_EBIT_INTERNAL);
        }
        if (g < a.r.nt) a.sb.tile_n[a.r.t0 + g] = 0;
    }
}

// Keys and ranks of the stored particles after the host changed positions
// (new particles, state writes).  Stored particles may be in any order here, so
// the tiles' particle counts are first summed per block in shared memory (with
// at most kPrepTiles tiles in the range; else each warp adds its own).
constexpr int kPrepTiles = 2048;

__global__ void __launch_bounds__(256) k_prepare(StepArgs a, PState st)
{
    chain_wait();
    __shared__ int s_tile[kPrepTiles];
    const bool block_sums = a.r.nt <= kPrepTiles;
    if (block_sums)
        for (int t = threadIdx.x; t < a.r.nt; t += blockDim.x) s_tile[t] = 0;
    __syncthreads();
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    const int i = a.r.p0 + g;
    const bool valid = g < a.r.np;
    int key = 0, scene = a.r.s0;
    unsigned ebits = 0;
    if (valid) {
        int lo = a.r.s0, hi = a.r.s1 - 1;
        while (lo < hi) {
            int mid = (lo + hi + 1) >> 1;
            if (a.scenes[mid].p_begin <= i) lo = mid;
            else hi = mid - 1;
        }
        scene = lo;
    }
    const SceneDev sc = a.scenes[scene];
    if (valid) {
        unsigned ood = 0;
        float x[3];
        load_x(st, i, x);
        key = cell_key(sc, x[0], x[1], x[2], ood);
        if (ood) ebits |= MPM_EBIT_OUT_OF_DOMAIN;
    }
    const int rank = cell_rank_end(cell_rank_begin(a.sb, sc, key, valid, !block_sums));
    if (valid) {
        a.sb.key[i] = key;
        a.sb.rank[i] = rank;
        if (ebits) atomicOr(&a.err[scene], ebits);
        if (block_sums)
            atomicAdd(&s_tile[sc.tile_base + (((key >> 6) - sc.brick_base) >> a.sb.tile_shift) - a.r.t0], 1);
    }
    if (block_sums) {
        __syncthreads();
        for (int t = threadIdx.x; t < a.r.nt; t += blockDim.x)
            if (s_tile[t]) atomicAdd(&a.sb.tile_n[a.r.t0 + t], s_tile[t]);
    }
}

// ------------------------------------------------------------------ P2G
//
// Warps work on their own chunks of sorted slots, without barriers:
//   A. one lane per particle: weights and coefficients into a record in the warp's
//      share of the shared memory, and the runs of slots with the same base cell
//      (the slots are in cell order);
//   B. one lane per (run, node plane x = i) sums its particles' contributions to the
//      9 nodes (i, j, k) of the cell in registers;
//   C. the sums of runs that are neighbours in z are joined by shuffles, and each node
//      of the joined runs added to HBM with one vector reduction.
// What bounds it is the instruction issue of B (61 % of the cycles; 28.4 M warp
// instructions per launch on the 1M block) and the loads of A, which are copied one
// batch ahead.  Before, a CTA took a brick: ranks in its cells, work items, staged item
// sums and a 6^3 window, one behind the other with a barrier between: 35.7 M
// instructions, 13.5 us for a lone brick and so 66 us for the 1M block's 2,744 and 19 us
// for 64k particles.  Now 43 and 8.5 us, 5.9 us at 4k; PB-MPM's cycles at 131k 39 -> 16 us.
// The standard MPM's took shared-memory atomics, 97 us at 131k; now its whole substep
// takes 41 us.
// Joining halves the reductions, and with them the error of the sums: C of a falling 64k
// block is 4.8e-6 off after 25 substeps, as before; without, 5.4e-6.
// Tried: a lane per node column (j, k), three groups of lanes at a third of the chunk
// each: 56 us, every lane reads 18 floats per particle from shared memory; the layer's
// sums joined in a window of 3 x 6 x 6 nodes: 62 us.

constexpr int kP2GWarps = kP2GThreads / 32;
constexpr int kRawPlanes = 7;  // planes of the state that a lane reads

// shared bytes of a warp: records, the next particles' planes, scenes and first slots of the runs
__host__ __device__ constexpr int p2g_warp_bytes(int slots)
{
    return slots * (kRecPitch + 1) * (int)sizeof(float) + kRawPlanes * 32 * (int)sizeof(float4) + ((slots + 8) * (int)sizeof(short) + 15) / 16 * 16;
}

// Record of the particle in storage p, returning its base node's index (key):
//   fx wy[3] wz[3] -, then for MLS- and PB-MPM q0 q1 A00 A10, A01 A11 A02 A12,
//   q2 A20 A21 A22: the momentum of node (i, j, k) is W (q + A (i-1, j-1, k-1)) (offsets
//   from the middle node keep the terms that cancel small); for the standard MPM
//   m v[3] fy, T0 T1 T2 T3, T4 T5 fz - with T = dt V0 n tau.
// plane(k) returns plane k of the particle's state.
template <int MODE, class Plane>
__device__ __forceinline__ unsigned p2g_record(const StepArgs& a, const SceneDev& sc, int p, Plane plane, float4* rec,
                                               int& key)
{
    const int n = sc.n, nb = sc.nb;
    const float fn = (float)n, m = sc.m_p;
    int bc[3];
    float f[3], w[9], v[3], C[9], t6[6];
    const float4 x = plane(0), Fv = plane(3);
    v[0] = Fv.y; v[1] = Fv.z; v[2] = Fv.w;
    const auto get_F = [&](float* F) {
        const float4 u = plane(1), t = plane(2);
        F[0] = u.x; F[1] = u.y; F[2] = u.z; F[3] = u.w;
        F[4] = t.x; F[5] = t.y; F[6] = t.z; F[7] = t.w;
        F[8] = Fv.x;
    };
    if (MODE != kP2GStd) {
        const float4 u = plane(4), t = plane(5);
        C[0] = u.x; C[1] = u.y; C[2] = u.z; C[3] = u.w;
        C[4] = t.x; C[5] = t.y; C[6] = t.z; C[7] = t.w;
        C[8] = plane(6).x;
    }
    unsigned ebits = particle_weights(x.x, x.y, x.z, n, bc, f, w);
    key = (sc.brick_base + ((bc[0] >> 2) * nb + (bc[1] >> 2)) * nb + (bc[2] >> 2)) * 64 + (bc[0] & 3) * 16 +
          (bc[1] & 3) * 4 + (bc[2] & 3);
    if (MODE == kP2GConstraint) {
        float F[9];
        get_F(F);
        pb_constraint(F, a.dt, a.pb_beta, C);
#pragma unroll
        for (int q = 0; q < 6; ++q) t6[q] = 0.f;
    } else if (a.tau_valid) {
        const float4 u = plane(6), t = plane(7);
        t6[0] = u.y; t6[1] = u.z; t6[2] = u.w;
        t6[3] = t.x; t6[4] = t.y; t6[5] = t.z;
    } else {
        // stress of the current F (after host writes, or seeding a fused run)
        float F[9];
        get_F(F);
        const float mu = sc.pp_mat ? a.in.mu[p] : sc.mu, lam = sc.pp_mat ? a.in.lam[p] : sc.lam;
        ebits |= constitutive(a.model, 0, 0.f, mu, lam, F, t6);
    }
    rec[0] = make_float4(f[0], w[3], w[4], w[5]);
    rec[1] = make_float4(w[6], w[7], w[8], __int_as_float(key));
    if (MODE == kP2GStd) {
        const float kap = a.dt * sc.V0 * fn;  // dt V0 times the n of grad W = n dW/df
        rec[2] = make_float4(m * v[0], m * v[1], m * v[2], f[1]);
        rec[3] = make_float4(kap * t6[0], kap * t6[1], kap * t6[2], kap * t6[3]);
        rec[4] = make_float4(kap * t6[4], kap * t6[5], f[2], 0.f);
    } else {
        float q[3], Ad[9];
        const float fc[3] = {f[0] - 1.f, f[1] - 1.f, f[2] - 1.f};
        p2g_coeffs(m, a.dt * sc.V0 * 4.0f * fn * fn, 1.0f / fn, v, C, t6, fc, q, Ad);
        rec[2] = make_float4(q[0], q[1], Ad[0], Ad[3]);
        rec[3] = make_float4(Ad[1], Ad[4], Ad[2], Ad[5]);
        rec[4] = make_float4(q[2], Ad[6], Ad[7], Ad[8]);
    }
    return ebits;
}

template <int MODE>
__global__ void __launch_bounds__(kP2GThreads, 4) k_p2g(StepArgs a)
{
    chain_wait();
    extern __shared__ __align__(16) unsigned char p2g_smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int slots = a.p2g_slots, np = a.r.np;
    float4* rec = reinterpret_cast<float4*>(p2g_smem + warp * p2g_warp_bytes(slots));
    float4* raw = rec + slots * (kRecPitch / 4) + lane;
    int* s_scene = reinterpret_cast<int*>(raw - lane + kRawPlanes * 32);
    short* s_start = reinterpret_cast<short*>(s_scene + slots);
    if (active_bricks(a.sb) == 0) return;  // the sort found its bookkeeping inconsistent
    // planes that are read, and where they are staged: with the stored stress 0 and 3-7,
    // else 0-6
    const bool stored = MODE != kP2GConstraint && a.tau_valid;
    const auto at = [&](int k) { return raw + 32 * (k > 0 && stored ? k - 2 : k); };
    const auto copy_planes = [&](int p) {
        if (p >= 0) {
#pragma unroll
            for (int k = 0; k < kPlanes; ++k)
                if (stored ? (k == 0 || k == 3 || k > 5 || (MODE != kP2GStd && k > 3)) : k < 7)
                    cp_async16(at(k), a.in.q + (size_t)k * a.cap + p);
        }
        cp_async_commit();
    };
    // batches of 32 slots, chunk by chunk: storage index of the lane's slot (the lanes
    // beyond the chunk's last one repeat it), or -1 after the last chunk
    const int step = gridDim.x * kP2GWarps * slots;
    const auto source = [&](int base, int q0) {
        if (q0 >= min(slots, np - base)) {
            base += step;
            q0 = 0;
        }
        return base < np ? a.sb.perm[a.r.p0 + min(base + min(q0 + lane, slots - 1), np - 1)] : -1;
    };
    int p = source((blockIdx.x * kP2GWarps + warp) * slots, 0);
    copy_planes(p);
    for (int base = (blockIdx.x * kP2GWarps + warp) * slots; base < np; base += step) {
        const int cnt = min(slots, np - base);
        // A
        int runs = 0, last = -1;
        for (int q0 = 0; q0 < cnt; q0 += 32) {
            const int q = q0 + lane, s = a.r.p0 + base + min(q, cnt - 1);
            const int scene = scene_of_slot(a, s);
            const int p_next = source(base, q0 + 32);
            int key = -1;
            cp_async_wait<0>();
            if (q < cnt) {
                const unsigned ebits = p2g_record<MODE>(
                    a, a.scenes[scene], p, [&](int k) { return *at(k); }, rec + q * (kRecPitch / 4), key);
                s_scene[q] = scene;
                if (ebits) atomicOr(&a.err[scene], ebits);
            }
            p = p_next;
            copy_planes(p);
            const int up = __shfl_up_sync(kFull, key, 1);
            const bool head = q < cnt && key != (lane ? up : last);
            const unsigned heads = __ballot_sync(kFull, head);
            if (head) s_start[runs + __popc(heads & ((1u << lane) - 1u))] = (short)q;
            runs += __popc(heads);
            last = __shfl_sync(kFull, key, 31);
        }
        if (lane == 0) s_start[runs] = (short)cnt;
        __syncwarp();
        scatter_runs<MODE>(a, rec, s_scene, s_start, runs);
        __syncwarp();  // the records are rewritten
    }
    cp_async_wait<0>();
}

// ----------------------------------------------------------- grid update


// Nearest point q of segment [a, b] to p (endpoint projections keep the
// segment); returns |p - q|.
__device__ __forceinline__ float closest_on_segment_f(float p0, float p1, float p2, const float* a, const float* b,
                                                      float q[3])
{
    const float e0 = b[0] - a[0], e1 = b[1] - a[1], e2 = b[2] - a[2];
    const float L2 = e0 * e0 + e1 * e1 + e2 * e2;
    float u = L2 > 0.f ? ((p0 - a[0]) * e0 + (p1 - a[1]) * e1 + (p2 - a[2]) * e2) / L2 : 0.f;
    u = fminf(fmaxf(u, 0.f), 1.f);
    q[0] = a[0] + u * e0;
    q[1] = a[1] + u * e1;
    q[2] = a[2] + u * e2;
    const float d0 = p0 - q[0], d1 = p1 - q[1], d2 = p2 - q[2];
    return sqrtf(d0 * d0 + d1 * d1 + d2 * d2);
}

// Nearest point q of triangle (a, b, c) to p: the orthogonal projection when
// its barycentric coordinates (2x2 normal equations of the plane) lie inside
// (inside = true), else the nearest of the three edges' nearest points.
__device__ __forceinline__ float closest_on_triangle_f(float p0, float p1, float p2, const float* a, const float* b,
                                                       const float* c, float q[3], bool& inside)
{
    const float e0[3] = {b[0] - a[0], b[1] - a[1], b[2] - a[2]}, e1[3] = {c[0] - a[0], c[1] - a[1], c[2] - a[2]};
    const float ap[3] = {p0 - a[0], p1 - a[1], p2 - a[2]};
    const float d00 = e0[0] * e0[0] + e0[1] * e0[1] + e0[2] * e0[2];
    const float d01 = e0[0] * e1[0] + e0[1] * e1[1] + e0[2] * e1[2];
    const float d11 = e1[0] * e1[0] + e1[1] * e1[1] + e1[2] * e1[2];
    const float d20 = ap[0] * e0[0] + ap[1] * e0[1] + ap[2] * e0[2];
    const float d21 = ap[0] * e1[0] + ap[1] * e1[1] + ap[2] * e1[2];
    const float den = d00 * d11 - d01 * d01;
    inside = false;
    if (den > 0.f) {
        const float s = (d11 * d20 - d01 * d21) / den, t = (d00 * d21 - d01 * d20) / den;
        if (s >= 0.f && t >= 0.f && s + t <= 1.f) {
#pragma unroll
            for (int i = 0; i < 3; ++i) q[i] = a[i] + s * e0[i] + t * e1[i];
            inside = true;
            const float d0 = p0 - q[0], d1 = p1 - q[1], d2 = p2 - q[2];
            return sqrtf(d0 * d0 + d1 * d1 + d2 * d2);
        }
    }
    float qa[3], qb[3], qc[3];
    const float da = closest_on_segment_f(p0, p1, p2, a, b, qa), db = closest_on_segment_f(p0, p1, p2, b, c, qb),
                dc = closest_on_segment_f(p0, p1, p2, c, a, qc);
    float best = da;
    q[0] = qa[0]; q[1] = qa[1]; q[2] = qa[2];
    if (db < best) { best = db; q[0] = qb[0]; q[1] = qb[1]; q[2] = qb[2]; }
    if (dc < best) { best = dc; q[0] = qc[0]; q[1] = qc[1]; q[2] = qc[2]; }
    return best;
}

// Region of the triangle-mesh slicer at body point p (3 sticky spine, 1
// regular, 0 none) and its body-frame normal nl.
__device__ __forceinline__ int mesh_slicer_region(const RigidDev& R, float p0, float p1, float p2, float nl[3])
{
    float dsp = 3.4e38f;
    for (int k = 0; k + 1 < R.n_spine; ++k) {
        const float* a = R.shape.pts + 3 * R.shape.spine[k];
        const float* b = R.shape.pts + 3 * R.shape.spine[k + 1];
        float q[3];
        dsp = fminf(dsp, closest_on_segment_f(p0, p1, p2, a, b, q));
    }
    if (dsp < R.spine_radius + R.margin) return 3;
    float best = 3.4e38f, bq[3] = {0.f, 0.f, 0.f};
    int bt = -1;
    bool binside = false;
    for (int k = 0; k < R.n_tris; ++k) {
        const unsigned char* tv = R.shape.tris + 3 * k;
        float q[3];
        bool inside;
        const float l = closest_on_triangle_f(p0, p1, p2, R.shape.pts + 3 * tv[0], R.shape.pts + 3 * tv[1],
                                              R.shape.pts + 3 * tv[2], q, inside);
        if (l < best) { best = l; bq[0] = q[0]; bq[1] = q[1]; bq[2] = q[2]; bt = k; binside = inside; }
    }
    if (bt < 0 || !(best < 0.5f * R.thickness + R.margin)) return 0;
    if (binside) {
        const unsigned char* tv = R.shape.tris + 3 * bt;
        const float* a = R.shape.pts + 3 * tv[0];
        const float* b = R.shape.pts + 3 * tv[1];
        const float* c = R.shape.pts + 3 * tv[2];
        const float e0[3] = {b[0] - a[0], b[1] - a[1], b[2] - a[2]};
        const float e1[3] = {c[0] - a[0], c[1] - a[1], c[2] - a[2]};
        const float m0 = e0[1] * e1[2] - e0[2] * e1[1], m1 = e0[2] * e1[0] - e0[0] * e1[2],
                    m2 = e0[0] * e1[1] - e0[1] * e1[0];
        const float ln = sqrtf(m0 * m0 + m1 * m1 + m2 * m2);
        const float sg = ((p0 - bq[0]) * m0 + (p1 - bq[1]) * m1 + (p2 - bq[2]) * m2) >= 0.f ? 1.f : -1.f;
        nl[0] = sg * m0 / ln; nl[1] = sg * m1 / ln; nl[2] = sg * m2 / ln;
    } else if (best > 0.f) {
        nl[0] = (p0 - bq[0]) / best; nl[1] = (p1 - bq[1]) / best; nl[2] = (p2 - bq[2]) / best;
    }
    return 1;
}

// Region test of one rigid at world point x (Sec. IV).  Returns 0 none,
// 1 regular, 2 one-dimensional (segments), 3 sticky (slicer spine); n is the
// contact normal (zero when undefined) and t the 1D tangent.
// EXT: the launch has arcs or mesh slicers (a separate instance of the grid
// kernel, so that the common shapes keep their registers).
template <bool EXT>
__device__ int rigid_region(const RigidDev& R, const RigidPose& P, float3 x, float3& n, float3& t)
{
    const float dx0 = x.x - P.c[0], dx1 = x.y - P.c[1], dx2 = x.z - P.c[2];
    // body coordinates p = R^T (x - c)
    const float p0 = P.R[0] * dx0 + P.R[3] * dx1 + P.R[6] * dx2;
    const float p1 = P.R[1] * dx0 + P.R[4] * dx1 + P.R[7] * dx2;
    const float p2 = P.R[2] * dx0 + P.R[5] * dx1 + P.R[8] * dx2;
    float nl0 = 0.f, nl1 = 0.f, nl2 = 0.f, tl0 = 0.f, tl1 = 0.f, tl2 = 0.f;
    int code = 0;
    // a thread's segments (or a mesh's triangles) are looked at by the nodes near it only:
    // with a blade and a 32-segment thread in a slab of 262k particles a substep takes 53.9
    // us instead of 60.2
    const bool near = p0 >= R.lo[0] && p0 <= R.hi[0] && p1 >= R.lo[1] && p1 <= R.hi[1] && p2 >= R.lo[2] && p2 <= R.hi[2];
    if (R.type == MPM_SPHERE) {
        const float l = sqrtf(p0 * p0 + p1 * p1 + p2 * p2);
        if (l - R.radius < R.margin) {
            code = 1;
            if (l > 0.f) { nl0 = p0 / l; nl1 = p1 / l; nl2 = p2 / l; }
            else nl1 = 1.f;
        }
    } else if (R.type == MPM_BOX) {
        const float q0 = fabsf(p0) - R.half[0], q1 = fabsf(p1) - R.half[1], q2 = fabsf(p2) - R.half[2];
        const float o0 = fmaxf(q0, 0.f), o1 = fmaxf(q1, 0.f), o2 = fmaxf(q2, 0.f);
        const float out = sqrtf(o0 * o0 + o1 * o1 + o2 * o2);
        const float mx = fmaxf(q0, fmaxf(q1, q2));
        const float sdf = out + fminf(mx, 0.f);
        if (sdf < R.margin) {
            code = 1;
            if (out > 0.f) {
                nl0 = copysignf(o0 / out, p0);
                nl1 = copysignf(o1 / out, p1);
                nl2 = copysignf(o2 / out, p2);
                // copysignf(0, negative) gives -0: harmless
            } else if (q0 >= q1 && q0 >= q2) nl0 = p0 >= 0.f ? 1.f : -1.f;
            else if (q1 >= q2) nl1 = p1 >= 0.f ? 1.f : -1.f;
            else nl2 = p2 >= 0.f ? 1.f : -1.f;
        }
    } else if (R.type == MPM_QUAD_SLICER &&
               fabsf(p2) < (fmaxf(0.5f * R.thickness, R.spine_radius) + R.margin) * 1.000001f + 1e-30f) {
        // (beyond that distance from the blade plane neither the spine nor the faces
        // can hold the node: both distances are at least |p2|)
        const float A = R.half[0], Bh = R.half[1];
        const float es = fmaxf(fabsf(p0) - A, 0.f), et = p1 + Bh;
        const float dsp = sqrtf(es * es + et * et + p2 * p2);
        if (dsp < R.spine_radius + R.margin) {
            code = 3;
        } else {
            const float qs = fminf(fmaxf(p0, -A), A), qt = fminf(fmaxf(p1, -Bh), Bh);
            const float d0 = p0 - qs, d1 = p1 - qt, d2 = p2;
            const float l = sqrtf(d0 * d0 + d1 * d1 + d2 * d2);
            if (l < 0.5f * R.thickness + R.margin) {
                code = 1;
                if (fabsf(p0) <= A && fabsf(p1) <= Bh) nl2 = p2 >= 0.f ? 1.f : -1.f;
                else { nl0 = d0 / l; nl1 = d1 / l; nl2 = d2 / l; }
            }
        }
    } else if (EXT && R.type == MPM_ARC) {
        // nearest point of the arc (radius half[0], angles half[1] .. half[1] + half[2])
        const float Ra = R.half[0], th0 = R.half[1], sw = R.half[2];
        const float kTwoPi = 6.28318530717958647f;
        float th = th0;
        if (p0 != 0.f || p1 != 0.f) {
            float rel = fmodf(atan2f(p1, p0) - th0, kTwoPi);
            if (rel < 0.f) rel += kTwoPi;
            if (rel <= sw) {
                th = th0 + rel;
            } else {
                float s0, c0, s1, c1;
                sincosf(th0, &s0, &c0);
                sincosf(th0 + sw, &s1, &c1);
                const float a0 = p0 - Ra * c0, a1 = p1 - Ra * s0, b0 = p0 - Ra * c1, b1 = p1 - Ra * s1;
                th = (b0 * b0 + b1 * b1 < a0 * a0 + a1 * a1) ? th0 + sw : th0;
            }
        }
        float sn, cs;
        sincosf(th, &sn, &cs);
        const float d0 = p0 - Ra * cs, d1 = p1 - Ra * sn, d2 = p2;
        const float l = sqrtf(d0 * d0 + d1 * d1 + d2 * d2);
        if (l < R.radius + R.margin) {
            code = 2;
            if (l > 0.f) { nl0 = d0 / l; nl1 = d1 / l; nl2 = d2 / l; }
            tl0 = -sn;
            tl1 = cs;
        }
    } else if (EXT && R.type == MPM_MESH_SLICER && near) {
        float nl[3] = {0.f, 0.f, 0.f};
        code = mesh_slicer_region(R, p0, p1, p2, nl);
        nl0 = nl[0]; nl1 = nl[1]; nl2 = nl[2];
    } else if (R.type == MPM_SEGMENTS && near) {
        float best = 3.4e38f, bq0 = 0.f, bq1 = 0.f, bq2 = 0.f;
        int bs = -1;
        for (int s = 0; s + 1 < R.n_pts; ++s) {
            const float a0 = R.shape.pts[3 * s], a1 = R.shape.pts[3 * s + 1], a2 = R.shape.pts[3 * s + 2];
            const float e0 = R.shape.pts[3 * s + 3] - a0, e1 = R.shape.pts[3 * s + 4] - a1, e2 = R.shape.pts[3 * s + 5] - a2;
            const float L2 = e0 * e0 + e1 * e1 + e2 * e2;
            float u = L2 > 0.f ? ((p0 - a0) * e0 + (p1 - a1) * e1 + (p2 - a2) * e2) / L2 : 0.f;
            u = fminf(fmaxf(u, 0.f), 1.f);
            const float c0 = a0 + u * e0, c1 = a1 + u * e1, c2 = a2 + u * e2;
            const float d0 = p0 - c0, d1 = p1 - c1, d2 = p2 - c2;
            const float l = sqrtf(d0 * d0 + d1 * d1 + d2 * d2);
            if (l < best) { best = l; bq0 = c0; bq1 = c1; bq2 = c2; bs = s; }
        }
        if (bs >= 0 && best < R.radius + R.margin) {
            code = 2;
            if (best > 0.f) { nl0 = (p0 - bq0) / best; nl1 = (p1 - bq1) / best; nl2 = (p2 - bq2) / best; }
            const float e0 = R.shape.pts[3 * bs + 3] - R.shape.pts[3 * bs], e1 = R.shape.pts[3 * bs + 4] - R.shape.pts[3 * bs + 1],
                        e2 = R.shape.pts[3 * bs + 5] - R.shape.pts[3 * bs + 2];
            const float L = sqrtf(e0 * e0 + e1 * e1 + e2 * e2);
            if (L > 0.f) { tl0 = e0 / L; tl1 = e1 / L; tl2 = e2 / L; }
        }
    }
    n = f3(P.R[0] * nl0 + P.R[1] * nl1 + P.R[2] * nl2, P.R[3] * nl0 + P.R[4] * nl1 + P.R[5] * nl2,
           P.R[6] * nl0 + P.R[7] * nl1 + P.R[8] * nl2);
    t = f3(P.R[0] * tl0 + P.R[1] * tl1 + P.R[2] * tl2, P.R[3] * tl0 + P.R[4] * tl1 + P.R[5] * tl2,
           P.R[6] * tl0 + P.R[7] * tl1 + P.R[8] * tl2);
    return code;
}

// Contact correction (Sec. IV-A..C): sticky -> v_rel' = 0; otherwise keep a
// separating node (v_n >= 0), else v_rel' = c_d max(1 - mu_k |v_n| / |v_t|, 0) v_t
// with v_t the tangential part (regular) or the part along the 1D tangent.
// Returns whether the node was changed; dp = node momentum change.
template <bool EXT>
__device__ bool rigid_contact(const RigidDev& R, const RigidPose& P, float3 x, float m, float3& v, float3& dp)
{
    float3 n, t;
    const int code = rigid_region<EXT>(R, P, x, n, t);
    if (code == 0) return false;
    const float r0 = x.x - P.c[0], r1 = x.y - P.c[1], r2 = x.z - P.c[2];
    const float vr0 = R.vel[0] + R.omega[1] * r2 - R.omega[2] * r1;
    const float vr1 = R.vel[1] + R.omega[2] * r0 - R.omega[0] * r2;
    const float vr2 = R.vel[2] + R.omega[0] * r1 - R.omega[1] * r0;
    const float e0 = v.x - vr0, e1 = v.y - vr1, e2 = v.z - vr2;
    float n0 = 0.f, n1 = 0.f, n2 = 0.f;
    if (code != 3) {
        const bool has_n = (n.x * n.x + n.y * n.y + n.z * n.z) > 0.f;
        float vn = e0 * n.x + e1 * n.y + e2 * n.z;
        if (has_n && vn >= 0.f) return false;
        if (!has_n) vn = 0.f;
        float t0, t1, t2;
        if (code == 1) {
            t0 = e0 - vn * n.x; t1 = e1 - vn * n.y; t2 = e2 - vn * n.z;
        } else {
            const float a = e0 * t.x + e1 * t.y + e2 * t.z;
            t0 = a * t.x; t1 = a * t.y; t2 = a * t.z;
        }
        const float lt = sqrtf(t0 * t0 + t1 * t1 + t2 * t2);
        float scale = 0.f;
        if (lt > 0.f) scale = R.c_d * fmaxf(1.f - R.mu_k * fabsf(vn) / lt, 0.f);
        n0 = scale * t0; n1 = scale * t1; n2 = scale * t2;
    }
    dp = f3(m * (n0 - e0), m * (n1 - e1), m * (n2 - e2));
    v = f3(vr0 + n0, vr1 + n1, vr2 + n2);
    return true;
}

constexpr int kGridThreads = 256;  // 4 node bricks per iteration

// Grid update of node nid of node brick B (Eq. 3, contact, walls) against the scene's nr
// rigids, at the poses that the scan left; each warp adds its momentum to the rigids'
// impulses.  64 threads per brick, one node each.
// The node's P2G accumulator is reset later: loading and clearing the freshly reduced lines
// in one kernel measured far slower.
template <bool EXT>
__device__ __forceinline__ void grid_node(const StepArgs& a, int B, int scene, int nid, int lane, const RigidDev* rig,
                                          const RigidPose* pose, int nr)
{
    const SceneDev sc = a.scenes[scene];
    const int n = sc.n, lb = B - sc.brick_base;
    int bx, by, bz;
    brick_coords(sc.nb, sc.nb_log2, lb, bx, by, bz);
    const int gi = bx * 4 + (nid >> 4);
    const int gj = by * 4 + ((nid >> 2) & 3);
    const int gk = bz * 4 + (nid & 3);
    const int node = B * 64 + nid;
    const float4 g = a.G[node];
    float3 v = f3(0.f, 0.f, 0.f);
    const float dxs = 1.0f / (float)n;
    float dpr[kMaxRigids][3];
    unsigned touched = 0;
    if (g.x > 0.f) {
        v = f3(g.y / g.x + a.dt * a.gravity[0], g.z / g.x + a.dt * a.gravity[1], g.w / g.x + a.dt * a.gravity[2]);
        const float3 xI = f3(gi * dxs, gj * dxs, gk * dxs);
        for (int r = 0; r < nr; ++r) {
            float3 dp;
            if (rigid_contact<EXT>(rig[r], pose[r], xI, g.x, v, dp)) {
                touched |= 1u << r;
                dpr[r][0] = dp.x; dpr[r][1] = dp.y; dpr[r][2] = dp.z;
            }
        }
        const int lo = a.bound, hi = n - 1 - a.bound;
        if (gi < lo) v.x = fmaxf(v.x, 0.f);
        if (gi > hi) v.x = fminf(v.x, 0.f);
        if (gj < lo) {
            if (a.floor_sticky) v = f3(0.f, 0.f, 0.f);
            else v.y = fmaxf(v.y, 0.f);
        }
        if (gj > hi) v.y = fminf(v.y, 0.f);
        if (gk < lo) v.z = fmaxf(v.z, 0.f);
        if (gk > hi) v.z = fminf(v.z, 0.f);
    }
    a.V[node] = make_float4(v.x, v.y, v.z, g.x);
    a.sb.ccnt[node] = 0;
    if (nid == 0) {
        a.brick_epoch[B] = a.epoch[scene];
        // the histograms of the next substep start from zero (the sort has
        // read them; every non-empty brick is an active node brick)
        a.sb.cnt[B] = 0;
    }
    // impulse on each rigid: -(node momentum change), linear and angular
    for (int r = 0; r < nr; ++r) {
        const bool on = (touched >> r) & 1u;
        if (!__any_sync(kFull, on)) continue;
        float val[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (on) {
            const float d0 = -dpr[r][0], d1 = -dpr[r][1], d2 = -dpr[r][2];
            const float r0 = gi * dxs - pose[r].c[0], r1 = gj * dxs - pose[r].c[1], r2 = gk * dxs - pose[r].c[2];
            val[0] = d0; val[1] = d1; val[2] = d2;
            val[3] = r1 * d2 - r2 * d1;
            val[4] = r2 * d0 - r0 * d2;
            val[5] = r0 * d1 - r1 * d0;
        }
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            float x = val[c];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
            if (lane == 0 && x != 0.f) atomicAdd(&a.impulse[(scene * kMaxRigids + r) * 6 + c], (double)x);
        }
    }
}

// Grid update of a launch whose scenes have no rigid: no staging and no impulse
// sums, so a budget of 32 registers holds twice the resident CTAs of k_grid and
// the node bricks of a 1M-particle block are taken in one round.
__global__ void __launch_bounds__(kGridThreads, 8) k_grid_plain(StepArgs a)
{
    chain_wait();
    const int tid = threadIdx.x, lane = tid & 31, grp = tid >> 6, nid = tid & 63;
    const int n_nact = a.sb.counters[CTR_N_NACT];
    for (int base = blockIdx.x * 4; base < n_nact; base += gridDim.x * 4) {
        const int item = base + grp;
        if (item < n_nact)
            grid_node<false>(a, a.sb.nact_brick[item], a.sb.nact_scene[item], nid, lane, nullptr, nullptr, 0);
    }
}

// Reset of the P2G accumulator of the active node bricks once the grid update has
// read it, where no G2P follows that does it (the fused G2P + P2G, the reverse
// substeps).  Loading and clearing the lines that P2G's reductions just wrote in
// one kernel measured far slower than two kernels: 13.4 against 11.5 us per
// substep for the 1M block without rigids, 0.138 against 0.047 ms for the 256
// batched scenes with their blades.
__global__ void __launch_bounds__(kGridThreads, 8) k_grid_clear(StepArgs a)
{
    chain_wait();
    const int grp = threadIdx.x >> 6, nid = threadIdx.x & 63;
    const int n_nact = a.sb.counters[CTR_N_NACT];
    for (int base = blockIdx.x * 4; base < n_nact; base += gridDim.x * 4) {
        const int item = base + grp;
        if (item < n_nact) {
            const int B = a.sb.nact_brick[item];
            a.G[B * 64 + nid] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
}

// One scene's rigids are staged in shared memory (a thread's segments are walked over and
// over: slab_256k 53.4 us a substep staged, 54.8 not).  Those of many scenes are read
// where they are, by uniform loads that stay in L1: staged scene by scene, with a table of
// the CTA's bricks and barriers at each change - bricks come interleaved by scan tile - a
// substep of 256 scenes with their blades took 377 us, so 352.
template <bool EXT>
__global__ void __launch_bounds__(kGridThreads, 4) k_grid(StepArgs a)
{
    __shared__ RigidDev s_rig[kMaxRigids];
    __shared__ RigidPose s_pose[kMaxRigids];
    chain_wait();
    const int tid = threadIdx.x, lane = tid & 31, grp = tid >> 6, nid = tid & 63;
    const int n_nact = a.sb.counters[CTR_N_NACT];
    if (a.r.s1 - a.r.s0 == 1) {
        const int nr = a.scenes[a.r.s0].n_rigid;
        static_assert(sizeof(RigidDev) % sizeof(int) == 0 && sizeof(RigidPose) % sizeof(int) == 0, "copied in words");
        const int* rig = reinterpret_cast<const int*>(a.rigids + a.r.s0 * kMaxRigids);
        const int* pose = reinterpret_cast<const int*>(a.pose + a.r.s0 * kMaxRigids);
        for (int t = tid; t < nr * (int)(sizeof(RigidDev) / sizeof(int)); t += kGridThreads) reinterpret_cast<int*>(s_rig)[t] = rig[t];
        for (int t = tid; t < nr * (int)(sizeof(RigidPose) / sizeof(int)); t += kGridThreads)
            reinterpret_cast<int*>(s_pose)[t] = pose[t];
        __syncthreads();
        for (int base = blockIdx.x * 4; base < n_nact; base += gridDim.x * 4) {
            const int item = base + grp;
            if (item < n_nact) grid_node<EXT>(a, a.sb.nact_brick[item], a.r.s0, nid, lane, s_rig, s_pose, nr);
        }
        return;
    }
    for (int base = blockIdx.x * 4; base < n_nact; base += gridDim.x * 4) {
        const int item = base + grp;
        if (item >= n_nact) continue;
        const int scene = a.sb.nact_scene[item];
        grid_node<EXT>(a, a.sb.nact_brick[item], scene, nid, lane, a.rigids + scene * kMaxRigids, a.pose + scene * kMaxRigids,
                       a.scenes[scene].n_rigid);
    }
}

// ------------------------------------------------------------------ G2P
//
// One thread per sorted slot (Eq. 4, Eq. 9, Eq. 10, then the constitutive update,
// the last step of the G2P loop in Algorithm 1).

// Result of one particle: the caller stores it (store_particle).
struct G2POut {
    float x[3], v[3], C[9], F[9], t6[6];
    int id;
};

// G2P of a particle with position (and id) q0 from its stencil's velocities; the
// new position before the push-out.  stencil(bc) returns the node functor of base
// cell bc, old_F(F) reads the deformation gradient, early(x, C) takes the new
// x and C before the constitutive update (C stored there leaves it eight registers more).
template <int FLAGS, class Stencil, class OldF, class Early>
__device__ __forceinline__ unsigned g2p_particle(const StepArgs& a, const SceneDev& sc, const float4 q0, float mu, float lam,
                                                 Stencil stencil, OldF old_F, Early early, G2POut& o)
{
    const int n = sc.n;
    const float fn = (float)n, dt = a.dt;
    unsigned ebits = 0;
    int bc[3];
    float f[3], w[9], B[9];
    particle_weights(q0.x, q0.y, q0.z, n, bc, f, w);
    o.id = __float_as_int(q0.w);
    gather_velocity<FLAGS>(f, w, stencil(bc), o.v, B);
    // C = D^-1 sum N v (x_I - x_p)^T = 4/dx^2 * dx * B  (Eq. 9), or for the
    // standard MPM L = n B with the derivative weights (Eq. 5); x += dt v (Eq. 4)
    const float c4 = (FLAGS & kG2PStdGrad) ? fn : 4.0f * fn;
#pragma unroll
    for (int i = 0; i < 9; ++i) o.C[i] = B[i] * c4;
    o.x[0] = q0.x + dt * o.v[0];
    o.x[1] = q0.y + dt * o.v[1];
    o.x[2] = q0.z + dt * o.v[2];
    // F <- (I + dt C) F  (Eq. 10)
    float F[9];
    old_F(F);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float F0 = F[c], F1 = F[3 + c], F2 = F[6 + c];
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const float Fr = r == 0 ? F0 : (r == 1 ? F1 : F2);
            o.F[3 * r + c] = Fr + dt * (o.C[3 * r] * F0 + o.C[3 * r + 1] * F1 + o.C[3 * r + 2] * F2);
        }
    }
    early(o.x, o.C);
    float chk = q0.x + q0.y + q0.z + o.v[0] + o.v[1] + o.v[2];
    if (!(FLAGS & kG2PNoStress)) {
        ebits |= constitutive(a.model, a.plasticity, a.yield_stress, mu, lam, o.F, o.t6);
    } else {
#pragma unroll
        for (int i = 0; i < 6; ++i) o.t6[i] = 0.f;
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) chk += o.F[i];
    if (!isfinite(chk)) ebits |= MPM_EBIT_NONFINITE;
    return ebits;
}

// Planes 4 and 5 (C but its last component) of slot s.
__device__ __forceinline__ void store_C(const StepArgs& a, int s, const float C[9])
{
    const size_t cap = a.cap;
    float4* q = a.out.q + s;
    q[4 * cap] = make_float4(C[0], C[1], C[2], C[3]);
    q[5 * cap] = make_float4(C[4], C[5], C[6], C[7]);
}

// The other planes of slot s, and the material.
__device__ __forceinline__ void store_particle(const StepArgs& a, int pp_mat, float mu, float lam, int s, const G2POut& o)
{
    const size_t cap = a.cap;
    float4* q = a.out.q + s;
    q[0] = make_float4(o.x[0], o.x[1], o.x[2], __int_as_float(o.id));
    q[cap] = make_float4(o.F[0], o.F[1], o.F[2], o.F[3]);
    q[2 * cap] = make_float4(o.F[4], o.F[5], o.F[6], o.F[7]);
    q[3 * cap] = make_float4(o.F[8], o.v[0], o.v[1], o.v[2]);
    q[6 * cap] = make_float4(o.C[8], o.t6[0], o.t6[1], o.t6[2]);
    q[7 * cap] = make_float4(o.t6[3], o.t6[4], o.t6[5], 0.f);
    if (pp_mat) {
        a.out.mu[s] = mu;
        a.out.lam[s] = lam;
    }
}

__device__ __forceinline__ void material_of(const StepArgs& a, const SceneDev& sc, int p, float& mu, float& lam)
{
    mu = sc.mu;
    lam = sc.lam;
    if (sc.pp_mat) {
        mu = a.in.mu[p];
        lam = a.in.lam[p];
    }
}

// Copy the 6^3 window out of the 2x2x2 staged bricks into a linear array, so
// that the 27 nodes of a particle sit at constant offsets.
template <int BLOCK>
__device__ __forceinline__ void linearize_window(const float4* vw, float4* lin)
{
    for (int t = threadIdx.x; t < kWinNodes; t += BLOCK) {
        const int wi = t / 36, wj = (t / 6) % 6, wk = t % 6;
        lin[t] = vw[(((wi >> 2) << 2) | ((wj >> 2) << 1) | (wk >> 2)) * 64 + (wi & 3) * 16 + (wj & 3) * 4 + (wk & 3)];
    }
}

// Persistent CTAs, their warps taking chunks of 32 slots in turn (the chunks in
// flight then cover one window of the arrays, and neighbouring warps the same nodes).
// What bounds it is the chain permutation -> planes -> nodes -> rank of each
// particle: planes 0-3 of a warp's next chunk are copied to shared memory while it
// computes, its slots of the permutation are read two chunks ahead, and the rank's
// atomic is sent before the constitutive update.  Read through
// L1, the stencils need no staging, no barriers and no brick: one CTA per brick with
// its window copied to shared memory (46.1 M warp instructions at 62 % issue, the SMs
// idle for a sixth of the launch behind its last bricks) took 70.8 us on a 1M block
// and 18.8 us on a 64k one; this kernel 59.8 us and 9.5 us, the accumulator's reset
// (1.8 us in a kernel of its own) included.  Spills cost more than warps in flight bring:
// a substep of the 1M block takes 126.6 us with 80 registers (32 B spilled), 146.4 with
// 72 (144 B), 128.4 with 96.
// MINB = CTAs per SM the registers must allow: the larger budget (6 at 128
// threads, 3 at 256: 80 registers; 1 at 512: 128) or 1024/BLOCK (64 registers,
// more warps in flight).  FLAGS & kG2PSolids: some scene of the launch has a
// sphere or a box, so particles may need the push-out.
template <int BLOCK, int MINB, int FLAGS>
__global__ void __launch_bounds__(BLOCK, MINB) k_g2p(StepArgs a)
{
    chain_wait();
    constexpr bool SOLIDS = (FLAGS & kG2PSolids) != 0;
    constexpr int NW = BLOCK / 32;
    __shared__ float4 s_q[4][BLOCK];  // planes 0-3 of each thread's next particle
    __shared__ SolidPose s_pose[SOLIDS ? NW : 1][SOLIDS ? kMaxRigids : 1];  // a scene's rigids at the end of the substep
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // the accumulator of the active node bricks: the grid update has read it
    const int n_clear = a.sb.counters[CTR_N_NACT] * 64;
    for (int t = blockIdx.x * BLOCK + tid; t < n_clear; t += gridDim.x * BLOCK)
        a.G[a.sb.nact_brick[t >> 6] * 64 + (t & 63)] = make_float4(0.f, 0.f, 0.f, 0.f);
    // (no particle brick: the sort found its bookkeeping inconsistent)
    const int c1 = active_bricks(a.sb) ? (a.r.np + 31) >> 5 : 0;
    const int step = gridDim.x * NW;
    int c = blockIdx.x * NW + warp;
    const int p_end = a.r.p0 + a.r.np;
    const size_t cap = a.cap;
    // (the lanes beyond the last slot repeat it and store nothing)
    const auto slot_source = [&](int ch) { return ch < c1 ? a.sb.perm[min(a.r.p0 + ch * 32 + lane, p_end - 1)] : -1; };
    const auto copy_planes = [&](int p) {
        if (p >= 0) {
#pragma unroll
            for (int k = 0; k < 4; ++k) cp_async16(&s_q[k][tid], a.in.q + k * cap + p);
        }
        cp_async_commit();
    };
    int p = slot_source(c), p_next = slot_source(c + step);
    copy_planes(p);
    int posed = -1;
    for (; c < c1; c += step) {
        const int p_after = slot_source(c + 2 * step);
        const bool valid = a.r.p0 + c * 32 + lane < p_end;
        const int s = min(a.r.p0 + c * 32 + lane, p_end - 1);
        const int scene = scene_of_slot(a, s);
        const SceneDev& sc = a.scenes[scene];
        G2POut o;
        unsigned ood = 0;
        CellRank rank;
        float mu, lam;
        material_of(a, sc, p, mu, lam);
        cp_async_wait<0>();
        // new key and the atomics of the rank, whose answer is not needed before the end
        const auto sort_key = [&](const float* x) {
            const int key = cell_key(sc, x[0], x[1], x[2], ood);
            rank = cell_rank_begin(a.sb, sc, key, valid);
            if (valid) a.sb.key[s] = key;
        };
        unsigned ebits = g2p_particle<FLAGS>(
            a, sc, s_q[0][tid], mu, lam, [&](const int* bc) { return GridStencil<(FLAGS & kG2PReadOnly) != 0>(a.V, sc, bc); },
            [&](float* F) {
                const float4 u = s_q[1][tid], v = s_q[2][tid];
                F[0] = u.x; F[1] = u.y; F[2] = u.z; F[3] = u.w;
                F[4] = v.x; F[5] = v.y; F[6] = v.z; F[7] = v.w;
                F[8] = s_q[3][tid].x;
                copy_planes(p_next);
            },
            [&](const float* x, const float* C) {
                if (valid) store_C(a, s, C);
                if (!SOLIDS) sort_key(x);
            },
            o);
        __syncwarp();
        if (SOLIDS) {
            // push-out (Sec. IV-A), scene by scene of the chunk
            const int sc1 = __shfl_sync(kFull, scene, 31);
            for (int q = __shfl_sync(kFull, scene, 0); q <= sc1; ++q) {
                const int nr = a.scenes[q].n_rigid;
                if (nr == 0) continue;
                if (q != posed) stage_solids(a, q, s_pose[warp], lane);
                posed = q;
                __syncwarp();
                if (scene == q) push_out(s_pose[warp], nr, o.x);
                __syncwarp();
            }
            sort_key(o.x);
        }
        const int r = cell_rank_end(rank);
        if (valid) {
            store_particle(a, sc.pp_mat, mu, lam, s, o);
            a.sb.rank[s] = r;
            if (ood && !(ebits & MPM_EBIT_NONFINITE)) ebits |= MPM_EBIT_OUT_OF_DOMAIN;
            if (ebits) atomicOr(&a.err[scene], ebits);
        }
        p = p_next;
        p_next = p_after;
    }
    cp_async_wait<0>();
    // every read of the clocks of this CTA lies before the barrier
    walker_exit(a);
}

// ------------------------------------------------------- fused G2P + P2G
//
// G2P of substep k fused with P2G of substep k+1: each particle is read and
// written once per substep, and its new stress goes from registers straight
// into the next P2G.  The CTA of a brick scatters into an 8^3-node window
// around the brick (base cells may have moved by up to one cell): particles
// whose new base cell is still inside the brick use the per-cell register
// accumulation of k_p2g; the few that crossed a brick face use shared atomics
// into the window; any that moved farther use global atomics.

constexpr int kFusedThreads = 192;  // 64 cells x 3 slices
constexpr int kW8 = 8, kW8Nodes = kW8 * kW8 * kW8;

__global__ void __launch_bounds__(kFusedThreads, 4) k_g2p2g(StepArgs a)
{
    __shared__ __align__(128) float4 vw[2][8 * 64];
    __shared__ __align__(16) float4 lin[kWinNodes];
    __shared__ float rec[kRecFields][kFusedThreads];
    __shared__ float win[4][kW8Nodes];
    __shared__ short order[kFusedThreads];
    __shared__ int cell_cnt[64], cell_off[65];
    __shared__ __align__(8) unsigned long long bar[2];
    __shared__ int s_item[2];
    __shared__ SolidPose s_pose[kMaxRigids];  // the scene's rigids at the end of the substep
    __shared__ int s_pose_scene;
    const int tid = threadIdx.x;
    const int cell = tid & 63, slice = tid >> 6;
    const int cx = cell >> 4, cy = (cell >> 2) & 3, cz = cell & 3;
    const int n_act = active_bricks(a.sb);
    int* work = &a.sb.counters[CTR_WORK_G2P];
    if (tid == 0) s_pose_scene = -1;
    walker_init<kFusedThreads>(a, n_act, vw, bar, s_item, work);
    unsigned phase[2] = {0u, 0u};
    int buf = 0;
    for (;;) {
        const int item = s_item[buf];
        if (item >= n_act) break;
        for (int t = tid; t < 4 * kW8Nodes; t += kFusedThreads) (&win[0][0])[t] = 0.0f;
        if (tid < 64) cell_cnt[tid] = 0;
        if (!walker_next(a, n_act, vw, bar, s_item, work, buf, phase, item)) break;
        const int e = active_entry(a.sb, item);
        const int start = a.sb.act_start[e], count = a.sb.act_count[e], scene = a.sb.act_scene[e];
        const SceneDev sc = a.scenes[scene];
        const int n_solid = a.any_solid ? sc.n_rigid : 0;
        if (n_solid && scene != s_pose_scene) stage_solids(a, scene, s_pose, tid);
        const int n = sc.n, nb = sc.nb, lb = a.sb.act_brick[e] - sc.brick_base;
        int ox, oy, oz;
        brick_coords(nb, sc.nb_log2, lb, ox, oy, oz);
        ox *= 4; oy *= 4; oz *= 4;
        const float fn = (float)n, dxs = 1.0f / fn;
        const float m = sc.m_p;
        const float kA = a.dt * sc.V0 * 4.0f * fn * fn;
        linearize_window<kFusedThreads>(vw[buf], lin);
        __syncthreads();
        if (tid == 0 && n_solid) s_pose_scene = scene;
        unsigned ebits = 0;
        for (int k0 = 0; k0 < count; k0 += kFusedThreads) {
            const int k = k0 + tid;
            const bool valid = k < count;
            int key = 0, my_cell = -1, my_rank = 0;
            if (valid) {
                G2POut o;
                const int p = a.sb.perm[start + k];
                float mu, lam;
                material_of(a, sc, p, mu, lam);
                ebits |= g2p_particle<0>(
                    a, sc, plane(a.in, a.cap, 0, p), mu, lam,
                    [&](const int* bc) {
                        const int l0 = min(max(bc[0] - ox, 0), 3), l1 = min(max(bc[1] - oy, 0), 3),
                                  l2 = min(max(bc[2] - oz, 0), 3);
                        const float4* base = lin + (l0 * 36 + l1 * 6 + l2);
                        return [base](int i, int j, int kk) { return base[i * 36 + j * 6 + kk]; };
                    },
                    [&](float* F) { load_F(a.in, a.cap, p, F); }, [&](const float*, const float* C) { store_C(a, start + k, C); }, o);
                if (n_solid) push_out(s_pose, n_solid, o.x);
                store_particle(a, sc.pp_mat, mu, lam, start + k, o);
                // P2G of the next substep at the new position
                int bc[3];
                float f[3], w[9];
                const unsigned ood = particle_weights(o.x[0], o.x[1], o.x[2], n, bc, f, w);
                if (ood && !(ebits & MPM_EBIT_NONFINITE)) ebits |= ood;
                key = (sc.brick_base + ((bc[0] >> 2) * nb + (bc[1] >> 2)) * nb + (bc[2] >> 2)) * 64 +
                      ((bc[0] & 3) * 16 + (bc[1] & 3) * 4 + (bc[2] & 3));
                float q3[3], Ad[9];
                p2g_coeffs(m, kA, dxs, o.v, o.C, o.t6, f, q3, Ad);
                const int l0 = bc[0] - ox, l1 = bc[1] - oy, l2 = bc[2] - oz;
                if ((unsigned)l0 < 4u && (unsigned)l1 < 4u && (unsigned)l2 < 4u) {
                    put_record<kFusedThreads>(rec, tid, w, q3, Ad);
                    my_cell = (l0 * 4 + l1) * 4 + l2;
                    my_rank = atomicAdd(&cell_cnt[my_cell], 1);
                } else if (l0 >= -1 && l0 <= 4 && l1 >= -1 && l1 <= 4 && l2 >= -1 && l2 <= 4) {
                    // crossed a brick face: scatter into the window with shared atomics
#pragma unroll
                    for (int i = 0; i < 3; ++i)
#pragma unroll
                        for (int j = 0; j < 3; ++j)
#pragma unroll
                            for (int k2 = 0; k2 < 3; ++k2) {
                                const float W = w[i] * w[3 + j] * w[6 + k2];
                                const int node = ((l0 + 1 + i) * kW8 + (l1 + 1 + j)) * kW8 + (l2 + 1 + k2);
                                atomicAdd(&win[0][node], W * m);
                                atomicAdd(&win[1][node], W * (q3[0] + Ad[0] * i + Ad[1] * j + Ad[2] * k2));
                                atomicAdd(&win[2][node], W * (q3[1] + Ad[3] * i + Ad[4] * j + Ad[5] * k2));
                                atomicAdd(&win[3][node], W * (q3[2] + Ad[6] * i + Ad[7] * j + Ad[8] * k2));
                            }
                } else {
                    // moved more than a cell: straight to HBM
#pragma unroll
                    for (int i = 0; i < 3; ++i)
#pragma unroll
                        for (int j = 0; j < 3; ++j)
#pragma unroll
                            for (int k2 = 0; k2 < 3; ++k2) {
                                const float W = w[i] * w[3 + j] * w[6 + k2];
                                red_add_v4(&a.G[node_index(sc, bc[0] + i, bc[1] + j, bc[2] + k2)], W * m,
                                           W * (q3[0] + Ad[0] * i + Ad[1] * j + Ad[2] * k2),
                                           W * (q3[1] + Ad[3] * i + Ad[4] * j + Ad[5] * k2),
                                           W * (q3[2] + Ad[6] * i + Ad[7] * j + Ad[8] * k2));
                            }
                }
            }
            const int rank = cell_rank_end(cell_rank_begin(a.sb, sc, key, valid));
            if (valid) {
                a.sb.key[start + k] = key;
                a.sb.rank[start + k] = rank;
            }
            __syncthreads();
            scan_cells(cell_cnt, cell_off, tid);
            __syncthreads();
            if (my_cell >= 0) order[cell_off[my_cell] + my_rank] = (short)tid;
            __syncthreads();
            float acc_w[9], acc_p[9][3];
#pragma unroll
            for (int q = 0; q < 9; ++q) { acc_w[q] = 0.f; acc_p[q][0] = acc_p[q][1] = acc_p[q][2] = 0.f; }
            cell_accumulate<kFusedThreads>(rec, order, cell_off[cell], cell_off[cell + 1], slice, acc_w, acc_p);
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                if (acc_w[q] != 0.f) {
                    const int node = ((cx + 1 + slice) * kW8 + (cy + 1 + q / 3)) * kW8 + (cz + 1 + q % 3);
                    atomicAdd(&win[0][node], acc_w[q] * m);
                    atomicAdd(&win[1][node], acc_p[q][0]);
                    atomicAdd(&win[2][node], acc_p[q][1]);
                    atomicAdd(&win[3][node], acc_p[q][2]);
                }
            }
            __syncthreads();
            if (tid < 64) cell_cnt[tid] = 0;
            __syncthreads();
        }
        // window -> HBM (node (ox-1, oy-1, oz-1) + (wi, wj, wk))
        for (int t = tid; t < kW8Nodes; t += kFusedThreads) {
            const float mm = win[0][t];
            if (mm == 0.0f) continue;
            const int gi = ox - 1 + t / (kW8 * kW8), gj = oy - 1 + (t / kW8) % kW8, gk = oz - 1 + t % kW8;
            if (gi < 0 || gj < 0 || gk < 0 || gi >= n || gj >= n || gk >= n) continue;
            red_add_v4(&a.G[node_index(sc, gi, gj, gk)], mm, win[1][t], win[2][t], win[3][t]);
        }
        if (ebits) atomicOr(&a.err[scene], ebits);
        __syncthreads();
        buf ^= 1;
    }
    walker_exit(a);
}

// ---------------------------------------------------- PB-MPM cycle G2P
//
// G2P of a PB-MPM cycle (Sec. III-C): positions and F stay fixed during the
// cycles, so each particle's v = sum W v_I and APIC C = 4/dx^2 sum W v_I
// (x_I - x_p)^T are written back in place (storage order), where the next
// cycle's P2G reads them through the same permutation.  It also resets the
// accumulator for that P2G.

constexpr int kVcThreads = 128;

template <bool READ_ONLY>
__global__ void __launch_bounds__(kVcThreads) k_g2p_vc(StepArgs a)
{
    chain_wait();
    const int g = blockIdx.x * kVcThreads + threadIdx.x;
    const int n_clear = a.sb.counters[CTR_N_NACT] * 64;
    for (int t = g; t < n_clear; t += gridDim.x * kVcThreads)
        a.G[a.sb.nact_brick[t >> 6] * 64 + (t & 63)] = make_float4(0.f, 0.f, 0.f, 0.f);
    const int s = a.r.p0 + min(g, a.r.np - 1);
    const SceneDev sc = a.scenes[scene_of_slot(a, s)];
    if (g >= a.r.np || active_bricks(a.sb) == 0) return;
    const size_t cap = a.cap;
    const int p = a.sb.perm[s];
    float x[3], f[3], w[9], v[3], B[9];
    int bc[3];
    load_x(a.in, p, x);
    particle_weights(x[0], x[1], x[2], sc.n, bc, f, w);
    gather_velocity<0>(f, w, GridStencil<READ_ONLY>(a.V, sc, bc), v, B);
    const float c4 = 4.0f * (float)sc.n;
#pragma unroll
    for (int i = 0; i < 9; ++i) B[i] *= c4;
    float4* q = a.in.q + p;
    const float F8 = state_at(a.in, cap, kAtF + 8, p);
    q[3 * cap] = make_float4(F8, v[0], v[1], v[2]);
    q[4 * cap] = make_float4(B[0], B[1], B[2], B[3]);
    q[5 * cap] = make_float4(B[4], B[5], B[6], B[7]);
    state_at(a.in, cap, kAtC + 8, p) = B[8];
}

// ------------------------------------------------------- state I/O kernels
//
// x, v, C and F of one scene as arrays in particle-id order (null: not moved), all
// fields in one pass over the planes; a slot whose id is not of the scene (a substep that
// a device error cut short wrote none) is left out.  Particle ids are in no order by slot, so one side
// is scattered over HBM, and the sectors it half uses are the cost: one kernel a field
// took 105 us to write 1M particles' state and 255 us to read it, now 75 and 117 us;
// writing through records in id order instead, 177 us.

// particle ids by slot
__global__ void k_order(PState st, int p0, int np, int* dst)
{
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g < np) dst[g] = state_id(st, p0 + g);
}

// Inverse of a scene's slot -> id map: inv[id] = slot.
__global__ void k_id_inverse(PState st, int p0, int np, int* inv)
{
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= np) return;
    const int id = state_id(st, p0 + g);
    if ((unsigned)id < (unsigned)np) inv[id] = p0 + g;
}

constexpr int kIoBlock = 128;
constexpr int kIoFloats = 24;  // x, v, C, F

// The inverse, and the fields of each slot as one record of 96 contiguous bytes: reading
// records in id order then fetches whole sectors, where the planes' 16-byte words would
// use half of each.
__global__ void __launch_bounds__(kIoBlock) k_pack(PState st, int cap_, int p0, int np, int* inv, float4* rec)
{
    __shared__ float4 buf[kIoBlock * (kIoFloats / 4)];
    const int t = threadIdx.x, g0 = blockIdx.x * kIoBlock, cnt = min(kIoBlock, np - g0);
    const size_t cap = cap_;
    if (t < cnt) {
        const float4* q = st.q + (p0 + g0 + t);
        const float4 a = q[0], b = q[cap], c = q[2 * cap], d = q[3 * cap], e = q[4 * cap], f = q[5 * cap];
        const float C8 = q[6 * cap].x;
        const int id = __float_as_int(a.w);
        if ((unsigned)id < (unsigned)np) inv[id] = p0 + g0 + t;
        float4* r = buf + t * (kIoFloats / 4);
        r[0] = make_float4(a.x, a.y, a.z, d.y);
        r[1] = make_float4(d.z, d.w, e.x, e.y);
        r[2] = make_float4(e.z, e.w, f.x, f.y);
        r[3] = make_float4(f.z, f.w, C8, b.x);
        r[4] = make_float4(b.y, b.z, b.w, c.x);
        r[5] = make_float4(c.y, c.z, c.w, d.x);
    }
    __syncthreads();
    for (int i = t; i < cnt * (kIoFloats / 4); i += kIoBlock) rec[(size_t)(p0 + g0) * (kIoFloats / 4) + i] = buf[i];
}

// Planes of slot s to the fields' entries (px, pv: 3 floats, pC, pF: 9; null: not wanted).
__device__ __forceinline__ void planes_to_fields(const PState& st, size_t cap, int s, float4 q0, float* px, float* pv, float* pC,
                                                 float* pF)
{
    const float4* q = st.q + s;
    const auto put4 = [](float* d, float4 a) { d[0] = a.x; d[1] = a.y; d[2] = a.z; d[3] = a.w; };
    if (px) { px[0] = q0.x; px[1] = q0.y; px[2] = q0.z; }
    if (pv || pF) {
        const float4 a = q[3 * cap];
        if (pv) { pv[0] = a.y; pv[1] = a.z; pv[2] = a.w; }
        if (pF) pF[8] = a.x;
    }
    if (pF) {
        const float4 a = q[cap], b = q[2 * cap];
        put4(pF, a);
        put4(pF + 4, b);
    }
    if (pC) {
        const float4 a = q[4 * cap], b = q[5 * cap];
        pC[8] = q[6 * cap].x;
        put4(pC, a);
        put4(pC + 4, b);
    }
}

// The other way.  Plane 6 also holds the stress, which a write makes void.
__device__ __forceinline__ void fields_to_planes(const PState& st, size_t cap, int s, int id, const float* px, const float* pv,
                                                 const float* pC, const float* pF)
{
    float4* q = st.q + s;
    const auto get4 = [](const float* d) { return make_float4(d[0], d[1], d[2], d[3]); };
    if (px) q[0] = make_float4(px[0], px[1], px[2], __int_as_float(id));
    if (pv || pF) {
        float4 a = pv && pF ? make_float4(0.f, 0.f, 0.f, 0.f) : q[3 * cap];
        if (pv) { a.y = pv[0]; a.z = pv[1]; a.w = pv[2]; }
        if (pF) a.x = pF[8];
        q[3 * cap] = a;
    }
    if (pF) {
        q[cap] = get4(pF);
        q[2 * cap] = get4(pF + 4);
    }
    if (pC) {
        q[4 * cap] = get4(pC);
        q[5 * cap] = get4(pC + 4);
        q[6 * cap] = make_float4(pC[8], 0.f, 0.f, 0.f);
    }
}

// One lane per slot at the planes, in order.  Reading the state, the warp stores the entries
// of its particles, wherever their ids say, with neighbouring lanes at neighbouring floats (a
// lane a particle, 64k particles took 33 us, now 26).  Writing it, each lane loads its own
// particle's (with the loads in the order of the floats 1M particles took 128 us, so 75).
__global__ void __launch_bounds__(kIoBlock) k_arrays_by_slot(PState st, int cap, int p0, int np, Fields h)
{
    __shared__ float buf[kIoBlock / 32][kIoFloats * 32];
    const int lane = threadIdx.x & 31;
    float* const mine = buf[threadIdx.x >> 5];
    const int g = blockIdx.x * kIoBlock + threadIdx.x, cnt = min(32, np - g + lane);
    const bool own = lane < cnt;
    const int s = p0 + g;
    const float4 q0 = own ? st.q[s] : make_float4(0.f, 0.f, 0.f, 0.f);
    const int id = __float_as_int(q0.w);
    float* const first[4] = {mine, mine + 3 * 32, mine + 6 * 32, mine + 15 * 32};
    const auto entry = [&](int f) { return h.f[f] ? first[f] + lane * (f < 2 ? 3 : 9) : nullptr; };
    if (own) planes_to_fields(st, cap, s, q0, entry(0), entry(1), entry(2), entry(3));
    __syncwarp();
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        if (!h.f[f]) continue;
        const int k = f < 2 ? 3 : 9;
#pragma unroll
        for (int i = 0; i < k; ++i) {
            const int at = i * 32 + lane, particle = at / k, to = __shfl_sync(kFull, id, particle);
            if (particle < cnt && (unsigned)to < (unsigned)np) h.f[f][(size_t)to * k + (at - particle * k)] = first[f][at];
        }
    }
}

__global__ void __launch_bounds__(kIoBlock) k_state_by_slot(PState st, int cap, int p0, int np, Fields h)
{
    const int g = blockIdx.x * kIoBlock + threadIdx.x;
    if (g >= np) return;
    const int s = p0 + g, id = state_id(st, s);
    if ((unsigned)id >= (unsigned)np) return;
    const size_t i = id;
    fields_to_planes(st, cap, s, id, h.f[0] ? h.f[0] + 3 * i : nullptr, h.f[1] ? h.f[1] + 3 * i : nullptr,
                     h.f[2] ? h.f[2] + 9 * i : nullptr, h.f[3] ? h.f[3] + 9 * i : nullptr);
}

// A CTA per kIoBlock consecutive ids: the arrays move as whole 16-byte words of one
// contiguous chunk each (they may be pinned host memory, over the host link), through
// shared memory; the particles' side, planes or records, is the scattered one.  (Pinned
// arrays are read and written from the planes: with records x of 4M particles took 429 us
// to read, so 311, and all fields 2,247, so 2,151.)
template <bool OUT, bool RECORDS>
__global__ void __launch_bounds__(kIoBlock) k_fields_by_id(PState st, int cap, int p0, int np, const int* __restrict__ inv,
                                                           const float4* rec, Fields h)
{
    __shared__ __align__(16) float buf[kIoFloats * kIoBlock];
    const int t = threadIdx.x;
    const int g0 = blockIdx.x * kIoBlock;
    const int cnt = min(kIoBlock, np - g0);
    // the slot of id g0 + t (ids are a permutation of the scene's slots)
    const int s = t < cnt ? inv[g0 + t] : p0;
    const bool own = t < cnt && (unsigned)(s - p0) < (unsigned)np;
    float* const first[4] = {buf, buf + 3 * kIoBlock, buf + 6 * kIoBlock, buf + 15 * kIoBlock};
    const auto entry = [&](int f) { return h.f[f] ? first[f] + t * (f < 2 ? 3 : 9) : nullptr; };
    if (OUT && !RECORDS) {
        if (own)
            planes_to_fields(st, cap, s, h.f[0] ? st.q[s] : make_float4(0.f, 0.f, 0.f, 0.f), entry(0), entry(1), entry(2), entry(3));
        __syncthreads();
    }
    if (OUT && RECORDS) {
        if (own) {
            float r[kIoFloats];
#pragma unroll
            for (int k = 0; k < kIoFloats / 4; ++k) {
                const float4 a = rec[(size_t)s * (kIoFloats / 4) + k];
                r[4 * k] = a.x; r[4 * k + 1] = a.y; r[4 * k + 2] = a.z; r[4 * k + 3] = a.w;
            }
#pragma unroll
            for (int f = 0, at = 0; f < 4; at += f < 2 ? 3 : 9, ++f)
#pragma unroll
                for (int c = 0; c < (f < 2 ? 3 : 9); ++c) first[f][t * (f < 2 ? 3 : 9) + c] = r[at + c];
        }
        __syncthreads();
    }
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        if (!h.f[f]) continue;
        const int k = f < 2 ? 3 : 9;
        float *chunk = h.f[f] + (size_t)g0 * k, *b = first[f];
        float *src = OUT ? b : chunk, *dst = OUT ? chunk : b;
        if (cnt == kIoBlock && (reinterpret_cast<uintptr_t>(chunk) & 15u) == 0) {
            for (int i = t; i < k * kIoBlock / 4; i += kIoBlock)
                reinterpret_cast<float4*>(dst)[i] = reinterpret_cast<const float4*>(src)[i];
        } else {
            for (int i = t; i < cnt * k; i += kIoBlock) dst[i] = src[i];
        }
    }
    if (!OUT) {
        __syncthreads();
        if (own) fields_to_planes(st, cap, s, g0 + t, entry(0), entry(1), entry(2), entry(3));
    }
}

__global__ void k_set_rigid(RigidDev d, RigidDev* dst)
{
    static_assert(sizeof(RigidDev) % sizeof(int) == 0, "copied in words");
    for (int i = threadIdx.x; i < (int)(sizeof(RigidDev) / sizeof(int)); i += blockDim.x)
        reinterpret_cast<int*>(dst)[i] = reinterpret_cast<const int*>(&d)[i];
}

__global__ void k_init_particles(PState st, int cap, int p_at, int n, int id0, const float* x, const float* v,
                                 const float* E, const float* nu, float E0, float nu0)
{
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= n) return;
    const int s = p_at + g;
    for (int d = 0; d < 3; ++d) {
        state_at(st, cap, kAtX + d, s) = x[3 * (size_t)g + d];
        state_at(st, cap, kAtV + d, s) = v ? v[3 * (size_t)g + d] : 0.f;
    }
    for (int i = 0; i < 9; ++i) {
        state_at(st, cap, kAtC + i, s) = 0.f;
        state_at(st, cap, kAtF + i, s) = (i % 4 == 0) ? 1.f : 0.f;
    }
    const float e = E ? E[g] : E0, q = nu ? nu[g] : nu0;
    st.mu[s] = e / (2.f * (1.f + q));
    st.lam[s] = e * q / ((1.f + q) * (1.f - 2.f * q));
    state_id(st, s) = id0 + g;
}

__global__ void k_read_grid(const float4* V, const int* brick_epoch, const int* epoch, int scene, int n,
                            int brick_base, float* dst)
{
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long total = (long long)n * n * n;
    if (g >= total) return;
    const int nb = n / 4;
    const int brick = (int)(g >> 6), loc = (int)(g & 63);
    const int B = brick_base + brick;
    if (brick_epoch[B] != epoch[scene] - 1) return;
    const int bx = brick / (nb * nb), by = (brick / nb) % nb, bz = brick % nb;
    const int gi = bx * 4 + (loc >> 4), gj = by * 4 + ((loc >> 2) & 3), gk = bz * 4 + (loc & 3);
    const float4 v = V[(size_t)B * 64 + loc];
    float* o = dst + (((size_t)gi * n + gj) * n + gk) * 4;
    o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
}

// ------------------------------------------------------------- launchers

static int n_blocks(long long n, int t) { return (int)((n + t - 1) / t); }

cudaError_t launch_prepare(const StepArgs& a, const PState& st, cudaStream_t s)
{
    if (a.r.np == 0) return cudaSuccess;
    launch_chain(a.r.np, k_prepare, n_blocks(a.r.np, 256), 256, 0, s, a, st);
    return cudaGetLastError();
}

cudaError_t launch_reset_histogram(const SortBufs& sb, int bricks, int tiles, int np, cudaStream_t s)
{
    launch_chain(np, k_reset_histogram, n_blocks(max(bricks, 32), 256), 256, 0, s, sb, bricks, tiles);
    return cudaGetLastError();
}

cudaError_t launch_scan(const StepArgs& a, cudaStream_t s)
{
    launch_chain(a.r.np, k_scan, a.r.nt, kScanThreads, 0, s, a);
    return cudaGetLastError();
}

cudaError_t launch_sort(const StepArgs& a, cudaStream_t s)
{
    cudaError_t e = launch_scan(a, s);
    if (e != cudaSuccess) return e;
    launch_chain(a.r.np, k_scatter, n_blocks(max(a.r.np, a.r.nt), 256 * kScatterPer), 256, 0, s, a);
    return cudaGetLastError();
}

cudaError_t prepare_kernels()
{
    const int most = kP2GWarps * p2g_warp_bytes(kP2GMaxSlots);
    cudaError_t e = cudaFuncSetAttribute(k_p2g<kP2GStress>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_p2g<kP2GConstraint>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_p2g<kP2GStd>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    // G2P of large launches keeps to the shared memory it needs: the rest is L1, which holds
    // the nodes (4M block 461 -> 449 us a substep, 256 scenes 382 -> 376)
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_g2p<128, 6, kG2PReadOnly>, cudaFuncAttributePreferredSharedMemoryCarveout, 25);
    return e;
}

cudaError_t launch_p2g(const StepArgs& a, cudaStream_t s)
{
    const int c = min(a.p2g_ctas, n_blocks(max(a.r.np, 1), kP2GWarps * a.p2g_slots));
    const size_t smem = kP2GWarps * p2g_warp_bytes(a.p2g_slots);
    if (a.solver == MPM_SOLVER_PB) launch_chain(a.r.np, k_p2g<kP2GConstraint>, c, kP2GThreads, smem, s, a);
    else if (a.solver == MPM_SOLVER_STANDARD) launch_chain(a.r.np, k_p2g<kP2GStd>, c, kP2GThreads, smem, s, a);
    else launch_chain(a.r.np, k_p2g<kP2GStress>, c, kP2GThreads, smem, s, a);
    return cudaGetLastError();
}

cudaError_t launch_g2p_vc(const StepArgs& a, cudaStream_t s)
{
    if (a.r.np == 0) return cudaSuccess;
    const int c = n_blocks(a.r.np, kVcThreads);
    if (a.r.np < kChainBelow) launch_chain(a.r.np, k_g2p_vc<false>, c, kVcThreads, 0, s, a);
    else launch_alone(k_g2p_vc<true>, c, kVcThreads, 0, s, a);
    return cudaGetLastError();
}

cudaError_t launch_grid(const StepArgs& a, cudaStream_t s, bool clear)
{
    if (!a.any_rigid) launch_chain(a.r.np, k_grid_plain, a.grid_plain_ctas, kGridThreads, 0, s, a);
    else if (a.rigid_ext) launch_chain(a.r.np, k_grid<true>, a.grid_ctas, kGridThreads, 0, s, a);
    else launch_chain(a.r.np, k_grid<false>, a.grid_ctas, kGridThreads, 0, s, a);
    if (clear) launch_chain(a.r.np, k_grid_clear, a.grid_plain_ctas, kGridThreads, 0, s, a);
    return cudaGetLastError();
}

// Only the shapes that small launches take by default exist with ordinary loads too, for
// programmatic launches (GridStencil).
template <int FLAGS>
static void launch_g2p_variant(const StepArgs& a, cudaStream_t s)
{
    const int c = min(a.g2p_ctas, n_blocks(max(a.r.np, 1), a.g2p_threads));
    constexpr int RO = FLAGS | kG2PReadOnly;
    if (a.g2p_regs64) {
        switch (a.g2p_threads) {
        case 128: launch_alone(k_g2p<128, 8, RO>, c, 128, 0, s, a); break;
        case 512: launch_alone(k_g2p<512, 2, RO>, c, 512, 0, s, a); break;
        default: launch_alone(k_g2p<256, 4, RO>, c, 256, 0, s, a); break;
        }
    } else {
        switch (a.g2p_threads) {
        case 128: launch_alone(k_g2p<128, 6, RO>, c, 128, 0, s, a); break;
        case 512: launch_alone(k_g2p<512, 1, RO>, c, 512, 0, s, a); break;
        default:
            if (a.r.np < kChainBelow) launch_chain(a.r.np, k_g2p<256, 3, FLAGS>, c, 256, 0, s, a);
            else launch_alone(k_g2p<256, 3, RO>, c, 256, 0, s, a);
            break;
        }
    }
}

// The one shape of the standard-MPM and PB-MPM variants.
template <int FLAGS>
static void launch_g2p_128(const StepArgs& a, cudaStream_t s)
{
    const int c = min(a.g2p_ctas, n_blocks(max(a.r.np, 1), 128));
    if (a.r.np < kChainBelow) launch_chain(a.r.np, k_g2p<128, 6, FLAGS>, c, 128, 0, s, a);
    else launch_alone(k_g2p<128, 6, FLAGS | kG2PReadOnly>, c, 128, 0, s, a);
}

// The standard-MPM and PB-MPM variants exist in one launch shape only (128
// threads, 80 registers): the MLS-MPM shapes are what the tuner explores.
cudaError_t launch_g2p(const StepArgs& a, cudaStream_t s)
{
    // the push-out variant only where a scene has a solid shape: blades, needles and
    // segments push nothing out
    if (a.solver == MPM_SOLVER_STANDARD) {
        if (a.any_solid) launch_g2p_128<kG2PStdGrad | kG2PSolids>(a, s);
        else launch_g2p_128<kG2PStdGrad>(a, s);
    } else if (a.solver == MPM_SOLVER_PB) {
        if (a.any_solid) launch_g2p_128<kG2PNoStress | kG2PSolids>(a, s);
        else launch_g2p_128<kG2PNoStress>(a, s);
    } else if (a.any_solid) {
        launch_g2p_variant<kG2PSolids>(a, s);
    } else {
        launch_g2p_variant<0>(a, s);
    }
    return cudaGetLastError();
}

cudaError_t launch_g2p2g(const StepArgs& a, cudaStream_t s)
{
    k_g2p2g<<<a.fused_ctas, kFusedThreads, 0, s>>>(a);
    return cudaGetLastError();
}

int occupancy_grid()
{
    int b = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_grid<true>, kGridThreads, 0);
    return b;
}

int occupancy_grid_plain()
{
    int b = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_grid_plain, kGridThreads, 0);
    return b;
}

int occupancy_g2p2g()
{
    int b = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_g2p2g, kFusedThreads, 0);
    return b;
}

cudaError_t launch_order(const PState& st, int p0, int np, int* dst, cudaStream_t s)
{
    if (np == 0) return cudaSuccess;
    k_order<<<n_blocks(np, 256), 256, 0, s>>>(st, p0, np, dst);
    return cudaGetLastError();
}

cudaError_t launch_fields(const PState& st, const PState& spare, int cap, int p0, int np, int* inv, const Fields& h, bool out,
                          bool host, cudaStream_t s)
{
    if (np == 0) return cudaSuccess;
    // the records (whole sectors) leave plane 0 alone: a substep that a device error skipped
    // leaves the spare buffer unwritten and current, and its ids are indexes
    float4* rec = spare.q + (((size_t)cap + 1) & ~(size_t)1);
    int fields = 0;
    size_t bytes = 0;
    for (int f = 0; f < 4; ++f)
        if (h.f[f]) {
            ++fields;
            bytes += (size_t)np * sizeof(float) * (f < 2 ? 3 : 9);
        }
    if (out && host) {
        k_id_inverse<<<n_blocks(np, 256), 256, 0, s>>>(st, p0, np, inv);
        k_fields_by_id<true, false><<<n_blocks(np, kIoBlock), kIoBlock, 0, s>>>(st, cap, p0, np, inv, rec, h);
    } else if (out && fields >= 3 && bytes >= kIoRecordsFrom) {
        k_pack<<<n_blocks(np, kIoBlock), kIoBlock, 0, s>>>(st, cap, p0, np, inv, rec);
        k_fields_by_id<true, true><<<n_blocks(np, kIoBlock), kIoBlock, 0, s>>>(st, cap, p0, np, inv, rec, h);
    } else if (out) {
        k_arrays_by_slot<<<n_blocks(np, kIoBlock), kIoBlock, 0, s>>>(st, cap, p0, np, h);
    } else if (host) {
        k_id_inverse<<<n_blocks(np, 256), 256, 0, s>>>(st, p0, np, inv);
        k_fields_by_id<false, false><<<n_blocks(np, kIoBlock), kIoBlock, 0, s>>>(st, cap, p0, np, inv, rec, h);
    } else {
        k_state_by_slot<<<n_blocks(np, kIoBlock), kIoBlock, 0, s>>>(st, cap, p0, np, h);
    }
    return cudaGetLastError();
}

cudaError_t launch_set_rigid(const RigidDev& d, RigidDev* dst, cudaStream_t s)
{
    k_set_rigid<<<1, 128, 0, s>>>(d, dst);
    return cudaGetLastError();
}

cudaError_t launch_init_particles(const PState& st, int cap, int p_at, int n, int id0, const float* x, const float* v,
                                  const float* E, const float* nu, float E0, float nu0, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    k_init_particles<<<n_blocks(n, 256), 256, 0, s>>>(st, cap, p_at, n, id0, x, v, E, nu, E0, nu0);
    return cudaGetLastError();
}

cudaError_t launch_read_grid(const float4* V, const int* brick_epoch, const int* epoch, const SceneDev*, int scene,
                             int n, int brick_base, float* dst, cudaStream_t s)
{
    const long long total = (long long)n * n * n;
    k_read_grid<<<n_blocks(total, 256), 256, 0, s>>>(V, brick_epoch, epoch, scene, n, brick_base, dst);
    return cudaGetLastError();
}

int occupancy_p2g(int slots)
{
    int b = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_p2g<kP2GStress>, kP2GThreads, kP2GWarps * p2g_warp_bytes(slots));
    return b;
}

int occupancy_g2p(int threads, int regs64)
{
    // the variant with the push-out uses the same registers and a little more
    // shared memory; its occupancy bounds both
    int b = 0;
    if (regs64) {
        if (threads == 128) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_g2p<128, 8, kG2PSolids | kG2PReadOnly>, 128, 0);
        else if (threads == 512) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_g2p<512, 2, kG2PSolids | kG2PReadOnly>, 512, 0);
        else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_g2p<256, 4, kG2PSolids | kG2PReadOnly>, 256, 0);
    } else {
        if (threads == 128) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_g2p<128, 6, kG2PSolids | kG2PReadOnly>, 128, 0);
        else if (threads == 512) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_g2p<512, 1, kG2PSolids | kG2PReadOnly>, 512, 0);
        else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_g2p<256, 3, kG2PSolids | kG2PReadOnly>, 256, 0);
    }
    return b;
}

}  // namespace mpm
