// Device helpers shared by the forward and adjoint transfer kernels: PTX
// wrappers (mbarrier, bulk-copy TMA, vector reductions), brick keys and ranks,
// B-spline weights, P2G coefficients, per-cell accumulation, halo staging.
#pragma once

#include "mpm_kernels.cuh"

namespace mpm {

// ------------------------------------------------------------ PTX helpers

__device__ __forceinline__ unsigned smem_u32(const void* p)
{
    return static_cast<unsigned>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void red_add_v4(float4* addr, float a, float b, float c, float d)
{
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(addr), "f"(a), "f"(b), "f"(c), "f"(d)
                 : "memory");
}

__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_mbar_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void fence_proxy_async()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(unsigned long long* bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, unsigned bytes, unsigned long long* bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(unsigned long long* bar, unsigned parity)
{
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait on an mbarrier phase; false when the bound ran out.
__device__ __forceinline__ bool mbar_wait_bounded(unsigned long long* bar, unsigned parity)
{
    for (int it = 0; it < (1 << 22); ++it)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

// Small launches of the substep chain are made programmatic: a kernel's CTAs come up
// while the one before it still runs, and wait here for its end and its writes (every
// thread, before its first access); the next kernel may come up at once.  Elsewhere both
// do nothing.
__device__ __forceinline__ void chain_wait()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <class... P, class... A>
void launch_chain(int np, void (*k)(P...), int ctas, int threads, size_t smem, cudaStream_t s, A... args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute programmatic;
    programmatic.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    programmatic.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &programmatic;
    cfg.numAttrs = np < kChainBelow ? 1 : 0;
    cudaLaunchKernelEx(&cfg, k, args...);
}

// A launch that is never programmatic: the kernel comes up when the one before it has ended.
template <class... P, class... A>
void launch_alone(void (*k)(P...), int ctas, int threads, size_t smem, cudaStream_t s, A... args)
{
    k<<<ctas, threads, smem, s>>>(args...);
}

constexpr unsigned kFull = 0xffffffffu;

// ----------------------------------------------------- brick key + rank

// Sort key of a particle: its brick (global index) x 64 + its base cell inside
// the brick, which is the index of its stencil's first node.
__device__ __forceinline__ int cell_key(const SceneDev& sc, float x0, float x1, float x2, unsigned& ood)
{
    int c0, c1, c2;
    ood |= (unsigned)(base_cell(x0, sc.n, c0) | base_cell(x1, sc.n, c1) | base_cell(x2, sc.n, c2));
    const int brick = sc.brick_base + ((c0 >> 2) * sc.nb + (c1 >> 2)) * sc.nb + (c2 >> 2);
    return brick * 64 + ((c0 & 3) * 16 + (c1 & 3) * 4 + (c2 & 3));
}

// Rank of a particle within its cell, which also counts the cell's, the brick's and
// the scan tile's particles for the next substep's sort: runs of lanes with the same
// cell take consecutive ranks from one atomic (all 32 lanes call it; `valid` marks
// lanes with a particle).  Particles come in the cell order of a substep ago, so a
// warp holds a handful of runs.  key is the particle's cell_key.  add_tile = false
// leaves the tile's count to the caller (which then aggregates it itself).
// In two parts: the atomic's answer is not waited for before the second.
struct CellRank {
    int base, first;  // the run's first rank (at its first lane), the run's first lane
};

__device__ __forceinline__ CellRank cell_rank_begin(const SortBufs& sb, const SceneDev& sc, int key, bool valid,
                                                    bool add_tile = true)
{
    const int lane = threadIdx.x & 31;
    if (!valid) key = -64;
    const int prev = __shfl_up_sync(kFull, key, 1);
    const bool head = lane == 0 || prev != key, bhead = lane == 0 || (prev >> 6) != (key >> 6);
    const unsigned heads = __ballot_sync(kFull, head), bheads = __ballot_sync(kFull, bhead);
    const unsigned upto = 0xffffffffu >> (31 - lane);  // this lane and the ones before it
    const auto run = [&](unsigned h) { return ((h & ~upto) ? __ffs(h & ~upto) - 1 : 32) - lane; };
    CellRank r{0, 31 - __clz(heads & upto)};
    if (valid && head) r.base = atomicAdd(&sb.ccnt[key], run(heads));
    if (valid && bhead) {
        const int brick = key >> 6, np = run(bheads);
        atomicAdd(&sb.cnt[brick], np);
        if (add_tile) atomicAdd(&sb.tile_n[sc.tile_base + ((brick - sc.brick_base) >> sb.tile_shift)], np);
    }
    return r;
}

__device__ __forceinline__ int cell_rank_end(const CellRank& r)
{
    return __shfl_sync(kFull, r.base, r.first) + (int)(threadIdx.x & 31) - r.first;
}

// The active particle bricks: those of at least kBigBrick particles fill the list
// from its front, the others from its back.
__device__ __forceinline__ int active_bricks(const SortBufs& sb) { return sb.counters[CTR_N_BIG] + sb.counters[CTR_N_SMALL]; }

__device__ __forceinline__ int active_entry(const SortBufs& sb, int item)
{
    const int n_big = sb.counters[CTR_N_BIG];
    return item < n_big ? item : sb.list_size - 1 - (item - n_big);
}

// ------------------------------------------------------ transfer helpers

constexpr int kRecFields = 21;  // w0[3] w1[3] w2[3] q[3] Ad[9]

// Base cells, fractional offsets and quadratic B-spline weights of a position.
__device__ __forceinline__ unsigned particle_weights(float x0, float x1, float x2, int n, int b[3], float f[3],
                                                     float w[9])
{
    const float fn = (float)n;
    const unsigned ood = base_cell(x0, n, b[0]) | base_cell(x1, n, b[1]) | base_cell(x2, n, b[2]);
    f[0] = __fmaf_rn(x0, fn, -(float)b[0]);
    f[1] = __fmaf_rn(x1, fn, -(float)b[1]);
    f[2] = __fmaf_rn(x2, fn, -(float)b[2]);
    bspline(f[0], w);
    bspline(f[1], w + 3);
    bspline(f[2], w + 6);
    return ood ? MPM_EBIT_OUT_OF_DOMAIN : 0u;
}

// P2G coefficients (Eq. 8 with the APIC particle momentum, M^-1 = 4/dx^2 of
// Eq. 7, V sigma = V0 tau): the momentum a particle gives node (i,j,k) of its
// stencil is W_ijk (q + Ad (i,j,k)) with Ad = (m C - dt V0 M^-1 tau) dx and
// q = m v - Ad f, so that Ad ((i,j,k) - f) = A (x_I - x_p).
__device__ __forceinline__ void p2g_coeffs(float m, float kA, float dxs, const float v[3], const float C[9],
                                           const float t6[6], const float f[3], float q[3], float Ad[9])
{
    const float tau[9] = {t6[0], t6[1], t6[2], t6[1], t6[3], t6[4], t6[2], t6[4], t6[5]};
#pragma unroll
    for (int i = 0; i < 9; ++i) Ad[i] = (m * C[i] - kA * tau[i]) * dxs;
#pragma unroll
    for (int r = 0; r < 3; ++r) q[r] = m * v[r] - (Ad[3 * r] * f[0] + Ad[3 * r + 1] * f[1] + Ad[3 * r + 2] * f[2]);
}

template <int N>
__device__ __forceinline__ void put_record(float (*rec)[N], int k, const float w[9], const float q[3], const float Ad[9])
{
#pragma unroll
    for (int i = 0; i < 9; ++i) rec[i][k] = w[i];
#pragma unroll
    for (int i = 0; i < 3; ++i) rec[9 + i][k] = q[i];
#pragma unroll
    for (int i = 0; i < 9; ++i) rec[12 + i][k] = Ad[i];
}

// Phase B of the per-cell accumulation: thread (cell, slice) adds the
// contributions of the particles of its cell (order[beg..end)) to the 9 nodes
// cell + (slice, j, k) in registers.
template <int N>
__device__ __forceinline__ void cell_accumulate(const float (*rec)[N], const short* order, int beg, int end, int slice,
                                                float acc_w[9], float acc_p[9][3])
{
    const float si = (float)slice;
    for (int j = beg; j < end; ++j) {
        const int k = order[j];
        const float wi = rec[slice][k];
        const float wy[3] = {rec[3][k], rec[4][k], rec[5][k]};
        const float wz[3] = {rec[6][k], rec[7][k], rec[8][k]};
        // r(j,k) = q + Ad (slice, j, k)
        const float r0 = rec[9][k] + si * rec[12][k], r1 = rec[10][k] + si * rec[15][k], r2 = rec[11][k] + si * rec[18][k];
        const float a01 = rec[13][k], a11 = rec[16][k], a21 = rec[19][k];
        const float a02 = rec[14][k], a12 = rec[17][k], a22 = rec[20][k];
#pragma unroll
        for (int jj = 0; jj < 3; ++jj) {
            const float wij = wi * wy[jj];
            const float s0 = r0 + a01 * jj, s1 = r1 + a11 * jj, s2 = r2 + a21 * jj;
#pragma unroll
            for (int kk = 0; kk < 3; ++kk) {
                const float W = wij * wz[kk];
                const int q = jj * 3 + kk;
                acc_w[q] += W;
                acc_p[q][0] += W * (s0 + a02 * kk);
                acc_p[q][1] += W * (s1 + a12 * kk);
                acc_p[q][2] += W * (s2 + a22 * kk);
            }
        }
    }
}

// Exclusive scan of the 64 per-cell counts by warp 0.
__device__ __forceinline__ void scan_cells(const int* cell_cnt, int* cell_off, int tid)
{
    if (tid < 32) {
        const int c_a = cell_cnt[2 * tid], c_b = cell_cnt[2 * tid + 1];
        int incl = c_a + c_b;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int t = __shfl_up_sync(kFull, incl, d);
            if (tid >= d) incl += t;
        }
        const int excl = incl - c_a - c_b;
        cell_off[2 * tid] = excl;
        cell_off[2 * tid + 1] = excl + c_a;
        if (tid == 31) cell_off[64] = incl;
    }
}

// Scene of slot s (scenes own consecutive slots): two warp-wide probes of the
// scenes' first slots for the warp's first slot, then the few lanes of later scenes
// step on.  Every lane of the warp calls it.
__device__ __forceinline__ int scene_of_slot(const StepArgs& a, int s)
{
    if (a.r.s1 - a.r.s0 == 1) return a.r.s0;
    const int lane = threadIdx.x & 31, s_first = __shfl_sync(kFull, s, 0);
    int lo = a.r.s0, len = a.r.s1 - a.r.s0;
    while (len > 1) {  // p_begin never decreases: the last scene that starts at or before s_first
        const int step = (len + 31) >> 5, at = lane * step;
        const bool le = at < len && a.scenes[lo + at].p_begin <= s_first;
        const int k = 31 - __clz(__ballot_sync(kFull, le) | 1u);
        lo += k * step;
        len = min(step, len - k * step);
    }
    while (lo + 1 < a.r.s1 && a.scenes[lo + 1].p_begin <= s) ++lo;
    return lo;
}

__device__ __forceinline__ void cp_async16(float4* dst, const float4* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }

template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

constexpr int kRecPitch = 20;  // floats per record: an odd number of 16-byte words

// MODE: kP2GStress (MLS-MPM: the Kirchhoff stress, stored by G2P or computed
// from F), kP2GConstraint (PB-MPM: the co-rotational constraint replaces C
// and there is no stress term) or kP2GStd (standard MPM, Sec. III-A: W m v and the
// internal-force impulse -dt V0 tau grad W, Eq. 2, 3).  kP2GAdj: the reverse of G2P
// adds three values and no mass.
enum { kP2GStress = 0, kP2GConstraint = 1, kP2GStd = 2, kP2GAdj = 3 };

// Adds a record's contributions to the nodes (i, j, k) of plane i: (p_x, p_y) in
// acc_a[3 j + k], (p_z, weight) in acc_b.
template <int MODE>
__device__ __forceinline__ void p2g_add(const float4* rec, int i, float2 acc_a[9], float2 acc_b[9])
{
    const auto two = [](float s) { return make_float2(s, s); };
    const float4 r0 = rec[0], r1 = rec[1], r2 = rec[2], r3 = rec[3], r4 = rec[4];
    const float wy[3] = {r0.y, r0.z, r0.w}, wz[3] = {r1.x, r1.y, r1.z};
    // w_i(f) = alpha + beta (f - gamma)^2
    const float gam = i == 0 ? 1.5f : (i == 1 ? 1.0f : 0.5f), bet = i == 1 ? -1.0f : 0.5f, alp = i == 1 ? 0.75f : 0.0f;
    const float e = r0.x - gam, wi = __fmaf_rn(bet * e, e, alp);
    if (MODE == kP2GStd) {
        // p = (wx m v - dwx T_x) wy wz - wx (T_y dwy wz + T_z wy dwz)
        const float dwx = 2.f * bet * e;
        const float mv[3] = {r2.x, r2.y, r2.z}, T[9] = {r3.x, r3.y, r3.z, r3.y, r3.w, r4.x, r3.z, r4.x, r4.y};
        float dy[3], dz[3];
        bspline_d(r2.w, dy);
        bspline_d(r4.z, dz);
        float A[3], B[3], C[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            A[c] = wi * mv[c] - dwx * T[3 * c];
            B[c] = wi * T[3 * c + 1];
            C[c] = wi * T[3 * c + 2];
        }
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            float P[3], Q[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                P[c] = wy[j] * A[c] - dy[j] * B[c];
                Q[c] = -wy[j] * C[c];
            }
            const float W = wi * wy[j];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const int q = 3 * j + k;
                acc_a[q] = __ffma2_rn(make_float2(P[0], P[1]), two(wz[k]), acc_a[q]);
                acc_a[q] = __ffma2_rn(make_float2(Q[0], Q[1]), two(dz[k]), acc_a[q]);
                acc_b[q] = __ffma2_rn(make_float2(P[2], W), two(wz[k]), acc_b[q]);
                acc_b[q].x = __fmaf_rn(Q[2], dz[k], acc_b[q].x);
            }
        }
        return;
    }
    const float si = (float)(i - 1);
    const float2 a1 = make_float2(r3.x, r3.y), a2 = make_float2(r3.z, r3.w);
    const float2 v01 = __ffma2_rn(two(si), make_float2(r2.z, r2.w), make_float2(r2.x, r2.y));
    const float v2 = __fmaf_rn(si, r4.y, r4.x);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const float wij = wi * wy[j], fj = (float)(j - 1);
        const float2 s01 = j == 1 ? v01 : __ffma2_rn(two(fj), a1, v01);
        const float s2 = j == 1 ? v2 : __fmaf_rn(fj, r4.z, v2);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float W = wij * wz[k], fk = (float)(k - 1);
            const int q = 3 * j + k;
            const float2 u01 = k == 1 ? s01 : __ffma2_rn(two(fk), a2, s01);
            const float2 u2w = make_float2(k == 1 ? s2 : __fmaf_rn(fk, r4.w, s2), 1.0f);
            acc_a[q] = __ffma2_rn(two(W), u01, acc_a[q]);
            acc_b[q] = __ffma2_rn(two(W), u2w, acc_b[q]);
        }
    }
}

// Phases B and C of P2G: the records' contributions to the nodes, summed by run (of
// records of one base cell; run r starts at s_start[r]) and node plane i, joined where
// runs are neighbours in z, and added to G.  Called by a whole warp.
template <int MODE>
__device__ __forceinline__ void scatter_runs(const StepArgs& a, const float4* rec, const int* s_scene, const short* s_start,
                                             int runs)
{
    const int lane = threadIdx.x & 31;
    for (int job0 = 0; job0 < 3 * runs; job0 += 32) {
        const int job = job0 + lane, run = min(job / 3, runs - 1), i = job - (job / 3) * 3, beg = s_start[run];
        const bool own = job < 3 * runs;
        const int end = own ? s_start[run + 1] : beg;
        float2 acc_a[9], acc_b[9];
#pragma unroll
        for (int q = 0; q < 9; ++q) acc_a[q] = acc_b[q] = make_float2(0.f, 0.f);
        for (int q = beg; q < end; ++q) p2g_add<MODE>(rec + q * (kRecPitch / 4), i, acc_a, acc_b);
        __syncwarp();
        const int key = __float_as_int(rec[beg * (kRecPitch / 4) + 1].w);
        const int ly = (key >> 2) & 3, lz = key & 3;
        // C: three lanes on lies the next run; where its cell is the next one in z
        // (of the brick), its nodes 0 and 1 are this run's 1 and 2
        const int before = __shfl_up_sync(kFull, key, 3);
        const bool joined = own && lane >= 3 && lz > 0 && before == key - 1;
        const bool last = !(__shfl_down_sync(kFull, joined, 3) && lane < 29);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const auto join = [&](float v0, float& v1, float v2) {
                const float c2 = __shfl_up_sync(kFull, v2, 3);
                if (joined) v1 += c2;
                const float c1 = __shfl_up_sync(kFull, v1, 3);
                return joined ? v0 + c1 : v0;
            };
            float2 *p = acc_a + 3 * j, *q = acc_b + 3 * j;
            p[0].x = join(p[0].x, p[1].x, p[2].x);
            p[0].y = join(p[0].y, p[1].y, p[2].y);
            q[0].x = join(q[0].x, q[1].x, q[2].x);
            q[0].y = join(q[0].y, q[1].y, q[2].y);
        }
        if (own) {
            const SceneDev& sc = a.scenes[s_scene[beg]];
            const int nb = sc.nb, lx = ((key >> 4) & 3) + i;
            const float m = sc.m_p;
            float4* g = a.G + (key + i * 16 + (lx > 3 ? (nb * nb - 1) * 64 : 0));
#pragma unroll
            for (int q = 0; q < 9; ++q)
                if (q % 3 == 0 || last) {
                    float4* to = g + ((q / 3) * 4 + q % 3 + (ly + q / 3 > 3 ? nb * 64 - 16 : 0) + (lz + q % 3 > 3 ? 60 : 0));
                    if (MODE == kP2GAdj) red_add_v4(to, acc_a[q].x, acc_a[q].y, acc_b[q].x, 0.f);
                    else red_add_v4(to, acc_b[q].y * m, acc_a[q].x, acc_a[q].y, acc_b[q].x);
                }
        }
    }
}

// Variants of the forward G2P (template flags).
enum {
    kG2PSolids = 1,    // push particles out of solid rigids (some scene has a sphere or a box)
    kG2PStdGrad = 2,   // standard MPM: L = sum v_I grad phi^T instead of the APIC C (Eq. 5)
    kG2PNoStress = 4,  // PB-MPM: no constitutive update (no stress is stored)
    kG2PReadOnly = 8   // nodes through the read-only path (GridStencil): for launch_alone only
};

// Velocity and affine matrix gathered at a position:
//   v = sum W v_I,  B_rc = sum W v_I,r (o_c - f_c),  W = wx_i wy_j wz_k
// (kG2PStdGrad: the basis gradient in cell units instead, B_rc = sum v_I,r dW/df_c),
// contracted separably over k, then j, then i; x and y go in paired FMAs.  The
// velocities are taken relative to the middle node's, whose share is known (sum W = 1,
// B = 0): a bulk motion then leaves no rounding in B.
// node(i, j, k) returns (v, m) of the stencil's nodes.
template <int FLAGS, class Node>
__device__ __forceinline__ void gather_velocity(const float f[3], const float w[9], Node node, float v[3], float B[9])
{
    const float* wy = w + 3;
    const float* wz = w + 6;
    float wyd[3], wzd[3];
    if (FLAGS & kG2PStdGrad) {
        bspline_d(f[1], wyd);
        bspline_d(f[2], wzd);
    } else {
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            wyd[q] = wy[q] * ((float)q - f[1]);
            wzd[q] = wz[q] * ((float)q - f[2]);
        }
    }
    const auto two = [](float s) { return make_float2(s, s); };
    const float4 mid = node(1, 1, 1);
    float2 vp = two(0.f), B0 = two(0.f), B1 = two(0.f), B2 = two(0.f);  // x, y rows
    float vz = 0.f, Bz0 = 0.f, Bz1 = 0.f, Bz2 = 0.f;                    // z row
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        // weight of plane i (as bspline) and its derivative or moment
        const float fi = (float)i;
        const float e = f[0] - (1.5f - 0.5f * fi);
        const float wx = i == 1 ? 0.75f - e * e : 0.5f * e * e;
        const float wxd = (FLAGS & kG2PStdGrad) ? (i == 1 ? -2.f * e : e) : wx * (fi - f[0]);
        float2 A = two(0.f), Ay = two(0.f), Az = two(0.f);
        float zA = 0.f, zAy = 0.f, zAz = 0.f;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            float2 p = two(0.f), d = two(0.f);
            float zp = 0.f, zd = 0.f;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const float4 g = node(i, j, k);
                const float2 xy = __fadd2_rn(make_float2(g.x, g.y), make_float2(-mid.x, -mid.y));
                const float z = g.z - mid.z;
                p = __ffma2_rn(two(wz[k]), xy, p);
                d = __ffma2_rn(two(wzd[k]), xy, d);
                zp = __fmaf_rn(wz[k], z, zp);
                zd = __fmaf_rn(wzd[k], z, zd);
            }
            A = __ffma2_rn(two(wy[j]), p, A);
            Ay = __ffma2_rn(two(wyd[j]), p, Ay);
            Az = __ffma2_rn(two(wy[j]), d, Az);
            zA = __fmaf_rn(wy[j], zp, zA);
            zAy = __fmaf_rn(wyd[j], zp, zAy);
            zAz = __fmaf_rn(wy[j], zd, zAz);
        }
        vp = __ffma2_rn(two(wx), A, vp);
        B0 = __ffma2_rn(two(wxd), A, B0);
        B1 = __ffma2_rn(two(wx), Ay, B1);
        B2 = __ffma2_rn(two(wx), Az, B2);
        vz = __fmaf_rn(wx, zA, vz);
        Bz0 = __fmaf_rn(wxd, zA, Bz0);
        Bz1 = __fmaf_rn(wx, zAy, Bz1);
        Bz2 = __fmaf_rn(wx, zAz, Bz2);
    }
    v[0] = vp.x + mid.x; v[1] = vp.y + mid.y; v[2] = vz + mid.z;
    B[0] = B0.x; B[1] = B1.x; B[2] = B2.x;
    B[3] = B0.y; B[4] = B1.y; B[5] = B2.y;
    B[6] = Bz0; B[7] = Bz1; B[8] = Bz2;
}

// Nodes of a base cell's stencil in the brick layout, read through L1.  READ_ONLY: by the
// read-only path, which is for data that nothing writes while the kernel lives; a programmatic
// launch comes up while the grid update still writes the nodes, and chain_wait orders ordinary
// accesses only.  A substep with the one and the other: 123.1 and 124.7 us at 1M particles,
// 411 and 419 at 4M (530 and 565 with 64 registers), 24.0 and 24.3 at 64k.
template <bool READ_ONLY>
struct GridStencil {
    const float4* V;
    int x0, sx, o[6];  // first x, stride of bricks along x, node offsets along y and z (with the scene's first node)
    __device__ __forceinline__ GridStencil(const float4* V_, const SceneDev& sc, const int bc[3]) : V(V_), x0(bc[0])
    {
        const int sy = sc.nb * 64;
        sx = sc.nb * sy;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const int y = bc[1] + i, z = bc[2] + i;
            o[i] = (y >> 2) * sy + (y & 3) * 4 + sc.brick_base * 64;
            o[3 + i] = (z >> 2) * 64 + (z & 3);
        }
    }
    __device__ __forceinline__ float4 operator()(int i, int j, int k) const
    {
        const int x = x0 + i, ox = (x >> 2) * sx + (x & 3) * 16;
        const float4* at = V + (ox + o[j] + o[3 + k]);
        return READ_ONLY ? __ldg(at) : *at;
    }
};

// Global node index of node (gi, gj, gk) of a scene (brick layout).
__device__ __forceinline__ int node_index(const SceneDev& sc, int gi, int gj, int gk)
{
    const int brick = sc.brick_base + ((gi >> 2) * sc.nb + (gj >> 2)) * sc.nb + (gk >> 2);
    return brick * 64 + (gi & 3) * 16 + (gj & 3) * 4 + (gk & 3);
}

__device__ __forceinline__ void issue_halo(const StepArgs& a, int item, float4* dst, unsigned long long* bar)
{
    item = active_entry(a.sb, item);
    const int b = a.sb.act_brick[item];
    const SceneDev& sc = a.scenes[a.sb.act_scene[item]];
    const int nb = sc.nb, lb = b - sc.brick_base;
    int bx, by, bz;
    brick_coords(nb, sc.nb_log2, lb, bx, by, bz);
    fence_proxy_async();
    unsigned bytes = 0;
#pragma unroll
    for (int o = 0; o < 8; ++o)
        if (bx + (o >> 2) < nb && by + ((o >> 1) & 1) < nb && bz + (o & 1) < nb) bytes += 64 * sizeof(float4);
    mbar_expect_tx(bar, bytes);
#pragma unroll
    for (int o = 0; o < 8; ++o) {
        const int ex = bx + (o >> 2), ey = by + ((o >> 1) & 1), ez = bz + (o & 1);
        if (ex < nb && ey < nb && ez < nb)
            bulk_g2s(dst + o * 64, &a.V[(sc.brick_base + (ex * nb + ey) * nb + ez) * 64], 64 * sizeof(float4), bar);
    }
}

// Shared prologue of the brick-walking kernels: mbarriers, first halo.
template <int BLOCK>
__device__ __forceinline__ void walker_init(const StepArgs& a, int n_act, float4 (*vw)[8 * 64], unsigned long long* bar,
                                            int* s_item, int* work)
{
    const int tid = threadIdx.x;
    if (tid == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        fence_mbar_init();
        const int first = atomicAdd(work, 1);
        s_item[0] = first;
        if (first < n_act) issue_halo(a, first, vw[0], &bar[0]);
    }
    __syncthreads();
}

// The lists of this substep are done with: keep their sizes for mpm_phase_stats
// and start the next scan's from empty.
__device__ __forceinline__ void reset_lists(const SortBufs& sb)
{
    sb.counters[CTR_LAST_ACT] = active_bricks(sb);
    sb.counters[CTR_LAST_NACT] = sb.counters[CTR_N_NACT];
    sb.counters[CTR_N_BIG] = sb.counters[CTR_N_SMALL] = sb.counters[CTR_N_NACT] = 0;
}

// Epilogue of the forward G2P launches, run by one warp of every CTA on its
// way out: the last CTA to finish advances the scene clocks and substep counters
// (read by the next grid update and the state readback).  No CTA of the launch
// reads a clock after it has counted itself out, so the clocks stay constant
// while G2P evaluates rigid poses at the end of the substep.
__device__ __forceinline__ void count_out(const StepArgs& a)
{
    const int lane = threadIdx.x & 31;
    int done = 0;
    if (lane == 0) {
        __threadfence();
        done = atomicAdd(&a.sb.counters[CTR_DONE_G2P], 1);
    }
    if (__shfl_sync(kFull, done, 0) != (int)gridDim.x - 1) return;
    __threadfence();
    for (int s = a.r.s0 + lane; s < a.r.s1; s += 32) {
        a.t_scene[s] += (double)a.dt;
        a.epoch[s] += 1;
    }
    if (lane == 0) {
        a.sb.counters[CTR_DONE_G2P] = 0;
        reset_lists(a.sb);
    }
}

__device__ __forceinline__ void walker_exit(const StepArgs& a)
{
    __syncthreads();
    if (threadIdx.x < 32) count_out(a);
}

// Centre and rotation matrix of a rigid at clock t_now.
__device__ __forceinline__ void rigid_pose_at(const RigidDev& src, double t_now, float c[3], float R[9])
{
    const float tau = (float)(t_now - src.t_set);
#pragma unroll
    for (int i = 0; i < 3; ++i) c[i] = src.c0[i] + tau * src.vel[i];
    // q(tau) = exp(tau omega / 2) * q0
    const float wx = src.omega[0], wy = src.omega[1], wz = src.omega[2];
    const float wn = sqrtf(wx * wx + wy * wy + wz * wz);
    float qw = src.q0[0], qx = src.q0[1], qy = src.q0[2], qz = src.q0[3];
    if (wn > 0.f) {
        float sh, ch;
        sincosf(0.5f * wn * tau, &sh, &ch);
        const float ax = wx / wn * sh, ay = wy / wn * sh, az = wz / wn * sh;
        const float nw = ch * qw - ax * qx - ay * qy - az * qz;
        const float nx = ch * qx + ax * qw + ay * qz - az * qy;
        const float ny = ch * qy - ax * qz + ay * qw + az * qx;
        const float nz = ch * qz + ax * qy - ay * qx + az * qw;
        qw = nw; qx = nx; qy = ny; qz = nz;
    }
    quat_to_mat(qw, qx, qy, qz, R);
}

// Poses at the end of the substep (clock + dt) of the solid rigids of a scene,
// staged in shared memory by the threads tid < kMaxRigids of a group; the rigid
// slots in use (shapes other than sphere and box are staged with type -1).
__device__ __forceinline__ void stage_solids(const StepArgs& a, int scene, SolidPose* poses, int tid)
{
    const int nr = a.scenes[scene].n_rigid;
    if (tid < nr) {
        const RigidDev& src = a.rigids[scene * kMaxRigids + tid];
        SolidPose& P = poses[tid];
        P.type = (src.type == MPM_SPHERE || src.type == MPM_BOX) ? src.type : -1;
        rigid_pose_at(src, a.t_scene[scene] + (double)a.dt, P.c, P.R);
        P.radius = src.radius;
#pragma unroll
        for (int i = 0; i < 3; ++i) P.half[i] = src.half[i];
    }
}

// Particle push-out (Sec. IV-A): a particle that ends the substep inside a
// solid rigid (sdf < 0 at the rigid's pose at the end of the substep) moves
// to the nearest surface point, x - sdf(x) n(x); rigids in id order.  Blades
// and line segments push nothing out (the tissue closes around them).
__device__ __forceinline__ void push_out(const SolidPose* poses, int nr, float x[3])
{
    for (int r = 0; r < nr; ++r) {
        const SolidPose& P = poses[r];
        if (P.type == MPM_SPHERE) {
            const float d0 = x[0] - P.c[0], d1 = x[1] - P.c[1], d2 = x[2] - P.c[2];
            const float l = sqrtf(d0 * d0 + d1 * d1 + d2 * d2);
            if (l < P.radius) {
                if (l > 0.f) {
                    const float k = P.radius / l;
                    x[0] = P.c[0] + k * d0;
                    x[1] = P.c[1] + k * d1;
                    x[2] = P.c[2] + k * d2;
                } else {  // at the centre: along the body y axis
                    x[0] = P.c[0] + P.radius * P.R[1];
                    x[1] = P.c[1] + P.radius * P.R[4];
                    x[2] = P.c[2] + P.radius * P.R[7];
                }
            }
        } else if (P.type == MPM_BOX) {
            const float d0 = x[0] - P.c[0], d1 = x[1] - P.c[1], d2 = x[2] - P.c[2];
            float p[3] = {P.R[0] * d0 + P.R[3] * d1 + P.R[6] * d2, P.R[1] * d0 + P.R[4] * d1 + P.R[7] * d2,
                          P.R[2] * d0 + P.R[5] * d1 + P.R[8] * d2};
            const float q0 = fabsf(p[0]) - P.half[0], q1 = fabsf(p[1]) - P.half[1], q2 = fabsf(p[2]) - P.half[2];
            if (q0 < 0.f && q1 < 0.f && q2 < 0.f) {
                // nearest face: the axis of the largest q (ties to the lower axis)
                const int ax = (q0 >= q1 && q0 >= q2) ? 0 : (q1 >= q2 ? 1 : 2);
                p[ax] = p[ax] >= 0.f ? P.half[ax] : -P.half[ax];
                x[0] = P.c[0] + P.R[0] * p[0] + P.R[1] * p[1] + P.R[2] * p[2];
                x[1] = P.c[1] + P.R[3] * p[0] + P.R[4] * p[1] + P.R[5] * p[2];
                x[2] = P.c[2] + P.R[6] * p[0] + P.R[7] * p[1] + P.R[8] * p[2];
            }
        }
    }
}

// Prefetch the next brick's halo and wait for this one; false on timeout (the
// CTA must then return).
__device__ __forceinline__ bool walker_next(const StepArgs& a, int n_act, float4 (*vw)[8 * 64], unsigned long long* bar,
                                            int* s_item, int* work, int buf, unsigned* phase, int item)
{
    if (threadIdx.x == 0) {
        const int next = atomicAdd(work, 1);
        s_item[buf ^ 1] = next;
        if (next < n_act) issue_halo(a, next, vw[buf ^ 1], &bar[buf ^ 1]);
    }
    const bool ok = mbar_wait_bounded(&bar[buf], phase[buf]);
    if (__syncthreads_or(!ok)) {
        if (threadIdx.x == 0) atomicOr(&a.err[a.sb.act_scene[active_entry(a.sb, item)]], MPM_EBIT_TIMEOUT);
        mbar_wait_bounded(&bar[buf], phase[buf]);  // let copies in flight land before leaving
        mbar_wait_bounded(&bar[buf ^ 1], phase[buf ^ 1]);
        return false;
    }
    phase[buf] ^= 1u;
    return true;
}

}  // namespace mpm
