// Kernel parameter blocks and host-side launchers of the forward substep.
#pragma once

#include "mpm_device.cuh"

namespace mpm {

struct Range {
    int s0, s1;     // scene range [s0, s1)
    int bb0, nbr;   // global brick range [bb0, bb0 + nbr)
    int t0, nt;     // scan tile range [t0, t0 + nt)
    int p0, np;     // particle range [p0, p0 + np)
};

struct SortBufs {
    int* key;       // [cap] brick x 64 + base cell of each stored particle (next substep)
    int* rank;      // [cap] rank of the particle within its cell
    int* perm;      // [cap] sorted slot -> storage index
    int* cnt;       // [bricks] particles per brick (next substep)
    int* ccnt;      // [bricks * 64] particles per cell (next substep); the scan turns an active
                    // brick's into the cells' first slots
    int* act_brick; // [list_size] active particle bricks: those of at least kBigBrick particles from
                    // the front, the others from the back (active_entry)
    int* act_start;
    int* act_count;
    int* act_scene;
    int* nact_brick;// [bricks] active node bricks
    int* nact_scene;
    int* counters;  // [CTR_COUNT]
    int* tile_n;    // [tiles] particles per scan tile of the next substep, added up by the key
                    // producers, read by the scan and cleared by the scatter
    int tile_shift; // log2 of the bricks per scan tile
    int list_size;  // entries of the active-brick lists (all bricks)
};

struct StepArgs {
    Range r;
    SortBufs sb;
    const SceneDev* scenes;
    const RigidDev* rigids;      // [n_scenes * kMaxRigids]
    RigidPose* pose;             // [n_scenes * kMaxRigids] at the scenes' clocks, by the scan
    double* impulse;             // [n_scenes * kMaxRigids * 6]
    double* t_scene;             // [n_scenes] scene clocks
    int* epoch;                  // [n_scenes] substep counters
    int* brick_epoch;            // [bricks] substep of the last grid update of a node brick
    unsigned* err;               // [n_scenes]
    float4* G;                   // P2G accumulator (m, mv)
    float4* V;                   // node (v, m)
    PState in, out;
    int cap;
    float dt;
    float gravity[3];
    int bound, floor_sticky;
    int model, plasticity;
    float yield_stress;
    int g2p_ctas;                // most CTAs of the persistent G2P kernel
    int p2g_ctas, grid_ctas;     // CTAs of the persistent P2G and grid kernels
    int grid_plain_ctas;         // CTAs of the grid kernel of launches without rigids
    int fused_ctas;              // CTAs of the fused G2P + P2G kernel
    int p2g_slots;               // slots that a P2G warp stages at once
    int g2p_threads, g2p_regs64;
    int tau_valid;               // P2G reads the stored stress (else recomputes it from F)
    int any_rigid;               // some scene of the range has a rigid (contact in the grid update)
    int rigid_ext;               // some scene of the range has an arc or a mesh slicer
    int any_solid;               // some scene of the range has a sphere or a box (particle push-out)
    int solver;                  // MPM_SOLVER_*
    float pb_beta;               // PB-MPM constraint blend
};

constexpr int kStateFloats = 34;  // eight float4 planes, mu, lam
constexpr int kP2GThreads = 192;  // six warps, each with slots of its own
constexpr int kP2GMaxSlots = 64;
constexpr int kScanThreads = 256;
// A scan tile holds 64 bricks or more: its CTA also turns the cells' counts of its particle
// bricks into first slots, a warp a brick, which is what takes long.  With 256 bricks or more
// a substep took 127.5 us on the 1M block (now 118.0: tiles of 128, see mpm_create), 33.2 with
// the indenter at 100k (31.7), 22.1 at 16k (20.9).
constexpr int kMinTileShift = 6;
// Launches of fewer particles are made programmatic (launch_chain).  A substep with and
// without: 19.6 and 21.0 us at 4k particles, 22.2 and 23.8 at 16k, 22.4 and 23.7 at 32k, 24.3
// and 24.9 at 48k; 26.4 and 25.1 at 64k, 134 and 128 at 1M, where CTAs that wait take the
// place of CTAs that work.
constexpr int kChainBelow = 48 << 10;
constexpr int kScatterPer = 4;  // particles per thread of the counting-sort scatter
// Particle bricks of at least this many particles come first in the active list,
// so the fused kernel, whose CTAs take bricks in turn, ends on small ones (a shorter tail)
constexpr int kBigBrick = 256;

cudaError_t launch_prepare(const StepArgs& a, const PState& st, cudaStream_t s);
// zero the brick histogram, the tile counts and the list sizes (all scenes)
cudaError_t launch_reset_histogram(const SortBufs& sb, int bricks, int tiles, int np, cudaStream_t s);
// the scan alone serves launches that bring a permutation of their own
cudaError_t launch_scan(const StepArgs& a, cudaStream_t s);
cudaError_t launch_sort(const StepArgs& a, cudaStream_t s);
cudaError_t launch_p2g(const StepArgs& a, cudaStream_t s);
cudaError_t prepare_kernels();  // shared-memory sizes of P2G and G2P (once per device, before any launch)
// clear: reset the P2G accumulator afterwards (G2P does it otherwise)
cudaError_t launch_grid(const StepArgs& a, cudaStream_t s, bool clear);
cudaError_t launch_g2p(const StepArgs& a, cudaStream_t s);
cudaError_t launch_g2p_vc(const StepArgs& a, cudaStream_t s);   // PB-MPM cycle G2P (v, C in place)
cudaError_t launch_g2p2g(const StepArgs& a, cudaStream_t s);
int occupancy_g2p2g();
int occupancy_grid();
int occupancy_grid_plain();

// state I/O helpers
cudaError_t launch_init_particles(const PState& st, int cap, int p_at, int n, int id0, const float* x,
                                  const float* v, const float* E, const float* nu, float E0, float nu0,
                                  cudaStream_t s);
// x, v, C, F (null: not moved) of one scene as arrays in particle-id order
struct Fields {
    float* f[4];
};
// Three or more fields whose arrays hold this many bytes are read into device memory through
// records, all others by slot, in one kernel: the entries that a warp scatters come together
// in L2 (129 MB) while it holds the arrays.  A read through records and by slot: x, v, C and F
// 128 and 117 us at 1M particles (101 MB), 189 and 230 at 1.5M, 475 and 755 at 4M; x, C and F
// 180 and 187 at 1.5M; x, v and C 226 and 194 at 2M, 448 and 499 at 4M; C and F 454 and 449 at
// 4M, 2,072 and 1,910 at 16M; x alone 114 and 27 at 1M, 397 and 44 at 4M.
constexpr size_t kIoRecordsFrom = 120'000'000;
// state -> arrays (out) or arrays -> state; inv: scratch of np ints, spare: the state's other
// buffer (all but its plane 0 is scratch); host: the arrays are pinned host memory
cudaError_t launch_fields(const PState& st, const PState& spare, int cap, int p0, int np, int* inv, const Fields& h, bool out,
                          bool host, cudaStream_t s);
cudaError_t launch_order(const PState& st, int p0, int np, int* dst, cudaStream_t s);  // ids by slot
cudaError_t launch_set_rigid(const RigidDev& d, RigidDev* dst, cudaStream_t s);
cudaError_t launch_read_grid(const float4* V, const int* brick_epoch, const int* epoch, const SceneDev* scenes,
                             int scene, int n, int brick_base, float* dst, cudaStream_t s);
int occupancy_p2g(int slots);
int occupancy_g2p(int threads, int regs64);

}  // namespace mpm
