// mppi_internal.h - types shared by the kernels and the C ABI implementation.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <atomic>

namespace mppi {

// Largest block of the single-plan rollout kernel: it is compiled for 896 lanes per SM (at
// most 72 registers a thread), as one block of 896 or several smaller ones.  One block per SM
// matters: two co-resident blocks of one wave do not progress alike (the second ran ~16 %
// slower), and the second then finished alone at half occupancy.
constexpr int MAX_ROLLOUT_THREADS = 896;

// Largest block of the batched planner's rollout kernel (two per SM).
constexpr int BATCH_MAX_THREADS = 448;

// Every value finite: no exponent field all ones (inf, NaN).  Adding one unit of the exponent
// field to the masked exponent carries into the top bit only from all ones, so the pass is
// integer and, or and add without branches, and the compiler vectorises it.
inline bool finite_all(const double* v, size_t n) {
    const uint64_t exp_mask = 0x7ff0000000000000ull, exp_one = 0x0010000000000000ull;
    uint64_t bad = 0;
    for (size_t i = 0; i < n; ++i) {
        uint64_t bits;
        memcpy(&bits, v + i, sizeof(bits));
        bad |= (bits & exp_mask) + exp_one;
    }
    return (bad >> 63) == 0;
}

// set() the first time the calling thread's current device needs it.  A kernel's attributes (here its
// opt-in to more than 48 KB of dynamic shared memory) belong to one device, while the contexts of several
// devices, driven from several threads, share the process: done holds a bit per device.  A device past
// the last bit sets it on every launch.
template <typename Set>
inline cudaError_t once_per_device(std::atomic<unsigned long long>& done, Set set) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = dev >= 0 && dev < 64 ? 1ull << dev : 0ull;
    if (done.load(std::memory_order_acquire) & bit) return cudaSuccess;
    e = set(dev);
    if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_release);
    return e;
}

// Per-context device record: iteration counter, status and the reduction results.
struct __align__(16) DevState {
    unsigned long long iter;     // next iteration index (low 32 bits enter the Philox counter)
    int32_t flags;               // FLAG_* raised by kernels
    int32_t status;              // mppi_status of the last iteration
    double s_min;                // lowest sample cost
    double eta;                  // sum of softmin weights
    int32_t argmin;
    int32_t n_finite;
    unsigned int ticket;         // last-block-done counter of the argmin reduction (rollout kernel)
    int32_t jb0;                 // reference segment closest to x0
    unsigned long long jkey;     // packed (distance bits, index) for the jb0 search
    float4 x0f;                  // (0, 0, yaw0, v0): x0 in the local frame
    unsigned long long iter_used;  // iteration index of the last finished iteration
    int32_t moving;              // some obstacle circle has a nonzero velocity
    float delta0f;               // steering angle of x0 (model 1)
    int32_t multi_head;          // the reference polyline has segments of more than one heading
    int32_t pad_;
};

// Byte offsets of the arrays in the scene blob that the rollout kernel stages into
// shared memory with one bulk copy.  Every offset is a multiple of 16.
struct SceneLayout {
    int T, n_ref, n_seg, n_l1, n_l2, n_circ;   // chunks of REF_L1 segments, groups of REF_L2 chunks
    int off_ctl;     // float4 [T]       (u_a, u_d, g_a, g_d): nominal controls and control-cost slopes
    int off_c0;      // float  [T]       1/2 u^T R u
    int off_vert;    // float2 [n_ref]   vertices, local frame
    int off_seg;     // float4 [n_seg]   (ex, ey, ex/|e|^2, ey/|e|^2)
    int off_head;    // float  [n_seg]   heading of each segment
    int off_cert;    // float  [n_ref]   squared distance up to which the window of three settles the search
    // the circles are stored sorted by their key s = p . d (p: the first centre, d: the axis, circle_axis)
    int off_circ;    // float4 [n_circ]  (x, y, r, (d_safe_0 + r + r_ego)^2 when d_safe is constant)
    int off_vel;     // float2 [n_circ]  velocities
    int off_disp;    // float  [n_circ]  bound on the distance a centre moves in one step
    int off_proj;    // float4           (dx, dy, 0, 0): unit direction of the lane (first to last vertex)
    int off_order;   // int    [n_circ]  input index of each sorted circle (its column of the centre table)
    int off_skey;    // float  [n_circ]  the sorted keys
    int bytes;       // the staged part (all of the above), a multiple of 16
    // after the staged part, read from global memory (through L1) by the search outside its window:
    int off_l1;      // float4 [n_l1]    level-1 chunk boxes
    int off_l2;      // float4 [n_l2]    level-2 boxes (REF_L2 chunks each)
    int off_pbox;    // float4 [n_ref]   box of the vertices 0 .. i
    int off_sbox;    // float4 [n_ref]   box of the vertices i .. n_ref - 1
    int total;       // the whole scene buffer, a multiple of 16
};

// Per-plan constants in the precision the kernels use.
struct PlanConst {
    int K, T;
    float dt, dt_over_L;
    float sig_a, sig_d, amin, amax, dmin, dmax;
    float w_dist, w_target, w_yaw, w_speed, w_safe, w_terminal;
    float v_ref, v_max;
    int vcap;
    float d_safe_c, d_safe_0;
    int collision_only;
    int n_ego;
    int ego_same_radius;     // all ego radii equal: the band limit is per circle
    float ego_off[8], ego_rad[8];
    float ego_omin, ego_omax, ego_rmax;   // extent of the ego circles along the heading, largest radius
    int ref_mode;
    int has_table;           // per-step centre table given
    uint32_t key0, key1, session;
    // double-precision parameters of the update and the optimal rollout
    double lam, dt_d, wheelbase_d, amin_d, amax_d, dmin_d, dmax_d, v_max_d;
    double g_a, g_d;         // (1 + alpha) R_a, (1 + alpha) R_d
    double half_Ra, half_Rd; // R / 2
    int sg_enable, shift;
    // last, so the members above keep their offsets (the weighted-sum kernel measurably
    // slows down when they move)
    int model;               // 0: control (a, delta); 1: state carries delta, control (a, omega)
    int cost_to_go;          // 1: per-step weights from the cost still to come
    double dt_over_wb_d;     // dt / wheelbase
    float inv_lam_f;         // 1 / lambda
    uint32_t k_offset;       // global index of sample 0 (a K-slice of a partitioned plan; else 0)
};

SceneLayout make_layout(int T, int n_ref, int n_circ);

// Samples per k-tile of the weighted sum: 256 threads of WS_J samples each.
constexpr int WSUM_KT = 2048;

// Blocks of wsum_kernel an SM holds (its launch bounds): 32 registers a thread, but 40 where the weights
// change with the step (ctg) and in tiles of one step.
__host__ __device__ constexpr int wsum_blocks_per_sm(int tt, bool ctg) { return ctg || tt == 1 ? 6 : 8; }

// Steps per tile of the weighted sum (PlanBuffers::tt_len) for a plan of n_kt k-tiles.  A tile's time
// grows with its steps plus about one more (weights, reduction, ticket), and the tiles run in rounds of
// the blocks the GPU holds, so the rule takes the length with the fewest rounds x (steps + 1); the longest
// among equals.  (The longest of 8, 4, 2, 1 with six tiles per SM left 1.3 rounds at 65,536 x 200: 32 us,
// with 6 steps in one round 27; 262,144 x 100 69 -> 57 us; both with the 32 registers that eight blocks
// per SM need, which the kernel had outgrown.)
inline int wsum_tile_steps(int K, int T, int n_kt, int n_sm, int noise_bf16, int ctg) {
    const bool staged = noise_bf16 && !ctg && K % 4 == 0;
    int best = 1;
    long long cost = -1;
    for (int tt : {1, 2, 3, 4, 6, 8}) {
        // the staged tiles (eight blocks an SM) also share its memory: with three steps and more they hold the
        // same 24 steps an SM, so six and eight are never the cheapest and have no staged kernel
        const int fit = (224 * 1024) / (tt * WSUM_KT * 4 + 2048);
        const long long slots = (long long)n_sm * (!staged ? wsum_blocks_per_sm(tt, ctg != 0) : fit < 8 ? fit : 8);
        const long long tiles = (long long)n_kt * ((T + tt - 1) / tt), rounds = (tiles + slots - 1) / slots;
        const long long c = rounds * (tt + 1);
        if (cost < 0 || c <= cost) {
            cost = c;
            best = tt;
        }
    }
    return best;
}

// The plan's parameters allow the specialised rollout step (rollout_sample's SIMPLE): three ego
// circles of one radius, a constant safety band, no collision-only switch, no speed cap, the
// segment form of the closest waypoint, no centre table, the 4-state model with whole-cost weights.
inline bool simple_plan(const PlanConst& pc) {
    return pc.n_ego == 3 && pc.ego_same_radius && pc.d_safe_c == 0.0f && !pc.collision_only && !pc.vcap &&
           pc.ref_mode == 0 && !pc.has_table && pc.model == 0 && !pc.cost_to_go;
}

struct PlanBuffers {
    DevState* state;
    unsigned char* scene;    // SceneLayout::bytes
    float2* table;           // [T][n_circ] centres, local frame (when given)
    void* z;                 // [T][K] float2 or bf16x2
    double* S;               // [K]
    float* w;                // [K] softmin weights
    double* eta_part;        // [n_wblk]
    ulonglong2* kmin_part;   // [K] per rollout block: (cost order key, (finite count << 32) | index)
    double* du_part;         // [n_kt][T][2]
    double* du;              // [T][2] sum over the k-tiles (wsum's last block per step tile), or null
    unsigned* tt_count;      // [n_tt] k-tile blocks done per step tile (zero between launches)
    double* U;               // [T][2] nominal controls (the warm start)
    unsigned long long* stats;  // [7] work counters (STATS launches only)
    unsigned* fix_count;     // bfloat16 noise: pairs whose rounding is taken again in binary64
    uint2* fix_list;         // [NOISE_FIX_CAP] their (step pair j, sample k); null: decided in place
    float* ctg_prefix;       // [T][K] cost of steps 0..t-1 per sample (cost-to-go form), or null
    float* wt;               // [T][K] per-step softmin weights (cost-to-go form)
    double* eta_t;           // [T] per-step normalisers (cost-to-go form)
    int n_wblk, n_kt, n_tt, kt_size;
    int tt_len;              // steps per step tile of the weighted sum (<= WS_TT)
    int n_sm;                // SMs of the device
};

// Shared memory each rollout block builds after the staged blob: the circle index (a float4
// of scalars and CIRC_BUCKETS + 1 bucket starts into the sorted circles) and the context of
// the closest-point search's out-of-line path.
constexpr int CIRC_BUCKETS = 64;

constexpr int CIRC_INDEX_BYTES = 16 + 4 * ((CIRC_BUCKETS + 1 + 3) & ~3);
constexpr int SEARCH_CTX_BYTES = 112;

__host__ __device__ inline size_t block_extra_bytes(const SceneLayout&) {
    return (size_t)CIRC_INDEX_BYTES + SEARCH_CTX_BYTES;
}

// Per-thread slots after the block's extras: the compensated steering angle of the
// steering-rate model (float2 per thread of the block), kept out of the registers of the
// other model; none for the 4-state model.
__host__ __device__ inline size_t steer_slots_bytes(int threads, bool model1) {
    return model1 ? (size_t)8 * threads : 0;
}

// Capacity of the deferred bfloat16 rounding list (pairs beyond it are decided in place).
constexpr unsigned NOISE_FIX_CAP = 1u << 16;

struct PlanInputs {
    const double* x0;        // [4]
    const double* ref;       // [n_ref][2]
    const double* circ;      // [n_circ][5]
    const double* centres;   // [T][n_circ][2] or null
    int n_ref, n_circ;
    double* u_out;           // [T][2]
    double* x_out;           // [T+1][4]
    DevState* state_out = nullptr;   // when set, finalize copies the device record here (pinned host)
};

// Launch the whole iteration (prep, noise, rollout, reductions, update) on a stream.
// ev: optional array of N_KERNELS + 1 events; ev_mode 1 records them around every kernel
// (per-kernel timing: the prep stage is the prep + noise launch, the noise stage the bf16
// fix-up, the argmin stage empty since the rollout kernel ends with the argmin), 2 only ev[2]
// and ev[3] around the rollout (the rest stays chained).
constexpr int N_KERNELS = 7;   // prep, noise, rollout, argmin, weights, wsum, finalize
// inject: status flags written into the device record between the rollout and the weights
// (debug: the failure path without a fault; 0 = none; the source must outlive the launch).
cudaError_t launch_iteration(const PlanConst& pc, const SceneLayout& L, const PlanBuffers& b,
                             const PlanInputs& in, int group, int threads, int noise_bf16, cudaStream_t st,
                             cudaEvent_t* ev = nullptr, int ev_mode = 1, const int* inject = nullptr);

// The iteration split at the two exchanges of a K-partitioned plan (each context holds the
// slice of samples k_offset .. k_offset + K - 1): costs (prep, noise, rollout with the slice's
// S_min and argmin), sums (softmin weights against the global S_min and the weighted noise
// sums), finalize (update, smoothing, x*, warm start from the summed eta and du).
cudaError_t launch_slice_costs(const PlanConst& pc, const SceneLayout& L, const PlanBuffers& b,
                               const PlanInputs& in, int group, int threads, int noise_bf16, cudaStream_t st);
cudaError_t launch_slice_sums(const PlanConst& pc, const SceneLayout& L, const PlanBuffers& b, int noise_bf16,
                              cudaStream_t st);
cudaError_t launch_slice_finalize(const PlanConst& pc, const PlanBuffers& b, const PlanInputs& in, cudaStream_t st);

// prep + noise only (no change to the warm start or the iteration counter) and the
// reset of the fields prep accumulates into; used by the autotuner.
cudaError_t launch_prep_noise(const PlanConst& pc, const SceneLayout& L, const PlanBuffers& b,
                              const PlanInputs& in, int noise_bf16, cudaStream_t st);
cudaError_t launch_reset_state(DevState* st, cudaStream_t s);

// Bounds-checking debug build (MPPI_CHECKS): the index violations counted by the kernels of
// each translation unit since the last call (then reset; 0 in the normal build), and a kernel
// with two out-of-range indices that the checks must count (a4: 4 ints, out: 1 int).
cudaError_t take_check_hits_kernels(unsigned long long* hits);
cudaError_t take_check_hits_batch(unsigned long long* hits);
cudaError_t run_check_selftest(int* a4, int* out, cudaStream_t st);

// Raw Philox words for n counters (device buffers).
cudaError_t launch_philox(uint2 key, const uint4* ctr, uint4* out, int n, cudaStream_t st);

// Rollout kernel only (for timing and tuning); requires prep and noise of the same plan.
cudaError_t launch_rollout(const PlanConst& pc, const SceneLayout& L, const PlanBuffers& b, int group,
                           int threads, int noise_bf16, cudaStream_t st);

// Rollout with work counters (1 lane per sample): accumulates into b.stats.
cudaError_t launch_rollout_stats(const PlanConst& pc, const SceneLayout& L, const PlanBuffers& b, int noise_bf16,
                                 cudaStream_t st);

// Dynamic shared memory of a rollout block: the staged blob, the extras the block builds and
// the steering slots (threads of the block; model1: the steering-rate model).
size_t rollout_smem_bytes(const SceneLayout& L, int threads, bool model1);

// Resident rollout blocks per SM for a launch shape (0 if it cannot launch).
// ext: the steering-rate model or the cost-to-go form is on (PlanConst model / cost_to_go)
int rollout_max_blocks_per_sm(int group, int threads, int noise_bf16, size_t smem, bool ext);

}  // namespace mppi
