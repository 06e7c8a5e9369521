// mppi_batch.cu - many independent MPPI iterations per launch (the batched planner).
//
// A submission carries n plans with their own K, T, reference, obstacles and warm-start
// slot.  All n are computed by one fixed sequence of kernels captured once in a CUDA
// graph: per-plan scene preparation, noise over the flattened (plan, step pair, sample)
// space, ONE persistent rollout kernel whose blocks pull (plan, sample block) tiles, longest
// plans first, from an atomic counter and re-stage a plan's scene into shared memory by
// TMA only when the plan changes, per-plan reductions, and per-plan smoothing and optimal
// rollout.  The per-sample arithmetic is the single-plan path's (mppi_iter.cuh), so a
// plan's result does not depend on which other plans share its submission.
//
// Warm starts live in device slots shared by all pipelines; a pipeline (stream + buffers
// + graph) holds one submission in flight, so several submissions can overlap.
#include <cooperative_groups.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "mppi.h"
#include "mppi_device.cuh"
#include "mppi_internal.h"
#include "mppi_iter.cuh"

namespace mppi {

// One plan of a submission (device descriptor).
struct __align__(16) BatchInst {
    PlanConst pc;
    SceneLayout L;
    int slot;
    int n_kt;             // k-tiles of the weighted sum
    int simple;           // the parameters allow the specialised rollout step (simple_plan)
    int pad_;
    long long z_off;      // noise offset (pairs)
    long long s_off;      // sample offset (S, w)
    long long scene_off;  // bytes
    long long in_off;     // doubles: x0 | ref | circ | centres
    long long table_off;  // float2
    long long out_off;    // doubles: u [T][2] | x [T+1][4]
    long long du_off;     // doubles: [n_kt][T][2]
};

struct __align__(16) BatchHeader {
    int n;                       // plans in this submission
    int n_tiles;                 // rollout tiles
    unsigned tile_counter;       // next rollout tile (zeroed before the rollout kernel)
    int flags;                   // FLAG_TIMEOUT
    long long noise_total;       // sum over plans of noise_units(K, T)
    long long wsum_total;        // sum over plans of ceil(T / tt_len) * n_kt
    int tt_len;                  // steps per tile of the weighted sum: 8, 4, 2 or 1
    int pad_[3];
};

// Per-plan results written by the batched finalize.
struct __align__(16) OutInfo {
    double s_min, eta;
    int argmin, n_finite, status, pad;
    unsigned long long iter;
};

struct BatchArgs {
    BatchHeader* hdr;
    const BatchInst* inst;
    const long long* noise_prefix;   // [n + 1]
    const long long* wsum_prefix;    // [n + 1]
    const int2* tiles;               // (plan, first sample)
    const double* in;                // inputs arena
    double* out;                     // outputs arena (pinned host memory)
    OutInfo* info;                   // [n] (pinned host memory)
    DevState* slots;
    double* slot_U;                  // [max_slots][max_T][2]
    int max_T;
    unsigned char* scene;
    float2* table;
    void* z;
    double* S;
    float* w;
    double* du;
};

template <typename I>
__device__ __forceinline__ int find_plan(const I* prefix, int n, I q) {
    int lo = 0, hi = n;  // prefix[lo] <= q < prefix[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (prefix[mid] <= q) lo = mid;
        else hi = mid;
    }
    return lo;
}

__device__ __forceinline__ void plan_views(const BatchArgs& a, const BatchInst& d, PlanInputs& in, PlanBuffers& b) {
    const double* x = a.in + d.in_off;
    in.x0 = x;
    in.ref = x + 4;
    in.circ = x + 4 + 2 * d.L.n_ref;
    in.centres = d.pc.has_table ? x + 4 + 2 * d.L.n_ref + 5 * d.L.n_circ : nullptr;
    in.n_ref = d.L.n_ref;
    in.n_circ = d.L.n_circ;
    in.u_out = a.out + d.out_off;
    in.x_out = a.out + d.out_off + 2 * d.pc.T;
    memset(&b, 0, sizeof(b));
    b.state = a.slots + d.slot;
    b.scene = a.scene + d.scene_off;
    b.table = a.table + d.table_off;
    b.S = a.S + d.s_off;
    b.w = a.w + d.s_off;
    b.du_part = a.du + d.du_off;
    b.U = a.slot_U + (size_t)d.slot * a.max_T * 2;
    b.eta_part = &b.state->eta;
    b.n_wblk = 1;
    b.n_kt = d.n_kt;
    b.kt_size = 256 * WS_J;
}

// Preparation and noise of every plan in one launch: prep needs the inputs and noise only the seed
// and the counter, so they run side by side.  The first prep_blocks blocks take the preparation units
// (per plan: shares of its certificates, more of them the fewer plans there are, then one unit per phase
// of prep_scene), the others the noise units of 256 samples x NOISE_PAIRS step pairs: a unit finds its
// plan once, where a search and a 64-bit division per pair made up a third of the time.  256 plans,
// 1.46e8 rollout-steps: prep 248 + noise 1095 us apart, 840 us together; 12 plans: 49 + 47, together 46 us.
constexpr int CERT_SHARES_MIN = 8, CERT_SHARES_MAX = 64;
constexpr int NOISE_PAIRS = 4;

inline __host__ __device__ long long noise_units(int K, int T) {
    return (long long)((K + 255) / 256) * (((T + 1) / 2 + NOISE_PAIRS - 1) / NOISE_PAIRS);
}

template <bool BF16>
__global__ void __launch_bounds__(256, 8) batch_prep_noise_kernel(BatchArgs a, int prep_blocks) {
    const int n = a.hdr->n;
    if ((int)blockIdx.x < prep_blocks) {
        const int shares = min(max(prep_blocks / n - PREP_PHASES, CERT_SHARES_MIN), CERT_SHARES_MAX);
        const int units = shares + PREP_PHASES;
        for (int u = blockIdx.x; u < n * units; u += prep_blocks) {
            const BatchInst& d = a.inst[u / units];
            const int row = u % units;
            PlanInputs in;
            PlanBuffers b;
            plan_views(a, d, in, b);
            if (row < shares)
                prep_cert(d.pc, d.L, in, b, row, shares, min((d.L.n_ref + shares - 1) / shares, CERT_ITEMS));
            else
                prep_scene(d.pc, d.L, in, b, threadIdx.x, blockDim.x, row - shares);
            __syncthreads();
        }
        return;
    }
    __shared__ int pre[1025];
    for (int i = threadIdx.x; i <= n; i += blockDim.x) pre[i] = (int)a.noise_prefix[i];
    __syncthreads();
    using NT = typename NoiseT<BF16>::type;
    const int total = (int)a.hdr->noise_total, stride = gridDim.x - prep_blocks;
    for (int q = blockIdx.x - prep_blocks; q < total; q += stride) {
        const int i = find_plan(pre, n, q);
        const BatchInst& d = a.inst[i];
        const int K = d.pc.K, T = d.pc.T, nkb = (K + 255) / 256;
        const int local = q - pre[i], jb = local / nkb, k = (local - jb * nkb) * 256 + (int)threadIdx.x;
        if (k >= K) continue;
        const uint32_t it = (uint32_t)a.slots[d.slot].iter;
        NT* z = reinterpret_cast<NT*>(a.z) + d.z_off + k;
        const int j1 = min((jb + 1) * NOISE_PAIRS, (T + 1) / 2);
        for (int j = jb * NOISE_PAIRS; j < j1; ++j) {
            const uint4 wv = philox4x32_10(make_uint4((uint32_t)j, (uint32_t)k, it, d.pc.session),
                                           make_uint2(d.pc.key0, d.pc.key1));
            z[(size_t)(2 * j) * K] = make_noise<BF16>(uniform24(wv.x), uniform24(wv.y));
            if (2 * j + 1 < T) z[(size_t)(2 * j + 1) * K] = make_noise<BF16>(uniform24(wv.z), uniform24(wv.w));
        }
    }
}

// G lanes per sample; TIME: they split the steps, else the work of each step (rollout_sample).  A plan
// whose parameters allow it and whose circles are static takes the specialised step, as in the
// single-plan kernel (one lane per sample and the time splits: the shapes in use).
template <int G, bool TIME, bool BF16>
__global__ void __launch_bounds__(BATCH_MAX_THREADS, 2) batch_rollout_kernel(BatchArgs a) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ unsigned long long bar;
    __shared__ PlanConst s_pc;
    __shared__ SceneLayout s_L;
    __shared__ float4 s_x0;
    __shared__ int s_tile, s_plan, s_moving, s_multi, s_jb0, s_simple;
    if (threadIdx.x == 0) {
        bulk_init(&bar);
        s_plan = -1;
    }
    __syncthreads();
    pdl_wait();
    uint32_t phase = 0;
    const int n_tiles = a.hdr->n_tiles;
    using NT = typename NoiseT<BF16>::type;
    for (;;) {
        if (threadIdx.x == 0) s_tile = (int)atomicAdd(&a.hdr->tile_counter, 1u);
        __syncthreads();
        const int tile = s_tile;
        if (tile >= n_tiles) {
            pdl_trigger();
            break;
        }
        const int2 td = a.tiles[tile];
        if (td.x != s_plan) {
            __syncthreads();   // every thread has read s_plan and is done with the previous scene
            if (threadIdx.x == 0) {
                const BatchInst& d = a.inst[td.x];
                s_pc = d.pc;
                s_L = d.L;
                const DevState* st = a.slots + d.slot;
                s_x0 = st->x0f;
                s_moving = st->moving;
                s_simple = d.simple && !st->moving;
                s_multi = st->multi_head;
                s_jb0 = (int)(st->jkey & 0xffffffffu);
                s_plan = td.x;
                bulk_issue(smem, a.scene + d.scene_off, d.L.bytes, &bar);
            }
            __syncthreads();
            if (!__syncthreads_and(bulk_wait(&bar, phase, &a.hdr->flags))) return;
            check_smem(s_L, false);
            phase ^= 1u;
            build_index(s_pc, smem, a.scene + a.inst[td.x].scene_off, s_L, s_multi != 0, (TIME || G == 1) && s_simple);
        }
        const BatchInst& d = a.inst[td.x];
        const int k = td.y + (int)threadIdx.x / G;   // G lanes per sample
        const NT* z = reinterpret_cast<const NT*>(a.z) + d.z_off;
        if ((TIME || G == 1) && s_simple)
            rollout_sample<G, TIME, BF16, false, false, TIME || G == 1>(s_pc, s_L, smem, z, a.table + d.table_off, s_x0,
                                                                        0.0f, false, s_multi != 0, s_jb0, k,
                                                                        a.S + d.s_off, nullptr);
        else
            rollout_sample<G, TIME, BF16, false, false>(s_pc, s_L, smem, z, a.table + d.table_off, s_x0, 0.0f,
                                                        s_moving != 0, s_multi != 0, s_jb0, k, a.S + d.s_off, nullptr);
        __syncthreads();
    }
}

// S_min with its index, the softmin weights and their sum: one cluster of blocks per plan, each block a
// run of samples (the runs depend on K alone, so a plan's sums do not depend on its batch).  As two
// kernels of one block a plan these took 38 + 48 us for 12 plans and 39 + 56 us for 256, waiting on
// loads; 15 and 51 us as one.
constexpr int WEIGHT_BLOCKS = 8;

__global__ void __cluster_dims__(WEIGHT_BLOCKS, 1, 1) __launch_bounds__(256) batch_weights_kernel(BatchArgs a) {
    __shared__ KeyRec s_rec;
    __shared__ double s_sum;
    pdl_wait();
    pdl_trigger();
    const int i = blockIdx.y;
    if (i >= a.hdr->n) return;               // the whole cluster
    cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    const BatchInst& d = a.inst[i];
    DevState* st = a.slots + d.slot;
    const double* S = a.S + d.s_off;
    float* w = a.w + d.s_off;
    const int K = d.pc.K, run = (K + WEIGHT_BLOCKS - 1) / WEIGHT_BLOCKS;
    const int k0 = blockIdx.x * run, k1 = min(K, k0 + run);
    KeyRec r{~0ull, 0x7fffffff, 0};
    for (int k = k0 + threadIdx.x; k < k1; k += blockDim.x) {
        const double s = S[k];
        if (isfinite(s)) r = key_combine(r, KeyRec{order_key(s), k, 1});
    }
    r = block_keymin(r);
    if (threadIdx.x == 0) s_rec = r;
    cl.sync();
    r = KeyRec{~0ull, 0x7fffffff, 0};
    for (int q = 0; q < WEIGHT_BLOCKS; ++q) r = key_combine(r, *cl.map_shared_rank(&s_rec, q));
    const double smin = r.n > 0 ? key_value(r.key) : (double)INFINITY;
    double acc = 0.0;
    for (int k = k0 + threadIdx.x; k < k1; k += blockDim.x) {
        const float wk = softmin_weight(S[k], smin, d.pc.inv_lam_f);
        w[k] = wk;
        acc += widen(wk);
    }
    acc = block_sum_d(acc);
    if (threadIdx.x == 0) s_sum = acc;
    cl.sync();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        acc = 0.0;
        for (int q = 0; q < WEIGHT_BLOCKS; ++q) acc += *cl.map_shared_rank(&s_sum, q);
        st->s_min = smin;
        st->argmin = r.n > 0 ? r.i : -1;
        st->n_finite = r.n;
        st->eta = acc;
    }
    cl.sync();                               // no block leaves while its sum is read
}

// The steps per tile come with the submission (BatchHeader::tt_len): fewer where the batch has too few
// tiles to fill the GPU (one plan: 32 us with 8 steps, now 8).  The sums do not depend on it.  Bound by
// load latency, so by warps in flight: eight blocks per SM (256 plans: 308 us; with 48 registers and
// five blocks per SM 480 us).
template <bool BF16>
__global__ void __launch_bounds__(256, 8) batch_wsum_kernel(BatchArgs a) {
    __shared__ int pre[1025];
    pdl_wait();
    pdl_trigger();
    const int n = a.hdr->n, tt = a.hdr->tt_len;
    for (int i = threadIdx.x; i <= n; i += blockDim.x) pre[i] = (int)a.wsum_prefix[i];
    __syncthreads();
    using NT = typename NoiseT<BF16>::type;
    for (int q = blockIdx.x; q < (int)a.hdr->wsum_total; q += gridDim.x) {
        const int i = find_plan(pre, n, q);
        const BatchInst& d = a.inst[i];
        const int local = q - pre[i];
        const int ti = local / d.n_kt, kt = local - ti * d.n_kt;
        const float4* ctl = reinterpret_cast<const float4*>(a.scene + d.scene_off + d.L.off_ctl);
        wsum_tile<BF16>(d.pc, ctl, reinterpret_cast<const NT*>(a.z) + d.z_off, a.w + d.s_off, kt, ti * tt, 256 * WS_J,
                        a.du + d.du_off, nullptr, 0, tt);
    }
}

__global__ void __launch_bounds__(1024) batch_finalize_kernel(BatchArgs a) {
    pdl_wait();
    const int i = blockIdx.x;
    if (i >= a.hdr->n) return;
    const BatchInst& d = a.inst[i];
    PlanInputs in;
    PlanBuffers b;
    plan_views(a, d, in, b);
    if (threadIdx.x == 0 && (a.hdr->flags & FLAG_TIMEOUT)) atomicOr(&b.state->flags, FLAG_TIMEOUT);
    __syncthreads();
    finalize_block(d.pc, b, in);
    __syncthreads();
    if (threadIdx.x == 0) {
        const DevState* st = b.state;
        OutInfo o;
        o.s_min = st->s_min;
        o.eta = st->eta;
        o.argmin = st->argmin;
        o.n_finite = st->n_finite;
        o.status = st->status;
        o.pad = 0;
        o.iter = st->iter_used;
        a.info[i] = o;
    }
}

template <int G, bool TIME, bool BF16>
static cudaError_t set_rollout_smem(size_t smem) {
    return cudaFuncSetAttribute(batch_rollout_kernel<G, TIME, BF16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(smem < 48 * 1024 ? 48 * 1024 : smem));
}

template <int G, bool TIME, bool BF16>
static int batch_blocks_per_sm(int threads, size_t smem) {
    int n = 0;
    if (set_rollout_smem<G, TIME, BF16>(smem) != cudaSuccess) return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, batch_rollout_kernel<G, TIME, BF16>, threads, smem) !=
        cudaSuccess)
        return 0;
    return n;
}

// Lanes per sample as the group value: g > 0 split the work of each step, g < 0 split the steps.
#define MPPI_BATCH_GROUPS(X) X(1, 1, false) X(2, 2, false) X(4, 4, false) X(8, 8, false) X(16, 16, false) \
    X(32, 32, false) X(-2, 2, true) X(-4, 4, true) X(-8, 8, true) X(-16, 16, true)

// The shared-memory attribute must already be set (batch_max_blocks does it), so this
// only launches and may be captured into a graph.
template <bool BF16>
static cudaError_t launch_batch_rollout_b(const BatchArgs& a, int G, int threads, int blocks, size_t smem,
                                          cudaStream_t st) {
    switch (G) {
#define CASE(gv, g, time)                                                            \
    case gv: {                                                                       \
        return launch_chained(batch_rollout_kernel<g, time, BF16>, dim3(blocks), dim3(threads), smem, st, a); \
    }
        MPPI_BATCH_GROUPS(CASE)
#undef CASE
        default: return cudaErrorInvalidValue;
    }
}

static int batch_max_blocks(int G, int bf16, int threads, size_t smem) {
    switch (G) {
#define CASE(gv, g, time)                                                                                    \
    case gv: return bf16 ? batch_blocks_per_sm<g, time, true>(threads, smem) : batch_blocks_per_sm<g, time, false>(threads, smem);
        MPPI_BATCH_GROUPS(CASE)
#undef CASE
        default: return 0;
    }
}

static int lanes_of(int G) { return G < 0 ? -G : G; }

// Debug build: the index violations this translation unit's kernels counted (then reset).
cudaError_t take_check_hits_batch(unsigned long long* hits) {
#ifdef MPPI_CHECKS
    cudaError_t e = cudaMemcpyFromSymbol(hits, g_check_hits, sizeof(unsigned long long));
    const unsigned long long zero = 0;
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_check_hits, &zero, sizeof(zero));
    return e;
#else
    *hits = 0;
    return cudaSuccess;
#endif
}

}  // namespace mppi

using namespace mppi;

namespace {

constexpr int ALIGN = 256;
size_t up(size_t x) { return (x + ALIGN - 1) / ALIGN * ALIGN; }

struct Pipeline {
    cudaStream_t stream = nullptr;
    cudaEvent_t done = nullptr;
    // the kernel sequence, captured once per rollout launch shape (a few: the launch rule has five)
    struct Graph {
        cudaGraphExec_t exec;
        int G, threads;
    };
    std::vector<Graph> graphs;
    // device buffers
    unsigned char* d_stage = nullptr;   // header | inst | prefixes | tiles | inputs
    unsigned char* scene = nullptr;
    float2* table = nullptr;
    void* z = nullptr;
    double* S = nullptr;
    float* w = nullptr;
    double* du = nullptr;
    // host staging
    unsigned char* h_stage = nullptr;
    unsigned char* h_out = nullptr;
    size_t stage_used = 0;
    std::vector<mppi_request*> pending;
    std::vector<long long> out_offsets;
    std::vector<long long> s_offsets;   // per plan of the last submission: offset of its costs in S
    std::vector<int> s_counts;          // and its K (kept after the wait for mppi_batch_get_costs)
    bool busy = false;
    BatchArgs args{};
};

}  // namespace

struct mppi_batch {
    int device = 0;
    int max_slots = 0, max_batch = 0, max_T = 0, max_ref = 0, max_circ = 0, noise_bf16 = 0;
    long long max_samples = 0, max_steps = 0, max_tiles = 0;
    size_t max_scene = 0, rollout_smem = 0, max_in = 0, max_out = 0, stage_bytes = 0, out_bytes = 0;
    // offsets inside the staging buffer
    size_t off_inst = 0, off_npre = 0, off_wpre = 0, off_tiles = 0, off_in = 0;
    DevState* slots = nullptr;
    double* slot_U = nullptr;
    int G = 0, threads = 0, n_sm = 0;   // launch shape of the rollout for the submission at hand
    // where it comes from: the launch rule, mppi_batch_set_launch, or mppi_batch_autotune on a
    // submission of tuned_samples samples
    enum { SHAPE_RULE, SHAPE_SET, SHAPE_TUNED } shape = SHAPE_RULE;
    int set_G = 0, set_threads = 0;
    long long tuned_samples = 0;
    std::vector<Pipeline> pipes;
    std::string err;
    std::mutex mu;
};

static thread_local std::string g_batch_err;

static int bfail(mppi_batch* b, int status, const std::string& msg) {
    if (b) b->err = msg;
    g_batch_err = msg;
    return status;
}

#define BCK(call, what)                                                                           \
    do {                                                                                          \
        cudaError_t e_ = (call);                                                                  \
        if (e_ != cudaSuccess) return bfail(B, MPPI_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e_)); \
    } while (0)

// the single-plan path's parameter conversion, validation and sizes
namespace mppi {
int check_params_shared(const mppi_params* p, std::string& why);
PlanConst make_const_shared(const mppi_params& p);
}  // namespace mppi

static void free_pipe(Pipeline& p) {
    void* dev[] = {p.d_stage, p.scene, p.table, p.z, p.S, p.w, p.du};
    for (void* q : dev)
        if (q) cudaFree(q);
    if (p.h_stage) cudaFreeHost(p.h_stage);
    if (p.h_out) cudaFreeHost(p.h_out);
    for (auto& g : p.graphs) cudaGraphExecDestroy(g.exec);
    if (p.done) cudaEventDestroy(p.done);
    if (p.stream) cudaStreamDestroy(p.stream);
}

static void free_batch(mppi_batch* B) {
    for (auto& p : B->pipes) free_pipe(p);
    if (B->slots) cudaFree(B->slots);
    if (B->slot_U) cudaFree(B->slot_U);
}

static size_t out_elems(int T) { return 2 * (size_t)T + 4 * (size_t)(T + 1); }

extern "C" {

int mppi_batch_create(int32_t max_slots, int32_t max_batch, int64_t max_samples, int64_t max_rollout_steps,
                      int32_t max_T, int32_t max_ref, int32_t max_circ, int32_t noise_bf16, int32_t pipelines,
                      int device, mppi_batch** out) {
    if (!out) return bfail(nullptr, MPPI_ERR_ARG, "out is NULL");
    *out = nullptr;
    if (max_slots < 1 || max_batch < 1 || max_batch > 1024 || max_samples < 1 || max_rollout_steps < 1 ||
        max_T < 1 || max_T > MPPI_MAX_T || max_ref < 2 || max_ref > MPPI_MAX_REF || max_circ < 0 ||
        max_circ > MPPI_MAX_CIRC || pipelines < 1 || pipelines > 16)
        return bfail(nullptr, MPPI_ERR_ARG, "batch capacities out of range");
    mppi_batch* B = new (std::nothrow) mppi_batch();
    if (!B) return bfail(nullptr, MPPI_ERR_OOM, "host allocation failed");
    B->device = device;
    B->max_slots = max_slots;
    B->max_batch = max_batch;
    B->max_T = max_T;
    B->max_ref = max_ref;
    B->max_circ = max_circ;
    B->noise_bf16 = noise_bf16 ? 1 : 0;
    B->max_samples = max_samples;
    B->max_steps = max_rollout_steps;
    B->max_tiles = max_samples / 16 + max_batch;
    const SceneLayout Lmax = make_layout(max_T, max_ref, max_circ);
    B->max_scene = up((size_t)Lmax.total);
    B->rollout_smem = up(rollout_smem_bytes(Lmax, BATCH_MAX_THREADS, false));   // blob and the boxes built after it
    B->max_in = 4 + 2 * (size_t)max_ref + 5 * (size_t)max_circ + 2 * (size_t)max_T * max_circ;
    B->max_out = out_elems(max_T);
    auto bail = [&](int st) {
        free_batch(B);
        delete B;
        return st;
    };
    cudaError_t e = cudaSetDevice(device);
    if (e != cudaSuccess) return bail(bfail(nullptr, MPPI_ERR_CUDA, std::string("cudaSetDevice: ") + cudaGetErrorString(e)));
    cudaDeviceGetAttribute(&B->n_sm, cudaDevAttrMultiProcessorCount, device);
    int max_smem = 0;
    cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
    if (B->rollout_smem + 1024 > (size_t)max_smem)
        return bail(bfail(nullptr, MPPI_ERR_CAPACITY, "scene of max_T, max_ref, max_circ exceeds shared memory"));
    // staging layout
    size_t o = up(sizeof(BatchHeader));
    B->off_inst = o;  o += up(sizeof(BatchInst) * (size_t)max_batch);
    B->off_npre = o;  o += up(sizeof(long long) * ((size_t)max_batch + 1));
    B->off_wpre = o;  o += up(sizeof(long long) * ((size_t)max_batch + 1));
    B->off_tiles = o; o += up(sizeof(int2) * (size_t)B->max_tiles);
    B->off_in = o;    o += up(sizeof(double) * B->max_in * (size_t)max_batch);
    B->stage_bytes = o;
    B->out_bytes = up(sizeof(double) * B->max_out * (size_t)max_batch) + up(sizeof(OutInfo) * (size_t)max_batch);
    if (cudaMalloc(&B->slots, sizeof(DevState) * (size_t)max_slots) != cudaSuccess ||
        cudaMalloc(&B->slot_U, sizeof(double) * 2 * (size_t)max_T * max_slots) != cudaSuccess)
        return bail(bfail(nullptr, MPPI_ERR_OOM, "slot allocation failed"));
    std::vector<DevState> s0((size_t)max_slots);
    memset(s0.data(), 0, sizeof(DevState) * s0.size());
    for (auto& s : s0) s.jkey = ~0ull;
    if (cudaMemcpy(B->slots, s0.data(), sizeof(DevState) * s0.size(), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(B->slot_U, 0, sizeof(double) * 2 * (size_t)max_T * max_slots) != cudaSuccess)
        return bail(bfail(nullptr, MPPI_ERR_CUDA, "slot initialisation failed"));
    const long long max_kt_tiles = max_samples / (256 * WS_J) + max_batch;
    B->pipes.resize((size_t)pipelines);
    for (auto& p : B->pipes) {
        const size_t zb = (size_t)max_rollout_steps * (B->noise_bf16 ? 4 : 8);
        bool ok = cudaStreamCreateWithFlags(&p.stream, cudaStreamNonBlocking) == cudaSuccess &&
                  cudaEventCreateWithFlags(&p.done, cudaEventDisableTiming) == cudaSuccess &&
                  cudaMalloc(&p.d_stage, B->stage_bytes) == cudaSuccess &&
                  cudaMalloc(&p.scene, B->max_scene * (size_t)max_batch) == cudaSuccess &&
                  cudaMalloc(&p.table, sizeof(float2) * (size_t)max_T * std::max(max_circ, 1) * max_batch) ==
                      cudaSuccess &&
                  cudaMalloc(&p.z, zb) == cudaSuccess && cudaMalloc(&p.S, sizeof(double) * max_samples) == cudaSuccess &&
                  cudaMalloc(&p.w, sizeof(float) * max_samples) == cudaSuccess &&
                  cudaMalloc(&p.du, sizeof(double) * 2 * (size_t)max_T * max_kt_tiles) == cudaSuccess &&
                  cudaMallocHost(&p.h_stage, B->stage_bytes) == cudaSuccess &&
                  cudaMallocHost(&p.h_out, B->out_bytes) == cudaSuccess;
        if (!ok) {
            cudaGetLastError();
            return bail(bfail(nullptr, MPPI_ERR_OOM, "pipeline allocation failed"));
        }
        BatchArgs& a = p.args;
        a.hdr = reinterpret_cast<BatchHeader*>(p.d_stage);
        a.inst = reinterpret_cast<const BatchInst*>(p.d_stage + B->off_inst);
        a.noise_prefix = reinterpret_cast<const long long*>(p.d_stage + B->off_npre);
        a.wsum_prefix = reinterpret_cast<const long long*>(p.d_stage + B->off_wpre);
        a.tiles = reinterpret_cast<const int2*>(p.d_stage + B->off_tiles);
        a.in = reinterpret_cast<const double*>(p.d_stage + B->off_in);
        // finalize writes u*, x* and the records into the pinned output buffer: nothing is copied back
        unsigned char* h_out_dev = nullptr;
        if (cudaHostGetDevicePointer(&h_out_dev, p.h_out, 0) != cudaSuccess) {
            cudaGetLastError();
            return bail(bfail(nullptr, MPPI_ERR_CUDA, "pinned host buffers are not mapped for the device"));
        }
        a.out = reinterpret_cast<double*>(h_out_dev);
        a.info = reinterpret_cast<OutInfo*>(h_out_dev + up(sizeof(double) * B->max_out * (size_t)max_batch));
        a.slots = B->slots;
        a.slot_U = B->slot_U;
        a.max_T = max_T;
        a.scene = p.scene;
        a.table = p.table;
        a.z = p.z;
        a.S = p.S;
        a.w = p.w;
        a.du = p.du;
    }
    *out = B;
    return MPPI_OK;
}

int mppi_batch_destroy(mppi_batch* B) {
    if (!B) return MPPI_OK;
    cudaSetDevice(B->device);
    for (auto& p : B->pipes)
        if (p.stream) cudaStreamSynchronize(p.stream);
    free_batch(B);
    delete B;
    return MPPI_OK;
}

}  // extern "C"

// Builds the staging image of a submission in p.h_stage; returns the status.
static void choose_shape(mppi_batch* B, long long samples);

static int build_submission(mppi_batch* B, Pipeline& p, mppi_request* req, int n, bool choose = false) {
    if (n < 1 || n > B->max_batch) return bfail(B, MPPI_ERR_CAPACITY, "number of plans outside [1, max_batch]");
    std::vector<char> used((size_t)B->max_slots, 0);
    BatchHeader* H = reinterpret_cast<BatchHeader*>(p.h_stage);
    BatchInst* I = reinterpret_cast<BatchInst*>(p.h_stage + B->off_inst);
    long long* npre = reinterpret_cast<long long*>(p.h_stage + B->off_npre);
    long long* wpre = reinterpret_cast<long long*>(p.h_stage + B->off_wpre);
    int2* tiles = reinterpret_cast<int2*>(p.h_stage + B->off_tiles);
    double* inp = reinterpret_cast<double*>(p.h_stage + B->off_in);
    long long z_off = 0, s_off = 0, in_off = 0, table_off = 0, out_off = 0, du_off = 0, scene_off = 0;
    long long noise = 0, wsum = 0, n_tiles = 0;
    p.out_offsets.assign((size_t)n, 0);
    p.s_offsets.assign((size_t)n, 0);
    p.s_counts.assign((size_t)n, 0);
    std::vector<std::pair<double, int>> cost((size_t)n);
    for (int i = 0; i < n; ++i) {
        mppi_request& r = req[i];
        std::string why;
        if (!r.params || check_params_shared(r.params, why) != MPPI_OK)
            return bfail(B, MPPI_ERR_ARG, "plan " + std::to_string(i) + ": " + (r.params ? why : "params NULL"));
        const mppi_params& pr = *r.params;
        if (pr.model != 0 || pr.cost_to_go != 0)
            return bfail(B, MPPI_ERR_ARG, "the batch engine runs model 0 with whole-cost weights");
        if (pr.noise_bf16 != B->noise_bf16) return bfail(B, MPPI_ERR_ARG, "noise precision differs from the batch's");
        if (r.slot < 0 || r.slot >= B->max_slots || used[(size_t)r.slot])
            return bfail(B, MPPI_ERR_ARG, "slot out of range or used twice in one submission");
        used[(size_t)r.slot] = 1;
        if (!r.x0 || !r.ref_xy || !r.u_out || !r.x_out || (r.n_circ > 0 && !r.circ) || r.n_ref < 2 || r.n_circ < 0)
            return bfail(B, MPPI_ERR_ARG, "plan " + std::to_string(i) + ": bad arrays");
        if (pr.T > B->max_T || r.n_ref > B->max_ref || r.n_circ > B->max_circ)
            return bfail(B, MPPI_ERR_CAPACITY, "plan " + std::to_string(i) + ": size above the batch capacity");
        const int T = pr.T, K = pr.K;
        const size_t nr = 2 * (size_t)r.n_ref, nc = 5 * (size_t)r.n_circ, nt = r.centres ? 2 * (size_t)T * r.n_circ : 0;
        if (!finite_all(r.x0, 4) || !finite_all(r.ref_xy, nr) || (nc && !finite_all((const double*)r.circ, nc)) ||
            (nt && !finite_all(r.centres, nt)))
            return bfail(B, MPPI_ERR_ARG, "plan " + std::to_string(i) + ": non-finite input");
        BatchInst& d = I[i];
        memset(&d, 0, sizeof(d));
        d.pc = make_const_shared(pr);
        d.pc.has_table = nt ? 1 : 0;
        d.L = make_layout(T, r.n_ref, r.n_circ);
        d.slot = r.slot;
        d.n_kt = (K + 256 * WS_J - 1) / (256 * WS_J);
        d.simple = simple_plan(d.pc) ? 1 : 0;
        d.z_off = z_off;
        d.s_off = s_off;
        d.scene_off = scene_off;
        d.in_off = in_off;
        d.table_off = table_off;
        d.out_off = out_off;
        d.du_off = du_off;
        double* x = inp + in_off;
        memcpy(x, r.x0, 4 * sizeof(double));
        memcpy(x + 4, r.ref_xy, nr * sizeof(double));
        if (nc) memcpy(x + 4 + nr, r.circ, nc * sizeof(double));
        if (nt) memcpy(x + 4 + nr + nc, r.centres, nt * sizeof(double));
        npre[i] = noise;
        noise += noise_units(K, T);
        p.out_offsets[(size_t)i] = out_off;
        p.s_offsets[(size_t)i] = s_off;
        p.s_counts[(size_t)i] = K;
        z_off += (long long)K * T;
        s_off += K;
        scene_off += (long long)up((size_t)d.L.total);
        in_off += (long long)(4 + nr + nc + nt);
        table_off += (long long)T * std::max(r.n_circ, 1);
        out_off += (long long)out_elems(T);
        du_off += 2LL * T * d.n_kt;
        cost[(size_t)i] = {(double)T * (700.0 + 20.0 * r.n_circ + 2.0 * r.n_ref / 16.0), i};
    }
    if (s_off > B->max_samples || z_off > B->max_steps || noise > 0x7fffffffLL)
        return bfail(B, MPPI_ERR_CAPACITY, "submission above the batch's sample or rollout-step capacity");
    npre[n] = noise;
    // steps per tile of the weighted sum: the longest of 8, 4, 2, 1 that still gives six tiles per SM
    int tt = WS_TT;
    for (;; tt /= 2) {
        wsum = 0;
        for (int i = 0; i < n; ++i) {
            wpre[i] = wsum;
            wsum += (long long)((I[i].pc.T + tt - 1) / tt) * I[i].n_kt;
        }
        wpre[n] = wsum;
        if (tt == 1 || wsum >= 6LL * B->n_sm) break;
    }
    // rollout tiles, most expensive plans first
    if (choose) choose_shape(B, s_off);
    const int spt = B->threads / lanes_of(B->G);   // samples per rollout tile
    std::stable_sort(cost.begin(), cost.end(), [](const auto& a, const auto& b) { return a.first > b.first; });
    for (auto& c : cost) {
        const int i = c.second;
        for (int k0 = 0; k0 < I[i].pc.K; k0 += spt) {
            if (n_tiles >= B->max_tiles) return bfail(B, MPPI_ERR_CAPACITY, "too many rollout tiles");
            tiles[n_tiles++] = make_int2(i, k0);
        }
    }
    memset(H, 0, sizeof(*H));
    H->n = n;
    H->n_tiles = (int)n_tiles;
    H->noise_total = noise;
    H->wsum_total = wsum;
    H->tt_len = tt;
    // the staged region is contiguous up to the end of the used inputs
    p.stage_used = B->off_in + sizeof(double) * (size_t)in_off;
    return MPPI_OK;
}

static cudaError_t launch_batch_prep_noise(mppi_batch* B, Pipeline& p) {
    const int prep = B->n_sm * 4, grid = prep + B->n_sm * 8;
    if (B->noise_bf16) batch_prep_noise_kernel<true><<<grid, 256, 0, p.stream>>>(p.args, prep);
    else batch_prep_noise_kernel<false><<<grid, 256, 0, p.stream>>>(p.args, prep);
    return cudaGetLastError();
}

static cudaError_t enqueue_kernels(mppi_batch* B, Pipeline& p, int per_sm) {
    const BatchArgs& a = p.args;
    const cudaStream_t st = p.stream;
    cudaError_t e;
    const int grid = B->n_sm * 8;
    if ((e = launch_batch_prep_noise(B, p)) != cudaSuccess) return e;
    // (the tile counter starts at zero: the submission's header is copied before every launch)
    const size_t smem = B->rollout_smem;
    if (B->noise_bf16) e = launch_batch_rollout_b<true>(a, B->G, B->threads, B->n_sm * per_sm, smem, st);
    else e = launch_batch_rollout_b<false>(a, B->G, B->threads, B->n_sm * per_sm, smem, st);
    if (e != cudaSuccess) return e;
    if ((e = launch_chained(batch_weights_kernel, dim3(WEIGHT_BLOCKS, B->max_batch), dim3(256), 0, st, a)) != cudaSuccess)
        return e;
    e = B->noise_bf16 ? launch_chained(batch_wsum_kernel<true>, dim3(grid), dim3(256), 0, st, a)
                      : launch_chained(batch_wsum_kernel<false>, dim3(grid), dim3(256), 0, st, a);
    if (e != cudaSuccess) return e;
    // one thread per step of the longest plan
    return launch_chained(batch_finalize_kernel, dim3(B->max_batch), dim3((B->max_T + 31) / 32 * 32), 0, st, a);
}

// The launch shape of a submission of `samples` samples.  A shape set by hand holds always, a tuned one
// for submissions within a factor of two of the one it was tuned on (a server's micro-batches range
// from one plan to all of them).  Otherwise the lanes of a sample split its steps as far as the
// submission stays within LANES_PER_SM lanes: measured on mixes of 1 to 256 plans, the widest such split
// was the fastest or within 3 % of it (1 plan of 8192 samples: 8 lanes 102 us, one lane 163; 16 plans,
// 98,304 samples: 2 lanes 389 us, 4 lanes 440; 31 plans, 189,440 samples: one lane 515 us, 8 lanes 717).
// Blocks of 448 threads from four tiles a block on (256 plans: 4.15 ms against 4.25 with 256), 256 below
// (finer tiles balance uneven plans: 12 plans 310 us against 318).
constexpr int LANES_PER_SM = 1300;

struct Shape {
    int G, threads;
};

static Shape rule_shape(const mppi_batch* B, long long samples) {
    int lanes = 1;
    while (lanes < 16 && samples * lanes * 2 <= (long long)B->n_sm * LANES_PER_SM) lanes *= 2;
    const bool full = samples * lanes >= 4LL * 2 * B->n_sm * BATCH_MAX_THREADS;
    return {lanes > 1 ? -lanes : 1, full ? BATCH_MAX_THREADS : 256};
}

static void choose_shape(mppi_batch* B, long long samples) {
    const bool tuned = B->shape == mppi_batch::SHAPE_TUNED && samples <= 2 * B->tuned_samples &&
                       2 * samples >= B->tuned_samples;
    const Shape s = B->shape == mppi_batch::SHAPE_SET || tuned ? Shape{B->set_G, B->set_threads} : rule_shape(B, samples);
    B->G = s.G;
    B->threads = s.threads;
}

// The kernel sequence of a pipeline for the launch shape at hand, captured when it is first needed.
static cudaError_t ensure_graph(mppi_batch* B, Pipeline& p, cudaGraphExec_t* exec) {
    for (auto& g : p.graphs)
        if (g.G == B->G && g.threads == B->threads) {
            *exec = g.exec;
            return cudaSuccess;
        }
    // configure function attributes outside the capture
    const int per_sm = batch_max_blocks(B->G, B->noise_bf16, B->threads, B->rollout_smem);
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamBeginCapture(p.stream, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return e;
    cudaError_t ek = enqueue_kernels(B, p, per_sm);
    e = cudaStreamEndCapture(p.stream, &g);
    if (ek != cudaSuccess) {
        if (g) cudaGraphDestroy(g);
        return ek;
    }
    if (e != cudaSuccess) return e;
    e = cudaGraphInstantiate(exec, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) return e;
    p.graphs.push_back({*exec, B->G, B->threads});
    return cudaSuccess;
}

extern "C" {

int mppi_batch_submit(mppi_batch* B, mppi_request* req, int32_t n, int32_t* ticket) {
    if (!B || !req || !ticket) return bfail(B, MPPI_ERR_ARG, "NULL argument");
    std::lock_guard<std::mutex> lock(B->mu);
    BCK(cudaSetDevice(B->device), "cudaSetDevice");
    int pi = -1;
    for (size_t i = 0; i < B->pipes.size(); ++i)
        if (!B->pipes[i].busy) {
            pi = (int)i;
            break;
        }
    if (pi < 0) return bfail(B, MPPI_ERR_CAPACITY, "every pipeline has a submission in flight");
    Pipeline& p = B->pipes[(size_t)pi];
    int rc = build_submission(B, p, req, n, true);
    if (rc != MPPI_OK) return rc;
    cudaGraphExec_t graph = nullptr;
    BCK(ensure_graph(B, p, &graph), "graph capture");
    BCK(cudaMemcpyAsync(p.d_stage, p.h_stage, p.stage_used, cudaMemcpyHostToDevice, p.stream), "input copy");
    BCK(cudaGraphLaunch(graph, p.stream), "graph launch");
    BCK(cudaEventRecord(p.done, p.stream), "event record");
    p.pending.assign((size_t)n, nullptr);
    for (int i = 0; i < n; ++i) p.pending[(size_t)i] = &req[i];
    p.busy = true;
    *ticket = pi;
    return MPPI_OK;
}

int mppi_batch_wait(mppi_batch* B, int32_t ticket) {
    if (!B || ticket < 0 || ticket >= (int)B->pipes.size()) return bfail(B, MPPI_ERR_ARG, "bad ticket");
    Pipeline& p = B->pipes[(size_t)ticket];
    if (!p.busy) return bfail(B, MPPI_ERR_ARG, "ticket has no submission in flight");
    BCK(cudaSetDevice(B->device), "cudaSetDevice");
    cudaError_t e = cudaEventSynchronize(p.done);
    std::lock_guard<std::mutex> lock(B->mu);
    p.busy = false;
    if (e != cudaSuccess) return bfail(B, MPPI_ERR_CUDA, std::string("batch: ") + cudaGetErrorString(e));
    const OutInfo* info = reinterpret_cast<const OutInfo*>(p.h_out + up(sizeof(double) * B->max_out * (size_t)B->max_batch));
    const double* outs = reinterpret_cast<const double*>(p.h_out);
    int worst = MPPI_OK;
    for (size_t i = 0; i < p.pending.size(); ++i) {
        mppi_request& r = *p.pending[i];
        const OutInfo& o = info[i];
        r.status = o.status;
        if (o.status == MPPI_OK) {
            const int T = r.params->T;
            memcpy(r.u_out, outs + p.out_offsets[i], 2 * (size_t)T * sizeof(double));
            memcpy(r.x_out, outs + p.out_offsets[i] + 2 * T, 4 * (size_t)(T + 1) * sizeof(double));
        } else if (worst == MPPI_OK) {
            worst = o.status;
        }
        if (r.info) {
            r.info->argmin = o.argmin;
            r.info->n_finite = o.n_finite;
            r.info->s_min = o.s_min;
            r.info->eta = o.eta;
            r.info->iter = o.iter;
        }
    }
    p.pending.clear();
    if (worst != MPPI_OK) return bfail(B, worst, "some plans of the submission failed (see their status)");
    return MPPI_OK;
}

}  // extern "C"

// 1 when the submission on the ticket's pipeline has finished on the device, 0 while it runs,
// MPPI_ERR_* on a bad ticket or a failed query (the server's watchdog polls it).
int batch_ticket_done(mppi_batch* B, int32_t ticket) {
    if (!B || ticket < 0 || ticket >= (int)B->pipes.size()) return MPPI_ERR_ARG;
    Pipeline& p = B->pipes[(size_t)ticket];
    if (!p.busy) return MPPI_ERR_ARG;
    if (cudaSetDevice(B->device) != cudaSuccess) return MPPI_ERR_CUDA;
    const cudaError_t e = cudaEventQuery(p.done);
    if (e == cudaSuccess) return 1;
    if (e == cudaErrorNotReady) return 0;
    return MPPI_ERR_CUDA;
}

extern "C" {

int mppi_batch_plan(mppi_batch* B, mppi_request* req, int32_t n) {
    int32_t t = -1;
    int rc = mppi_batch_submit(B, req, n, &t);
    if (rc != MPPI_OK) return rc;
    return mppi_batch_wait(B, t);
}

int mppi_batch_autotune(mppi_batch* B, mppi_request* req, int32_t n, int32_t* group, int32_t* block) {
    if (!B || !req) return bfail(B, MPPI_ERR_ARG, "NULL argument");
    BCK(cudaSetDevice(B->device), "cudaSetDevice");
    Pipeline& p = B->pipes[0];
    if (p.busy) return bfail(B, MPPI_ERR_CAPACITY, "pipeline 0 has a submission in flight");
    // the shapes a caller can set, at least 16 samples per tile, then the rule's own for this submission
    // (16 lanes splitting the steps, up to some 12,000 samples, is only the rule's): the fastest of all is
    // kept, the fastest that mppi_batch_set_launch takes is reported
    std::vector<Shape> shapes;
    for (int g : {1, 2, 4, 8, 16, 32, -2, -4, -8})
        for (int th : {64, 128, 256, BATCH_MAX_THREADS})
            if (th / lanes_of(g) >= 16) shapes.push_back({g, th});
    const size_t n_set = shapes.size();
    float best = INFINITY, best_set = INFINITY;
    Shape kept{0, 0}, reported{0, 0};
    cudaEvent_t e0, e1;
    BCK(cudaEventCreate(&e0), "cudaEventCreate");
    BCK(cudaEventCreate(&e1), "cudaEventCreate");
    int rc = MPPI_OK;
    // (the passes change neither the warm starts nor the counters of the slots)
    B->G = 4;
    B->threads = 128;
    rc = build_submission(B, p, req, n);     // refuses what a submission refuses
    cudaError_t e = cudaSuccess;
    long long samples = 0;
    for (int i = 0; i < n && rc == MPPI_OK; ++i) samples += req[i].params->K;
    shapes.push_back(rule_shape(B, samples));
    if (shapes.back().G != -16) shapes.pop_back();     // timed among the others
    // The preparation and the rollout chained to it, as a submission runs them: by itself the rollout of a
    // few tiles can be faster in a shape that is slower there (2048 x 150, 8 lanes in blocks of 128: 44 to 69
    // us alone, and the submission 115 us against 93 with the rule's 57 us).  ms: the mean of the passes.
    const auto time_shape = [&](const Shape& sh, int passes, float& ms) -> cudaError_t {
        ms = INFINITY;
        const int per_sm = batch_max_blocks(sh.G, B->noise_bf16, sh.threads, B->rollout_smem);
        if (per_sm < 1) return cudaSuccess;
        B->G = sh.G;
        B->threads = sh.threads;
        rc = build_submission(B, p, req, n);           // tiles depend on samples per tile
        if (rc != MPPI_OK) return cudaSuccess;
        cudaError_t err = cudaMemcpyAsync(p.d_stage, p.h_stage, p.stage_used, cudaMemcpyHostToDevice, p.stream);
        float sum = 0.0f;
        for (int r = 0; r < passes && err == cudaSuccess; ++r) {
            float once = 0.0f;
            if (err == cudaSuccess) err = cudaMemsetAsync(&p.args.hdr->tile_counter, 0, sizeof(unsigned), p.stream);
            if (err == cudaSuccess) err = cudaEventRecord(e0, p.stream);
            if (err == cudaSuccess) err = launch_batch_prep_noise(B, p);
            if (err == cudaSuccess)
                err = B->noise_bf16
                          ? launch_batch_rollout_b<true>(p.args, sh.G, sh.threads, B->n_sm * per_sm, B->rollout_smem, p.stream)
                          : launch_batch_rollout_b<false>(p.args, sh.G, sh.threads, B->n_sm * per_sm, B->rollout_smem, p.stream);
            if (err == cudaSuccess) err = cudaEventRecord(e1, p.stream);
            if (err == cudaSuccess) err = cudaEventSynchronize(e1);
            if (err == cudaSuccess) err = cudaEventElapsedTime(&once, e0, e1);
            sum += once;
        }
        if (err == cudaSuccess) ms = sum / (float)passes;
        return err;
    };
    // one pass of each shape, then more of those within a third of the best: six where they are short (and
    // scatter by a tenth), else four
    std::vector<float> took(shapes.size(), INFINITY);
    float first = INFINITY;
    for (size_t i = 0; i < shapes.size() && rc == MPPI_OK && e == cudaSuccess; ++i) {
        e = time_shape(shapes[i], 1, took[i]);
        first = std::min(first, took[i]);
    }
    const float limit = 1.35f * first;
    for (size_t i = 0; i < shapes.size() && rc == MPPI_OK && e == cudaSuccess; ++i)
        if (took[i] <= limit) e = time_shape(shapes[i], first < 0.3f ? 6 : 4, took[i]);
    for (size_t i = 0; i < shapes.size(); ++i) {
        if (took[i] < best) {
            best = took[i];
            kept = shapes[i];
        }
        if (i < n_set && took[i] < best_set) {
            best_set = took[i];
            reported = shapes[i];
        }
    }
    // leave the slots as they were: the preparation only accumulated the per-iteration fields
    for (int i = 0; i < n && rc == MPPI_OK && e == cudaSuccess; ++i) e = launch_reset_state(B->slots + req[i].slot, p.stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(p.stream);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (rc != MPPI_OK) return rc;
    if (e == cudaSuccess && reported.G == 0) e = cudaErrorInvalidConfiguration;
    if (e != cudaSuccess) return bfail(B, MPPI_ERR_CUDA, std::string("batch autotune: ") + cudaGetErrorString(e));
    B->shape = mppi_batch::SHAPE_TUNED;
    B->set_G = kept.G;
    B->set_threads = kept.threads;
    B->tuned_samples = samples;
    if (group) *group = reported.G;
    if (block) *block = reported.threads;
    return MPPI_OK;
}

int mppi_batch_set_launch(mppi_batch* B, int32_t group, int32_t block) {
    if (!B) return bfail(B, MPPI_ERR_ARG, "NULL argument");
    bool known = false;
#define CASE(gv, g, time) known |= group == gv;
    MPPI_BATCH_GROUPS(CASE)
#undef CASE
    known = known && group != -16;      // the launch rule's own (choose_shape)
    if (!known || block < 32 || block > BATCH_MAX_THREADS || block % 32 != 0 || block / lanes_of(group) < 16)
        return bfail(B, MPPI_ERR_ARG, "group must be 1..32 or -2, -4, -8; block a multiple of 32 up to 448 with "
                                      "at least 16 samples per block");
    for (auto& p : B->pipes)
        if (p.busy) return bfail(B, MPPI_ERR_CAPACITY, "a submission is in flight");
    BCK(cudaSetDevice(B->device), "cudaSetDevice");
    if (batch_max_blocks(group, B->noise_bf16, block, B->rollout_smem) < 1)
        return bfail(B, MPPI_ERR_CAPACITY, "launch shape does not fit the shared memory of a block");
    B->shape = mppi_batch::SHAPE_SET;
    B->set_G = group;
    B->set_threads = block;
    return MPPI_OK;
}

int mppi_batch_set_controls(mppi_batch* B, int32_t slot, const double* U, int32_t T, uint64_t iter) {
    if (!B || !U || slot < 0 || slot >= B->max_slots || T < 1 || T > B->max_T) return bfail(B, MPPI_ERR_ARG, "bad argument");
    if (!finite_all(U, 2 * (size_t)T)) return bfail(B, MPPI_ERR_ARG, "non-finite controls");
    BCK(cudaSetDevice(B->device), "cudaSetDevice");
    BCK(cudaMemcpy(B->slot_U + (size_t)slot * B->max_T * 2, U, sizeof(double) * 2 * T, cudaMemcpyHostToDevice),
        "controls copy");
    unsigned long long it = iter;
    BCK(cudaMemcpy(&B->slots[slot].iter, &it, sizeof(it), cudaMemcpyHostToDevice), "iter copy");
    return MPPI_OK;
}

int mppi_batch_get_controls(mppi_batch* B, int32_t slot, double* U, int32_t T, uint64_t* iter) {
    if (!B || !U || slot < 0 || slot >= B->max_slots || T < 1 || T > B->max_T) return bfail(B, MPPI_ERR_ARG, "bad argument");
    BCK(cudaSetDevice(B->device), "cudaSetDevice");
    BCK(cudaMemcpy(U, B->slot_U + (size_t)slot * B->max_T * 2, sizeof(double) * 2 * T, cudaMemcpyDeviceToHost),
        "controls copy");
    unsigned long long it = 0;
    BCK(cudaMemcpy(&it, &B->slots[slot].iter, sizeof(it), cudaMemcpyDeviceToHost), "iter copy");
    if (iter) *iter = it;
    return MPPI_OK;
}

int mppi_batch_get_costs(mppi_batch* B, int32_t ticket, int32_t i, double* S, int32_t K) {
    if (!B || !S || ticket < 0 || ticket >= (int)B->pipes.size()) return bfail(B, MPPI_ERR_ARG, "bad argument");
    std::lock_guard<std::mutex> lock(B->mu);
    Pipeline& p = B->pipes[(size_t)ticket];
    if (p.busy) return bfail(B, MPPI_ERR_CAPACITY, "the pipeline has a submission in flight");
    if (i < 0 || i >= (int)p.s_counts.size() || K != p.s_counts[(size_t)i])
        return bfail(B, MPPI_ERR_ARG, "no such plan in the pipeline's last submission, or K differs");
    BCK(cudaSetDevice(B->device), "cudaSetDevice");
    BCK(cudaMemcpy(S, p.S + p.s_offsets[(size_t)i], sizeof(double) * (size_t)K, cudaMemcpyDeviceToHost), "costs copy");
    return MPPI_OK;
}

const char* mppi_batch_last_error(mppi_batch* B) { return B ? B->err.c_str() : g_batch_err.c_str(); }

}  // extern "C"
