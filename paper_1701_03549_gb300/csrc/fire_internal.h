// Internal declarations shared by the C ABI (fire_api.cu) and the kernels
// (fire_kernels.cu).  Not part of the public interface.
#pragma once

#include <cstddef>
#include <cstdint>
#include <string>
#include <vector>

#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include "fire.h"
#include "fire_device.cuh"

namespace fire {

// Device-resident landscape.  Covariates are row-major per cell; the
// non-burnable and target bitmaps are tile-major: tile (ti, tj) of the
// ceil(H/32) x ceil(W/32) tiling owns 32 consecutive words, word r holding
// row 32 ti + r, bit i holding column 32 tj + i.  Cells of a tile that lie
// outside the grid are marked non-burnable and not in the target.
struct MapDev {
    int H, W, TH, TW, ntiles;
    const float4 *feat;         // (psi, sig, cos wind, sin wind) per cell
    const float2 *wdiag;        // cos(wind - 45 deg), cos(wind - 135 deg) per cell
    // Fixed-point covariates of the simulation's screen (fx 0: some burnable cell
    // is out of their range and the float-pair screen runs).  A wind raster of
    // one value in all burnable cells (bit for bit) has the same cosine and sine
    // there: the simulation then reads them from here and only (psi, sig) per
    // cell, 10 bytes with the flags; else (psi, sig, cos, sin), 18 bytes.  What
    // cannot burn is never read, so it has no say in either.
    int fx, uniform_wind;
    int cw, sw;                 // scale 2^30, uniform wind
    const int2 *fx2;            // (psi, sig) per cell, uniform wind
    const int4 *fx4;            // (psi, sig, cos, sin) per cell
    const uint16_t *cfl;        // bit d<8 uphill from source d, 8 forest, 9 burnable
    const uint32_t *blk;        // non-burnable bitmap, ntiles * 32 words
    const uint2 *init;          // every word of blk twice: a simulation's initial
                                // state (X, Y), ntiles * 32 pairs
    const uint32_t *tgt;        // target bitmap, ntiles * 32 words
    const uint32_t *tgt_count;  // |A|, one word
};

struct SimLaunch {
    MapDev map;                // the map when `maps` is NULL
    const MapDev *maps;        // device map table (multi-map launches)
    int nmaps;
    const int32_t *map_of_sim; // map index per simulation (NULL: map 0)
    const uint32_t *order;     // processing order of the simulations (NULL: 0..n-1)
    int ntiles_max;            // largest map of the launch (sizes buffers)
    int n;
    const fire_params *params;
    const fire_cell *ign;
    const uint64_t *seeds;
    fire_result *out;
    int32_t *burn_step;        // nullable
    uint32_t *burnt_bits;      // nullable; single-map launches only: the final
                               // burnt words (tile-major, blocked cells
                               // cleared), ntiles * 32 words per simulation
    uint32_t *work_counter;    // zeroed before a launch of fewer blocks than
                               // simulations (reset_counter)
    uint32_t *gstate;          // global-state variant: block_words words per block
    size_t block_words;        // 0: 2 * ntiles_max * 32 (the (X, Y) pairs)
    const uint8_t *burn_time;  // burn-time variant: steps each cell burns
                               // (1..250, others clamped); its blocks keep X, Y,
                               // two "still burning" planes and one fuel byte
                               // per cell in their global state
    const uint32_t *long_burn; // burn-time variant: tile-major bit plane of the
                               // cells that burn 2 steps or more (only these
                               // keep a fuel count)
    uint32_t *error_word;      // set nonzero when a bounded wait runs out
    uint32_t max_steps;        // 0 = no cap
    int qcap;                  // candidate-queue capacity (entries)
    int cell_uniform;          // 1: one uniform per target cell (Sec. 2.3)
};

// Largest batch ordered longest-first (the ranking is quadratic in n).
constexpr int kLongestFirstMax = 8192;

// Cell-flag bits.
constexpr uint16_t kFlagForest = 1u << 8;
constexpr uint16_t kFlagBurnable = 1u << 9;

// Per-simulation shared state of the simulation kernel's block.
struct SimShared {
    uint4 rk[5];          // Philox round keys: (k0, k1) of round 2j, then 2j + 1
    double beta[5];
    ScreenParams sp;
    FxParams fx;
    int use_fx;           // the map and the parameters fit the fixed-point screen
    uint32_t key0, key1;
    uint32_t first;       // the block's first simulation, then ~0
    int sim;
    int skip;
    int timeout;
    uint32_t count[3];    // worklist lengths, slot t % 3 for step t
    uint32_t newflag[3];  // some cell burning at step t (slot t % 3)
    uint32_t qcount[2];   // candidate-queue reservations of step t (t & 1)
    uint32_t qvalid[2];   // end of the valid queue prefix of step t (t & 1)
    uint32_t trials, status, last_new;
    uint32_t burnt, inter;
    uint32_t hard_cap;
    int nmark;
    // floor((2^32 - 1) / TW): k / TW = (k + 1) m >> 32 for every tile index
    // k < FIRE_MAX_TILES and TW <= FIRE_MAX_TILES (checked exhaustively)
    uint32_t tw_magic;
    MapDev map;                   // map of the current simulation
    unsigned long long mbar;
};

// Shared-memory layout of the simulation kernel (identical on host/device):
// header, worklist mark bits (2 per tile), three worklists of uint16 tile
// indices, the block's candidate queue (qcap uint32 entries), then, in the
// shared-state variant, the (X, Y) state pairs.
struct SimLayout {
    size_t header, marks, lists, queue, planes, total;
};

__host__ __device__ inline size_t align_up(size_t x, size_t a)
{
    return (x + a - 1) / a * a;
}

__host__ __device__ inline SimLayout sim_layout(int ntiles, int qcap,
                                                bool smem_state)
{
    SimLayout L;
    L.header = 0;
    L.marks = align_up(sizeof(SimShared), 16);
    L.lists = align_up(L.marks + 4 * (size_t)((ntiles + 15) / 16), 16);
    L.queue = align_up(L.lists + 3 * 2 * (size_t)ntiles, 16);
    L.planes = align_up(L.queue + 4 * (size_t)qcap, 128);
    L.total = smem_state ? L.planes + 2 * (size_t)ntiles * 128 : L.planes;
    return L;
}

// Launchers (fire_kernels.cu).  All are asynchronous on `st`.
// flags: [0] the wind varies among burnable cells; [1] a burnable cell is out of
// the fixed-point range; [2], [3] cosine and sine (float bits) of the wind in the
// first burnable cell; [4] that cell's index (~0: there is none).
cudaError_t launch_features(int H, int W, const uint8_t *veg, const float *elev,
                            const float *slope, const float *aspect,
                            const float *wind, float4 *feat, float2 *wdiag,
                            uint16_t *cfl, uint32_t *flags, cudaStream_t st);
// Fixed-point covariates of every cell into fx2 or fx4 (the other one NULL).
cudaError_t launch_fx(long long n, const float4 *feat, int2 *fx2, int4 *fx4,
                      cudaStream_t st);
cudaError_t launch_blocked(const MapDev &m, const uint8_t *veg, uint32_t *blk,
                           uint2 *init, cudaStream_t st);
cudaError_t launch_target(const MapDev &m, const uint8_t *burnt, uint32_t *tgt,
                          uint32_t *tgt_count, cudaStream_t st);
cudaError_t launch_simulate(const SimLaunch &a, bool smem_state, int nwarps,
                            int grid, size_t smem_bytes, cudaStream_t st);
// The burn-time variant (global-memory state only).
cudaError_t launch_simulate_burn(const SimLaunch &a, int nwarps, int grid,
                                 size_t smem_bytes, cudaStream_t st);
// Clears the work counter for a launch of `grid` blocks over n simulations, if
// that launch reads it: with a block per simulation it does not.
inline cudaError_t reset_counter(uint32_t *counter, long long grid, int n, cudaStream_t st)
{
    return grid < n ? cudaMemsetAsync(counter, 0, 4, st) : cudaSuccess;
}
// Tile-major bit plane of the cells whose burn time is 2 or more; stats (zeroed by
// the launcher): [0] there is such a cell, [1] the fires with b0 > 0, which spread
// across the wind and against it likelier than not and so fill the map.
cudaError_t launch_long_burn(const MapDev &m, const uint8_t *burn_time, int n,
                             const fire_params *params, uint32_t *plane,
                             uint32_t *stats, cudaStream_t st);
// Words of one block's global state in the burn-time variant.
inline size_t burn_block_words(int ntiles, long long HW)
{
    return 4 * (size_t)ntiles * 32 + (size_t)((HW + 15) / 16) * 4;
}
// Threads per block the simulation kernel is compiled for (upper bound).
constexpr int kSimMaxThreads = 512;
const void *simulate_kernel_ptr(bool smem_state);
const void *simulate_burn_kernel_ptr();
cudaError_t launch_longest_first(const MapDev &m, int n, const fire_params *params,
                                 float *key, uint32_t *order, cudaStream_t st);
cudaError_t launch_fitness(const fire_result *r, int n, int kind, double *out,
                           cudaStream_t st);
// Counting sort of simulations by rank[map_of_sim[i]] (counts: nmaps + 1).
cudaError_t launch_order(int n, const int32_t *map_of_sim, int nmaps,
                         const int32_t *rank, uint32_t *counts, uint32_t *order,
                         cudaStream_t st);
cudaError_t launch_thresholds(const MapDev &m, const double *beta_dev,
                              int64_t *out, cudaStream_t st);
cudaError_t launch_probabilities(const MapDev &m, const double *beta_dev,
                                 float *p32, double *p64, cudaStream_t st);
cudaError_t launch_features_export(const MapDev &m, float *psi, float *sig,
                                   float *cw, float *sw, uint16_t *cfl,
                                   cudaStream_t st);
cudaError_t launch_screen_selftest(uint64_t n, uint64_t seed,
                                   unsigned long long *counts,
                                   unsigned long long *max_dp_bits,
                                   cudaStream_t st);
cudaError_t launch_philox_blocks(uint64_t n, uint4 ctr, uint2 key,
                                 uint32_t *out, cudaStream_t st);

struct LaunchPlan {
    int nwarps, qcap;
    bool smem_state;
    SimLayout L;
    int grid;
};

}  // namespace fire

// Launch-shape record of the autotuner (per map tile count).
struct TuneEntry {
    int ntiles, warps, bps, queue, state;
    float ms;
};

// A captured CUDA graph and the call it replays.
struct GraphEntry {
    std::vector<unsigned long long> key;
    cudaGraphExec_t exec;
    unsigned epoch;
};

// Opaque handles of the C ABI (definitions shared by the host sources).
struct fire_ctx {
    int device = 0;
    int num_sms = 0;
    size_t max_smem_optin = 0, smem_per_sm = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    int warps_per_block = 0;   // 0: heuristic
    int blocks_per_sm = 0;     // 0: as many as fit
    int queue_entries = 0;     // 0: default
    int state_mode = 0;        // FIRE_STATE_*
    std::string err;
    // device scratch
    uint32_t *counter = nullptr;     // work counter + error word
    uint32_t *host_error = nullptr;  // pinned copy of the error word (fire_sync)
    void *staging = nullptr;         // inputs / outputs of host-pointer calls
    size_t staging_bytes = 0;
    uint32_t *gstate = nullptr;      // global-state simulation buffers
    size_t gstate_bytes = 0;
    size_t gstate_refused = 0;       // smallest size that failed (0: none yet)
    void *host_pinned = nullptr;     // pinned bounce buffer
    size_t host_pinned_bytes = 0;
    void *table = nullptr;           // map table + map ranks (multi-map calls)
    size_t table_bytes = 0;
    void *order = nullptr;           // bucket counts + processing order
    size_t order_bytes = 0;
    void *lpt = nullptr;             // longest-first keys + order (single map)
    size_t lpt_bytes = 0;
    std::vector<TuneEntry> tuned;    // autotuned launch shapes
    std::vector<GraphEntry> graphs;  // captured calls
    unsigned epoch = 0;              // bumped when a device buffer moves
    int fail_alloc_after = -1;       // test hook: fail that growth (-1: off)
    void *burn_aux = nullptr;        // burn-time calls: long-burn plane + flag
    size_t burn_aux_bytes = 0;
};

struct fire_map {
    fire_ctx *ctx = nullptr;
    fire::MapDev dev{};
    float cell_m = 0.f;
    float4 *feat = nullptr;
    float2 *wdiag = nullptr;
    void *fx = nullptr;
    uint16_t *cfl = nullptr;
    uint32_t *blk = nullptr;
    uint2 *init = nullptr;
    uint32_t *tgt = nullptr;
    uint32_t *tgt_count = nullptr;
    std::vector<uint8_t> burnable_host;
};


namespace fire {
// Host helpers shared by the C ABI sources (fire_api.cu).
int set_err(fire_ctx *ctx, int code, const char *fmt, ...);
int cuda_err(fire_ctx *ctx, cudaError_t e, const char *what);
int ensure_device(fire_ctx *ctx);
// keep: the old buffer stays until the new one is there, and if it cannot be had.
int grow_device(fire_ctx *ctx, void **buf, size_t *cap, size_t need,
                const char *what, bool keep = false);
size_t round16(size_t x);
bool valid_map(const fire_map *m);
int noalloc_take_error(int device, bool *set);
// Launch shape of the simulation kernel (burn: the burn-time variant, whose
// state is always in global memory; fixed_scratch: no state buffer can be
// grown, so a state that fits in shared memory goes there).
int plan_launch(fire_ctx *ctx, int ntiles, long long n, LaunchPlan *p,
                bool burn = false, bool fixed_scratch = false,
                long long spreading = 0);
// plan_launch, with ctx->gstate grown for it (not for the burn-time variant).
int plan_with_state(fire_ctx *ctx, int ntiles, long long n, LaunchPlan *p);
// Launch that may begin while the kernel before it on the stream drains
// (programmatic stream serialisation).  The kernel calls pdl_wait() before it
// touches anything an earlier kernel wrote or reads; what comes before that
// (barriers, tensor memory, weights, which no kernel of a pass writes) overlaps
// the predecessor's last CTAs.
template <class Kernel, class... Args>
cudaError_t launch_pdl(Kernel kern, dim3 grid, int threads, size_t smem, cudaStream_t st,
                       Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

// The network's head on the top layer's activations: probabilities, and with
// target the per-pixel gradient g and the loss terms (summed by k_loss_sum).
struct HeadArgs {
    const float *wh;       // w[128], then the bias
    float *prob;
    const float *target;   // nullable
    float inv_count;
    float *g, *term;
};
cudaError_t launch_conv_tma(int mode, const uint16_t *in, const uint16_t *w,
                            const float *bias, uint4 *bits, uint16_t *out,
                            int n, int S, int lgS, int d, const HeadArgs *head,
                            uint32_t *err, cudaStream_t st);
// Bias and head gradients are sums over all pixels.  An FP32 atomic addition rounds
// the running total, so they are added in kSumSlots slots of kSums floats, a block's
// partial sums into the slot of its number, and the slots together in double
// precision at the end (k_round_sums).  Error against 64-bit sums of the same terms,
// of the norm: 32 samples at S = 32, bias 2.9e-8 and head 3.5e-8 (one slot: 1.7e-7
// and 3.4e-7); 8 at S = 256, 4.2e-7 (the tensor core's chains) and 5.0e-8 (4.6e-7 and
// 6.5e-7).  The launch that adds them also hands out the loss, which was a copy.
constexpr int kSums = FIRE_NET_LAYERS * 128 + 129, kSumSlots = 16;
cudaError_t launch_conv1_tma(const uint16_t *x, const uint16_t *w, const float *bias,
                             uint16_t *out, uint4 *bits, int n, int S, int lgS, uint32_t *err,
                             cudaStream_t st);
cudaError_t launch_wgrad_tma(const uint16_t *dz, const uint16_t *in, int cin, float *dw,
                             float *db, int n, int S, int lgS, int d, uint32_t *err,
                             cudaStream_t st);
int launch_batch(fire_ctx *ctx, const fire_map *m, int n,
                 const fire_params *dparams, const fire_cell *dign,
                 const uint64_t *dseeds, uint32_t max_steps, uint32_t flags,
                 fire_result *dout, int32_t *dsteps, uint32_t *dbits);
}  // namespace fire

// NVTX range named after the C-ABI entry point, open for the call's
// duration (profilers such as Nsight show the library's calls on the host
// timeline; without a tool attached each range costs a no-op call).
struct NvtxScope {
    explicit NvtxScope(const char *name) { nvtxRangePushA(name); }
    ~NvtxScope() { nvtxRangePop(); }
    NvtxScope(const NvtxScope &) = delete;
    NvtxScope &operator=(const NvtxScope &) = delete;
};
#define FIRE_NVTX(name) NvtxScope fire_nvtx_scope_(name)

#define CUDA_TRY(ctx, expr, what)                                   \
    do {                                                            \
        cudaError_t e_ = (expr);                                    \
        if (e_ != cudaSuccess) return fire::cuda_err(ctx, e_, what); \
    } while (0)
