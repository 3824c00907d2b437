// TMA-fed implicit-GEMM convolutions of the surrogate network on tcgen05
// tensor cores: the 128 -> 128 layers forward and input gradient
// (k_conv_pair), the weight and bias gradients of all layers (k_wgrad_strip)
// and the first layer forward (k_conv1).
//
// In each, one thread issues tensor-map copies of shifted NHWC activation
// boxes (channels, x, y, sample; out-of-range elements read as zero, which is
// the convolution's zero padding) that land swizzled, in the tensor core's
// canonical layouts; one issues MMAs into a tensor-memory accumulator and
// commits them to the barriers that hand the stages back; warps drain the
// accumulator (tensor memory -> registers -> stores).  Every wait is bounded;
// on a timeout the CTA records an error, waits (bounded) for its own copies
// and MMAs in flight, frees its tensor memory and returns.
#include "fire_internal.h"
#include "fire_tc.cuh"

#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <mutex>

namespace fire {
namespace convtma {

constexpr int kSlabs = 18;                      // 9 taps x 2 channel halves
// Epilogues: forward (bias + ReLU), input gradient (ReLU mask of the layer
// below), forward with the network's head behind it.
constexpr int kFwd = 0, kDgrad = 1, kFwdHead = 2;

struct Epi {
    const float *bias;        // forward
    // [P][4] where activations are positive, channel c in bit (c % 32) / 2 + 16 (c
    // % 2) of word c / 32: forward, of the output (nullable, written); input
    // gradient, of the layer below
    uint4 *bits;
    uint16_t *out;            // [P][128] BF16
    HeadArgs head;
};

__device__ __forceinline__ uint64_t desc_sw128(uint32_t saddr)
{
    uint64_t d = (uint64_t)((saddr & 0x3ffffu) >> 4);
    d |= (uint64_t)1 << 16;                 // LBO (unused for swizzled K-major)
    d |= (uint64_t)(1024 >> 4) << 32;       // SBO: 8 rows x 128 B
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;                 // SWIZZLE_128B
    return d;
}

__device__ __forceinline__ void expect_tx(void *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(
                     tc::smem_addr(bar)),
                 "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void tma_4d(uint32_t dst, const CUtensorMap *map, int c0,
                                       int c1, int c2, int c3, void *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::"
        "bytes [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3),
        "r"(tc::smem_addr(bar))
        : "memory");
}

__device__ __forceinline__ void tma_5d(uint32_t dst, const CUtensorMap *map, int c0,
                                       int c1, int c2, int c3, int c4, void *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::"
        "bytes [%0], [%1, {%2, %3, %4, %5, %6}], [%7];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3),
        "r"(c4), "r"(tc::smem_addr(bar))
        : "memory");
}

__device__ __forceinline__ void tma_2d(uint32_t dst, const CUtensorMap *map, int c0,
                                       int c1, void *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::"
        "bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1),
        "r"(tc::smem_addr(bar))
        : "memory");
}

__device__ __forceinline__ uint32_t pack2(float a, float b)
{
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t *>(&h);
}

// 32 bytes of one row per thread: whole sectors, where 16-byte accesses of
// rows 256 bytes apart touch every sector twice.
__device__ __forceinline__ void st_global32(void *p, const uint32_t v[8])
{
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p),
                 "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]),
                 "r"(v[6]), "r"(v[7])
                 : "memory");
}

// One lane of a converged warp.
__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "elect.sync _|p, 0xffffffff;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(p));
    return p != 0;
}

__device__ __forceinline__ bool all_ok(bool ok)
{
    return __all_sync(0xffffffffu, ok);
}

// --- CTA-pair primitives (cta_group::2) -------------------------------------

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\t"
                 "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Address in the shared window of CTA 0 of the pair of a local address.
__device__ __forceinline__ uint32_t leader_addr(const void *p)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(tc::smem_addr(p)));
    return r;
}

__device__ __forceinline__ void mbar_arrive(void *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_addr(bar))
                 : "memory");
}

__device__ __forceinline__ void arrive_cluster(uint32_t cluster_addr)
{
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(
                     cluster_addr)
                 : "memory");
}

// Tensor-map copies into this CTA's shared memory whose bytes count on a
// barrier of either CTA of the pair.
__device__ __forceinline__ void tma_4d_pair(uint32_t dst, const CUtensorMap *map,
                                            int c0, int c1, int c2, int c3,
                                            uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.tile."
        "mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3),
        "r"(bar)
        : "memory");
}

__device__ __forceinline__ void tma_5d_pair(uint32_t dst, const CUtensorMap *map,
                                            int c0, int c1, int c2, int c3, int c4,
                                            uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.5d.cta_group::2.shared::cluster.global.tile."
        "mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], [%7];" ::"r"(
            dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3),
        "r"(c4), "r"(bar)
        : "memory");
}

__device__ __forceinline__ void tma_2d_pair(uint32_t dst, const CUtensorMap *map,
                                            int c0, int c1, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile."
        "mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar)
        : "memory");
}

__device__ __forceinline__ void mma_bf16_pair(uint32_t d_tmem, uint64_t adesc,
                                              uint64_t bdesc, uint32_t idesc,
                                              bool accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.u32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(
            d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"((uint32_t)accumulate)
        : "memory");
}

// The four K = 16 steps of a 64-wide slab.
__device__ __forceinline__ void issue4(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc,
                                       uint32_t idesc, bool accumulate)
{
#pragma unroll
    for (int kk = 0; kk < 4; ++kk)
        mma_bf16_pair(d_tmem, adesc + kk * 2, bdesc + kk * 2, idesc, accumulate || kk > 0);
}

// Arrives on the barrier at this offset in both CTAs once the MMAs issued so
// far are done.
__device__ __forceinline__ void commit_pair(void *bar)
{
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster."
        "multicast::cluster.b64 [%0], %1;" ::"r"(tc::smem_addr(bar)),
        "h"((uint16_t)3)
        : "memory");
}

__device__ __forceinline__ void tmem_alloc_pair(uint32_t *dst_smem, uint32_t ncols)
{
    asm volatile(
        "tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
            tc::smem_addr(dst_smem)),
        "r"(ncols)
        : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" :::
                     "memory");
}

__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr),
                 "r"(ncols)
                 : "memory");
}

// How the pair convolution streams a layer's activations (conv_shape): strips
// of `px` pixels x 64 channels, each serving `taps` taps (the three of a row,
// or one), in `na` shared-memory stages.
//
// step > 0: the tile's 128 pixels are laid out so that a tap's shift by d pixels
// is a shift by `step` pixels of the tile itself, and what it shifts in from
// beyond is the zero padding: `gap` zero pixels between the stages.  Pixel m of
// the tile is pixel (m / fold) * outer + (m mod fold) * inner of the image.
//   Row combs (d >= S / 16): `fold` = 128 d / S neighbouring pixels at every
//     multiple of d of one row; a shift is one tooth.
//   Columns (S < 128): 128 / S whole rows, column by column; a shift is d
//     columns.
struct StripShape {
    int taps, px, na;
    int step, gap, fold, outer, inner, cols;   // cols: columns, else comb
};

constexpr int kWHalf = 64 * 128;                // 64 weight rows x 64 BF16
constexpr int kWBytes = kSlabs * kWHalf;        // one CTA's half of the weights
constexpr int kStripRoom = 80 * 1024;
constexpr int kMaxA = 5;
constexpr int kEpiWarps = 4;
constexpr int kPairThreads = 32 * (kEpiWarps + 3);
constexpr int kPairSmem = kWBytes + kStripRoom + 3072;   // + alignment, barriers

struct PairShared {
    unsigned long long afull[kMaxA], aempty[kMaxA], wfull[kSlabs];
    unsigned long long tfull[2], tempty[2], done;
    uint32_t tmem_slot;
    int fail, issued, used;
    float bias[128], head[129];
};
static_assert(sizeof(PairShared) <= 2048, "barrier area");

__device__ __forceinline__ float bf16_lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t u)
{
    return __uint_as_float(u & 0xffff0000u);
}

// Probability, gradient and loss term of pixel p from the head's 16 partial
// sums of eight channels each (added in the order of k_head, whose 16 lanes
// hold one each).
__device__ __forceinline__ void head_pixel(const HeadArgs &hd, float bias,
                                           const float part[16], size_t p)
{
    float v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = part[i] + part[i + 8];
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] += v[i + 4];
    const float z = ((v[0] + v[2]) + (v[1] + v[3])) + bias;
    const float y = 1.0f / (1.0f + expf(-z));
    hd.prob[p] = y;
    if (hd.target) {
        const float t = hd.target[p];
        hd.term[p] = fmaxf(z, 0.0f) - t * z + log1pf(expf(-fabsf(z)));
        hd.g[p] = (y - t) * hd.inv_count;
    }
}

// Epilogue of one accumulator row (pixel p, 128 channels in tensor memory at
// taddr): forward, bias and ReLU; input gradient, zero where the layer
// below's activation is not positive (mask: its bits); BF16 stores.  s_head: the
// head's weights and bias.
template <int kMode>
__device__ __forceinline__ void pair_epilogue(const Epi &epi, const float *s_bias,
                                              const float *s_head, uint32_t taddr,
                                              size_t p, uint4 mask)
{
    uint16_t *orow = epi.out + p * 128;
    float part[16];
    uint32_t words[4] = {mask.x, mask.y, mask.z, mask.w};
#pragma unroll
    for (int c0 = 0; c0 < 128; c0 += 32) {
        float v[32];
        tc::tmem_ld32(taddr + (uint32_t)c0, v);
        uint32_t pk[16];
        if (kMode != kDgrad) {
#pragma unroll
            for (int j = 0; j < 16; ++j)
                pk[j] = pack2(fmaxf(v[2 * j] + s_bias[c0 + 2 * j], 0.0f),
                              fmaxf(v[2 * j + 1] + s_bias[c0 + 2 * j + 1], 0.0f));
            if (epi.bits) {
                uint32_t w = 0;   // a half that is not zero carries into its sign
#pragma unroll
                for (int j = 0; j < 16; ++j)
                    w |= (((pk[j] & 0x7fff7fffu) + 0x7fff7fffu) & 0x80008000u) >> (15 - j);
                words[c0 / 32] = w;
            }
        } else {
            const uint32_t w = words[c0 / 32];
#pragma unroll
            for (int j = 0; j < 16; ++j)
                pk[j] = pack2(v[2 * j], v[2 * j + 1]) & (((w >> j) & 0x10001u) * 0xffffu);
        }
        if (kMode == kFwdHead) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                float z = 0.0f;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    z = fmaf(bf16_lo(pk[4 * q + j]), s_head[c0 + 8 * q + 2 * j], z);
                    z = fmaf(bf16_hi(pk[4 * q + j]), s_head[c0 + 8 * q + 2 * j + 1], z);
                }
                part[c0 / 8 + q] = z;
            }
        }
        st_global32(orow + c0, pk);
        st_global32(orow + c0 + 16, pk + 8);
    }
    if (kMode != kDgrad && epi.bits)
        epi.bits[p] = make_uint4(words[0], words[1], words[2], words[3]);
    if (kMode == kFwdHead) head_pixel(epi.head, s_head[128], part, p);
}

// Convolution of a 128 -> 128 layer on CTA pairs (cta_group::2).  The pair
// computes 256 pixels x 128 channels, each CTA its own 128 pixels (rows of A)
// with 64 rows of the weights (half of B, read by the tensor cores of both
// SMs).  The K loop runs over the taps and the two 64-channel halves, in this
// order.
//
// What bounds it, and why this shape (8 x 256 x 256, 154.6 GFLOP a layer):
//  * half the weights are 144 KB, so they are loaded once and stay: only
//    activations stream.  Distinct data reaches an SM from L2 at no more than
//    about 30 bytes per clock when all SMs read (9 TB/s), and a 16 KB box per
//    tap and half needs 64; a strip of 128 + 2 d pixels that serves the three
//    taps of a row needs 6 to 8 KB per tap and half.  Wide dilations (32, 64) have
//    no room for four such strips and take combs of 128 pixels (StripShape); where
//    those can't be had (teeth below 8 pixels, or separate rows), three strips or a
//    box per tap.
//  * the issuing thread's own instructions: with waits, commits and
//    descriptor arithmetic per 64-wide slab it took 500 clocks a slab
//    whatever the MMA count, against 256 for the slab's MMAs.  Waits and
//    commits per row of taps, unrolled, leave the tensor core the bound.
// Measured (one layer): 84 us for d <= 16 (1840 TFLOP/s) and, with combs, for
// d = 32; 108 us for d = 64 (combs, three stages); the input gradients 83 and 105
// with the layer below's ReLU mask as bits, 96 and 114 when they read its
// activations for it (32 KB more into an SM per tile).  One 128-pixel tile per
// CTA with boxes per tap and streamed weights took 136 us for every d, and 158
// for the input gradients.
//
// Persistent: one pair per two SMs walks pairs of tiles.  In both CTAs one
// thread issues the strip copies, whose bytes count on the leader's barrier
// (CTA 0), one loads the weights, four warps drain the accumulator; a warp of
// the leader issues the MMAs into one of two 128-column accumulators, so that
// a tile's epilogue runs under the next tile's MMAs.
//
// sign = +1: forward (source pixel p + off(t)); -1: input gradient (p - off(t)).
// A strip serves kTaps taps (StripShape).  kComb: kTaps is 3 and the tiles are
// combs or columns.
template <int kTaps, int kMode, bool kComb>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kPairThreads, 1)
    k_conv_pair(const __grid_constant__ CUtensorMap act,
                const __grid_constant__ CUtensorMap wts, Epi epi, StripShape sp, int S,
                int lgS, int d, int sign, int npairs, uint32_t *err)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    const uint32_t raw = tc::smem_addr(smem_raw);
    const uint32_t wbase = (raw + 1023u) & ~1023u;
    const uint32_t abase = wbase + kWBytes;
    PairShared &sh = *reinterpret_cast<PairShared *>(smem_raw + (wbase - raw) + kWBytes +
                                                     kStripRoom);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = (int)cluster_rank();
    const int pair0 = blockIdx.x >> 1, pstep = gridDim.x >> 1;
    constexpr int kGroups = 9 / kTaps;
    const int na = sp.na;
    const uint32_t strip = (uint32_t)sp.px * 128;    // from one stage to the next
    const uint32_t copied = kComb ? 128 * 128 : strip;
    if (kComb) {
        // the zero gaps: before each stage's 128 pixels, and behind the last
        uint4 *const gap = reinterpret_cast<uint4 *>(smem_raw + (abase - raw));
        const int n16 = sp.gap * 8;
        for (int i = tid; i < (na + 1) * n16; i += kPairThreads)
            gap[(i / n16) * (strip >> 4) + i % n16] = make_uint4(0u, 0u, 0u, 0u);
        tc::fence_proxy_async();
    }
    if (kMode != kDgrad && tid < 128) sh.bias[tid] = epi.bias[tid];
    if (kMode == kFwdHead && tid <= 128) sh.head[tid] = epi.head.wh[tid];
    if (warp == kEpiWarps) tmem_alloc_pair(&sh.tmem_slot, 256);
    if (tid == 0) {
        for (int i = 0; i < kMaxA; ++i) {
            tc::mbar_init(&sh.afull[i], 1);
            tc::mbar_init(&sh.aempty[i], 1);
        }
        for (int i = 0; i < kSlabs; ++i) tc::mbar_init(&sh.wfull[i], 1);
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(&sh.tfull[i], 1);
            tc::mbar_init(&sh.tempty[i], 2 * kEpiWarps);   // of both CTAs
        }
        tc::mbar_init(&sh.done, 1);
        sh.fail = 0;
        sh.issued = sh.used = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc::fence_before_sync();
    __syncthreads();
    cluster_sync();   // the barriers of both CTAs are set up
    tc::fence_after_sync();
    const uint32_t tmem = sh.tmem_slot;

    if (warp == kEpiWarps) {
        // strip loader: strip g of the pair's sequence uses stage g mod na
        pdl_wait();
        const bool leader = elect_one();
        int g = 0, st = 0;
        uint32_t ph = 1;   // parity of the stage's last release
        bool ok = true;
        for (int pr = pair0; ok && pr < npairs; pr += pstep) {
            const int m0 = (2 * pr + rank) * 128;
            const int b = m0 >> (2 * lgS);
            const int y0 = (m0 >> lgS) & (S - 1), x0 = m0 & (S - 1);
            for (int q = 0; ok && q < kGroups; ++q) {
                const int dy = sign * ((kTaps == 3 ? q : q / 3) - 1) * d;
                const int dx = kTaps == 3 ? -d : sign * (q % 3 - 1) * d;
                for (int half = 0; half < 2; ++half, ++g) {
                    if (g >= na) ok = all_ok(tc::mbar_wait_bounded(&sh.aempty[st], ph));
                    ok = all_ok(ok && !*(volatile int *)&sh.fail);
                    if (!ok) break;
                    if (leader) {
                        if (rank == 0) expect_tx(&sh.afull[st], 2 * copied);
                        if (kComb)
                            tma_5d_pair(abase + st * strip + sp.gap * 128, &act, half * 64,
                                        sp.cols ? y0 + dy : (x0 >> 7) * sp.fold, 0,
                                        sp.cols ? 0 : y0 + dy, b,
                                        leader_addr(&sh.afull[st]));
                        else
                            tma_4d_pair(abase + st * strip, &act, half * 64, x0 + dx,
                                        y0 + dy, b, leader_addr(&sh.afull[st]));
                    }
                    __syncwarp();
                    if (++st == na) st = 0, ph ^= 1;
                }
            }
        }
        if (leader) {
            if (!ok) atomicOr(&sh.fail, 1);
            sh.issued = g;
        }
        __syncwarp();
    } else if (warp == kEpiWarps + 1) {
        // this CTA's half of the weights: rows 64 rank .. 64 rank + 63 (no
        // kernel that can still be running writes them)
        const bool leader = elect_one();
        for (int s = 0; s < kSlabs; ++s) {
            if (leader) {
                if (rank == 0) expect_tx(&sh.wfull[s], 2 * kWHalf);
                tma_2d_pair(wbase + s * kWHalf, &wts, s * 64, 64 * rank,
                            leader_addr(&sh.wfull[s]));
            }
            __syncwarp();
        }
    } else if (warp == kEpiWarps + 2) {
        if (rank == 0) {
            // MMA issuer: pair number `it` of this cluster accumulates in
            // buffer it & 1, once the epilogues have drained its last use.
            // One thread's instruction latency is what an MMA every 64 clocks
            // competes with, so the waits and commits are per group of taps,
            // the slabs of a group are unrolled, and the whole warp walks the
            // loop and votes on its waits, which keeps the operand descriptors
            // warp-uniform; one elected lane issues.
            constexpr uint32_t idesc = tc::idesc_bf16(256, 128);
            const uint64_t adesc = desc_sw128(abase), wdesc = desc_sw128(wbase);
            const uint32_t strip16 = strip >> 4;
            // rows of a strip: a tap's shift (a multiple of 128 bytes; the
            // 128-byte swizzle goes by address, so any row may come first)
            const int shift = kComb ? sp.step : d;
            const uint32_t row0 = (kComb ? sp.gap - sp.step : 0) * 8 +
                                  (sign > 0 ? 0 : (kTaps - 1) * (uint32_t)shift * 8);
            const int rowstep = sign * shift * 8;
            const bool leader = elect_one();
            int it = 0, ast = 0, ag = 0;
            uint32_t aph = 0;
            bool ok = true;
            for (int pr = pair0; ok && pr < npairs; pr += pstep, ++it) {
                const int acc = it & 1;
                if (it >= 2)
                    ok = all_ok(tc::mbar_wait_bounded(&sh.tempty[acc], ((it >> 1) - 1) & 1));
                const uint32_t td = tmem + (uint32_t)(acc * 128);
                for (int q = 0; ok && q < kGroups; ++q) {
                    // the strips of the two channel halves
                    const int st0 = ast, st1 = ast + 1 == na ? 0 : ast + 1;
                    const uint32_t ph1 = ast + 1 == na ? aph ^ 1 : aph;
                    if (it == 0)
                        for (int s = 2 * kTaps * q; ok && s < 2 * kTaps * (q + 1); ++s)
                            ok = all_ok(tc::mbar_wait_bounded(&sh.wfull[s], 0));
                    ok = ok && all_ok(tc::mbar_wait_bounded(&sh.afull[st0], aph));
                    if (!ok) break;
                    tc::fence_after_sync();
                    const uint64_t a0 = adesc + st0 * strip16 + row0;
                    const uint64_t a1 = adesc + st1 * strip16 + row0;
                    const uint64_t w0 = wdesc + q * (2 * kTaps * (kWHalf >> 4));
                    // the first tap's first half starts without the second strip,
                    // and the first strip is released before the last half: what
                    // three strips need to keep one in flight (d = 64 at S = 256:
                    // 110 us against 128)
                    if (kTaps == 3) {
                        if (leader) issue4(td, a0, w0, idesc, q > 0);
                        __syncwarp();
                    }
                    ok = all_ok(tc::mbar_wait_bounded(&sh.afull[st1], ph1));
                    if (!ok) break;
                    tc::fence_after_sync();
                    if (leader) {
#pragma unroll
                        for (int j = 0; j < kTaps; ++j) {
                            if (j > 0 || kTaps == 1)
                                issue4(td, a0 + j * rowstep, w0 + 2 * j * (kWHalf >> 4),
                                       idesc, q > 0 || j > 0);
                            if (j == kTaps - 1) commit_pair(&sh.aempty[st0]);
                            issue4(td, a1 + j * rowstep,
                                   w0 + (2 * j + 1) * (kWHalf >> 4), idesc, true);
                        }
                        commit_pair(&sh.aempty[st1]);
                        if (q == kGroups - 1) commit_pair(&sh.tfull[acc]);
                    }
                    __syncwarp();
                    ag += 2;
                    ast += 2;
                    if (ast >= na) ast -= na, aph ^= 1;
                }
            }
            if (leader) {
                if (!ok) atomicOr(&sh.fail, 1);
                sh.used = ag;
                commit_pair(&sh.done);   // arrives once every issued MMA is done
            }
            __syncwarp();
        }
    } else {
        // epilogue: pair number `it` is read from buffer it & 1
        pdl_wait();
        int it = 0;
        for (int pr = pair0; pr < npairs; pr += pstep, ++it) {
            const int acc = it & 1;
            const int tile = 2 * pr + rank, m = warp * 32 + lane;
            size_t p = (size_t)tile * 128 + m;
            if (kComb) {
                // a comb's first pixel: its row's, then its tooth's
                const size_t first = sp.cols ? (size_t)tile * 128
                                             : ((size_t)(tile >> (lgS - 7)) << lgS) +
                                                   (tile & ((S >> 7) - 1)) * sp.fold;
                const int q = m / sp.fold;
                p = first + q * sp.outer + (m - q * sp.fold) * sp.inner;
            }
            const uint4 mask = kMode == kDgrad ? epi.bits[p] : make_uint4(0, 0, 0, 0);
            if (*(volatile int *)&sh.fail ||
                !tc::mbar_wait_bounded(&sh.tfull[acc], (it >> 1) & 1)) {
                atomicOr(&sh.fail, 1);
                break;
            }
            tc::fence_after_sync();
            pair_epilogue<kMode>(epi, sh.bias, sh.head,
                                 tmem + ((uint32_t)(warp * 32) << 16) +
                                     (uint32_t)(acc * 128),
                                 p, mask);
            tc::fence_before_sync();
            __syncwarp();
            if (lane == 0) arrive_cluster(leader_addr(&sh.tempty[acc]));
        }
    }
    __syncthreads();
    if (tid == 0) {
        if (sh.fail) {
            atomicOr(err, 1u);
            // copies of either CTA still in flight must land before the pair
            // leaves: the leader waits for those it can see (bounded), both
            // for a time far above a copy's
            if (rank == 0)
                for (int g = sh.used; g < sh.issued; ++g)
                    tc::mbar_wait_bounded(&sh.afull[g % na], (g / na) & 1);
            const long long t0 = clock64();
            while (clock64() - t0 < (1ll << 24)) {}
        }
        // every MMA of the pair has completed
        tc::mbar_wait_bounded(&sh.done, 0);
    }
    tc::fence_before_sync();
    __syncthreads();
    cluster_sync();   // neither CTA leaves while the other may signal it
    tc::fence_after_sync();
    if (warp == kEpiWarps) tmem_dealloc_pair(tmem, 256);
}

// Weight and bias gradients of a layer of Cin input channels (128 or 16):
// dW[o][(t, i)] += sum_p dz[p, o] in[p + off(t), i], db[o] += sum_p dz[p, o].
// Both operands are MN-major (channels within 128 or 32 bytes of a pixel,
// pixels along K).  A slab is L pixels: dz, and strips of `in` with d pixels
// on either side of each row, so that the three taps of a row of taps are one
// operand: N = 3 taps x 64 (16) channels, the taps d pixels apart (the
// leading-dimension stride; swizzles go by address, so a tap may start at any
// pixel).  Where a strip of separate rows would be wider than three boxes
// (d >= S) it is three boxes, one per tap.  A CTA takes a range of slabs and,
// with 128 channels, one row of taps and both channel halves (2 x N = 192),
// with 16 all three rows (3 x N = 48); a column of ones beside them gives the
// bias gradient in the same pass, shared out over the rows' CTAs.
//
// What bounds it (128 channels, 8 x 256 x 256, 154.6 GFLOP): the copies into
// shared memory, 64 to 68 KB per 128 pixels at 30 bytes a clock for 1536 clocks
// of MMAs (halving the MMAs saves a fifth; sharing dz by multicast in clusters of
// three saves nothing and leaves 14 SMs idle), then shared memory, which a 128 x
// 192 x 16 MMA reads at 107 bytes a clock.  Rows are taken in chains y, y + d, y +
// 2d, so that the three rows of taps read a row of `in` one slab row apart and not
// d: 275 MB from DRAM instead of 508 at d = 16, a training step 2075 us instead of
// 2095; with combs 2060.  86 us a layer with the bias (d = 64, two stages: 92).
// One tap per CTA with a box per operand loaded 32 KB per 64 pixels and tap: 119
// us, and another 27 us for a bias pass over dz.  16 channels: 31 us (bound by
// reading dz, 134 MB) against 204 on register-staged tiles.
struct WgradShape {
    int L, lgw;        // pixels of a slab, log2 pixels of its rows
    int pitch;         // pixels from one row of a strip to the next
    int nbox, box;     // boxes of a strip and the bytes of one
    int tap;           // bytes from one tap to the next
    int strip, stages;
    int lgm;           // log2 rows of a chain of rows d apart, 0: rows in order
    int fold;          // comb: pixels of a tooth, and of the gaps around the strip
};

constexpr int kMaxWgStages = 6;
constexpr int kWgThreads = 192;
constexpr int kOnesBytes = 2048;
constexpr int kWgRoom = 227 * 1024 - 2048 - kOnesBytes;   // beside alignment, barriers

struct WgradShared {
    unsigned long long full[kMaxWgStages], empty[kMaxWgStages], done;
    uint32_t tmem_slot;
    int fail, issued, used;
};

__device__ __forceinline__ uint64_t desc_mn(uint32_t saddr, uint32_t lbo, uint32_t sbo,
                                            uint32_t swizzle)
{
    uint64_t d = (uint64_t)((saddr & 0x3ffffu) >> 4);
    d |= (uint64_t)(lbo >> 4) << 16;        // next 64 (16) MN elements
    d |= (uint64_t)(sbo >> 4) << 32;        // next 8 K rows
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)swizzle << 61;           // 2: 128 bytes, 6: 32 bytes
    return d;
}

template <int Cin, int kSteps>
__global__ void __launch_bounds__(kWgThreads, 1)
    k_wgrad_strip(const __grid_constant__ CUtensorMap dzm,
                  const __grid_constant__ CUtensorMap inm, float *dw, float *db, int S,
                  int lgS, int d, WgradShape sp, int slabs_total, int slabs_per,
                  uint32_t *err)
{
    constexpr int kB = Cin == 128 ? 2 : 3;          // strips of a slab
    constexpr int kCh = Cin == 128 ? 64 : 16;       // channels of a strip
    constexpr int kN = 3 * kCh;
    constexpr uint32_t kRow = kCh * 2;              // bytes of a pixel
    constexpr uint32_t kSwizzle = Cin == 128 ? 2 : 6;
    constexpr int kBiasCol = kB * kN;
    constexpr int kCols = Cin == 128 ? 512 : 256;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    const uint32_t raw = tc::smem_addr(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    unsigned char *const sm = smem_raw + (base - raw);
    WgradShared &sh = *reinterpret_cast<WgradShared *>(sm + kWgRoom + kOnesBytes);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr uint32_t kDz = kSteps * 16 * 256;     // bytes of a dz slab
    const uint32_t stage = kDz + kB * (uint32_t)sp.strip;
    // the CTAs of one pixel range are neighbours: their dz requests meet on the way
    const int dyi = Cin == 128 ? (int)blockIdx.x : 0;
    const int s0 = blockIdx.y * slabs_per;
    const int ns = min(slabs_total - s0, slabs_per);
    // slabs whose bias this CTA sums: all, or those of its residue mod 3
    const int nbias = Cin == 128 ? (s0 + ns + 2 - dyi) / 3 - (s0 + 2 - dyi) / 3 : ns;

    if (warp == 4) {
        tc::tmem_alloc(&sh.tmem_slot, kCols);
        tc::tmem_relinquish();
    }
    for (int i = tid; i < kOnesBytes / 4; i += kWgThreads)
        reinterpret_cast<uint32_t *>(sm + kWgRoom)[i] = 0x3f803f80u;
    // zeros of the combs' gaps: no copy writes there
    for (int i = tid; i < sp.stages * kB * 2 * sp.fold * 8; i += kWgThreads) {
        const int gap = i / (sp.fold * 8), strip = gap >> 1;
        unsigned char *const at = sm + (strip / kB) * stage + kDz + (strip % kB) * sp.strip +
                                  (gap & 1) * (sp.strip - sp.fold * 128);
        reinterpret_cast<uint4 *>(at)[i - gap * (sp.fold * 8)] = make_uint4(0, 0, 0, 0);
    }
    tc::fence_proxy_async();
    if (tid == 0) {
        for (int i = 0; i < kMaxWgStages; ++i) {
            tc::mbar_init(&sh.full[i], 1);
            tc::mbar_init(&sh.empty[i], 1);
        }
        tc::mbar_init(&sh.done, 1);
        sh.fail = sh.issued = sh.used = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = sh.tmem_slot;
    pdl_wait();

    if (warp == 4) {
        const bool leader = elect_one();
        int st = 0, s = 0;
        uint32_t ph = 1;
        bool ok = true;
        for (; s < ns; ++s) {
            if (s >= sp.stages) ok = all_ok(tc::mbar_wait_bounded(&sh.empty[st], ph));
            ok = all_ok(ok && !*(volatile int *)&sh.fail);
            if (!ok) break;
            if (leader) {
                const int p0 = (s0 + s) * (kSteps * 16);
                const int b = p0 >> (2 * lgS);
                const int k = (p0 >> lgS) & (S - 1), x = p0 & (S - 1);
                // 128 channels: row k of the order, y = k with lgm = 0
                const int y = (k & ((1 << sp.lgm) - 1)) * d + (k >> sp.lgm);
                const uint32_t sa = base + st * stage;
                expect_tx(&sh.full[st], kDz + kB * sp.nbox * sp.box);
                if (sp.fold) {
                    const int xi = (x >> 7) * sp.fold, yi = y + (dyi - 1) * d;
                    tma_5d(sa, &dzm, 0, xi, 0, y, b, &sh.full[st]);
                    tma_5d(sa + kDz / 2, &dzm, 64, xi, 0, y, b, &sh.full[st]);
                    const uint32_t in0 = sa + kDz + sp.fold * 128;
                    tma_5d(in0, &inm, 0, xi, 0, yi, b, &sh.full[st]);
                    tma_5d(in0 + sp.strip, &inm, 64, xi, 0, yi, b, &sh.full[st]);
                } else {
                    tma_4d(sa, &dzm, 0, x, y, b, &sh.full[st]);
                    tma_4d(sa + kDz / 2, &dzm, 64, x, y, b, &sh.full[st]);
                }
                for (int i = 0; i < kB && !sp.fold; ++i) {
                    const int c = Cin == 128 ? 64 * i : 0;
                    const int yi = y + (Cin == 128 ? dyi - 1 : i - 1) * d;
                    for (int t = 0; t < sp.nbox; ++t)
                        tma_4d(sa + kDz + i * sp.strip + t * sp.box, &inm, c,
                               x + (t - 1) * d, yi, b, &sh.full[st]);
                }
            }
            __syncwarp();
            if (++st == sp.stages) st = 0, ph ^= 1;
        }
        if (leader) {
            if (!ok) atomicOr(&sh.fail, 1);
            sh.issued = s;
        }
        __syncwarp();
    } else if (warp == 5) {
        constexpr uint32_t idesc = tc::idesc_bf16(128, kN) | (1u << 15) | (1u << 16);
        constexpr uint32_t idesc1 = tc::idesc_bf16(128, 16) | (1u << 15) | (1u << 16);
        const uint64_t ad = desc_mn(base, kDz / 2, 1024, 2);
        const uint64_t bd = desc_mn(base + kDz, sp.tap, 8 * kRow, kSwizzle);
        const uint64_t od = desc_mn(base + kWgRoom, 1024, 1024, 2);
        const uint32_t strip16 = (uint32_t)sp.strip >> 4;
        uint32_t row16[kSteps];   // first pixel of each 16 within a strip
#pragma unroll
        for (int j = 0; j < kSteps; ++j)
            row16[j] = (uint32_t)(((16 * j) >> sp.lgw) * sp.pitch +
                                  ((16 * j) & ((1 << sp.lgw) - 1))) * (kRow / 16);
        const bool leader = elect_one();
        int st = 0, s = 0, nb = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (; s < ns; ++s) {
            ok = all_ok(tc::mbar_wait_bounded(&sh.full[st], ph));
            if (!ok) break;
            tc::fence_after_sync();
            const uint32_t off = (uint32_t)st * (stage >> 4);
            const bool bias = Cin != 128 || (s0 + s) % 3 == dyi;
            if (leader) {
#pragma unroll
                for (int j = 0; j < kSteps; ++j)
#pragma unroll
                    for (int i = 0; i < kB; ++i)
                        tc::mma_bf16(tmem + i * kN, ad + off + j * 128,
                                     bd + off + i * strip16 + row16[j], idesc,
                                     s > 0 || j > 0);
                // together: between the others each cost 110 clocks
                if (bias)
#pragma unroll
                    for (int j = 0; j < kSteps; ++j)
                        tc::mma_bf16(tmem + kBiasCol, ad + off + j * 128, od, idesc1,
                                     nb > 0 || j > 0);
                tc::mma_commit(&sh.empty[st]);
            }
            __syncwarp();
            nb += bias;
            if (++st == sp.stages) st = 0, ph ^= 1;
        }
        if (leader) {
            if (!ok) atomicOr(&sh.fail, 1);
            sh.used = s;
            tc::mma_commit(&sh.done);   // arrives once every issued MMA is done
        }
        __syncwarp();
    }
    if (!tc::mbar_wait_bounded(&sh.done, 0)) atomicOr(&sh.fail, 1);
    __syncthreads();
    tc::fence_after_sync();

    if (ns > 0 && !sh.fail) {
        // kPiece columns at a time through shared memory (the stages are free),
        // so that a warp's atomics cover whole sectors
        constexpr int kPiece = Cin == 128 ? 64 : kN;
        constexpr int kLd = kPiece + 4;
        float *stg = reinterpret_cast<float *>(sm);
        const uint32_t lanes = tmem + ((uint32_t)(warp * 32) << 16);
#pragma unroll 1
        for (int q = 0; q < kB * kN / kPiece; ++q) {
            if (warp < 4) {
                float *row = stg + (warp * 32 + lane) * kLd;
                float v[32];
                tc::tmem_ld32(lanes + q * kPiece, v);
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    *reinterpret_cast<float4 *>(row + 4 * j) =
                        make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
                if (Cin == 128) tc::tmem_ld32(lanes + q * kPiece + 32, v);
                else tc::tmem_ld16(lanes + q * kPiece + 32, v);
#pragma unroll
                for (int j = 0; j < (kPiece - 32) / 4; ++j)
                    *reinterpret_cast<float4 *>(row + 32 + 4 * j) =
                        make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
            }
            __syncthreads();
            // piece q: channel half q / 3 of tap (row of taps, q % 3), or row q
            const int col = Cin == 128 ? (dyi * 3 + q % 3) * 128 + (q / 3) * 64 : q * kN;
            for (int e = tid; e < 128 * (kPiece / 4); e += kWgThreads) {
                const int o = e / (kPiece / 4), c = (e - o * (kPiece / 4)) * 4;
                const float4 f = *reinterpret_cast<const float4 *>(stg + o * kLd + c);
                // 16-byte aligned: rows, taps and channels are multiples of four
                atomicAdd(reinterpret_cast<float4 *>(dw + (size_t)o * (9 * Cin) + col + c), f);
            }
            __syncthreads();
        }
        if (warp < 4 && nbias > 0) {
            float v[16];
            tc::tmem_ld16(lanes + kBiasCol, v);
            atomicAdd(db + (blockIdx.y % kSumSlots) * kSums + warp * 32 + lane, v[0]);
        }
    } else if (sh.fail && tid == 0) {
        atomicOr(err, 1u);
        for (int s = sh.used; s < sh.issued; ++s)
            tc::mbar_wait_bounded(&sh.full[s % sp.stages], (s / sp.stages) & 1);
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 4) tc::tmem_dealloc(tmem, kCols);
}

// First layer (16 -> 128 channels): K = 9 taps x 16 channels, one 128 x 128 x
// 16 MMA per tap, in tap order; rows of 32 bytes, 32-byte swizzle.  Bound by
// writing the activations (134 MB at 8 x 256 x 256, 20 us of fallback copy
// bandwidth), so the kernel is built around its epilogue: one persistent CTA
// per SM, the weights loaded once, four tensor-memory accumulators, two groups
// of four epilogue warps on alternate tiles.  A tile's input is three strips
// of 130 pixels, one per row of taps (S >= 128), or nine boxes, one per tap.
// 37.6 us; one tile per CTA, four to an SM, spent its time setting up: 95 us.
constexpr int kC1Tile = 128 * 32;                 // 128 rows x 16 BF16
constexpr int kC1Threads = 320;
constexpr int kC1Stages = 4;

struct C1Shared {
    unsigned long long full[kC1Stages], empty[kC1Stages], wfull;
    unsigned long long tfull[4], tempty[4], done;
    uint32_t tmem_slot;
    int fail, issued, used;
    float bias[128];
};
static_assert(sizeof(C1Shared) <= 1024, "barrier area");

__device__ __forceinline__ uint64_t desc_sw32(uint32_t saddr)
{
    uint64_t d = (uint64_t)((saddr & 0x3ffffu) >> 4);
    d |= (uint64_t)1 << 16;                 // LBO (unused for swizzled K-major)
    d |= (uint64_t)(256 >> 4) << 32;        // SBO: 8 rows x 32 B
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)6 << 61;                 // SWIZZLE_32B
    return d;
}

// kBoxes: 3 strips of 130 pixels (5 KB apart) or 9 boxes of 128 (4 KB).
template <int kBoxes>
__global__ void __launch_bounds__(kC1Threads, 1)
    k_conv1(const __grid_constant__ CUtensorMap act,
            const __grid_constant__ CUtensorMap wts, Epi epi, int S, int lgS, int ntiles,
            uint32_t *err)
{
    constexpr uint32_t kBoxStep = kBoxes == 3 ? 5120 : kC1Tile;
    constexpr uint32_t kBoxTx = kBoxes == 3 ? 130 * 32 : kC1Tile;
    constexpr uint32_t kStage = kBoxes * kBoxStep;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    const uint32_t raw = tc::smem_addr(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    const uint32_t wbase = base + kC1Stages * kStage;
    C1Shared &sh = *reinterpret_cast<C1Shared *>(smem_raw + (base - raw) +
                                                 kC1Stages * kStage + 9 * kC1Tile);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (warp == 8) {
        tc::tmem_alloc(&sh.tmem_slot, 512);
        tc::tmem_relinquish();
    }
    if (tid == 0) {
        for (int i = 0; i < kC1Stages; ++i) {
            tc::mbar_init(&sh.full[i], 1);
            tc::mbar_init(&sh.empty[i], 1);
        }
        tc::mbar_init(&sh.wfull, 1);
        for (int i = 0; i < 4; ++i) {
            tc::mbar_init(&sh.tfull[i], 1);
            tc::mbar_init(&sh.tempty[i], 4);
        }
        tc::mbar_init(&sh.done, 1);
        sh.fail = sh.issued = sh.used = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // the optimiser's step, which writes weights and biases, may be the kernel
    // before this one
    pdl_wait();
    if (tid < 128) sh.bias[tid] = epi.bias[tid];
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = sh.tmem_slot;

    if (warp == 8) {
        // loader
        const bool leader = elect_one();
        if (leader) {
            expect_tx(&sh.wfull, 9 * kC1Tile);
            for (int t = 0; t < 9; ++t)
                tma_2d(wbase + t * kC1Tile, &wts, t * 16, 0, &sh.wfull);
        }
        __syncwarp();
        int g = 0;
        bool ok = true;
        for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++g) {
            const int st = g % kC1Stages;
            if (g >= kC1Stages)
                ok = all_ok(tc::mbar_wait_bounded(&sh.empty[st], ((g / kC1Stages) - 1) & 1));
            ok = all_ok(ok && !*(volatile int *)&sh.fail);
            if (!ok) break;
            if (leader) {
                const int m0 = tile * 128;
                const int b = m0 >> (2 * lgS);
                const int y = (m0 >> lgS) & (S - 1), x = m0 & (S - 1);
                const uint32_t sa = base + st * kStage;
                expect_tx(&sh.full[st], kBoxes * kBoxTx);
                for (int i = 0; i < kBoxes; ++i)
                    tma_4d(sa + i * kBoxStep, &act, 0,
                           x + (kBoxes == 3 ? -1 : i % 3 - 1),
                           y + (kBoxes == 3 ? i - 1 : i / 3 - 1), b, &sh.full[st]);
            }
            __syncwarp();
        }
        if (leader) {
            if (!ok) atomicOr(&sh.fail, 1);
            sh.issued = g;
        }
        __syncwarp();
    } else if (warp == 9) {
        // MMA issuer: tile number g of this CTA accumulates in buffer g mod 4
        constexpr uint32_t idesc = tc::idesc_bf16(128, 128);
        const uint64_t ad = desc_sw32(base), wd = desc_sw32(wbase);
        const bool leader = elect_one();
        int g = 0;
        bool ok = all_ok(tc::mbar_wait_bounded(&sh.wfull, 0));
        for (int tile = blockIdx.x; ok && tile < ntiles; tile += gridDim.x, ++g) {
            const int st = g % kC1Stages, acc = g & 3;
            if (g >= 4) ok = all_ok(tc::mbar_wait_bounded(&sh.tempty[acc], ((g >> 2) - 1) & 1));
            ok = ok && all_ok(tc::mbar_wait_bounded(&sh.full[st], (g / kC1Stages) & 1));
            if (!ok) break;
            tc::fence_after_sync();
            const uint64_t a0 = ad + st * (kStage >> 4);
            if (leader) {
#pragma unroll
                for (int t = 0; t < 9; ++t)
                    tc::mma_bf16(tmem + acc * 128,
                                 a0 + (kBoxes == 3 ? (t / 3) * (kBoxStep >> 4) + (t % 3) * 2
                                                   : t * (kBoxStep >> 4)),
                                 wd + t * (kC1Tile >> 4), idesc, t > 0);
                tc::mma_commit(&sh.empty[st]);
                tc::mma_commit(&sh.tfull[acc]);
            }
            __syncwarp();
        }
        if (leader) {
            if (!ok) atomicOr(&sh.fail, 1);
            sh.used = g;
            tc::mma_commit(&sh.done);   // arrives once every issued MMA is done
        }
        __syncwarp();
    } else {
        // epilogue: warps 0..3 the even tiles of this CTA, 4..7 the odd ones
        const int q = warp & 3;
        for (int g = warp >> 2, tile = blockIdx.x + (warp >> 2) * gridDim.x; tile < ntiles;
             g += 2, tile += 2 * gridDim.x) {
            const int acc = g & 3;
            if (*(volatile int *)&sh.fail ||
                !tc::mbar_wait_bounded(&sh.tfull[acc], (g >> 2) & 1)) {
                atomicOr(&sh.fail, 1);
                break;
            }
            tc::fence_after_sync();
            pair_epilogue<kFwd>(epi, sh.bias, nullptr,
                                tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * 128),
                                (size_t)tile * 128 + q * 32 + lane,
                                make_uint4(0, 0, 0, 0));
            tc::fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.tempty[acc]);
        }
    }
    __syncthreads();
    if (tid == 0) {
        if (sh.fail) {
            atomicOr(err, 1u);
            // copies issued but never consumed must land before the CTA leaves
            tc::mbar_wait_bounded(&sh.wfull, 0);
            for (int g = sh.used; g < sh.issued; ++g)
                tc::mbar_wait_bounded(&sh.full[g % kC1Stages], (g / kC1Stages) & 1);
        }
        tc::mbar_wait_bounded(&sh.done, 0);
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (warp == 8) tc::tmem_dealloc(tmem, 512);
}

// --- host: tensor maps ------------------------------------------------------

PFN_cuTensorMapEncodeTiled_v12000 encoder()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        cudaDriverEntryPointQueryResult q;
        void *p = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000,
                                             cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    });
    return fn;
}

// NHWC activations [n][S][S][128] BF16; box 64 channels x `pix` pixels
// (a run of one row, or whole rows when S < pix).
bool map_act(CUtensorMap *m, const uint16_t *ptr, int n, int S, int pix = 128)
{
    auto fn = encoder();
    if (!fn) return false;
    const cuuint64_t dims[4] = {128, (cuuint64_t)S, (cuuint64_t)S, (cuuint64_t)n};
    const cuuint64_t strides[3] = {256, (cuuint64_t)S * 256, (cuuint64_t)S * S * 256};
    const cuuint32_t bx = S >= 128 || S >= pix ? pix : S, by = pix / bx;
    const cuuint32_t box[4] = {64, bx, by, 1};
    const cuuint32_t es[4] = {1, 1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<uint16_t *>(ptr), dims,
              strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Strips of the pair convolution.  Three taps share a strip when a CTA's 128
// pixels lie in one row (S >= 128) and its stages fit: two strips serve a row
// of taps, and with four the next row's are on their way (dilations up to 16:
// 84.5 us a layer at 8 x 256 x 256; three strips of 192 pixels, d = 32, took 126
// and a box per tap, d = 64, 135).  Combs stream 128 pixels per strip whatever d
// and fit three or four from d = 32 on (85.8 and 110 us); their teeth are 128 d
// / S pixels wide and whole 1 KB groups.  Columns do the same for S < 128 while
// d < S and three fit (32 x 32 x 32: 14.2 us a layer, 15.7 with a box per tap).
StripShape conv_shape(int S, int d)
{
    StripShape sp{};
    sp.taps = 3;
    const auto gapped = [&](int step) {   // stages between gaps of >= step pixels
        sp.step = step;
        sp.gap = (step + 7) / 8 * 8;
        sp.px = 128 + sp.gap;
        sp.na = std::min(4, (kStripRoom - sp.gap * 128) / (sp.px * 128));
    };
    if (S < 128) {
        const int rows = 128 / S;
        gapped(d * rows);
        sp.fold = rows;
        sp.outer = 1;
        sp.inner = S;
        sp.cols = 1;
        if (d < S && sp.na >= 3) return sp;
    } else {
        const int tooth = 128 * d / S, px = 128 + (2 * d + 7) / 8 * 8;
        const int na = std::min(4, kStripRoom / (px * 128));
        if (na < 4 && d < S && tooth >= 8) {
            gapped(tooth);
            sp.fold = tooth;
            sp.outer = d;
            sp.inner = 1;
            if (sp.na >= 3 && sp.na >= na) return sp;
        }
        sp = StripShape{};
        sp.taps = 3;
        sp.px = px;
        sp.na = na;
        if (na >= 3) return sp;
    }
    sp = StripShape{};
    sp.taps = 1;
    sp.px = 128;
    sp.na = kMaxA;
    return sp;
}

// NHWC activations of 128 channels for a gapped strip: combs split x into (x mod
// d, x / d), box 64 channels x one tooth at all S / d multiples of one row;
// columns take y before x, box 64 channels x 128 / S rows x S columns.
bool map_gapped(CUtensorMap *m, const uint16_t *ptr, int n, int S, int d,
                const StripShape &sp)
{
    auto fn = encoder();
    if (!fn) return false;
    const cuuint64_t row = (cuuint64_t)S * 256, img = (cuuint64_t)S * row;
    const cuuint64_t N = (cuuint64_t)n, s = (cuuint64_t)S;
    const cuuint64_t teeth = sp.cols ? s : (cuuint64_t)(S / d);
    const cuuint64_t dims[5] = {128, sp.cols ? s : (cuuint64_t)d, teeth, sp.cols ? 1 : s, N};
    const cuuint64_t strides[4] = {sp.cols ? row : 256,
                                   sp.cols ? 256 : (cuuint64_t)d * 256,
                                   sp.cols ? img : row, img};
    const cuuint32_t box[5] = {64, (cuuint32_t)sp.fold, (cuuint32_t)teeth, 1, 1};
    const cuuint32_t es[5] = {1, 1, 1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<uint16_t *>(ptr), dims,
              strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// NHWC tensor of 128 (box 64, 128-byte swizzle) or 16 channels (32-byte
// swizzle); box w x h pixels.
bool map_nhwc(CUtensorMap *m, const uint16_t *ptr, int ch, int n, int S, int w, int h)
{
    auto fn = encoder();
    if (!fn) return false;
    const cuuint64_t row = (cuuint64_t)ch * 2;
    const cuuint64_t dims[4] = {(cuuint64_t)ch, (cuuint64_t)S, (cuuint64_t)S, (cuuint64_t)n};
    const cuuint64_t strides[3] = {row, (cuuint64_t)S * row, (cuuint64_t)S * S * row};
    const cuuint32_t box[4] = {ch == 128 ? 64u : 16u, (cuuint32_t)w, (cuuint32_t)h, 1};
    const cuuint32_t es[4] = {1, 1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<uint16_t *>(ptr), dims,
              strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
              ch == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_32B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Slabs and strips of the weight gradient: 128 pixels where two stages fit,
// else 64.  Rows of more than a slab are taken as combs (k_conv_pair) where the
// teeth are whole 1 KB groups: 64 KB a slab whatever d, where strips of
// neighbours take 32 KB + 256 (128 + 2 d) bytes (training step at S = 256: 2075 us
// with strips, 2069 with combs of 16 pixels or more, 2060 with combs of 8).
WgradShape wgrad_shape(int S, int d, int cin)
{
    const int strips = cin == 128 ? 2 : 3, row = cin == 128 ? 128 : 32;
    if (cin == 128 && S >= 256 && d < S && S % d == 0 && 128 * d / S >= 8) {
        WgradShape sp{};
        sp.L = 128;
        sp.lgw = 7;
        sp.fold = 128 * d / S;
        sp.pitch = 128 + 2 * sp.fold;
        sp.nbox = 1;
        sp.box = 128 * 128;
        sp.tap = sp.fold * 128;
        sp.strip = sp.pitch * 128;
        sp.stages = std::min(kMaxWgStages, kWgRoom / (128 * 256 + 2 * sp.strip));
        while (d << sp.lgm < S) ++sp.lgm;
        if (sp.stages >= 2) return sp;
    }
    for (int L = 128;; L = 64) {
        WgradShape sp{};
        const int w = S < L ? S : L, R = L / w;
        sp.L = L;
        while ((1 << sp.lgw) < w) ++sp.lgw;
        const bool one = w + 2 * d <= 256 && w + 2 * d < 3 * w;
        sp.pitch = one ? w + 2 * d : w;
        sp.nbox = one ? 1 : 3;
        sp.box = R * sp.pitch * row;
        sp.tap = one ? d * row : sp.box;
        sp.strip = (sp.nbox * sp.box + 1023) / 1024 * 1024;
        sp.stages = std::min(kMaxWgStages, kWgRoom / (L * 256 + strips * sp.strip));
        if (w == L && cin == 128) {   // chains of S / d rows
            while ((d << (sp.lgm + 1)) <= S) ++sp.lgm;
            if (d << sp.lgm != S) sp.lgm = 0;
        }
        if (sp.stages >= 2 || L == 64) return sp;
    }
}

// First-layer weights [128 rows][144] BF16; box 16 x 128.
bool map_w144(CUtensorMap *m, const uint16_t *ptr)
{
    auto fn = encoder();
    if (!fn) return false;
    const cuuint64_t dims[2] = {144, 128};
    const cuuint64_t strides[1] = {144 * 2};
    const cuuint32_t box[2] = {16, 128};
    const cuuint32_t es[2] = {1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<uint16_t *>(ptr), dims,
              strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_32B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Weights [128 rows][1152] BF16; box 64 x 64 (one CTA's half of a slab).
bool map_wts(CUtensorMap *m, const uint16_t *ptr)
{
    auto fn = encoder();
    if (!fn) return false;
    const cuuint64_t dims[2] = {1152, 128};
    const cuuint64_t strides[1] = {1152 * 2};
    const cuuint32_t box[2] = {64, 64};
    const cuuint32_t es[2] = {1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<uint16_t *>(ptr), dims,
              strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace convtma

// Forward (mode 0: out = ReLU(conv(in) + bias)) or input gradient (mode 1:
// out = conv^T(in), zero where the layer below's bits are) of a 128 -> 128 layer
// over n samples; forward with bits writes its own (Epi)
// (head: forward only, the network's head on the result)
// of S x S (S a power of two >= 16).  `w` is W[o][t][i] (forward) or
// Wt[i][t][o] (input gradient), 16-byte aligned.
cudaError_t launch_conv_tma(int mode, const uint16_t *in, const uint16_t *w,
                            const float *bias, uint4 *bits, uint16_t *out,
                            int n, int S, int lgS, int d, const HeadArgs *head,
                            uint32_t *err, cudaStream_t st)
{
    using namespace convtma;
    if (S < 16 || (S & (S - 1)) || ((uintptr_t)in & 15) || ((uintptr_t)w & 15))
        return cudaErrorInvalidValue;
    const StripShape sp = conv_shape(S, d);
    CUtensorMap ma, mw;
    if (!(sp.step ? map_gapped(&ma, in, n, S, d, sp) : map_act(&ma, in, n, S, sp.px)) ||
        !map_wts(&mw, w))
        return cudaErrorInvalidValue;
    Epi e{bias, bits, out, head ? *head : HeadArgs{}};
    int dev = 0, nsm = 0;
    cudaError_t attr = cudaGetDevice(&dev);
    if (attr == cudaSuccess)
        attr = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    using Kernel = decltype(&k_conv_pair<3, kFwd, true>);
    static const Kernel kerns[3][3] = {   // mode x (boxes, strips, combs)
        {k_conv_pair<1, kFwd, false>, k_conv_pair<3, kFwd, false>,
         k_conv_pair<3, kFwd, true>},
        {k_conv_pair<1, kDgrad, false>, k_conv_pair<3, kDgrad, false>,
         k_conv_pair<3, kDgrad, true>},
        {k_conv_pair<1, kFwdHead, false>, k_conv_pair<3, kFwdHead, false>,
         k_conv_pair<3, kFwdHead, true>}};
    const Kernel kern = kerns[mode != 0 ? kDgrad : head ? kFwdHead : kFwd]
                             [sp.step ? 2 : sp.taps == 3 ? 1 : 0];
    if (attr == cudaSuccess)
        attr = cudaFuncSetAttribute(
            kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kPairSmem);
    if (attr != cudaSuccess) return attr;
    // S >= 16: whole pairs of 128-pixel tiles
    const int npairs = (int)((long long)n * S * S / 256);
    return launch_pdl(kern, dim3(2 * std::min(npairs, nsm / 2)), kPairThreads, kPairSmem, st,
                      ma, mw, e, sp, S, lgS, d, mode == 0 ? 1 : -1, npairs, err);
}

// Weight gradient, added into dw[128][9 cin] (FP32, cleared by the caller), and
// bias gradient, added into db[128] of kSumSlots slots, of a layer of cin = 16 or
// 128 input channels: dz [n][S][S][128] and in [n][S][S][cin] BF16, S a power of two >=
// 16; the pixel range is split over the SMs.
cudaError_t launch_wgrad_tma(const uint16_t *dz, const uint16_t *in, int cin, float *dw,
                             float *db, int n, int S, int lgS, int d, uint32_t *err,
                             cudaStream_t st)
{
    using namespace convtma;
    if (S < 16 || (S & (S - 1)) || (cin != 16 && cin != 128) || ((uintptr_t)dz & 15) ||
        ((uintptr_t)in & 15) || ((uintptr_t)dw & 15))
        return cudaErrorInvalidValue;
    const WgradShape sp = wgrad_shape(S, d, cin);
    CUtensorMap mz, mi;
    const int w = 1 << sp.lgw;
    StripShape comb{};
    comb.fold = sp.fold;
    if (sp.fold ? !map_gapped(&mz, dz, n, S, d, comb) || !map_gapped(&mi, in, n, S, d, comb)
                : !map_nhwc(&mz, dz, 128, n, S, w, sp.L / w) ||
                      !map_nhwc(&mi, in, cin, n, S, sp.pitch, sp.L / w))
        return cudaErrorInvalidValue;
    const bool eight = sp.L == 128;
    const auto kern = cin == 128 ? (eight ? k_wgrad_strip<128, 8> : k_wgrad_strip<128, 4>)
                                 : (eight ? k_wgrad_strip<16, 8> : k_wgrad_strip<16, 4>);
    int dev = 0, nsm = 0;
    cudaError_t attr = cudaGetDevice(&dev);
    if (attr == cudaSuccess)
        attr = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const int smem = 227 * 1024;
    if (attr == cudaSuccess)
        attr = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (attr != cudaSuccess) return attr;
    const int total = (int)((long long)n * S * S / sp.L);
    const int rows = cin == 128 ? 3 : 1;   // rows of taps, one per CTA
    const int per = (total + nsm / rows - 1) / (nsm / rows);
    return launch_pdl(kern, dim3(rows, (total + per - 1) / per), kWgThreads, smem, st, mz, mi,
                      dw, db, S, lgS, d, sp, total, per, err);
}

// First layer forward: out = ReLU(conv3x3(x, W1) + b1) for x [n][S][S][16]
// and W1 [128][9][16] (BF16, 16-byte aligned), S a power of two >= 16.
cudaError_t launch_conv1_tma(const uint16_t *x, const uint16_t *w, const float *bias,
                             uint16_t *out, uint4 *bits, int n, int S, int lgS,
                             uint32_t *err, cudaStream_t st)
{
    using namespace convtma;
    if (S < 16 || (S & (S - 1)) || ((uintptr_t)x & 15) || ((uintptr_t)w & 15))
        return cudaErrorInvalidValue;
    CUtensorMap ma, mw;
    const bool strips = S >= 128;   // a tile lies in one row
    const int bw = strips ? 130 : (S < 128 ? S : 128);
    if (!map_nhwc(&ma, x, 16, n, S, bw, strips ? 1 : 128 / bw) || !map_w144(&mw, w))
        return cudaErrorInvalidValue;
    Epi e{bias, bits, out, HeadArgs{}};
    const auto kern = strips ? k_conv1<3> : k_conv1<9>;
    const int smem = kC1Stages * (strips ? 3 * 5120 : 9 * kC1Tile) + 9 * kC1Tile + 2048;
    int dev = 0, nsm = 0;
    cudaError_t attr = cudaGetDevice(&dev);
    if (attr == cudaSuccess)
        attr = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (attr == cudaSuccess)
        attr = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (attr != cudaSuccess) return attr;
    const int ntiles = (int)((long long)n * S * S / 128);
    return launch_pdl(kern, dim3(std::min(ntiles, nsm)), kC1Threads, smem, st, ma, mw, e, S,
                      lgS, ntiles, err);
}

}  // namespace fire
