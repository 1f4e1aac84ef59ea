// labs_net.cu -- the learned proposal network (the library's addition: the paper has no
// learned component).  BF16 operands with FP32 accumulation on the 5th-generation tensor
// cores (tcgen05.mma, accumulators in TMEM, operands staged by TMA), hand-written
// forward, backward, loss and AdamW kernels.
//
// Network, per state of n free variables (positions p = 0..n-1):
//   x (3 features per position, padded to 16 channels)
//   a1..a3 = relu(conv(a_{l-1}) + b_l): Conv1d, 64 output channels, 7 taps, zero padding 3
//   h      = relu(W4 a3 + b4) per position;  score_p = w5 . h_p + b5   (flip score)
//   restart = w6 . mean_p(a3_p) + b6                                   (restart score)
// Loss per sample: wf * CE(softmax(score), t) + 0.5 (restart - y)^2, batch mean.
//
// Tiles.  A tile holds as many whole samples as fit 128 output rows (256 for n > 128) with
// three zero rows between them (the convolutions' padding), so nothing crosses a tile: one
// CTA carries it through all layers without leaving shared memory.  A tile's activations
// are kept as 16-byte rows of 8 channels, one column of rows per 8 channels ([column][row],
// rows 0-2 zero, row o+3 output row o), in shared and in global memory alike:
//   - as the K-major operand of a product over channels, tap k of a convolution is the same
//     operand with its start address 16 k bytes further;
//   - as the MN-major operand of a weight gradient (the reduction runs over rows), the same
//     columns serve without a transpose;
//   - a tile moves between global and shared memory as one contiguous copy.
// Weights are packed per layer as [K/8][64 outputs][8] bf16, the K-major layout of the second
// operand; the backward-data products use the tap-reversed transpose.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <mutex>

#include "labs_internal.cuh"
#include "labs_tc.cuh"
#include "labs_nvtx.h"

namespace labsgpu {
namespace net {

using bf16 = __nv_bfloat16;

constexpr int kC = 64, kTaps = 7, kCin = 16;
constexpr int oW1 = 0, oB1 = oW1 + kC * kCin * kTaps, oW2 = oB1 + kC, oB2 = oW2 + kC * kC * kTaps, oW3 = oB2 + kC,
              oB3 = oW3 + kC * kC * kTaps, oW4 = oB3 + kC, oB4 = oW4 + kC * kC, oW5 = oB4 + kC, oB5 = oW5 + kC,
              oW6 = oB5 + 1, oB6 = oW6 + kC, kParams = oB6 + 1;
// packed bf16 operand copies (element offsets)
constexpr int pWf1 = 0, pWf2 = pWf1 + kC * kTaps * kCin, pWf3 = pWf2 + kC * kTaps * kC, pWf4 = pWf3 + kC * kTaps * kC,
              pWb2 = pWf4 + kC * kC, pWb3 = pWb2 + kC * kTaps * kC, pWb4 = pWb3 + kC * kTaps * kC, pW5 = pWb4 + kC * kC,
              pW6 = pW5 + kC, kPacked = pW6 + kC;

namespace {

constexpr int kTcThreads = 128;  // threads of a tile group: one TMEM lane (output row) each

// Attempts of the kernels' waits, by what is waited for (a test builds this file with none).
// A wait that gives up is repeated once, with kWaitTries attempts, so that nothing is left under
// way where that can be helped; then it marks a word of its tile group's that the group's
// threads read only between two of their barriers which no such mark can come between, so that
// they leave together; and it sets the pass's error word.  (A reduction in the group's barriers
// instead of the mark took 1 to 2% of a pass, a test around the epilogue after a wait up to 25%
// in spilled registers: until the group leaves, its epilogues run on whatever there is.)
#ifndef LABS_NET_TRIES_WEIGHTS
#define LABS_NET_TRIES_WEIGHTS kWaitTries
#endif
#ifndef LABS_NET_TRIES_TILES
#define LABS_NET_TRIES_TILES kWaitTries
#endif
#ifndef LABS_NET_TRIES_PRODUCTS
#define LABS_NET_TRIES_PRODUCTS kWaitTries
#endif
constexpr int kTriesWeights = LABS_NET_TRIES_WEIGHTS, kTriesTiles = LABS_NET_TRIES_TILES,
              kTriesProducts = LABS_NET_TRIES_PRODUCTS;

// A tile of MT x 128 output rows.
template <int MT>
struct Tile {
    static constexpr int M = 128 * MT;
    static constexpr int RP = M + 9;            // rows per column: 3 zero rows on each side, 1 (mod 8) rows
                                                // so that the columns of a row use different banks
    static constexpr int COL = RP * 16;         // bytes per column
    static constexpr int ACT = 8 * COL;         // bytes of 64 channels
};

__host__ __device__ inline int tile_rows(int n) { return n <= 128 ? 128 : 256; }
__host__ __device__ inline int tile_samples(int n) { return (tile_rows(n) + 3) / (n + 3); }
__host__ __device__ inline int64_t tile_count(int64_t B, int n)
{
    const int k = tile_samples(n);
    return (B + k - 1) / k;
}

// Where an output row of a tile stands: its sample (of the tile) and position, in if it is
// one.
struct RowPos {
    int k, p;
    bool in;
    __device__ RowPos(int o, int n, int K) : k(o / (n + 3)), p(o % (n + 3)), in(false) { in = p < n && k < K; }
};

__device__ __forceinline__ void group_sync(int id)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(kTcThreads) : "memory");
}

__device__ __forceinline__ uint32_t pack2(float a, float b)
{
    const __nv_bfloat162 r = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&r);
}
__device__ __forceinline__ float lo_f(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float hi_f(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

__device__ __forceinline__ void sts128(uint32_t a, uint4 v)
{
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ uint4 lds128(uint32_t a)
{
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "r"(a)
                 : "memory");
    return v;
}

__device__ __forceinline__ float4 lds_f4(uint32_t a)
{
    const uint4 v = lds128(a);
    return make_float4(__uint_as_float(v.x), __uint_as_float(v.y), __uint_as_float(v.z), __uint_as_float(v.w));
}

// Instruction descriptor of kind::f16 with both operands MN-major (bits 15 and 16).
__host__ __device__ constexpr uint32_t idesc_bf16_f32_mn(int M, int N)
{
    return idesc_bf16_f32(M, N) | (1u << 15) | (1u << 16);
}

// D (128 rows, 64 columns at TMEM address d) = TAPS-tap product of the rows from byte
// address a (column pitch COL) with the packed weights at w.  One warp, uniform arguments.
template <int CIN, int TAPS, int COL>
__device__ __forceinline__ void issue_product(uint32_t elected, uint32_t d, uint32_t a, uint32_t w)
{
    constexpr uint32_t id = idesc_bf16_f32(128, kC);
    const uint64_t ad = smem_desc(a, COL, 128), wd = smem_desc(w, 1024, 128);  // addresses in 16-byte units
#pragma unroll
    for (int k = 0; k < TAPS; ++k)
#pragma unroll
        for (int s2 = 0; s2 < CIN / 16; ++s2)
            tc_mma_bf16(elected, d, ad + (k + 2 * s2 * (COL / 16)), wd + (k * (CIN / 8) + 2 * s2) * 64, id, (k | s2) != 0);
}

// D (128 x 64 at TMEM address d) += over the rows r < M: A columns (16 of them, pitch COL,
// from address a) x G columns (8, from address g): a weight gradient, both operands
// MN-major (the next 8 rows 128 bytes on, the next 8 channels one column on).
template <int M, int COL>
__device__ __forceinline__ void issue_wgrad(uint32_t elected, uint32_t d, uint32_t a, uint32_t g, bool fresh)
{
    constexpr uint32_t id = idesc_bf16_f32_mn(128, kC);
    const uint64_t ad = smem_desc(a, 128, COL), gd = smem_desc(g, 128, COL);
#pragma unroll
    for (int ks = 0; ks < M / 16; ++ks) tc_mma_bf16(elected, d, ad + 16 * ks, gd + 16 * ks, id, !fresh || ks > 0);
}

// This thread's 64 accumulators (TMEM lane 32 (warp mod 4) + lane).
__device__ __forceinline__ void load_acc(uint32_t d, int wq, float (&acc)[64])
{
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        float v[16];
        tmem_ld16(d + ((uint32_t)(32 * wq) << 16) + 16 * q, v);
#pragma unroll
        for (int i = 0; i < 16; ++i) acc[16 * q + i] = v[i];
    }
    tc_wait_ld();
}

// Sums v over the warp's 32 lanes: lane l returns the sums of entries 2l and 2l+1 (each
// round exchanges half of what a lane still holds).
__device__ __forceinline__ float2 warp_colsum(float (&v)[64], int lane)
{
#pragma unroll
    for (int h = 32, off = 16; h >= 2; h >>= 1, off >>= 1) {
        const bool up = (lane & off) != 0;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const float keep = up ? v[i + h] : v[i], give = up ? v[i] : v[i + h];
            v[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, give, off);
        }
    }
    return make_float2(v[0], v[1]);
}

__device__ __forceinline__ void add2(float2& a, float2 b)
{
    a.x += b.x;
    a.y += b.y;
}

// Adds a lane's channel sums (2 lane, 2 lane + 1) to the CTA's.
__device__ __forceinline__ void add_channels(float* sums, int lane, float2 v)
{
    atomicAdd(sums + 2 * lane, v.x);
    atomicAdd(sums + 2 * lane + 1, v.y);
}

// ------------------------------------------------------------------ forward
//
// One kernel from the inputs to the scores: conv1..3, the MLP and the heads of a tile stay
// in shared memory (a convolution's result overwrites its input once its product has
// completed), the weights of all layers are loaded once per CTA.  NG tile groups of 128
// threads share a CTA and its weights, each with its own tile, accumulators and barriers,
// so one group's epilogue runs beside another's products.  TRAIN goes on to the loss and the
// gradients that need the scores of whole samples: the softmax, dh, the MLP's and the heads'
// gradients and da3; a1, a2 and da3 go to global memory for the convolutions' backward
// kernels, a3 and h never leave the CTA.
//
// What bounds it: shared-memory bandwidth -- the products read 6 KB per 128 x 64 x 16
// product, 67 products a tile, and the epilogues about a third as much again (8192 samples
// of n = 128: 157 us; the products alone would take 110).  It replaces one launch per layer
// over global activations (70 MB read and written per layer of 4096 samples) that a memset
// cleared before every pass: scoring 8192 states 172 us with the features, from 950.
template <int MT, bool TRAIN>
struct FwdShape {
    using T = Tile<MT>;
    static constexpr int NG = TRAIN ? (MT == 1 ? 2 : 1) : (MT == 1 ? 3 : 2);
    static constexpr int THREADS = NG * kTcThreads;
    static constexpr int W1 = 0, W2 = W1 + kTaps * kCin * 128, W3 = W2 + kTaps * kC * 128, W4 = W3 + kTaps * kC * 128,
                         WB4 = W4 + kC * 128, W_END = TRAIN ? WB4 + kC * 128 : WB4;
    static constexpr int X0 = 0, ACT = 2 * T::COL, DH = ACT + T::ACT;  // within a group
    static constexpr int GROUP = TRAIN ? DH + T::ACT : DH;
    static constexpr int GROUPS = W_END;
    static constexpr int MISC = GROUPS + NG * GROUP;
    // misc: biases b1..b4, w5, w6 (float), barriers, the TMEM slot; then per group scores and ds
    // (M floats each) and dr per sample (M/4 floats), the CTA's sums of b3, b4, w5, w6 gradients
    static constexpr int BIAS = MISC, BAR = BIAS + 6 * kC * 4, SC = BAR + 64;
    static constexpr int SCB = (2 * T::M + T::M / 4 + 32) * 4;
    static constexpr int SUMS = SC + (TRAIN ? NG * SCB : 0);
    static constexpr int SMEM = SUMS + (TRAIN ? 4 * kC * 4 : 0) + 128;  // + alignment slack
    // Accumulators of dW4 per group, taken in turn by its tiles: two per SM either way.  A chain
    // of products loses what the tensor core's additions round toward zero, so it is kept as
    // short as two CTAs per SM had it (one accumulator above n = 128 made it twice as long).
    static constexpr int ACC4 = 2 / NG > 1 ? 2 / NG : 1;
    static constexpr int TMEM_USED = NG * MT * 64 + (TRAIN ? NG * ACC4 * 64 : 0);
    static constexpr int TMEM = TMEM_USED <= 128 ? 128 : 256;
};

// A wait gave up: the pass's error word (its gradients become NaN) and, in a walk, the
// context's status.
__device__ __forceinline__ void net_failed(int* err, DevStatus* status)
{
    atomicExch(err, 1);
    if (status != nullptr) atomicCAS(&status->error, 0, LABS_ECUDA);
}

struct FwdArgs {
    const float* x;
    const bf16* wpk;
    const float* prm;
    float* score;
    float* restart;
    int* err;
    DevStatus* status;  // of the walk's context, or null
    int64_t B;
    int n;
    // training
    const int32_t* target;
    const float* y;
    const float* wf;
    bf16 *X0, *A1, *A2, *dA3;  // tiles in global memory
    float* part4;              // [accumulator x CTA x group][64 channels][64 outputs] partial dW4
    float* grad;
    float* loss;
};

// Row o of a tile: 64 bf16 values (as 32 words) to the columns at address col (this row's
// first 16 bytes) and, when g is given, to the same place of a tile in global memory.
template <int COL>
__device__ __forceinline__ void store_row(uint32_t col, unsigned char* g, const uint32_t (&w)[32])
{
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const uint4 v = make_uint4(w[4 * c], w[4 * c + 1], w[4 * c + 2], w[4 * c + 3]);
        if (col != 0u) sts128(col + c * COL, v);
        if (g != nullptr) *reinterpret_cast<uint4*>(g + c * COL) = v;
    }
}

// Zero rows of a tile in global memory (rows outside its output rows), by the first threads
// of a group.
template <int MT, int COLS>
__device__ __forceinline__ void zero_pad_rows(unsigned char* g, int t)
{
    if (t < 9) {
        const int r = t < 3 ? t : Tile<MT>::M + t;
#pragma unroll
        for (int c = 0; c < COLS; ++c) *reinterpret_cast<uint4*>(g + c * Tile<MT>::COL + 16 * r) = make_uint4(0u, 0u, 0u, 0u);
    }
}

template <int MT, bool TRAIN>
__global__ void __launch_bounds__(FwdShape<MT, TRAIN>::THREADS, 1) net_forward_kernel(FwdArgs a)
{
    using S = FwdShape<MT, TRAIN>;
    using T = Tile<MT>;
    extern __shared__ unsigned char tc_smem_raw[];
    unsigned char* sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(tc_smem_raw) + 127) & ~uintptr_t(127));
    const uint32_t sb = smem_addr(sm);
    const int t = threadIdx.x % kTcThreads, grp = threadIdx.x / kTcThreads, wq = t >> 5, lane = t & 31;
    float* bias = reinterpret_cast<float*>(sm + S::BIAS);
    const uint32_t s_bias = sb + S::BIAS;
    const uint32_t bar_w = sb + S::BAR, bar = bar_w + 8 + 8 * grp, slot = sb + S::BAR + 48;
    volatile int* failed = reinterpret_cast<volatile int*>(sm + S::BAR + 32) + grp;  // the group's mark
    const uint32_t gx = sb + S::GROUPS + grp * S::GROUP + S::X0, ga = sb + S::GROUPS + grp * S::GROUP + S::ACT,
                   gd = sb + S::GROUPS + grp * S::GROUP + S::DH;
    float* s_score = reinterpret_cast<float*>(sm + S::SC + grp * S::SCB);
    float* s_ds = s_score + T::M;
    float* s_dr = s_ds + T::M;
    float* sums = reinterpret_cast<float*>(sm + S::SUMS);  // b3, b4, w5, w6
    const int n = a.n, K = tile_samples(n);
    const int64_t tiles = tile_count(a.B, n);

    for (int i = threadIdx.x; i < kC; i += S::THREADS) {
        bias[i] = a.prm[oB1 + i];
        bias[kC + i] = a.prm[oB2 + i];
        bias[2 * kC + i] = a.prm[oB3 + i];
        bias[3 * kC + i] = a.prm[oB4 + i];
        bias[4 * kC + i] = __bfloat162float(a.wpk[pW5 + i]);
        bias[5 * kC + i] = __bfloat162float(a.wpk[pW6 + i]);
    }
    if (TRAIN)
        for (int i = threadIdx.x; i < 4 * kC; i += S::THREADS) sums[i] = 0.f;
    for (int i = threadIdx.x; i < S::NG * S::GROUP / 16; i += S::THREADS)
        sts128(sb + S::GROUPS + 16 * i, make_uint4(0u, 0u, 0u, 0u));
    if (threadIdx.x < 32) tmem_alloc(slot, S::TMEM);
    if (t == 0) *failed = 0;
    if (threadIdx.x == 0) {
        mbar_init(bar_w, 1);
        for (int g = 0; g < S::NG; ++g) mbar_init(bar_w + 8 + 8 * g, 1);
        mbar_init_fence();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(sm + S::BAR + 48);
    const uint32_t acc0 = tmem + grp * MT * 64, acc4 = tmem + S::NG * MT * 64 + grp * S::ACC4 * 64;
    // the group's first warp issues its products, from uniform values
    const bool issuer = uniform(wq) == 0;
    const uint32_t u_sb = uniform(sb), u_gx = uniform(gx), u_ga = uniform(ga), u_bar = uniform(bar), u_acc0 = uniform(acc0),
                   u_acc4 = uniform(acc4);
    if (threadIdx.x == 0) {
        mbar_arrive_expect_tx(bar_w, S::W_END);
        bulk_copy_g2s(sb + S::W1, a.wpk + pWf1, S::W2 - S::W1, bar_w);
        bulk_copy_g2s(sb + S::W2, a.wpk + pWf2, S::W3 - S::W2, bar_w);
        bulk_copy_g2s(sb + S::W3, a.wpk + pWf3, S::W4 - S::W3, bar_w);
        bulk_copy_g2s(sb + S::W4, a.wpk + pWf4, kC * 128, bar_w);
        if (TRAIN) bulk_copy_g2s(sb + S::WB4, a.wpk + pWb4, kC * 128, bar_w);
    }
    bool ok = !__syncthreads_or(!mbar_wait(bar_w, 0, kTriesWeights));
    uint32_t phase = 0;
    int done = 0;           // tiles of this group
    float2 gw6 = {0.f, 0.f};  // this warp's samples: the gradients of w6's channels 2 lane and 2 lane + 1
    float gb5 = 0.f, gb6 = 0.f, lsum = 0.f;
    const float inv = TRAIN ? 1.f / (float)a.B : 0.f;

    // this thread's output rows: sample of the tile (K: none) and position
    int rk[MT], rpos[MT];
#pragma unroll
    for (int mt = 0; mt < MT; ++mt) {
        const RowPos rp(t + 128 * mt, n, K);
        rk[mt] = rp.in ? rp.k : -1;
        rpos[mt] = rp.p;
    }
    // the group's inputs of a tile: three features per row
    float xin[MT][3];
    auto fetch = [&](int64_t tile) {
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
            const int64_t b = tile * K + rk[mt];
            const bool in = rk[mt] >= 0 && tile < tiles && b < a.B;
#pragma unroll
            for (int f = 0; f < 3; ++f) xin[mt][f] = in ? a.x[(b * 3 + f) * n + rpos[mt]] : 0.f;
        }
    };
    // waits for the group's products; a wait that gives up ends the group's work with this tile
    auto wait_products = [&]() {
        if (!mbar_wait(bar, phase, kTriesProducts)) {
            mbar_wait(bar, phase);
            *failed = 1;
        }
        phase ^= 1;
        tc_fence_after();
    };
    // the epilogue's shared-memory rows are visible to the next product, the accumulators read
    auto rows_ready = [&]() {
        fence_async_shared();
        tc_fence_before();
        group_sync(1 + grp);
        tc_fence_after();
    };

    const int64_t stride = (int64_t)gridDim.x * S::NG;
    int64_t tile = (int64_t)grp * gridDim.x + blockIdx.x;
    fetch(tile);
    for (; tile < tiles && ok; tile += stride, ++done) {
        unsigned char* const gA1 = TRAIN ? reinterpret_cast<unsigned char*>(a.A1) + tile * T::ACT : nullptr;
        unsigned char* const gA2 = TRAIN ? reinterpret_cast<unsigned char*>(a.A2) + tile * T::ACT : nullptr;
        unsigned char* const gA3 = TRAIN ? reinterpret_cast<unsigned char*>(a.dA3) + tile * T::ACT : nullptr;
        if (TRAIN) {
            zero_pad_rows<MT, 8>(gA1, t);
            zero_pad_rows<MT, 8>(gA2, t);
            zero_pad_rows<MT, 8>(gA3, t);
            zero_pad_rows<MT, 1>(reinterpret_cast<unsigned char*>(a.X0) + tile * T::COL, t);
        }
        bool in[MT];
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
            const int o = t + 128 * mt;
            in[mt] = rk[mt] >= 0 && tile * K + rk[mt] < a.B;
            const uint4 v = make_uint4(pack2(xin[mt][0], xin[mt][1]), pack2(xin[mt][2], 0.f), 0u, 0u);
            sts128(gx + 16 * (o + 3), v);
            if (TRAIN) *reinterpret_cast<uint4*>(reinterpret_cast<unsigned char*>(a.X0) + tile * T::COL + 16 * (o + 3)) = v;
        }
        rows_ready();
        if (issuer) {
            const uint32_t el = elect_one();
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
                issue_product<kCin, kTaps, T::COL>(el, u_acc0 + 64 * mt, u_gx + 2048 * mt, u_sb + S::W1);
            tc_commit(el, u_bar);
        }
        fetch(tile + stride);
        // conv1..3: bias, ReLU, the rows replace the layer's input
#pragma unroll 1
        for (int l = 0; l < 3; ++l) {
            wait_products();
            unsigned char* const gl = l == 0 ? gA1 : l == 1 ? gA2 : nullptr;
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) {
                float acc[64];
                load_acc(acc0 + 64 * mt, wq, acc);
                const int o = t + 128 * mt;
                uint32_t w[32];
#pragma unroll
                for (int q = 0; q < 16; ++q) {
                    const float4 bv = lds_f4(s_bias + 4 * (l * kC + 4 * q));
                    w[2 * q] = in[mt] ? pack2(fmaxf(acc[4 * q] + bv.x, 0.f), fmaxf(acc[4 * q + 1] + bv.y, 0.f)) : 0u;
                    w[2 * q + 1] = in[mt] ? pack2(fmaxf(acc[4 * q + 2] + bv.z, 0.f), fmaxf(acc[4 * q + 3] + bv.w, 0.f)) : 0u;
                }
                store_row<T::COL>(ga + 16 * (o + 3), gl ? gl + 16 * (o + 3) : nullptr, w);
            }
            rows_ready();
            if (issuer) {
                const uint32_t el = elect_one();
#pragma unroll
                for (int mt = 0; mt < MT; ++mt) {
                    if (l < 2)
                        issue_product<kC, kTaps, T::COL>(el, u_acc0 + 64 * mt, u_ga + 2048 * mt,
                                                         u_sb + (l == 0 ? S::W2 : S::W3));
                    else
                        issue_product<kC, 1, T::COL>(el, u_acc0 + 64 * mt, u_ga + 48 + 2048 * mt, u_sb + S::W4);
                }
                tc_commit(el, u_bar);
            }
        }
        // restart scores from the pooled a3 (beside the MLP's product): a warp per sample,
        // lane l sums channels 2l and 2l+1 over the positions
        for (int k = wq; k < K; k += 4) {
            const int64_t b = tile * K + k;
            if (b >= a.B) break;
            const uint32_t col = ga + (lane >> 2) * T::COL + 4 * (lane & 3) + 16 * (k * (n + 3) + 3);
            float ma = 0.f, mb = 0.f;
            // in the order of the positions, 16 loads ahead of their additions (the loads may
            // run past the sample, within the CTA's memory; what they read there is dropped)
            for (int p0 = 0; p0 < n; p0 += 16) {
                uint32_t v[16];
#pragma unroll
                for (int i = 0; i < 16; ++i)
                    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v[i]) : "r"(col + 16 * (p0 + i)) : "memory");
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    if (p0 + i >= n) v[i] = 0u;
                    ma += lo_f(v[i]);
                    mb += hi_f(v[i]);
                }
            }
            ma /= (float)n;
            mb /= (float)n;
            float r = ma * bias[5 * kC + 2 * lane] + mb * bias[5 * kC + 2 * lane + 1];
#pragma unroll
            for (int off = 16; off; off >>= 1) r += __shfl_xor_sync(0xFFFFFFFFu, r, off);
            r += a.prm[oB6];
            if (TRAIN) {
                const float e = r - a.y[b], dr = e * inv;
                gw6.x += ma * dr;
                gw6.y += mb * dr;
                if (lane == 0) {
                    s_dr[k] = dr;
                    gb6 += dr;
                    lsum += 0.5f * e * e * inv;
                }
            } else if (lane == 0) {
                a.restart[b] = r;
            }
        }
        wait_products();
        uint32_t h[TRAIN ? MT : 1][32];
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
            float acc[64];
            load_acc(acc0 + 64 * mt, wq, acc);
            const int o = t + 128 * mt;
            float sacc = 0.f;
#pragma unroll
            for (int q = 0; q < 16; ++q) {
                const float4 bv = lds_f4(s_bias + 4 * (3 * kC + 4 * q)), wv = lds_f4(s_bias + 4 * (4 * kC + 4 * q));
                const float b4[4] = {bv.x, bv.y, bv.z, bv.w}, w5[4] = {wv.x, wv.y, wv.z, wv.w};
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const int i = 2 * q + j;
                    const uint32_t w = pack2(fmaxf(acc[2 * i] + b4[2 * j], 0.f), fmaxf(acc[2 * i + 1] + b4[2 * j + 1], 0.f));
                    if (TRAIN) h[mt][i] = w;
                    sacc += lo_f(w) * w5[2 * j] + hi_f(w) * w5[2 * j + 1];
                }
            }
            sacc += a.prm[oB5];
            if (TRAIN)
                s_score[o] = sacc;
            else if (in[mt])
                a.score[(tile * K + rk[mt]) * n + rpos[mt]] = sacc;
        }
        if constexpr (TRAIN) {
            group_sync(1 + grp);
            // softmax cross-entropy and its gradient, a warp per sample
            for (int k = wq; k < K; k += 4) {
                const int64_t b = tile * K + k;
                if (b >= a.B) break;
                const float* s = s_score + k * (n + 3);
                float m = -INFINITY;
                for (int p = lane; p < n; p += 32) m = fmaxf(m, s[p]);
#pragma unroll
                for (int off = 16; off; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, off));
                float z = 0.f;
                for (int p = lane; p < n; p += 32) z += expf(s[p] - m);
#pragma unroll
                for (int off = 16; off; off >>= 1) z += __shfl_xor_sync(0xFFFFFFFFu, z, off);
                const int tg = min(max(a.target[b], 0), n - 1);
                const float w = a.wf[b];
                for (int p = lane; p < n; p += 32)
                    s_ds[k * (n + 3) + p] = w * (expf(s[p] - m) / z - (p == tg ? 1.f : 0.f)) * inv;
                if (lane == 0) lsum += w * (logf(z) + m - s[tg]) * inv;
            }
            group_sync(1 + grp);
            // dh = w5 ds where h > 0; gradients of w5, b5 and b4
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) {
                const int o = t + 128 * mt;
                const float ds = in[mt] ? s_ds[o] : 0.f;
                gb5 += ds;
                float v[64];
                uint32_t w[32];
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    v[2 * i] = lo_f(h[mt][i]) * ds;
                    v[2 * i + 1] = hi_f(h[mt][i]) * ds;
                }
                add_channels(sums + 2 * kC, lane, warp_colsum(v, lane));
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    w[i] = pack2(lo_f(h[mt][i]) > 0.f ? bias[4 * kC + 2 * i] * ds : 0.f,
                                 hi_f(h[mt][i]) > 0.f ? bias[4 * kC + 2 * i + 1] * ds : 0.f);
                    if (!in[mt]) w[i] = 0u;
                    v[2 * i] = lo_f(w[i]);
                    v[2 * i + 1] = hi_f(w[i]);
                }
                store_row<T::COL>(gd + 16 * (o + 3), nullptr, w);
                add_channels(sums + kC, lane, warp_colsum(v, lane));
            }
            rows_ready();
            if (issuer) {
                const uint32_t el = elect_one(), u_gd = u_ga + T::ACT;
#pragma unroll
                for (int mt = 0; mt < MT; ++mt)
                    issue_product<kC, 1, T::COL>(el, u_acc0 + 64 * mt, u_gd + 48 + 2048 * mt, u_sb + S::WB4);
                // dW4: its rows 64-127 (the columns after a3's, i.e. dh's) are dropped
                issue_wgrad<T::M, T::COL>(el, u_acc4 + 64 * (done % S::ACC4), u_ga + 48, u_gd + 48, done < S::ACC4);
                tc_commit(el, u_bar);
            }
            wait_products();
            // da3 = (W4^T dh + w6 dr / n) where a3 > 0; gradient of b3
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) {
                float acc[64];
                load_acc(acc0 + 64 * mt, wq, acc);
                const int o = t + 128 * mt;
                const float pdr = in[mt] ? s_dr[rk[mt]] / (float)n : 0.f;
                uint32_t w[32];
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const uint4 q = lds128(ga + c * T::COL + 16 * (o + 3));
                    const uint32_t mw[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int i = 8 * c + 2 * j;
                        const float v0 = acc[i] + bias[5 * kC + i] * pdr, v1 = acc[i + 1] + bias[5 * kC + i + 1] * pdr;
                        w[4 * c + j] = pack2(lo_f(mw[j]) > 0.f ? v0 : 0.f, hi_f(mw[j]) > 0.f ? v1 : 0.f);
                    }
                }
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    if (!in[mt]) w[i] = 0u;
                    acc[2 * i] = lo_f(w[i]);
                    acc[2 * i + 1] = hi_f(w[i]);
                }
                store_row<T::COL>(0u, gA3 + 16 * (o + 3), w);
                add_channels(sums, lane, warp_colsum(acc, lane));
            }
        }
        tc_fence_before();
        group_sync(1 + grp);
        tc_fence_after();
        // the same for the whole group: the mark is made before this barrier, or after the next
        // tile's first one
        ok = *failed == 0;
    }
    if (!ok) {
        mbar_wait(bar_w, 0);  // the weights' copies end before the CTA does
        if (t == 0) net_failed(a.err, a.status);
        if (!TRAIN) {
            // the scores that this group owes, from the tile it gave up at
            for (tile = (int64_t)grp * gridDim.x + blockIdx.x + max(done - 1, 0) * stride; tile < tiles; tile += stride) {
#pragma unroll
                for (int mt = 0; mt < MT; ++mt)
                    if (rk[mt] >= 0 && tile * K + rk[mt] < a.B) {
                        a.score[(tile * K + rk[mt]) * n + rpos[mt]] = NAN;
                        a.restart[tile * K + rk[mt]] = NAN;
                    }
            }
        }
    }
    if constexpr (TRAIN) {
        add_channels(sums + 3 * kC, lane, gw6);
#pragma unroll
        for (int off = 16; off; off >>= 1) gb5 += __shfl_xor_sync(0xFFFFFFFFu, gb5, off);
        if (lane == 0) {
            atomicAdd(a.grad + oB5, gb5);
            atomicAdd(a.grad + oB6, gb6);
            atomicAdd(a.loss, lsum);
        }
        // this group's partial dW4 (channel x output)
        for (int q = 0; q < S::ACC4; ++q) {
            if (q > 0 && tiles <= gridDim.x * S::NG) break;  // no tile took it
            const int64_t slot4 = ((int64_t)q * gridDim.x + blockIdx.x) * S::NG + grp;
            float4* dst = reinterpret_cast<float4*>(a.part4 + slot4 * kC * kC) + t * (kC / 4);
            const bool used = done > q;  // the same for the group: the load is warp-wide
            float acc[64];
            if (used) load_acc(acc4 + 64 * q, wq, acc);
#pragma unroll
            for (int i = 0; i < 16; ++i)
                if (t < kC)
                    dst[i] = used ? make_float4(acc[4 * i], acc[4 * i + 1], acc[4 * i + 2], acc[4 * i + 3])
                                  : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (TRAIN && threadIdx.x < kC) {
        atomicAdd(a.grad + oB3 + threadIdx.x, sums[threadIdx.x]);
        atomicAdd(a.grad + oB4 + threadIdx.x, sums[kC + threadIdx.x]);
        atomicAdd(a.grad + oW5 + threadIdx.x, sums[2 * kC + threadIdx.x]);
        atomicAdd(a.grad + oW6 + threadIdx.x, sums[3 * kC + threadIdx.x]);
    }
    if (threadIdx.x < 32) {
        tc_fence_after();
        tmem_dealloc(tmem, S::TMEM);
    }
}

// ------------------------------------------------------------------ backward of a convolution
//
// Per tile, from the gradient G of a convolution's output (rows outside the positions zero)
// and its input IN:
//   dIN = (G convolved with the tap-reversed transpose) where IN > 0,
//   dW[o][c][k] += sum over rows r of G[r][o] IN[r + k][c],
//   the bias gradient of the layer below (the column sums of dIN).
// FIRST: IN is a1, and dIN = da1 stays in shared memory for conv1's weight gradient against
// the inputs; else dIN goes to global memory.
//
// A warp of its own issues every product: the weight gradient's accumulators are shared by
// the CTA's tile groups, and one thread's products on an accumulator complete in order.  The
// weight gradient takes taps in pairs (M = 128): the tile of IN is loaded twice, the second
// copy one row up and right behind the first, so that columns 8-15 of the operand are the
// next tap's.  conv1's takes one column (8 channels, 3 in use) per tap from 8 copies of the
// inputs, each one row further up.
// CTAs per SM's turn: a weight gradient's accumulator takes the products of a CTA's tiles one
// after the other, and the tensor core's FP32 additions round toward zero, an error that
// grows with their number.  304 CTAs add about 110 products each at 4096 samples of n = 128;
// with 152 the gradients of W2 and W3 were 2e-6 to 3e-6 away (2-norm) from those with 304,
// with 608 1e-6 the other way.  The second turn costs a training step of 4096 20 us (417
// from 396): weights loaded and partial sums written twice as often.
constexpr int kBwdCtas = 2;

template <int MT, bool FIRST>
struct BwdShape {
    using T = Tile<MT>;
    static constexpr int NG = MT == 1 ? (FIRST ? 2 : 3) : 1;
    static constexpr int THREADS = NG * kTcThreads + 32;
    static constexpr int WB = 0, GROUPS = kTaps * kC * 128;
    // the 8 input copies (column k one row further up than column k-1; the operand's columns
    // 8-15 fall on G and their rows of the result are dropped), G, IN, IN one row up (its
    // first row lies 16 bytes before it)
    static constexpr int XC = 0, G = FIRST ? 8 * T::COL : 0, IN = G + T::ACT, GROUP = IN + 2 * T::ACT;
    // barriers, the TMEM slot, the CTA's mark (a part of it gave up), two marks per group
    static constexpr int BAR = GROUPS + NG * GROUP, MARKS = BAR + 152, SUMS = BAR + 192;
    static_assert(4 + 8 * NG <= SUMS - MARKS, "marks");
    static constexpr int SMEM = SUMS + kC * 4 + 128;
    static constexpr int ACC_W = 0, ACC_W1 = 256, ACC_D = FIRST ? 320 : 256;  // TMEM columns
    static constexpr int TMEM = 512;
    static_assert(ACC_D + NG * MT * 64 <= TMEM, "TMEM columns");
};

struct BwdArgs {
    const bf16 *G, *IN, *X0, *wb;
    bf16* dIN;
    float* part;   // [CTA][448][64] partial dW (row tap * 64 + channel)
    float* part1;  // FIRST: [CTA][64][64] partial dW1 (row tap * 8 + channel)
    float* db;
    int* err;
    int64_t tiles;
    int64_t B;
    int n;
};

template <int MT, bool FIRST>
__global__ void __launch_bounds__(BwdShape<MT, FIRST>::THREADS, 1) conv_backward_kernel(BwdArgs a)
{
    using S = BwdShape<MT, FIRST>;
    using T = Tile<MT>;
    extern __shared__ unsigned char tc_smem_raw[];
    unsigned char* sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(tc_smem_raw) + 127) & ~uintptr_t(127));
    const uint32_t sb = smem_addr(sm);
    const int t = threadIdx.x % kTcThreads, wq = t >> 5, lane = t & 31;
    const int grp = (int)uniform(threadIdx.x / kTcThreads);
    const bool issuer = grp == S::NG;
    // barriers per group: operands loaded, dIN product done, weight gradient done, da1 ready,
    // conv1's weight gradient done
    const uint32_t bar_w = sb + S::BAR, bars = bar_w + 8, slot = sb + S::BAR + 144;
    auto full = [&](int g) { return bars + 40 * g; };
    auto dbar = [&](int g) { return bars + 40 * g + 8; };
    auto wbar = [&](int g) { return bars + 40 * g + 16; };
    auto rbar = [&](int g) { return bars + 40 * g + 24; };
    auto fbar = [&](int g) { return bars + 40 * g + 32; };
    volatile int* failed = reinterpret_cast<volatile int*>(sm + S::MARKS);
    float* sums = reinterpret_cast<float*>(sm + S::SUMS);
    auto buf = [&](int g) { return sb + S::GROUPS + g * S::GROUP; };
    if (threadIdx.x < kC) sums[threadIdx.x] = 0.f;
    // the operands' unwritten rows and columns hold finite values
    for (int i = threadIdx.x; i < S::NG * S::GROUP / 16; i += S::THREADS)
        sts128(sb + S::GROUPS + 16 * i, make_uint4(0u, 0u, 0u, 0u));
    if (issuer) tmem_alloc(slot, S::TMEM);
    if (threadIdx.x <= 2 * S::NG) failed[threadIdx.x] = 0;
    if (threadIdx.x == 0) {
        mbar_init(bar_w, 1);
        for (int i = 0; i < 5 * S::NG; ++i) mbar_init(bars + 8 * i, 1);
        mbar_init_fence();
    }
    fence_async_shared();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(sm + S::BAR + 144);
    const int64_t first = (int64_t)blockIdx.x, stride = (int64_t)gridDim.x * S::NG;
    auto tile_of = [&](int g, int it) { return first + (int64_t)g * gridDim.x + it * stride; };
    // one thread: the group's operands of a tile
    auto load = [&](int g, int64_t tile) {
        const uint32_t b = buf(g), f = full(g);
        const unsigned char* src = reinterpret_cast<const unsigned char*>(a.IN) + tile * T::ACT;
        mbar_arrive_expect_tx(f, 3 * T::ACT + (FIRST ? 8 * T::COL : 0));
        bulk_copy_g2s(b + S::G, reinterpret_cast<const unsigned char*>(a.G) + tile * T::ACT, T::ACT, f);
        bulk_copy_g2s(b + S::IN, src, T::ACT, f);
        bulk_copy_g2s(b + S::IN + T::ACT - 16, src, T::ACT, f);
        if (FIRST)
            for (int k = 0; k < 8; ++k)
                bulk_copy_g2s(b + S::XC + k * (T::COL - 16),
                              reinterpret_cast<const unsigned char*>(a.X0) + tile * T::COL, T::COL, f);
    };
    int loads = 0;  // a group's first thread: its tiles' copies
    if (issuer) {
        // the whole warp, with uniform values; one lane issues.  Its waits are over, too, once a
        // group has given up
        auto wait = [&](uint32_t bar, uint32_t parity, int tries) {
            return __all_sync(0xFFFFFFFFu, mbar_wait(bar, parity, tries)) != 0;
        };
        uint32_t last = 0, last_parity = 0;  // the barrier of the last products, its phase
        const uint32_t el = elect_one(), u_sb = uniform(sb), u_tmem = uniform(tmem), u_bars = uniform(bars);
        bool fresh = true, fresh1 = true;
        if (el) {
            mbar_arrive_expect_tx(bar_w, kTaps * kC * 128);
            bulk_copy_g2s(sb + S::WB, a.wb, kTaps * kC * 128, bar_w);
            for (int g = 0; g < S::NG; ++g)
                if (tile_of(g, 0) < a.tiles) load(g, tile_of(g, 0));
        }
        __syncwarp();
        bool ok = wait(bar_w, 0, kTriesWeights);
        for (int it = 0; ok && tile_of(0, it) < a.tiles; ++it) {
            for (int g = 0; ok && g < S::NG && tile_of(g, it) < a.tiles; ++g) {
                const uint32_t b = u_sb + S::GROUPS + g * S::GROUP, br = u_bars + 40 * g;
                ok = wait(br, it & 1, kTriesTiles);
                if (!ok) break;
                tc_fence_after();
#pragma unroll
                for (int mt = 0; mt < MT; ++mt)
                    issue_product<kC, kTaps, T::COL>(el, u_tmem + S::ACC_D + 64 * (g * MT + mt), b + S::G + 2048 * mt,
                                                     u_sb + S::WB);
                tc_commit(el, br + 8);
#pragma unroll
                for (int q = 0; q < 4; ++q)  // taps 2q, 2q+1 (the eighth is dropped)
                    issue_wgrad<T::M, T::COL>(el, u_tmem + S::ACC_W + 64 * q, b + S::IN + 32 * q, b + S::G + 48, fresh);
                fresh = false;
                tc_commit(el, br + 16);
                last = br + 16, last_parity = it & 1;
            }
            if (FIRST)
                for (int g = 0; ok && g < S::NG && tile_of(g, it) < a.tiles; ++g) {
                    const uint32_t b = u_sb + S::GROUPS + g * S::GROUP, br = u_bars + 40 * g;
                    ok = wait(br + 24, it & 1, kTriesTiles);
                    if (!ok) break;
                    tc_fence_after();
                    issue_wgrad<T::M, T::COL>(el, u_tmem + S::ACC_W1, b + S::XC, b + S::G + 48, fresh1);
                    fresh1 = false;
                    tc_commit(el, br + 32);
                    last = br + 32, last_parity = it & 1;
                }
        }
        if (!ok) {
            *failed = 1;  // the groups' waits are over
            // the copies and products under way end before the CTA does (a commit covers all before it)
            mbar_wait(bar_w, 0);
            if (last != 0u) mbar_wait(last, last_parity);
        }
    } else {
        // Marks: a thread makes the one of its iteration's parity before the group's barrier,
        // all read it after the barrier, and the next iteration but one cannot make it before
        // they have: the same for the whole group.  What the first thread waits for after the
        // barrier (`late`) it tells in the next iteration.
        bool late = false;
        volatile int* const marks = failed + 1 + 2 * grp;
        auto await = [&](uint32_t bar, uint32_t parity) {  // over, too, once the issuer or a group has given up
            if (mbar_wait(bar, parity, kTriesProducts)) return true;
            if (*failed == 0) mbar_wait(bar, parity);
            return false;
        };
        if (t == 0 && tile_of(grp, 0) < a.tiles) loads = 1;  // (the issuer's)
        const int K = tile_samples(a.n);
        float2 gb = {0.f, 0.f};
        int rk[MT];
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) {
            const RowPos rp(t + 128 * mt, a.n, K);
            rk[mt] = rp.in ? rp.k : -1;
        }
        for (int it = 0; tile_of(grp, it) < a.tiles; ++it) {
            const int64_t tile = tile_of(grp, it);
            if (late || !await(dbar(grp), it & 1)) marks[it & 1] = 1;
            tc_fence_after();
            unsigned char* const gout = FIRST ? nullptr : reinterpret_cast<unsigned char*>(a.dIN) + tile * T::ACT;
            if (!FIRST) zero_pad_rows<MT, 8>(gout, t);
            if (FIRST) {
                // da1 takes G's place: the weight gradient has read it
                if (!late && !await(wbar(grp), it & 1)) marks[it & 1] = 1;
                tc_fence_after();
            }
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) {
                float acc[64];
                load_acc(tmem + S::ACC_D + 64 * (grp * MT + mt), wq, acc);
                const int o = t + 128 * mt;
                const bool in = rk[mt] >= 0 && tile * K + rk[mt] < a.B;
                uint32_t w[32];
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const uint4 q = lds128(buf(grp) + S::IN + c * T::COL + 16 * (o + 3));
                    const uint32_t mw[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int i = 8 * c + 2 * j;
                        w[4 * c + j] = pack2(lo_f(mw[j]) > 0.f ? acc[i] : 0.f, hi_f(mw[j]) > 0.f ? acc[i + 1] : 0.f);
                    }
                }
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    if (!in) w[i] = 0u;
                    acc[2 * i] = lo_f(w[i]);
                    acc[2 * i + 1] = hi_f(w[i]);
                }
                store_row<T::COL>(FIRST ? buf(grp) + S::G + 16 * (o + 3) : 0u, FIRST ? nullptr : gout + 16 * (o + 3), w);
                add2(gb, warp_colsum(acc, lane));
            }
            if (FIRST) {
                fence_async_shared();
                tc_fence_before();
                group_sync(1 + grp);
                if (marks[it & 1]) break;
                if (t == 0) {
                    mbar_arrive(rbar(grp));
                    late = !await(fbar(grp), it & 1);
                    if (tile_of(grp, it + 1) < a.tiles && !late) {
                        fence_async_shared();
                        load(grp, tile_of(grp, it + 1));
                        ++loads;
                    }
                }
            } else {
                tc_fence_before();
                group_sync(1 + grp);  // every row's mask has been read
                if (marks[it & 1]) break;
                if (t == 0) {
                    late = !await(wbar(grp), it & 1);
                    if (tile_of(grp, it + 1) < a.tiles && !late) {
                        fence_async_shared();
                        load(grp, tile_of(grp, it + 1));
                        ++loads;
                    }
                }
            }
        }
        if (late || marks[0] || marks[1]) *failed = 1;
        add_channels(sums, lane, gb);
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (*failed) {
        if (loads > 0) mbar_wait(full(grp), (loads - 1) & 1);  // the tiles' copies end before the CTA does
        if (threadIdx.x == 0) net_failed(a.err, nullptr);
    } else if (grp == 0) {
        // every product has completed: each group's last waits covered its own
        for (int q = 0; q < 4; ++q) {
            float acc[64];
            load_acc(tmem + S::ACC_W + 64 * q, wq, acc);
            const int m = 128 * q + t;  // tap * 64 + channel
            if (m < kTaps * kC) {
                float4* dst = reinterpret_cast<float4*>(a.part + ((int64_t)blockIdx.x * kTaps * kC + m) * kC);
#pragma unroll
                for (int i = 0; i < 16; ++i) dst[i] = make_float4(acc[4 * i], acc[4 * i + 1], acc[4 * i + 2], acc[4 * i + 3]);
            }
        }
        if (FIRST) {
            float acc[64];
            load_acc(tmem + S::ACC_W1, wq, acc);
            if (t < 64) {
                float4* dst = reinterpret_cast<float4*>(a.part1 + ((int64_t)blockIdx.x * 64 + t) * kC);
#pragma unroll
                for (int i = 0; i < 16; ++i) dst[i] = make_float4(acc[4 * i], acc[4 * i + 1], acc[4 * i + 2], acc[4 * i + 3]);
            }
        }
    }
    if (threadIdx.x < kC) atomicAdd(a.db + threadIdx.x, sums[threadIdx.x]);
    tc_fence_before();
    __syncthreads();
    if (issuer) {
        tc_fence_after();
        tmem_dealloc(tmem, S::TMEM);
    }
}

// Gradients of W1..W4 from the CTAs' partial sums: 16 outputs x 4 of them per block, 16
// slices of the CTAs each.
struct ReduceArgs {
    const float *p1, *p2, *p3, *p4;
    int c23, c4;  // CTAs of the convolutions' partials, accumulators of W4's
    float* grad;
    float* loss;
    const int* err;  // nonzero: a wait of the pass gave up, everything it returns is NaN
};

__global__ void __launch_bounds__(256) wgrad_reduce_kernel(ReduceArgs a)
{
    __shared__ float4 sh[16][17];
    const bool failed = *a.err != 0;
    if (failed && blockIdx.x == 0) {
        // the gradients that are added up elsewhere
        for (int i = threadIdx.x; i < kParams; i += blockDim.x)
            if (!(i < oB1 || (i >= oW2 && i < oB2) || (i >= oW3 && i < oB3) || (i >= oW4 && i < oB4))) a.grad[i] = NAN;
        if (threadIdx.x == 0) *a.loss = NAN;
    }
    const int col = threadIdx.x & 15, sl = threadIdx.x >> 4;
    // rows of 64 outputs: W2 448, W3 448, W1 64 (tap * 8 + channel), W4 64
    int row = blockIdx.x, ctas = a.c23, rows = kTaps * kC;
    const float* p = a.p2;
    int which = 2;
    if (row >= 2 * kTaps * kC + 64) {
        which = 4, row -= 2 * kTaps * kC + 64, p = a.p4, ctas = a.c4, rows = 64;
    } else if (row >= 2 * kTaps * kC) {
        which = 1, row -= 2 * kTaps * kC, p = a.p1, rows = 64;
    } else if (row >= kTaps * kC) {
        which = 3, row -= kTaps * kC, p = a.p3;
    }
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int c = sl; c < ctas; c += 16) {
        const float4 v = reinterpret_cast<const float4*>(p + ((int64_t)c * rows + row) * kC)[col];
        s.x += v.x, s.y += v.y, s.z += v.z, s.w += v.w;
    }
    sh[sl][col] = s;
    __syncthreads();
    if (threadIdx.x < 64) {
        const int o = threadIdx.x;
        float t = 0.f;
        for (int k = 0; k < 16; ++k) t += reinterpret_cast<const float*>(&sh[k][o >> 2])[o & 3];
        if (failed) t = NAN;
        if (which == 4) {
            a.grad[oW4 + o * kC + row] = t;  // dW4[j][c]
        } else if (which == 1) {
            const int k = row >> 3, c = row & 7;
            if (k < kTaps) {
                a.grad[oW1 + (o * kCin + c) * kTaps + k] = t;
                a.grad[oW1 + (o * kCin + c + 8) * kTaps + k] = failed ? NAN : 0.f;  // channels 8-15 carry no input
            }
        } else {
            const int k = row / kC, c = row % kC;
            a.grad[(which == 2 ? oW2 : oW3) + (o * kC + c) * kTaps + k] = t;
        }
    }
}

// Packed bf16 copies of the float32 master weights (and the pass's error word cleared): element e of a layer's K x 64 operand is
// K index 8 (e / 512) + e % 8 of output (e / 8) % 64.
__global__ void pack_kernel(const float* __restrict__ prm, bf16* __restrict__ wpk, int* __restrict__ err)
{
    if (blockIdx.x == 0 && threadIdx.x == 0) *err = 0;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < kPacked; t += gridDim.x * blockDim.x) {
        float v;
        if (t < pWf2) {  // Wf1: K index k*16+c, W1[o][c][k]
            const int e = t - pWf1, o = (e >> 3) & 63, kk = 8 * (e >> 9) + (e & 7), k = kk / kCin, c = kk % kCin;
            v = prm[oW1 + (o * kCin + c) * kTaps + k];
        } else if (t < pWf4) {  // Wf2 / Wf3: K index k*64+c
            const int e = t - (t < pWf3 ? pWf2 : pWf3), o = (e >> 3) & 63, kk = 8 * (e >> 9) + (e & 7), k = kk / kC, c = kk % kC;
            v = prm[(t < pWf3 ? oW2 : oW3) + (o * kC + c) * kTaps + k];
        } else if (t < pWb2) {  // Wf4: K index c, W4[j][c]
            const int e = t - pWf4, o = (e >> 3) & 63, c = 8 * (e >> 9) + (e & 7);
            v = prm[oW4 + o * kC + c];
        } else if (t < pWb4) {  // Wb2 / Wb3: outputs c, K index k'*64+o, W[o][c][6-k']
            const int e = t - (t < pWb3 ? pWb2 : pWb3), c = (e >> 3) & 63, kk = 8 * (e >> 9) + (e & 7), kr = kk / kC, o = kk % kC;
            v = prm[(t < pWb3 ? oW2 : oW3) + (o * kC + c) * kTaps + (kTaps - 1 - kr)];
        } else if (t < pW5) {  // Wb4: outputs c, K index j, W4[j][c]
            const int e = t - pWb4, c = (e >> 3) & 63, j = 8 * (e >> 9) + (e & 7);
            v = prm[oW4 + j * kC + c];
        } else if (t < pW6) {
            v = prm[oW5 + (t - pW5)];
        } else {
            v = prm[oW6 + (t - pW6)];
        }
        wpk[t] = __float2bfloat16_rn(v);
    }
}

__device__ __forceinline__ bool is_weight(int i)
{
    return (i >= oW1 && i < oB1) || (i >= oW2 && i < oB2) || (i >= oW3 && i < oB3) || (i >= oW4 && i < oB4) ||
           (i >= oW5 && i < oB5) || (i >= oW6 && i < oB6);
}

__global__ void adamw_kernel(float* __restrict__ prm, const float* __restrict__ grad, float* __restrict__ m,
                             float* __restrict__ v, float lr, float wd, float c1, float c2)
{
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < kParams; i += gridDim.x * blockDim.x) {
        const float g = grad[i];
        const float mi = b1 * m[i] + (1.f - b1) * g;
        const float vi = b2 * v[i] + (1.f - b2) * g * g;
        m[i] = mi;
        v[i] = vi;
        const float mh = mi / c1, vh = vi / c2;
        const float decay = is_weight(i) ? wd : 0.f;
        prm[i] = prm[i] - lr * (mh / (sqrtf(vh) + eps) + decay * prm[i]);
    }
}

// He-uniform weights from Philox (key = seed, counter = (index, 0, 0, 3)), zero biases.
__global__ void init_kernel(float* __restrict__ prm, uint64_t seed)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < kParams; i += gridDim.x * blockDim.x) {
        int fan = 0;
        if (i >= oW1 && i < oB1) fan = 3 * kTaps;
        else if ((i >= oW2 && i < oB2) || (i >= oW3 && i < oB3)) fan = kC * kTaps;
        else if ((i >= oW4 && i < oB4) || (i >= oW5 && i < oB5) || (i >= oW6 && i < oB6)) fan = kC;
        if (fan == 0) {
            prm[i] = 0.f;
            continue;
        }
        uint32_t c0 = (uint32_t)i, c1 = 0, c2 = 0, c3 = 3u, k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
#pragma unroll
        for (int r = 0; r < 10; ++r) {
            if (r) {
                k0 += 0x9E3779B9u;
                k1 += 0xBB67AE85u;
            }
            const uint32_t hi0 = __umulhi(0xD2511F53u, c0), lo0 = 0xD2511F53u * c0;
            const uint32_t hi1 = __umulhi(0xCD9E8D57u, c2), lo1 = 0xCD9E8D57u * c2;
            const uint32_t y0 = hi1 ^ c1 ^ k0, y2 = hi0 ^ c3 ^ k1;
            c0 = y0;
            c1 = lo1;
            c2 = y2;
            c3 = lo0;
        }
        const float u = (float)(c0 >> 8) * (1.f / 16777216.f) * 2.f - 1.f;
        prm[i] = u * sqrtf(6.f / (float)fan);
    }
}

}  // namespace

// Workspace carve-up for a batch of B states of n free variables.
struct NetWs {
    bf16 *X0, *A1, *A2, *dA3, *dA2, *wpk;
    float *score, *restart, *loss;
    int* err;  // cleared by pack_kernel, set by a tensor-core kernel whose wait gave up
    float *part1, *part2, *part3, *part4;  // per-CTA partial weight gradients
    float* grad;  // gradients of a pass whose result overlaps its inputs
    size_t bytes;
};

static size_t align256(size_t x)
{
    return (x + 255) & ~(size_t)255;
}

// The kernels' bulk copies and 16-byte stores start on 16-byte boundaries of the workspace.
static bool aligned_ws(const void* ws)
{
    return ((uintptr_t)ws & 15) == 0;
}

// Memory that a pass reads while it writes its results: a result that overlaps some of it (in
// place of an input, say) goes to the workspace first and is copied at the end.
struct Span {
    const void* p;
    size_t bytes;
};

template <int N>
static bool apart(const void* out, size_t bytes, const Span (&in)[N])
{
    const uintptr_t a = (uintptr_t)out;
    bool ok = out != nullptr;
    for (const Span& s : in) ok = ok && (a + bytes <= (uintptr_t)s.p || (uintptr_t)s.p + s.bytes <= a);
    return ok;
}

static int sm_count()
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms > 0 ? sms : 1;
}

NetWs carve(void* base, int64_t B, int n)
{
    NetWs w;
    const size_t tiles = (size_t)tile_count(B, n), col = (size_t)(tile_rows(n) + 9) * 16, sms = (size_t)sm_count();
    // the CTAs that write partial sums: a small batch has fewer than the GPU could run (80 MB of
    // partials for all of them, 1 MB for one state)
    const size_t fwd = std::min(tiles, sms), bwd = std::min(tiles, kBwdCtas * sms);
    char* p = static_cast<char*>(base);
    size_t off = 0;
    auto take = [&](size_t bytes) {
        char* q = p ? p + off : nullptr;
        off += align256(bytes);
        return q;
    };
    w.X0 = (bf16*)take(tiles * col);
    w.A1 = (bf16*)take(tiles * 8 * col);
    w.A2 = (bf16*)take(tiles * 8 * col);
    w.dA3 = (bf16*)take(tiles * 8 * col);
    w.dA2 = (bf16*)take(tiles * 8 * col);
    w.wpk = (bf16*)take(kPacked * sizeof(bf16));
    w.score = (float*)take((size_t)B * n * 4);
    w.restart = (float*)take((size_t)B * 4);
    w.loss = (float*)take(4);
    w.err = (int*)take(4);
    w.part1 = (float*)take(bwd * 64 * kC * 4);
    w.part2 = (float*)take(bwd * kTaps * kC * kC * 4);
    w.part3 = (float*)take(bwd * kTaps * kC * kC * 4);
    w.part4 = (float*)take(fwd * 2 * kC * kC * 4);
    w.grad = (float*)take(kParams * 4);
    w.bytes = off;
    return w;
}

template <class S>
static int allow_smem(void (*fn)(FwdArgs))
{
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, S::SMEM) == cudaSuccess ? LABS_OK : LABS_ECUDA;
}

template <int MT, bool TRAIN>
static int launch_forward(const FwdArgs& a, int sms, cudaStream_t s)
{
    using S = FwdShape<MT, TRAIN>;
    static_assert(S::SMEM <= 227 * 1024, "shared memory");
    if (allow_smem<S>(net_forward_kernel<MT, TRAIN>)) return LABS_ECUDA;
    const int grid = (int)std::min<int64_t>(tile_count(a.B, a.n), sms);
    net_forward_kernel<MT, TRAIN><<<grid, S::THREADS, S::SMEM, s>>>(a);
    return cudaGetLastError() == cudaSuccess ? LABS_OK : LABS_ECUDA;
}

template <int MT, bool FIRST>
static int launch_conv_backward(const BwdArgs& a, int sms, cudaStream_t s)
{
    using S = BwdShape<MT, FIRST>;
    static_assert(S::SMEM <= 227 * 1024, "shared memory");
    if (cudaFuncSetAttribute(conv_backward_kernel<MT, FIRST>, cudaFuncAttributeMaxDynamicSharedMemorySize, S::SMEM) !=
        cudaSuccess)
        return LABS_ECUDA;
    const int grid = (int)std::min<int64_t>(a.tiles, kBwdCtas * sms);
    conv_backward_kernel<MT, FIRST><<<grid, S::THREADS, S::SMEM, s>>>(a);
    return cudaGetLastError() == cudaSuccess ? LABS_OK : LABS_ECUDA;
}

static FwdArgs forward_args(const float* prm, const float* x, const NetWs& w, int64_t B, int n, float* score, float* restart)
{
    FwdArgs a{};
    a.x = x;
    a.wpk = w.wpk;
    a.prm = prm;
    a.score = score;
    a.restart = restart;
    a.err = w.err;
    a.B = B;
    a.n = n;
    return a;
}

int pack(const float* prm, const NetWs& w, cudaStream_t s)
{
    pack_kernel<<<4 * sm_count(), 256, 0, s>>>(prm, w.wpk, w.err);
    return cudaGetLastError() == cudaSuccess ? LABS_OK : LABS_ECUDA;
}

int forward(const float* prm, const float* x, const NetWs& w, int64_t B, int n, float* score, float* restart, DevStatus* status,
            cudaStream_t s)
{
    int rc = pack(prm, w, s);
    if (rc) return rc;
    FwdArgs a = forward_args(prm, x, w, B, n, score, restart);
    a.status = status;
    return n <= 128 ? launch_forward<1, false>(a, sm_count(), s) : launch_forward<2, false>(a, sm_count(), s);
}

template <int MT>
static int gradients_tiles(FwdArgs a, const NetWs& w, float* grad, int sms, cudaStream_t s)
{
    int rc = launch_forward<MT, true>(a, sms, s);
    const int64_t tiles = tile_count(a.B, a.n);
    BwdArgs b{};
    b.err = w.err;
    b.tiles = tiles;
    b.B = a.B;
    b.n = a.n;
    b.G = w.dA3, b.IN = w.A2, b.wb = w.wpk + pWb3, b.dIN = w.dA2, b.part = w.part3, b.db = grad + oB2;
    if (!rc) rc = launch_conv_backward<MT, false>(b, sms, s);
    b.G = w.dA2, b.IN = w.A1, b.X0 = w.X0, b.wb = w.wpk + pWb2, b.dIN = nullptr, b.part = w.part2, b.part1 = w.part1;
    b.db = grad + oB1;
    if (!rc) rc = launch_conv_backward<MT, true>(b, sms, s);
    constexpr int NG = FwdShape<MT, true>::NG, ACC4 = FwdShape<MT, true>::ACC4;
    const int ctas = (int)std::min<int64_t>(tiles, sms), back = (int)std::min<int64_t>(tiles, kBwdCtas * sms);
    const ReduceArgs r{w.part1, w.part2, w.part3, w.part4, back, ctas * NG * (tiles > ctas * NG ? ACC4 : 1),
                       grad, a.loss, w.err};
    wgrad_reduce_kernel<<<2 * kTaps * kC + 128, 256, 0, s>>>(r);
    if (!rc && cudaGetLastError() != cudaSuccess) rc = LABS_ECUDA;
    return rc;
}

int gradients(const float* prm, const float* x, const NetWs& w, const int32_t* target, const float* y, const float* wf,
              float* grad, int64_t B, int n, cudaStream_t s)
{
    if (cudaMemsetAsync(grad, 0, kParams * sizeof(float), s) != cudaSuccess) return LABS_ECUDA;
    if (cudaMemsetAsync(w.loss, 0, sizeof(float), s) != cudaSuccess) return LABS_ECUDA;
    const int rc = pack(prm, w, s);
    if (rc) return rc;
    FwdArgs a = forward_args(prm, x, w, B, n, w.score, w.restart);
    a.target = target;
    a.y = y;
    a.wf = wf;
    a.X0 = w.X0;
    a.A1 = w.A1;
    a.A2 = w.A2;
    a.dA3 = w.dA3;
    a.part4 = w.part4;
    a.grad = grad;
    a.loss = w.loss;
    return n <= 128 ? gradients_tiles<1>(a, w, grad, sm_count(), s) : gradients_tiles<2>(a, w, grad, sm_count(), s);
}

int init_params(float* prm, uint64_t seed, cudaStream_t s)
{
    init_kernel<<<64, 256, 0, s>>>(prm, seed);
    return cudaGetLastError() == cudaSuccess ? LABS_OK : LABS_ECUDA;
}

int adamw(float* prm, const float* grad, float* m, float* v, int64_t t, float lr, float wd, cudaStream_t s)
{
    const float c1 = 1.f - powf(0.9f, (float)t), c2 = 1.f - powf(0.999f, (float)t);
    adamw_kernel<<<64, 256, 0, s>>>(prm, grad, m, v, lr, wd, c1, c2);
    return cudaGetLastError() == cudaSuccess ? LABS_OK : LABS_ECUDA;
}

}  // namespace net
}  // namespace labsgpu

namespace labsgpu {

size_t net_workspace_bytes(int64_t B, int n)
{
    return net::carve(nullptr, B, n).bytes;
}

int net_forward_ws(const float* params, const float* x, int64_t B, int n, void* ws, const float** scores,
                   const float** restart, DevStatus* status, void* stream)
{
    const net::NetWs w = net::carve(ws, B, n);
    const int rc = net::forward(params, x, w, B, n, w.score, w.restart, status, (cudaStream_t)stream);
    if (scores) *scores = w.score;
    if (restart) *restart = w.restart;
    return rc;
}

}  // namespace labsgpu

using namespace labsgpu;

extern "C" {

int labs_net_sizes(int32_t n, int64_t batch, size_t* param_count, size_t* workspace_bytes)
{
    if (n < 2 || n > kMaxN || batch < 0) return LABS_EINVAL;
    if (param_count) *param_count = net::kParams;
    if (workspace_bytes) *workspace_bytes = net::carve(nullptr, batch, n).bytes;
    return LABS_OK;
}

int labs_net_init(float* dev_params, uint64_t seed, void* cuda_stream)
{
    LABS_API_RANGE();
    if (!dev_params) return LABS_EINVAL;
    return net::init_params(dev_params, seed, (cudaStream_t)cuda_stream);
}

int labs_net_forward(const float* dev_params, const float* dev_x, int64_t batch, int32_t n, float* dev_scores,
                     float* dev_restart, void* dev_ws, size_t ws_bytes, void* cuda_stream)
{
    LABS_API_RANGE();
    if (!dev_params || !dev_x || n < 2 || n > kMaxN || batch < 0 || batch > INT32_MAX) return LABS_EINVAL;
    if (batch == 0) return LABS_OK;
    const net::NetWs w = net::carve(dev_ws, batch, n);
    if (!dev_ws || ws_bytes < w.bytes) return LABS_ENOMEM;
    if (!net::aligned_ws(dev_ws)) return LABS_EINVAL;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    const size_t sb = (size_t)batch * n * 4, rb = (size_t)batch * 4;
    const net::Span in[] = {{dev_params, net::kParams * 4}, {dev_x, 3 * sb}, {dev_ws, ws_bytes}};
    float* const score = net::apart(dev_scores, sb, in) ? dev_scores : w.score;
    float* const restart = net::apart(dev_restart, rb, in) ? dev_restart : w.restart;
    int rc = net::forward(dev_params, dev_x, w, batch, n, score, restart, nullptr, s);
    if (!rc && dev_scores && score != dev_scores)
        rc = cudaMemcpyAsync(dev_scores, score, sb, cudaMemcpyDeviceToDevice, s) ? LABS_ECUDA : 0;
    if (!rc && dev_restart && restart != dev_restart)
        rc = cudaMemcpyAsync(dev_restart, restart, rb, cudaMemcpyDeviceToDevice, s) ? LABS_ECUDA : 0;
    return rc;
}

int labs_net_gradients(const float* dev_params, const float* dev_x, const int32_t* dev_target, const float* dev_y,
                       const float* dev_wf, int64_t batch, int32_t n, float* dev_grads, float* dev_loss, void* dev_ws,
                       size_t ws_bytes, void* cuda_stream)
{
    LABS_API_RANGE();
    if (!dev_params || !dev_x || !dev_target || !dev_y || !dev_wf || !dev_grads || n < 2 || n > kMaxN || batch < 1 ||
        batch > INT32_MAX)
        return LABS_EINVAL;
    const net::NetWs w = net::carve(dev_ws, batch, n);
    if (!dev_ws || ws_bytes < w.bytes) return LABS_ENOMEM;
    if (!net::aligned_ws(dev_ws)) return LABS_EINVAL;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    const size_t gb = net::kParams * 4, rb = (size_t)batch * 4;
    const net::Span in[] = {{dev_params, gb}, {dev_x, 3 * n * rb}, {dev_target, rb}, {dev_y, rb}, {dev_wf, rb}};
    float* const grad = net::apart(dev_grads, gb, in) ? dev_grads : w.grad;
    int rc = net::gradients(dev_params, dev_x, w, dev_target, dev_y, dev_wf, grad, batch, n, s);
    if (!rc && grad != dev_grads)
        rc = cudaMemcpyAsync(dev_grads, grad, gb, cudaMemcpyDeviceToDevice, s) ? LABS_ECUDA : 0;
    if (!rc && dev_loss) rc = cudaMemcpyAsync(dev_loss, w.loss, 4, cudaMemcpyDeviceToDevice, s) ? LABS_ECUDA : 0;
    return rc;
}

int labs_net_adamw(float* dev_params, const float* dev_grads, float* dev_m, float* dev_v, int64_t t, float lr,
                   float weight_decay, void* cuda_stream)
{
    LABS_API_RANGE();
    if (!dev_params || !dev_grads || !dev_m || !dev_v || t < 1) return LABS_EINVAL;
    return net::adamw(dev_params, dev_grads, dev_m, dev_v, t, lr, weight_decay, (cudaStream_t)cuda_stream);
}

}  // extern "C"
