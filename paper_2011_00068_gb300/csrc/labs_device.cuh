// labs_device.cuh -- device code shared by the kernel translation units: random starts,
// lane groups, the rows, table and neighbourhood of a walker on FP32 (the learned walk, the
// first starts, the long sequences; the other walks and the row kernels evaluate the
// neighbourhood in the form of labs_step.cuh).  Not part of the public ABI.
//
// A lane group owns one walker (or one input row): the whole warp, a part of it when
// several walkers share a warp, or a CTA.  A walker's sequence is kept in shared
// memory split by parity, because for even lags every term of the neighbourhood
// evaluation pairs positions of equal parity:
//   A0[u] = s_{2u}   (u = 0..n-1),   A1[u] = s_{2u+1}   (u = 0..n-2),
// and its even-lag autocorrelations (odd lags vanish by Eq. 4) as the symmetric table
//   E[d] = C_{2|d|}  (0 < |d| < n),  E[0] = 0.
//
// dISL of free variable i = 2v+p (class p, index v), q = L-1-i its mirror, c = n-1:
//   flipping {i, q} changes C_k, k even, by dC_k = -4 s_i u_k with
//   u_k = s_{i+k}[i+k != q] + s_{i-k} (out-of-range s = 0; the pair (i,q) is excluded
//   because both of its ends flip), so with Eq. 2
//   dISL_i = sum_k dC_k (2 C_k + dC_k)
//          = -8 s_i (X_i - s_q C_{q-i}) + 16 (N_i - 1) + 32 (P_i - [3i >= L-1] s_q s_{3i-L+1})
//   X_i = sum_{j != i, j = i mod 2} s_j C_{|j-i|}      (a Toeplitz product: X_v = sum_u A_p[u] E[u-v])
//   P_i = sum_{k even, 2 <= k <= i} s_{i+k} s_{i-k}
//   N_i = number of positions of the parity of i, minus one (n-1 for even i, n-2 for odd i).
//   The centre flips alone: dC_k = -2 s_c (s_{c+k} + s_{c-k}), so
//   dISL_c = -4 s_c X_c + 16 floor(c/2).
// X costs n(n-1)/2 multiply-adds per class, i.e. about one per (flip, even lag) pair of
// the neighbourhood (Algorithm 1's loop over the (L+1)/2 free variables), and is the hot
// loop.  The first half of a tile holds the even class, the second half the odd class;
// each lane owns R consecutive outputs v0..v0+R-1 and slides a window of R values of E
// along u.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <climits>
#include <cstdint>

#include "labs_internal.cuh"

namespace labsgpu {

namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;

#ifndef LABS_TOEPLITZ_UNROLL
#define LABS_TOEPLITZ_UNROLL 2  // u-blocks of the Toeplitz loop unrolled together
#endif
constexpr int kToeplitzUnroll = LABS_TOEPLITZ_UNROLL;

#ifndef LABS_WALK_MIN_BLOCKS
#define LABS_WALK_MIN_BLOCKS 2  // CTAs of 8 warps per SM the walk kernel is compiled for (2 measured fastest)
#endif

// ------------------------------------------------------------------ Philox4x32-10
// Salmon, Moraes, Dror, Shaw, "Parallel random numbers: as easy as 1, 2, 3" (SC'11):
// ten rounds of two 32x32->64 multiplies with a Weyl-sequence key schedule.
__device__ __forceinline__ void philox(uint32_t& c0, uint32_t& c1, uint32_t& c2, uint32_t& c3,
                                       uint32_t k0, uint32_t k1)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r) {
            k0 += 0x9E3779B9u;
            k1 += 0xBB67AE85u;
        }
        const uint32_t m0 = 0xD2511F53u, m1 = 0xCD9E8D57u;
        uint32_t hi0 = __umulhi(m0, c0), lo0 = m0 * c0;
        uint32_t hi1 = __umulhi(m1, c2), lo1 = m1 * c2;
        uint32_t y0 = hi1 ^ c1 ^ k0, y2 = hi0 ^ c3 ^ k1;
        c0 = y0;
        c1 = lo1;
        c2 = y2;
        c3 = lo0;
    }
}

// Word j (j < 8) of the free-variable bits of start r of walker g: Philox block
// (g, r, j/4, 0) under key (seed lo, seed hi), word j%4; bits >= n cleared.
__device__ __forceinline__ uint32_t start_word(uint64_t seed, uint32_t g, uint32_t r, int j, int n)
{
    uint32_t c0 = g, c1 = r, c2 = (uint32_t)(j >> 2), c3 = 0u;
    philox(c0, c1, c2, c3, (uint32_t)seed, (uint32_t)(seed >> 32));
    uint32_t w = (j & 3) == 0 ? c0 : (j & 3) == 1 ? c1 : (j & 3) == 2 ? c2 : c3;
    int lo = 32 * j;
    if (n <= lo) return 0u;
    if (n - lo >= 32) return w;
    return w & ((1u << (n - lo)) - 1u);
}

__device__ __forceinline__ uint64_t global_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void raise_error(DevStatus* st, int code, int detail)
{
    if (atomicCAS(&st->error, 0, code) == 0) st->error_detail = detail;
}

// A group of TILE lanes that runs one walker (or one row): the whole warp (TILE = 32)
// or a half warp (TILE = 16, two walkers per warp).  Every warp-level primitive of the
// walk goes through it with the tile's own lane mask, so the two halves of a warp may
// take different paths.
template <int TILE>
struct Tile {
    static constexpr int kSize = TILE;
    static constexpr int kHalf = TILE / 2;  // lanes per parity class
    static constexpr unsigned kLow = TILE == 32 ? 0xFFFFFFFFu : ((1u << TILE) - 1u);
    int lane;       // 0 .. TILE-1
    int base;       // warp lane of the tile's lane 0
    unsigned mask;  // the tile's lanes
    __device__ explicit Tile(int warp_lane)
        : lane(warp_lane & (TILE - 1)), base(warp_lane & ~(TILE - 1)), mask(kLow << (warp_lane & ~(TILE - 1)))
    {
    }
    __device__ __forceinline__ void sync() const { __syncwarp(mask); }
    __device__ __forceinline__ unsigned ballot(bool p) const { return (__ballot_sync(mask, p) >> base) & kLow; }
    __device__ __forceinline__ int shfl(int v, int src) const { return __shfl_sync(mask, v, base + src); }
    __device__ __forceinline__ uint32_t shfl(uint32_t v, int src) const { return __shfl_sync(mask, v, base + src); }
    __device__ __forceinline__ int rmin(int v) const { return __reduce_min_sync(mask, v); }
    __device__ __forceinline__ int rmax(int v) const { return __reduce_max_sync(mask, v); }
    __device__ __forceinline__ int radd(int v) const { return __reduce_add_sync(mask, v); }
    __device__ __forceinline__ uint32_t rxor(uint32_t v) const { return __reduce_xor_sync(mask, v); }
    __device__ __forceinline__ unsigned rminu(unsigned v) const { return __reduce_min_sync(mask, v); }
};

// Two walkers per warp advancing in lockstep (lanes 16h..16h+15 belong to walker h):
// the same interface as Tile<16>, built from full-warp collectives in which each half
// contributes the neutral value to the other half's reduction.  Only for converged
// code: both halves must reach every call.
struct Pair {
    static constexpr int kSize = 16;
    static constexpr int kHalf = 8;
    int lane;  // 0 .. 15
    int h;     // which walker of the warp
    int base;  // 16 h
    __device__ explicit Pair(int warp_lane) : lane(warp_lane & 15), h(warp_lane >> 4), base(warp_lane & 16) {}
    __device__ __forceinline__ void sync() const { __syncwarp(); }
    __device__ __forceinline__ unsigned ballot(bool p) const { return (__ballot_sync(kFull, p) >> base) & 0xFFFFu; }
    __device__ __forceinline__ int shfl(int v, int src) const { return __shfl_sync(kFull, v, base + src); }
    __device__ __forceinline__ uint32_t shfl(uint32_t v, int src) const { return __shfl_sync(kFull, v, base + src); }
    __device__ __forceinline__ int rmin(int v) const
    {
        const int a = __reduce_min_sync(kFull, h ? INT_MAX : v), b = __reduce_min_sync(kFull, h ? v : INT_MAX);
        return h ? b : a;
    }
    __device__ __forceinline__ unsigned rminu(unsigned v) const
    {
        const unsigned a = __reduce_min_sync(kFull, h ? 0xFFFFFFFFu : v), b = __reduce_min_sync(kFull, h ? v : 0xFFFFFFFFu);
        return h ? b : a;
    }
    __device__ __forceinline__ int rmax(int v) const
    {
        const int a = __reduce_max_sync(kFull, h ? INT_MIN : v), b = __reduce_max_sync(kFull, h ? v : INT_MIN);
        return h ? b : a;
    }
    __device__ __forceinline__ int radd(int v) const
    {
        const int a = __reduce_add_sync(kFull, h ? 0 : v), b = __reduce_add_sync(kFull, h ? v : 0);
        return h ? b : a;
    }
    __device__ __forceinline__ uint32_t rxor(uint32_t v) const
    {
        const uint32_t a = __reduce_xor_sync(kFull, h ? 0u : v), b = __reduce_xor_sync(kFull, h ? v : 0u);
        return h ? b : a;
    }
};

// Four walkers per warp advancing in lockstep (lanes 8h..8h+7 belong to walker h): the
// reductions are butterflies of xor-shuffles that stay inside each group of 8 lanes, so
// one sequence serves all four walkers.  Only for converged code.
struct Quad {
    static constexpr int kSize = 8;
    static constexpr int kHalf = 4;
    int lane;  // 0 .. 7
    int h;     // which walker of the warp
    int base;  // 8 h
    __device__ explicit Quad(int warp_lane) : lane(warp_lane & 7), h(warp_lane >> 3), base(warp_lane & 24) {}
    __device__ __forceinline__ void sync() const { __syncwarp(); }
    __device__ __forceinline__ unsigned ballot(bool p) const { return (__ballot_sync(kFull, p) >> base) & 0xFFu; }
    __device__ __forceinline__ int shfl(int v, int src) const { return __shfl_sync(kFull, v, base + src); }
    __device__ __forceinline__ uint32_t shfl(uint32_t v, int src) const { return __shfl_sync(kFull, v, base + src); }
    __device__ __forceinline__ int rmin(int v) const
    {
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) v = min(v, __shfl_xor_sync(kFull, v, o));
        return v;
    }
    __device__ __forceinline__ unsigned rminu(unsigned v) const
    {
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) v = min(v, __shfl_xor_sync(kFull, v, o));
        return v;
    }
    __device__ __forceinline__ int rmax(int v) const
    {
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(kFull, v, o));
        return v;
    }
    __device__ __forceinline__ int radd(int v) const
    {
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
        return v;
    }
    __device__ __forceinline__ uint32_t rxor(uint32_t v) const
    {
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) v ^= __shfl_xor_sync(kFull, v, o);
        return v;
    }
};

// Per-walker views of the shared-memory layout.
struct View {
    float* A0;    // A0[-apad .. alen-apad)
    float* A1;
    float2* G;    // G[y] = (E[y], E[y+1]), y in [-gpad, glen-gpad)
    uint32_t* B;  // bit-packed classes and reversals, 4 x bvec words
    __half* H0;   // FP16 copies of A0 and A1 for the tensor-core Toeplitz product (null:
    __half* H1;   // none); every write of a row entry writes its copy too
    int* wide;    // long tensor-core layout: nonzero when some |E| is above 2^11 (null: none)
    int gpad;
    int bvec;
};

__device__ __forceinline__ View make_view(int* base, const WarpSmem& L)
{
    View v;
    v.A0 = reinterpret_cast<float*>(base) + L.apad;
    v.A1 = reinterpret_cast<float*>(base) + L.alen + L.apad;
    v.G = reinterpret_cast<float2*>(base + L.goff) + L.gpad;
    v.B = reinterpret_cast<uint32_t*>(base + L.boff);
    v.H0 = L.hlen ? reinterpret_cast<__half*>(base + L.hoff) + L.hpad : nullptr;
    v.H1 = L.hlen ? reinterpret_cast<__half*>(base + L.hoff + L.hlen) + L.hpad : nullptr;
    v.wide = L.foff ? base + L.foff : nullptr;
    v.gpad = L.gpad;
    v.bvec = L.bvec;
    return v;
}

// Row entry u of class p (and its FP16 copy, when the layout keeps one).
__device__ __forceinline__ void set_row(const View& V, int p, int u, float s)
{
    (p ? V.A1 : V.A0)[u] = s;
    if (V.H0 != nullptr) (p ? V.H1 : V.H0)[u] = __float2half_rn(s);
}

// Integers above 2^11 in magnitude are not all FP16 numbers: a table that holds one is
// marked, and its Toeplitz product takes the FP32 pipes until the rows are rebuilt.
__device__ __forceinline__ void note_wide(const View& V, float e)
{
    if (V.wide != nullptr && fabsf(e) > 2048.f) *V.wide = 1;
}

// E[m] = e (m >= 1) in every pair of G that holds it, mirrored to E[-m].
__device__ __forceinline__ void set_E(const View& V, int m, float e)
{
    V.G[m].x = e;
    V.G[m - 1].y = e;
    if (m <= V.gpad) V.G[-m].x = e;
    if (m < V.gpad) V.G[-m - 1].y = e;
}

// Zeroes the walker's rows, table and bit vectors.
template <class TL>
__device__ __forceinline__ void clear_rows(int* base, const WarpSmem& L, const TL& t)
{
    int4* b4 = reinterpret_cast<int4*>(base);
    for (int i = t.lane; i < L.words / 4; i += TL::kSize) b4[i] = make_int4(0, 0, 0, 0);
    t.sync();
}

// Fills A0/A1 from the free-variable bits (word j of the bits lives in tile lane j's
// `word`), by Eq. 4: s_j = x_j for j <= c, s_{c+t} = (-1)^t x_{c-t}.
template <class TL>
__device__ __forceinline__ void rows_from_bits(const View& V, uint32_t word, int L, int n, const TL& t)
{
    const int c = n - 1;
    for (int j0 = 0; j0 < L; j0 += TL::kSize) {
        const int j = j0 + t.lane;
        int f = j <= c ? j : 2 * c - j;
        if (j >= L) f = 0;
        const uint32_t w = t.shfl(word, f >> 5);
        if (j < L) {
            const int x = ((w >> (f & 31)) & 1u) ? -1 : 1;
            const int s = (j > c && ((j - c) & 1)) ? -x : x;
            set_row(V, j & 1, j >> 1, (float)s);
        }
    }
    t.sync();
}

// Bit-packed classes: B[p*bvec + k] holds bits 32k..32k+31 of class p (bit u set
// <=> A_p[u] = -1); B[(2+p)*bvec + k] the same for the reversed class (bit u is
// class entry n_p-1-u).  Zero beyond the class length.  A lane group wider than a warp
// (one walker per CTA) builds one word per warp and round.
template <class TL>
__device__ __forceinline__ void bits_from_rows(const View& V, int n, const TL& t)
{
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        const float* A = p ? V.A1 : V.A0;
        const int np = p ? n - 1 : n;
        if constexpr (TL::kSize > 32) {
            const int wl = t.lane & 31;
            for (int k = t.lane >> 5; k < V.bvec; k += TL::kSize / 32) {
                const int u = 32 * k + wl;
                const uint32_t w = __ballot_sync(kFull, u < np && A[u] < 0.f);
                const uint32_t r = __ballot_sync(kFull, u < np && A[np - 1 - u] < 0.f);
                if (wl == 0) {
                    V.B[p * V.bvec + k] = w;
                    V.B[(2 + p) * V.bvec + k] = r;
                }
            }
        } else {
            // words beyond the class (and its zero word) stay zero: every caller cleared
            // them and no walker of another length shares this walker's memory since
            const int nwd = min(V.bvec, (np + 31) / 32 + 1);
            for (int k = 0; k < nwd; ++k) {
                uint32_t w = 0, r = 0;
#pragma unroll
                for (int h = 0; h < 32 / TL::kSize; ++h) {
                    const int u = 32 * k + TL::kSize * h + t.lane;
                    const uint32_t bw = t.ballot(u < np && A[u] < 0.f);
                    const uint32_t br = t.ballot(u < np && A[np - 1 - u] < 0.f);
                    w |= (TL::kSize == 32) ? bw : (bw << (TL::kSize * h));
                    r |= (TL::kSize == 32) ? br : (br << (TL::kSize * h));
                }
                if (t.lane == 0) {
                    V.B[p * V.bvec + k] = w;
                    V.B[(2 + p) * V.bvec + k] = r;
                }
            }
        }
    }
    t.sync();
}

// Even-lag autocorrelations (Eq. 1) into E and the ISL (Eq. 2) from the bit-packed
// classes: for each class, sum_u a_u a_{u+m} = (n_p - m) - 2 #{u : a_u != a_{u+m}}.
template <class TL>
__device__ __forceinline__ int build_table(const View& V, int n, const TL& t)
{
    bits_from_rows(V, n, t);
    int part = 0;
    const uint32_t* x0 = V.B;
    const uint32_t* x1 = V.B + V.bvec;
    // lags m = mb + g kSize, g < 4, together (eight independent counts), both classes in
    // one pass over the words (lengths n - m and n - 1 - m, same shift)
    constexpr int kG = 4;
    for (int mb = 1 + t.lane; mb < n; mb += kG * TL::kSize) {
        int c0[kG], c1[kG];
#pragma unroll
        for (int g = 0; g < kG; ++g) c0[g] = c1[g] = 0;
        for (int k = 0; 32 * k < n - mb; ++k) {
#pragma unroll
            for (int g = 0; g < kG; ++g) {
                const int m = mb + g * TL::kSize, len0 = n - m, v0 = len0 - 32 * k, v1 = v0 - 1;
                if (v0 > 0) {
                    const int q = m >> 5, r = m & 31;
                    const uint32_t m0 = v0 >= 32 ? ~0u : (1u << v0) - 1u;
                    const uint32_t m1 = v1 >= 32 ? ~0u : (v1 > 0 ? (1u << v1) - 1u : 0u);
                    c0[g] += __popc((x0[k] ^ __funnelshift_r(x0[k + q], x0[k + q + 1], r)) & m0);
                    c1[g] += __popc((x1[k] ^ __funnelshift_r(x1[k + q], x1[k + q + 1], r)) & m1);
                }
            }
        }
#pragma unroll
        for (int g = 0; g < kG; ++g) {
            const int m = mb + g * TL::kSize;
            if (m < n) {
                const int len0 = n - m, len1 = len0 - 1;
                const int d = len0 - 2 * c0[g] + (len1 > 0 ? len1 - 2 * c1[g] : 0);
                set_E(V, m, (float)d);
                if constexpr (TL::kSize > 32) note_wide(V, (float)d);
                part += d * d;
            }
        }
    }
    t.sync();
    return t.radd(part);
}

// Lane layout of the neighbourhood: the first half of the tile holds the even class,
// the second half the odd class; lane l of a half owns outputs v0 .. v0+R-1.
template <class TL, int R>
struct Outs {
    int p, v0;
    __device__ explicit Outs(const TL& t) : p(t.lane / TL::kHalf), v0((t.lane % TL::kHalf) * R) {}
};

// X_v = sum_u A_p[u] E[u-v] for the lane's R outputs v = v0..v0+R-1 (the Toeplitz
// product), on the FP32 pipes with packed pairs: accumulator r holds the partial sums
// of X_{v0+r} over even u (.x) and odd u (.y), so one __ffma2_rn multiplies the pair
// (A[u], A[u+1]) by G[u-v] = (E[u-v], E[u+1-v]).  The window win[j] = G[u-v0-j] slides
// two positions per pair of u: two 8-byte loads per R packed FMAs.  All operands and
// partial sums are integers below 2^24, so the result is exact.
// Outputs C0 .. C0+RC-1 of the lane's block (G already offset by -v0).
template <int R, int C0, int RC>
__device__ __forceinline__ void toeplitz_part(const float* A, const float2* G, int nu, float (&X)[R])
{
    float2 acc[RC], win[RC];
#pragma unroll
    for (int r = 0; r < RC; ++r) {
        acc[r] = make_float2(0.f, 0.f);
        win[r] = G[-C0 - r];
    }
#pragma unroll kToeplitzUnroll
    for (int u = 0; u < nu; u += 8) {
        const float4 a0 = *reinterpret_cast<const float4*>(A + u);
        const float4 a1 = *reinterpret_cast<const float4*>(A + u + 4);
        const float2 ap[4] = {make_float2(a0.x, a0.y), make_float2(a0.z, a0.w), make_float2(a1.x, a1.y),
                              make_float2(a1.z, a1.w)};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
#pragma unroll
            for (int r = 0; r < RC; ++r) acc[r] = __ffma2_rn(ap[q], win[r], acc[r]);
#pragma unroll
            for (int j = RC - 1; j >= 2; --j) win[j] = win[j - 2];
            if (RC >= 2) win[1] = G[u + 2 * q + 1 - C0];
            win[0] = G[u + 2 * q + 2 - C0];
        }
    }
#pragma unroll
    for (int r = 0; r < RC; ++r) X[C0 + r] = acc[r].x + acc[r].y;
}

// All R outputs in one pass over u.
template <class TL, int R>
__device__ __forceinline__ void toeplitz(const View& V, int n, const Outs<TL, R>& o, float (&X)[R])
{
    const float* A = o.p ? V.A1 : V.A0;
    toeplitz_part<R, 0, R>(A, V.G - o.v0, (n + 7) & ~7, X);
}

// The Toeplitz product on the tensor cores.  In blocks of 16, u = 16 s + j and v = 16 t + i,
// it is
//   X_t = sum_d T_d A_{t+d},   T_d[i][j] = E[16 d + j - i],   A_s[j] = A_p[16 s + j],
// a sum over the block diagonals d of a 16 x 16 Toeplitz block of the table times the
// row blocks d further.  One mma.sync.m16n8k16 per diagonal takes T_d (rows i, columns
// j) and, as its 8 columns, the row blocks of output blocks t = 0..3 of both classes
// (columns 0-3 class 0, 4-7 class 1); d runs from -(T-1) to S-1 for the T output and S
// row blocks.  The table's entries are rounded to FP16 as they are loaded (|E| < 2^11
// is exact), the rows come from their FP16 copies (A = 0, +-1), and the products
// accumulate in FP32: every partial sum is an integer below 2^24, so the result equals
// the FP32 product's.  Reads outside the class meet the rows' zero padding, and E is
// finite (zero) beyond the table.
__device__ __forceinline__ uint32_t half2_bits(float2 v)
{
    const __half2 h = __float22half2_rn(v);  // .x in the low half
    return *reinterpret_cast<const uint32_t*>(&h);
}

__device__ __forceinline__ void mma_16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                          uint32_t b0, uint32_t b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// One block diagonal of one walker: T_d from the table pairs at gy (and the pair 8 below,
// carried in am8), the row blocks' FP16 pairs at ab.
__device__ __forceinline__ void tc_diag(float (&d)[4], const float2* gy, const uint32_t* ab, uint32_t& am8)
{
    const uint32_t a0 = half2_bits(gy[0]), a2 = half2_bits(gy[8]);
    mma_16816(d, a0, am8, a2, a0, ab[0], ab[4]);
    am8 = a2;
}

// One walker on one warp: the output blocks form M = ceil(T/4)
// column groups of 4 blocks per class (M <= 2 for n <= 256), and for group m the block
// diagonals run from -(4m+3) (or -(T-1)) up to S-1-4m.  Two accumulator chains (two
// groups, or the even and odd diagonals of a lone group; integer partial sums, so the
// split does not change the result).  The results go through the walker's scratch X[2][xp]
// to the lanes' R outputs.
template <class LG, int R>
__device__ __forceinline__ void toeplitz_tc1(const View& V, const WarpSmem& SL, int n, const Outs<LG, R>& o,
                                             const LG& t, float (&X)[R])
{
    const int l = threadIdx.x & 31, g = l >> 2, tq = l & 3;
    const int S = (n + 15) >> 4, T = (((n + 1) >> 1) + 15) >> 4, M = (T + 3) >> 2;
    const int pb = g >> 2, tb = g & 3, px = tq >> 1, tx = 2 * (tq & 1);
    int* const base = reinterpret_cast<int*>(V.A0) - SL.apad;
    const float2* G = reinterpret_cast<const float2*>(base + SL.goff) + SL.gpad + (2 * tq - g);
    const uint32_t* H = reinterpret_cast<const uint32_t*>(base + SL.hoff + pb * SL.hlen) + (SL.hpad >> 1) + 8 * tb + tq;
    float* xs = reinterpret_cast<float*>(base + SL.roff) + px * SL.xp + g;
    const int dloA = -min(3, T - 1), dhi = S - 1;  // group 0: d = dloA .. dhi
    if (M > 1) {
        // both groups together: a diagonal's table fragment is loaded once for both
        const int dlo = -(T - 1), dhiB = dhi - 4;  // group 1: d = dlo .. dhiB
        const float2* gy = G + 16 * dlo;
        const uint32_t* ab = H + 8 * dlo;  // group 0's operand; group 1's is 32 words further
        float dA[4] = {0.f, 0.f, 0.f, 0.f}, dB[4] = {0.f, 0.f, 0.f, 0.f};
        uint32_t am = half2_bits(gy[-8]);
        for (int d = dlo; d <= dhi; ++d) {
            const uint32_t a0 = half2_bits(gy[0]), a2 = half2_bits(gy[8]);
            if (d >= dloA) mma_16816(dA, a0, am, a2, a0, ab[0], ab[4]);
            if (d <= dhiB) mma_16816(dB, a0, am, a2, a0, ab[32], ab[36]);
            am = a2;
            gy += 16;
            ab += 8;
        }
        const int tB = tx + 4;
        xs[16 * tx] = dA[0];
        xs[16 * tx + 8] = dA[2];
        xs[16 * tx + 16] = dA[1];
        xs[16 * tx + 24] = dA[3];
        if (tB < T) {
            xs[16 * tB] = dB[0];
            xs[16 * tB + 8] = dB[2];
        }
        if (tB + 1 < T) {
            xs[16 * tB + 16] = dB[1];
            xs[16 * tB + 24] = dB[3];
        }
    } else {
        const int nd = dhi - dloA + 1;
        const float2* gy = G + 16 * dloA;
        const uint32_t* ab = H + 8 * dloA;
        float d0[4] = {0.f, 0.f, 0.f, 0.f}, d1[4] = {0.f, 0.f, 0.f, 0.f};
        uint32_t am = half2_bits(gy[-8]);
        int k = 0;
        for (; k + 1 < nd; k += 2) {
            tc_diag(d0, gy, ab, am);
            tc_diag(d1, gy + 16, ab + 8, am);
            gy += 32;
            ab += 16;
        }
        if (k < nd) tc_diag(d0, gy, ab, am);
        if (tx < T) {
            xs[16 * tx] = d0[0] + d1[0];
            xs[16 * tx + 8] = d0[2] + d1[2];
        }
        if (tx + 1 < T) {
            xs[16 * tx + 16] = d0[1] + d1[1];
            xs[16 * tx + 24] = d0[3] + d1[3];
        }
    }
    t.sync();
    const float* xr = reinterpret_cast<const float*>(base + SL.roff) + o.p * SL.xp + o.v0;
#pragma unroll
    for (int r = 0; r < R; ++r) X[r] = xr[r];
}

// The product of a walker that a CTA of W warps owns (n > 256, M = ceil(T/4) >= 3 column
// groups).  A warp's operands are what bounds it, so it takes GC = 2 to 4 column groups at
// once, and the diagonals in chunks of four: group m + 1 needs at diagonal d the row
// blocks that group m needs at d + 4, so a chunk's row fragments, loaded once by ldmatrix
// (two MMAs' operands each), pass through a ring to the next group a chunk later, and the
// table fragments of a diagonal serve all GC groups: 10 loads for 16 MMAs (two row words
// and, for every second MMA, two table pairs to convert before, with tests of the diagonal
// around each).  608 walkers x 512 steps at L = 4095: 11.2 ms from 17.2; the tensor pipe is
// now busy 45% of the time, the rest is the step around it.  Chunk k of a set of groups that
// starts at m0 has d = 4k .. 4k+3 and the row blocks 4 (k + m0 + j) + 0..6 for group j;
// k runs from -(m0 + GC), where the last group meets its first row block, to C - m0, C
// the chunk of the last row block; what lies outside the class meets the rows' zeros.
template <int GC>
__device__ __forceinline__ void tc_chunks(float (&acc)[GC][4], const float2* gy, uint32_t ha, int nk)
{
    uint32_t F[GC][8];
    const auto load = [&](uint32_t (&f)[8], uint32_t a) {
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                     : "=r"(f[0]), "=r"(f[1]), "=r"(f[2]), "=r"(f[3])
                     : "r"(a));
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                     : "=r"(f[4]), "=r"(f[5]), "=r"(f[6]), "=r"(f[7])
                     : "r"(a + 64u));
    };
#pragma unroll
    for (int j = 0; j < GC - 1; ++j) {
        load(F[j], ha);
        ha += 128u;
    }
    uint32_t am = half2_bits(gy[-8]);
    for (;;) {
#pragma unroll
        for (int s = 0; s < GC; ++s) {
            load(F[(s + GC - 1) % GC], ha);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t a0 = half2_bits(gy[16 * i]), a2 = half2_bits(gy[16 * i + 8]);
#pragma unroll
                for (int j = 0; j < GC; ++j)
                    mma_16816(acc[j], a0, am, a2, a0, F[(s + j) % GC][2 * i], F[(s + j) % GC][2 * i + 1]);
                am = a2;
            }
            gy += 64;
            ha += 128u;
            if (--nk == 0) return;
        }
    }
}

// One set's chunks k0 .. k0 + nk - 1, added to the integer sums xs (whole numbers, so the
// order of the warps' additions does not change them).
template <int GC>
__device__ __forceinline__ void tc_set(const float2* G, uint32_t H, int* xs, int m0, int k0, int nk, int T, int tx)
{
    float acc[GC][4];
#pragma unroll
    for (int j = 0; j < GC; ++j)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[j][q] = 0.f;
    tc_chunks<GC>(acc, G + 64 * k0, H + 128u * (uint32_t)(k0 + m0), nk);
#pragma unroll
    for (int j = 0; j < GC; ++j) {
        const int t0 = tx + 4 * (m0 + j);
        if (t0 < T) {
            atomicAdd(xs + 16 * t0, __float2int_rn(acc[j][0]));
            atomicAdd(xs + 16 * t0 + 8, __float2int_rn(acc[j][2]));
        }
        if (t0 + 1 < T) {
            atomicAdd(xs + 16 * t0 + 16, __float2int_rn(acc[j][1]));
            atomicAdd(xs + 16 * t0 + 24, __float2int_rn(acc[j][3]));
        }
    }
}

// The sets (Q = ceil(M/4), of ceil or floor M/Q groups) and their chunks are one line of
// work, cut into W equal pieces.  The sums start at zero (long_clear) and are zeroed again
// as they are read.
template <class LB, int R>
__device__ __forceinline__ void toeplitz_long(const View& V, const WarpSmem& SL, int n, const Outs<LB, R>& o,
                                              const LB& t, float (&X)[R])
{
    constexpr int W = LB::kSize / 32;
    const int warp = __shfl_sync(kFull, (int)(threadIdx.x >> 5), 0);
    const int l = threadIdx.x & 31, g = l >> 2, tq = l & 3, px = tq >> 1, tx = 2 * (tq & 1);
    const int S = (n + 15) >> 4, T = (((n + 1) >> 1) + 15) >> 4, M = (T + 3) >> 2;
    const int C = (S - 1) >> 2, Q = (M + 3) >> 2, few = M / Q, more = M - few * Q;
    int* const base = reinterpret_cast<int*>(V.A0) - SL.apad;
    const float2* G = V.G + (2 * tq - g);
    // ldmatrix row of this lane: operand column l & 7 (class, block), half block (l >> 3) & 1,
    // the chunk's even or odd diagonal l >> 4
    const uint32_t H =
        (uint32_t)__cvta_generic_to_shared(reinterpret_cast<__half*>(base + SL.hoff + ((l >> 2) & 1) * SL.hlen) +
                                           SL.hpad + 16 * ((l & 3) + (l >> 4)) + 8 * ((l >> 3) & 1));
    int* const xi = base + SL.roff;
    int* const xs = xi + px * SL.xp + g;
    const int total = Q * (C + 1) + M;  // chunks of all sets: C + 1 + their groups
    int at = warp * total / W, left = (warp + 1) * total / W - at;
    for (int q = 0, m0 = 0; q < Q && left > 0; ++q) {
        const int gc = few + (q < more ? 1 : 0), nk = C + 1 + gc;
        if (at < nk) {
            const int k0 = at - (m0 + gc), take = min(nk - at, left);
            if (gc == 4) tc_set<4>(G, H, xs, m0, k0, take, T, tx);
            else if (gc == 3) tc_set<3>(G, H, xs, m0, k0, take, T, tx);
            else tc_set<2>(G, H, xs, m0, k0, take, T, tx);
            left -= take;
            at = nk;
        }
        at -= nk;
        m0 += gc;
    }
    t.sync();
    int* xr = xi + o.p * SL.xp + o.v0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        X[r] = (float)xr[r];
        xr[r] = 0;
    }
}

// The product of a walker that a CTA of four warps owns with no more column groups than warps:
// a warp takes one group, its even and odd diagonals as the two chains (toeplitz_tc1's form),
// and no sums meet; the pieces of toeplitz_long are too short there for its ring.  608 walkers x
// 256 steps of L = 513 / 769 / 897 0.881 / 1.065 / 1.122 ms like this and 0.911 / 1.079 / 1.106
// with toeplitz_long, best-first x 128 2.21 / 2.75 / 2.84 and 2.25 / 2.80 / 2.85: the line lies
// between the last two.  (The PSL walk, on eight warps there, keeps toeplitz_long: 3.61 ms at
// L = 513, 3.65 like this.)
constexpr int kGroupsMaxN = 400;
template <class LB, int R>
__device__ __forceinline__ void toeplitz_groups(const View& V, const WarpSmem& SL, int n, const Outs<LB, R>& o,
                                                const LB& t, float (&X)[R])
{
    const int m = threadIdx.x >> 5, l = threadIdx.x & 31, g = l >> 2, tq = l & 3;
    const int S = (n + 15) >> 4, T = (((n + 1) >> 1) + 15) >> 4, M = (T + 3) >> 2;
    const int pb = g >> 2, tb = g & 3, px = tq >> 1, tx = 2 * (tq & 1);
    int* const base = reinterpret_cast<int*>(V.A0) - SL.apad;
    float* const xf = reinterpret_cast<float*>(base + SL.roff);
    if (m < M) {
        const int dlo = -min(4 * m + 3, T - 1), nd = S - 4 * m - dlo;  // d = dlo .. S-1-4m
        const float2* gy = V.G + (2 * tq - g) + 16 * dlo;
        const uint32_t* ab = reinterpret_cast<const uint32_t*>(base + SL.hoff + pb * SL.hlen) + (SL.hpad >> 1) +
                             8 * (tb + 4 * m + dlo) + tq;
        float d0[4] = {0.f, 0.f, 0.f, 0.f}, d1[4] = {0.f, 0.f, 0.f, 0.f};
        uint32_t am = half2_bits(gy[-8]);
        int k = 0;
        for (; k + 1 < nd; k += 2) {
            tc_diag(d0, gy, ab, am);
            tc_diag(d1, gy + 16, ab + 8, am);
            gy += 32;
            ab += 16;
        }
        if (k < nd) tc_diag(d0, gy, ab, am);
        float* const xs = xf + px * SL.xp + g;
        const int t0 = tx + 4 * m;
        if (t0 < T) {
            xs[16 * t0] = d0[0] + d1[0];
            xs[16 * t0 + 8] = d0[2] + d1[2];
        }
        if (t0 + 1 < T) {
            xs[16 * t0 + 16] = d0[1] + d1[1];
            xs[16 * t0 + 24] = d0[3] + d1[3];
        }
    }
    t.sync();
    const float* const xr = xf + o.p * SL.xp + o.v0;
#pragma unroll
    for (int r = 0; r < R; ++r) X[r] = xr[r];
}

// The Toeplitz product of a lane group that owns one walker: on the tensor cores when
// the layout holds the FP16 rows and the results' scratch (and the table's entries are
// FP16 numbers), else on the FP32 pipes.
template <class LG, int R>
__device__ __forceinline__ void toeplitz_one(const View& V, const WarpSmem& SL, int n, const Outs<LG, R>& o,
                                             const LG& t, float (&X)[R])
{
    if constexpr (LG::kSize > 32) {
        if (SL.xp != 0 && *V.wide == 0) {
            // (lane blocks that such a length can have; a context of longer ones takes the other)
            if constexpr (LG::kSize == 128 && R <= 5) {
                if (n <= kGroupsMaxN) {
                    toeplitz_groups(V, SL, n, o, t, X);
                    return;
                }
            }
            toeplitz_long(V, SL, n, o, t, X);
            return;
        }
    } else if constexpr (LG::kSize == 32) {
        if (SL.xp != 0) {
            toeplitz_tc1(V, SL, n, o, t, X);
            return;
        }
    }
    toeplitz(V, n, o, X);
}

// P_v = sum_{m=1}^{v} A_p[v+m] A_p[v-m] from scratch for the lane's outputs, from the
// bit-packed classes (built by build_table): the pairs compare bits v+1.. of the
// class with bits n_p-v.. of the reversed class, P_v = v - 2 #{mismatches}.
template <class TL, int R>
__device__ __forceinline__ void p_direct(const View& V, int n, const Outs<TL, R>& o, float (&P)[R])
{
    const int np = o.p ? n - 1 : n;
    const int nv = o.p ? (n >> 1) : ((n + 1) >> 1);
    const uint32_t* x = V.B + o.p * V.bvec;
    const uint32_t* xr = V.B + (2 + o.p) * V.bvec;
    // the R outputs word by word (independent chains); output v compares v bits
    int cnt[R];
#pragma unroll
    for (int r = 0; r < R; ++r) cnt[r] = 0;
    const int vtop = min(o.v0 + R - 1, nv - 1);
    for (int k = 0; 32 * k < vtop; ++k) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int v = o.v0 + r;
            const int valid = v - 32 * k;
            if (v < nv && valid > 0) {
                const uint32_t a = __funnelshift_r(x[k + ((v + 1) >> 5)], x[k + ((v + 1) >> 5) + 1], (v + 1) & 31);
                const uint32_t b = __funnelshift_r(xr[k + ((np - v) >> 5)], xr[k + ((np - v) >> 5) + 1], (np - v) & 31);
                const uint32_t mk = valid >= 32 ? ~0u : (1u << valid) - 1u;
                cnt[r] += __popc((a ^ b) & mk);
            }
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int v = o.v0 + r;
        P[r] = (v >= nv || v == 0) ? 0.f : (float)(v - 2 * cnt[r]);
    }
}

// Change of P for a move that negates class-pb entries w1 and w2 (w2 < 0: centre, one
// entry).  A pair (v+m, v-m) with exactly one negated end changes by -2 x its old
// product; pairs with both ends negated are unchanged.  Reads A before the flip.
template <class TL, int R>
__device__ __forceinline__ void p_update(const View& V, int n, const Outs<TL, R>& o, float (&P)[R], int pb, int w1,
                                         int w2)
{
    if (o.p != pb) return;
    const float* A = pb ? V.A1 : V.A0;
    const int nv = pb ? (n >> 1) : ((n + 1) >> 1);
    const float a1 = A[w1];
    const float a2 = w2 >= 0 ? A[w2] : 0.f;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int v = o.v0 + r;
        if (v >= nv) continue;
        float d = 0.f;
        const int t1 = 2 * v - w1;
        if (v != w1 && t1 != w2) d = a1 * A[t1];
        if (w2 >= 0) {
            const int t2 = 2 * v - w2;
            if (v != w2 && t2 != w1) d = fmaf(a2, A[t2], d);
        }
        P[r] = fmaf(-2.f, d, P[r]);
    }
}

// dl[r] = dISL of free variable i = 2(v0+r)+p, or INT_MAX where that output does not
// exist.  Formula in the header comment; evaluated in exact float arithmetic (all
// terms are integers below 2^24) and converted once.
template <class TL, int R>
__device__ __forceinline__ void assemble(const View& V, int n, const Outs<TL, R>& o, const float (&X)[R],
                                         const float (&P)[R], int (&dl)[R])
{
    const int p = o.p;
    const float* A = p ? V.A1 : V.A0;
    const int nv = p ? (n >> 1) : ((n + 1) >> 1);
    const int c = n - 1;
    const float base = (float)(16 * ((p ? n - 2 : n - 1) - 1));
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int v = o.v0 + r;
        if (v >= nv) {
            dl[r] = INT_MAX;
            continue;
        }
        const int i = 2 * v + p;
        const float av = A[v];
        if (i == c) {
            dl[r] = __float2int_rn(fmaf(-4.f * av, X[r], (float)(16 * (c >> 1))));
            continue;
        }
        const float sq = A[n - 1 - v - p];
        const float ck0 = V.G[c - i].x;
        const int t = 3 * v + p - n + 1;
        const float corr = t >= 0 ? sq * A[t] : 0.f;
        dl[r] = __float2int_rn(fmaf(-8.f * av, fmaf(-sq, ck0, X[r]), fmaf(32.f, P[r] - corr, base)));
    }
}

// Rebuilds the walker's rows and table from its bits; returns the ISL.
template <class TL>
__device__ __forceinline__ int load_rows(int* base, const WarpSmem& SL, const View& V, uint32_t word, int L, int n,
                                         const TL& t)
{
    clear_rows(base, SL, t);
    rows_from_bits(V, word, L, n, t);
    return build_table(V, n, t);
}

// HT fingerprint (Zobrist): XOR of the keys of the free variables equal to -1.
template <class TL>
__device__ __forceinline__ uint64_t fingerprint_all(uint32_t word, const uint64_t* zk, int n, const TL& t)
{
    uint64_t f = 0;
    const int nr = (n + TL::kSize - 1) & ~(TL::kSize - 1);
    for (int i0 = 0; i0 < nr; i0 += TL::kSize) {
        const int i = i0 + t.lane;
        const uint32_t w = t.shfl(word, i0 >> 5);
        if (i < n && ((w >> (i & 31)) & 1u)) f ^= __ldg(zk + i);
    }
    const uint32_t lo = t.rxor((uint32_t)f);
    const uint32_t hi = t.rxor((uint32_t)(f >> 32));
    return (uint64_t)lo | ((uint64_t)hi << 32);
}

// Registers of one walker while its tile runs it.
struct Walker {
    uint32_t word;   // tile lane j < 8: bits word j
    uint64_t fp;
    int isl, best_isl, since, stag;
    uint32_t restart_idx, gen;
    int restarts, overflows, blocked;
    int64_t steps, best_step, target_step;
};

struct WalkEnv {
    const KParams* p;
    uint64_t* T;       // this walker's HT
    uint64_t tmask;
    const uint64_t* zk;
    WalkerState* st;
    int L, n, patience;
    uint32_t g;
    // learned mode (null when off): proposed restart state and its flag
    uint32_t* slot;
    int32_t* slot_valid;
    // replay dumps of a traced walker in learned mode (null when off)
    uint32_t* rdump;   // [cap][8]
    int64_t* rdump_idx;
    int32_t* rdump_count;
    int dump_cap;
};

__device__ __forceinline__ bool target_met(const KParams& p, int L, int isl)
{
    if (p.target_num <= 0 || p.target_den <= 0) return false;
    return (int64_t)p.target_den * L * L >= 2 * (int64_t)p.target_num * isl;
}

// PSL objective: the current sequence's PSL, and the PSL halves of the (PSL, ISL)
// pairs of the best sequence and of the best since the last (re)start.
struct PslTrack {
    int psl, best_psl, since_psl;
};

// Lower (PSL, ISL) pair, compared lexicographically.
__device__ __forceinline__ bool psl_better(int psl, int isl, int psl0, int isl0)
{
    return psl < psl0 || (psl == psl0 && isl < isl0);
}

// max |C_{2m}| over m = 1..n-1 from the table: the PSL of a skew-symmetric sequence
// (Section 1; its odd-lag C_k vanish).
template <class TL>
__device__ __forceinline__ int table_psl(const View& V, int n, const TL& t)
{
    int mx = 0;
    for (int m = 1 + t.lane; m < n; m += TL::kSize) mx = max(mx, abs(__float2int_rn(V.G[m].x)));
    return t.rmax(mx);
}

// Best-sequence update: strictly lower ISL, or under the PSL objective (ps != null) a
// strictly lower (PSL, ISL) pair.
template <class TL>
__device__ __forceinline__ void note_best(const WalkEnv& env, Walker& w, const TL& t, PslTrack* ps = nullptr)
{
    const bool better = ps ? psl_better(ps->psl, w.isl, ps->best_psl, w.best_isl) : w.isl < w.best_isl;
    if (better) {
        w.best_isl = w.isl;
        if (ps) ps->best_psl = ps->psl;
        w.best_step = w.steps;
        if (t.lane < kBitWords) env.st->best[t.lane] = w.word;
    }
    if (w.target_step < 0 && target_met(*env.p, env.L, w.isl)) w.target_step = w.steps;
}

// Algorithm 1 start: random skew-symmetric S (restart index w.restart_idx), its ISL,
// insert it into HT (a fresh generation: its home slot is free), best update.
template <class TL>
__device__ void start_walker(const WalkEnv& env, Walker& w, int* base, const WarpSmem& SL, const View& V,
                             const TL& t, bool proposed = false, PslTrack* ps = nullptr)
{
    const int lane = t.lane;
    if (proposed) {
        // learned mode: the restart state chosen by the proposal pass replaces the draw
        w.word = lane < kBitWords ? env.slot[lane] : 0u;
        if (env.rdump != nullptr) {
            const int k = *env.rdump_count;
            if (k < env.dump_cap) {
                if (lane < kBitWords) env.rdump[(int64_t)k * kBitWords + lane] = w.word;
                if (lane == 0) env.rdump_idx[k] = w.restart_idx;
            }
            t.sync();
            if (lane == 0) *env.rdump_count = k + 1;
        }
        t.sync();
        if (lane == 0) *env.slot_valid = 0;
    } else {
        w.word = lane < kBitWords ? start_word(env.p->seed, env.g, w.restart_idx, lane, env.n) : 0u;
    }
    w.isl = load_rows(base, SL, V, w.word, env.L, env.n, t);
    w.fp = fingerprint_all(w.word, env.zk, env.n, t);
    if (lane == 0) env.T[w.fp & env.tmask] = (w.fp & ~kGenMask) | w.gen;
    t.sync();
    w.since = w.isl;
    w.stag = 0;
    if (ps) {
        ps->psl = table_psl(V, env.n, t);
        ps->since_psl = ps->psl;
    }
    note_best(env, w, t, ps);
}

template <class TL>
__device__ void restart_walker(const WalkEnv& env, Walker& w, int* base, const WarpSmem& SL, const View& V,
                               const TL& t, PslTrack* ps = nullptr)
{
    w.restart_idx += 1;
    w.restarts += 1;
    w.gen += 1;
    if (w.gen > kGenMask) {
        const int64_t slots = (int64_t)env.tmask + 1;
        for (int64_t i = t.lane; i < slots; i += TL::kSize) env.T[i] = 0ull;
        t.sync();
        w.gen = 1;
    }
    int prop = 0;
    if (t.lane == 0 && env.slot_valid != nullptr) prop = *env.slot_valid != 0;
    const bool proposed = t.shfl(prop, 0) != 0;
    start_walker(env, w, base, SL, V, t, proposed, ps);
}

// Stop requests from the host-written control block (mapped host memory, slow to
// read).  One lane (`reader`) reads the deadline and the cancel flag when a walk call
// starts; after that it re-reads the cancel flag at every poll without waiting for it:
// the value lands while the steps run and is acted on at the next poll, kCheckEvery
// steps later.  The deadline is compared with %globaltimer at every poll.
struct StopCheck {
    uint64_t deadline = ~0ull;
    int next = 0;
    __device__ __forceinline__ void start(const KParams& p, bool reader)
    {
        if (reader && p.ctrl != nullptr) {
            deadline = p.ctrl->deadline_ns;
            next = p.ctrl->stop;
        }
    }
    // LABS_ECANCELLED, LABS_ETIMEOUT or 0, in the reader lane (0 elsewhere)
    __device__ __forceinline__ int poll(const KParams& p, bool reader)
    {
        int why = 0;
        if (reader && p.ctrl != nullptr) {
            if (next) why = LABS_ECANCELLED;
            else if (global_ns() >= deadline) why = LABS_ETIMEOUT;
            next = p.ctrl->stop;
        }
        return why;
    }
};

// Result of probing HT for one candidate.
struct Probe {
    bool visited;
    int64_t slot;  // insertion slot when not visited, -1 when no free slot within the cap
};

// Full linear probe of f: up to `cap` slots, TILE at a time.
template <class TL>
__device__ __forceinline__ Probe probe_full(const WalkEnv& env, uint64_t f, uint32_t gen, int cap, const TL& t)
{
    const uint64_t tag = (f & ~kGenMask) | gen;
    Probe pr{false, -1};
    for (int s0 = 0; s0 < cap; s0 += TL::kSize) {
        const int s = s0 + t.lane;
        uint64_t e = 0;
        if (s < cap) e = env.T[(f + (uint64_t)s) & env.tmask];
        const bool match = e == tag;
        const unsigned bal = t.ballot(s < cap && (((e & kGenMask) != gen) || match));
        if (bal) {
            const int fl = __ffs(bal) - 1;
            pr.visited = t.shfl(match ? 1 : 0, fl) != 0;
            pr.slot = (int64_t)((f + (uint64_t)(s0 + fl)) & env.tmask);
            break;
        }
    }
    return pr;
}

// Lowest (dl, i) among the lane outputs not in `excl` (every lane of the tile gets the
// result; bi = -1 when none is left).
template <class TL, int R>
__device__ __forceinline__ void tile_argmin(const int (&dl)[R], uint32_t excl, const Outs<TL, R>& o,
                                            const TL& t, int& bd, int& bi)
{
    int lm = INT_MAX, li = INT_MAX;
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (!((excl >> r) & 1u) && dl[r] < lm) {
            lm = dl[r];
            li = 2 * (o.v0 + r) + o.p;
        }
    bd = t.rmin(lm);
    bi = bd == INT_MAX ? -1 : t.rmin(lm == bd ? li : INT_MAX);
}

template <class TL, int R>
__device__ __forceinline__ void exclude(uint32_t& excl, int bi, const TL& t)
{
    const int vb = bi >> 1, pb = bi & 1;
    if (t.lane == pb * TL::kHalf + vb / R) excl |= 1u << (vb % R);
}

// Order-preserving map of a float score to int32 (the learned ordering compares these).
__device__ __forceinline__ int score_key(float f)
{
    const int k = __float_as_int(f);
    return k >= 0 ? k : (k ^ 0x7FFFFFFF);
}

// S <- S_f for free variable bi: the table E (C_{2m} += -4 s_i (s_{i-2m} + s_{i+2m}),
// the mirror's own term left out, -2 s_c (..) at the centre), P and the two row
// entries, all from the values before the flip.  Ends without a tile barrier.
template <class TL, int R>
__device__ __forceinline__ void flip_rows_table(const View& V, int n, const Outs<TL, R>& o, float (&P)[R], int bi,
                                                const TL& t)
{
    const int lane = t.lane, c = n - 1;
    const int pb = bi & 1, vb = bi >> 1;
    float* Ab = pb ? V.A1 : V.A0;
    const float as = Ab[vb];
    const bool centre = bi == c;
    const int vq = n - 1 - vb - pb;
    float dd[R];
#pragma unroll
    for (int k = 0; k < R; ++k) {  // lags 2m, m = lane+1+TILE k < n (n <= TILE R)
        const int m = lane + 1 + TL::kSize * k;
        dd[k] = 0.f;
        if (m < n) {
            float up = Ab[vb + m];
            if (!centre && vb + m == vq) up = 0.f;
            const float dn = Ab[vb - m];
            dd[k] = ((centre ? -2.f : -4.f) * as) * (up + dn);
        }
    }
    p_update(V, n, o, P, pb, vb, centre ? -1 : vq);
    t.sync();
#pragma unroll
    for (int k = 0; k < R; ++k) {
        const int m = lane + 1 + TL::kSize * k;
        if (m < n) {
            const float e = V.G[m].x + dd[k];
            set_E(V, m, e);
            if constexpr (TL::kSize > 32) note_wide(V, e);
        }
    }
    if (lane == 0) {
        set_row(V, pb, vb, -as);
        if (!centre) set_row(V, pb, vq, -Ab[vq]);
    }
}

// What a walk call records besides the trajectory.
struct StepExtras {
    const float* scores;  // learned flip scores for the first step of this call, or null
    int tau;              // learned candidates: dISL <= min dISL + tau
    float* sdump;         // replay dump of the scores used (traced walker), or null
    int64_t* sdump_step;
    int32_t* sdump_count;
    int dump_cap, n_max;
    labs_log_record* rec; // log record of this chunk, or null
};

template <class TL, int R>
__device__ void walk_steps(const WalkEnv& env, Walker& w, int64_t until, int* base, const WarpSmem& SL,
                           const View& V, int trace_slot, int64_t trace_start, const StepExtras& ex,
                           const TL& t)
{
    const KParams& p = *env.p;
    const int lane = t.lane, n = env.n;
    const Outs<TL, R> o(t);
    const int cap = p.probe_cap;
    constexpr int S = TL::kSize / 2;  // probe slots per candidate in the two-candidate round
    float P[R];
    p_direct(V, n, o, P);
    const int64_t first_step = w.steps;
    int log_first = 0, log_min = w.isl;
    bool log_live = true;
    StopCheck stop;
    stop.start(p, lane == 0);
    if (ex.rec != nullptr) {
        if (lane < kBitWords) ex.rec->bits[lane] = w.word;
        if (lane == 0) {
            ex.rec->isl = w.isl;
            ex.rec->L = env.L;
            ex.rec->walker = env.g;
            ex.rec->step = w.steps;
        }
    }
    while (w.steps < until) {
        if ((w.steps & (kCheckEvery - 1)) == 0) {
            const int why = t.shfl(stop.poll(p, lane == 0), 0);
            if (why) {
                if (lane == 0) raise_error(p.status, why, (int)env.g);
                break;
            }
        }
        int dl[R];
        {
            float X[R];
            toeplitz_one(V, SL, n, o, t, X);
            assemble(V, n, o, X, P, dl);
        }

        // Best admissible flip: lowest (dISL, i) whose result is not in HT.  Two
        // candidates are probed per round, TILE/2 slots each (half the tile per
        // candidate); a longer chain falls back to a full probe.  The chosen flip is
        // the best one in about 40% of the steps and one of the best two in about 86%
        // (L = 201).
        uint32_t excl = 0;
        int best_i = -1, best_d = 0;
        int64_t slot = -1;
        uint64_t fnew = 0;
        if (ex.scores != nullptr && w.steps == first_step) {
            // Learned step: among the flips with dISL <= min dISL + tau, try them by
            // (score descending, i ascending) first; the plain order follows.
            int lm = INT_MAX;
#pragma unroll
            for (int r = 0; r < R; ++r) lm = min(lm, dl[r]);
            const int dmin = t.rmin(lm);
            const int thr = dmin > INT_MAX - ex.tau ? INT_MAX - 1 : dmin + ex.tau;
            int keys[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int i = 2 * (o.v0 + r) + o.p;
                keys[r] = dl[r] <= thr ? score_key(ex.scores[i]) : INT_MIN;
            }
            if (ex.sdump != nullptr) {
                const int k = *ex.sdump_count;
                if (k < ex.dump_cap) {
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const int i = 2 * (o.v0 + r) + o.p;
                        if (dl[r] != INT_MAX) ex.sdump[(int64_t)k * ex.n_max + i] = ex.scores[i];
                    }
                    if (lane == 0) ex.sdump_step[k] = w.steps;
                }
                t.sync();
                if (lane == 0) *ex.sdump_count = k + 1;
                t.sync();
            }
            for (;;) {
                int lk = INT_MIN, li = INT_MAX, ld = INT_MAX;
#pragma unroll
                for (int r = 0; r < R; ++r)
                    if (!((excl >> r) & 1u) && keys[r] > lk && dl[r] != INT_MAX) {
                        lk = keys[r];
                        li = 2 * (o.v0 + r) + o.p;
                        ld = dl[r];
                    }
                const int km = t.rmax(lk);
                if (km == INT_MIN) break;
                const int bi = t.rmin(lk == km ? li : INT_MAX);
                const int bd = t.rmin(li == bi ? ld : INT_MAX);
                const uint64_t f = w.fp ^ __ldg(env.zk + bi);
                const Probe pr = probe_full(env, f, w.gen, cap, t);
                if (!pr.visited) {
                    best_i = bi;
                    best_d = bd;
                    slot = pr.slot;
                    fnew = f;
                    break;
                }
                exclude<TL, R>(excl, bi, t);
            }
        }
        for (; best_i < 0;) {
            int d0, i0, d1, i1;
            tile_argmin(dl, excl, o, t, d0, i0);
            if (i0 < 0) break;
            uint32_t ex1 = excl;
            exclude<TL, R>(ex1, i0, t);
            tile_argmin(dl, ex1, o, t, d1, i1);
            const int hs = lane % S;
            const int mine = lane < S ? i0 : i1;
            bool hit = false, match = false;
            if (mine >= 0 && hs < cap) {
                const uint64_t f = w.fp ^ __ldg(env.zk + mine);
                const uint64_t e = env.T[(f + (uint64_t)hs) & env.tmask];
                match = e == ((f & ~kGenMask) | w.gen);
                hit = ((e & kGenMask) != w.gen) || match;
            }
            const unsigned bal = t.ballot(hit);
            const int cand[2] = {i0, i1};
            const int cdl[2] = {d0, d1};
            bool chosen = false;
#pragma unroll
            for (int g = 0; g < 2; ++g) {
                if (cand[g] < 0) break;
                const uint64_t fg = w.fp ^ __ldg(env.zk + cand[g]);
                const unsigned b = (bal >> (S * g)) & ((1u << S) - 1u);
                Probe pr;
                if (b) {
                    const int fl = __ffs(b) - 1;
                    pr.visited = t.shfl(match ? 1 : 0, S * g + fl) != 0;
                    pr.slot = (int64_t)((fg + (uint64_t)fl) & env.tmask);
                } else if (cap > S) {
                    pr = probe_full(env, fg, w.gen, cap, t);
                } else {
                    pr.visited = false;
                    pr.slot = -1;
                }
                if (!pr.visited) {
                    best_i = cand[g];
                    best_d = cdl[g];
                    slot = pr.slot;
                    fnew = fg;
                    chosen = true;
                    break;
                }
                exclude<TL, R>(excl, cand[g], t);
            }
            if (chosen) break;
        }

        w.steps += 1;
        int code;
        if (best_i < 0) {
            // Every neighbour is in HT: restart without a move.
            w.blocked += 1;
            restart_walker(env, w, base, SL, V, t);
            p_direct(V, n, o, P);
            code = LABS_TRACE_BLOCKED;
        } else {
            flip_rows_table(V, n, o, P, best_i, t);
            const bool stored = slot >= 0;
            if (lane == 0 && stored) env.T[slot] = (fnew & ~kGenMask) | w.gen;
            if (lane == (best_i >> 5)) w.word ^= 1u << (best_i & 31);
            t.sync();
            w.fp = fnew;
            w.isl += best_d;
            if (!stored) w.overflows += 1;
            note_best(env, w, t);
            if (w.isl < w.since) {
                w.since = w.isl;
                w.stag = 0;
            } else {
                w.stag += 1;
            }
            code = best_i;
            if (w.stag >= env.patience || !stored) {
                restart_walker(env, w, base, SL, V, t);
                p_direct(V, n, o, P);
                code |= LABS_TRACE_RESTART;
            }
        }
        if (trace_slot >= 0 && lane == 0) {
            const int64_t s = w.steps - 1 - trace_start;
            if (s >= 0 && s < p.status->trace_capacity) {
                p.status->trace_code[trace_slot * p.status->trace_capacity + s] = code;
                p.status->trace_isl[trace_slot * p.status->trace_capacity + s] = w.isl;
            }
        }
        if (ex.rec != nullptr && log_live) {
            // lowest ISL at the end of the chunk's steps before its first restart step
            if (w.steps == first_step + 1) log_first = code;
            if (code == LABS_TRACE_BLOCKED || (code & LABS_TRACE_RESTART)) log_live = false;
            else log_min = min(log_min, w.isl);
        }
    }
    if (ex.rec != nullptr && lane == 0) {
        ex.rec->first = log_first;
        ex.rec->min_isl = log_min;
    }
}

__device__ void load_walker(const WalkerState* st, Walker& w, int lane)
{
    w.word = lane < kBitWords ? st->cur[lane] : 0u;
    w.fp = st->fp;
    w.isl = st->isl;
    w.best_isl = st->best_isl;
    w.since = st->since_best;
    w.stag = st->stagnation;
    w.restart_idx = st->restart_idx;
    w.gen = st->gen;
    w.restarts = st->restarts;
    w.overflows = st->overflows;
    w.blocked = st->blocked;
    w.steps = st->steps_done;
    w.best_step = st->best_step;
    w.target_step = st->target_step;
}

__device__ void save_scalars(WalkerState* st, const Walker& w);

__device__ void save_walker(WalkerState* st, const Walker& w, int lane)
{
    if (lane < kBitWords) st->cur[lane] = w.word;
    if (lane == 0) save_scalars(st, w);
}

// Everything of the walker state but the bits (one thread).
__device__ void save_scalars(WalkerState* st, const Walker& w)
{
    {
        st->fp = w.fp;
        st->isl = w.isl;
        st->best_isl = w.best_isl;
        st->since_best = w.since;
        st->stagnation = w.stag;
        st->restart_idx = w.restart_idx;
        st->gen = w.gen;
        st->restarts = w.restarts;
        st->overflows = w.overflows;
        st->blocked = w.blocked;
        st->steps_done = w.steps;
        st->best_step = w.best_step;
        st->target_step = w.target_step;
    }
}

// dISL + 1.5 * 2^23 in fp32 has the bit pattern 0x4B400000 + dISL (|dISL| < 2^22 for L <=
// 511): the integer sits in the low bits without a conversion.
constexpr float kIntBias = 12582912.f;  // 1.5 * 2^23
constexpr int kKeyBias = 1 << 22;       // walk keys: dISL = (key >> 8) - kKeyBias

// ISL at or below which the target merit factor is met (-1: no target).
__device__ __forceinline__ int target_isl(const KParams& p, int L)
{
    if (p.target_num <= 0 || p.target_den <= 0) return -1;
    return (int)min((int64_t)INT_MAX, (int64_t)p.target_den * L * L / (2 * (int64_t)p.target_num));
}

// Lowest and highest 64-bit value of the warp's lanes (the best-first search's queue keys).
__device__ __forceinline__ uint64_t warp_min64(uint64_t v)
{
    const unsigned hi = __reduce_min_sync(kFull, (unsigned)(v >> 32));
    const unsigned lo = __reduce_min_sync(kFull, (unsigned)(v >> 32) == hi ? (unsigned)v : 0xFFFFFFFFu);
    return ((uint64_t)hi << 32) | lo;
}

__device__ __forceinline__ uint64_t warp_max64(uint64_t v)
{
    const unsigned hi = __reduce_max_sync(kFull, (unsigned)(v >> 32));
    const unsigned lo = __reduce_max_sync(kFull, (unsigned)(v >> 32) == hi ? (unsigned)v : 0u);
    return ((uint64_t)hi << 32) | lo;
}

// A new S that differs from S in at most this many free variables is reached by that
// many incremental flips (a neighbour of S, about half the steps, by one) rather than
// a rebuild from its bits; about four of five steps at L = 101..151, each flip costing about
// a sixth of a rebuild.
constexpr int kBestFirstMaxFlips = 5;

// ------------------------------------------------------------ PSL objective walk

// Order key of a flip under the PSL objective: PSL' << 43 | ISL' << 13 | i (PSL' < 2^21,
// ISL' < 2^30, i < 2^13 for every length served).
__device__ __forceinline__ uint64_t psl_key(int psl, int isl, int i)
{
    return ((uint64_t)psl << 43) | ((uint64_t)(uint32_t)isl << 13) | (uint64_t)i;
}
__device__ __forceinline__ int psl_key_i(uint64_t k) { return (int)(k & 0x1FFFu); }
__device__ __forceinline__ int psl_key_isl(uint64_t k) { return (int)((k >> 13) & 0x3FFFFFFFull); }
__device__ __forceinline__ int psl_key_psl(uint64_t k) { return (int)(k >> 43); }

// A pointer into shared memory that the compiler keeps in a register: without this the loops
// below computed theirs anew from the layout (a select of the class, the base of shared memory)
// in every iteration, 36 times a step at L = 513.
template <class T>
__device__ __forceinline__ const T* held_shared(const T* p)
{
    uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    asm volatile("" : "+r"(a));
    return static_cast<const T*>(__cvta_shared_to_generic(a));
}

// The same PSL values for the lane block R = 7 in one pass: s_{i-2m} and s_{i+2m} of the
// R outputs in two windows of R values that slide one class entry per lag (three shared
// loads per lag), and the mirror's term dropped by a compare and select per lag term.
template <class TL, int R>
__device__ __forceinline__ void psl_eval_select(const View& V, int n, const Outs<TL, R>& o, int (&pl)[R])
{
    const float* A = held_shared((o.p ? V.A1 : V.A0) + o.v0);
    const float2* G = held_shared(V.G);
    const int c = n - 1;
    float cs[R], mx[R], lo[R], hi[R];
    int q0[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = 2 * (o.v0 + r) + o.p;
        cs[r] = (i == c ? -2.f : -4.f) * A[r];
        q0[r] = c - i;
        mx[r] = 0.f;
    }
    // lo[e mod R] = A[-e] for e = m-R+1 .. m, hi[e mod R] = A[e] for e = m .. m+R-1
#pragma unroll
    for (int k = 1; k < R; ++k) lo[k] = A[R - k];
#pragma unroll
    for (int e = 0; e + 1 < R; ++e) hi[e] = A[e];
    for (int m0 = 0; m0 < n; m0 += R) {
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const int m = m0 + j;
            if (m >= n) break;
            lo[j] = A[-m];
            hi[(j + R - 1) % R] = A[m + R - 1];
            if (m == 0) continue;
            const float C = G[m].x;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float a = lo[(j - r + R) % R];
                const float b = m == q0[r] ? 0.f : hi[(j + r) % R];
                mx[r] = fmaxf(mx[r], fabsf(fmaf(cs[r], a + b, C)));
            }
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) pl[r] = (int)mx[r];
}

// PSL of every neighbour S_i for the lane's outputs i = 2(v0+r)+p: flipping s_i and its
// mirror s_{L-1-i} changes C_{2m} by -4 s_i (s_{i-2m} + s_{i+2m}) with the mirror's own
// term (i+2m = L-1-i, i.e. m = c-i) left out, or by -2 s_c (s_{c-2m} + s_{c+2m}) at the
// centre; the odd-lag C_k stay zero.  pl[r] = max_m |C_{2m} + dC_{2m}(i)| over
// m = 1..n-1 (Section 1's PSL).
// psl_ring takes the outputs C0 .. C0+RC-1 of the lane (block start w0 = v0 + C0).
// Output r takes lag m = t - 2r at iteration t, so that every output of the pass meets
// its mirror at the same iteration t* = c - p - 2 w0 (where m = c - i): there one
// multiplier z = 0 drops the mirror term of all of them, and a lag term costs three
// instructions (FMA, FMA, max of the absolute value).  s_{i-2m} = A_p[w0 + 3r - t],
// C_{2m} = E[t - 2r] and s_{i+2m} = A_p[w0 + t - r] come from three register rings of
// P = 3 RC - 2 entries indexed by t mod P (one new shared load each per iteration, the
// loop unrolled by P so that the ring indices are constants).  Lags outside 1..n-1 (the
// first 2 RC - 2 and the last iterations) are masked in the blocks that hold them.
// Exact in fp32: every value is an integer of magnitude below 2^10.
// Compiled by itself (not inlined): its registers are then the same whatever surrounds it.
// Inlined beside the tensor-core product its ring lost register banks (dispatch stalls 0.44 an
// issue from 0.32).  608 walkers x 128 steps of the long PSL walk, inlined / like this: L = 513
// 4.10 / 3.61 ms, 1025 7.17 / 6.22, 2047 20.8 / 16.3, 4095 60.7 / 55.2, 11263 437 / 410.
template <class TL, int R, int C0, int RC>
__device__ __noinline__ void psl_ring(const View& V, int n, const Outs<TL, R>& o, int (&pl)[R])
{
    constexpr int P = 3 * RC - 2;
    const int w0 = o.v0 + C0;
    const float* A = held_shared((o.p ? V.A1 : V.A0) + w0);
    const float2* G = held_shared(V.G);
    const int c = n - 1;
    const int tstar = c - o.p - 2 * w0;
    const int tend = n - 1 + 2 * (RC - 1);
    float cs[RC], mx[RC], ra[P], rc[P], rb[P];
#pragma unroll
    for (int r = 0; r < RC; ++r) {
        const int i = 2 * (w0 + r) + o.p;
        cs[r] = (i == c ? -2.f : -4.f) * A[r];
        mx[r] = 0.f;
    }
    // entries e = -P+1 .. -1 (read only by masked lags)
#pragma unroll
    for (int k = 1; k < P; ++k) {
        ra[k] = A[P - k];
        rc[k] = G[k - P].x;
        rb[k] = A[k - P];
    }
    for (int t0 = 0; t0 <= tend; t0 += P) {
        if (t0 >= 2 * RC - 1 && t0 + P - 1 <= c) {
#pragma unroll
            for (int j = 0; j < P; ++j) {
                const int t = t0 + j;
                ra[j] = A[-t];
                rc[j] = G[t].x;
                rb[j] = A[t];
                const float z = t == tstar ? 0.f : 1.f;
#pragma unroll
                for (int r = 0; r < RC; ++r) {
                    const float cp = fmaf(cs[r], fmaf(rb[(j - r + P) % P], z, ra[(j - 3 * r + 3 * P) % P]),
                                          rc[(j - 2 * r + 2 * P) % P]);
                    mx[r] = fmaxf(mx[r], fabsf(cp));
                }
            }
        } else {
#pragma unroll
            for (int j = 0; j < P; ++j) {
                const int t = t0 + j;
                if (t > tend) break;
                ra[j] = A[-t];
                rc[j] = G[t].x;
                rb[j] = A[t];
                const float z = t == tstar ? 0.f : 1.f;
#pragma unroll
                for (int r = 0; r < RC; ++r) {
                    const float cp = fmaf(cs[r], fmaf(rb[(j - r + P) % P], z, ra[(j - 3 * r + 3 * P) % P]),
                                          rc[(j - 2 * r + 2 * P) % P]);
                    const int m = t - 2 * r;
                    if (m >= 1 && m <= c) mx[r] = fmaxf(mx[r], fabsf(cp));
                }
            }
        }
    }
#pragma unroll
    for (int r = 0; r < RC; ++r) pl[C0 + r] = (int)mx[r];
}

// All R outputs of the lane: one ring pass up to R = 6; wider lane blocks, whose three
// rings of 3R - 2 entries would not fit the registers, take the compare-and-select form
// at R = 7 (2% faster there when a walk of two per warp had that lane block) and two ring
// passes of (R+1)/2 and R - (R+1)/2 outputs from R = 9 (each pass reloads its rings:
// about twice the shared loads of one pass, but three instructions per lag term instead
// of a compare and select per term; 21-40% faster for the long lane blocks 9 and 11).
template <class TL, int R>
__device__ __forceinline__ void psl_eval(const View& V, int n, const Outs<TL, R>& o, int (&pl)[R])
{
    if constexpr (R == 7) {
        psl_eval_select<TL, R>(V, n, o, pl);
    } else if constexpr (R >= 8) {
        constexpr int H = (R + 1) / 2;
        psl_ring<TL, R, 0, H>(V, n, o, pl);
        psl_ring<TL, R, H, R - H>(V, n, o, pl);
    } else {
        psl_ring<TL, R, 0, R>(V, n, o, pl);
    }
}

// Lowest 64-bit value of the lane group: the lowest high word, then the lowest low word
// among the lanes that hold it.
template <class LG>
__device__ __forceinline__ uint64_t group_min64(uint64_t v, const LG& t)
{
    const uint32_t hi = t.rminu((uint32_t)(v >> 32));
    const uint32_t lo = t.rminu((uint32_t)(v >> 32) == hi ? (uint32_t)v : 0xFFFFFFFFu);
    return ((uint64_t)hi << 32) | lo;
}

template <int TILE, int RMAX>
__global__ void __launch_bounds__(256, LABS_WALK_MIN_BLOCKS) walk_learned_kernel(KParams p, int chunk_index)
{
    extern __shared__ __align__(16) int smem[];
    const WarpSmem SL = warp_smem(p.n_max, TILE);
    const Tile<TILE> t(threadIdx.x & 31);
    const int slot_id = threadIdx.x / TILE;  // walker slot of this tile in the CTA
    int* base = smem + slot_id * SL.words;
    const View V = make_view(base, SL);
    const int64_t target = p.status->target_steps;
    for (;;) {
        uint32_t q = 0;
        if (t.lane == 0) q = atomicAdd(&p.queue[chunk_index], 1u);
        const int64_t wi = (int64_t)t.shfl(q, 0);
        if (wi >= p.W) break;
        WalkerState* st = p.states + wi;
        const int64_t steps_done = st->steps_done;
        const int64_t until = min(target, steps_done + (int64_t)p.chunk_steps);
        if (steps_done >= until) continue;
        const DevGroup G = p.groups[st->group];
        WalkEnv env;
        env.p = &p;
        env.tmask = (1ull << p.tabu_log2) - 1ull;
        env.T = p.tabu + ((uint64_t)wi << p.tabu_log2);
        env.zk = p.zkeys + G.zkey_off;
        env.st = st;
        env.L = G.L;
        env.n = G.n;
        env.patience = p.patience > 0 ? p.patience : 2 * G.n;
        env.g = (uint32_t)wi;
        Walker w;
        load_walker(st, w, t.lane);
        const int trace_slot = st->trace_slot;
        const int64_t trace_start = trace_slot >= 0 ? p.trace_start[trace_slot] : 0;
        const int isl = load_rows(base, SL, V, w.word, G.L, G.n, t);
        if (isl != w.isl) {
            if (t.lane == 0) raise_error(p.status, LABS_ESTATE, (int)wi);
            continue;
        }
        StepExtras ex;
        ex.scores = nullptr;
        ex.sdump = nullptr;
        ex.rec = nullptr;
        ex.tau = 0;
        ex.dump_cap = 0;
        ex.n_max = p.n_max;
        env.slot = nullptr;
        env.slot_valid = nullptr;
        env.rdump = nullptr;
        env.rdump_idx = nullptr;
        env.rdump_count = nullptr;
        env.dump_cap = 0;
        DevStatus* S = p.status;
        if (S->learned) {
            env.slot = S->l_slot + wi * kBitWords;
            env.slot_valid = S->l_slot_valid + wi;
            if (S->l_score_step[wi] == steps_done) {
                ex.scores = S->l_scores + wi * p.n_max;
                ex.tau = S->l_tau;
            }
            if (trace_slot >= 0 && S->d_scores != nullptr) {
                ex.sdump = S->d_scores + (int64_t)trace_slot * S->d_cap * p.n_max;
                ex.sdump_step = S->d_score_step + (int64_t)trace_slot * S->d_cap;
                ex.sdump_count = S->d_score_count + trace_slot;
                ex.dump_cap = S->d_cap;
                env.rdump = S->d_restart + (int64_t)trace_slot * S->d_cap * kBitWords;
                env.rdump_idx = S->d_restart_idx + (int64_t)trace_slot * S->d_cap;
                env.rdump_count = S->d_restart_count + trace_slot;
                env.dump_cap = S->d_cap;
            }
        }
        if (S->log != nullptr && p.chunk_steps > 0) {
            const int64_t since = steps_done - S->log_start;
            if (since >= 0 && since % p.chunk_steps == 0) {
                const int64_t idx = (since / p.chunk_steps) * p.W + wi;
                if (idx < S->log_capacity) ex.rec = S->log + idx;
            }
        }
        constexpr int R2 = RMAX > 2 ? RMAX - 2 : 1;
        const bool full = RMAX <= 2 || block_R(G.n, TILE) >= RMAX;
        if (full)
            walk_steps<Tile<TILE>, RMAX>(env, w, until, base, SL, V, trace_slot, trace_start, ex, t);
        else
            walk_steps<Tile<TILE>, R2>(env, w, until, base, SL, V, trace_slot, trace_start, ex, t);
        save_walker(st, w, t.lane);
        t.sync();
    }
}


}  // namespace
}  // namespace labsgpu
