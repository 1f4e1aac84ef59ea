// labs_rows.cu -- the neighbourhood of Algorithm 1 for a batch of skew-symmetric rows
// (labs_neighbor_delta, L <= LABS_MAX_L) and for a batch of states (labs_features), on the
// step of labs_step.cuh: two rows per warp up to n = 160 free variables, one above.
//
// A row is seen once, so everything is built from the row itself:
//   - a lane takes 16 consecutive bytes, i.e. eight entries of each parity class: as FP16
//     they go into the product's rows in one 16-byte store per class, their signs into one
//     byte of the class's bit vector (bit u set <=> A_p[u] = -1), and the bytes are checked
//     to be +-1;
//   - the Eq. 4 check on the bit vectors: class p of a skew-symmetric row is a palindrome
//     when c + p is even and an antipalindrome when it is odd (entries u and n_p-1-u are
//     positions c-j and c+j of the sequence), so its vector reversed over its n_p bits
//     equals itself, or itself with every bit inverted;
//   - C^(p)_m from popcounts of the class against itself shifted by m, over half of the
//     pairs: with a_{n_p-1-u} = s_p a_u the pairs (u, u+m) and (n_p-1-u-m, n_p-1-u) have the
//     same product, and the pair in the middle (n_p - m odd) has product s_p, so with t
//     mismatches among the first h = floor((n_p - m)/2) pairs
//       C^(p)_m = 2 h - 4 t + [n_p - m odd] s_p;
//   - E_m = C^(0)_m + C^(1)_m and Z_m (labs_step.cuh) as one FP16 pair from the two sums.
// Then the step's product and dISL of every output, which go through shared memory so that
// a row leaves in whole 64- or 128-byte lines.
//
// What bounds it: instruction issue (three quarters of the slots), with the shared-memory
// pipe (two thirds) and the logic unit close behind.  A pair of rows at L = 201 issues about
// 900 warp instructions; the kernels this replaces (bytes one by one through ballots, FP32 or
// converted tables, popcounts over all pairs, a P value per output, results stored as the
// lanes held them) 1277.  2^20 rows of L = 201: 524 us from 810; 2^18 rows: L = 255 148 us,
// L = 303 231, L = 511 352.
#include "labs_async.cuh"
#include "labs_launch.h"
#include "labs_step.cuh"

#include <algorithm>

namespace labsgpu {

namespace {

// Staging of input rows: each warp copies the bytes of its next rows (rows r0 .. r0+k-1,
// global bytes [r0 L, (r0+k) L)) into one of two shared-memory buffers with one bulk
// copy while it evaluates the current rows from the other buffer.  A bulk copy moves
// 16-byte aligned blocks, so the copy covers [floor16(r0 L), ceil16((r0+k) L)), cut at
// the last 16-byte boundary of the input (the few bytes past it, and every byte when the
// input is not 16-byte aligned, are read from global memory directly).
__host__ __device__ inline int stage_bytes(int L, int rows)
{
    return (rows * L + 32 + 15) & ~15;
}

struct StageRange {
    int64_t a0, a1;  // staged global bytes [a0, a1); a1 <= a0: none
};

__device__ __forceinline__ StageRange stage_range(int64_t r0, int rows, int L, int64_t total)
{
    const int64_t e = min((r0 + rows) * (int64_t)L, total);
    StageRange g;
    g.a0 = (r0 * L) & ~(int64_t)15;
    g.a1 = min((e + 15) & ~(int64_t)15, total & ~(int64_t)15);
    return g;
}

// Issued by one lane: the copy of rows r0 .. r0+rows-1 into the buffer at shared address
// dst, counted on barrier bar (an arrival without bytes when nothing is staged).
__device__ __forceinline__ void stage_rows(const int8_t* seqs, int64_t r0, int rows, int L, int64_t total,
                                           uint32_t dst, uint32_t bar)
{
    const StageRange g = stage_range(r0, rows, L, total);
    fence_async_shared();  // earlier reads of the buffer come before the copy's writes
    if (g.a1 > g.a0) {
        const uint32_t bytes = (uint32_t)(g.a1 - g.a0);
        mbar_arrive_expect_tx(bar, bytes);
        bulk_copy_g2s(dst, seqs + g.a0, bytes, bar);
    } else {
        mbar_arrive(bar);
    }
}

// Sign bits of the four bytes of t, in order: bits 28-31 of the product.
__device__ __forceinline__ uint32_t sign_bits(uint32_t t)
{
    return (t & 0x80808080u) * 0x00204081u;
}

// Two of the four bytes of t (sel: their places, between the bytes of 0x64646464) as FP16:
// 0x6480 + b is 1152 + b.
__device__ __forceinline__ uint32_t byte_halves(uint32_t flipped, uint32_t sel)
{
    return as_u32(__hsub2(as_half2(__byte_perm(flipped, 0x64646464u, sel)), as_half2(0x64806480u)));
}

// Bits of class entries below np in word k.
__device__ __forceinline__ uint32_t class_mask(int np, int k)
{
    const int w = np - 32 * k;
    return w >= 32 ? ~0u : (w <= 0 ? 0u : (1u << w) - 1u);
}

// Whether the class's bits reversed over its np bits differ from themselves with `invert`
// applied: nonzero where they do (np >= 32 (NW-1)).
template <int NW>
__device__ __forceinline__ uint32_t mirror_diff(const uint32_t (&x)[NW], int np, uint32_t invert)
{
    uint32_t rv[NW + 1], diff = 0;
#pragma unroll
    for (int k = 0; k < NW; ++k) rv[k] = __brev(x[NW - 1 - k]);
    rv[NW] = 0u;
    const int sh = 32 * NW - np;  // 0 .. 32
#pragma unroll
    for (int k = 0; k < NW; ++k)
        diff |= __funnelshift_rc(rv[k], rv[k + 1], sh) ^ x[k] ^ (invert & (k < NW - 1 ? ~0u : class_mask(np, k)));
    return diff;
}

// One lane of a row evaluation.  LG: Pair (two rows per warp) or Tile<32>; R = step_R(n, lanes
// per row) outputs per lane; NW = ceil(n/32) words per class.
template <class LG, int R, int NW>
struct RowLane {
    static constexpr int NL = LG::kSize, W = 32 / NL;
    using LAY = StepLayout<NL, R, false>;
    static constexpr int IT = (4 * NW + NL - 1) / NL;  // pieces of 16 positions per lane
    StepLane<LAY, LG, R> a;
    int lane, n, c;
    // this lane's constants: its lags m = lane (mod NL) all have the parity of the lane
    int h0, h1;      // half the pairs at lag `lane`
    uint32_t kc;     // FP16 bits of 1536 + C^(p) at lag `lane` before its mismatches, class 1 high
    uint32_t zs0, zs1;  // (E, Z) = C^(0) (1, z0) + C^(1) (1, z1)
    uint32_t gp, gm, zp, rowa, bita, sga, res;
    int v0;
    int rc;          // this lane's output that is the centre

    __device__ __forceinline__ RowLane(int wb0, int n_, const LG& t, const Outs<LG, R>& o)
        : a(wb0, n_, t, o), lane(t.lane), n(n_), c(n_ - 1), v0(o.v0)
    {
        constexpr StepSmem SL = LAY::SL;
        const int wb = a.wb, odd0 = (n - lane) & 1, odd1 = odd0 ^ 1, sgn0 = (c & 1) ? -1 : 1;
        h0 = (n - lane) >> 1;
        h1 = (n - 1 - lane) >> 1;
        kc = 0x66006600u + (uint32_t)(2 * h0 + odd0 * sgn0) + ((uint32_t)(2 * h1 - odd1 * sgn0) << 16);
        // Z takes 3 times the lag's own class p = (c - m) mod 2, with the sign (-1)^m
        const uint32_t zs = (lane & 1) ? 0x80000000u : 0u, own = ((c - lane) & 1) ? 0x3C000000u : 0x42000000u;
        zs0 = (own | 0x3C00u) ^ zs;
        zs1 = ((own ^ 0x7E000000u) | 0x3C00u) ^ zs;
        gp = sbyte(wb + SL.g + lane);
        gm = sbyte(wb + SL.g - lane);
        zp = sbyte(wb + SL.z) + 2 * lane;
        rowa = sbyte(wb + SL.h0) + 16 * lane;
        bita = sbyte(wb + SL.b) + lane;
        sga = sbyte(wb + SL.b + o.p * SL.bvec + (o.v0 >> 5));
        rc = o.p == (c & 1) ? (c >> 1) - o.v0 : -1;
        res = sbyte(wb + SL.r8) + 4 * (2 * o.v0 + o.p);
    }

    // Every row writes the same entries: the padding is cleared once.
    __device__ __forceinline__ void clear() const
    {
        constexpr StepSmem SL = LAY::SL;
        for (int i = lane; i < SL.words / 4; i += NL) sts_v4(sbyte(a.wb) + 16 * i, 0u, 0u, 0u, 0u);
    }

    // Class words, and the signs of the lane's outputs (bit r; above the class anything).
    __device__ __forceinline__ uint32_t classes(uint32_t (&x0)[NW], uint32_t (&x1)[NW]) const
    {
        constexpr StepSmem SL = LAY::SL;
#pragma unroll
        for (int k = 0; k < NW; ++k) {
            x0[k] = lds_u32(sbyte(a.wb + SL.b) + 4 * k);
            x1[k] = lds_u32(sbyte(a.wb + SL.b + SL.bvec) + 4 * k);
        }
        return __funnelshift_r(lds_u32(sga), lds_u32(sga + 4), v0 & 31);
    }

    // Table and Z: lags m = lane + NL j + 32 q.
    __device__ __forceinline__ void table(const uint32_t (&x0)[NW], const uint32_t (&x1)[NW]) const
    {
        constexpr StepSmem SL = LAY::SL;
        const uint32_t ez0 = half_bits(6 - c + (c & 1)) << 16;  // lag 0: E = 0, Z of the centre
#pragma unroll
        for (int j = 0; j < 32 / NL; ++j) {
            uint32_t s0[NW], s1[NW];
#pragma unroll
            for (int k = 0; k < NW; ++k) {
                s0[k] = __funnelshift_r(x0[k], k + 1 < NW ? x0[k + 1] : 0u, lane + NL * j);
                s1[k] = __funnelshift_r(x1[k], k + 1 < NW ? x1[k + 1] : 0u, lane + NL * j);
            }
#pragma unroll
            for (int q = 0; q < NW; ++q) {
                const int m0 = 32 * q + NL * j;  // m = m0 + lane
                int t0 = 0, t1 = 0;
#pragma unroll
                for (int k = 0; 2 * k < NW - q; ++k) {
                    // pairs 32 k .. of the first h: n > 32 (NW - 1) and m < 32 (q + 1)
                    uint32_t d0 = x0[k] ^ s0[k + q], d1 = x1[k] ^ s1[k + q];
                    if (32 * (k + 1) > 16 * (NW - q - 2)) {
                        const int b0 = h0 - m0 / 2 - 32 * k, b1 = h1 - m0 / 2 - 32 * k;
                        d0 &= __funnelshift_lc(~0u, 0u, k ? max(b0, 0) : b0);
                        d1 &= __funnelshift_lc(~0u, 0u, k ? max(b1, 0) : b1);
                    }
                    t0 += __popc(d0);
                    t1 += __popc(d1);
                }
                const uint32_t cc = kc - (uint32_t)m0 * 0x00010001u - 4u * ((uint32_t)t0 + ((uint32_t)t1 << 16));
                const __half2 ch = __hsub2(as_half2(cc), as_half2(0x66006600u));
                uint32_t ez =
                    as_u32(__hfma2(__high2half2(ch), as_half2(zs1), __hmul2(__low2half2(ch), as_half2(zs0))));
                if (m0 == 0) ez = lane == 0 ? ez0 : ez;
                if (q < NW - 1) {  // n > 32 (NW - 1): the lag exists
                    sts_u16(gp + 4 * m0, ez);
                    sts_u16(gp + 4 * m0 - 2, ez);
                    sts_u16(zp + 2 * m0, ez >> 16);
                    if (m0 + NL - 1 < SL.gneg) {
                        sts_u16(gm - 4 * m0, ez);
                        sts_u16(gm - 4 * m0 - 2, ez);
                    } else if (m0 <= SL.gneg) {
                        sts_u16_if(m0 + lane <= SL.gneg, gm - 4 * m0, ez);
                        sts_u16_if(m0 + lane < SL.gneg, gm - 4 * m0 - 2, ez);
                    }
                } else {
                    const bool in = lane < n - m0;
                    sts_u16_if(in, gp + 4 * m0, ez);
                    sts_u16_if(in, gp + 4 * m0 - 2, ez);
                    sts_u16_if(in, zp + 2 * m0, ez >> 16);
                    if (m0 <= SL.gneg) {
                        sts_u16_if(in && m0 + lane <= SL.gneg, gm - 4 * m0, ez);
                        sts_u16_if(in && m0 + lane < SL.gneg, gm - 4 * m0 - 2, ez);
                    }
                }
            }
        }
    }

    // The product and the outputs' dISL, int32 i of the row at result(i):
    //   dISL = -8 s_i (X_i + 4 sg s_{3i-L+1}) + 8 Z_m + 16 (N_p - 2), the centre -4 s_c;
    // the FP32 value dISL + 1.5 2^23 holds the integer in its low bits.
    __device__ __forceinline__ void values(uint32_t sgn, int wl) const
    {
        __syncwarp();
        step_toeplitz(a.prod, wl);  // ends with a warp barrier
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float x = lds_f32(a.xr + 4 * r), z = lds_f16(a.zr - 4 * r), s3 = lds_f16(a.sr + 6 * r);
            const float y = __uint_as_float(__float_as_uint(fmaf(a.sig4, s3, x)) ^ ((sgn << (31 - r)) & 0x80000000u));
            const float v = fmaf(r == rc ? -4.f : -8.f, y, fmaf(8.f, z, a.bias));
            sts_u32(res + 8 * r, __float_as_uint(v) - __float_as_uint(kIntBias));
        }
        __syncwarp();
    }

    __device__ __forceinline__ uint32_t result(int i) const { return sbyte(a.wb + LAY::SL.r8) + 4 * i; }
};

template <class LG, int R>
constexpr int row_ctas()
{
    return LG::kSize == 16 && R > 7 ? 2 : 3;  // of eight warps per SM
}

// STAGED: rows come through the staging buffers after the rows' shared memory.
template <class LG, int R, int NW, bool STAGED>
__global__ void __launch_bounds__(256, row_ctas<LG, R>())
    rows_kernel(const int8_t* __restrict__ seqs, int64_t batch, int L, int32_t* __restrict__ out, DevStatus* status)
{
    using RL = RowLane<LG, R, NW>;
    constexpr int NL = RL::NL, W = RL::W, IT = RL::IT;
    constexpr StepSmem SL = RL::LAY::SL;
    extern __shared__ __align__(16) int smem[];
    const int n = (L + 1) / 2, c = n - 1;
    const LG t(threadIdx.x & 31);
    const int lane = t.lane, wl = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const Outs<LG, R> o(t);
    const RL rl(warp * W * SL.words, n, t, o);
    rl.clear();

    const int SB = stage_bytes(L, W);
    const int8_t* stg = reinterpret_cast<const int8_t*>(smem + (blockDim.x >> 5) * W * SL.words) + warp * (2 * SB + 16);
    const uint32_t sdst = smem_addr(stg), bar = sdst + 2 * SB;  // two buffers, then two barriers
    const int64_t total = batch * (int64_t)L;
    const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    const int64_t first = W * ((int64_t)blockIdx.x * (blockDim.x >> 5) + warp);
    if (STAGED) {
        if (wl == 0) {
            mbar_init(bar, 1);
            mbar_init(bar + 8, 1);
            mbar_init_fence();
        }
        __syncwarp();
        if (wl == 0 && first < batch) stage_rows(seqs, first, W, L, total, sdst, bar);
    }
    __syncwarp();

    int it = 0;
    for (int64_t r0 = first; r0 < batch; r0 += W * nwarps, ++it) {
        const int b = it & 1;
        StageRange g{0, 0};
        if (STAGED) {
            const int64_t next = r0 + W * nwarps;
            const bool more = next < batch;
            if (wl == 0 && more) stage_rows(seqs, next, W, L, total, sdst + (b ^ 1) * SB, bar + 8 * (b ^ 1));
            if (!__all_sync(kFull, mbar_wait(bar + 8 * b, (it >> 1) & 1))) {
                if (wl == 0 && status) raise_error(status, LABS_ECUDA, (int)r0);
                if (more) mbar_wait(bar + 8 * (b ^ 1), ((it + 1) >> 1) & 1);  // the copy in flight
                return;
            }
            g = stage_range(r0, W, L, total);
        }
        const int64_t row = r0 + group_of(t);
        const bool has = row < batch;
        const int64_t rs = row * (int64_t)L, lim = g.a1 - rs;
        const int8_t* src = seqs + rs;
        const uint32_t srow = sdst + b * SB + (uint32_t)(rs - g.a0);
        // rows held whole by the staging buffer (all but the input's last few bytes) are
        // read from there in words; the choice is the same for the whole warp
        const bool whole = STAGED && __all_sync(kFull, has && lim >= L);
        uint32_t bad = 0;
#pragma unroll
        for (int q = 0; q < IT; ++q) {
            const int piece = lane + NL * q;
            if (IT * NL == 4 * NW || piece < 4 * NW) {
                uint32_t w[4];
                const int left = L - 16 * piece;  // bytes of the row from here on
                if (whole) {
                    // a piece past the row reads its first bytes, which the mask takes away
                    const uint32_t at = srow + (left > 0 ? 16 * piece : 0), w4 = at & ~3u;
                    uint32_t v[5];
#pragma unroll
                    for (int k = 0; k < 5; ++k) v[k] = lds_u32(w4 + 4 * k);
#pragma unroll
                    for (int k = 0; k < 4; ++k) w[k] = __funnelshift_r(v[k], v[k + 1], 8 * (at & 3u));
                } else {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        w[k] = 0u;
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const int j = 16 * piece + 4 * k + e;
                            if (has && j < L) {
                                const int8_t s = STAGED && j < lim ? stg[b * SB + (rs - g.a0) + j] : src[j];
                                w[k] |= (uint32_t)(uint8_t)s << (8 * e);
                            }
                        }
                    }
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    // bytes of the row in this word; every one of them is 1 or 255
                    const uint32_t m = __funnelshift_lc(~0u, 0u, max(8 * (left - 4 * k), 0));
                    w[k] &= m;
                    const uint32_t neg = (w[k] >> 7) & 0x01010101u;
                    bad |= w[k] ^ ((m & 0x01010101u) | ((neg << 8) - neg));
                }
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    const uint32_t lo = __byte_perm(w[0], w[1], p ? 0x7531 : 0x6420);
                    const uint32_t hi = __byte_perm(w[2], w[3], p ? 0x7531 : 0x6420);
                    const uint32_t fl = lo ^ 0x80808080u, fh = hi ^ 0x80808080u;
                    sts_v4(rl.rowa + 4 * p * SL.hc + 16 * NL * q, byte_halves(fl, 0x4140), byte_halves(fl, 0x4342),
                           byte_halves(fh, 0x4140), byte_halves(fh, 0x4342));
                    sts_u8(rl.bita + 4 * p * SL.bvec + NL * q, (sign_bits(lo) >> 28) | ((sign_bits(hi) >> 24) & 0xF0u));
                }
            }
        }
        __syncwarp();
        uint32_t x0[NW], x1[NW];
        const uint32_t sgn = rl.classes(x0, x1);
        const uint32_t f0 = (c & 1) ? ~0u : 0u;  // antipalindromic class: all bits inverted
        bad |= mirror_diff<NW>(x0, n, f0) | mirror_diff<NW>(x1, n - 1, ~f0);
        // the ballot is a full-warp collective: both halves take it, with or without a row (no
        // row: no bytes, not valid)
        const bool valid = t.ballot(bad != 0u) == 0u;
        rl.table(x0, x1);
        rl.values(sgn, wl);
        int32_t* dst = out + row * (int64_t)n;
        const uint32_t res = rl.result(lane);
        if (__all_sync(kFull, has && valid)) {
#pragma unroll
            for (int k = 0; k < R; ++k)
                if (NL * (k + 1) <= 32 * (NW - 1) + 1 || lane < n - NL * k)
                    dst[lane + NL * k] = (int)lds_u32(res + 4 * NL * k);
        } else if (has) {
            if (!valid && lane == 0 && status) atomicAdd(&status->invalid_rows, 1);
            for (int i = lane; i < n; i += NL) dst[i] = valid ? (int)lds_u32(rl.result(i)) : INT_MIN;
        }
        // the warp barriers before the next rows' product order its overwrites of X and the
        // staged results; the rows, Z and this staging buffer were last read before the one above
    }
}

// Network inputs of states given by their free-variable bits (8 words each, `stride` words
// apart): x[b][0][i] = s_i, x[b][1][i] = C_{2(i+1)}/sqrt(L) (0 for i = n-1), x[b][2][i] =
// dISL_i/(8L).  As the rows, with the pieces of 16 positions from the bits: those above the
// centre are the mirror's, reversed, with the sign (-1)^(j-c).  Scoring 8192 states of n =
// 128 takes 172 us with this kernel and took 209 with one warp per state on the FP32 product
// (40 us of it); a training step of 4096 records is 21 us shorter.
template <class LG, int R, int NW>
__global__ void __launch_bounds__(256, row_ctas<LG, R>())
    features_kernel(const uint32_t* __restrict__ bits, int64_t stride, int64_t count, int L, float* __restrict__ x)
{
    using RL = RowLane<LG, R, NW>;
    constexpr int NL = RL::NL, W = RL::W, IT = RL::IT;
    constexpr StepSmem SL = RL::LAY::SL;
    const int n = (L + 1) / 2, c = n - 1;
    const LG t(threadIdx.x & 31);
    const int lane = t.lane, wl = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const Outs<LG, R> o(t);
    const RL rl(warp * W * SL.words, n, t, o);
    rl.clear();
    const float sq = sqrtf((float)L), inv8L = (float)(8 * L);
    const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    __syncwarp();
    for (int64_t b0 = W * ((int64_t)blockIdx.x * (blockDim.x >> 5) + warp); b0 < count; b0 += W * nwarps) {
        const int64_t b = b0 + group_of(t);
        const bool has = b < count;
        const uint32_t* src = bits + (has ? b : b0) * stride;  // no state: the first one's again
        // bits v .. v+31 of the state, for v >= -31 (zero below 0 and from 32 kBitWords on)
        const auto window = [&](int v) {
            const int k = v >> 5;
            const uint32_t lo = k >= 0 && k < kBitWords ? __ldg(src + k) : 0u;
            const uint32_t hi = k + 1 >= 0 && k + 1 < kBitWords ? __ldg(src + k + 1) : 0u;
            return __funnelshift_r(lo, hi, v & 31);
        };
#pragma unroll
        for (int q = 0; q < IT; ++q) {
            const int piece = lane + NL * q, j0 = 16 * piece;
            if (IT * NL == 4 * NW || piece < 4 * NW) {
                // bit e: s_{j0+e} = -1.  Up to the centre the state's bits, above it bit 2c - j
                uint32_t w = window(j0);
                if (j0 + 15 > c) {
                    const uint32_t alt = ((j0 - c) & 1) ? 0x5555u : 0xAAAAu;  // j - c odd
                    const uint32_t up = (__brev(window(2 * c - j0 - 15)) >> 16) ^ alt;
                    const uint32_t own = __funnelshift_lc(~0u, 0u, max(c + 1 - j0, 0));
                    w = (w & own) | (up & ~own);
                }
                const int left = L - j0;  // positions of the row from here on
                w &= __funnelshift_lc(~0u, 0u, min(max(left, 0), 16));
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    uint32_t y = (w >> p) & 0x5555u;
                    y = (y | y >> 1) & 0x3333u;
                    y = (y | y >> 2) & 0x0F0Fu;
                    y = (y | y >> 4) & 0x00FFu;
                    const int live = (left + 1 - p) >> 1;  // entries of the class from here on
                    uint32_t hp[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const uint32_t two = y >> 2 * k;
                        const uint32_t v = (two << 15 & 0x8000u) | (two << 30 & 0x80000000u) | 0x3C003C00u;
                        hp[k] = v & (2 * k + 1 < live ? ~0u : 2 * k < live ? 0xFFFFu : 0u);
                    }
                    sts_v4(rl.rowa + 4 * p * SL.hc + 16 * NL * q, hp[0], hp[1], hp[2], hp[3]);
                    sts_u8(rl.bita + 4 * p * SL.bvec + NL * q, y);
                }
            }
        }
        __syncwarp();
        uint32_t x0[NW], x1[NW];
        const uint32_t sgn = rl.classes(x0, x1);
        rl.table(x0, x1);
        rl.values(sgn, wl);
        if (has) {
            float* xb = x + b * 3 * n;
            for (int i = lane; i < n; i += NL) {
                xb[i] = (__ldg(src + (i >> 5)) >> (i & 31)) & 1u ? -1.f : 1.f;
                xb[n + i] = i < n - 1 ? lds_f16(sbyte(rl.a.wb + SL.g) + 4 * (i + 1)) / sq : 0.f;
                xb[2 * n + i] = (float)(int)lds_u32(rl.result(i)) / inv8L;
            }
        }
        __syncwarp();  // the next state's table comes after this one's reads
    }
}

using RowsFn = void (*)(const int8_t*, int64_t, int, int32_t*, DevStatus*);
using FeaturesFn = void (*)(const uint32_t*, int64_t, int64_t, int, float*);

// A kernel and the shared memory of one of its warps' rows.  (The layout is a loop over all
// lengths: worked out in every call instead of by the compiler it took 1.5 us of a 4 us call.)
template <class Fn>
struct RowKernel {
    Fn fn = nullptr;
    size_t warp_bytes = 0;
};
template <class LG, int R>
constexpr size_t row_warp_bytes()
{
    constexpr StepSmem SL = step_smem(LG::kSize, R);
    return (size_t)(32 / LG::kSize) * SL.words * sizeof(int);
}

// (lane block, words per class) of every length: step_R(n, lanes per row), ceil(n/32)
#define LABS_ROW_CASES(CASE)                                                                                       \
    CASE(Pair, 1, 1) CASE(Pair, 2, 1) CASE(Pair, 3, 2) CASE(Pair, 5, 2) CASE(Pair, 5, 3) CASE(Pair, 6, 3)          \
    CASE(Pair, 7, 4) CASE(Pair, 9, 4) CASE(Pair, 10, 5) CASE(Tile<32>, 7, 6) CASE(Tile<32>, 7, 7)                  \
    CASE(Tile<32>, 9, 8)

template <bool STAGED>
RowKernel<RowsFn> rows_fn(int key)
{
    switch (key) {
#define LABS_ROW_CASE(LG, R, NW) \
    case 16 * R + NW: return {rows_kernel<LG, R, NW, STAGED>, row_warp_bytes<LG, R>()};
        LABS_ROW_CASES(LABS_ROW_CASE)
#undef LABS_ROW_CASE
        default: return {};
    }
}

RowKernel<FeaturesFn> features_fn(int key)
{
    switch (key) {
#define LABS_ROW_CASE(LG, R, NW) \
    case 16 * R + NW: return {features_kernel<LG, R, NW>, row_warp_bytes<LG, R>()};
        LABS_ROW_CASES(LABS_ROW_CASE)
#undef LABS_ROW_CASE
        default: return {};
    }
}

// Warps of a CTA for `units` warps of work: eight; a batch that leaves SMs without a CTA is
// spread over more, smaller ones (64 rows of L = 255, back to back: 6.1 us a call on the
// device, 8.2 as four CTAs).
int row_warps(int64_t units, int sms)
{
    int warps = 8;
    while (warps > 1 && units <= (int64_t)(warps / 2) * sms) warps /= 2;
    return warps;
}

}  // namespace

int launch_delta(const int8_t* seqs, int64_t batch, int32_t L, int32_t* out, DevStatus* status, void* stream)
{
    if (batch == 0) return LABS_OK;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int n = (L + 1) / 2, tile = n <= 160 ? 16 : 32, rows = 32 / tile, R = step_R(n, tile);
    const int64_t units = (batch + rows - 1) / rows;
    const int warps = row_warps(units, sms);
    const int key = 16 * R + (n + 31) / 32;
    const RowKernel<RowsFn> plain = rows_fn<false>(key);
    if (plain.fn == nullptr) return LABS_EINVAL;
    const size_t warp_bytes = plain.warp_bytes;
    const size_t stage = 2 * (size_t)stage_bytes(L, rows) + 16;
    // staged rows need a 16-byte aligned input, and are used where they keep as many CTAs
    // of eight warps on an SM as the rows alone (three, two with lane blocks 9 and 10)
    const size_t sm_bytes = 226 * 1024 / 8;
    const size_t cap = tile == 32 || R <= 7 ? 3 : 2;  // the kernels' launch bounds
    const bool staged = ((uintptr_t)seqs & 15) == 0 &&
                        std::min(cap, sm_bytes / (warp_bytes + stage)) >= std::min(cap, sm_bytes / warp_bytes);
    const RowsFn fn = staged ? rows_fn<true>(key).fn : plain.fn;
    const size_t smem = warps * (warp_bytes + (staged ? stage : 0));
    if (smem > 48 * 1024 && allow_shared((const void*)fn, 0) != cudaSuccess) return LABS_ECUDA;
    // more CTAs than fit at once (up to 8 per SM): measured faster than one resident wave
    const int64_t need = (units + warps - 1) / warps, most = (int64_t)sms * 8;
    fn<<<(int)std::min(need, most), warps * kWarp, smem, (cudaStream_t)stream>>>(seqs, batch, L, out, status);
    return cudaGetLastError() == cudaSuccess ? LABS_OK : LABS_ECUDA;
}

int launch_features(const uint32_t* bits, int64_t stride, int64_t count, int32_t L, float* x, void* stream)
{
    if (count == 0) return LABS_OK;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int n = (L + 1) / 2, tile = n <= 160 ? 16 : 32, rows = 32 / tile, R = step_R(n, tile);
    const auto [fn, warp_bytes] = features_fn(16 * R + (n + 31) / 32);
    if (fn == nullptr) return LABS_EINVAL;
    const int64_t units = (count + rows - 1) / rows;
    const int warps = row_warps(units, sms);
    const size_t smem = warps * warp_bytes;
    if (smem > 48 * 1024 && allow_shared((const void*)fn, 0) != cudaSuccess) return LABS_ECUDA;
    const int64_t need = (units + warps - 1) / warps, most = (int64_t)sms * 8;
    fn<<<(int)std::min(need, most), warps * kWarp, smem, (cudaStream_t)stream>>>(bits, stride, count, L, x);
    return cudaGetLastError() == cudaSuccess ? LABS_OK : LABS_ECUDA;
}

}  // namespace labsgpu
