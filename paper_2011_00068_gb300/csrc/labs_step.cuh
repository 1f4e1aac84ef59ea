// labs_step.cuh -- the walk's step (Algorithm 1, self-avoiding form) for lengths up to
// LABS_MAX_L under the ISL or the PSL objective: four, two or one walkers per warp (LG =
// Quad, Pair or Tile<32>), the Toeplitz product on the tensor cores in all three.  The step
// rule is the one stated at labs_walk in labs.h.  Included by the labs_walk*.cu units (but
// 32l) and, for the layout, the product and the outputs, by labs_rows.cu.
//
// The neighbourhood in the form this step evaluates.  With p = i mod 2, v = i / 2, n_p
// entries in class p, c = n-1, m = c - i and sg = (-1)^m:
//   class p is a palindrome (sg = +1) or an antipalindrome (sg = -1), a_{n_p-1-u} = sg a_u
//   (Eq. 4), so the mirror is s_q = sg s_i, and P_i of labs_device.cuh is the class's
//   autocorrelation at lag m: C^(p)_m = 2 sg P_i + sg.  Putting both into the formula there
//   (C_{q-i} = C^(0)_m + C^(1)_m at the same lag m) leaves
//     dISL_i = -8 s_i (X_i + 4 sg s_{3i-L+1}) + 8 Z_m + 16 (N_p - 2)
//     Z_m    = sg (3 C^(p)_m + C^(1-p)_m)
//   and for the centre (m = 0) the same expression with -4 s_c in place of -8 s_i and
//   Z_0 = 6 - c + (c mod 2).
// So nothing but the table E, the sums Z and the rows is carried from step to step: a move
// changes C^(pb) of the flipped class at every lag by one vector of sums, which updates E
// and Z alike, and no per-output P exists.
//
// Exactness: E, Z and the rows are FP16 integers (|E| < 512, |Z| <= 4 * 256), the updates
// are FP16 FMAs on integers below 2048, the product and the assembly are FP32 on integers
// below 2^24: every result is the exact integer.
//
// What bounds it.  A step of two walkers in one warp issues about 540 warp instructions and
// moves about 170 wavefronts through the shared-memory pipe (L = 201), which is the busiest
// unit (three quarters of its peak); the HT probe's round trip to HBM is covered by 24
// warps per SM.  The step it replaces (FP32 rows and pair table, P per output, table
// operands converted on load, 128 registers and 16 warps per SM) issued 1017.  16384
// walkers x 10^4 steps at L = 201: 63.9 ms from 120.7; 16384 x 2000 at L = 501: 35.2 from
// 58.0; 52 lengths 201..303 x 512 walkers x 2000: 29.9 from 63.4.
#pragma once

#include "labs_device.cuh"

namespace labsgpu {
namespace {

// ------------------------------------------------------------------ shared memory
//
// Shared memory is addressed by 32-bit byte addresses (explicit ld/st.shared), with the
// layout a compile-time constant: a lane keeps a few base registers and every offset is an
// immediate of the access.  Word offsets below are relative to the CTA's dynamic shared
// memory; sbyte turns one into an address.
__device__ __forceinline__ uint32_t sbyte(int word)
{
    extern __shared__ __align__(16) int smem[];
    return (uint32_t)__cvta_generic_to_shared(smem) + 4u * (uint32_t)word;
}
__device__ __forceinline__ uint32_t lds_u32(uint32_t a)
{
    uint32_t v;
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ float lds_f32(uint32_t a)
{
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ float lds_f16(uint32_t a)  // an FP16 value as FP32
{
    float f;
    asm volatile("{\n\t.reg .b16 h;\n\tld.shared.b16 h, [%1];\n\tcvt.f32.f16 %0, h;\n\t}" : "=f"(f) : "r"(a) : "memory");
    return f;
}
__device__ __forceinline__ void sts_u32(uint32_t a, uint32_t v)
{
    asm volatile("st.shared.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void sts_f32(uint32_t a, float v)
{
    asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void sts_u16(uint32_t a, uint32_t v)
{
    asm volatile("st.shared.u16 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void sts_u8(uint32_t a, uint32_t v)
{
    asm volatile("st.shared.u8 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void sts_v2(uint32_t a, uint32_t x, uint32_t y)
{
    asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(a), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void sts_v4(uint32_t a, uint32_t x, uint32_t y, uint32_t z, uint32_t w)
{
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(x), "r"(y), "r"(z), "r"(w) : "memory");
}
// Predicated forms (no branch).
__device__ __forceinline__ void sts_u16_if(bool p, uint32_t a, uint32_t v)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %2, 0;\n\t@q st.shared.u16 [%0], %1;\n\t}" ::"r"(a),
                 "r"(v), "r"((uint32_t)p)
                 : "memory");
}
__device__ __forceinline__ void sts_f32_if(bool p, uint32_t a, float v)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %2, 0;\n\t@q st.shared.f32 [%0], %1;\n\t}" ::"r"(a), "f"(v),
                 "r"((uint32_t)p)
                 : "memory");
}
__device__ __forceinline__ void sts_v4_if(bool p, uint32_t a, uint32_t x, uint32_t y, uint32_t z, uint32_t w)
{
    asm volatile(
        "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %5, 0;\n\t@q st.shared.v4.b32 [%0], {%1, %2, %3, %4};\n\t}" ::"r"(a), "r"(x),
        "r"(y), "r"(z), "r"(w), "r"((uint32_t)p)
        : "memory");
}
__device__ __forceinline__ void stg_u64_if(bool p, uint64_t* a, uint64_t v)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %2, 0;\n\t@q st.global.b64 [%0], %1;\n\t}" ::"l"(a), "l"(v),
                 "r"((uint32_t)p)
                 : "memory");
}

__device__ __forceinline__ __half2 as_half2(uint32_t x)
{
    return *reinterpret_cast<__half2*>(&x);
}
__device__ __forceinline__ uint32_t as_u32(__half2 x)
{
    return *reinterpret_cast<uint32_t*>(&x);
}
__device__ __forceinline__ uint32_t half_bits(int v)
{
    return __half_as_ushort(__int2half_rn(v));
}
constexpr uint32_t kHalfInf = 0x7C00u;  // an FP16 infinity: no such output, or not a candidate

// Four 8x8 blocks of 16-bit entries; lane l gives the address (bytes) of row l % 8 of
// block l / 8 and receives entries 2 (l % 4), 2 (l % 4) + 1 of row l / 4 of every block.
__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t (&r)[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}

// The lane of the thread, read once (the compiler would otherwise read it again where it
// runs out of registers).
__device__ __forceinline__ int lane_id()
{
    int l;
    asm volatile("mov.u32 %0, %%laneid;" : "=r"(l));
    return l;
}

// Compile-time shape of a step with lane group LG and lane block R.  The product runs the
// row and output blocks of the largest n with this lane block: a shorter class is zero
// beyond its end.
template <class LG, int R>
struct StepShape {
    static constexpr int NL = LG::kSize;              // lanes per walker
    static constexpr int NMAX = step_n(NL, R);
    static constexpr int S = (NMAX + 15) / 16, T = ((NMAX + 1) / 2 + 15) / 16;
    static constexpr int W = 32 / NL;                 // walkers per warp
    static constexpr int M = step_groups(NL, R);      // column groups of 4 output blocks
    static constexpr int NB = step_lag_blocks(NL, R); // blocks of 8 lags per lane
    static constexpr int OUTS = (NL / 2) * R;         // outputs per class (existing or not)
    static constexpr int TB = (OUTS + 15) / 16 < 4 * M ? (OUTS + 15) / 16 : 4 * M;
};

// Layout of a kernel's walkers: that of its largest lane block.
template <int NL, int RMAX, bool PSL>
struct StepLayout {
    static constexpr StepSmem SL = step_smem(NL, RMAX, PSL);
    static constexpr bool kPsl = PSL;
};

// ------------------------------------------------------------------ rebuild from bits

// Rows, table and Z of the walker at word offset wb from its free-variable bits (word j in
// lane j of the tile); returns the ISL, and under the PSL objective max |C_{2m}|.  Every
// word of the walker's shared memory is rewritten.
template <class LAY, class TL>
__device__ int step_build(int wb, uint32_t word, int L, int n, const TL& t, int* psl)
{
    constexpr StepSmem SL = LAY::SL;
    constexpr int NL = TL::kSize;
    const int c = n - 1;
    const uint32_t base = sbyte(wb);
    for (int i = t.lane; i < SL.words / 4; i += NL) sts_v4(base + 16 * i, 0u, 0u, 0u, 0u);
    t.sync();
    // Z of outputs that do not exist (m < 0)
    for (int i = t.lane; i < SL.zneg / 2; i += NL) sts_u32(base + 4 * (SL.z - SL.zneg / 2 + i), kHalfInf | (kHalfInf << 16));
    // rows (both copies) and coefficients
    for (int j0 = 0; j0 < L; j0 += NL) {
        const int j = j0 + t.lane;
        int f = j <= c ? j : 2 * c - j;
        if (j >= L) f = 0;
        const uint32_t w = t.shfl(word, f >> 5);
        if (j < L) {
            const int x = ((w >> (f & 31)) & 1u) ? -1 : 1;
            const int s = (j > c && ((j - c) & 1)) ? -x : x;
            const uint32_t a = base + 4 * (SL.h0 + (j & 1) * SL.hc) + 2 * (j >> 1);
            sts_u16(a, s < 0 ? 0xBC00u : 0x3C00u);
            sts_u16(a + 4 * SL.ks - 2, s < 0 ? 0xBC00u : 0x3C00u);
            if (j <= c) sts_f32(base + 4 * (SL.r8 + (j & 1) * SL.xp + (j >> 1)), (float)((j == c ? -4 : -8) * s));
        }
    }
    t.sync();
    // bit vectors of the classes: word k of class p at b + p bvec + k
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        const int np = n - p;
        const uint32_t row = base + 4 * (SL.h0 + p * SL.hc);
        for (int k = 0; 32 * k < np; ++k) {
            uint32_t w = 0;
#pragma unroll
            for (int h = 0; h < 32 / NL; ++h) {
                const int u = 32 * k + NL * h + t.lane;
                const uint32_t b = t.ballot(u < np && lds_f16(row + 2 * min(u, np)) < 0.f);
                w |= NL == 32 ? b : (b << (NL * h));
            }
            if (t.lane == 0) sts_u32(base + 4 * (SL.b + p * SL.bvec + k), w);
        }
    }
    t.sync();
    // autocorrelations of both classes at every lag, four lags per lane and pass
    int part = 0, top = 0;
    const uint32_t x0 = base + 4 * SL.b, x1 = x0 + 4 * SL.bvec;
    constexpr int kG = 4;
    for (int mb = 1 + t.lane; mb < n; mb += kG * NL) {
        int c0[kG], c1[kG];
#pragma unroll
        for (int g = 0; g < kG; ++g) c0[g] = c1[g] = 0;
        for (int k = 0; 32 * k < n - mb; ++k) {
#pragma unroll
            for (int g = 0; g < kG; ++g) {
                const int m = mb + g * NL, v0 = n - m - 32 * k, v1 = v0 - 1;
                if (v0 > 0) {
                    const int q = 4 * (k + (m >> 5)), r = m & 31;
                    const uint32_t m0 = v0 >= 32 ? ~0u : (1u << v0) - 1u;
                    const uint32_t m1 = v1 >= 32 ? ~0u : (v1 > 0 ? (1u << v1) - 1u : 0u);
                    c0[g] += __popc((lds_u32(x0 + 4 * k) ^ __funnelshift_r(lds_u32(x0 + q), lds_u32(x0 + q + 4), r)) & m0);
                    c1[g] += __popc((lds_u32(x1 + 4 * k) ^ __funnelshift_r(lds_u32(x1 + q), lds_u32(x1 + q + 4), r)) & m1);
                }
            }
        }
#pragma unroll
        for (int g = 0; g < kG; ++g) {
            const int m = mb + g * NL;
            if (m < n) {
                const int a0 = (n - m) - 2 * c0[g], a1 = m < c ? (c - m) - 2 * c1[g] : 0;
                const int d = a0 + a1;
                part += d * d;
                if (LAY::kPsl) top = max(top, abs(d));
                const uint32_t e = half_bits(d), gb = base + 4 * SL.g;
                sts_u16(gb + 4 * m, e);
                sts_u16(gb + 4 * m - 2, e);
                if (m <= SL.gneg) sts_u16(gb - 4 * m, e);
                if (m < SL.gneg) sts_u16(gb - 4 * m - 2, e);
                // Z_m = sg (3 C^(p) + C^(1-p)), p = (c - m) mod 2
                const int z = ((c - m) & 1) ? 3 * a1 + a0 : 3 * a0 + a1;
                sts_u16(base + 4 * SL.z + 2 * m, half_bits((m & 1) ? -z : z));
            }
        }
    }
    if (t.lane == 0) sts_u16(base + 4 * SL.z, half_bits(6 - c + (c & 1)));
    t.sync();
    if (LAY::kPsl) *psl = t.rmax(top);
    return t.radd(part);
}

// ------------------------------------------------------------------ Toeplitz product

__device__ __forceinline__ void mma_16816_zero(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                               uint32_t b0, uint32_t b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%10, %10, %10, %10};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
}

// Addresses of a lane in the product (bytes).
template <class LAY, class LG, int R>
struct StepProduct {
    using SH = StepShape<LG, R>;
    uint32_t gy;  // first operand word of the table
    uint32_t ha;  // its ldmatrix row, first diagonal
    uint32_t xw;  // its first result
    __device__ StepProduct(int wb0, int l)
    {
        constexpr StepSmem SL = LAY::SL;
        const int g = l >> 2, tq = l & 3;
        gy = sbyte(wb0 + SL.g + 2 * tq - g - 16 * (SH::T - 1));
        // operand rows: class row/4, block order 0, 2, 1, 3 (so that a store of the results
        // takes neighbouring blocks); K half kh; first or second operand ob
        const int row = l & 7, kh = (l >> 3) & 1, ob = l >> 4;
        const int blk = ((row >> 1) & 1) | ((row & 1) << 1);
        int hb = wb0 + SL.h0 + (row >> 2) * SL.hc + 8 * (blk - (SH::T - 1)) + 4 * kh;
        if (SH::W * SH::M == 1) hb += 8 * ob;   // the next diagonal
        else if (SH::M == 2) hb += 32 * ob;     // the next column group
        else hb += SL.words * ob;               // the next walker
        ha = sbyte(hb);
        xw = sbyte(wb0 + SL.x + (tq >> 1) * SL.xp + 16 * (tq & 1) + g);
    }
};

// X_v for all outputs of the warp's W walkers into their scratch: the block-diagonal sum
// of toeplitz_tc1 (labs_device.cuh), with the table kept as FP16 pairs G[y] = (E[y],
// E[y+1]) (one 4-byte load per operand register, no conversion) and the row blocks of
// two (walker, column group) operands loaded by one ldmatrix per diagonal.
template <class LAY, class LG, int R>
__device__ __forceinline__ void step_toeplitz(const StepProduct<LAY, LG, R>& a, int l)
{
    using SH = StepShape<LG, R>;
    constexpr StepSmem SL = LAY::SL;
    constexpr int W = SH::W, M = SH::M, OPS = W * M, S = SH::S, T = SH::T, nd = S + T - 1;
    constexpr int WB = 4 * SL.words;  // bytes per walker
    float d[OPS == 1 ? 2 : OPS][4];
    uint32_t am[W];
#pragma unroll
    for (int w = 0; w < W; ++w) am[w] = lds_u32(a.gy - 32u + w * WB);
    if constexpr (OPS == 1) {
        // one operand: the even and the odd diagonals are the two chains
#pragma unroll
        for (int k = 0; k < 4; ++k) d[1][k] = 0.f;
#pragma unroll
        for (int k = 0; k < nd; k += 2) {
            uint32_t b[4];
            ldmatrix_x4(a.ha + 32 * k, b);
            const uint32_t a0 = lds_u32(a.gy + 64 * k), a2 = lds_u32(a.gy + 64 * k + 32);
            if (k == 0)
                mma_16816_zero(d[0], a0, am[0], a2, a0, b[0], b[1]);
            else
                mma_16816(d[0], a0, am[0], a2, a0, b[0], b[1]);
            am[0] = a2;
            if (k + 1 < nd) {
                const uint32_t a4 = lds_u32(a.gy + 64 * k + 64), a6 = lds_u32(a.gy + 64 * k + 96);
                mma_16816(d[1], a4, a2, a6, a4, b[2], b[3]);
                am[0] = a6;
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) d[0][k] += d[1][k];
    } else {
#pragma unroll
        for (int k = 0; k < nd; ++k) {
            uint32_t b[OPS / 2][4];
#pragma unroll
            for (int q = 0; q < OPS / 2; ++q) ldmatrix_x4(a.ha + 32 * k + (M == 2 ? q * WB : 2 * q * WB), b[q]);
#pragma unroll
            for (int w = 0; w < W; ++w) {
                const uint32_t a0 = lds_u32(a.gy + 64 * k + w * WB), a2 = lds_u32(a.gy + 64 * k + w * WB + 32);
#pragma unroll
                for (int m = 0; m < M; ++m) {
                    // group m of block diagonal d = k - (T-1): its row blocks t + d, t = 4m ..
                    // 4m+3, are all zero unless some lie in 0 .. S-1
                    const int o = w * M + m, first = T - 1 - (4 * m + 3) > 0 ? T - 1 - (4 * m + 3) : 0;
                    const uint32_t b0 = b[o >> 1][2 * (o & 1)], b1 = b[o >> 1][2 * (o & 1) + 1];
                    if (k == first)
                        mma_16816_zero(d[o], a0, am[w], a2, a0, b0, b1);
                    else if (k > first && 4 * m + k - (T - 1) < S)
                        mma_16816(d[o], a0, am[w], a2, a0, b0, b1);
                }
                am[w] = a2;
            }
        }
    }
    // this lane's accumulator columns: class tq/2, blocks tq mod 2 and 2 further
#pragma unroll
    for (int o = 0; o < OPS; ++o) {
        const int w = o / M, m = o % M;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const uint32_t xw = a.xw + w * WB + 256 * m + 128 * k;
            if (4 * m + 2 * k + 1 < SH::TB || (4 * m + 2 * k < SH::TB && !(l & 1))) {
                sts_f32(xw, d[o][k]);
                sts_f32(xw + 32, d[o][2 + k]);
            }
        }
    }
    __syncwarp();
}

// ------------------------------------------------------------------ walker state

// What a step reads of its walker; everything else stays in WalkerState and is touched
// only when it changes (a new best, a restart, an overflow).
struct StepWalker {
    uint32_t word;  // group lane j < 8: bits word j
    uint64_t fp;
    int isl, best, since, stag;
    uint32_t gen;
    int tisl;       // the target's ISL while it has not been met, else -1
    int psl, best_psl, since_psl;  // PSL objective: the PSL halves of the (PSL, ISL) pairs
};

template <bool PSL>
struct StepKey {
    using type = unsigned;
};
template <>
struct StepKey<true> {
    using type = uint64_t;
};

// Strictly lower objective: the ISL, or the (PSL, ISL) pair.
template <bool PSL>
__device__ __forceinline__ bool step_better(int psl, int isl, int psl0, int isl0)
{
    if constexpr (PSL) return psl_better(psl, isl, psl0, isl0);
    return isl < isl0;
}

struct StepEnv {
    const KParams* p;
    uint64_t* T;         // this walker's HT (a valid table for a group without a walker)
    const uint64_t* zk;
    int n, patience;
    uint32_t g;
    __device__ __forceinline__ WalkerState* state() const { return p->states + g; }
};

// The step loops count from the warp's phase, its first walker's step count modulo kCheckEvery,
// so that stop requests are asked for at the same steps whatever the chunks.  (The question
// waits for host memory: asked at every chunk's start, it took a third of a one-step chunk's
// time, 16384 walkers of L = 201 173 us a chunk from 118.  The phase is read again where it is
// needed, which is rare: held, it cost a register and 1.4% of the walk at L = 201.)
template <class LG>
__device__ __forceinline__ int step_phase(const StepEnv& env, const LG& t)
{
    uint32_t h = 0;  // (a group past the last walker stands on one that exists: any valid state)
    if constexpr (LG::kSize < 32) h = min((uint32_t)t.h, env.g);
    return (int)env.p->states[env.g - h].steps_done & (kCheckEvery - 1);
}

// The lags of a lane: E and Z at lags 4 (lane + NL b) .. +3 as FP16 pairs.
template <int NB>
struct StepLags {
    uint32_t e[NB][2], z[NB][2];
};

template <class LAY, class LG, int R>
__device__ __forceinline__ void step_load_lags(int wb, int lane, StepLags<StepShape<LG, R>::NB>& lg)
{
    constexpr StepSmem SL = LAY::SL;
    constexpr int NL = LG::kSize;
#pragma unroll
    for (int b = 0; b < StepShape<LG, R>::NB; ++b) {
        const bool in = 4 * (lane + NL * b) < SL.gpos;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            lg.e[b][j] = in ? lds_u32(sbyte(wb + SL.g + 4 * (lane + NL * b) + 2 * j)) : 0u;
            lg.z[b][j] = lds_u32(sbyte(wb + SL.z + 2 * (lane + NL * b) + j));
        }
    }
}

// Algorithm 1's start for the walker's next restart index: the random (or the learned
// mode's proposed) sequence, its rows, its HT insertion (the generation is fresh: its home
// slot is free).
template <class LAY, class TL>
__device__ __forceinline__ void step_restart(const StepEnv& env, StepWalker& w, int wb, int64_t steps, const TL& t)
{
    const KParams& p = *env.p;
    const int lane = t.lane;
    const uint32_t tmask = (1u << p.tabu_log2) - 1u;
    WalkerState* st = env.state();
    const uint32_t ridx = st->restart_idx + 1;
    DevStatus* S = p.status;
    int prop = 0;
    if (S->learned) prop = S->l_slot_valid[env.g];
    const int tslot = S->learned && S->d_restart != nullptr ? st->trace_slot : -1;
    t.sync();
    if (lane == 0) {
        st->restart_idx = ridx;
        st->restarts += 1;
    }
    w.gen += 1;
    if (w.gen > kGenMask) {
        for (int64_t i = lane; i <= (int64_t)tmask; i += TL::kSize) env.T[i] = 0ull;
        t.sync();
        w.gen = 1;
    }
    if (prop) {
        w.word = lane < kBitWords ? S->l_slot[(int64_t)env.g * kBitWords + lane] : 0u;
        if (tslot >= 0) {
            const int k = S->d_restart_count[tslot];
            const int64_t e = (int64_t)tslot * S->d_cap + k;
            if (k < S->d_cap) {
                if (lane < kBitWords) S->d_restart[e * kBitWords + lane] = w.word;
                if (lane == 0) S->d_restart_idx[e] = ridx;
            }
            t.sync();
            if (lane == 0) S->d_restart_count[tslot] = k + 1;
        }
        t.sync();
        if (lane == 0) S->l_slot_valid[env.g] = 0;
    } else {
        w.word = lane < kBitWords ? start_word(p.seed, env.g, ridx, lane, env.n) : 0u;
    }
    w.isl = step_build<LAY>(wb, w.word, 2 * env.n - 1, env.n, t, &w.psl);
    w.fp = fingerprint_all(w.word, env.zk, env.n, t);
    if (lane == 0) env.T[(uint32_t)w.fp & tmask] = (w.fp & ~kGenMask) | w.gen;
    t.sync();
    w.since = w.isl;
    w.since_psl = w.psl;
    w.stag = 0;
    if (step_better<LAY::kPsl>(w.psl, w.isl, w.best_psl, w.best)) {
        w.best = w.isl;
        w.best_psl = w.psl;
        if (lane == 0) st->best_step = steps;
        if (lane < kBitWords) st->best[lane] = w.word;
    }
    if (w.isl <= w.tisl) {
        w.tisl = -1;
        if (lane == 0) st->target_step = steps;
    }
}

// The two lowest of a walker's keys (b1 <= b2 the lane's own two lowest).
template <class LG>
__device__ __forceinline__ void step_min2(unsigned b1, unsigned b2, const LG& t, unsigned& k0, unsigned& k1)
{
    if constexpr (LG::kSize == 8) {
        // one butterfly carries both: half the latency of two
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
            const unsigned c1 = __shfl_xor_sync(kFull, b1, o), c2 = __shfl_xor_sync(kFull, b2, o);
            const unsigned hi = max(b1, c1);
            b1 = min(b1, c1);
            b2 = min(min(b2, c2), hi);
        }
        k0 = b1;
        k1 = b2;
    } else {
        k0 = t.rminu(b1);
        k1 = t.rminu(b1 == k0 ? b2 : b1);
    }
}

template <class LG>
__device__ __forceinline__ void step_min2(uint64_t b1, uint64_t b2, const LG& t, uint64_t& k0, uint64_t& k1)
{
    k0 = group_min64(b1, t);
    k1 = group_min64(b1 == k0 ? b2 : b1, t);
}

// Keys: the plain walk's 32 bits (below 2^31 for a candidate), or under the PSL objective
// the PSL above them (below 2^63).
__device__ __forceinline__ bool key_none(unsigned k) { return (int)k < 0; }
__device__ __forceinline__ bool key_none(uint64_t k) { return (int64_t)k < 0; }
template <class LG>
__device__ __forceinline__ unsigned group_min(unsigned v, const LG& t) { return t.rminu(v); }
template <class LG>
__device__ __forceinline__ uint64_t group_min(uint64_t v, const LG& t) { return group_min64(v, t); }

// The lane's two lowest keys (all ones where there are fewer).
template <class KT, int R>
__device__ __forceinline__ void key_top2(const KT (&key)[R], KT& b1, KT& b2)
{
    b1 = key[0];
    b2 = ~(KT)0;
#pragma unroll
    for (int r = 1; r < R; ++r) {
        b2 = min(b2, max(b1, key[r]));
        b1 = min(b1, key[r]);
    }
}

template <class LG>
__device__ __forceinline__ int group_of(const LG& t)
{
    if constexpr (LG::kSize == 32)
        return 0;
    else
        return t.h;
}

// The rest of the candidate search when the two best candidates' first HT slots did not
// settle it (a chain longer than the probed slots, or both states visited): the walkers
// with need set try their keys above floor one by one with full probes and insert the
// state they choose.  kc: the chosen key, all ones when every neighbour is in HT; stored:
// the state found a free slot.
template <class LG, class KT, int R>
__device__ __forceinline__ void step_search(const StepEnv& env, uint64_t fp, uint32_t gen, const KT (&key)[R], KT floor,
                                            bool need, const LG& t, KT& kc, bool& stored)
{
    constexpr KT none = ~(KT)0;
    const KParams& p = *env.p;
    const uint32_t tmask = (1u << p.tabu_log2) - 1u;
    const int cap = p.probe_cap;
    do {
        KT b = none;
#pragma unroll
        for (int r = 0; r < R; ++r) b = min(b, key[r] > floor ? key[r] : none);
        const KT k = group_min(need ? b : none, t);
        if (key_none(k)) need = false;  // no candidate left (or the walker is done)
        const uint64_t f = fp ^ (need ? __ldg(env.zk + ((uint32_t)k & 0xFFu)) : 0ull);
        const uint64_t tag = (f & ~kGenMask) | gen;
        bool found = !need;
        for (int s0 = 0; s0 < cap; s0 += LG::kSize) {
            const int s = s0 + t.lane;
            const uint32_t at = ((uint32_t)f + (uint32_t)s) & tmask;
            uint64_t e = 0;
            const bool live = !found && s < cap;
            if (live) e = env.T[at];
            const bool match = live && e == tag;
            const unsigned bal = t.ballot(live && ((((uint32_t)e & (uint32_t)kGenMask) != gen) || match));
            const unsigned mat = t.ballot(match);
            if (bal && !found) {
                found = true;
                const unsigned first = bal & (0u - bal);
                if (mat & first) {
                    floor = k;  // visited
                } else {
                    kc = k;
                    stored = true;
                    need = false;
                    if ((1u << t.lane) == first) env.T[at] = tag;
                }
            }
        }
        if (need && !found) {  // no free slot within the cap: taken, not inserted
            kc = k;
            need = false;
        }
    } while (__any_sync(kFull, need));
}

// Log record of walker wi's chunk that starts at step steps0, or null.
__device__ __forceinline__ labs_log_record* step_record(const KParams& p, int64_t wi, int64_t steps0)
{
    const DevStatus* S = p.status;
    if (S->log == nullptr || p.chunk_steps <= 0) return nullptr;
    const int64_t since = steps0 - S->log_start;
    if (since < 0 || since % p.chunk_steps != 0) return nullptr;
    const int64_t idx = (since / p.chunk_steps) * p.W + wi;
    return idx < S->log_capacity ? S->log + idx : nullptr;
}

// Trace and log of one step (one lane of a walker that has either); false once the log
// record is complete.
__device__ __forceinline__ bool step_note(const StepEnv& env, int it, int code, int isl, unsigned extras)
{
    const KParams& p = *env.p;
    const WalkerState* st = env.state();
    const int64_t steps0 = st->steps_done;
    if (extras & 1u) {
        const DevStatus* D = p.status;
        const int64_t slot = st->trace_slot, s = steps0 + it - p.trace_start[slot];
        if (s >= 0 && s < D->trace_capacity) {
            D->trace_code[slot * D->trace_capacity + s] = code;
            D->trace_isl[slot * D->trace_capacity + s] = isl;
        }
    }
    if (extras & 2u) {
        // lowest ISL at the end of the chunk's steps before its first restart step
        labs_log_record* rec = step_record(p, env.g, steps0);
        if (it == 0) rec->first = code;
        if (code == LABS_TRACE_BLOCKED || (code & LABS_TRACE_RESTART)) return false;
        if (isl < rec->min_isl) rec->min_isl = isl;
    }
    return true;
}

// ------------------------------------------------------------------ PSL of the neighbours
//
// Flipping output v of class p changes C_{2m} by ms (a_{v+m} + a_{v-m}), ms = -4 s_i (centre
// -2 s_c), the mirror's own term a_{v+m} (m = c - i) left out: by at most 8.  So of all lags
// only those within 8 of the sequence's PSL can decide a neighbour's unless the neighbour is
// better than the sequence, and then those within 8 of the best neighbour's bound: about 31
// and 1.4 of 100 lags at L = 201 (28% of the steps need the second band).  The lags of a
// band are listed in shared memory (lag and C as one word) and every lane takes its R
// outputs through them in FP16 pairs, exact on these small integers.  All lags of all
// outputs in FP32 took 59.5 ms for 16384 walkers x 1000 steps at L = 201.

// Lists the walker's lags with lo <= |C| < hi (both groups of a warp together: returns the
// longer list's length, the shorter one filled with lag n, whose terms are all zero).
template <class LAY, class LG, int R>
__device__ __forceinline__ int psl_list(uint32_t list, const StepLags<StepShape<LG, R>::NB>& lg, int n, int lo, int hi,
                                        const LG& t)
{
    constexpr int NL = LG::kSize;
    const uint32_t lob = half_bits(max(lo, 0)), hib = half_bits(max(hi, 0));
    const unsigned below = ((1u << t.lane) - 1u);
    int count = 0;
#pragma unroll
    for (int b = 0; b < StepShape<LG, R>::NB; ++b)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t e = (j & 1) ? lg.e[b][j >> 1] >> 16 : lg.e[b][j >> 1] & 0xFFFFu, ab = e & 0x7FFFu;
            const int m = 4 * (t.lane + NL * b) + j;
            const bool in = ab >= lob && ab < hib && m > 0 && m < n;
            const unsigned bal = t.ballot(in);
            if (in) sts_u32(list + 4 * (count + __popc(bal & below)), (uint32_t)m | (e << 16));
            count += __popc(bal);
        }
    const int top = __reduce_max_sync(kFull, count);
    for (int k = count + t.lane; k < top; k += NL) sts_u32(list + 4 * k, (uint32_t)n);
    __syncwarp();
    return top;
}

// Takes the lane's outputs through a list: mx = max(mx, |C'|), outputs 2j and 2j+1 in pair j.
template <class LAY, class LG, int R>
__device__ __forceinline__ void psl_terms(uint32_t list, int top, uint32_t rows, int v0, int z0, uint32_t corr,
                                          const uint32_t (&ms)[(R + 1) / 2], uint32_t (&mx)[(R + 1) / 2])
{
    constexpr StepSmem SL = LAY::SL;
    constexpr int J = (R + 1) / 2;
    for (int k = 0; k < top; ++k) {
        const uint32_t w = lds_u32(list + 4 * k);
        const int m = (int)(w & 0xFFFFu);
        const uint32_t c2 = __byte_perm(w, w, 0x3232);
        // entries v0 + m and v0 - m have the same parity: the same copy; entry u of copy 1 is
        // at half u - 1
        const uint32_t r = rows + ((v0 + m) & 1 ? 4 * SL.ks - 2 : 0);
        const uint32_t up = r + 2 * (v0 + m), dn = r + 2 * (v0 - m);
        // the output whose mirror this lag reaches (its a_{v+m} is sg s_i): z / 2, if even
        const int z = z0 - m;
        const uint32_t cx = as_u32(__hadd2(as_half2(c2), as_half2((z & 2) ? corr << 16 : corr)));
        const int zj = (z & 1) ? -1 : z >> 2;
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const __half2 s2 = __hadd2(as_half2(lds_u32(up + 4 * j)), as_half2(lds_u32(dn + 4 * j)));
            const __half2 e = __hfma2(as_half2(ms[j]), s2, as_half2(zj == j ? cx : c2));
            mx[j] = as_u32(__hmax2(as_half2(mx[j]), __habs2(e)));
        }
    }
}

// ------------------------------------------------------------------ parts of a step

// A lane's base addresses and constants.
template <class LAY, class LG, int R>
struct StepLane {
    using SH = StepShape<LG, R>;
    StepProduct<LAY, LG, R> prod;
    uint32_t xr;      // results; coefficients at a fixed distance
    uint32_t zr, sr;  // Z and s_{3i-L+1} of the outputs
    uint32_t rows, gw, zw;
    float sig4, bias;
    uint32_t ib;  // free variables i of outputs 0-3, one byte each
    int hw4;      // row words from here on are zero in both copies
    int wb, n;
    __device__ __forceinline__ StepLane(int wb0, int n_, const LG& t, const Outs<LG, R>& o)
        : prod(wb0, t.lane + t.base), wb(wb0 + group_of(t) * LAY::SL.words), n(n_)
    {
        constexpr StepSmem SL = LAY::SL;
        const int c = n - 1;
        xr = sbyte(wb + SL.x + o.p * SL.xp + o.v0);
        // a lane without outputs reads Z below 0 (no output) and any finite row entry
        zr = sbyte(wb + SL.z) + 2 * max(c - o.p - 2 * o.v0, -1);
        sr = sbyte(wb + SL.h0 + o.p * SL.hc) + 2 * (2 * o.v0 + o.p <= c ? 3 * o.v0 + o.p - n + 1 : 0);
        rows = sbyte(wb + SL.h0);
        gw = sbyte(wb + SL.g + 4 * t.lane);
        zw = sbyte(wb + SL.z + 2 * t.lane);
        sig4 = ((c - o.p) & 1) ? -4.f : 4.f;
        bias = (float)(16 * (n - o.p - 3)) + kIntBias;  // 16 (N_p - 2), N_p = n - 1 - p
        ib = (uint32_t)(2 * o.v0 + o.p) * 0x01010101u + 0x06040200u;
        hw4 = 4 * ((n + 1) >> 1);
    }
};

// Keys (dISL + 2^22) << 8 | i of the lane's outputs after step_toeplitz, ascending in (dISL,
// i): the FP32 value dISL + 1.5 2^23 holds the integer in its low bits, and one byte
// permute puts i below its low three bytes.  Outputs that do not exist or are marked have
// an infinite Z, whose bytes give a key of at least 2^31.  ms (MS): -8 s_i / 2 as FP16 pairs.
template <bool MS, class LAY, class LG, int R>
__device__ __forceinline__ void step_keys(const StepLane<LAY, LG, R>& a, unsigned (&key)[R], uint32_t (&ms)[(R + 1) / 2])
{
    constexpr StepSmem SL = LAY::SL;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const float x = lds_f32(a.xr + 4 * r), r8 = lds_f32(a.xr - 4u * (uint32_t)(SL.x - SL.r8) + 4 * r);
        const float z = lds_f16(a.zr - 4 * r), s3 = lds_f16(a.sr + 6 * r);
        const float v = fmaf(r8, fmaf(a.sig4, s3, x), fmaf(8.f, z, a.bias));
        key[r] = __byte_perm(__float_as_uint(v), r < 4 ? a.ib : r < 8 ? a.ib + 0x08080808u : a.ib + 0x10101010u,
                             0x2104 + (r & 3));
        if (MS) {
            const uint32_t h = __half_as_ushort(__float2half_rn(0.5f * r8));
            ms[r >> 1] = (r & 1) ? ms[r >> 1] | (h << 16) : h;
        }
    }
}

// Flips free variable bi (and its mirror) of the walkers with `moves` in rows, coefficients,
// table and Z; neg: 0x80000000 where s_i = -1 before the flip.  mark: the flipped output is
// no candidate of the next step (the lags' next store of Z takes the mark away).   The flipped entries read as 0 while the sums are
// taken, which leaves out the pairs whose two ends both flip and lag 0.
template <class LAY, class LG, int R>
__device__ __forceinline__ void step_flip(const StepLane<LAY, LG, R>& a, StepLags<StepShape<LG, R>::NB>& lg, bool moves,
                                          int bi, uint32_t neg, bool mark, const LG& t)
{
    constexpr StepSmem SL = LAY::SL;
    constexpr int NL = LG::kSize, NB = StepShape<LG, R>::NB;
    const int lane = t.lane, n = a.n, c = n - 1;
    const int pb = bi & 1, vb = bi >> 1, vq = n - 1 - pb - vb;
    const bool centre = bi == c, same = ((pb ^ c) & 1) == 0;  // same: sg = +1 in the flipped class
    const uint32_t rb = a.rows + (pb ? 4 * SL.hc : 0);
    const bool writer = moves && lane < 2;  // lane 0 writes s_i, lane 1 its mirror
    const uint32_t ea = rb + 2 * (lane ? vq : vb);
    sts_u16_if(writer, ea, 0u);
    sts_u16_if(writer, ea + 4 * SL.ks - 2, 0u);
    __syncwarp();
    {
        // at lag m the flipped class's autocorrelation changes by -2 s_i (a_{vb+m} +
        // a_{vb-m}) for each flipped end, in all coef (a_{vb+m} + sg a_{vq+m}), coef = -4
        // s_i (centre: -2 s_c): a_{vb-m} = sg a_{vq+m}
        const __half2 coef = as_half2(moves ? (centre ? 0xC000C000u : 0xC400C400u) ^ (neg | neg >> 16) : 0u);
        const __half2 sig = as_half2(same ? 0x3C003C00u : 0xBC00BC00u);
        // Z: 3 x the lag's own class, 1 x the other, sign (-1)^m
        const __half2 cz = __hmul2(coef, as_half2(same ? 0xBC004200u : 0xC2003C00u));
        const uint32_t ub = rb + ((vb & 1) ? 4 * SL.ks : 0), qb = rb + ((vq & 1) ? 4 * SL.ks : 0);
        const int uo = 2 * (vb & ~1) + 8 * lane, qo = 2 * (vq & ~1) + 8 * lane;
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const uint32_t u = ub + min(uo + 8 * NL * b, a.hw4), q = qb + min(qo + 8 * NL * b, a.hw4);
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const __half2 s2 = __hfma2(sig, as_half2(lds_u32(q + 4 * j)), as_half2(lds_u32(u + 4 * j)));
                lg.e[b][j] = as_u32(__hfma2(coef, s2, as_half2(lg.e[b][j])));
                lg.z[b][j] = as_u32(__hfma2(cz, s2, as_half2(lg.z[b][j])));
            }
        }
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            // the lag after the lane's block: the next lane's first (the next block's first
            // lane for the last one)
            const uint32_t give = lane == 0 ? (b + 1 < NB ? lg.e[b + 1 < NB ? b + 1 : b][0] : 0u) : lg.e[b][0];
            const uint32_t nx = __shfl_sync(kFull, give, t.base + ((lane + 1) & (NL - 1)));
            const uint32_t e0 = lg.e[b][0], e1 = lg.e[b][1];
            const uint32_t o0 = __byte_perm(e0, e1, 0x5432), o1 = __byte_perm(e1, nx, 0x5432);
            if (4 * NL * (b + 1) <= SL.gpos)
                sts_v4(a.gw + 16 * NL * b, e0, o0, e1, o1);
            else
                sts_v4_if(lane < SL.gpos / 4 - NL * b, a.gw + 16 * NL * b, e0, o0, e1, o1);
            if (4 * NL * b < SL.gneg) {
                // the mirror: G[-m-1] is G[m] with its halves exchanged
                const uint32_t m = a.gw - 32 * lane - 16 - 16 * NL * b;
                const uint32_t r0 = __byte_perm(o1, o1, 0x1032), r1 = __byte_perm(e1, e1, 0x1032),
                               r2 = __byte_perm(o0, o0, 0x1032), r3 = __byte_perm(e0, e0, 0x1032);
                if (4 * NL * (b + 1) <= SL.gneg)
                    sts_v4(m, r0, r1, r2, r3);
                else
                    sts_v4_if(lane < SL.gneg / 4 - NL * b, m, r0, r1, r2, r3);
            }
            sts_v2(a.zw + 8 * NL * b, lg.z[b][0], lg.z[b][1]);
        }
    }
    __syncwarp();
    // s_i and, with the class's sign, its mirror, both negated: an entry is +1 exactly when
    // s_i (lane 1: sg s_i) was -1
    const uint32_t s = (neg != 0u) == (lane == 0 || same) ? 0x3C00u : 0xBC00u;
    sts_u16_if(writer, ea, s);
    sts_u16_if(writer, ea + 4 * SL.ks - 2, s);
    const bool first = moves && lane == 0;
    sts_f32_if(first, sbyte(a.wb + SL.r8) + (pb ? 4 * SL.xp : 0) + 4 * vb,
               __uint_as_float((centre ? 0x40800000u : 0x41000000u) | neg));
    if (mark) sts_u16_if(first, sbyte(a.wb + SL.z) + 2 * (c - bi), kHalfInf);
}

// 0x80000000 where free variable i of the walker's bits is -1.
template <class LG>
__device__ __forceinline__ uint32_t step_sign(uint32_t word, int i, const LG& t)
{
    return (t.shfl(word, i >> 5) << (31 - (i & 31))) & 0x80000000u;
}

// ------------------------------------------------------------------ the walk's steps

// Advances the warp's walkers by up to len steps each (one per lane group; `real`: the
// group has one), from shared state built by step_build.  RT is the tile type a group
// restarts with (divergently).  extras: bit 0 the walker is traced, bit 1 its chunk is
// logged.  Returns the steps taken.
//
// AHEAD (few walkers): with a warp or two on a scheduler nothing covers the latency of the HT
// lookup, which was half of a step.  The states of all neighbours are known when a step
// starts, so every lane loads the first HT slot of each of its R outputs then, under the
// product; what is found visited leaves the keys, and the lowest key left is the move (an
// occupied first slot of another state sends the walker to step_search).  n loads a step
// instead of one or two: only while the walkers' HT traffic is small (kAheadSlots).
template <class LAY, class LG, class RT, int R, bool AHEAD = false>
__device__ __forceinline__ int walk_lockstep(const StepEnv& env, StepWalker& w, int len, bool real, int wb0,
                                             unsigned extras, const LG& t, const RT& tt)
{
    constexpr StepSmem SL = LAY::SL;
    constexpr int NL = LG::kSize, NB = StepShape<LG, R>::NB;
    constexpr int S = NL / 2;  // HT slots probed per candidate in a round
    constexpr bool PSL = LAY::kPsl;
    using KT = typename StepKey<PSL>::type;
    const KParams& p = *env.p;
    const int lane = t.lane, l = lane + t.base, n = env.n, c = n - 1;
    const Outs<LG, R> o(t);
    const StepLane<LAY, LG, R> a(wb0, n, t, o);
    const int wb = a.wb;
    StepLags<NB> lg;
    step_load_lags<LAY, LG, R>(wb, lane, lg);
    StopCheck stop;
    stop.start(p, l == 0);
    const uint32_t tmask = (1u << p.tabu_log2) - 1u;
    uint64_t zkr[AHEAD ? R : 1], ent[AHEAD ? R : 1];
    if constexpr (AHEAD) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int i = 2 * (o.v0 + r) + o.p;
            zkr[r] = i <= c ? __ldg(env.zk + i) : 0ull;
        }
    }
    int it = __shfl_sync(kFull, step_phase(env, t), 0);
    len += it;
    const int top = __reduce_max_sync(kFull, real ? len : 0);
    for (; it < top; ++it) {
        const bool act = real && it < len;
        if ((it & (kCheckEvery - 1)) == 0) {
            const int why = __shfl_sync(kFull, stop.poll(p, l == 0), 0);
            if (why) {
                if (act && lane == 0) raise_error(p.status, why, (int)env.g);
                break;
            }
        }
        if constexpr (AHEAD) {
#pragma unroll
            for (int r = 0; r < R; ++r) ent[r] = env.T[(uint32_t)(w.fp ^ zkr[r]) & tmask];
        }
        step_toeplitz<LAY, LG, R>(a.prod, l);

        // The move back to the state just left is marked (that state is always in HT).  Under
        // the PSL objective the PSL (as FP16 bits, which order as the integers do) goes above
        // the key.
        KT key[R];
        {
            unsigned kl[R];
            uint32_t ms[(R + 1) / 2];
            step_keys<PSL>(a, kl, ms);
            if constexpr (PSL) {
                uint32_t mx[(R + 1) / 2];
#pragma unroll
                for (int j = 0; j < (R + 1) / 2; ++j) mx[j] = 0u;
                const uint32_t list = sbyte(wb + SL.x), prow = sbyte(wb + SL.h0 + o.p * SL.hc);
                const uint32_t corr = ((c - o.p) & 1) ? 0xC400u : 0x4400u;  // 4 sg
                const int z0 = c - o.p - 2 * o.v0;
                __syncwarp();  // the list takes the results' place
                int top_k = psl_list<LAY, LG, R>(list, lg, n, w.psl - 8, 0x7FF, t);
                psl_terms<LAY, LG, R>(list, top_k, prow, o.v0, z0, corr, ms, mx);
                uint32_t lb = 0x7FFFu;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const uint32_t h = (r & 1) ? mx[r >> 1] >> 16 : mx[r >> 1] & 0xFFFFu;
                    lb = min(lb, (int)kl[r] < 0 ? 0x7FFFu : h);
                }
                lb = t.rminu(lb);
                const int low = (int)__half2float(__ushort_as_half((unsigned short)lb));
                if (__any_sync(kFull, act && low < w.psl)) {
                    __syncwarp();
                    const bool more = low < w.psl;
                    top_k = psl_list<LAY, LG, R>(list, lg, n, more ? low - 7 : 0, more ? w.psl - 8 : 0, t);
                    psl_terms<LAY, LG, R>(list, top_k, prow, o.v0, z0, corr, ms, mx);
                }
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const uint32_t h = (r & 1) ? mx[r >> 1] >> 16 : mx[r >> 1] & 0xFFFFu;
                    key[r] = ((uint64_t)(h | (uint32_t)((int)kl[r] >> 31)) << 32) | kl[r];
                }
            } else {
#pragma unroll
                for (int r = 0; r < R; ++r) key[r] = kl[r];
            }
        }
        // Best admissible flip: the lowest key whose state is not in HT.  The two lowest
        // are probed at once, the first S HT slots of each by one half of the walker's
        // lanes; that settles nearly every step, step_search does the others.
        KT kc;
        uint32_t at;
        uint64_t tag;
        bool stored = true, insert;  // insert: this lane writes the chosen state to HT
        if constexpr (AHEAD) {
            uint32_t occ = 0;  // outputs whose first slot holds a state of this start
            KT b = ~(KT)0;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const uint64_t tr = ((w.fp ^ zkr[r]) & ~kGenMask) | w.gen;
                if (ent[r] == tr) key[r] = ~(KT)0;
                occ |= ((uint32_t)ent[r] & (uint32_t)kGenMask) == w.gen ? 1u << r : 0u;
                b = min(b, key[r]);
            }
            kc = group_min(b, t);
            if (key_none(kc)) kc = ~(KT)0;
            const int i0 = (int)((uint32_t)kc & 0xFFu), r0 = (i0 >> 1) - o.v0;
            const bool other = act && kc != ~(KT)0 && (i0 & 1) == o.p && (unsigned)r0 < (unsigned)R && ((occ >> r0) & 1u);
            const uint64_t f = w.fp ^ __ldg(env.zk + i0);
            at = (uint32_t)f & tmask;
            tag = (f & ~kGenMask) | w.gen;
            insert = lane == 0;
            if (__any_sync(kFull, other)) {
                const bool need = t.ballot(other) != 0u;
                KT ks = ~(KT)0;
                bool st = false;
                step_search(env, w.fp, w.gen, key, (KT)0, need, t, ks, st);
                if (need) {
                    kc = ks;
                    stored = st;
                    insert = false;
                }
            }
        } else {
            KT b1, b2, k0, k1;
            key_top2(key, b1, b2);
            step_min2(b1, b2, t, k0, k1);
            const int hs = lane & (S - 1);
            const KT km = lane >= S ? k1 : k0;
            const bool live = act && !key_none(km) && hs < p.probe_cap;
            // a key without an output reads past the length's fingerprint keys, within the workspace
            const uint64_t f = w.fp ^ __ldg(env.zk + ((uint32_t)km & 0xFFu));
            at = ((uint32_t)f + (uint32_t)hs) & tmask;
            tag = (f & ~kGenMask) | w.gen;
            const uint64_t e = env.T[at];
            const bool match = live && e == tag;
            const unsigned hb = __ballot_sync(kFull, match || (live && ((uint32_t)e & (uint32_t)kGenMask) != w.gen));
            const unsigned mb = __ballot_sync(kFull, match);
            {
                // pick: the lane that saw the free slot of the chosen state (0: not settled)
                const unsigned g0 = hb & (((1u << S) - 1u) << t.base), g1 = hb & (((1u << S) - 1u) << (t.base + S));
                const unsigned p0 = g0 & (0u - g0), p1 = g1 & (0u - g1);  // each candidate's first hit
                const bool v0 = (p0 & mb) != 0u, v1 = (p1 & mb) != 0u;
                kc = v0 ? k1 : k0;
                const unsigned pick = v0 ? (v1 ? 0u : p1) : p0;
                insert = (pick >> l) == 1u;
                if (__any_sync(kFull, act && pick == 0u)) {
                    const bool need = act && pick == 0u;
                    KT ks = ~(KT)0;
                    bool st = false;
                    step_search(env, w.fp, w.gen, key, v0 ? (v1 ? k1 : k0) : (KT)0, need, t, ks, st);
                    if (need) {
                        kc = ks;
                        stored = st;
                    }
                }
            }
        }
        const bool moves = act && kc != ~(KT)0;
        stg_u64_if(moves && insert, env.T + at, tag);

        // Apply the move (walkers that have one).
        const int bi = moves ? (int)((uint32_t)kc & 0xFFu) : 0;
        const uint32_t neg = step_sign(w.word, bi, t);
        const uint64_t zk = __ldg(env.zk + bi);
        step_flip(a, lg, moves, bi, neg, true, t);
        bool again = act;
        if (moves) {
            if (lane == (bi >> 5)) w.word ^= 1u << (bi & 31);
            w.fp ^= zk;
            w.isl += (int)((uint32_t)kc >> 8) - kKeyBias;
            if constexpr (PSL) w.psl = (int)__half2float(__ushort_as_half((unsigned short)((uint64_t)kc >> 32)));
            w.stag += 1;
            if (step_better<PSL>(w.psl, w.isl, w.since_psl, w.since)) {
                w.since = w.isl;
                w.since_psl = w.psl;
                w.stag = 0;
            }
            again = w.stag >= env.patience || !stored;
        }
        if (moves && (step_better<PSL>(w.psl, w.isl, w.best_psl, w.best) || w.isl <= w.tisl)) {
            WalkerState* st = env.state();
            const int64_t steps = st->steps_done + (it - step_phase(env, t)) + 1;
            if (step_better<PSL>(w.psl, w.isl, w.best_psl, w.best)) {
                w.best = w.isl;
                w.best_psl = w.psl;
                if (lane == 0) st->best_step = steps;
                if (lane < kBitWords) st->best[lane] = w.word;
            }
            if (w.isl <= w.tisl) {
                w.tisl = -1;
                if (lane == 0) st->target_step = steps;
            }
        }
        if (again) {  // several walkers per warp: divergent, only this group restarts
            WalkerState* st = env.state();
            if (lane == 0) {
                if (!moves)
                    st->blocked += 1;
                else if (!stored)
                    st->overflows += 1;
            }
            step_restart<LAY>(env, w, wb, st->steps_done + (it - step_phase(env, t)) + 1, tt);
            step_load_lags<LAY, LG, R>(wb, lane, lg);
        }
        __syncwarp();
        if (extras && act && lane == 0) {
            const int code = !moves ? LABS_TRACE_BLOCKED : again ? bi | LABS_TRACE_RESTART : bi;
            if (!step_note(env, it - step_phase(env, t), code, w.isl, extras)) extras &= ~2u;
        }
    }
    return min(it, len) - __shfl_sync(kFull, step_phase(env, t), 0);
}

// ------------------------------------------------------------------ best-first search
//
// Algorithm 1 as printed (impxLast, Section 3): the neighbourhood of S fills a queue of
// LABS_QUEUE_SIZE evaluated neighbours ordered by merit factor and the next S is the queue's
// first entry (the readings are stated with labs_walk in labs.h).  One walker per warp; lane
// l holds queue entry l as a 64-bit key
//   ISL << 36 | (steps done before the step that produced it) << 8 | i
// (ascending = the queue order; ~0 = empty) and the entry's free variables live in global
// memory.  A new S that differs from S in at most kBestFirstMaxFlips free variables is
// reached by that many flips, any other by a rebuild from its bits.
//
// What bounds it: the queue's insertions and the move, not the neighbourhood (about 3
// insertions a step, each a minimum over the warp and an HT lookup).  16384 walkers x 1000
// steps at L = 201: 35.9 ms, 51.6 on FP32 rows and table at 16 warps per SM (38.7 before the
// entries' fingerprints were kept and the candidates' HT lines prefetched).
template <class LAY, int R>
__device__ __forceinline__ int walk_bestfirst(const StepEnv& env, StepWalker& w, int len, bool real, int wb,
                                              unsigned extras, const Tile<32>& t)
{
    static_assert(LABS_QUEUE_SIZE == 32, "one queue entry per lane");
    using LG = Tile<32>;
    const KParams& p = *env.p;
    const int lane = t.lane, n = env.n;
    const Outs<LG, R> o(t);
    const StepLane<LAY, LG, R> a(wb, n, t, o);
    const int cap = p.probe_cap;
    const uint32_t tmask = (1u << p.tabu_log2) - 1u;
    uint64_t* const qkey = p.pq_key + (int64_t)env.g * LABS_QUEUE_SIZE;
    uint32_t* const qbits = p.pq_bits + (int64_t)env.g * LABS_QUEUE_SIZE * kBitWords;
    uint64_t qk = qkey[lane];
    // the entry's fingerprint (kept beside its key while the chunk runs)
    uint64_t qf = 0ull;
    if (qk != ~0ull)
        for (int j = 0; 32 * j < n; ++j)
            for (uint32_t x = qbits[lane * kBitWords + j]; x; x &= x - 1u) qf ^= __ldg(env.zk + 32 * j + __ffs(x) - 1);
    __syncwarp();
    // xLastovka's second table (null when off): slot f mod size holds
    // (generation << 40) | (~f mod 2^40) of an evaluated neighbour f
    uint64_t* const T2 = p.tabu2 != nullptr ? p.tabu2 + (env.T - p.tabu) : nullptr;
    constexpr uint64_t kLow40 = 0xFFFFFFFFFFull;
    int64_t hits = 0;
    int it = step_phase(env, t);
    const int64_t steps0 = env.state()->steps_done - it;  // before step it = 0
    StepLags<StepShape<LG, R>::NB> lg;
    step_load_lags<LAY, LG, R>(wb, lane, lg);
    StopCheck stop;
    stop.start(p, lane == 0);
    len = real ? len + it : 0;
    for (; it < len; ++it) {
        if ((it & (kCheckEvery - 1)) == 0) {
            const int why = t.shfl(stop.poll(p, lane == 0), 0);
            if (why) {
                if (lane == 0) raise_error(p.status, why, (int)env.g);
                break;
            }
        }
        const uint64_t e = (uint64_t)(steps0 + it);
        step_toeplitz<LAY, LG, R>(a.prod, lane);
        unsigned key[R];
        {
            uint32_t ms[(R + 1) / 2];
            step_keys<false>(a, key, ms);
        }
        if (T2 != nullptr) {
            // neighbours the table holds are skipped (their keys dropped); every other one is
            // inserted once all lanes have looked (larger word kept: the table does not
            // depend on the order of the insertions)
            uint64_t ins[R];
            int h = 0;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                ins[r] = 0ull;
                if ((int)key[r] < 0) continue;
                const uint64_t f = w.fp ^ __ldg(env.zk + (key[r] & 0xFFu));
                const uint64_t tag = ((uint64_t)w.gen << 40) | (~f & kLow40);
                if (T2[(uint32_t)f & tmask] == tag) {
                    key[r] = 0xFFFFFFFFu;
                    ++h;
                } else {
                    ins[r] = f;
                }
            }
            hits += t.radd(h);
            t.sync();
#pragma unroll
            for (int r = 0; r < R; ++r)
                if ((int)key[r] >= 0)
                    atomicMax(reinterpret_cast<unsigned long long*>(T2 + ((uint32_t)ins[r] & tmask)),
                              (unsigned long long)(((uint64_t)w.gen << 40) | (~ins[r] & kLow40)));
            t.sync();
        }
        // Neighbours in queue order (ISL, then i: the packed keys' order) while they come
        // before the queue's last entry or the queue has a free place.  The last entry only
        // moves forward during the step, so neighbours after its value at the start cannot
        // enter; the others are looked up in HT as the insertion reaches them (HT does not
        // change during the insertion).  A new key orders behind the queue's of equal ISL (its
        // step is later, or its i is higher), so a candidate comes before the last entry
        // exactly when its ISL is lower.
        unsigned qempty = t.ballot(qk == ~0ull);
        uint64_t last = qempty ? ~0ull : warp_max64(qk);
        unsigned limit = 0x80000000u;  // keys below it may enter
        if (!qempty) {
            const int64_t d = (int64_t)(last >> 36) - w.isl + kKeyBias;
            limit = d <= 0 ? 0u : (unsigned)min(d << 8, (int64_t)0x80000000ll);
        }
        // the HT lines of the lanes' lowest candidates are on their way before the insertion
        // asks for them one after the other
        {
            unsigned b = key[0];
#pragma unroll
            for (int r = 1; r < R; ++r) b = min(b, key[r]);
            if (b < limit)
                asm volatile("prefetch.global.L1 [%0];" ::"l"(env.T + ((uint32_t)(w.fp ^ __ldg(env.zk + (b & 0xFFu))) & tmask)));
        }
        unsigned floor = 0u;
        for (;;) {
            unsigned b = 0x80000000u;
#pragma unroll
            for (int r = 0; r < R; ++r) b = min(b, key[r] > floor ? key[r] : 0x80000000u);
            const unsigned k = t.rminu(b);
            if (k >= limit) break;
            floor = k;
            const int i = (int)(k & 0xFFu);
            const uint64_t f = w.fp ^ __ldg(env.zk + i);
            {
                // HT lookup of this neighbour: up to probe_cap slots, four per round
                const uint64_t tag = (f & ~kGenMask) | w.gen;
                bool visited = false;
                for (int s0 = 0; s0 < cap; s0 += 4) {
                    const bool mine = lane < 4 && s0 + lane < cap;
                    const uint64_t x = mine ? env.T[((uint32_t)f + (uint32_t)(s0 + lane)) & tmask] : 0ull;
                    const unsigned bal = t.ballot(mine && ((((uint32_t)x & (uint32_t)kGenMask) != w.gen) || x == tag));
                    const unsigned mat = t.ballot(mine && x == tag);
                    if (bal) {
                        visited = (mat & bal & (0u - bal)) != 0u;
                        break;
                    }
                }
                if (visited) continue;
            }
            const int isl_f = w.isl + (int)(k >> 8) - kKeyBias;
            const uint64_t ck = ((uint64_t)isl_f << 36) | (e << 8) | (uint64_t)i;
            const int dst = __ffs(qempty ? qempty : t.ballot(qk == last)) - 1;
            if (lane == dst) {
                qk = ck;
                qf = f;
            }
            const uint32_t word = w.word ^ (lane == (i >> 5) ? 1u << (i & 31) : 0u);
            if (lane < kBitWords) qbits[dst * kBitWords + lane] = word;
            if (isl_f < w.best) {
                w.best = isl_f;
                if (lane == 0) env.state()->best_step = (int64_t)e + 1;
                if (lane < kBitWords) env.state()->best[lane] = word;
            }
            if (isl_f <= w.tisl) {
                w.tisl = -1;
                if (lane == 0) env.state()->target_step = (int64_t)e + 1;
            }
            qempty &= qempty - 1u;
            if (!qempty) {
                // the queue is full: the rest enter only below its last entry
                last = warp_max64(qk);
                const int64_t d = (int64_t)(last >> 36) - w.isl + kKeyBias;
                limit = d <= 0 ? 0u : (unsigned)min(d << 8, (int64_t)0x80000000ll);
            }
        }
        t.sync();
        // S <- the queue's first entry not in HT (entries that are get dropped)
        int code = LABS_TRACE_BLOCKED;
        bool again = true, moved = false;
        for (;;) {
            if (!t.ballot(qk != ~0ull)) break;  // empty queue: restart
            const uint64_t first = warp_min64(qk);
            const int src = __ffs(t.ballot(qk == first)) - 1;
            const uint32_t word = lane < kBitWords ? qbits[src * kBitWords + lane] : 0u;
            if (lane == src) qk = ~0ull;
            const bool nb = ((first >> 8) & 0xFFFFFFFull) == e;  // a neighbour of S
            const uint64_t f = ((uint64_t)t.shfl((uint32_t)(qf >> 32), src) << 32) | t.shfl((uint32_t)qf, src);
            const uint64_t tag = (f & ~kGenMask) | w.gen;
            bool visited = false;
            int64_t slot = -1;
            for (int s0 = 0; s0 < cap; s0 += 32) {
                const int s = s0 + lane;
                const uint64_t x = s < cap ? env.T[((uint32_t)f + (uint32_t)s) & tmask] : 0ull;
                const unsigned bal = t.ballot(s < cap && ((((uint32_t)x & (uint32_t)kGenMask) != w.gen) || x == tag));
                const unsigned mat = t.ballot(s < cap && x == tag);
                if (bal) {
                    visited = (mat & bal & (0u - bal)) != 0u;
                    slot = ((uint32_t)f + (uint32_t)(s0 + __ffs(bal) - 1)) & tmask;
                    break;
                }
            }
            if (visited) continue;
            // free variables in which the new S differs from S (1 for a neighbour)
            uint32_t diff = lane < kBitWords ? (word ^ w.word) : 0u;
            const int k = nb ? 1 : t.radd(__popc(diff));
            if (k <= kBestFirstMaxFlips) {
                // flip them one by one, lowest first
                for (int j = 0; j < k; ++j) {
                    const unsigned bl = t.ballot(diff != 0u);
                    const int sl = __ffs(bl) - 1;
                    const int fi = 32 * sl + t.shfl(__ffs(diff) - 1, sl);
                    const uint32_t neg = step_sign(w.word, fi, t);
                    step_flip(a, lg, true, fi, neg, false, t);
                    t.sync();
                    if (lane == sl) diff &= diff - 1u;
                }
            } else {
                int none;
                step_build<LAY>(wb, word, 2 * n - 1, n, t, &none);
                step_load_lags<LAY, LG, R>(wb, lane, lg);
            }
            moved = true;
            w.word = word;
            w.isl = (int)(first >> 36);
            w.fp = f;
            code = (int)(f & 0xFFFFu);
            if (slot >= 0) {
                if (lane == 0) env.T[slot] = tag;
                again = false;
            } else {
                code |= LABS_TRACE_RESTART;  // no free HT slot for the new S: restart
            }
            break;
        }
        if (again) {
            WalkerState* st = env.state();
            if (lane == 0) {
                if (moved)
                    st->overflows += 1;
                else
                    st->blocked += 1;
            }
            qk = ~0ull;
            const uint32_t gen0 = w.gen;
            step_restart<LAY>(env, w, wb, (int64_t)e + 1, t);
            if (T2 != nullptr && w.gen < gen0) {  // generations wrapped: HT was zeroed, so is T2
                for (int64_t i = lane; i <= (int64_t)tmask; i += 32) T2[i] = 0ull;
                t.sync();
            }
            step_load_lags<LAY, LG, R>(wb, lane, lg);
        }
        t.sync();
        if (extras && lane == 0) step_note(env, it - step_phase(env, t), code, w.isl, extras & 1u);
    }
    if (real) {
        qkey[lane] = qk;
        if (lane == 0) env.state()->cache_hits += hits;
    }
    return it - step_phase(env, t);
}

// CTAs of 8 warps per SM the walk kernels are compiled for: three (80 registers a thread),
// but two where three would not fit in shared memory (four walkers per warp, lane blocks
// from 7)
__host__ __device__ constexpr int step_ctas(int tile, int R, bool psl = false)
{
    return 3 * 8 * (32 / tile) * step_smem(tile, R, psl).words * 4 <= kSmemBudget ? 3 : 2;
}

// Runs the walkers of the queue: the warp takes W consecutive walkers; when their lengths
// differ (a group boundary) or fewer are left, it runs them one after the other with the
// other lane groups idle.
template <class LG, class RT, int RMAX, bool PSL = false, bool BEST = false, bool AHEAD = false>
__device__ __forceinline__ void walk_group(const KParams& p, int chunk_index)
{
    constexpr int NL = LG::kSize, W = 32 / NL;
    using LAY = StepLayout<NL, RMAX, PSL>;
    constexpr StepSmem SL = LAY::SL;
    const int l = lane_id();
    const LG t(l);
    const RT tt(l);
    const int h = group_of(t);
    const int wb0 = (int)(threadIdx.x >> 5) * W * SL.words;
    const int wb = wb0 + h * SL.words;
    const int64_t target = p.status->target_steps;
    for (;;) {
        uint32_t q = 0;
        if (l == 0) q = atomicAdd(&p.queue[chunk_index], (uint32_t)W);
        q = __shfl_sync(kFull, q, 0);
        if ((int64_t)q >= p.W) break;
        const int64_t mine_w = (int64_t)q + h;
        const bool exists = mine_w < p.W;
        const int my_n = exists ? p.groups[p.states[mine_w].group].n : -1;
        const int n0 = __shfl_sync(kFull, my_n, 0);
        const bool together = __all_sync(kFull, exists && my_n == n0);
        const int passes = together ? 1 : (int)min((int64_t)W, p.W - (int64_t)q);
        for (int pass = 0; pass < passes; ++pass) {
            // together: every group runs its walker; else pass k runs group k alone
            const bool mine = exists && (together || pass == h);
            // the idle groups mirror the running group's length so that loops match (a group
            // past the last walker stands on the running group's state and table, idle)
            const int64_t lead_w = together ? mine_w : (int64_t)q + pass;
            const DevGroup G = p.groups[p.states[lead_w].group];
            StepEnv env;
            env.p = &p;
            env.g = (uint32_t)(exists ? mine_w : lead_w);
            env.T = p.tabu + ((uint64_t)env.g << p.tabu_log2);
            env.zk = p.zkeys + G.zkey_off;
            env.n = G.n;
            env.patience = p.patience > 0 ? p.patience : 2 * G.n;
            WalkerState* const st = env.state();
            StepWalker w;
            w.word = t.lane < kBitWords ? st->cur[t.lane] : 0u;
            w.fp = st->fp;
            w.isl = st->isl;
            w.best = st->best_isl;
            w.since = st->since_best;
            w.stag = st->stagnation;
            w.gen = st->gen;
            w.tisl = st->target_step < 0 ? target_isl(p, G.L) : -1;
            const int64_t steps0 = st->steps_done;
            const int len = (int)min((int64_t)p.chunk_steps, max(target - steps0, (int64_t)0));
            bool real = mine && len > 0;
            w.psl = w.best_psl = w.since_psl = 0;
            const int isl = step_build<LAY>(wb, w.word, G.L, G.n, t, &w.psl);
            if (PSL) {
                w.best_psl = st->best_psl;
                w.since_psl = st->since_psl;
            }
            if (real && (isl != w.isl || (PSL && w.psl != st->psl))) {
                if (t.lane == 0) raise_error(p.status, LABS_ESTATE, (int)mine_w);
                real = false;
            }
            unsigned extras = real && st->trace_slot >= 0 ? 1u : 0u;
            labs_log_record* rec = real ? step_record(p, mine_w, steps0) : nullptr;
            if (rec != nullptr) {
                extras |= 2u;
                if (t.lane < kBitWords) rec->bits[t.lane] = w.word;
                if (t.lane == 0) {
                    rec->isl = w.isl;
                    rec->L = G.L;
                    rec->walker = env.g;
                    rec->step = steps0;
                    rec->first = 0;
                    rec->min_isl = w.isl;
                }
            }
            // lane block: step_R(n) when it is one of RMAX .. RMAX-3, else the smallest
            // bank-conflict-free one of those
            int R = step_R(G.n, NL);
            if (R < RMAX - 3) R = conflict_free_R(RMAX - 3, NL);
            int done;
            if constexpr (BEST) {
                if (R >= RMAX)
                    done = walk_bestfirst<LAY, RMAX>(env, w, len, real, wb0, extras, t);
                else
                    done = walk_bestfirst<LAY, (RMAX > 2 ? RMAX - 2 : 1)>(env, w, len, real, wb0, extras, t);
            } else if constexpr (NL == 32) {  // lane blocks are odd
                if (R >= RMAX)
                    done = walk_lockstep<LAY, LG, RT, RMAX, AHEAD>(env, w, len, real, wb0, extras, t, tt);
                else
                    done = walk_lockstep<LAY, LG, RT, (RMAX > 2 ? RMAX - 2 : 1), AHEAD>(env, w, len, real, wb0, extras, t, tt);
            } else if (R >= RMAX)
                done = walk_lockstep<LAY, LG, RT, RMAX, AHEAD>(env, w, len, real, wb0, extras, t, tt);
            else if (R == RMAX - 1)
                done = walk_lockstep<LAY, LG, RT, (RMAX > 1 ? RMAX - 1 : 1), AHEAD>(env, w, len, real, wb0, extras, t, tt);
            else if (R == RMAX - 2)
                done = walk_lockstep<LAY, LG, RT, (RMAX > 2 ? RMAX - 2 : 1), AHEAD>(env, w, len, real, wb0, extras, t, tt);
            else
                done = walk_lockstep<LAY, LG, RT, (RMAX > 3 ? RMAX - 3 : 1), AHEAD>(env, w, len, real, wb0, extras, t, tt);
            if (real) {
                if (t.lane < kBitWords) st->cur[t.lane] = w.word;
                if (t.lane == 0) {
                    st->fp = w.fp;
                    st->isl = w.isl;
                    st->best_isl = w.best;
                    st->since_best = w.since;
                    st->stagnation = w.stag;
                    st->gen = w.gen;
                    st->steps_done = steps0 + done;
                    if (PSL) {
                        st->psl = w.psl;
                        st->best_psl = w.best_psl;
                        st->since_psl = w.since_psl;
                    }
                }
            }
            __syncwarp();
        }
    }
}

}  // namespace
}  // namespace labsgpu
