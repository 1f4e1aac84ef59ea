// labs_enum.cu -- exhaustive search over skew-symmetric sequences of short odd length
// (L <= 63), the exact counterpart of the stochastic search for small L.
//
// The centre is fixed to s_c = +1 (negating a whole sequence keeps Eq. 4 and the ISL).
// Assignment a sets free variable i (i < c) to -1 when bit i of a is set.
//
// Every assignment's even-lag C_k come from bit vectors of its two parity classes.  Class p
// (n_p = n - p entries) is a palindrome or an antipalindrome (Eq. 4), a_{n_p-1-u} = sg_p a_u,
// so the pairs (u, u+m) of lag m repeat from both ends: with h = floor((n_p - m) / 2) pairs
// counted and d of them unequal, C^(p)_m = 2 h - 4 d, plus sg_p when n_p - m is odd (the
// middle pair).  h <= 16 for L <= 63: both classes' pairs share one 32-bit word and one
// popcount, and C_{2m} is a constant of the lag minus 4 popcounts.  The ISL (Eq. 2) is the
// sum of the squares (odd lags vanish).
//
// What bounds it: about 8 integer instructions per assignment and lag.  A thread takes its
// 2^low consecutive assignments kEnumLanes at a time, so that a lag's masks and constant
// are computed once for all of them.  The partial results are reduced by trees of one CTA
// each (one thread reading 1024 of them took 270 us).  L = 41: the two kernels take about
// 10 us of the call (333 before).
#include <cuda_runtime.h>

#include <climits>
#include <cstdint>
#include <mutex>

#include "labs_internal.cuh"
#include "labs_nvtx.h"

namespace labsgpu {

namespace {

constexpr int kEnumThreads = 128;
constexpr int kEnumMaxHighBits = 17;

__host__ __device__ inline int enum_low_bits(int free_bits)
{
    return free_bits > kEnumMaxHighBits ? free_bits - kEnumMaxHighBits : 0;
}

// Every second bit of a, from bit 0, packed.
__device__ __forceinline__ uint32_t even_bits(uint32_t a)
{
    a &= 0x55555555u;
    a = (a | (a >> 1)) & 0x33333333u;
    a = (a | (a >> 2)) & 0x0F0F0F0Fu;
    a = (a | (a >> 4)) & 0x00FF00FFu;
    return (a | (a >> 8)) & 0x0000FFFFu;
}

__device__ __forceinline__ uint32_t low_mask(int bits)  // 0 <= bits <= 32
{
    return bits >= 32 ? ~0u : (1u << bits) - 1u;
}

// Bit vector of class p of assignment a: free variables 2v + p, then their mirrors.
__device__ __forceinline__ uint32_t class_bits(uint32_t a, int n, int p)
{
    const int c = n - 1, np = n - p, nv = p ? n >> 1 : (n + 1) >> 1;  // nv entries are free (or the centre)
    const uint32_t lo = even_bits(a >> p) & low_mask(nv);
    uint32_t rev = __brev(lo) >> (32 - np);                           // entry np-1-u for entry u
    if ((c + p) & 1) rev = ~rev;                                      // antipalindrome
    return lo | (rev & low_mask(np) & ~low_mask(nv));
}

struct EnumBest {
    int isl;
    uint32_t first;
    unsigned long long count;
};

__device__ __forceinline__ void enum_take(EnumBest& b, int isl, uint32_t first, unsigned long long count)
{
    if (count == 0 || isl > b.isl) return;
    if (isl < b.isl) {
        b.isl = isl;
        b.count = 0;
        b.first = first;
    }
    b.count += count;
    b.first = min(b.first, first);
}

// Adds the whole CTA's results into thread 0's.
template <int THREADS>
__device__ __forceinline__ EnumBest enum_block_best(EnumBest b)
{
    __shared__ EnumBest sh[THREADS];
    sh[threadIdx.x] = b;
    for (int h = THREADS / 2; h > 0; h >>= 1) {
        __syncthreads();
        if ((int)threadIdx.x < h) {
            const EnumBest o = sh[threadIdx.x + h];
            enum_take(b, o.isl, o.first, o.count);
            sh[threadIdx.x] = b;
        }
    }
    return b;
}

// ISLs of the K assignments a0 .. a0+K-1.  (ISL <= sum of squares below 63: 2^17.)
template <int K>
__device__ __forceinline__ void enum_eval(uint32_t a0, int n, EnumBest& best)
{
    const int c = n - 1;
    uint32_t x0[K], x1[K];
    int isl[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        x0[k] = class_bits(a0 + k, n, 0);
        x1[k] = class_bits(a0 + k, n, 1);
        isl[k] = 0;
    }
    const int g0 = (c & 1) ? -1 : 1;  // sg of class 0; class 1 has the other sign
    for (int m = 1; m < n; ++m) {
        const int q0 = n - m, q1 = n - 1 - m, h0 = q0 >> 1, h1 = q1 >> 1;
        const uint32_t m0 = low_mask(h0), m1 = low_mask(h1);
        const int base = 2 * (h0 + h1) + ((q0 & 1) ? g0 : 0) + ((q1 & 1) ? -g0 : 0);
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const uint32_t d0 = (x0[k] ^ (x0[k] >> m)) & m0, d1 = (x1[k] ^ (x1[k] >> m)) & m1;
            const int cm = base - 4 * __popc(d0 | (d1 << 16));
            isl[k] += cm * cm;
        }
    }
#pragma unroll
    for (int k = 0; k < K; ++k) enum_take(best, isl[k], a0 + k, 1ull);
}

constexpr int kEnumLanes = 8;

__global__ void __launch_bounds__(kEnumThreads) enum_kernel(int L, EnumPart* parts)
{
    const int n = (L + 1) / 2, T = n - 1, low = enum_low_bits(T);
    const uint32_t high = blockIdx.x * kEnumThreads + threadIdx.x;
    EnumBest best{INT_MAX, ~0u, 0ull};
    if (high < (1u << (T - low))) {
        const uint32_t a0 = high << low;
        if (low >= 3) {
            for (uint32_t t = 0; t < (1u << low); t += kEnumLanes) enum_eval<kEnumLanes>(a0 + t, n, best);
        } else {
            for (uint32_t t = 0; t < (1u << low); ++t) enum_eval<1>(a0 + t, n, best);
        }
    }
    best = enum_block_best<kEnumThreads>(best);
    if (threadIdx.x == 0) {
        parts[blockIdx.x].min_isl = best.isl;
        parts[blockIdx.x].count = best.count;
        parts[blockIdx.x].first = best.first;
    }
}

constexpr int kEnumReduceThreads = 256;

__global__ void __launch_bounds__(kEnumReduceThreads) enum_reduce_kernel(const EnumPart* parts, int nparts, EnumPart* out)
{
    EnumBest best{INT_MAX, ~0u, 0ull};
    for (int t = threadIdx.x; t < nparts; t += kEnumReduceThreads)
        enum_take(best, (int)parts[t].min_isl, (uint32_t)parts[t].first, parts[t].count);
    best = enum_block_best<kEnumReduceThreads>(best);
    if (threadIdx.x == 0) {
        out->min_isl = best.isl;
        out->count = best.count;
        out->first = best.first;
    }
}

}  // namespace

int enum_blocks(int L)
{
    const int n = (L + 1) / 2;
    const int T = n - 1;
    const uint64_t nhigh = 1ull << (T - enum_low_bits(T));
    return (int)((nhigh + kEnumThreads - 1) / kEnumThreads);
}

// Scratch: one EnumPart per block plus the final result.
size_t enum_scratch_bytes(int L)
{
    return sizeof(EnumPart) * (size_t)(enum_blocks(L) + 1);
}

int enum_run(int L, EnumPart* scratch, void* stream, EnumPart* host_out)
{
    const int blocks = enum_blocks(L);
    cudaStream_t s = (cudaStream_t)stream;
    enum_kernel<<<blocks, kEnumThreads, 0, s>>>(L, scratch);
    enum_reduce_kernel<<<1, kEnumReduceThreads, 0, s>>>(scratch, blocks, scratch + blocks);
    if (cudaGetLastError() != cudaSuccess) return LABS_ECUDA;
    if (cudaMemcpyAsync(host_out, scratch + blocks, sizeof(EnumPart), cudaMemcpyDeviceToHost, s) != cudaSuccess)
        return LABS_ECUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return LABS_ECUDA;
    return LABS_OK;
}

// ------------------------------------------------ allocation-free variant
//
// labs_enumerate_noalloc runs the same two kernels with their scratch (the per-block
// partial results and the final result) in the file-scope array below instead of a
// caller buffer.  The array is part of the library image: every GPU that loads the
// library holds its kNoAllocParts * 32 bytes (33,280 bytes) until the process exits.
// Host code cannot use the array's name as a device address, so the first call on
// each device looks the address up with cudaGetSymbolAddress (with that device
// current) and keeps it per device.  A device reset (cudaDeviceReset) unloads the
// module and invalidates a kept address: a call whose CUDA work fails drops the kept
// address of its device, and the next call looks it up again.
constexpr int kNoAllocParts = 1040;  // enum_blocks(63) + 1 = 1025 fit
constexpr int kNoAllocDevices = 64;
static __device__ __align__(256) EnumPart g_noalloc_scratch[kNoAllocParts];

namespace {
std::mutex g_noalloc_mutex;
EnumPart* g_noalloc_addr[kNoAllocDevices] = {};
}  // namespace

}  // namespace labsgpu

extern "C" int labs_enumerate_noalloc(int32_t L, int64_t* min_isl, uint64_t* count, uint64_t* first_assignment,
                                      void* cuda_stream)
{
    LABS_API_RANGE();
    using namespace labsgpu;
    if (L < 3 || L > 63 || (L & 1) == 0) return LABS_EINVAL;
    const int blocks = enum_blocks(L);
    if (blocks + 1 > kNoAllocParts) return LABS_ENOMEM;  // needs more scratch than the static array holds
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return LABS_ECUDA;
    if (dev < 0 || dev >= kNoAllocDevices) return LABS_EINVAL;
    EnumPart* scratch = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_noalloc_mutex);
        if (g_noalloc_addr[dev] == nullptr) {
            void* addr = nullptr;
            if (cudaGetSymbolAddress(&addr, g_noalloc_scratch) != cudaSuccess || addr == nullptr) return LABS_ECUDA;
            g_noalloc_addr[dev] = static_cast<EnumPart*>(addr);
        }
        scratch = g_noalloc_addr[dev];
    }
    auto forget = [dev]() {
        std::lock_guard<std::mutex> lock(g_noalloc_mutex);
        g_noalloc_addr[dev] = nullptr;
    };
    // The array keeps the previous call's contents; clear the part this call uses.
    cudaStream_t s = (cudaStream_t)cuda_stream;
    if (cudaMemsetAsync(scratch, 0, sizeof(EnumPart) * (size_t)(blocks + 1), s) != cudaSuccess) {
        forget();
        return LABS_ECUDA;
    }
    EnumPart r;
    const int rc = enum_run(L, scratch, cuda_stream, &r);
    if (rc) {
        if (rc == LABS_ECUDA) forget();
        return rc;
    }
    if (min_isl) *min_isl = r.min_isl;
    if (count) *count = r.count;
    if (first_assignment) *first_assignment = r.first;
    return LABS_OK;
}
