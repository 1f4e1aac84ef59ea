// labs_kernels.cu -- sm_103a kernels of the skew-symmetric LABS search
// (Brest & Boskovic, arXiv 2011.00068): walker starts, the ISL of rows, learned-proposal
// support, reductions and the launchers.  The walks themselves are in labs_step.cuh (the
// learned mode's in labs_device.cuh), instantiated by the labs_walk*.cu units, and in
// labs_long.cu; the row neighbourhoods and the network's inputs in labs_rows.cu.
#include <algorithm>

#include "labs_device.cuh"
#include "labs_launch.h"

namespace labsgpu {

namespace {

// Start of every walker (restart index 0, HT generation 1; HT zeroed by the caller).
__global__ void __launch_bounds__(512) reset_kernel(KParams p)
{
    extern __shared__ __align__(16) int smem[];
    const WarpSmem SL = warp_smem(p.n_max, 32);
    const Tile<32> t(threadIdx.x & 31);
    const int warp = threadIdx.x >> 5;
    int* base = smem + warp * SL.words;
    const View V = make_view(base, SL);
    const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t wi = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp; wi < p.W; wi += nwarps) {
        int gidx = 0;
        for (int g = 0; g < p.nG; ++g)
            if (wi >= p.groups[g].first && wi < p.groups[g].first + p.groups[g].count) gidx = g;
        const DevGroup G = p.groups[gidx];
        WalkerState* st = p.states + wi;
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
        env.slot = nullptr;
        env.slot_valid = nullptr;
        env.rdump = nullptr;
        env.rdump_idx = nullptr;
        env.rdump_count = nullptr;
        env.dump_cap = 0;
        Walker w;
        w.restart_idx = 0;
        w.gen = 1;
        w.restarts = w.overflows = w.blocked = 0;
        w.steps = 0;
        w.best_isl = INT_MAX;
        w.best_step = 0;
        w.target_step = -1;
        PslTrack ps;
        ps.best_psl = INT_MAX;
        start_walker(env, w, base, SL, V, t, false, p.mode == 3 ? &ps : nullptr);
        save_walker(st, w, t.lane);
        if (p.best_first) p.pq_key[wi * LABS_QUEUE_SIZE + t.lane] = ~0ull;  // empty queue
        if (t.lane == 0) {
            st->group = gidx;
            st->trace_slot = -1;
            st->psl = p.mode == 3 ? ps.psl : -1;
            st->best_psl = p.mode == 3 ? ps.best_psl : -1;
            st->since_psl = p.mode == 3 ? ps.since_psl : -1;
        }
        t.sync();
    }
}

__global__ void prep_walk_kernel(DevStatus* st, uint32_t* queue, int64_t steps, int nchunks)
{
    if (blockIdx.x == 0 && threadIdx.x == 0) st->target_steps += steps;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < nchunks; j += gridDim.x * blockDim.x)
        queue[j] = 0u;
}

__global__ void zobrist_kernel(uint64_t* zkeys, int64_t off, int L, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint32_t c0 = (uint32_t)i, c1 = (uint32_t)L, c2 = 0u, c3 = 2u;
    philox(c0, c1, c2, c3, kZobristKey0, kZobristKey1);
    zkeys[off + i] = (uint64_t)c0 | ((uint64_t)c1 << 32);
}

// --------------------------------------------------------- batch kernels (rows)

// Eq. 2 for arbitrary +-1 rows from bit vectors (bit u set <=> s_u = -1):
//   C_k = (L - k) - 2 #{u < L - k : s_u != s_{u+k}},
// the count by popcounts of the vector against itself shifted by k.  An ISL above INT32_MAX
// (long rows only) is reported as -2 with LABS_ERANGE.
//
// What bounds it: NW (NW + 1) / 2 words per lane and row (NW = ceil(L/32)), a popcount (16
// lanes per clock and SM), an XOR and an addition each.  From six words up three of them
// are added in carry-save form first (two popcounts for three), which moves work from the
// popcounts to the logic unit; from three words up measured slower (76 against 72 us), never
// (76 us) too.  2^18 rows of L = 255: 72 us (the sums of int products from 4-byte copies it
// replaces: 1507); L = 201 64, L = 511 238.
__device__ __forceinline__ void isl_store(int32_t* out, int64_t row, bool ok, long long isl, DevStatus* status)
{
    out[row] = !ok ? -1 : isl > INT_MAX ? -2 : (int32_t)isl;
    if (!ok && status) atomicAdd(&status->invalid_rows, 1);
    if (ok && isl > INT_MAX && status) raise_error(status, LABS_ERANGE, (int)row);
}

// Set bits of NWORDS words.
template <int NWORDS>
__device__ __forceinline__ int popc_sum(const uint32_t* w)
{
    if constexpr (NWORDS == 0) {
        return 0;
    } else if constexpr (NWORDS < 6) {
        return __popc(w[0]) + popc_sum<NWORDS - 1>(w + 1);
    } else {
        const uint32_t s = w[0] ^ w[1] ^ w[2], m = (w[0] & w[1]) | (w[2] & (w[0] | w[1]));
        return __popc(s) + 2 * __popc(m) + popc_sum<NWORDS - 3>(w + 3);
    }
}

template <int NW, int Q>
__device__ __forceinline__ int isl_lags(const uint32_t (&x)[NW], const uint32_t (&s)[NW], uint32_t mprev, uint32_t mlast,
                                        int L, int r)
{
    if constexpr (Q == NW) {
        return 0;
    } else {
        // lag 32 Q + r: word k against shifted word k + Q, the last two cut to the pairs
        // that exist
        constexpr int N = NW - Q;
        uint32_t w[N];
#pragma unroll
        for (int k = 0; k < N; ++k) {
            w[k] = x[k] ^ s[k + Q];
            if (k == N - 2) w[k] &= mprev;
            if (k == N - 1) w[k] &= mlast;
        }
        int c = L - 32 * Q - r;
        if constexpr (Q == NW - 1) c = max(c, 0);  // only here may a lane's lag lie past the row
        c -= 2 * popc_sum<N>(w);
        if (Q == 0 && r == 0) c = 0;  // lag 0 is not part of the ISL
        return c * c + isl_lags<NW, Q + 1>(x, s, mprev, mlast, L, r);
    }
}

// One warp per row, L <= 512: the row's NW = ceil(L/32) words in registers of every lane,
// lane r counts the lags 32 q + r.  C^2 sums below 2^31 for L <= 512.
template <int NW>
__global__ void __launch_bounds__(256) isl_kernel(const int8_t* __restrict__ seqs, int64_t batch, int L,
                                                  int32_t* __restrict__ out, DevStatus* status)
{
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    int64_t row = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int tail = L - 32 * (NW - 1), v = tail - lane;  // pairs of the last word (lag 32 q + lane)
    const uint32_t mlast = v <= 0 ? 0u : (v >= 32 ? ~0u : (1u << v) - 1u);
    const uint32_t mprev = v >= 0 ? ~0u : (1u << (32 + v)) - 1u;
    int b[NW];
    auto fetch = [&](int64_t r) {
        const int8_t* src = seqs + r * (int64_t)L;
#pragma unroll
        for (int k = 0; k < NW; ++k) b[k] = k < NW - 1 || lane < tail ? src[32 * k + lane] : 1;
    };
    if (row < batch) fetch(row);
    for (; row < batch; row += nwarps) {
        uint32_t x[NW], s[NW], bad = 0u;
#pragma unroll
        for (int k = 0; k < NW; ++k) {
            bad |= (uint32_t)(b[k] + 1) & ~2u;  // 0 exactly for 1 and -1
            x[k] = __ballot_sync(kFull, b[k] < 0);
        }
        const bool ok = !__any_sync(kFull, bad != 0u);
        if (row + nwarps < batch) fetch(row + nwarps);  // the next row's bytes land meanwhile
#pragma unroll
        for (int k = 0; k < NW; ++k) s[k] = __funnelshift_r(x[k], k + 1 < NW ? x[k + 1] : 0u, lane);
        int part = isl_lags<NW, 0>(x, s, mprev, mlast, L, lane);
        part = __reduce_add_sync(kFull, part);
        if (lane == 0) isl_store(out, row, ok, part, status);
    }
}

// One CTA per row, L > 512: the words in shared memory; each warp takes word shifts q from
// both ends of the range (a large and a small count of words), lane r the lags 32 q + r.
__global__ void __launch_bounds__(256) isl_long_kernel(const int8_t* __restrict__ seqs, int64_t batch, int L,
                                                       int32_t* __restrict__ out, DevStatus* status)
{
    __shared__ uint32_t x[(LABS_MAX_L_LONG + 31) / 32 + 2];
    __shared__ long long sums[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, NW = (L + 31) / 32;
    for (int64_t row = blockIdx.x; row < batch; row += gridDim.x) {
        const int8_t* src = seqs + row * (int64_t)L;
        bool bad = false;
        for (int k = warp; k < NW + 2; k += 8) {
            const int j = 32 * k + lane, v = j < L ? src[j] : 1;
            bad |= v != 1 && v != -1;
            const uint32_t w = __ballot_sync(kFull, v < 0);
            if (lane == 0) x[k] = w;
        }
        const bool ok = !__syncthreads_or(bad);
        long long part = 0;
        for (int i = warp; i < NW; i += 8) {
            // shifts in the order 0, NW-1, 1, NW-2, ..
            const int q = (i & 1) ? NW - 1 - (i >> 1) : i >> 1;
            const int m = 32 * q + lane, pairs = L - m;
            int cnt = 0;
            uint32_t lo = x[q];
            for (int k = 0; k < NW - q; ++k) {
                const uint32_t hi = x[k + q + 1];
                uint32_t w = x[k] ^ __funnelshift_r(lo, hi, lane);
                const int v = pairs - 32 * k;  // pairs of this word and beyond
                if (v < 32) w &= v > 0 ? (1u << v) - 1u : 0u;
                cnt += __popc(w);
                lo = hi;
            }
            if (m > 0 && m < L) {
                const long long c = pairs - 2 * cnt;
                part += c * c;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(kFull, part, o);
        if (lane == 0) sums[warp] = part;
        __syncthreads();
        if (threadIdx.x == 0) {
            long long t = 0;
            for (int w = 0; w < 8; ++w) t += sums[w];
            isl_store(out, row, ok, t, status);
        }
        __syncthreads();
    }
}

// --------------------------------------------------- learned proposal support

// Restart candidates of walkers [first, first+count) of one length: candidate 0 is the
// walker's own next random start (what the plain walk would use); candidates c >= 1 are
// further random starts, Philox with key = seed and counter = (walker, next restart
// index, block, c) laid out as start_word's.  (Perturbations of the walker's best state
// were tried as candidates instead: the walkers then crowd around their old optima and
// found worse sequences, best F 6.81 against 7.23 at L = 255.)  Output bits [count][P][8].
__global__ void candidates_kernel(KParams p, int64_t first, int64_t count, int n, int P, uint32_t* __restrict__ out)
{
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < count * P;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t w = first + t / P;
        const int c = (int)(t % P);
        const WalkerState& st = p.states[w];
        const uint32_t ridx = st.restart_idx + 1;
        uint32_t bits[kBitWords];
        if (c == 0) {
#pragma unroll
            for (int j = 0; j < kBitWords; ++j) bits[j] = start_word(p.seed, (uint32_t)w, ridx, j, n);
        } else {
#pragma unroll
            for (int j = 0; j < kBitWords; ++j) {
                uint32_t c0 = (uint32_t)w, c1 = ridx, c2 = (uint32_t)(j >> 2), c3 = (uint32_t)c;
                philox(c0, c1, c2, c3, (uint32_t)p.seed, (uint32_t)(p.seed >> 32));
                const uint32_t v = (j & 3) == 0 ? c0 : (j & 3) == 1 ? c1 : (j & 3) == 2 ? c2 : c3;
                const int lo = 32 * j;
                bits[j] = n <= lo ? 0u : (n - lo >= 32 ? v : v & ((1u << (n - lo)) - 1u));
            }
        }
#pragma unroll
        for (int j = 0; j < kBitWords; ++j) out[t * kBitWords + j] = bits[j];
    }
}

// Per walker: the candidate with the highest restart score (ties: lowest c) becomes the
// walker's proposed restart state.
__global__ void select_kernel(KParams p, int64_t first, int64_t count, int P, const float* __restrict__ score,
                              const uint32_t* __restrict__ cand)
{
    DevStatus* S = p.status;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < count; t += (int64_t)gridDim.x * blockDim.x) {
        int best = 0;
        for (int c = 1; c < P; ++c)
            if (score[t * P + c] > score[t * P + best]) best = c;
        const int64_t w = first + t;
#pragma unroll
        for (int j = 0; j < kBitWords; ++j) S->l_slot[w * kBitWords + j] = cand[(t * P + best) * kBitWords + j];
        S->l_slot_valid[w] = 1;
    }
}

// Flip scores of walkers [first, first+count) for their current step.
__global__ void scores_kernel(KParams p, int64_t first, int64_t count, int n, const float* __restrict__ score)
{
    DevStatus* S = p.status;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < count * n; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t w = first + t / n;
        const int i = (int)(t % n);
        S->l_scores[w * p.n_max + i] = score[t];
        if (i == 0) S->l_score_step[w] = p.states[w].steps_done;
    }
}

// Training labels of log records: target = the flip of the first step (0 when the step
// moved nowhere), wf = 1 when the ISL fell below the start ISL later in the chunk,
// y = L^2 / (2 min_isl) / 8 (the merit factor reached, scaled).
__global__ void labels_kernel(const labs_log_record* __restrict__ rec, int64_t count, int32_t* __restrict__ target,
                              float* __restrict__ y, float* __restrict__ wf)
{
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < count; t += (int64_t)gridDim.x * blockDim.x) {
        const labs_log_record r = rec[t];
        const bool moved = r.first >= 0;
        target[t] = moved ? (r.first & 0xFFFF) : 0;
        wf[t] = (moved && r.min_isl < r.isl) ? 1.f : 0.f;
        y[t] = (float)r.L * (float)r.L / (2.f * (float)r.min_isl) / 8.f;
    }
}

// ------------------------------------------------------------ reductions, tracing

// Objective of a walker's best sequence: its ISL, or (PSL << 32) | ISL under the PSL
// objective.
__device__ __forceinline__ unsigned long long best_objective(const KParams& p, const WalkerState& st)
{
    const unsigned long long isl = (uint32_t)st.best_isl;
    return p.mode == 3 ? ((unsigned long long)(uint32_t)st.best_psl << 32) | isl : isl;
}

// Lowest objective over the walkers of length L (0: all), into status->best_obj.
__global__ void best_obj_kernel(KParams p, int L)
{
    for (int64_t wi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; wi < p.W;
         wi += (int64_t)gridDim.x * blockDim.x) {
        const WalkerState& st = p.states[wi];
        if (L != 0 && p.groups[st.group].L != L) continue;
        atomicMin(&p.status->best_obj, best_objective(p, st));
    }
}

// Lowest (best ISL, walker); under the PSL objective only among the walkers whose
// objective equals status->best_obj (best_obj_kernel ran first).
__global__ void best_kernel(KParams p, int L)
{
    for (int64_t wi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; wi < p.W;
         wi += (int64_t)gridDim.x * blockDim.x) {
        const WalkerState& st = p.states[wi];
        if (L != 0 && p.groups[st.group].L != L) continue;
        if (p.mode == 3 && best_objective(p, st) != p.status->best_obj) continue;
        const unsigned long long key = ((unsigned long long)(uint32_t)st.best_isl << 32) |
                                       (unsigned long long)(uint32_t)wi;
        atomicMin(&p.status->best_key, key);
    }
}

__global__ void stats_kernel(KParams p, int L)
{
    for (int64_t wi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; wi < p.W;
         wi += (int64_t)gridDim.x * blockDim.x) {
        const WalkerState& st = p.states[wi];
        const DevGroup& G = p.groups[st.group];
        if (L != 0 && G.L != L) continue;
        DevStatus* s = p.status;
        atomicAdd(&s->st_steps, (unsigned long long)st.steps_done);
        atomicAdd(&s->st_evals, (unsigned long long)st.steps_done * (unsigned long long)G.n);
        atomicAdd(&s->st_restarts, (unsigned long long)st.restarts);
        atomicAdd(&s->st_overflows, (unsigned long long)st.overflows);
        atomicAdd(&s->st_blocked, (unsigned long long)st.blocked);
        atomicAdd(&s->st_cache_hits, (unsigned long long)st.cache_hits);
        if (st.target_step >= 0) {
            atomicAdd(&s->st_at_target, 1ull);
            atomicMin(&s->st_target_step, (long long)st.target_step);
        }
        if (p.mode == 3) {
            atomicMin(&s->best_obj, best_objective(p, st));
            continue;
        }
        const unsigned long long key = ((unsigned long long)(uint32_t)st.best_isl << 32) |
                                       (unsigned long long)(uint32_t)wi;
        atomicMin(&s->best_key, key);
    }
}

__global__ void trace_clear_kernel(KParams p)
{
    for (int64_t wi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; wi < p.W;
         wi += (int64_t)gridDim.x * blockDim.x)
        p.states[wi].trace_slot = -1;
}

__global__ void trace_set_kernel(KParams p, const int64_t* ids, int k, int32_t* code, int32_t* isl,
                                 int64_t capacity)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j == 0) {
        p.status->trace_code = code;
        p.status->trace_isl = isl;
        p.status->trace_capacity = capacity;
    }
    if (j < k) {
        const int64_t wi = ids[j];
        p.states[wi].trace_slot = j;
        p.trace_start[j] = p.states[wi].steps_done;
    }
}

__global__ void time_probe_kernel(unsigned long long* out)
{
    *out = global_ns();
}

int status_of(cudaError_t e)
{
    return e == cudaSuccess ? LABS_OK : LABS_ECUDA;
}

}  // namespace

// ------------------------------------------------------------------- launchers

int launch_zobrist(const KParams&, uint64_t* zkeys, const DevGroup* host_groups, int nG, void* stream)
{
    for (int g = 0; g < nG; ++g) {
        const DevGroup& G = host_groups[g];
        zobrist_kernel<<<(G.n + 127) / 128, 128, 0, (cudaStream_t)stream>>>(zkeys, G.zkey_off, G.L, G.n);
    }
    return status_of(cudaGetLastError());
}

int launch_reset(const KParams& p, int grid, int block, void* stream)
{
    const size_t smem = (size_t)(block / kWarp) * warp_smem(p.n_max, 32).words * sizeof(int);
    if (allow_shared((const void*)reset_kernel) != cudaSuccess) return LABS_ECUDA;
    reset_kernel<<<grid, block, smem, (cudaStream_t)stream>>>(p);
    return status_of(cudaGetLastError());
}

int launch_prep_walk(const KParams& p, int64_t steps, int nchunks, void* stream)
{
    prep_walk_kernel<<<(nchunks + 255) / 256, 256, 0, (cudaStream_t)stream>>>(p.status, p.queue, steps,
                                                                              nchunks);
    return status_of(cudaGetLastError());
}

static WalkFn walk_fn(int tile, int rmax, int mode)
{
    if (mode == 4) return tile == 8 ? walk_fn8f(rmax) : tile == 16 ? walk_fn16f(rmax) : walk_fn32f(rmax);
    if (tile == 8) return rmax <= 6 ? walk_fn8a(rmax) : walk_fn8b(rmax);
    if (tile == 16 && mode == 3) return rmax <= 5 ? walk_fn16p(rmax) : walk_fn16q(rmax);
    if (tile == 16) return rmax <= 5 ? walk_fn16a(rmax) : walk_fn16b(rmax);
    switch (mode) {
        case 1: return walk_fn32l(rmax);
        case 2: return walk_fn32b(rmax);
        case 3: return walk_fn32p(rmax);
        default: return walk_fn32(rmax);
    }
}

// Lane block and shared memory per warp of a walk kernel (mode 1: the learned mode, 4: the
// plain walk's kernels for few walkers).
static int walk_R(int n_max, int tile, int mode)
{
    return mode != 1 ? step_R(n_max, tile) : block_R(n_max, tile);
}

static size_t walk_warp_bytes(int n_max, int tile, int mode)
{
    const int words = mode != 1 ? step_smem(tile, step_R(n_max, tile), mode == 3).words : warp_smem(n_max, tile).words;
    return (size_t)words * sizeof(int) * (kWarp / tile);
}

int walk_kernel_config(int n_max, int tile, int mode, int warps_per_cta, int* ctas_per_sm, int* regs)
{
    const WalkFn fn = walk_fn(tile, walk_R(n_max, tile, mode), mode);
    const size_t smem_bytes = walk_warp_bytes(n_max, tile, mode) * (size_t)warps_per_cta;
    int dev = 0, most = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return LABS_ECUDA;
    *ctas_per_sm = 0;
    if (smem_bytes > (size_t)most) return LABS_EINVAL;
    cudaFuncAttributes fa;
    if (allow_shared((const void*)fn, &fa) != cudaSuccess) return LABS_ECUDA;
    if (regs) *regs = fa.numRegs;
    if (warps_per_cta * kWarp > fa.maxThreadsPerBlock) return LABS_EINVAL;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, fn, warps_per_cta * kWarp, smem_bytes);
    return status_of(e);
}

int launch_walk_chunk(const KParams& p, int chunk_index, int grid, int warps_per_cta, void* stream)
{
    const WalkFn fn = walk_fn(p.tile, walk_R(p.n_max, p.tile, p.mode), p.mode == 0 && p.ahead ? 4 : p.mode);
    const size_t smem_bytes = walk_warp_bytes(p.n_max, p.tile, p.mode) * (size_t)warps_per_cta;
    fn<<<grid, warps_per_cta * kWarp, smem_bytes, (cudaStream_t)stream>>>(p, chunk_index);
    return status_of(cudaGetLastError());
}

static int row_grid(int64_t batch, int warps)
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    int64_t need = (batch + warps - 1) / warps;
    int64_t cap = (int64_t)sms * 8;
    return (int)(need < cap ? need : cap);
}

template <int NW>
static void launch_isl_words(int nw, const int8_t* seqs, int64_t batch, int32_t L, int32_t* out, DevStatus* status,
                             cudaStream_t s)
{
    if constexpr (NW <= 16) {
        if (nw == NW)
            isl_kernel<NW><<<row_grid(batch, 8), 256, 0, s>>>(seqs, batch, L, out, status);
        else
            launch_isl_words<NW + 1>(nw, seqs, batch, L, out, status, s);
    }
}

int launch_isl(const int8_t* seqs, int64_t batch, int32_t L, int32_t* out, DevStatus* status, void* stream)
{
    if (batch == 0) return LABS_OK;
    if (L <= 512)
        launch_isl_words<1>((L + 31) / 32, seqs, batch, L, out, status, (cudaStream_t)stream);
    else
        isl_long_kernel<<<row_grid(batch, 1), 256, 0, (cudaStream_t)stream>>>(seqs, batch, L, out, status);
    return status_of(cudaGetLastError());
}

int launch_best(const KParams& p, int32_t L, void* stream)
{
    if (p.mode == 3) best_obj_kernel<<<256, 256, 0, (cudaStream_t)stream>>>(p, L);
    best_kernel<<<256, 256, 0, (cudaStream_t)stream>>>(p, L);
    return status_of(cudaGetLastError());
}

int launch_stats(const KParams& p, int32_t L, void* stream)
{
    stats_kernel<<<256, 256, 0, (cudaStream_t)stream>>>(p, L);
    if (p.mode == 3) best_kernel<<<256, 256, 0, (cudaStream_t)stream>>>(p, L);
    return status_of(cudaGetLastError());
}

int launch_trace_arm(const KParams& p, const int64_t* dev_ids, int32_t k, int32_t* code, int32_t* isl,
                     int64_t capacity, void* stream)
{
    trace_clear_kernel<<<256, 256, 0, (cudaStream_t)stream>>>(p);
    trace_set_kernel<<<(k + 255) / 256 + 1, 256, 0, (cudaStream_t)stream>>>(p, dev_ids, k, code, isl, capacity);
    return status_of(cudaGetLastError());
}

int launch_candidates(const KParams& p, int64_t first, int64_t count, int n, int P, uint32_t* out, void* stream)
{
    candidates_kernel<<<256, 256, 0, (cudaStream_t)stream>>>(p, first, count, n, P, out);
    return status_of(cudaGetLastError());
}

int launch_select(const KParams& p, int64_t first, int64_t count, int P, const float* score, const uint32_t* cand,
                  void* stream)
{
    select_kernel<<<256, 256, 0, (cudaStream_t)stream>>>(p, first, count, P, score, cand);
    return status_of(cudaGetLastError());
}

int launch_scores(const KParams& p, int64_t first, int64_t count, int n, const float* score, void* stream)
{
    scores_kernel<<<256, 256, 0, (cudaStream_t)stream>>>(p, first, count, n, score);
    return status_of(cudaGetLastError());
}

int launch_labels(const labs_log_record* rec, int64_t count, int32_t* target, float* y, float* wf, void* stream)
{
    labels_kernel<<<256, 256, 0, (cudaStream_t)stream>>>(rec, count, target, y, wf);
    return status_of(cudaGetLastError());
}

int launch_time_probe(unsigned long long* dev_out, void* stream)
{
    time_probe_kernel<<<1, 1, 0, (cudaStream_t)stream>>>(dev_out);
    return status_of(cudaGetLastError());
}

}  // namespace labsgpu
