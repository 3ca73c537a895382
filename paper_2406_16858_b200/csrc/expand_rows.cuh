// Expansion of rows whose logits a thread-block cluster can hold in registers (included by expand.cu).
//
// A cluster of up to eight blocks serves one row: every thread loads its 16 to 64 logits at once, the block
// takes their softmax sum and its k best keys from registers, and the blocks' keys and sums meet in the first
// block's shared memory, which ranks the row's children and writes the tree level.  The last row of a sequence
// to finish ranks the next frontier.  Against a list of partials per tile in global memory, merged by the last
// block to arrive, that leaves one global hand-over of k numbers per row where there were two of k keys per tile,
// and the rows of a step are merged side by side.
//
// What bounds it: at one sequence the chain load - sums - candidates - cluster barrier - row - ticket - frontier,
// with many rows the logits' way from memory (64 KB in flight per block, two blocks per SM).
#pragma once

#include <cooperative_groups.h>

namespace eagle2 {

constexpr int kRowThreads = 256;
constexpr int kRowWarps = kRowThreads / kWarp;
constexpr int kRowMaxCluster = 8;
constexpr int kRowGroups = 32;   // groups of eight threads, whose maxima give the bar
static_assert(kRowGroups * 8 == kRowThreads && EAGLE2_MAX_K <= kRowGroups, "the bar is one of the groups' maxima");
constexpr int kRowCand = 512;  // candidates a block ranks; more (ties, rows of -inf) go through exact selection

// How many of n keys are above `mine`; W neighbouring lanes share the comparisons (all of them get the count).
template <int W>
__device__ __forceinline__ int count_above(const unsigned long long* keys, int n, unsigned long long mine) {
    int c = 0;
#pragma unroll 8
    for (int j = threadIdx.x & (W - 1); j < n; j += W) c += keys[j] > mine;
#pragma unroll
    for (int o = 1; o < W; o <<= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    return c;
}

// 2^d for a whole d <= 0 (0 below the smallest normal number; NaN stays), exactly
__device__ __forceinline__ float pow2_whole(float d) { return d >= -126.f ? __int_as_float(((int)d + 127) << 23) : d * 0.f; }

// The node a row belongs to and its value; a frontier entry outside the level before is reported.
__device__ __forceinline__ int parent_of_row(const int32_t* frontier, const double* tree_value, int b, int row, int k, int s, long long N,
                                             int* parent, double* value) {
    const long long prev_base = s >= 2 ? (long long)k + (long long)(s - 2) * k * k : 0;
    const long long prev_count = s >= 2 ? (long long)k * k : k;
    *parent = frontier[(long long)b * k + row];
    if (*parent < prev_base || *parent >= prev_base + prev_count) {
        *parent = (int)prev_base;
        return EAGLE2_STATUS_BAD_TREE;
    }
    *value = tree_value[(long long)b * N + *parent];
    return 0;
}

// Writes the children of a row whose k best keys (0: none) and log-sum-exp are known to the block; the block of a
// sequence that does so last ranks the next frontier.
__device__ __forceinline__ void hand_on_row(const unsigned long long* s_row, double lse, int parent, double parent_value, int b, int row, int k,
                                            int n_s, long long N, long long base, int by_confidence, int32_t* tree_token,
                                            int32_t* tree_parent, double* tree_value, int32_t* frontier, int* counters,
                                            unsigned long long* codes, unsigned long long* s_code, int* s_flag, int status,
                                            int32_t* d_status) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // A lane per child: what the row hands on is written by one warp, whose first lane announces it without another
    // meeting of the block.
    if (tid < k && s_row[tid]) {
        const long long at = (long long)b * N + base + (long long)row * k + tid;
        const double confidence = (double)key_value(s_row[tid]) - lse;  // log c_i
        const double v = parent_value + confidence;
        tree_token[at] = (int32_t)key_index(s_row[tid]);
        tree_parent[at] = parent;
        tree_value[at] = v;
        // the next frontier is ranked by value, or by confidence alone in the ablation
        if (n_s > 1) codes[((size_t)b * n_s + row) * k + tid] = order_code_f64(by_confidence ? confidence : v);
    }
    if (n_s == 1 && tid < k) frontier[(long long)b * k + tid] = (int32_t)(base + tid);  // a row's children are in order
    if (status) raise_status(d_status, status);
    if (n_s == 1) return;

    // ---- last row of the sequence: the next frontier, by (value desc, index asc) ----------------------------
    const int n_new = n_s * k;
    if (warp == 0) {
        __syncwarp();
        if (lane == 0) {
            __threadfence();  // cumulative: covers the stores of the warp's other lanes
            *s_flag = atomicAdd(counters + b, 1) == n_s - 1;
            if (*s_flag) counters[b] = 0;
        }
    }
    __syncthreads();
    if (!*s_flag) return;
    __threadfence();
    for (int i = tid; i < n_new; i += kRowThreads) s_code[i] = __ldcg(codes + (size_t)b * n_new + i);
    __syncthreads();
    for (int i = tid >> 1; i < (n_new + 15 & ~15); i += kRowThreads / 2) {  // two threads a candidate
        const unsigned long long ci = i < n_new ? s_code[i] : 0ull;
        int place = 0;
#pragma unroll 8
        for (int j = tid & 1; j < n_new; j += 2) {
            const unsigned long long cj = s_code[j];
            place += (cj > ci) || (cj == ci && j < i);
        }
        place += __shfl_xor_sync(0xffffffffu, place, 1);
        if ((tid & 1) == 0 && i < n_new && place < k) frontier[(long long)b * k + place] = (int32_t)(base + i);
    }
}

template <int NF, bool VEC>
__global__ void __launch_bounds__(kRowThreads, NF == 16 ? 2 : 3)
expand_rows_kernel(const float* __restrict__ draft_logits, long long batch_stride, int V, int k, int D, int s, int n_s,
                   int by_confidence, int32_t* __restrict__ tree_token, int32_t* __restrict__ tree_parent,
                   double* __restrict__ tree_value, int32_t* __restrict__ frontier, int* __restrict__ counters,
                   unsigned long long* __restrict__ codes, int32_t* d_status) {
    namespace cg = cooperative_groups;
    constexpr int NE = 4 * NF, kSlice = kRowThreads * NE;
    constexpr float kLog2e = 1.4426950408889634f;
    cg::cluster_group cluster = cg::this_cluster();
    const int cs = (int)cluster.num_blocks(), me = (int)cluster.block_rank();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    __shared__ unsigned long long s_cand[kRowCand];
    __shared__ unsigned long long s_in[kRowMaxCluster * EAGLE2_MAX_K];  // first block: every block's k best
    __shared__ float2 s_stats[kRowMaxCluster];                          // first block: every block's (reference, sum)
    __shared__ unsigned long long s_row[EAGLE2_MAX_K];                  // first block: the row's k best
    __shared__ unsigned long long s_best[kRowWarps], s_code[EAGLE2_MAX_K * EAGLE2_MAX_K];
    __shared__ float s_wref[kRowWarps], s_wsum[kRowWarps];
    __shared__ __align__(16) float s_top[kRowGroups];
    __shared__ int s_n, s_flag;
    __shared__ double s_lse;

    if (cs > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");  // (waited for before the first remote store)
    if (tid == 0) s_n = 0;
    if (tid < k) s_row[tid] = 0ull;
    const int line = blockIdx.x / cs, row = line % n_s, b = line / n_s;
    const float* z = draft_logits + (long long)b * batch_stride + (long long)row * V;
    const int lo = me * kSlice;
    auto token_of = [&](int j) { return lo + (VEC ? ((j >> 2) * kRowThreads + tid) * 4 + (j & 3) : j * kRowThreads + tid); };
    chain_wait();
    chain_release();
    float x[NE];
    if (VEC) {
#pragma unroll
        for (int i = 0; i < NF; ++i) {
            const int e = token_of(4 * i);
            float4 v = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
            if (e < V) v = __ldcs(reinterpret_cast<const float4*>(z + e));
            x[4 * i] = v.x, x[4 * i + 1] = v.y, x[4 * i + 2] = v.z, x[4 * i + 3] = v.w;
        }
    } else {
#pragma unroll
        for (int j = 0; j < NE; ++j) {
            const int e = token_of(j);
            x[j] = e < V ? __ldcs(z + e) : -INFINITY;
        }
    }
    // the row's node and its value, needed when the row is complete
    const long long N = nodes_of(k, D);
    const long long base = s ? (long long)k + (long long)(s - 1) * k * k : 0;
    int parent = -1, status = 0;
    double parent_value = 0.0;
    if (s && me == 0) status |= parent_of_row(frontier, tree_value, b, row, k, s, N, &parent, &parent_value);

    // ---- maxima --------------------------------------------------------------------------
    float gm[NF];  // of four elements each
#pragma unroll
    for (int i = 0; i < NF; ++i) gm[i] = fmaxf(fmaxf(x[4 * i], x[4 * i + 1]), fmaxf(x[4 * i + 2], x[4 * i + 3]));
    float tm = gm[0];
#pragma unroll
    for (int i = 1; i < NF; ++i) tm = fmaxf(tm, gm[i]);
    float um = tm;  // of eight threads
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) um = fmaxf(um, __shfl_xor_sync(0xffffffffu, um, o));
    if ((lane & 7) == 0) s_top[tid >> 3] = um;
    float wmax = fmaxf(um, __shfl_xor_sync(0xffffffffu, um, 8));
    wmax = fmaxf(wmax, __shfl_xor_sync(0xffffffffu, wmax, 16));

    // ---- the sum of exponentials -----------------------------------------------------------------------
    // Relative to the warp's maximum in base 2, rounded up to a whole number: factors between references are exact.
    float wref = ceilf(wmax * kLog2e);
    float part[4] = {0.f, 0.f, 0.f, 0.f};
    if (fabsf(wmax) < kFarLogit) {
        const float2 scale2 = make_float2(kLog2e, kLog2e), neg2 = make_float2(-wref, -wref);
#pragma unroll
        for (int j = 0; j < NE; j += 2) {
            const float2 a = __ffma2_rn(make_float2(x[j], x[j + 1]), scale2, neg2);
            part[j & 2] += fast_ex2(a.x), part[(j & 2) + 1] += fast_ex2(a.y);
        }
    } else {
        wref = -INFINITY;
#pragma unroll
        for (int j = 0; j < NE; ++j)
            if (x[j] != x[j]) part[0] = x[j];  // a NaN is seen all the same
    }
    const float wsum = warp_sum_f32((part[0] + part[1]) + (part[2] + part[3]));
    if (lane == 0) {
        s_wref[warp] = wref, s_wsum[warp] = wsum;
        if (!(wsum == wsum) || wmax == INFINITY) status |= EAGLE2_STATUS_NONFINITE_LOGIT;
    }
    __syncthreads();

    // ---- the bar ------------------------------------------------------------------------------------------
    // The k-th largest of the 32 groups' maxima is a value that k elements reach: so does the block's k-th best, and
    // about 32 ln(32 / (32 - k)) elements do (12 for k = 10).  Every warp works it out for itself.  (The k-th of the
    // threads' maxima leaves 10, but takes a sort per warp and another meeting of the block: 0.7 us of a call's 8.)
    float bar;
    {
        const float mine = s_top[lane];
        int above = 0;
#pragma unroll
        for (int j = 0; j < kRowGroups; j += 4) {
            const float4 t = *reinterpret_cast<const float4*>(s_top + j);
            above += (t.x > mine) + (t.y > mine) + (t.z > mine) + (t.w > mine);
        }
        bar = order_decode(__reduce_min_sync(0xffffffffu, above < k ? order_code(mine) : ~0u));
    }

    // ---- the block's candidates ------------------------------------------------------------------------
    if (tm >= bar) {
#pragma unroll
        for (int i = 0; i < NF; ++i) {
            if (!(gm[i] >= bar)) continue;
            int c = 0;
#pragma unroll
            for (int e = 0; e < 4; ++e) c += x[4 * i + e] >= bar && token_of(4 * i + e) < V;
            int at = atomicAdd(&s_n, c);
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (x[4 * i + e] >= bar && token_of(4 * i + e) < V) {
                    if (at < kRowCand) s_cand[at] = make_key(x[4 * i + e], (uint32_t)token_of(4 * i + e));
                    ++at;
                }
        }
    }
    __syncthreads();
    int n = s_n;
    if (n > kRowCand) {
        // exact: k times the largest key below the last one taken
        unsigned long long last = ~0ull;
        for (int r = 0; r < k; ++r) {
            unsigned long long best = 0ull;
#pragma unroll
            for (int j = 0; j < NE; ++j) {
                const int e = token_of(j);
                const unsigned long long key = e < V ? make_key(x[j], (uint32_t)e) : 0ull;
                best = key < last && key > best ? key : best;
            }
            best = warp_max_u64(best);
            if (lane == 0) s_best[warp] = best;
            __syncthreads();
            best = 0ull;
#pragma unroll
            for (int w = 0; w < kRowWarps; ++w) best = s_best[w] > best ? s_best[w] : best;
            if (tid == 0) s_cand[r] = best;
            last = best;
            __syncthreads();
            if (best == 0ull) break;
        }
        n = k;
        __syncthreads();
    }
    // ranked by counting (keys differ); straight into the first block's memory
    if (cs > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    unsigned long long* to = cs > 1 ? cluster.map_shared_rank(s_in, 0) : s_in;
    for (int i = tid >> 2; i < (n + 7 & ~7); i += kRowThreads / 4) {  // four threads share a key's comparisons
        const unsigned long long mine = i < n ? s_cand[i] : 0ull;
        const int rank = count_above<4>(s_cand, n, mine);
        if ((tid & 3) == 0 && rank < k && mine) to[me * k + rank] = mine;
    }
    if (tid >= n && tid < k) to[me * k + tid] = 0ull;
    if (warp == kRowWarps - 1) {
        const float ref = lane < kRowWarps ? s_wref[lane] : -INFINITY;
        const float cref = warp_max_f32(ref);
        const float csum = warp_sum_f32(ref > -INFINITY ? s_wsum[lane] * pow2_whole(ref - cref) : 0.f);
        if (lane == 0) {
            float2* st = cs > 1 ? cluster.map_shared_rank(s_stats, 0) : s_stats;
            st[me] = make_float2(cref, csum);
        }
    }
    if (cs > 1) cluster.sync();
    else __syncthreads();
    if (me != 0) {
        if (status) raise_status(d_status, status);
        return;
    }

    // ---- first block: the row's children -----------------------------------------------------------------
    const int n_in = cs * k;  // <= 256
    if (warp == kRowWarps - 1) {  // the row's log-sum-exp, in double
        const float2 st = lane < cs ? s_stats[lane] : make_float2(-INFINITY, 0.f);
        float m = st.x;
#pragma unroll
        for (int o = kRowMaxCluster / 2; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        double sum = st.x > -INFINITY ? (double)(st.y * pow2_whole(st.x - m)) : 0.0;
#pragma unroll
        for (int o = kRowMaxCluster / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        const uint32_t best = __reduce_max_sync(0xffffffffu, lane < cs ? (uint32_t)(s_in[lane * k] >> 32) : 0u);
        if (lane == 0) {
            const float top = best ? order_decode(best) : -INFINITY;
            s_lse = fabsf(top) < kFarLogit ? (double)m * 0.69314718055994530942 + log(sum) : (double)top;
            if (!(top > -INFINITY)) status |= EAGLE2_STATUS_NONFINITE_LOGIT;
        }
    }
    // (the last warp is busy with the sum; the others rank, two threads a key)
    constexpr int kRankers = kRowThreads - kWarp;
    if (tid < kRankers)
        for (int i = tid >> 1; i < (n_in + 15 & ~15); i += kRankers / 2) {
            const unsigned long long mine = i < n_in ? s_in[i] : 0ull;
            const int rank = count_above<2>(s_in, n_in, mine);
            if ((tid & 1) == 0 && mine && rank < k) s_row[rank] = mine;
        }
    __syncthreads();
    hand_on_row(s_row, s_lse, parent, parent_value, b, row, k, n_s, N, base, by_confidence, tree_token, tree_parent, tree_value, frontier,
                counters, codes, s_code, &s_flag, status, d_status);
}

// Finishes a step whose rows were ranked by another kernel in parts (the LM head that ranks its own logits: a part per
// SM with the part's k best keys and its maximum and sum of exponentials).  A block per row; a row's `slots` places are
// filled up to chunks_lo below split_row and chunks_hi from there on.  Keys of a row differ, but for the empty ones, 0.
// What bounds it is the chain load - bar - candidates - row - ticket - frontier.
constexpr int kPartKeysPerThread = 16;
__global__ void __launch_bounds__(kRowThreads)
expand_parts_kernel(int slots, int split_row, int chunks_lo, int chunks_hi, const double2* __restrict__ stats,
                    const unsigned long long* __restrict__ keys, int k, int D, int s, int n_s, int32_t* __restrict__ tree_token,
                    int32_t* __restrict__ tree_parent, double* __restrict__ tree_value, int32_t* __restrict__ frontier,
                    int* __restrict__ counters, unsigned long long* __restrict__ codes, int32_t* d_status) {
    __shared__ unsigned long long s_cand[kRowCand], s_code[EAGLE2_MAX_K * EAGLE2_MAX_K];
    __shared__ unsigned long long s_row[EAGLE2_MAX_K], s_best[kRowWarps];
    __shared__ __align__(16) uint32_t s_top[kRowGroups];
    __shared__ float s_wmax[kRowWarps];
    __shared__ double s_wsum[kRowWarps], s_lse;
    __shared__ int s_n, s_flag;
    chain_wait();
    chain_release();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int line = blockIdx.x, row = line % n_s, b = line / n_s;
    const int chunks = line < split_row ? chunks_lo : chunks_hi, n_in = chunks * k;
    const unsigned long long* in = keys + (size_t)line * slots * k;
    unsigned long long mine[kPartKeysPerThread], best = 0ull;
#pragma unroll
    for (int t = 0; t < kPartKeysPerThread; ++t) {
        const int i = tid + t * kRowThreads;
        mine[t] = i < n_in ? in[i] : 0ull;
    }
    const double2 part = tid < chunks ? stats[(size_t)line * slots + tid] : make_double2(-INFINITY, 0.0);
    const long long N = nodes_of(k, D), base = s ? (long long)k + (long long)(s - 1) * k * k : 0;
    int parent = -1, status = 0;
    double parent_value = 0.0;
    if (s) status |= parent_of_row(frontier, tree_value, b, row, k, s, N, &parent, &parent_value);
    if (tid == 0) s_n = 0;
    if (tid < k) s_row[tid] = 0ull;
#pragma unroll
    for (int t = 0; t < kPartKeysPerThread; ++t) best = mine[t] > best ? mine[t] : best;
    uint32_t um = (uint32_t)(best >> 32);  // of eight threads, by value
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) um = max(um, __shfl_xor_sync(0xffffffffu, um, o));
    if ((lane & 7) == 0) s_top[tid >> 3] = um;
    const float wmax = warp_max_f32((float)part.x);  // (the maxima are 32-bit values)
    if (lane == 0) s_wmax[warp] = wmax;
    __syncthreads();

    // the bar, as for a row of logits
    uint32_t bar;
    {
        const uint32_t v = s_top[lane];
        int above = 0;
#pragma unroll
        for (int j = 0; j < kRowGroups; j += 4) {
            const uint4 t = *reinterpret_cast<const uint4*>(s_top + j);
            above += (t.x > v) + (t.y > v) + (t.z > v) + (t.w > v);
        }
        bar = __reduce_min_sync(0xffffffffu, above < k ? v : ~0u);
    }
    if ((uint32_t)(best >> 32) >= bar) {
#pragma unroll
        for (int t = 0; t < kPartKeysPerThread; ++t)
            if (mine[t] && (uint32_t)(mine[t] >> 32) >= bar) {
                const int at = atomicAdd(&s_n, 1);
                if (at < kRowCand) s_cand[at] = mine[t];
            }
    }
    // the parts' sums, in double
    float m = s_wmax[0];
#pragma unroll
    for (int w = 1; w < kRowWarps; ++w) m = fmaxf(m, s_wmax[w]);
    const double wsum = warp_sum_f64(part.x > -INFINITY ? part.y * exp(part.x - (double)m) : 0.0);
    if (lane == 0) s_wsum[warp] = wsum;
    __syncthreads();
    int n = s_n;
    if (n > kRowCand) {  // hundreds of equal logits: k times the largest key below the last one taken
        unsigned long long last = ~0ull;
        for (int r = 0; r < k; ++r) {
            unsigned long long top = 0ull;
#pragma unroll
            for (int t = 0; t < kPartKeysPerThread; ++t) top = mine[t] < last && mine[t] > top ? mine[t] : top;
            top = warp_max_u64(top);
            if (lane == 0) s_best[warp] = top;
            __syncthreads();
            top = 0ull;
#pragma unroll
            for (int w = 0; w < kRowWarps; ++w) top = s_best[w] > top ? s_best[w] : top;
            if (tid == 0) s_cand[r] = top;
            last = top;
            __syncthreads();
        }
        n = k;
    }
    if (tid == kRowThreads - 1) {
        double sum = 0.0;
#pragma unroll
        for (int w = 0; w < kRowWarps; ++w) sum += s_wsum[w];
        s_lse = (double)m + log(sum);
        if (!(m > -INFINITY)) status |= EAGLE2_STATUS_NONFINITE_LOGIT;
    }
    for (int i = tid >> 2; i < (n + 7 & ~7); i += kRowThreads / 4) {  // four threads share a key's comparisons
        const unsigned long long key = i < n ? s_cand[i] : 0ull;
        const int rank = count_above<4>(s_cand, n, key);
        if ((tid & 3) == 0 && rank < k && key) s_row[rank] = key;
    }
    __syncthreads();
    hand_on_row(s_row, s_lse, parent, parent_value, b, row, k, n_s, N, base, 0, tree_token, tree_parent, tree_value, frontier, counters,
                codes, s_code, &s_flag, status, d_status);
}

// Slices: the shortest (most blocks) that keep the launch on the device at once; else the longest.
// Many rows of a large vocabulary are left to the tiles, which keep more of memory's bandwidth busy (six steps at
// V = 128256, 1 / 2 / 4 / 8 / 16 / 32 sequences of ten rows: 78 / 107 / 140 / 199 / 238 / 293 us in tiles, 72 / 80 /
// 116 / 159 / 258 / 454 us this way; at V = 32000 69 / 73 / 77 / 109 / 145 / 224 against 56 / 57 / 64 / 78 / 115 /
// 163 us, 64 sequences 306 against 263).
static bool expand_rows_shape(long long rows, int V, int* nf, int* cs) {
    if (V > kRowMaxCluster * kRowThreads * 64 || (rows > 128 && V > 2 * kRowThreads * 64)) return false;
    for (*nf = 4;; *nf *= 2) {
        *cs = (V + kRowThreads * 4 * *nf - 1) / (kRowThreads * 4 * *nf);
        if (*nf == 16 || *cs == 1 || (*cs <= kRowMaxCluster && rows * *cs <= 2LL * sm_count())) return true;
    }
}

template <bool VEC>
static int launch_expand_rows(const float* logits, long long batch_stride, int B, int V, int k, int D, int s, int n_s,
                              int by_confidence, int nf, int cs, int32_t* token, int32_t* parent, double* value, int32_t* frontier,
                              int* counters, unsigned long long* codes, int32_t* d_status, cudaStream_t st) {
    auto kern = nf == 4 ? expand_rows_kernel<4, VEC> : nf == 8 ? expand_rows_kernel<8, VEC> : expand_rows_kernel<16, VEC>;
    return launch_chained(kern, dim3((unsigned)((long long)B * n_s * cs)), dim3(kRowThreads), 0, st, (unsigned)cs, logits, batch_stride,
                          V, k, D, s, n_s, by_confidence, token, parent, value, frontier, counters, codes, d_status);
}

}  // namespace eagle2
