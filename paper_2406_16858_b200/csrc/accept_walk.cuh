// Acceptance at temperature > 0, one walk per sequence (included by accept.cu; the rule and the
// closed form of its rounds are stated there).
//
// One thread-block cluster walks one sequence's tree from the root: it reads the current node's target
// and draft rows into registers (a block holds a contiguous slice of the vocabulary), runs the node's
// rejection chain, goes to the accepted child, and draws the extra token from the weights it still holds
// where the walk stops.  Only the rows on the walk are read - two or three nodes of a typical tree's
// twenty expanded ones - and there is no second launch.  What bounds it is latency: per node one trip to
// memory and one exchange across the cluster for the softmax sums, and one exchange per rejected child.
//   - Rows live in registers, not in shared memory: a round is 4 * NF multiply-adds per thread.
//   - Exponentials are relative to the warp's own maximum, so that maxima and sums cross the cluster in
//     one exchange instead of two; a warp's factor to the common maximum joins its normalisation.
//   - An exchange is one remote store per warp and peer, one cluster barrier, and a warp-wide sum of all
//     blocks' warps in a fixed order: every warp of every block carries the same scalars.
//   - Child i of the node lives in lane i of every warp; its p and q come from the thread that holds its
//     token, so that the corrections for removed tokens cancel bit for bit.
#pragma once

#include <cooperative_groups.h>
#include <math.h>

#include <type_traits>

#include "common.cuh"

namespace eagle2 {

constexpr int kWalkThreads = 512;
constexpr int kWalkWarps = kWalkThreads / kWarp;
constexpr int kWalkMaxCluster = 8;
constexpr int kWalkEntries = kWalkWarps * kWalkMaxCluster;  // one per warp of the cluster

struct WalkSums {  // a warp's contribution to the softmax sums of a node (sum_q: without the node's children), and its
                   // largest logits
    double sum_p, sum_q;
    float max_p, max_q;
};
struct WalkChild {  // a child's token as its holder has it: unnormalised, with the largest logits of the holder's warp
    float ep, eq, mp, mq;
};

__device__ __forceinline__ void prefetch_l2(const float* p, uint32_t bytes) {  // both multiples of 16
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

__device__ __forceinline__ float exp2_approx(float x) {  // 2 ulp; -inf gives 0
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// The exponent of 2 that a warp's exponentials are taken relative to, from its largest logit; to_log2: log2(e) / T.
// (Rounded on its own: the tokens' exponents and the factors between warps have to mean the same number.)
// Far from zero (up to the largest numbers a float holds: masks often are its lowest) that product overflows or is
// rounded by more than the exponents' own differences, so that there differences are taken before the product.
constexpr float kWalkFar = 4194304.f;  // 2^22: the product's rounding is at most 1/4
__device__ __forceinline__ float walk_reference(float max_logit, float to_log2) {
    return max_logit > -INFINITY ? __fmul_rn(max_logit, to_log2) : 0.f;  // (a warp without mass: any number does)
}
__device__ __forceinline__ bool walk_near(float max_logit, float to_log2) { return fabsf(walk_reference(max_logit, to_log2)) < kWalkFar; }
// Factor from one warp's reference to that of the warp with the row's largest logit; FAR: one of the row's is far (rare:
// kept out of the way of the code that a launch runs through once and cold).
static __device__ __noinline__ float walk_factor_far(float max_logit, float row_max, float to_log2) {
    const float ref_w = walk_reference(max_logit, to_log2), ref_r = walk_reference(row_max, to_log2);
    const bool near_w = fabsf(ref_w) < kWalkFar, near_r = fabsf(ref_r) < kWalkFar;
    if (near_w && near_r) return exp2_approx(ref_w - ref_r);
    if (near_w) return exp2_approx(fmaf(-row_max, to_log2, ref_w));
    if (near_r) return exp2_approx(fmaf(max_logit, to_log2, -ref_r));
    return max_logit == row_max ? 1.f : exp2_approx((max_logit - row_max) * to_log2);
}
template <bool FAR>
__device__ __forceinline__ float walk_factor(float max_logit, float row_max, float to_log2) {
    if (FAR) return walk_factor_far(max_logit, row_max, to_log2);
    return exp2_approx(walk_reference(max_logit, to_log2) - walk_reference(row_max, to_log2));
}
// A thread's N logits, in place, to exponentials relative to its warp's reference; their sum (in two chains).
template <int N>
__device__ __forceinline__ float walk_exponentials(float (&x)[N], float max_logit, float to_log2) {
    float t[2] = {0.f, 0.f}, ref = walk_reference(max_logit, to_log2);
    if (__builtin_expect(!walk_near(max_logit, to_log2), 0)) {
        ref = 0.f;
#pragma unroll
        for (int j = 0; j < N; ++j) x[j] -= max_logit;
    }
#pragma unroll
    for (int j = 0; j < N; ++j) x[j] = exp2_approx(fmaf(x[j], to_log2, -ref)), t[j & 1] += x[j];
    return t[0] + t[1];
}
// Probability mass in units of 2^-54: integer sums do not depend on their order, and two additions over the
// warp's lanes (27 bits each) take a quarter of the time of five shuffled steps in 64-bit floating point.
__device__ __forceinline__ unsigned long long mass_to_fixed(float v) {
    const float hi = floorf(v * 134217728.f);
    return ((unsigned long long)(uint32_t)hi << 27) + (unsigned long long)(uint32_t)((v * 134217728.f - hi) * 134217728.f);
}
__device__ __forceinline__ unsigned long long warp_sum_fixed(unsigned long long v) {
    const uint32_t lo = __reduce_add_sync(0xffffffffu, (uint32_t)v & 0x7ffffffu);
    const uint32_t hi = __reduce_add_sync(0xffffffffu, (uint32_t)(v >> 27));
    return ((unsigned long long)hi << 27) + lo;
}

template <int NF, bool VEC, bool FULLQ>
__global__ void __launch_bounds__(kWalkThreads, 1)
accept_walk_kernel(const float* __restrict__ target_logits, long long t_stride,
                   const float* __restrict__ draft_logits_all, long long d_stride,
                   const int32_t* __restrict__ sel_index, const int32_t* __restrict__ sel_parent,
                   const int32_t* __restrict__ sel_token, const int32_t* __restrict__ n_sel,
                   const float* __restrict__ u_accept, const float* __restrict__ u_bonus, int V, int k, int D, int m,
                   float inv_t, int32_t* __restrict__ acc_len, int32_t* __restrict__ acc_path,
                   int32_t* __restrict__ bonus_token, int32_t* d_status) {
    namespace cg = cooperative_groups;
    constexpr int NE = 4 * NF;                     // tokens per thread
    constexpr int kSlice = kWalkThreads * NE;      // tokens per block
    constexpr int PER = VEC ? 4 : 1;               // consecutive tokens per thread and group
    constexpr int GROUPS = NE / PER;               // ascending order: group, thread, token in group
    cg::cluster_group cluster = cg::this_cluster();
    const int cs = (int)cluster.num_blocks(), me = (int)cluster.block_rank();
    const int b = blockIdx.x / cs;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    __shared__ WalkSums s_sums[2][kWalkEntries];
    __shared__ unsigned long long s_fixed[2][kWalkEntries];
    __shared__ double s_mass[kWalkEntries];
    __shared__ WalkChild s_kid[2][EAGLE2_MAX_K];
    __shared__ int s_par[EAGLE2_MAX_M], s_tok[EAGLE2_MAX_M], s_idx[EAGLE2_MAX_M];
    __shared__ float s_u[EAGLE2_MAX_M];
    __shared__ short s_list[kWalkWarps][EAGLE2_MAX_K];
    __shared__ double s_seg[GROUPS * kWalkWarps];
    __shared__ int s_found, s_last;

    chain_wait();
    chain_release();
    const int ns = min(n_sel[b], m);
    int status = 0;
    if (tid < m) {
        s_par[tid] = sel_parent[(long long)b * m + tid];
        s_tok[tid] = sel_token[(long long)b * m + tid];
        s_u[tid] = u_accept[(long long)b * m + tid];
        if (FULLQ) {  // which draft row a node's children come from: one that is there, whatever the index says
            int idx = sel_index[(long long)b * m + tid];
            if (tid < ns && (idx < 0 || idx >= nodes_of(k, D))) idx = 0, status = EAGLE2_STATUS_BAD_TREE;
            s_idx[tid] = idx;
        }
    }
    if (tid == 0) s_found = 0x7fffffff, s_last = -1;
    if (cs > 1) cluster.sync();  // every block runs before any remote store
    else __syncthreads();

    const int lo = me * kSlice;
    // token held in element j of this thread
    auto token_of = [&](int j) { return lo + (VEC ? ((j >> 2) * kWalkThreads + tid) * 4 + (j & 3) : j * kWalkThreads + tid); };
    // the element of this thread that holds token t, or -1
    auto element_of = [&](int t) {
        const int o = t - lo;
        if (o < 0 || o >= kSlice) return -1;
        if (VEC) return ((o >> 2) % kWalkThreads) == tid ? ((o >> 2) / kWalkThreads) * 4 + (o & 3) : -1;
        return (o % kWalkThreads) == tid ? o / kWalkThreads : -1;
    };
    auto meet = [&]() {  // remote and local stores before it are visible behind it
        if (cs > 1) cluster.sync();
        else __syncthreads();
    };
    // Mass (at most 1 in all) of a value per thread over the whole cluster; the same bits in every warp.
    int parity = 0;
    auto mass_of_all = [&](float v) {
        const unsigned long long w = warp_sum_fixed(mass_to_fixed(v));
        if (lane < cs) *cluster.map_shared_rank(&s_fixed[parity][me * kWalkWarps + warp], lane) = w;
        meet();
        unsigned long long r = 0;
        for (int i = lane; i < cs * kWalkWarps; i += 32) r += s_fixed[parity][i];
        parity ^= 1;
        return (double)warp_sum_fixed(r) * (1.0 / (double)(1ull << 54));
    };

    const float to_log2 = inv_t * 1.4426950408889634f;  // logits to exponents of 2
    int cur = -1, len = 0, node = 0, bad = 0;
    float p[NE], q[FULLQ ? NE : 1];
    for (;; ++node) {
        // ---- the node's children: lane i of every warp holds child i -----------------------------------
        int nc = 0;
        if (len < D) {
            for (int x0 = 0; x0 < ns; x0 += 32) {
                const int x = x0 + lane;
                const bool is = x < ns && x > cur && s_par[x] == cur;
                const unsigned bal = __ballot_sync(0xffffffffu, is);
                const int at = nc + __popc(bal & ((1u << lane) - 1u));
                if (is && at < EAGLE2_MAX_K) s_list[warp][at] = (short)x;
                nc += __popc(bal);
            }
            nc = min(nc, EAGLE2_MAX_K);
            __syncwarp();
        }
        const int kid = lane < nc ? s_list[warp][lane] : -1;
        const int kid_tok = kid >= 0 ? s_tok[kid] : -1;
        const float kid_u = kid >= 0 ? s_u[kid] : 0.f;
        __syncwarp();

        // ---- rows into registers (beyond the vocabulary: -inf) -----------------------------------------
        const bool with_q = FULLQ && nc > 0;
        const float* zp = target_logits + (long long)b * t_stride + (long long)(cur + 1) * V;
        const float* zq = nullptr;
        if (with_q) {
            const int row = draft_row_of_child(s_idx[s_list[warp][0]], k);
            zq = draft_logits_all + (long long)b * d_stride + (long long)row * V;
        }
        if (VEC) {
#pragma unroll
            for (int i = 0; i < NF; ++i) {
                const int e = token_of(4 * i);
                float4 a = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY), c = a;
                if (e < V) {
                    a = __ldcs(reinterpret_cast<const float4*>(zp + e));
                    if (with_q) c = __ldcs(reinterpret_cast<const float4*>(zq + e));
                }
                p[4 * i] = a.x, p[4 * i + 1] = a.y, p[4 * i + 2] = a.z, p[4 * i + 3] = a.w;
                if (FULLQ) q[4 * i] = c.x, q[4 * i + 1] = c.y, q[4 * i + 2] = c.z, q[4 * i + 3] = c.w;
            }
        } else {
#pragma unroll
            for (int j = 0; j < NE; ++j) {
                const int e = token_of(j);
                p[j] = e < V ? __ldcs(zp + e) : -INFINITY;
                if (FULLQ) q[j] = e < V && with_q ? __ldcs(zq + e) : -INFINITY;
            }
        }
        // While this node is worked on, the rows of its first child - the likeliest to be accepted - come
        // into L2.
        if (VEC && nc > 0 && warp == 0 && lo < V) {
            const int first = s_list[0][0];
            int grand = -1;
            if (FULLQ) {
                for (int x0 = 0; x0 < ns && grand < 0; x0 += 32) {
                    const int x = x0 + lane;
                    const unsigned bal = __ballot_sync(0xffffffffu, x < ns && s_par[x] == first);
                    if (bal) grand = x0 + __ffs(bal) - 1;
                }
            }
            const uint32_t bytes = (uint32_t)(min(kSlice, V - lo) * 4);
            if (lane == 0) {
                prefetch_l2(target_logits + (long long)b * t_stride + (long long)(first + 1) * V + lo, bytes);
                if (grand >= 0)
                    prefetch_l2(draft_logits_all + (long long)b * d_stride + (long long)draft_row_of_child(s_idx[grand], k) * V + lo, bytes);
            }
        }

        // ---- exponentials relative to the warp's maxima, their sums across the cluster -----------------
        float mp = -INFINITY, mq = -INFINITY;
#pragma unroll
        for (int j = 0; j < NE; ++j) {
            mp = fmaxf(mp, p[j]);
            if (FULLQ) mq = fmaxf(mq, q[j]);
        }
        mp = warp_max_f32(mp);
        if (FULLQ) mq = warp_max_f32(mq);
        const double wp = warp_sum_f64((double)walk_exponentials<NE>(p, mp, to_log2));
        float tq = 0.f;
        if (FULLQ && with_q) tq = walk_exponentials<FULLQ ? NE : 1>(q, mq, to_log2);
        uint32_t mine = 0u;  // the elements of this thread that are children's tokens
        for (int i = 0; i < nc; ++i) {  // the holder of a child's token tells every block
            const int t = __shfl_sync(0xffffffffu, kid_tok, i);
            const int j = element_of(t);
            if (j >= 0 && t < V) {
                mine |= 1u << j;
                WalkChild c = {0.f, 0.f, mp, mq};
#pragma unroll
                for (int u = 0; u < NE; ++u)
                    if (u == j) {
                        c.ep = p[u];
                        if (FULLQ) c.eq = q[u];
                    }
                for (int r = 0; r < cs; ++r) *cluster.map_shared_rank(&s_kid[node & 1][i], r) = c;
            }
        }
        // q's sum leaves the children out: what is left of q after rejections is then a sum of what is left, where one
        // minus the rejected children's share would be nothing but rounding behind a child that holds nearly all of it.
        if (FULLQ && mine) {
            float t[2] = {0.f, 0.f};
#pragma unroll
            for (int j = 0; j < NE; ++j) t[j & 1] += (mine >> j) & 1u ? 0.f : q[j];
            tq = t[0] + t[1];
        }
        const double wq = FULLQ ? warp_sum_f64((double)tq) : 0.0;
        if (lane < cs) {
            WalkSums* dst = cluster.map_shared_rank(&s_sums[node & 1][me * kWalkWarps + warp], lane);
            dst->sum_p = wp, dst->sum_q = wq, dst->max_p = mp, dst->max_q = mq;
        }
        meet();
        // (a warp without mass has sum 0 and no largest logit; a NaN or +inf logit makes its sum NaN)
        constexpr int kPerLane = kWalkEntries / 32;
        double gs_p[kPerLane], gs_q[kPerLane];
        float gm_p[kPerLane], gm_q[kPerLane], gp = -INFINITY, gq = -INFINITY;
        bool far = false;
#pragma unroll
        for (int u = 0; u < kPerLane; ++u) {
            const int i = lane + 32 * u;
            WalkSums w = {0.0, 0.0, -INFINITY, -INFINITY};
            if (i < cs * kWalkWarps) w = s_sums[node & 1][i];
            gs_p[u] = w.sum_p, gs_q[u] = w.sum_q, gm_p[u] = w.max_p, gm_q[u] = w.max_q;
            gp = fmaxf(gp, w.max_p);
            if (FULLQ) gq = fmaxf(gq, w.max_q);
            far |= !walk_near(w.max_p, to_log2) | (FULLQ && !walk_near(w.max_q, to_log2));
        }
        far = __any_sync(0xffffffffu, far);
        gp = order_decode(__reduce_max_sync(0xffffffffu, order_code(gp)));
        if (FULLQ) gq = order_decode(__reduce_max_sync(0xffffffffu, order_code(gq)));
        double sum_p = 0.0, sum_q = 0.0;  // (sum_q: without the children, which are added below)
        // Factors: of this warp's exponentials, of the child's in this lane (0 for a warp without mass, which has no
        // largest logit, and for a token without any).
        float fp = 0.f, fq = 0.f, kid_p = 0.f, kid_q = 0.f;
        WalkChild child = {0.f, 0.f, 0.f, 0.f};
        if (lane < nc) {
            if (kid_tok >= 0 && kid_tok < V) child = s_kid[node & 1][lane];
            else bad = 1;
        }
        auto weigh = [&](auto far_tag) {
            constexpr bool FAR = decltype(far_tag)::value;
#pragma unroll
            for (int u = 0; u < kPerLane; ++u) {
                if (gs_p[u] != 0.0) sum_p += gs_p[u] * (double)walk_factor<FAR>(gm_p[u], gp, to_log2);
                if (FULLQ && gs_q[u] != 0.0) sum_q += gs_q[u] * (double)walk_factor<FAR>(gm_q[u], gq, to_log2);
            }
            if (mp > -INFINITY) fp = walk_factor<FAR>(mp, gp, to_log2);
            if (FULLQ && mq > -INFINITY) fq = walk_factor<FAR>(mq, gq, to_log2);
            if (child.ep > 0.f) kid_p = walk_factor<FAR>(child.mp, gp, to_log2);
            if (FULLQ && child.eq > 0.f) kid_q = walk_factor<FAR>(child.mq, gq, to_log2);
        };
        if (__builtin_expect(far, 0)) weigh(std::true_type{});
        else weigh(std::false_type{});
        // What is left of q behind child i, lane i: the sum without children and the children after it (a token counts
        // where it first is).  Sums and scan go side by side.
        double behind = 0.0;  // of this lane's child and those after it
        if (FULLQ) {
            const unsigned same = __match_any_sync(0xffffffffu, kid_tok);
            if (lane < nc && __ffs(same) - 1 == lane) behind = (double)child.eq * (double)kid_q;
        }
#pragma unroll
        for (int s = 0; s < 5; ++s) {
            sum_p += __shfl_xor_sync(0xffffffffu, sum_p, 16 >> s);
            if (FULLQ) {
                sum_q += __shfl_xor_sync(0xffffffffu, sum_q, 16 >> s);
                const double add = __shfl_down_sync(0xffffffffu, behind, 1 << s);
                if (lane + (1 << s) < 32) behind += add;
            }
        }
        double left = 0.0;
        if (FULLQ) {
            const double after = __shfl_down_sync(0xffffffffu, behind, 1);
            left = sum_q + (lane < 31 ? after : 0.0);
            sum_q += __shfl_sync(0xffffffffu, behind, 0);
        }
        // (a row whose largest logit overflows when divided by the temperature counts as one that was not finite)
        bad |= !(sum_p > 0.0) | !(fabsf(gp * inv_t) < INFINITY);
        if (FULLQ && with_q) bad |= !(sum_q > 0.0) | !(fabsf(gq * inv_t) < INFINITY);
        const float c_p = (float)(1.0 / sum_p), c_q = with_q ? (float)(1.0 / sum_q) : 0.f;
        if (FULLQ) left *= with_q ? 1.0 / sum_q : 0.0;
        // what this warp's exponentials have to be multiplied with to be probabilities, and the children's
        fp = fp > 0.f ? fp * c_p : 0.f, fq = fq > 0.f ? fq * c_q : 0.f;
        const float q_to_p = fp > 0.f ? fminf(fq / fp, 1e30f) : 0.f;  // q in units of the warp's p
        kid_p = child.ep > 0.f ? child.ep * (kid_p * c_p) : 0.f;
        if (FULLQ) kid_q = child.eq > 0.f ? child.eq * (kid_q * c_q) : 0.f;

        // ---- the rejection chain over the node's children ----------------------------------------------
        int taken = -1;
        if (FULLQ) {
            // (alpha, beta): the target in force is max(p - alpha q, 0) / beta; rest: what is left of q.
            // A token that leaves q keeps the alpha in force then: its holder folds that into its p.
            double alpha = 0.0, beta = 1.0, rest = 1.0;
            for (int i = 0; i < nc; ++i) {
                const double pf = (double)__shfl_sync(0xffffffffu, kid_p, i), qf = (double)__shfl_sync(0xffffffffu, kid_q, i);
                const double have = fmax(pf - alpha * qf, 0.0);
                // u < min(1, (have / beta) / (qf / rest)) without the divisions; off q's support: u < (have > 0)
                const double u = (double)__shfl_sync(0xffffffffu, kid_u, i);
                if (qf > 0.0 && rest > 0.0 ? u * qf * beta < have * rest : have > 0.0) {
                    taken = i;
                    break;
                }
                const double alpha_new = alpha + (rest > 0.0 ? beta / rest : 0.0);  // residual after rejecting child i
                double mass = 1.0;
                if (i < nc - 1) {  // (nothing is tested after the last child: only alpha is needed)
                    const float an = (float)alpha_new * q_to_p;
                    float part[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                    for (int j = 0; j < NE; ++j) part[j & 3] += fmaxf(fmaf(-an, q[j], p[j]), 0.f);
                    mass = mass_of_all(((part[0] + part[1]) + (part[2] + part[3])) * fp);
                }
                if (mass > 0.0) alpha = alpha_new, beta = mass;  // zero residual mass: the target stays
                rest = __shfl_sync(0xffffffffu, left, i);
                const int e = element_of(__shfl_sync(0xffffffffu, kid_tok, i));
                if (e >= 0) {
                    const float ai = (float)alpha * q_to_p;
#pragma unroll
                    for (int j = 0; j < NE; ++j)
                        if (j == e) p[j] = fmaxf(fmaf(-ai, q[j], p[j]), 0.f), q[j] = 0.f;
                }
            }
            if (taken < 0 && nc > 0) {
                const float al = (float)alpha * q_to_p;
#pragma unroll
                for (int j = 0; j < NE; ++j) p[j] = fmaxf(fmaf(-al, q[j], p[j]), 0.f);
            }
        } else {
            double removed_p = 0.0;  // accept with p(x), then take x out of p
            for (int i = 0; i < nc; ++i) {
                const double px = (double)__shfl_sync(0xffffffffu, kid_p, i);
                const double rest = 1.0 - removed_p;
                const double pj = rest > 0.0 ? px / rest : 0.0;
                if ((double)__shfl_sync(0xffffffffu, kid_u, i) < (pj < 1.0 ? pj : 1.0)) {
                    taken = i;
                    break;
                }
                if ((rest - px) > 0.0) {  // zero residual mass: keep p as it is
                    removed_p += px;
                    const int e = element_of(__shfl_sync(0xffffffffu, kid_tok, i));
                    if (e >= 0) {
#pragma unroll
                        for (int j = 0; j < NE; ++j)
                            if (j == e) p[j] = 0.f;
                    }
                }
            }
        }
        if (taken >= 0) {
            cur = __shfl_sync(0xffffffffu, kid, taken);
            if (me == 0 && tid == 0) acc_path[(long long)b * D + len] = cur;
            ++len;
            continue;
        }

        // the walk stops here: the weights of the extra token's law
#pragma unroll
        for (int j = 0; j < NE; ++j) p[j] *= fp;
        break;
    }
    if (bad) status |= EAGLE2_STATUS_NONFINITE_LOGIT;
    raise_status(d_status, status);
    if (me == 0 && tid == 0) {
        acc_len[b] = len;
        for (int j = len; j < D; ++j) acc_path[(long long)b * D + j] = -1;
    }

    // ---- the extra token: inverse CDF in ascending token id ----------------------------------------------
    // The warp sums of the block's segments (group, warp), then the blocks' totals across the cluster.
    double mine = 0.0;
#pragma unroll
    for (int gi = 0; gi < GROUPS; ++gi) {
        float t = 0.f;
#pragma unroll
        for (int c = 0; c < PER; ++c) t += p[gi * PER + c];
        mine += (double)t;
    }
    mine = warp_sum_f64(mine);
    if (lane < cs) *cluster.map_shared_rank(&s_mass[me * kWalkWarps + warp], lane) = mine;
    meet();
    // lane r of every warp holds the total of block r, then the total up to it
    double block_total = 0.0;
    {
        double t[kWalkMaxCluster];
#pragma unroll
        for (int r = 0; r < kWalkMaxCluster; ++r) t[r] = r < cs ? s_mass[r * kWalkWarps + (lane & (kWalkWarps - 1))] : 0.0;
#pragma unroll
        for (int o = kWalkWarps / 2; o > 0; o >>= 1)
#pragma unroll
            for (int r = 0; r < kWalkMaxCluster; ++r) t[r] += __shfl_xor_sync(0xffffffffu, t[r], o);
#pragma unroll
        for (int r = 0; r < kWalkMaxCluster; ++r)
            if (r == lane) block_total = t[r];
    }
    double incl = block_total;
#pragma unroll
    for (int o = 1; o < kWalkMaxCluster; o <<= 1) {
        const double add = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += add;
    }
    const double total = __shfl_sync(0xffffffffu, incl, kWalkMaxCluster - 1);
    const double thr = (double)u_bonus[b] * total;
    const unsigned crossed = __ballot_sync(0xffffffffu, lane < cs && incl > thr);
    const unsigned massive = __ballot_sync(0xffffffffu, lane < cs && block_total > 0.0);
    // (rounding may leave no block beyond the threshold: then the last one with weight has the token)
    const int pick = crossed ? __ffs(crossed) - 1 : (massive ? 31 - __clz(massive) : 0);
    if (me == pick) {
        const double before = pick ? __shfl_sync(0xffffffffu, incl, pick - 1) : 0.0;
        int last = -1;
#pragma unroll
        for (int gi = 0; gi < GROUPS; ++gi) {
            double t = 0.0;
#pragma unroll
            for (int c = 0; c < PER; ++c) {
                t += (double)p[gi * PER + c];
                if (p[gi * PER + c] > 0.f) last = token_of(gi * PER + c);
            }
            t = warp_sum_f64(t);
            if (lane == 0) s_seg[gi * kWalkWarps + warp] = t;
        }
        last = __reduce_max_sync(0xffffffffu, last);
        if (lane == 0 && last >= 0) atomicMax(&s_last, last);
        __syncthreads();
        // Which segment passes the threshold: a lane adds up a run of consecutive segments, the warp the lanes.
        constexpr int kRun = (GROUPS * kWalkWarps + 31) / 32;
        double seg[kRun], upto_lane = 0.0;
#pragma unroll
        for (int u = 0; u < kRun; ++u) {
            const int sg = lane * kRun + u;
            seg[u] = sg < GROUPS * kWalkWarps ? s_seg[sg] : 0.0;
            upto_lane += seg[u];
        }
        const double own_run = upto_lane;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double add = __shfl_up_sync(0xffffffffu, upto_lane, o);
            if (lane >= o) upto_lane += add;
        }
        double run_l = before + (upto_lane - own_run);  // mass before the segment looked at
        int seg_l = -1;
#pragma unroll
        for (int u = 0; u < kRun; ++u)
            if (seg_l < 0) {
                if (run_l + seg[u] > thr) seg_l = lane * kRun + u;
                else run_l += seg[u];
            }
        const unsigned past = __ballot_sync(0xffffffffu, seg_l >= 0);
        if (past) {
            const int src = __ffs(past) - 1;
            const int sg = __shfl_sync(0xffffffffu, seg_l, src);
            const double run = __shfl_sync(0xffffffffu, run_l, src);
            if (sg % kWalkWarps == warp) {
                const int gi = sg / kWalkWarps;
                double w4[PER], local = 0.0;
                int e0 = 0;
#pragma unroll
                for (int u = 0; u < GROUPS; ++u)
                    if (u == gi) {
                        e0 = token_of(u * PER);
#pragma unroll
                        for (int c = 0; c < PER; ++c) w4[c] = (double)p[u * PER + c], local += w4[c];
                    }
                double upto = local;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const double add = __shfl_up_sync(0xffffffffu, upto, o);
                    if (lane >= o) upto += add;
                }
                double at = run + (upto - local);
                int found = 0x7fffffff;
#pragma unroll
                for (int c = 0; c < PER; ++c) {
                    at += w4[c];
                    if (at > thr && w4[c] > 0.0) found = min(found, e0 + c);
                }
                if (!__any_sync(0xffffffffu, found != 0x7fffffff)) {  // rounding: the segment's last token with weight
                    int tail = -1;
#pragma unroll
                    for (int c = 0; c < PER; ++c)
                        if (w4[c] > 0.0) tail = e0 + c;
                    tail = __reduce_max_sync(0xffffffffu, tail);
                    if (tail >= 0) found = tail;
                }
                if (found != 0x7fffffff) atomicMin(&s_found, found);
            }
        }
        __syncthreads();
        if (tid == 0) bonus_token[b] = s_found != 0x7fffffff ? s_found : max(s_last, 0);
    }
    if (cs > 1) cluster.sync();  // no block leaves while another may still read or write its memory
}

}  // namespace eagle2
