// branch.cu -- Pruner, batch_pick_out and batch_split of Algorithm 2
// (Section 3 overview and Section 3.1), bit-exact and deterministic.
//
//   k_branch_plan_cl  one problem: a thread-block cluster plans the pool (the FP64
//                   prune test, the pick-out selection as the exact k-th smallest
//                   of the composite keys (order(ub), id) and (order(lb), id) by
//                   8-bit radix selection, the stable ranks of picked and unpicked
//                   survivors by warp ballots); k_branch_plan_small the same for
//                   at most 256 rows, by counting.
//   k_branch_plan   several problems: the same with one CTA per problem.
//   k_branch_write  a few lanes per pool row: the widest coordinate (argmax over the
//                   lanes, lowest index on ties), the FP32 midpoint, and the
//                   coalesced writes of two children or of the unpicked row.
#include <cooperative_groups.h>

#include "bab_internal.cuh"
#include "kernels.cuh"
#include "select.cuh"

namespace bab {

constexpr int kPlanThreads = 1024;
constexpr int kPickFlag = 1 << 30;

// Problem pb's quota, and the part of it that is taken by upper bound.
__device__ __forceinline__ void plan_quota(const BranchArgs &a, int pb, int &n_pick, int &n1)
{
    n_pick = a.n_pick;
    n1 = a.n1;
    if (a.n_pick_dev) {
        n_pick = a.n_pick_dev[pb] < 0 ? 0 : a.n_pick_dev[pb];
        n1 = (int)ceil((double)a.eta * n_pick);
        n1 = n1 > n_pick ? n_pick : n1;
    }
}

__global__ void __launch_bounds__(kPlanThreads) k_branch_plan(BranchArgs a)
{
    __shared__ unsigned hist[256];
    __shared__ uint32_t sh_pk;
    __shared__ uint64_t sh_pid;
    __shared__ int sh_rem, sh_done;
    __shared__ int wsum[2][kPlanThreads / 32];
    __shared__ int red[kPlanThreads / 32];
    const int n = live_count(a.n, a.d_n);
    // this CTA's problem and its rows
    const int pb = blockIdx.x;
    const BatchDesc &B = a.batch;
    auto mine = [&](int i) { return B.prob == nullptr || row_problem(B, i) == pb; };
    const double inc = a.inc_val[pb];
    int n_pick, n1;
    plan_quota(a, pb, n_pick, n1);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

    // prune (strict, in FP64; a NaN bound is kept and latched as BAB_ERR_NUMERIC)
    int cnt = 0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        if (!mine(i)) continue;
        const float lbi = a.lb[i];
        if (lbi != lbi) set_status(a.status, BAB_ERR_NUMERIC);
        const uint8_t k = !((double)lbi > inc);
        a.keep[i] = k;
        cnt += k;
    }
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xFFFFFFFFu, cnt, o);
    if (lane == 0) red[warp] = cnt;
    __syncthreads();
    int ns = 0;
    for (int w = 0; w < kPlanThreads / 32; ++w) ns += red[w];
    __syncthreads();

    const bool all = ns <= n_pick;
    Thresh T1, T2;
    T1.none = T2.none = true;
    const float *key2 = a.lb;  // the rest of the quota is chosen on the lower bound
    if (!all) {
        const uint8_t *keep = a.keep;
        T1 = radix_select(n, a.ub, a.id, [&](int i) { return mine(i) && keep[i] != 0; }, n1, hist, &sh_pk, &sh_pid,
                          &sh_rem, &sh_done);
        const float *ub = a.ub;
        const uint64_t *ids = a.id;
        auto cand = [&](int i) { return mine(i) && keep[i] != 0 && !le_thresh(float_order(ub[i]), ids[i], T1); };
        T2 = radix_select(n, key2, a.id, cand, n_pick - n1, hist, &sh_pk, &sh_pid, &sh_rem, &sh_done);
    }

    // stable ranks of picked and unpicked survivors
    int base_p = 0, base_r = 0;
    const unsigned lt = (1u << lane) - 1u;
    for (int c0 = 0; c0 < n; c0 += blockDim.x) {
        const int i = c0 + threadIdx.x;
        bool kp = false, pk = false;
        const bool own = i < n && mine(i);
        if (own) {
            kp = a.keep[i] != 0;
            const bool by_ub = le_thresh(float_order(a.ub[i]), a.id[i], T1);
            pk = kp && (all || by_ub || le_thresh(float_order(key2[i]), a.id[i], T2));
        }
        const bool rs = kp && !pk;
        const unsigned bp = __ballot_sync(0xFFFFFFFFu, pk), br = __ballot_sync(0xFFFFFFFFu, rs);
        if (lane == 0) {
            wsum[0][warp] = __popc(bp);
            wsum[1][warp] = __popc(br);
        }
        __syncthreads();
        int op = 0, orr = 0, tp = 0, tr = 0;
        for (int w = 0; w < kPlanThreads / 32; ++w) {
            if (w < warp) {
                op += wsum[0][w];
                orr += wsum[1][w];
            }
            tp += wsum[0][w];
            tr += wsum[1][w];
        }
        if (own) {
            if (pk) a.dest[i] = (base_p + op + __popc(bp & lt)) | kPickFlag;
            else if (rs) a.dest[i] = base_r + orr + __popc(br & lt);
            else a.dest[i] = -1;
        }
        base_p += tp;
        base_r += tr;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        a.pcounts[2 * pb] = base_p;
        a.pcounts[2 * pb + 1] = base_r;
    }
}

// ---------------------------------------------------------------------------
// One problem
// ---------------------------------------------------------------------------
__device__ __forceinline__ void plan_totals(const BranchArgs &a, int picked, int rest)
{
    a.d_counts[0] = 2 * picked;
    a.d_counts[1] = rest;
    a.d_counts[2] = 2 * picked + rest;
    a.poff[0] = 0;
    a.poff[1] = 2 * picked;
    if (a.pcounts) {
        a.pcounts[0] = picked;
        a.pcounts[1] = rest;
    }
}

// At most kSmallPlan rows, one per thread: a row is among the k smallest composite keys when fewer than k candidates
// have a smaller one, so each selection is one count over the rows, without a branch (the others carry the largest key).
// 48 rows: 28 us by radix passes -> 5 us; the whole call at 256 rows: 29 to 37 us by radix passes, 39 to 46 with a branch
// a row, 17 without (the host's launches).
constexpr int kSmallPlan = 256;

__global__ void __launch_bounds__(kSmallPlan) k_branch_plan_small(BranchArgs a)
{
    __shared__ uint32_t key[kSmallPlan];
    __shared__ uint64_t ids[kSmallPlan];
    __shared__ int wsum[2][kSmallPlan / 32];
    __shared__ float wmn[kSmallPlan / 32], wmx[kSmallPlan / 32];
    const int n = live_count(a.n, a.d_n);
    const int i = threadIdx.x, lane = i & 31, warp = i >> 5;
    const bool row = i < n;
    int n_pick, n1;
    plan_quota(a, 0, n_pick, n1);
    const float lb = row ? a.lb[i] : 0.f, ub = row ? a.ub[i] : 0.f;
    const uint64_t id = row ? a.id[i] : 0;
    if (row && lb != lb) set_status(a.status, BAB_ERR_NUMERIC);  // a NaN bound is kept and latched
    const bool kp = row && !((double)lb > a.inc_val[0]);
    if (row) a.keep[i] = kp;
    const int ns = __syncthreads_count(kp);
    bool pk = kp;
    if (ns > n_pick) {
        // among the rows flagged `in`, whether this one is one of the k smallest by (order(v), id)
        auto smallest = [&](bool in, float v, int k) {
            const uint32_t mk = float_order(v);
            key[i] = in ? mk : 0xFFFFFFFFu;
            ids[i] = in ? id : ~0ull;
            __syncthreads();
            int less = 0;
            if (k > 0) {
#pragma unroll 8
                for (int j = 0; j < n; ++j) less += (key[j] < mk) | ((key[j] == mk) & (ids[j] < id));
            }
            __syncthreads();
            return in && less < k;
        };
        const bool by_ub = smallest(kp, ub, n1);
        const bool cand = kp && !by_ub;
        float v2 = lb;
        if (a.pick_rule == 1) {
            // min-max scaling over the candidates' (non-NaN) lower bounds, then each candidate's race key
            float mn = cand && lb == lb ? lb : INFINITY, mx = cand && lb == lb ? lb : -INFINITY;
            for (int o = 16; o > 0; o >>= 1) {
                mn = fminf(mn, __shfl_xor_sync(0xFFFFFFFFu, mn, o));
                mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));
            }
            if (lane == 0) {
                wmn[warp] = mn;
                wmx[warp] = mx;
            }
            __syncthreads();
            for (int w = 0; w < kSmallPlan / 32; ++w) {
                mn = fminf(mn, wmn[w]);
                mx = fmaxf(mx, wmx[w]);
            }
            if (cand && lb == lb) v2 = pick_key(lb, mn, mx, a.temperature, a.pick_seed, id);
            if (cand) a.pick_keys[i] = v2;
        }
        const bool by_lb = smallest(cand, v2, n_pick - n1);
        pk = by_ub || by_lb;
    }
    const bool rs = kp && !pk;
    const unsigned lt = (1u << lane) - 1u;
    const unsigned bp = __ballot_sync(0xFFFFFFFFu, pk), br = __ballot_sync(0xFFFFFFFFu, rs);
    __syncthreads();
    if (lane == 0) {
        wsum[0][warp] = __popc(bp);
        wsum[1][warp] = __popc(br);
    }
    __syncthreads();
    int op = 0, orr = 0, tp = 0, tr = 0;
    for (int w = 0; w < kSmallPlan / 32; ++w) {
        if (w < warp) {
            op += wsum[0][w];
            orr += wsum[1][w];
        }
        tp += wsum[0][w];
        tr += wsum[1][w];
    }
    if (row) a.dest[i] = pk ? ((op + __popc(bp & lt)) | kPickFlag) : rs ? orr + __popc(br & lt) : -1;
    if (i == 0) plan_totals(a, tp, tr);
}

// A cluster of 1 to 8 CTAs, each with a contiguous share of the rows: the histograms of a radix pass are summed over the
// CTAs' shared memory (distributed shared memory), one cluster barrier a pass, and every CTA finds the same digit; the
// ranks start from the other CTAs' counts.  A pass stops the selection as soon as its digit's rows are all needed.
// What bounds it is the latency of a pass, not bytes: 60000 rows took one CTA 473 us, the cluster 84 us reading its share
// again in every pass and 51 us with the rows in registers (at most kPlanItems a thread).
constexpr int kPlanCTAs = 8;
constexpr int kPlanItems = 8;  // rows a thread keeps in registers

struct PlanShared {
    unsigned hist[2][256];
    unsigned wtot[8];
    int part[2][2];
    float mn, mx;
    int wsum[2][kPlanThreads / 32];
    float wmn[kPlanThreads / 32], wmx[kPlanThreads / 32];
    int digit, rem, done;
};

// ITEMS > 0: the share is at most ITEMS rows a thread, their keys and identifiers loaded once and kept in registers;
// 0: any share, read again in every pass.
template <int ITEMS>
__global__ void __launch_bounds__(kPlanThreads) k_branch_plan_cl(BranchArgs a)
{
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    __shared__ PlanShared sh;
    const int n = live_count(a.n, a.d_n), share = (n + C - 1) / C;
    const int i0 = min(n, rank * share), i1 = min(n, i0 + share);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const double inc = a.inc_val[0];
    int n_pick, n1;
    plan_quota(a, 0, n_pick, n1);
    // (a lone CTA needs neither the cluster's barriers nor its view of the shared memory: ties among 600 rows 43 -> 36 us)
    auto sync = [&]() {
        if (C > 1) cluster.sync();
        else __syncthreads();
    };
    auto of = [&](auto *p, int q) { return C > 1 ? cluster.map_shared_rank(p, q) : p; };
    // the sum of a value over the block's threads (every thread gets it)
    auto block_sum = [&](int v) {
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
        if (lane == 0) sh.wsum[0][warp] = v;
        __syncthreads();
        int t = sh.wsum[0][lane];
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xFFFFFFFFu, t, o);
        __syncthreads();
        return t;
    };

    // A row's order-preserving keys of ub and of lb (or its race key), its identifier and whether it survives; row it of
    // this thread is i0 + it * kPlanThreads + tid.
    struct Row {
        uint32_t ub, v2;
        uint64_t id;
        bool kept;
    };
    constexpr int R = ITEMS > 0 ? ITEMS : 1;
    uint32_t r_ub[R], r_v2[R], r_kept = 0;
    uint64_t r_id[R];
    // prune (strict, in FP64; a NaN bound is kept and latched as BAB_ERR_NUMERIC)
    auto prune = [&](int i, float lbi) {
        if (lbi != lbi) set_status(a.status, BAB_ERR_NUMERIC);
        const bool k = !((double)lbi > inc);
        a.keep[i] = k;
        return k;
    };
    int cnt = 0;
    if (ITEMS > 0) {
        float v[R];
#pragma unroll
        for (int it = 0; it < R; ++it) {
            const int i = i0 + it * kPlanThreads + tid;
            v[it] = i < i1 ? a.lb[i] : 0.f;
            r_ub[it] = i < i1 ? float_order(a.ub[i]) : 0u;
            r_id[it] = i < i1 ? a.id[i] : 0ull;
        }
#pragma unroll
        for (int it = 0; it < R; ++it) {
            const int i = i0 + it * kPlanThreads + tid;
            r_v2[it] = float_order(v[it]);
            if (i < i1 && prune(i, v[it])) {
                r_kept |= 1u << it;
                ++cnt;
            }
        }
    } else {
        for (int i = i0 + tid; i < i1; i += kPlanThreads) cnt += prune(i, a.lb[i]);
    }
    bool race = false;  // v2 is the race key from here on
    // every row of the share in turn, all threads of the block together: f(row's index, its data); kept is false beyond
    // the share
    auto each = [&](auto f) {
        if (ITEMS > 0) {
#pragma unroll
            for (int it = 0; it < R; ++it) {
                if (it * kPlanThreads >= i1 - i0) break;  // (the same for the whole block)
                Row r{r_ub[it], r_v2[it], r_id[it], ((r_kept >> it) & 1u) != 0};
                f(i0 + it * kPlanThreads + tid, it, r);
            }
        } else {
            for (int b = i0; b < i1; b += kPlanThreads) {
                const int i = b + tid;
                Row r{0u, 0u, 0ull, i < i1 && a.keep[i] != 0};
                if (r.kept) {
                    r.ub = float_order(a.ub[i]);
                    r.v2 = float_order(race ? a.pick_keys[i] : a.lb[i]);
                    r.id = a.id[i];
                }
                f(i, 0, r);
            }
        }
    };
    cnt = block_sum(cnt);
    if (tid == 0) sh.part[0][0] = cnt;
    sync();
    int ns = 0;
    for (int q = 0; q < C; ++q) ns += *of(&sh.part[0][0], q);

    const bool all = ns <= n_pick;
    Thresh T1, T2;
    T1.none = T2.none = true;
    int parity = 0;
    // the kth smallest (1-based) composite key (key(row), id) among the rows accepted by filt, over the whole cluster
    auto select = [&](auto key_of, auto filt, int kth) {
        Thresh T;
        T.none = kth <= 0;
        T.key = 0;
        T.id = 0;
        if (T.none) return T;
        int rem = kth;
        for (int pass = 0; pass < 12; ++pass, parity ^= 1) {
            unsigned *hist = sh.hist[parity];
            if (tid < 256) hist[tid] = 0;
            __syncthreads();
            each([&](int, int, const Row &r) {
                const uint32_t key = key_of(r);
                const bool in = filt(r) && prefix_match(key, r.id, T.key, T.id, pass);
                const uint32_t dg = digit_of(key, r.id, pass);
                // (the leading digits of most rows agree: one addition for the warp then)
                const unsigned m = __ballot_sync(0xFFFFFFFFu, in);
                if (m == 0) return;
                const int first = __ffs(m) - 1;
                const uint32_t d0 = __shfl_sync(0xFFFFFFFFu, dg, first);
                if (__all_sync(0xFFFFFFFFu, !in || dg == d0)) {
                    if (lane == first) atomicAdd(&hist[d0], (unsigned)__popc(m));
                } else if (in) {
                    atomicAdd(&hist[dg], 1u);
                }
            });
            sync();  // every CTA's histogram complete
            unsigned h = 0, inclusive = 0;
            if (tid < 256) {
#pragma unroll
                for (int q = 0; q < kPlanCTAs; ++q)
                    if (q < C) h += of(hist, q)[tid];
                inclusive = h;
                for (int o = 1; o < 32; o *= 2) {
                    const unsigned v = __shfl_up_sync(0xFFFFFFFFu, inclusive, o);
                    if (lane >= o) inclusive += v;
                }
                if (lane == 31) sh.wtot[warp] = inclusive;
            }
            __syncthreads();
            if (tid < 256) {
                for (int w = 0; w < warp; ++w) inclusive += sh.wtot[w];
                const bool here = inclusive >= (unsigned)rem && inclusive - h < (unsigned)rem;
                const bool none = tid == 255 && inclusive < (unsigned)rem;  // fewer candidates than asked for: all
                if (here || none) {
                    sh.digit = tid;
                    sh.rem = rem - (int)(none ? inclusive : inclusive - h);
                    sh.done = here && h == (unsigned)(rem - (int)(inclusive - h));
                }
            }
            __syncthreads();
            const uint32_t D = (uint32_t)sh.digit;
            rem = sh.rem;
            const bool done = sh.done != 0;
            if (pass < 4) T.key |= D << (24 - 8 * pass);
            else T.id |= (uint64_t)D << (56 - 8 * (pass - 4));
            if (done) {
                // every row with this prefix is needed
                if (pass < 4) {
                    T.key |= pass == 3 ? 0u : 0xFFFFFFFFu >> (8 * (pass + 1));
                    T.id = ~0ull;
                } else if (pass < 11) {
                    T.id |= ~0ull >> (8 * (pass - 3));
                }
                parity ^= 1;
                break;
            }
        }
        return T;
    };
    if (!all) {
        T1 = select([](const Row &r) { return r.ub; }, [](const Row &r) { return r.kept; }, n1);
        auto cand = [&](const Row &r) { return r.kept && !le_thresh(r.ub, r.id, T1); };
        if (a.pick_rule == 1) {
            // min-max scaling over the candidates' (non-NaN) lower bounds, then each candidate's race key
            float mn = INFINITY, mx = -INFINITY;
            each([&](int, int, const Row &r) {
                const float v = float_unorder(r.v2);
                if (cand(r) && v == v) {
                    mn = fminf(mn, v);
                    mx = fmaxf(mx, v);
                }
            });
            for (int o = 16; o > 0; o >>= 1) {
                mn = fminf(mn, __shfl_xor_sync(0xFFFFFFFFu, mn, o));
                mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));
            }
            if (lane == 0) {
                sh.wmn[warp] = mn;
                sh.wmx[warp] = mx;
            }
            __syncthreads();
            if (tid == 0) {
                for (int w = 1; w < kPlanThreads / 32; ++w) {
                    mn = fminf(mn, sh.wmn[w]);
                    mx = fmaxf(mx, sh.wmx[w]);
                }
                sh.mn = mn;
                sh.mx = mx;
            }
            sync();
            mn = INFINITY;
            mx = -INFINITY;
            for (int q = 0; q < C; ++q) {
                mn = fminf(mn, *of(&sh.mn, q));
                mx = fmaxf(mx, *of(&sh.mx, q));
            }
            each([&](int i, int it, const Row &r) {
                if (!cand(r)) return;
                float v = float_unorder(r.v2);
                v = v == v ? pick_key(v, mn, mx, a.temperature, a.pick_seed, r.id) : v;
                a.pick_keys[i] = v;
                if (ITEMS > 0) r_v2[it] = float_order(v);
            });
            race = true;
            __syncthreads();
        }
        T2 = select([](const Row &r) { return r.v2; }, cand, n_pick - n1);
    }

    // stable ranks of picked and unpicked survivors: the share's counts, the shares before it, then row by row
    auto picked = [&](const Row &r) { return r.kept && (all || le_thresh(r.ub, r.id, T1) || le_thresh(r.v2, r.id, T2)); };
    int cp = 0, cr = 0;
    each([&](int, int, const Row &r) {
        const bool pk = picked(r);
        cp += pk;
        cr += r.kept && !pk;
    });
    cp = block_sum(cp);
    cr = block_sum(cr);
    if (tid == 0) {
        sh.part[1][0] = cp;
        sh.part[1][1] = cr;
    }
    sync();
    int base_p = 0, base_r = 0, tp = 0, tr = 0;
    for (int q = 0; q < C; ++q) {
        const int *o = of(&sh.part[1][0], q);
        if (q < rank) {
            base_p += o[0];
            base_r += o[1];
        }
        tp += o[0];
        tr += o[1];
    }
    const unsigned lt = (1u << lane) - 1u;
    each([&](int i, int, const Row &r) {
        const bool pk = picked(r), rs = r.kept && !pk;
        const unsigned bp = __ballot_sync(0xFFFFFFFFu, pk), br = __ballot_sync(0xFFFFFFFFu, rs);
        if (lane == 0) {
            sh.wsum[0][warp] = __popc(bp);
            sh.wsum[1][warp] = __popc(br);
        }
        __syncthreads();
        // warp prefix of the warps' counts
        const int vp = sh.wsum[0][lane], vr = sh.wsum[1][lane];
        int ip = vp, ir = vr;
        for (int o = 1; o < 32; o *= 2) {
            const int xp = __shfl_up_sync(0xFFFFFFFFu, ip, o), xr = __shfl_up_sync(0xFFFFFFFFu, ir, o);
            if (lane >= o) {
                ip += xp;
                ir += xr;
            }
        }
        const int op = __shfl_sync(0xFFFFFFFFu, ip - vp, warp), orr = __shfl_sync(0xFFFFFFFFu, ir - vr, warp);
        if (i < i1) a.dest[i] = pk ? ((base_p + op + __popc(bp & lt)) | kPickFlag) : rs ? base_r + orr + __popc(br & lt) : -1;
        base_p += __shfl_sync(0xFFFFFFFFu, ip, 31);
        base_r += __shfl_sync(0xFFFFFFFFu, ir, 31);
        __syncthreads();
    });
    if (rank == 0 && tid == 0) plan_totals(a, tp, tr);
    sync();  // no CTA leaves while another may still read its shared memory
}

// Several problems: output offsets of each problem's children and unpicked rows, and the totals.
__global__ void k_branch_offsets(BranchArgs a)
{
    if (threadIdx.x != 0) return;
    const int P = a.batch.P;
    long long tp = 0, tr = 0;
    for (int p = 0; p < P; ++p) {
        tp += a.pcounts[2 * p];
        tr += a.pcounts[2 * p + 1];
    }
    long long cp = 0, cr = 2 * tp;
    for (int p = 0; p < P; ++p) {
        a.poff[2 * p] = (int)cp;
        a.poff[2 * p + 1] = (int)cr;
        cp += 2 * a.pcounts[2 * p];
        cr += a.pcounts[2 * p + 1];
    }
    if (2 * tp + tr > a.cap_out) set_status(a.status, BAB_ERR_SHAPE);  // rows beyond cap_out are dropped
    a.d_counts[0] = (int)(2 * tp);
    a.d_counts[1] = (int)tr;
    a.d_counts[2] = (int)(2 * tp + tr);
}

// VEC coordinates per lane (4: every row is 16-byte aligned), LPR lanes per row.
template <int VEC, int LPR>
__global__ void __launch_bounds__(256) k_branch_write(BranchArgs a)
{
    const int n = live_count(a.n, a.d_n);
    const int lane = threadIdx.x % LPR;
    const int row = blockIdx.x * (256 / LPR) + threadIdx.x / LPR;
    const unsigned group = LPR == 32 ? 0xFFFFFFFFu : ((1u << (LPR % 32)) - 1u) << ((threadIdx.x & 31) / LPR * LPR);
    if (row >= n) return;
    const int d = a.d;
    const float *lo = a.lo + (size_t)row * d, *hi = a.hi + (size_t)row * d;
    // one row's coordinates j .. j + VEC - 1
    struct Part {
        float v[VEC];
    };
    auto load = [](const float *p) {
        Part q;
        if (VEC == 4) {
            const float4 t = *reinterpret_cast<const float4 *>(p);
            q.v[0] = t.x;
            q.v[1 % VEC] = t.y;
            q.v[2 % VEC] = t.z;
            q.v[3 % VEC] = t.w;
        } else {
            q.v[0] = *p;
        }
        return q;
    };
    auto store = [](float *p, const Part &q) {
        if (VEC == 4) *reinterpret_cast<float4 *>(p) = make_float4(q.v[0], q.v[1 % VEC], q.v[2 % VEC], q.v[3 % VEC]);
        else *p = q.v[0];
    };
    const int j0 = lane * VEC;
    Part l0{}, h0{};
    if (j0 < d) {
        // (before the row's destination is known: few rows are pruned)
        l0 = load(lo + j0);
        h0 = load(hi + j0);
    }
    const int dst = a.dest[row];
    if (dst < 0) return;
    const int pb = row_problem(a.batch, row);
    const int dp = a.batch.H ? a.k * problem_H(a.batch, pb, 0) : d;  // coordinates the problem uses
    const uint64_t id = a.id[row];
    if (!(dst & kPickFlag)) {
        const size_t o = (size_t)a.poff[2 * pb + 1] + dst;
        if (o >= (size_t)a.cap_out) return;
        if (a.out_prob && lane == 0) a.out_prob[o] = pb;
        if (a.out_split_dim && lane == 0) a.out_split_dim[o] = a.split_dim ? a.split_dim[row] : -1;
        for (int j = j0; j < d; j += LPR * VEC) {
            store(a.out_lo + o * d + j, j == j0 ? l0 : load(lo + j));
            store(a.out_hi + o * d + j, j == j0 ? h0 : load(hi + j));
        }
        if (a.out_row_u)
            for (int j = j0; j < d; j += LPR * VEC) store(a.out_row_u + o * d + j, load(a.row_u + (size_t)row * d + j));
        if (lane == 0) {
            a.out_id[o] = id;
            a.out_lb[o] = a.lb[row];
            a.out_ub[o] = a.ub[row];
        }
        return;
    }
    // widest coordinate, lowest index on ties
    float wb = -1.f;
    int jb = 0x7FFFFFFF;
    const int given = a.split_dim ? a.split_dim[row] : -1;  // the sample-imbalance choice, when given
    if (!(given >= 0 && given < dp))
        for (int j = j0; j < dp; j += LPR * VEC) {
            const Part l = j == j0 ? l0 : load(lo + j), h = j == j0 ? h0 : load(hi + j);
#pragma unroll
            for (int e = 0; e < VEC; ++e) {
                const float w = __fsub_rn(h.v[e], l.v[e]);
                if (j + e < dp && w > wb) {
                    wb = w;
                    jb = j + e;
                }
            }
        }
    for (int o = LPR / 2; o > 0; o >>= 1) {
        const float w2 = __shfl_xor_sync(group, wb, o);
        const int j2 = __shfl_xor_sync(group, jb, o);
        if (w2 > wb || (w2 == wb && j2 < jb)) {
            wb = w2;
            jb = j2;
        }
    }
    if (given >= 0 && given < dp) jb = given;
    if (jb >= dp) jb = 0;  // a problem without coordinates (H_p = 0) splits nothing meaningful
    const float mid = __fmul_rn(0.5f, __fadd_rn(lo[jb], hi[jb]));
    const size_t o0 = (size_t)a.poff[2 * pb] + 2 * (size_t)(dst & ~kPickFlag);
    if (o0 + 1 >= (size_t)a.cap_out) return;
    if (a.out_prob && lane == 0) a.out_prob[o0] = a.out_prob[o0 + 1] = pb;
    if (a.out_split_dim && lane == 0) a.out_split_dim[o0] = a.out_split_dim[o0 + 1] = -1;
    for (int j = j0; j < d; j += LPR * VEC) {
        const Part l = j == j0 ? l0 : load(lo + j), h = j == j0 ? h0 : load(hi + j);
        Part lm = l, hm = h;
#pragma unroll
        for (int e = 0; e < VEC; ++e)
            if (j + e == jb) lm.v[e] = hm.v[e] = mid;
        store(a.out_lo + o0 * d + j, l);
        store(a.out_hi + o0 * d + j, hm);
        store(a.out_lo + (o0 + 1) * d + j, lm);
        store(a.out_hi + (o0 + 1) * d + j, h);
    }
    if (a.out_row_u)
        for (int j = j0; j < d; j += LPR * VEC) {
            const Part v = load(a.row_u + (size_t)row * d + j);
            store(a.out_row_u + o0 * d + j, v);
            store(a.out_row_u + (o0 + 1) * d + j, v);
        }
    if (lane == 0) {
        a.out_id[o0] = child_id(id, 0);
        a.out_id[o0 + 1] = child_id(id, 1);
        a.out_lb[o0] = a.out_lb[o0 + 1] = a.lb[row];
        a.out_ub[o0] = a.out_ub[o0 + 1] = a.ub[row];
    }
}

// The splitting heuristic of Section 3.1, one warp per box: the top_k samples of smallest (cost, m) (selected
// in increasing order, each the smallest key above the previous), their coordinates re-drawn from the counter
// sampler, per dimension the counts below / above the midpoint and the score (hi - lo) |n_lo - n_up|; the
// largest score (lowest j on ties), or the widest dimension when no dimension is imbalanced.
__global__ void __launch_bounds__(256) k_split_dims(int d, const float *lo, const float *hi, const uint64_t *id,
                                                    int n, const int *d_n, uint64_t seed, const float *costs, int M,
                                                    int top_k, int *split_dim)
{
    __shared__ int tops[8][64];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int box = blockIdx.x * 8 + wib;
    if (box >= live_count(n, d_n)) return;
    const float *c = costs + (size_t)box * M;
    unsigned long long prev = 0;
    for (int q = 0; q < top_k; ++q) {
        unsigned long long best = ~0ull;
        for (int m = lane; m < M; m += 32) {
            const unsigned long long key = ((unsigned long long)float_order(c[m]) << 32) | (unsigned)m;
            if ((q == 0 || key > prev) && key < best) best = key;
        }
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long other = __shfl_xor_sync(0xFFFFFFFFu, best, o);
            best = other < best ? other : best;
        }
        prev = best;
        if (lane == 0) tops[wib][q] = (int)(best & 0xFFFFFFFFu);
    }
    __syncwarp();
    const uint64_t hb = box_hash(seed, id[box]);
    const float *bl = lo + (size_t)box * d, *bh = hi + (size_t)box * d;
    float sb = 0.f;
    int jb = 0x7FFFFFFF;
    for (int j = lane; j < d; j += 32) {
        const float mid = __fmul_rn(0.5f, __fadd_rn(bl[j], bh[j]));
        int nlo = 0, nup = 0;
        for (int q = 0; q < top_k; ++q) {
            const float u = draw_sample(hb, (uint32_t)tops[wib][q], (uint32_t)j, bl[j], bh[j]);
            nlo += u <= mid;
            nup += u >= mid;
        }
        const float sc = __fmul_rn(__fsub_rn(bh[j], bl[j]), (float)abs(nlo - nup));
        if (sc > sb) {
            sb = sc;
            jb = j;
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        const float s2 = __shfl_xor_sync(0xFFFFFFFFu, sb, o);
        const int j2 = __shfl_xor_sync(0xFFFFFFFFu, jb, o);
        if (s2 > sb || (s2 == sb && j2 < jb)) {
            sb = s2;
            jb = j2;
        }
    }
    if (!(sb > 0.f)) {
        // no imbalance: the widest dimension, lowest index on ties
        float wb = -1.f;
        jb = 0x7FFFFFFF;
        for (int j = lane; j < d; j += 32) {
            const float w = __fsub_rn(bh[j], bl[j]);
            if (w > wb) {
                wb = w;
                jb = j;
            }
        }
        for (int o = 16; o > 0; o >>= 1) {
            const float w2 = __shfl_xor_sync(0xFFFFFFFFu, wb, o);
            const int j2 = __shfl_xor_sync(0xFFFFFFFFu, jb, o);
            if (w2 > wb || (w2 == wb && j2 < jb)) {
                wb = w2;
                jb = j2;
            }
        }
    }
    if (lane == 0) split_dim[box] = jb;
}

cudaError_t launch_split_dims(int d, const float *lo, const float *hi, const uint64_t *id, int n, const int *d_n,
                              uint64_t seed, const float *costs, int M, int top_k, int *split_dim, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    if (top_k < 1 || top_k > 64 || top_k > M) return cudaErrorInvalidValue;
    k_split_dims<<<(n + 7) / 8, 256, 0, st>>>(d, lo, hi, id, n, d_n, seed, costs, M, top_k, split_dim);
    return cudaGetLastError();
}

cudaError_t launch_prune_branch(const BranchArgs &a, cudaStream_t st)
{
    if (a.batch.P > 1) {
        k_branch_plan<<<a.batch.P, kPlanThreads, 0, st>>>(a);
        k_branch_offsets<<<1, 32, 0, st>>>(a);
    } else if (a.n <= kSmallPlan) {
        k_branch_plan_small<<<1, kSmallPlan, 0, st>>>(a);
    } else {
        // a CTA per 2048 rows (two a thread), at most kPlanCTAs
        int C = 1;
        while (C < kPlanCTAs && C * 2 * kPlanThreads < a.n) C *= 2;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)C);
        cfg.blockDim = dim3(kPlanThreads);
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)C;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        cudaError_t e = a.n <= C * kPlanItems * kPlanThreads ? cudaLaunchKernelEx(&cfg, k_branch_plan_cl<kPlanItems>, a)
                                                             : cudaLaunchKernelEx(&cfg, k_branch_plan_cl<0>, a);
        if (e != cudaSuccess) return e;
    }
    if (a.n > 0) {
        // rows of whole, aligned 16-byte words: the fewest lanes (8, 16 or 32) that take a row in one pass; else a warp a
        // row, a coordinate a lane
        auto al = [](const void *p) { return ((uintptr_t)p & 15) == 0; };
        const bool vec = a.d % 4 == 0 && al(a.lo) && al(a.hi) && al(a.out_lo) && al(a.out_hi) && al(a.row_u) && al(a.out_row_u);
        auto run = [&](auto kern, int lpr) { kern<<<(a.n + 256 / lpr - 1) / (256 / lpr), 256, 0, st>>>(a); };
        if (!vec) run(k_branch_write<1, 32>, 32);
        else if (a.d <= 32) run(k_branch_write<4, 8>, 8);
        else if (a.d <= 64) run(k_branch_write<4, 16>, 16);
        else run(k_branch_write<4, 32>, 32);
    }
    return cudaGetLastError();
}

}  // namespace bab
