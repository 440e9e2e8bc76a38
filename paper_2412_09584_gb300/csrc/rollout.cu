// rollout.cu -- sampled search (Section 3.3, batch_search with uniform samples)
// and the FP64 incumbent re-score (the incumbent update of Algorithm 2).
//
// k_rollout_fp32 (batched problems and search-integrated bounds; the other FP32
// rollouts are rollout_rows.cu's): a persistent kernel.  A tile is R samples of one box; a CTA
// keeps the whole forward network image in shared memory for all H steps and
// all of its tiles, and carries the R states x_t and running costs in shared
// memory.  Per step it draws u_t (counter-based, so nothing is read from
// memory), runs the L dense layers as register-blocked FP32 products over the
// tile, adds the residual, and reduces the per-row cost with warp shuffles.
// A tile's best (f, m) is folded into its box with a 64-bit atomicMin on
// (order(f) << 32 | m), which keeps the lowest m among equal values.
#include <atomic>

#include <cooperative_groups.h>

#include "bab_internal.cuh"
#include "kernels.cuh"

namespace bab {

__device__ __forceinline__ unsigned long long umin64(unsigned long long a, unsigned long long b) { return a < b ? a : b; }

template <int R, int NT, bool WSMEM, int MINB>
__global__ void __launch_bounds__(NT, MINB) k_rollout_fp32(RolloutArgs a)
{
    extern __shared__ float4 smem4[];
    float *sm = reinterpret_cast<float *>(smem4);
    const NetDesc &N = a.net;
    const int s = N.s, k = N.k, L = N.L, d = a.d;
    const int ld = N.maxw_p;
    const float *img = a.fwd;
    float *p = sm;
    if (WSMEM) {
        for (int i = threadIdx.x; i < N.img_floats / 4; i += NT)
            smem4[i] = reinterpret_cast<const float4 *>(a.fwd)[i];
        img = sm;
        p += N.img_floats;
    }
    float *act0 = p; p += R * ld;
    float *act1 = p; p += R * ld;
    float *xs = p; p += R * pad4(s);
    float *us = p; p += R * pad4(k);
    float *blo = p; p += pad4(d);
    float *bhi = p; p += pad4(d);
    float *cost = p; p += R;
    float *goal = p; p += pad4(s);
    float *ps = p; p += 2 * R;  // pusher position per row (obstacle cost)
    __shared__ unsigned long long red[NT / 32];

    const int nlive = live_count(a.n, a.d_n);
    const int tpb = (a.M + R - 1) / R;
    const long long ntiles = (long long)nlive * tpb;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int Kp1 = pad4(s + k);
    const bool emit = a.emp_pre_lo != nullptr;
    const int Hm = a.batch.Hmax;

    for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int box = (int)(tile / tpb);
        const int m0 = (int)(tile % tpb) * R;
        const int rv = a.M - m0 < R ? a.M - m0 : R;  // rows holding real samples
        // the box's problem: its weights, start, goal, horizon and rho
        const int pb = row_problem(a.batch, box);
        if (!WSMEM) img = a.fwd + (size_t)pb * N.img_floats;
        const int Hb = problem_H(a.batch, pb, a.H), db = k * Hb;
        const float rho = problem_rho(a.batch, pb, a.rho);
        const float *x0 = a.x0 + (size_t)pb * s;
        __syncthreads();  // previous tile fully consumed
        for (int i = threadIdx.x; i < s; i += NT) goal[i] = a.goal[(size_t)pb * s + i];
        for (int j = threadIdx.x; j < db; j += NT) {
            blo[j] = a.lo[(size_t)box * d + j];
            bhi[j] = a.hi[(size_t)box * d + j];
        }
        for (int i = threadIdx.x; i < R * s; i += NT) xs[(i / s) * pad4(s) + i % s] = x0[i % s];
        for (int r = threadIdx.x; r < R; r += NT) {
            cost[r] = 0.f;
            ps[2 * r] = a.cost.p0x;
            ps[2 * r + 1] = a.cost.p0y;
        }
        const uint64_t hb = box_hash(a.seed, a.id[box]);
        __syncthreads();
        for (int t = 0; t < Hb; ++t) {
            // input rows [x_t | u_t | 0]
            for (int i = threadIdx.x; i < R * Kp1; i += NT) {
                const int r = i / Kp1, c = i % Kp1;
                float v;
                if (c < s) {
                    v = xs[r * pad4(s) + c];
                } else if (c < s + k) {
                    const int j = t * k + (c - s);
                    v = a.cem_mu ? cem_sample(hb, (uint32_t)a.cem_it, (uint32_t)(m0 + r), (uint32_t)j,
                                              a.cem_mu[(size_t)box * d + j], a.cem_sigma[(size_t)box * d + j], blo[j],
                                              bhi[j])
                                 : draw_sample(hb, (uint32_t)(m0 + r), (uint32_t)j, blo[j], bhi[j]);
                    us[r * pad4(k) + (c - s)] = v;
                } else {
                    v = 0.f;
                }
                act0[r * ld + c] = v;
            }
            __syncthreads();
            float *in = act0, *out = act1;
            for (int l = 1; l <= L; ++l) {
                const int Kp = pad4(N.dims[l - 1]), Np = pad4(N.dims[l]);
                dense_rows_auto<R, NT>(in, ld, img + N.fwd_w[l], img + N.fwd_b[l], Kp, Np, out, ld, l < L && !emit);
                __syncthreads();
                if (emit && l < L) {
                    // search-integrated bounds: the tile's extremes of each pre-activation, then the ReLU
                    const int dl = N.dims[l];
                    for (int c = threadIdx.x; c < Np; c += NT) {
                        float mn = INFINITY, mx = -INFINITY;
                        for (int r = 0; r < R; ++r) {
                            const float v = out[r * ld + c];
                            if (r < rv) {
                                mn = fminf(mn, v);
                                mx = fmaxf(mx, v);
                            }
                            out[r * ld + c] = fmaxf(v, 0.f);
                        }
                        if (c < dl) {
                            const size_t e = ((size_t)box * Hm + t) * N.sumh + N.hoff[l] + c;
                            atomicMin(&a.emp_pre_lo[e], float_order(mn));
                            atomicMax(&a.emp_pre_hi[e], float_order(mx));
                        }
                    }
                    __syncthreads();
                }
                float *tmp = in; in = out; out = tmp;
            }
            // `in` holds the network output: residual step and the step cost of each row (one thread per row,
            // state terms then action terms in index order, so the value has a plain sequential definition)
            for (int r = threadIdx.x; r < R; r += NT) {
                float c = 0.f;
                if (a.cost.kind == 0) {
                    for (int i = 0; i < s; ++i) {
                        const float x = xs[r * pad4(s) + i] + in[r * ld + i];
                        xs[r * pad4(s) + i] = x;
                        const float e = x - goal[i];
                        c = fmaf(e, e, c);
                    }
                } else {
                    // the pusher moves by u_t, then the state cost at t + 1 (Appendix D.4)
                    ps[2 * r] = __fadd_rn(ps[2 * r], us[r * pad4(k)]);
                    ps[2 * r + 1] = __fadd_rn(ps[2 * r + 1], us[r * pad4(k) + 1]);
                    for (int i = 0; i < s; ++i) xs[r * pad4(s) + i] = __fadd_rn(xs[r * pad4(s) + i], in[r * ld + i]);
                    c = obstacle_cost_f32(a.cost, t + 1, s, xs + r * pad4(s), goal, ps[2 * r], ps[2 * r + 1]);
                }
                for (int j = 0; j < k; ++j) {
                    const float u = us[r * pad4(k) + j];
                    c = fmaf(rho * u, u, c);
                }
                cost[r] += c;
            }
            __syncthreads();
            if (emit) {
                // search-integrated bounds of the state x_{t+1}
                for (int i = threadIdx.x; i < s; i += NT) {
                    float mn = INFINITY, mx = -INFINITY;
                    for (int r = 0; r < rv; ++r) {
                        const float v = xs[r * pad4(s) + i];
                        mn = fminf(mn, v);
                        mx = fmaxf(mx, v);
                    }
                    const size_t e = ((size_t)box * (Hm + 1) + t + 1) * s + i;
                    atomicMin(&a.emp_x_lo[e], float_order(mn));
                    atomicMax(&a.emp_x_hi[e], float_order(mx));
                }
            }
        }
        if (a.costs)
            for (int r = threadIdx.x; r < rv; r += NT) a.costs[(size_t)box * a.M + m0 + r] = cost[r];
        // best (f, m) of the tile
        unsigned long long best = ~0ull;
        for (int r = threadIdx.x; r < R; r += NT)
            if (m0 + r < a.M) best = umin64(best, ((unsigned long long)float_order(cost[r]) << 32) | (unsigned)(m0 + r));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) best = umin64(best, __shfl_xor_sync(0xFFFFFFFFu, best, o));
        if (lane == 0) red[warp] = best;
        __syncthreads();
        if (threadIdx.x == 0) {
            unsigned long long b = red[0];
            for (int w = 1; w < NT / 32; ++w) b = umin64(b, red[w]);
            atomicMin(&a.keys[box], b);
        }
    }
}

__global__ void k_fill_u64(unsigned long long *p, int n, unsigned long long v)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) p[i] = v;
}

// ub[i] and best_u[i] from the packed per-box minimum; the argmin sample is re-drawn.
__global__ void k_rollout_finalize(RolloutArgs a)
{
    const int nlive = live_count(a.n, a.d_n);
    const int box = blockIdx.x;
    if (box >= nlive) return;
    const unsigned long long key = a.keys[box];
    const uint32_t m = (uint32_t)(key & 0xFFFFFFFFu);
    if (threadIdx.x == 0) a.ub[box] = float_unorder((uint32_t)(key >> 32));
    if (!a.best_u) return;
    const uint64_t hb = box_hash(a.seed, a.id[box]);
    const int db = a.net.k * problem_H(a.batch, row_problem(a.batch, box), a.H);
    for (int j = threadIdx.x; j < a.d; j += blockDim.x)
        a.best_u[(size_t)box * a.d + j] =
            j < db ? draw_sample(hb, m, (uint32_t)j, a.lo[(size_t)box * a.d + j], a.hi[(size_t)box * a.d + j]) : 0.f;
}

// Incumbent update: the box with the smallest ub (lowest index on ties) has its best_u re-evaluated in FP64; if the
// value beats *inc_val, it becomes the incumbent.  One row is a chain of H x L layers, so what bounds it is the FP64
// rate of the SMs it runs on (two multiply-adds per clock each) and, once that is spread, each layer's latency.  A
// cluster of kIncCTAs CTAs shares every layer's outputs (one CTA for the smallest networks): each CTA keeps its rows of
// every layer's weights in shared memory as doubles for all steps, an output's sum is split over ks lanes (strided over
// the inputs, added by shuffles), lane by lane written into the CTAs' shared memory (distributed shared memory), and
// one cluster barrier closes the layer.  The outputs alternate between two buffers without restarting at a step: a CTA
// at most one layer ahead then writes the buffer that nobody reads.  The control flow depends only on values every CTA
// of the cluster computes alike, so all of them reach the same barriers.
// Pushing network (20 steps): 603 -> 146 us (one CTA before); object manipulation (40 steps): 1136 -> 488 us (the
// weights read from L2 at every step before); tiny network (5 steps), one CTA: 39 -> 28 us.
constexpr int kIncCTAs = 16;  // a non-portable cluster size; 8 where the GPU cannot place 16
constexpr int kIncThreads = 256;
constexpr int kIncActions = 1024;  // action coordinates kept in shared memory (a longer plan is read as it goes)

// Lanes per output of a layer with ni inputs of which a CTA computes `chunk` outputs: the power of two that takes the
// fewest clocks.  A warp's FP64 instruction holds the SM's FP64 unit for 16 clocks (and a warp waits longer than that
// for its own result), the additions across lanes like the multiply-adds, so few lanes are best.
__host__ __device__ inline int incumbent_lanes(int chunk, int ni)
{
    int best = 1, cost = 1 << 30;
    for (int ks = 1, lg = 0; ks <= 32 && chunk * ks <= kIncThreads; ks *= 2, ++lg) {
        const int warps = (chunk * ks + 31) / 32, c = ((ni + ks - 1) / ks + 4 + lg) * (warps > 2 ? 16 * warps : 40);
        if (c < cost) {
            cost = c;
            best = ks;
        }
    }
    return best;
}

// The same where the weights are read through L2: two at least, so that a warp's load touches fewer rows (128 problems of
// the pushing network, one CTA each, 20 steps: one lane 1301 us, two 1164).
__host__ __device__ inline int incumbent_lanes_l2(int chunk, int ni)
{
    const int ks = incumbent_lanes(chunk, ni);
    return ks == 1 && 2 * chunk <= kIncThreads ? 2 : ks;
}

// doubles of shared memory a CTA of a cluster of ncta needs: its rows of every layer's weights (ni + lanes apart, so
// that the outputs of a warp read different banks) and their biases
__host__ __device__ inline size_t incumbent_doubles(const NetDesc &N, int ncta)
{
    size_t f = 0;
    for (int l = 1; l <= N.L; ++l) {
        const int chunk = (N.dims[l] + ncta - 1) / ncta;
        f += (size_t)chunk * (N.dims[l - 1] + incumbent_lanes(chunk, N.dims[l - 1]) + 1);
    }
    return f;
}

// WSMEM: the CTA's rows fit in shared memory (else they are read through L2).
template <bool WSMEM>
__global__ void __launch_bounds__(kIncThreads) k_incumbent_fp64(RolloutArgs a)
{
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank(), ncta = (int)cluster.num_blocks();
    const NetDesc &N = a.net;
    const int nlive = live_count(a.n, a.d_n);
    // one cluster per problem: its rows, weights, start, goal, horizon, rho and incumbent
    const int pb = blockIdx.x / ncta;
    const float *raw = a.raw + (size_t)pb * N.raw_floats;
    const float *x0 = a.x0 + (size_t)pb * N.s, *goal = a.goal + (size_t)pb * N.s;
    const int Hb = problem_H(a.batch, pb, a.H);
    const float rho = problem_rho(a.batch, pb, a.rho);
    double *inc_val = a.inc_val + pb;
    float *inc_u = a.inc_u + (size_t)pb * a.d;
    extern __shared__ double wsh[];  // WSMEM: per layer this CTA's rows [chunk][ni], then their biases [chunk]
    __shared__ unsigned long long red[kIncThreads / 32];
    __shared__ double act[2][kMaxWidth];
    __shared__ double xin[kMaxWidth], xs[kMaxWidth], gl[kMaxWidth];
    __shared__ float us[kIncActions];
    __shared__ double f_sh;
    __shared__ int row_sh, ks_sh[kMaxLayers + 1];
    const int lane = threadIdx.x & 31;
    if (threadIdx.x >= 1 && (int)threadIdx.x <= N.L) {
        const int chunk = (N.dims[threadIdx.x] + ncta - 1) / ncta;
        ks_sh[threadIdx.x] = WSMEM ? incumbent_lanes(chunk, N.dims[threadIdx.x - 1]) : incumbent_lanes_l2(chunk, N.dims[threadIdx.x - 1]);
    }
    unsigned long long best = ~0ull;
#pragma unroll 8
    for (int i = threadIdx.x; i < nlive; i += kIncThreads)
        if (row_problem(a.batch, i) == pb)
            best = umin64(best, ((unsigned long long)float_order(a.ub[i]) << 32) | (unsigned)i);
    if (WSMEM) {
        double *w = wsh;
        for (int l = 1; l <= N.L; ++l) {
            const int no = N.dims[l], ni = N.dims[l - 1], chunk = (no + ncta - 1) / ncta, q0 = rank * chunk;
            const int mine = min(chunk, no - q0), ldw = ni + incumbent_lanes(chunk, ni);  // (mine may be <= 0)
#pragma unroll 4
            for (int i = threadIdx.x; i < mine * ni; i += kIncThreads) {
                const int r = i / ni;
                w[r * ldw + (i - r * ni)] = (double)raw[N.raw_w[l] + (size_t)q0 * ni + i];
            }
            w += chunk * ldw;
            for (int i = threadIdx.x; i < mine; i += kIncThreads) w[i] = (double)raw[N.raw_b[l] + q0 + i];
            w += chunk;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) best = umin64(best, __shfl_xor_sync(0xFFFFFFFFu, best, o));
    if (lane == 0) red[threadIdx.x >> 5] = best;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long b = red[0];
        for (int w = 1; w < kIncThreads / 32; ++w) b = umin64(b, red[w]);
        row_sh = (b == ~0ull) ? -1 : (int)(b & 0xFFFFFFFFu);
        f_sh = 0.0;
    }
    __syncthreads();
    const int row = row_sh;
    if (row < 0) return;  // the same in every CTA of the cluster
    const float *u = a.best_u + (size_t)row * a.d;
    const int s = N.s, k = N.k;
    double px = (double)a.cost.p0x, py = (double)a.cost.p0y;  // pusher position (obstacle cost; lane 0)
    double f = 0.0;  // the first warp's partial sums of the objective, added up at the end
    const bool u_sh = Hb * k <= kIncActions;
    if (u_sh)
        for (int j = threadIdx.x; j < Hb * k; j += kIncThreads) us[j] = u[j];
    for (int i = threadIdx.x; i < s; i += kIncThreads) gl[i] = (double)goal[i];
    for (int i = threadIdx.x; i < s; i += kIncThreads) xs[i] = (double)x0[i];
    for (int c = threadIdx.x; c < s + k; c += kIncThreads) xin[c] = c < s ? (double)x0[c] : (Hb > 0 ? (double)u[c - s] : 0.0);
    if (ncta > 1) cluster.sync();  // every CTA of the cluster runs before its shared memory is written
    else __syncthreads();
    int cur = 0;  // the buffer the next layer writes
    for (int t = 0; t < Hb; ++t) {
        const double *w = wsh;
        for (int l = 1; l <= N.L; ++l) {
            const int no = N.dims[l], ni = N.dims[l - 1];
            const double *in = l == 1 ? xin : act[cur ^ 1];
            // this CTA's outputs q0 .. q0 + chunk - 1 (chunk <= 256, the widest layer), ks lanes each
            const int chunk = (no + ncta - 1) / ncta, q0 = rank * chunk;
            const int ks = ks_sh[l], ldw = ni + ks;
            const int ql = (int)threadIdx.x / ks, sl = (int)threadIdx.x % ks, q = q0 + ql;
            const bool mine = ql < chunk && q < no;
            if (((int)threadIdx.x & ~31) < chunk * ks) {  // (whole warps)
                double pt[4] = {0.0, 0.0, 0.0, 0.0};
                if (mine) {
                    if (WSMEM) {
                        const double *wq = w + ql * ldw;
                        int c = sl;
                        for (; c + 3 * ks < ni; c += 4 * ks)
#pragma unroll
                            for (int e = 0; e < 4; ++e) pt[e] = fma(wq[c + e * ks], in[c + e * ks], pt[e]);
                        for (; c < ni; c += ks) pt[0] = fma(wq[c], in[c], pt[0]);
                    } else {
                        const float *wq = raw + N.raw_w[l] + (size_t)q * ni;
#pragma unroll 4
                        for (int c = sl; c < ni; c += ks) pt[0] = fma((double)wq[c], in[c], pt[0]);
                    }
                }
                double part = (pt[0] + pt[1]) + (pt[2] + pt[3]);
                for (int o = ks / 2; o > 0; o >>= 1) part += __shfl_xor_sync(0xFFFFFFFFu, part, o);
                if (mine) {
                    double v = (WSMEM ? w[chunk * ldw + ql] : (double)raw[N.raw_b[l] + q]) + part;
                    if (l < N.L && v < 0.0) v = 0.0;
                    // (every lane of the output holds the sum: lane r2 writes CTA r2's copy)
                    if (ncta == 1) {
                        if (sl == 0) act[cur][q] = v;
                    } else {
                        for (int r2 = sl; r2 < ncta; r2 += ks) cluster.map_shared_rank(&act[cur][0], r2)[q] = v;
                    }
                }
            }
            w += chunk * (ldw + 1);
            if (ncta > 1) cluster.sync();  // every CTA's copy of the layer output complete
            else __syncthreads();
            cur ^= 1;
        }
        // x_{t+1}, its cost and the next input row (every CTA its own copy)
        const double *z = act[cur ^ 1];
        if (threadIdx.x < 32) {
            for (int i = lane; i < s; i += 32) {
                const double x = xs[i] + z[i];
                xs[i] = x;
                xin[i] = x;
                if (a.cost.kind == 0) {
                    const double e = x - gl[i];
                    f = fma(e, e, f);
                }
            }
            for (int j = lane; j < k; j += 32) {
                const double uu = (double)(u_sh ? us[t * k + j] : u[t * k + j]);
                f = fma((double)rho * uu, uu, f);
            }
            if (a.cost.kind != 0) {
                __syncwarp();
                if (lane == 0) {
                    px += (double)u[t * k];
                    py += (double)u[t * k + 1];
                    f += obstacle_cost_f64(a.cost, t + 1, s, xs, goal, px, py);
                }
            }
        } else if (t + 1 < Hb) {
            for (int j = (int)threadIdx.x - 32; j < k; j += kIncThreads - 32)
                xin[s + j] = (double)(u_sh ? us[(t + 1) * k + j] : u[(t + 1) * k + j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) f += __shfl_xor_sync(0xFFFFFFFFu, f, o);
    if (rank != 0) return;
    if (threadIdx.x == 0) {
        f_sh = f;
        row_sh = (f < *inc_val) ? 1 : 0;
    }
    __syncthreads();
    if (row_sh) {
        for (int j = threadIdx.x; j < a.d; j += kIncThreads) inc_u[j] = u[j];
        if (threadIdx.x == 0) *inc_val = f_sh;
    }
}

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------
static size_t rollout_smem_bytes(const NetDesc &N, int R, int d, bool wsmem)
{
    size_t f = (wsmem ? (size_t)N.img_floats : 0) + 2 * (size_t)R * N.maxw_p + (size_t)R * pad4(N.s) +
               (size_t)R * pad4(N.k) + 2 * (size_t)pad4(d) + R + pad4(N.s) + 2 * (size_t)R;
    return f * sizeof(float);
}

template <int R, int NT, int MINB>
static cudaError_t launch_fp32_variant(const RolloutArgs &a, int num_sms, size_t budget, cudaStream_t st)
{
    // several problems: every tile reads its own problem's image through L1 / L2
    bool wsmem = a.batch.P <= 1 && rollout_smem_bytes(a.net, R, a.d, true) <= budget;
    size_t smem = rollout_smem_bytes(a.net, R, a.d, wsmem);
    if (smem > budget) return cudaErrorInvalidConfiguration;
    auto kern = wsmem ? k_rollout_fp32<R, NT, true, MINB> : k_rollout_fp32<R, NT, false, MINB>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int occ = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, NT, smem);
    if (e != cudaSuccess) return e;
    if (occ < 1) return cudaErrorInvalidConfiguration;
    const long long ntiles = (long long)a.n * ((a.M + R - 1) / R);
    const long long slots = (long long)num_sms * occ;
    const int grid = (int)(ntiles < slots ? ntiles : slots);
    kern<<<grid, NT, smem, st>>>(a);
    return cudaGetLastError();
}

int rollout_fp32_variants() { return 3; }

// variant 0: 64 samples x 256 threads per CTA, one CTA per SM (large networks, weights in shared memory); for one
// problem without search-integrated bounds k_rollout_rows;
// variant 1: 64 x 256 with at most 128 registers (two or more CTAs per SM for small networks);
// variant 2: 32 x 128, at most 128 registers.
cudaError_t launch_rollout_fp32(const RolloutArgs &a, int variant, int num_sms, cudaStream_t st)
{
    int dev;
    cudaGetDevice(&dev);
    int max_optin = 0;
    cudaDeviceGetAttribute(&max_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    const size_t budget = (size_t)max_optin - 1024;  // room for static shared memory
    // the register-tiled kernel unless another variant is set (512 boxes x 1024 samples x 20 steps of the pushing
    // network: 13.9 ms against 30.5 for the per-box tiles)
    const bool rows = variant <= 0 && rollout_rows_supported(a, budget);
    if (rollout_smem_bytes(a.net, 64, a.d, false) > budget) return cudaErrorInvalidConfiguration;
    if (a.n <= 0) return cudaSuccess;
    if (variant < 0) {
        // default: the register-capped variant once two CTAs' shared memory fits on an SM
        variant = rollout_smem_bytes(a.net, 64, a.d, true) * 2 + 2048 <= (size_t)max_optin ? 1 : 0;
    }
    k_fill_keys(a.keys, a.n, st);
    cudaError_t e;
    if (rows) e = launch_rollout_rows(a, num_sms, budget, st);
    else switch (variant) {
        case 1: e = launch_fp32_variant<64, 256, 2>(a, num_sms, budget, st); break;
        case 2: e = launch_fp32_variant<32, 128, 4>(a, num_sms, budget, st); break;
        default: e = launch_fp32_variant<64, 256, 1>(a, num_sms, budget, st); break;
    }
    if (e != cudaSuccess) return e;
    if (a.cem_mu) return cudaGetLastError();  // the cross-entropy search keeps its own best (launch_cem_step)
    launch_rollout_finalize(a, st);
    if (a.inc_val && (e = launch_incumbent(a, st)) != cudaSuccess) return e;
    return cudaGetLastError();
}

// Search-integrated bounds: key arrays start at the identities of min / max; after the rollout the keys turn
// back into floats in place, and x_0 (known exactly) is written.
__global__ void k_emp_init(uint32_t *lo, uint32_t *hi, long long n)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        lo[i] = 0xFFFFFFFFu;
        hi[i] = 0u;
    }
}

__global__ void k_emp_finish(uint32_t *lo, uint32_t *hi, long long n)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        lo[i] = __float_as_uint(float_unorder(lo[i]));
        hi[i] = __float_as_uint(float_unorder(hi[i]));
    }
}

__global__ void k_emp_x0(const RolloutArgs a)
{
    const int nlive = live_count(a.n, a.d_n), s = a.net.s, Hm = a.batch.Hmax;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < (long long)nlive * s;
         i += (long long)gridDim.x * blockDim.x) {
        const long long box = i / s;
        const int c = (int)(i % s);
        const float v = a.x0[(size_t)row_problem(a.batch, (int)box) * s + c];
        a.emp_x_lo[(size_t)box * (Hm + 1) * s + c] = __float_as_uint(v);
        a.emp_x_hi[(size_t)box * (Hm + 1) * s + c] = __float_as_uint(v);
    }
}

void launch_emp_init(const RolloutArgs &a, cudaStream_t st)
{
    const long long nh = (long long)a.n * a.batch.Hmax * a.net.sumh, nx = (long long)a.n * (a.batch.Hmax + 1) * a.net.s;
    if (nh > 0) k_emp_init<<<1024, 256, 0, st>>>(a.emp_pre_lo, a.emp_pre_hi, nh);
    k_emp_init<<<1024, 256, 0, st>>>(a.emp_x_lo, a.emp_x_hi, nx);
}

void launch_emp_finish(const RolloutArgs &a, cudaStream_t st)
{
    const long long nh = (long long)a.n * a.batch.Hmax * a.net.sumh, nx = (long long)a.n * (a.batch.Hmax + 1) * a.net.s;
    if (nh > 0) k_emp_finish<<<1024, 256, 0, st>>>(a.emp_pre_lo, a.emp_pre_hi, nh);
    k_emp_finish<<<1024, 256, 0, st>>>(a.emp_x_lo, a.emp_x_hi, nx);
    k_emp_x0<<<256, 256, 0, st>>>(a);
}

void k_fill_keys(unsigned long long *keys, int n, cudaStream_t st)
{
    if (n > 0) k_fill_u64<<<(n + 255) / 256, 256, 0, st>>>(keys, n, ~0ull);
}

void launch_rollout_finalize(const RolloutArgs &a, cudaStream_t st)
{
    if (a.n > 0) k_rollout_finalize<<<a.n, 128, 0, st>>>(a);
}

// The most shared memory the incumbent kernel takes.
constexpr size_t kIncMaxSmem = 200 * 1024;

// The kernel's attributes on the current device (the same for every launch, so that threads do not undo each other's) and
// a launch of `blocks` CTAs in clusters of ncta.
template <bool WSMEM>
static cudaError_t incumbent_config(int ncta, int blocks, size_t smem, cudaStream_t st, cudaLaunchConfig_t &cfg,
                                    cudaLaunchAttribute &attr)
{
    cudaError_t e = cudaSuccess;
    if (WSMEM)
        e = cudaFuncSetAttribute(k_incumbent_fp64<WSMEM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kIncMaxSmem);
    if (e == cudaSuccess && ncta > 8)
        e = cudaFuncSetAttribute(k_incumbent_fp64<WSMEM>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(kIncThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)ncta;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return e;
}

template <bool WSMEM>
static bool incumbent_placed(int ncta, size_t smem)
{
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr;
    int nclusters = 0;
    const bool ok = incumbent_config<WSMEM>(ncta, ncta, smem, nullptr, cfg, attr) == cudaSuccess &&
                    cudaOccupancyMaxActiveClusters(&nclusters, k_incumbent_fp64<WSMEM>, &cfg) == cudaSuccess && nclusters >= 1;
    if (!ok) cudaGetLastError();
    return ok;
}

template <bool WSMEM>
static cudaError_t incumbent_run(const RolloutArgs &a, int ncta, size_t smem, cudaStream_t st)
{
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr;
    const cudaError_t e = incumbent_config<WSMEM>(ncta, ncta * (a.batch.P > 1 ? a.batch.P : 1), smem, st, cfg, attr);
    return e != cudaSuccess ? e : cudaLaunchKernelEx(&cfg, k_incumbent_fp64<WSMEM>, a);
}

// Whether the current device places a 16-CTA cluster (non-portable size) with the most shared memory the kernel takes:
// asked at a device's first launch, which runs eagerly before any graph capture.
static bool incumbent_wide()
{
    constexpr int kDevices = 64;
    static std::atomic<int> known[kDevices];  // 0: not asked, 1: no, 2: yes
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevices) return false;
    int k = known[dev].load();
    if (k == 0) {
        k = incumbent_placed<true>(kIncCTAs, kIncMaxSmem) && incumbent_placed<false>(kIncCTAs, 0) ? 2 : 1;
        known[dev].store(k);
    }
    return k == 2;
}

cudaError_t launch_incumbent(const RolloutArgs &a, cudaStream_t st)
{
    if (a.n <= 0) return cudaSuccess;
    // One CTA where a step is at most 4096 multiply-adds (2048 clocks of one SM's FP64 rate, about the layers' cluster
    // barriers); else a cluster of kIncCTAs, or of 8 where the GPU does not place 16.  Several problems run side by side,
    // and their clusters share the SMs: a cluster each for up to 64 problems (32 with one step) of more than 512 P
    // multiply-adds a step.
    // Measured, cluster against one CTA, 20 steps: pushing network 2 problems 774 to 1279 us, 64 1038 to 1298, 128 1394
    // to 1301; 160 and 128 wide, 32 problems 643 to 711, 64 795 to 711; two 64-wide layers, 8 problems 318 to 316, 16 332
    // to 316; two 256-wide layers, 64 problems 2126 to 2515, 128 2585 to 2543.
    const NetDesc &N = a.net;
    long long macs = 0;
    for (int l = 1; l <= N.L; ++l) macs += (long long)N.dims[l] * N.dims[l - 1];
    const bool several = a.batch.P > 1;
    int ncta = macs > 4096 && (!several || (a.batch.P <= (a.H > 1 ? 64 : 32) && macs > 512LL * a.batch.P)) ? kIncCTAs : 1;
    if (ncta > 8 && !incumbent_wide()) ncta = 8;
    // Few steps are not worth the copy of the weights: of one CTA a single step, of several problems' CTAs one or two (512
    // problems of two 64-wide layers: one step 88 us with, 77 without; five steps 238 and 239), of several problems'
    // clusters a single one (8 such problems: 45.4 and 43.3 us; two steps 59.7 both).
    const int few = ncta == 1 ? (several ? 2 : 1) : (several ? 1 : 0);
    const size_t smem = incumbent_doubles(N, ncta) * sizeof(double);
    if (smem <= kIncMaxSmem && a.H > few) return incumbent_run<true>(a, ncta, smem, st);
    return incumbent_run<false>(a, ncta, 0, st);
}

}  // namespace bab
