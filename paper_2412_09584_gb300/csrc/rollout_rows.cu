// rollout_rows.cu -- the FP32 sampled search of one problem (Section 3.3, batch_search) with register tiles.
//
// k_rollout_rows is persistent: a tile is 64 consecutive samples of the call's n x M (so a tile may hold samples of
// several boxes, and a call with few samples per box fills its rows), owned by a group of warps with its own
// activation buffer and barriers.  The network image sits in shared memory for all steps and tiles, read by two
// groups of four warps (widths up to 128), or by one group of eight (wider layers; an image that does not fit is
// copied through a ring of spans ahead of its use).  Per layer every warp computes one block of the tile's outputs:
// lane (rg, cg) = (lane / 8, lane % 8) holds rows rg, rg + 4, .. and columns 4 cg .. 4 cg + 3 (and + 32) of it, two
// columns per FMA pair; the outputs stay in registers until the group has read its inputs, so one buffer serves
// every layer.
//
// What bounds it: FP32 FMAs, and the issue slots beside them.  Per input k a warp of 8 x 8 tiles issues 32 FMA pairs
// (64 cycles of its scheduler) and four 16-byte loads a lane; the former per-box tiles (4 x 8, weights read at a stride
// of two 16-byte words) spent more wavefronts of shared memory than cycles of FMAs.  Two groups, so that one's
// barriers, sample draws and costs run under the other's products.  512 boxes x 1024 samples x 20 steps of the pushing
// network: 30.5 -> 13.9 ms, 53 TFLOP/s of the 80 that FP32 FMAs reach (FMA pipe busy 71% of the cycles, shared memory
// 58%); 64 boxes x 256 samples x 5 steps of the tiny one: 32 -> 17 us.
//
// Every output is the FMA chain over the inputs in order from the bias, the cost the chain of its terms in order, as
// in k_rollout_fp32: the values are bit-identical.
#include "bab_internal.cuh"
#include "kernels.cuh"

namespace bab {

namespace {

constexpr int kRows = 64;            // samples per tile
constexpr int kThreads = 256;        // per CTA: groups x warps x 32
constexpr int kSpan = 32, kStages = 2;  // inputs per span of the ring

__device__ __forceinline__ float2 unpack2(unsigned long long v)
{
    return make_float2(__uint_as_float((uint32_t)v), __uint_as_float((uint32_t)(v >> 32)));
}
__device__ __forceinline__ float lane4(const float4 &v, int i) { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; }

// Leading dimension of the activation rows: 4 mod 8 floats (16-byte loads of neighbouring rows on distinct banks).
__host__ __device__ constexpr int act_ld(int maxw_p) { return ((maxw_p + 7) & ~7) + 4; }

// Shared-memory floats of one group.
__host__ __device__ inline size_t group_floats(const NetDesc &N)
{
    // activations, states [s][rows], actions [2][k][rows], cost, pusher position (2), box key (2), box
    return (size_t)kRows * (act_ld(N.maxw_p) + N.s + 2 * N.k + 6);
}

// acc += inputs k0 .. k1 - 1 (multiples of 4) of the thread's TR rows (4 apart) times its TN columns' weights.
// x: the thread's first row; w: input k0's weights at the thread's first column; hi: its second four columns exist.
template <int TR, int TN>
__device__ __forceinline__ void product(const float *__restrict__ x, int ld, const float *__restrict__ w, int Np, int k0,
                                        int k1, bool hi, unsigned long long (&acc)[TR][TN / 2])
{
#pragma unroll 2
    for (int k = k0; k < k1; k += 4) {
        float4 xv[TR];
#pragma unroll
        for (int i = 0; i < TR; ++i) xv[i] = *reinterpret_cast<const float4 *>(x + (size_t)4 * i * ld + k);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
            const float *wr = w + (size_t)(k - k0 + kk) * Np;
            unsigned long long wv[TN / 2];
            const float4 a = *reinterpret_cast<const float4 *>(wr);
            wv[0] = pack_f32x2(a.x, a.y);
            wv[1] = pack_f32x2(a.z, a.w);
            if (TN == 8) {
                const float4 b = hi ? *reinterpret_cast<const float4 *>(wr + 32) : make_float4(0.f, 0.f, 0.f, 0.f);
                wv[2 % (TN / 2)] = pack_f32x2(b.x, b.y);
                wv[3 % (TN / 2)] = pack_f32x2(b.z, b.w);
            }
#pragma unroll
            for (int i = 0; i < TR; ++i) {
                const float xs = lane4(xv[i], kk);
                const unsigned long long x2 = pack_f32x2(xs, xs);
#pragma unroll
                for (int j = 0; j < TN / 2; ++j) acc[i][j] = ffma2_rn(x2, wv[j], acc[i][j]);
            }
        }
    }
}

struct LayerArgs {
    float *act;
    const float *W, *bias;
    float *ring;
    int ld, Kp, Np;
    bool relu;
};

// One layer of a group's tile in blocks of 4 TR rows x 8 TN columns per warp (kRows / (4 TR) row blocks), in place.
template <int TR, int TN, bool STREAM>
__device__ __forceinline__ void layer(const LayerArgs &a, int grp, int tid, int nt)
{
    constexpr int RB = kRows / (4 * TR);
    const int warp = tid >> 5, lane = tid & 31, rg = lane >> 3, cg = lane & 7;
    const int r0 = (warp % RB) * 4 * TR + rg, c0 = (warp / RB) * 8 * TN + 4 * cg;
    const bool mine = c0 < a.Np, hi = TN == 8 && c0 + 32 < a.Np;
    const int Np = a.Np, Kp = a.Kp, ld = a.ld;
    unsigned long long acc[TR][TN / 2];
    {
        const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 b0 = mine ? *reinterpret_cast<const float4 *>(a.bias + c0) : z;
        const float4 b1 = hi ? *reinterpret_cast<const float4 *>(a.bias + c0 + 32) : z;
#pragma unroll
        for (int i = 0; i < TR; ++i) {
            acc[i][0] = pack_f32x2(b0.x, b0.y);
            acc[i][1] = pack_f32x2(b0.z, b0.w);
            if (TN == 8) {
                acc[i][2 % (TN / 2)] = pack_f32x2(b1.x, b1.y);
                acc[i][3 % (TN / 2)] = pack_f32x2(b1.z, b1.w);
            }
        }
    }
    const float *x = a.act + (size_t)r0 * ld;
    if (!STREAM) {
        if (mine) product<TR, TN>(x, ld, a.W + c0, Np, 0, Kp, hi, acc);
    } else {
        const int nspan = (Kp + kSpan - 1) / kSpan;
        auto fetch = [&](int q) {
            if (q < nspan) {
                const int k0 = q * kSpan, n4 = min(kSpan, Kp - k0) * Np / 4;
                const float4 *src = reinterpret_cast<const float4 *>(a.W + (size_t)k0 * Np);
                const uint32_t dst =
                    (uint32_t)__cvta_generic_to_shared(a.ring + (size_t)(q % kStages) * kSpan * kMaxWidth);
                for (int i = tid; i < n4; i += nt)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16 * i), "l"(src + i) : "memory");
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        fetch(0);
        for (int q = 0; q < nspan; ++q) {
            fetch(q + 1);  // its stage was last read before the barrier that closed the span before
            asm volatile("cp.async.wait_group 1;" ::: "memory");
            group_barrier(grp, nt);
            const int k0 = q * kSpan;
            if (mine)
                product<TR, TN>(x, ld, a.ring + (size_t)(q % kStages) * kSpan * kMaxWidth + c0, Np, k0,
                                min(Kp, k0 + kSpan), hi, acc);
            group_barrier(grp, nt);
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    if (!STREAM) group_barrier(grp, nt);  // every input read
    if (mine) {
        float *o = a.act + (size_t)r0 * ld + c0;
#pragma unroll
        for (int i = 0; i < TR; ++i)
#pragma unroll
            for (int h = 0; h < TN / 4; ++h) {
                if (h == 1 && !hi) continue;
                float2 p = unpack2(acc[i][2 * h]), q = unpack2(acc[i][2 * h + 1]);
                if (a.relu) {
                    p.x = fmaxf(p.x, 0.f);
                    p.y = fmaxf(p.y, 0.f);
                    q.x = fmaxf(q.x, 0.f);
                    q.y = fmaxf(q.y, 0.f);
                }
                *reinterpret_cast<float4 *>(o + (size_t)4 * i * ld + 32 * h) = make_float4(p.x, p.y, q.x, q.y);
            }
    }
    group_barrier(grp, nt);
}

// A layer of at most nt / 16 outputs (the network's last): one row and four columns per thread.
__device__ __forceinline__ void layer_narrow(const LayerArgs &a, int grp, int tid, int nt)
{
    const int r = tid % kRows, c0 = 4 * (tid / kRows), Np = a.Np;
    const bool mine = c0 < Np;
    unsigned long long acc[2] = {0ull, 0ull};
    if (mine) {
        const float4 b = *reinterpret_cast<const float4 *>(a.bias + c0);
        acc[0] = pack_f32x2(b.x, b.y);
        acc[1] = pack_f32x2(b.z, b.w);
        const float *x = a.act + (size_t)r * a.ld;
#pragma unroll 4
        for (int k = 0; k < a.Kp; k += 4) {
            const float4 xv = *reinterpret_cast<const float4 *>(x + k);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                const float4 w = *reinterpret_cast<const float4 *>(a.W + (size_t)(k + kk) * Np + c0);
                const float xs = lane4(xv, kk);
                const unsigned long long x2 = pack_f32x2(xs, xs);
                acc[0] = ffma2_rn(x2, pack_f32x2(w.x, w.y), acc[0]);
                acc[1] = ffma2_rn(x2, pack_f32x2(w.z, w.w), acc[1]);
            }
        }
    }
    group_barrier(grp, nt);
    if (mine) {
        float2 p = unpack2(acc[0]), q = unpack2(acc[1]);
        if (a.relu) {
            p.x = fmaxf(p.x, 0.f);
            p.y = fmaxf(p.y, 0.f);
            q.x = fmaxf(q.x, 0.f);
            q.y = fmaxf(q.y, 0.f);
        }
        *reinterpret_cast<float4 *>(a.act + (size_t)r * a.ld + c0) = make_float4(p.x, p.y, q.x, q.y);
    }
    group_barrier(grp, nt);
}

}  // namespace

template <int G, bool STREAM>
__global__ void __launch_bounds__(kThreads, 1) k_rollout_rows(RolloutArgs a)
{
    constexpr int TG = kThreads / G;
    extern __shared__ float4 smem4[];
    float *sm = reinterpret_cast<float *>(smem4);
    const NetDesc &N = a.net;
    const int s = N.s, k = N.k, L = N.L, d = a.d, H = a.H, M = a.M;
    const int ld = act_ld(N.maxw_p), Kp1 = pad4(s + k);
    const float *img = a.fwd;
    float *p = sm, *ring = nullptr;
    if (STREAM) {
        ring = p;
        p += (size_t)kStages * kSpan * kMaxWidth;
    } else {
        for (int i = threadIdx.x; i < N.img_floats / 4; i += kThreads)
            smem4[i] = reinterpret_cast<const float4 *>(a.fwd)[i];
        img = sm;
        p += N.img_floats;
    }
    __syncthreads();
    const int grp = threadIdx.x / TG, tid = threadIdx.x % TG;
    p += (size_t)grp * group_floats(N);
    float *act = p, *xs = act + kRows * ld, *us = xs + kRows * s, *cost = us + 2 * kRows * k, *ps = cost + kRows;
    uint64_t *hb = reinterpret_cast<uint64_t *>(ps + 2 * kRows);
    int *rowbox = reinterpret_cast<int *>(hb + kRows);

    const long long total = (long long)live_count(a.n, a.d_n) * M;
    const long long ntiles = (total + kRows - 1) / kRows;
    const float rho = a.rho;
    for (long long tile = blockIdx.x + (long long)gridDim.x * grp; tile < ntiles; tile += (long long)gridDim.x * G) {
        const long long g0 = tile * kRows;
        group_barrier(grp, TG);  // the last tile's rows are done with
        for (int r = tid; r < kRows; r += TG) {
            const long long g = g0 + r;
            const int box = (int)((g < total ? g : total - 1) / M);  // (rows past the end repeat the last box)
            rowbox[r] = box;
            hb[r] = box_hash(a.seed, a.id[box]);
            cost[r] = 0.f;
            ps[2 * r] = a.cost.p0x;
            ps[2 * r + 1] = a.cost.p0y;
        }
        for (int i = tid; i < kRows * s; i += TG) xs[i] = a.x0[i / kRows];
        group_barrier(grp, TG);
        for (int t = 0; t <= H; ++t) {
            // the first threads: state and cost of step t from the network's output, and the state part of the next
            // input row; the others: the actions u_t
            if (tid < kRows) {
                const int r = tid;
                float *row = act + (size_t)r * ld;
                if (t > 0) {
                    const float *u = us + (size_t)((t - 1) & 1) * kRows * k + r;
                    float c = 0.f;
                    if (a.cost.kind == 0) {
                        for (int i = 0; i < s; ++i) {
                            const float x = xs[i * kRows + r] + row[i];
                            xs[i * kRows + r] = x;
                            row[i] = x;
                            const float e = x - a.goal[i];
                            c = fmaf(e, e, c);
                        }
                    } else {
                        // the pusher moves by u_{t-1}, then the state cost at t (Appendix D.4)
                        ps[2 * r] = __fadd_rn(ps[2 * r], u[0]);
                        ps[2 * r + 1] = __fadd_rn(ps[2 * r + 1], u[kRows]);
                        for (int i = 0; i < s; ++i) {
                            const float x = __fadd_rn(xs[i * kRows + r], row[i]);
                            xs[i * kRows + r] = x;
                            row[i] = x;
                        }
                        c = obstacle_cost_f32(a.cost, t, s, row, a.goal, ps[2 * r], ps[2 * r + 1]);
                    }
                    for (int j = 0; j < k; ++j) {
                        const float v = u[j * kRows];
                        c = fmaf(rho * v, v, c);
                    }
                    cost[r] += c;
                } else {
                    for (int i = 0; i < s; ++i) row[i] = xs[i * kRows + r];
                }
            } else if (t < H) {
                float *u = us + (size_t)(t & 1) * kRows * k;
                for (int i = tid - kRows; i < kRows * (Kp1 - s); i += TG - kRows) {
                    const int r = i % kRows, j = i / kRows;
                    float v = 0.f;
                    if (j < k) {
                        const int box = rowbox[r];
                        const uint32_t m = (uint32_t)((g0 + r < total ? g0 + r : total - 1) - (long long)box * M);
                        const uint32_t q = (uint32_t)(t * k + j);
                        const size_t e = (size_t)box * d + q;
                        v = a.cem_mu ? cem_sample(hb[r], (uint32_t)a.cem_it, m, q, a.cem_mu[e], a.cem_sigma[e], a.lo[e],
                                                  a.hi[e])
                                     : draw_sample(hb[r], m, q, a.lo[e], a.hi[e]);
                        u[j * kRows + r] = v;
                    }
                    act[(size_t)r * ld + s + j] = v;
                }
            }
            if (t == H) break;
            group_barrier(grp, TG);
            for (int l = 1; l <= L; ++l) {
                LayerArgs la;
                la.act = act;
                la.W = img + N.fwd_w[l];
                la.bias = img + N.fwd_b[l];
                la.ring = ring;
                la.ld = ld;
                la.Kp = pad4(N.dims[l - 1]);
                la.Np = pad4(N.dims[l]);
                la.relu = l < L;
                if (G == 2) {
                    if (la.Np > 64) layer<8, 8, STREAM>(la, grp, tid, TG);
                    else if (la.Np > 32) layer<4, 8, STREAM>(la, grp, tid, TG);
                    else if (la.Np > 8) layer<4, 4, STREAM>(la, grp, tid, TG);
                    else layer_narrow(la, grp, tid, TG);
                } else {
                    if (la.Np > 128) layer<8, 8, STREAM>(la, grp, tid, TG);
                    else if (la.Np > 64) layer<4, 8, STREAM>(la, grp, tid, TG);
                    else if (la.Np > 32) layer<4, 4, STREAM>(la, grp, tid, TG);
                    else if (STREAM || la.Np > 16) layer<2, 4, STREAM>(la, grp, tid, TG);
                    else layer_narrow(la, grp, tid, TG);
                }
            }
        }
        // (cost[r] was written by this thread)
        if (tid < kRows) {
            const long long g = g0 + tid;
            const int box = rowbox[tid];
            const uint32_t m = (uint32_t)(g - (long long)box * M);
            unsigned long long key = ~0ull;
            if (g < total) {
                key = ((unsigned long long)float_order(cost[tid]) << 32) | m;
                if (a.costs) a.costs[(size_t)box * M + m] = cost[tid];
            }
            if (__match_any_sync(0xFFFFFFFFu, box) == 0xFFFFFFFFu) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const unsigned long long v = __shfl_xor_sync(0xFFFFFFFFu, key, o);
                    key = v < key ? v : key;
                }
                if ((tid & 31) == 0) atomicMin(&a.keys[box], key);
            } else if (g < total) {
                atomicMin(&a.keys[box], key);
            }
        }
    }
}

static size_t ring_bytes() { return (size_t)kStages * kSpan * kMaxWidth * 4; }

// Whether the kernel takes this call: one problem, no search-integrated bounds (their per-box extremes are gathered by
// k_rollout_fp32, a tile of which belongs to one box), and a group's buffers beside the image or the ring.
bool rollout_rows_supported(const RolloutArgs &a, size_t budget)
{
    const size_t img = (size_t)a.net.img_floats * 4, grp = group_floats(a.net) * 4;
    return a.batch.P <= 1 && !a.emp_pre_lo && (img + grp <= budget || ring_bytes() + grp <= budget);
}

// Two groups of four warps where every layer fits their tiles (width <= 128) and both buffers fit beside the image;
// else one group of eight with the image resident, or streamed.
cudaError_t launch_rollout_rows(const RolloutArgs &a, int num_sms, size_t budget, cudaStream_t st)
{
    const NetDesc &N = a.net;
    const size_t img = (size_t)N.img_floats * 4, grp = group_floats(N) * 4;
    int wide = 0;
    for (int l = 1; l <= N.L; ++l) wide = pad4(N.dims[l]) > wide ? pad4(N.dims[l]) : wide;
    const long long tiles = ((long long)a.n * a.M + kRows - 1) / kRows;
    const int grid = (int)(tiles < num_sms ? tiles : num_sms);
    auto run = [&](auto kern, size_t smem) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        kern<<<grid, kThreads, smem, st>>>(a);
        return cudaGetLastError();
    };
    if (wide <= 128 && img + 2 * grp <= budget) return run(k_rollout_rows<2, false>, img + 2 * grp);
    if (img + grp <= budget) return run(k_rollout_rows<1, false>, img + grp);
    return run(k_rollout_rows<1, true>, ring_bytes() + grp);
}

}  // namespace bab
