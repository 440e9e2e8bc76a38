// bound.cu -- lower bounds of the planning objective over boxes.
//
//   k_ibp        interval bound propagation (outward-rounded FP32) through the
//                H-step unrolled network: the pre-activation bounds that
//                Lemma 1 (Appendix B.1) needs, the state intervals, and, per
//                row k of every layer, S_k = sum_j |W_kj| max|a_j| over the
//                layer's input box (used to bound the rounding error of the
//                backward products).
//   k_rows       CROWN: Theorem 1 backward propagation of the tangent-linearised cost
//                through all H steps, then Theorem 2 in box form.  Constant
//                terms are accumulated with downward rounding (so they are
//                lower bounds by construction); the rounding error of the
//                coefficient vectors (the products A W_l, the relaxation
//                products, the state-coefficient updates) is bounded a
//                posteriori and subtracted as `margin`.
//                Its other form (FWD) is the adjoint, the forward pass of the relaxed
//                network from x_0 and the concretizing point u*, giving
//                dLB/dalpha = A_j z~_j.
//   k_adam       projected Adam ascent on alpha.
//
// In k_rows a CTA's warps form groups of a few boxes (rows) each that share the
// network image, in shared memory when it fits (otherwise it is read through L2);
// the rows move through the layers as register-blocked FP32 products (dense_rows),
// and each per-row reduction is one warp with shuffles.  k_ibp has its own tiles.
#include <cmath>

#include "bab_internal.cuh"
#include "kernels.cuh"

namespace bab {

constexpr int RB = 28;  // boxes whose working set must fit in shared memory for k_rows to take a network
constexpr int NT = 512;
constexpr float kTwoU = 1.1920930376163597e-07f;  // 2^-23 (1 + 2^-20): twice the unit roundoff, rounded up

// ---------------------------------------------------------------------------
// IBP
// ---------------------------------------------------------------------------
// Paired FP32 FMA with directed rounding: (a.x b.x + c.x, a.y b.y + c.y), each rounded down (RD) or up (RU);
// per element the same result as the scalar __fmaf_rd / __fmaf_ru.
__device__ __forceinline__ unsigned long long ffma2_rd(unsigned long long a, unsigned long long b, unsigned long long c)
{
    unsigned long long d;
    asm("fma.rm.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ unsigned long long ffma2_ru(unsigned long long a, unsigned long long b, unsigned long long c)
{
    unsigned long long d;
    asm("fma.rp.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ float half2f(unsigned long long v, int e)
{
    return __uint_as_float((uint32_t)(e ? v >> 32 : v));
}

constexpr int kIbpNT = 512;  // threads of k_ibp
constexpr int kIbpGroups = 4; // independent row groups of a CTA (weights in shared memory)

// Where a layer's outputs go: the interval bounds and S of step t to global memory (rows < nlive, columns < dl;
// no pre-activation bounds for the output layer, no S where the caller takes none), and the next layer's input
// (ReLU of the bounds, or the bounds of the output layer themselves) to the tile's shared-memory buffers.
struct IbpSink {
    float *pre_lo, *pre_hi, *S;  // at (box0 * H + t) of the [n][H][...] arrays, the layer's first column
    size_t rstride_h, rstride_s; // per row: H * sumh, H * (sumh + s)
    uint32_t *mask;              // [rows][2][4], zero before: bit (c / 4) % 32 of word [c / 128][c % 4] set where column
                                 // c's lower end is not 0 (the next layer's input)
    int dl, nrows;
    bool full;                   // every warp that stores has all 32 lanes storing
    bool hidden, vec_h, vec_s;   // vec: four columns from a multiple of 4 on are 16-byte aligned
};

// A layer's outputs of one thread: TR rows x TN columns, lower and upper sums and S, written to the sink and to the
// next layer's input.  Returns whether a value is not finite.
template <int TR, int TN>
__device__ __forceinline__ bool ibp_store(const float (&l)[TR][TN], const float (&h)[TR][TN], const float (&S)[TR][TN],
                                          int r0, int c0, int Np, int ld, float *__restrict__ zlo,
                                          float *__restrict__ zhi, const IbpSink &o)
{
    bool bad = false;
    // the lanes of a warp hold whole rows' segments of 4 seg columns (seg = 32, 16, .. 1): masks by ballot
    const int seg = Np / 4;
    const bool by_ballot = TN == 4 && (seg % 32 == 0 || (seg <= 16 && (seg & (seg - 1)) == 0 && o.full));
#pragma unroll
    for (int i = 0; i < TR; ++i) {
        const int r = r0 + i;
        const bool live = r < o.nrows;
        const bool whole = TN == 4 && c0 + 4 <= o.dl;
        if (live && o.S) {
            float *p = o.S + r * o.rstride_s + c0;
            if (whole && o.vec_s)
                *reinterpret_cast<float4 *>(p) = make_float4(S[i][0], S[i][1 % TN], S[i][2 % TN], S[i][3 % TN]);
            else
#pragma unroll
                for (int j = 0; j < TN; ++j)
                    if (c0 + j < o.dl) p[j] = S[i][j];
        }
        if (live && o.hidden) {
            float *pl = o.pre_lo + r * o.rstride_h + c0, *ph = o.pre_hi + r * o.rstride_h + c0;
            if (whole && o.vec_h) {
                *reinterpret_cast<float4 *>(pl) = make_float4(l[i][0], l[i][1 % TN], l[i][2 % TN], l[i][3 % TN]);
                *reinterpret_cast<float4 *>(ph) = make_float4(h[i][0], h[i][1 % TN], h[i][2 % TN], h[i][3 % TN]);
            } else
#pragma unroll
                for (int j = 0; j < TN; ++j)
                    if (c0 + j < o.dl) {
                        pl[j] = l[i][j];
                        ph[j] = h[i][j];
                    }
        }
        float vl[TN], vh[TN];
#pragma unroll
        for (int j = 0; j < TN; ++j) {
            const bool relu = o.hidden && c0 + j < o.dl;
            vl[j] = relu ? fmaxf(l[i][j], 0.f) : l[i][j];
            vh[j] = relu ? fmaxf(h[i][j], 0.f) : h[i][j];
            bad |= !(fabsf(l[i][j]) < INFINITY) || !(fabsf(h[i][j]) < INFINITY);
        }
        if (o.hidden) {
            uint32_t *mk = o.mask + 8 * r + 4 * (c0 >> 7);
            if (by_ballot) {
                uint32_t m[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) m[j] = __ballot_sync(0xFFFFFFFFu, vl[j % TN] != 0.f);
                if (seg < 32) {
                    const int first = (threadIdx.x & 31) & ~(seg - 1);
#pragma unroll
                    for (int j = 0; j < 4; ++j) m[j] = (m[j] >> first) & ((1u << seg) - 1u);
                }
                if ((threadIdx.x & 31 & (seg - 1)) == 0) *reinterpret_cast<uint4 *>(mk) = make_uint4(m[0], m[1], m[2], m[3]);
            } else {
#pragma unroll
                for (int j = 0; j < TN; ++j)
                    if (vl[j] != 0.f && c0 + j < Np) atomicOr(mk + ((c0 + j) & 3), 1u << ((c0 >> 2) & 31));
            }
        }
        if (TN == 4) {
            // (Np is a multiple of 4)
            *reinterpret_cast<float4 *>(zlo + r * ld + c0) = make_float4(vl[0], vl[1 % TN], vl[2 % TN], vl[3 % TN]);
            *reinterpret_cast<float4 *>(zhi + r * ld + c0) = make_float4(vh[0], vh[1 % TN], vh[2 % TN], vh[3 % TN]);
        } else {
#pragma unroll
            for (int j = 0; j < TN; ++j)
                if (c0 + j < Np) {
                    zlo[r * ld + c0 + j] = vl[j];
                    zhi[r * ld + c0 + j] = vh[j];
                }
        }
    }
    return bad;
}

// One input of a thread's TR x TN outputs, two columns per FMA pair:
//   lower += w+ a_lo + w- a_hi (rounded down),  upper += w+ a_hi + w- a_lo (rounded up),
//   V     += |w| max|a| for the first layer, |w| a_lo for the later ones (rounded up),
// w+ = max(w, 0), w- = min(w, 0).  One of the two products of a weight is an exact zero, so each sum has the bits of
// the one that takes the endpoint by the sign of the weight.  LOWER: some row's a_lo is not 0; without it only the
// products of the upper end are left.
template <int TR, int TN, bool FIRST, bool LOWER>
__device__ __forceinline__ void ibp_input(const float *__restrict__ wr, const float4 (&l4)[TR], const float4 (&h4)[TR], int kk, unsigned long long (&l2)[TR][TN / 2],
                                          unsigned long long (&h2)[TR][TN / 2], unsigned long long (&v2)[TR][TN / 2])
{
    constexpr int TP = TN / 2;
    float w[TN];
    if (TN == 4) {
        const float4 q = *reinterpret_cast<const float4 *>(wr);
        w[0] = q.x;
        w[1] = q.y;
        w[2 % TN] = q.z;
        w[3 % TN] = q.w;
    } else {
        const float2 q = *reinterpret_cast<const float2 *>(wr);
        w[0] = q.x;
        w[1] = q.y;
    }
    unsigned long long wp[TP], wn[TP], wa[TP];
#pragma unroll
    for (int j = 0; j < TP; ++j) {
        wp[j] = pack_f32x2(fmaxf(w[2 * j], 0.f), fmaxf(w[2 * j + 1], 0.f));
        wn[j] = pack_f32x2(fminf(w[2 * j], 0.f), fminf(w[2 * j + 1], 0.f));
        wa[j] = pack_f32x2(fabsf(w[2 * j]), fabsf(w[2 * j + 1]));
    }
#pragma unroll
    for (int i = 0; i < TR; ++i) {
        const float ah = kk == 0 ? h4[i].x : kk == 1 ? h4[i].y : kk == 2 ? h4[i].z : h4[i].w;
        const unsigned long long ah2 = pack_f32x2(ah, ah);
        if (!LOWER) {
#pragma unroll
            for (int j = 0; j < TP; ++j) {
                l2[i][j] = ffma2_rd(wn[j], ah2, l2[i][j]);
                h2[i][j] = ffma2_ru(wp[j], ah2, h2[i][j]);
            }
        } else {
            const float al = kk == 0 ? l4[i].x : kk == 1 ? l4[i].y : kk == 2 ? l4[i].z : l4[i].w;
            const float am = FIRST ? fmaxf(fabsf(al), fabsf(ah)) : al;
            const unsigned long long al2 = pack_f32x2(al, al), am2 = pack_f32x2(am, am);
#pragma unroll
            for (int j = 0; j < TP; ++j) {
                l2[i][j] = ffma2_rd(wn[j], ah2, ffma2_rd(wp[j], al2, l2[i][j]));
                h2[i][j] = ffma2_ru(wn[j], al2, ffma2_ru(wp[j], ah2, h2[i][j]));
                v2[i][j] = ffma2_ru(wa[j], am2, v2[i][j]);
            }
        }
    }
}

// The sums of one thread's TR x TN outputs over the inputs k0 <= k < k1 (multiples of 4, within one group of 128),
// in input order.  mask: bit (k / 4) % 32 of word k % 4 says whether some row's lower end of input k is not 0.  After
// a ReLU nearly all are 0 (90-100% on the pushing and object-manipulation networks), so most of a layer is two FMAs a
// weight and row: 3.2 cycles per scheduler (pairs; 4.0 with scalar FMAs) against 6.9 with all five, and 7.2-8 with
// the endpoints selected instead (the selects run on the half-wide ALU pipe).
template <int TR, int TN, bool FIRST, bool FINE>
__device__ __forceinline__ void ibp_span(const float *__restrict__ alo, const float *__restrict__ ahi, int ld,
                                         const float *__restrict__ W, int ldw, int k0, int k1, int r0,
                                         const uint32_t (&mask)[4], unsigned long long (&l2)[TR][TN / 2],
                                         unsigned long long (&h2)[TR][TN / 2], unsigned long long (&v2)[TR][TN / 2])
{
    const uint32_t some = mask[0] | mask[1] | mask[2] | mask[3];
#pragma unroll 1
    for (int k = k0; k < k1; k += 4) {
        float4 l4[TR], h4[TR];
        const int b = (k >> 2) & 31;
#pragma unroll
        for (int i = 0; i < TR; ++i) h4[i] = *reinterpret_cast<const float4 *>(ahi + (r0 + i) * ld + k);
        const float *wq = W + (size_t)(k - k0) * ldw;
        if (!FIRST && !((some >> b) & 1u)) {
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) ibp_input<TR, TN, FIRST, false>(wq + kk * ldw, l4, h4, kk, l2, h2, v2);
        } else {
#pragma unroll
            for (int i = 0; i < TR; ++i) l4[i] = *reinterpret_cast<const float4 *>(alo + (r0 + i) * ld + k);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
                if (FIRST || !FINE || ((mask[kk] >> b) & 1u))
                    ibp_input<TR, TN, FIRST, true>(wq + kk * ldw, l4, h4, kk, l2, h2, v2);
                else
                    ibp_input<TR, TN, FIRST, false>(wq + kk * ldw, l4, h4, kk, l2, h2, v2);
        }
    }
}

// The masks of inputs k .. k + 127 (k a multiple of 128) over rows r0 .. r0 + TR - 1.
template <int TR>
__device__ __forceinline__ void ibp_mask(const uint32_t *__restrict__ mask, int r0, int k, uint32_t (&m)[4])
{
    m[0] = m[1] = m[2] = m[3] = 0u;
#pragma unroll
    for (int i = 0; i < TR; ++i) {
        const uint4 q = *reinterpret_cast<const uint4 *>(mask + 8 * (r0 + i) + 4 * (k >> 7));
        m[0] |= q.x;
        m[1] |= q.y;
        m[2] |= q.z;
        m[3] |= q.w;
    }
}

// The sums turned into a thread's bounds and S.
template <int TR, int TN, bool FIRST>
__device__ __forceinline__ void ibp_unpack(const float *__restrict__ bias, unsigned long long (&l2)[TR][TN / 2],
                                           unsigned long long (&h2)[TR][TN / 2], unsigned long long (&v2)[TR][TN / 2],
                                           float (&l)[TR][TN], float (&h)[TR][TN], float (&S)[TR][TN])
{
#pragma unroll
    for (int i = 0; i < TR; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) {
            l[i][j] = half2f(l2[i][j / 2], j & 1);
            h[i][j] = half2f(h2[i][j / 2], j & 1);
            const float v = half2f(v2[i][j / 2], j & 1);
            S[i][j] = FIRST ? v : ibp_s(l[i][j], h[i][j], bias[j], v);
        }
}

// One layer with the weights in shared memory, TR rows x TN columns per thread and pass.
template <int TR, int TN, bool FIRST>
__device__ __forceinline__ bool ibp_dense(int tid, const float *__restrict__ alo, const float *__restrict__ ahi,
                                          const uint32_t *__restrict__ mask, int ld, int rb,
                                          const float *__restrict__ Wt, const float *__restrict__ bias, int Kp, int Np,
                                          float *__restrict__ zlo, float *__restrict__ zhi, const IbpSink &o)
{
    const int ngc = Np / TN;  // (Np is a multiple of 4)
    const int items = (rb / TR) * ngc;
    bool bad = false;
    for (int it = tid; it < items; it += kIbpNT / kIbpGroups) {
        const int rg = it / ngc, c0 = (it - rg * ngc) * TN, r0 = rg * TR;
        constexpr int TP = TN / 2;
        unsigned long long l2[TR][TP], h2[TR][TP], v2[TR][TP];
#pragma unroll
        for (int j = 0; j < TP; ++j)
#pragma unroll
            for (int i = 0; i < TR; ++i) {
                l2[i][j] = h2[i][j] = pack_f32x2(bias[c0 + 2 * j], bias[c0 + 2 * j + 1]);
                v2[i][j] = 0ull;
            }
        for (int k = 0; k < Kp; k += 128) {
            uint32_t m[4];
            ibp_mask<TR>(mask, r0, k, m);
            ibp_span<TR, TN, FIRST, true>(alo, ahi, ld, Wt + (size_t)k * Np + c0, Np, k, min(Kp, k + 128), r0, m, l2, h2, v2);
        }
        float l[TR][TN], h[TR][TN], S[TR][TN];
        ibp_unpack<TR, TN, FIRST>(bias + c0, l2, h2, v2, l, h, S);
        bad |= ibp_store<TR, TN>(l, h, S, r0, c0, Np, ld, zlo, zhi, o);
    }
    return bad;
}

// A later layer with few outputs (the network's last): one output per thread and pass, two chains of Kp FMAs whose
// latency is what the layer takes, so each input's endpoint is selected by the sign of the weight off the chain.
__device__ __forceinline__ bool ibp_dense_narrow(int tid, int nt, const float *__restrict__ alo,
                                                 const float *__restrict__ ahi, int ld, int rb,
                                                 const float *__restrict__ Wt, const float *__restrict__ bias, int Kp,
                                                 int Np, float *__restrict__ zlo, float *__restrict__ zhi, const IbpSink &o)
{
    bool bad = false;
    for (int it = tid; it < rb * Np; it += nt) {
        const int r = it / Np, c = it - r * Np;
        const float *al = alo + r * ld, *ah = ahi + r * ld, *w = Wt + c;
        float l[1][1], h[1][1], S[1][1];
        l[0][0] = h[0][0] = bias[c];
        S[0][0] = 0.f;
#pragma unroll 4
        for (int k = 0; k < Kp; k += 4) {
            const float4 h4 = *reinterpret_cast<const float4 *>(ah + k), l4 = *reinterpret_cast<const float4 *>(al + k);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                const float wk = w[(size_t)(k + kk) * Np];
                const float hi = kk == 0 ? h4.x : kk == 1 ? h4.y : kk == 2 ? h4.z : h4.w;
                const float lo = kk == 0 ? l4.x : kk == 1 ? l4.y : kk == 2 ? l4.z : l4.w;
                const bool pos = wk >= 0.f;
                l[0][0] = __fmaf_rd(wk, pos ? lo : hi, l[0][0]);
                h[0][0] = __fmaf_ru(wk, pos ? hi : lo, h[0][0]);
                S[0][0] = __fmaf_ru(fabsf(wk), lo, S[0][0]);
            }
        }
        S[0][0] = ibp_s(l[0][0], h[0][0], bias[c], S[0][0]);
        bad |= ibp_store<1, 1>(l, h, S, r, c, Np, ld, zlo, zhi, o);
    }
    return bad;
}

// The same layer where an input (or a weight) is not finite: 0 x inf must not reach the sums, so each input's
// endpoint is picked by the sign of the weight (the same bits for the rows that are finite).  One output per thread
// and pass.
__device__ __noinline__ bool ibp_dense_any(int tid, int nt, bool first, const float *__restrict__ alo,
                                           const float *__restrict__ ahi, int ld, int rb,
                                           const float *__restrict__ Wt, const float *__restrict__ bias, int Kp,
                                           int Np, float *__restrict__ zlo, float *__restrict__ zhi, const IbpSink &o)
{
    bool bad = false;
    for (int it = tid; it < rb * Np; it += nt) {
        const int r = it / Np, c = it - r * Np;
        float l[1][1], h[1][1], S[1][1];
        l[0][0] = h[0][0] = bias[c];
        S[0][0] = 0.f;
        for (int k = 0; k < Kp; ++k) {
            const float w = Wt[(size_t)k * Np + c], al = alo[r * ld + k], ah = ahi[r * ld + k];
            const bool pos = w >= 0.f;
            l[0][0] = __fmaf_rd(w, pos ? al : ah, l[0][0]);
            h[0][0] = __fmaf_ru(w, pos ? ah : al, h[0][0]);
            S[0][0] = __fmaf_ru(fabsf(w), first ? fmaxf(fabsf(al), fabsf(ah)) : al, S[0][0]);
        }
        if (!first) S[0][0] = ibp_s(l[0][0], h[0][0], bias[c], S[0][0]);
        bad |= ibp_store<1, 1>(l, h, S, r, c, Np, ld, zlo, zhi, o);
    }
    return bad;
}

// Weights beyond shared memory: the layer's forward image goes through a ring of kIbpStages stages of kIbpSpan
// inputs each, copied asynchronously while the stage before is multiplied; every thread owns the same TR x TN
// outputs throughout (rb / TR x Np / TN of them, at most kIbpNT).
constexpr int kIbpSpan = 32, kIbpStages = 2, kIbpStreamRows = 32;

template <int TR, int TN, bool FIRST>
__device__ __forceinline__ bool ibp_dense_stream(const float *__restrict__ alo, const float *__restrict__ ahi,
                                                 const uint32_t *__restrict__ mask, int ld,
                                                 float *__restrict__ ring, const float *__restrict__ Wt,
                                                 const float *__restrict__ bias, int Kp, int Np, int rb,
                                                 float *__restrict__ zlo, float *__restrict__ zhi, const IbpSink &o)
{
    const int ngc = Np / TN;
    const int rg = threadIdx.x / ngc, c0 = (threadIdx.x - rg * ngc) * TN, r0 = rg * TR;
    const bool mine = rg < rb / TR;
    const int nspan = (Kp + kIbpSpan - 1) / kIbpSpan;
    auto fetch = [&](int q) {
        if (q < nspan) {
            const int k0 = q * kIbpSpan, n4 = min(kIbpSpan, Kp - k0) * Np / 4;
            const float4 *src = reinterpret_cast<const float4 *>(Wt + (size_t)k0 * Np);
            const uint32_t dst =
                (uint32_t)__cvta_generic_to_shared(ring + (size_t)(q % kIbpStages) * kIbpSpan * kMaxWidth);
            for (int i = threadIdx.x; i < n4; i += kIbpNT)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16 * i), "l"(src + i) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    constexpr int TP = TN / 2;
    unsigned long long l2[TR][TP], h2[TR][TP], v2[TR][TP];
#pragma unroll
    for (int j = 0; j < TP; ++j) {
        const unsigned long long b2 = mine ? pack_f32x2(bias[c0 + 2 * j], bias[c0 + 2 * j + 1]) : 0ull;
#pragma unroll
        for (int i = 0; i < TR; ++i) {
            l2[i][j] = h2[i][j] = b2;
            v2[i][j] = 0ull;
        }
    }
    uint32_t m[4] = {0u, 0u, 0u, 0u};
    fetch(0);
    for (int q = 0; q < nspan; ++q) {
        fetch(q + 1);  // its stage was last read before the barrier that closed the span before
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();
        if (mine) {
            const int k0 = q * kIbpSpan;
            if (k0 % 128 == 0) ibp_mask<TR>(mask, r0, k0, m);
            ibp_span<TR, TN, FIRST, false>(alo, ahi, ld, ring + (size_t)(q % kIbpStages) * kIbpSpan * kMaxWidth + c0, Np, k0,
                                    min(Kp, k0 + kIbpSpan), r0, m, l2, h2, v2);
        }
        __syncthreads();
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (!mine) return false;
    float l[TR][TN], h[TR][TN], S[TR][TN];
    ibp_unpack<TR, TN, FIRST>(bias + c0, l2, h2, v2, l, h, S);
    return ibp_store<TR, TN>(l, h, S, r0, c0, Np, ld, zlo, zhi, o);
}

// Leading dimension of the tile's activation rows: 4 mod 8 floats, so that the 16-byte loads of different rows by
// one warp fall on different banks.
__host__ __device__ constexpr int ibp_ld(int maxw_p) { return ((maxw_p + 7) & ~7) + 4; }

// Shared-memory floats of one group of rb rows (a multiple of 4).
__host__ __device__ inline size_t ibp_rest_floats(const NetDesc &N, int rb)
{
    return (4 * (size_t)rb * ibp_ld(N.maxw_p) + 28 * (size_t)rb + 2 * (size_t)rb * pad4(N.s) + rb + 3) & ~size_t(3);
}

// Barrier of one row group (threads nt, barrier id g + 1), and whether any of its threads passed a nonzero v.
__device__ __forceinline__ int group_or(int g, int nt, int v)
{
    int r;
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.s32 p, %1, 0;\n\tbarrier.cta.red.or.pred q, %2, %3, p;\n\t"
                 "selp.s32 %0, 1, 0, q;\n\t}"
                 : "=r"(r)
                 : "r"(v), "r"(g + 1), "r"(nt)
                 : "memory");
    return r;
}

// Interval bounds of a tile of boxes.  The weights sit in shared memory and the CTA's warps form kIbpGroups groups of
// rb boxes each that share them and run on their own (buffers, barriers): while one group waits at a layer's end or
// walks the narrow output layer, the others multiply.  STREAM: the image does not fit; one group of rb boxes,
// ROWS of them if not 0.  tiles: two bits per layer, the tile of ibp_tile.  safe: some weight may not be finite.
// from: the grid's first box (0 with ROWS).
// What bounds it: issue slots and the latencies of a layer's ends (a step of the pushing network is four layers); the
// FMAs of the upper ends alone take 3.2 (4 x 4 outputs a thread) to 4.2 cycles (2 x 4) per weight and row.  Measured,
// all arrays written: pushing 3001 boxes 1079 -> 586 us; object manipulation, 16384 boxes, 51.4 -> 18.5 ms.
template <bool STREAM, int ROWS = 0>
__global__ void __launch_bounds__(kIbpNT, 1) k_ibp(BoundArgs a, int rb, int tiles, int vec_h, int vec_s, int safe, int from)
{
    const int first = ROWS ? 0 : from;
    constexpr int G = STREAM ? 1 : kIbpGroups, TG = kIbpNT / G;
    extern __shared__ float4 smem4[];
    float *sm = reinterpret_cast<float *>(smem4);
    const NetDesc &N = a.net;
    const int s = N.s, k = N.k, L = N.L, d = a.d, H = a.H, sumh = N.sumh;
    const int ld = ibp_ld(N.maxw_p), s4 = pad4(s);
    const int nlive = live_count(a.n, a.d_n, a.row0);
    if (first + (int)blockIdx.x * G * rb >= nlive) return;
    // a group's first warps do its narrow layers: spread the groups' over the schedulers (warp id modulo 4)
    const int grp = threadIdx.x / TG, tid = (threadIdx.x + 32 * grp) % TG;
    const int box0 = first + ((int)blockIdx.x * G + grp) * rb;
    const float *img = a.fwd;
    float *p = sm, *ring = nullptr;
    if (STREAM) {
        ring = p;
        p += (size_t)kIbpStages * kIbpSpan * kMaxWidth;
    } else {
        for (int i = threadIdx.x; i < N.img_floats / 4; i += kIbpNT)
            smem4[i] = reinterpret_cast<const float4 *>(a.fwd)[i];
        img = sm;
        p += N.img_floats;
        __syncthreads();
    }
    if (box0 >= nlive) return;
    p += (size_t)grp * ibp_rest_floats(N, rb);
    // activation buffers (lower and upper ends of buffer i), masks [3][rb][2][4] (IbpSink::mask), and per row: the
    // pusher position box of the obstacle cost (lo x, lo y, hi x, hi y), the state box, the bound so far
    float *act = p;
    auto buf_lo = [&](int i) { return act + 2 * i * rb * ld; };
    auto buf_hi = [&](int i) { return act + (2 * i + 1) * rb * ld; };
    uint32_t *masks = reinterpret_cast<uint32_t *>(act + 4 * rb * ld);
    float *pbx = act + 4 * rb * ld + 24 * rb, *xl = pbx + 4 * rb, *xu = xl + rb * s4, *lbacc = xu + rb * s4;
    int mcur = 0;

    const int lane = tid & 31, warp = tid >> 5;
    const int Kp1 = pad4(s + k);

    for (int i = tid; i < 24 * rb; i += TG) masks[i] = 0u;
    for (int i = tid; i < rb * s; i += TG) {
        const int r = i / s, c = i % s;
        xl[r * s4 + c] = a.x0[c];
        xu[r * s4 + c] = a.x0[c];
        if (box0 + r < nlive && a.x_lo) {
            a.x_lo[(size_t)(box0 + r) * (H + 1) * s + c] = a.x0[c];
            a.x_hi[(size_t)(box0 + r) * (H + 1) * s + c] = a.x0[c];
        }
    }
    for (int r = tid; r < rb; r += TG) {
        lbacc[r] = 0.f;
        pbx[4 * r] = pbx[4 * r + 2] = a.cost.p0x;
        pbx[4 * r + 1] = pbx[4 * r + 3] = a.cost.p0y;
    }
    group_or(grp, TG, 0);

    // a warp's rows are warp and warp + TG / 32 (rb is at most twice that); where a row's inputs fit the lanes, each
    // step's action bounds are loaded one step ahead
    const bool ahead = !STREAM && Kp1 <= 32;
    float ul[2] = {0.f, 0.f}, uh[2] = {0.f, 0.f};
    auto load_u = [&](int t) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int r = warp + i * (TG / 32);
            if (r < rb && box0 + r < nlive && t < H && lane >= s && lane < s + k) {
                ul[i] = a.lo[(size_t)(box0 + r) * d + t * k + (lane - s)];
                uh[i] = a.hi[(size_t)(box0 + r) * d + t * k + (lane - s)];
            }
        }
    };
    if (ahead) load_u(0);
    int cur = 0;
    for (int t = 0; t <= H; ++t) {
        // per row, one warp: x_t in [x_{t-1}] + [z_L] and the interval bound of its cost, then the next input row
        // [x_t | u_t | 0] and the bound of rho ||u_t||^2
        bool bad = false;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int r = warp + i * (TG / 32);
            if (r >= rb) break;
            const int box = box0 + r;
            const bool live = box < nlive;
            float v = 0.f, vu = 0.f;
            for (int c = lane; c < Kp1; c += 32) {
                float nl = 0.f, nh = 0.f;
                if (c < s) {
                    nl = xl[r * s4 + c];
                    nh = xu[r * s4 + c];
                    if (t > 0) {
                        nl = __fadd_rd(nl, buf_lo(cur)[r * ld + c]);
                        nh = __fadd_ru(nh, buf_hi(cur)[r * ld + c]);
                        xl[r * s4 + c] = nl;
                        xu[r * s4 + c] = nh;
                        if (live && a.x_lo) {
                            a.x_lo[((size_t)box * (H + 1) + t) * s + c] = nl;
                            a.x_hi[((size_t)box * (H + 1) + t) * s + c] = nh;
                        }
                        const float g = a.goal[c];
                        if (a.cost.kind == 0) {
                            v = __fadd_rd(v, sq_min_rd(__fsub_rd(nl, g), __fsub_ru(nh, g)));
                        } else {
                            // distance from g to the interval, rounded down, squared rounded down
                            const float e = fmaxf(fmaxf(__fsub_rd(nl, g), __fsub_rd(g, nh)), 0.f);
                            v = __fmaf_rd(e, e, v);
                        }
                    }
                } else if (c < s + k && live && t < H) {
                    nl = ahead ? ul[i] : a.lo[(size_t)box * d + t * k + (c - s)];
                    nh = ahead ? uh[i] : a.hi[(size_t)box * d + t * k + (c - s)];
                }
                bad |= !(fabsf(nl) < INFINITY) || !(fabsf(nh) < INFINITY);
                buf_lo(0)[r * ld + c] = nl;
                buf_hi(0)[r * ld + c] = nh;
            }
            if (t > 0) {
                v = warp_sum_rd(v);
                if (a.cost.kind == 1) {
                    // w_t times the distance from g to the box, then the penalties at their minima (rounded down)
                    __syncwarp();
                    float pen = 0.f;
                    const int nq = s / 2 + 1;
                    for (int q = lane; q < a.cost.n_obs * nq; q += 32) {
                        const int o = q / nq, kp = q % nq - 1;
                        pen = __fadd_rd(pen, kp < 0 ? penalty_min_rd(a.cost, o, pbx[4 * r], pbx[4 * r + 2],
                                                                     pbx[4 * r + 1], pbx[4 * r + 3])
                                                    : penalty_min_rd(a.cost, o, xl[r * s4 + 2 * kp], xu[r * s4 + 2 * kp],
                                                                     xl[r * s4 + 2 * kp + 1], xu[r * s4 + 2 * kp + 1]));
                    }
                    pen = warp_sum_rd(pen);
                    v = __fadd_rd(__fmul_rd(a.cost.w[t - 1], __fsqrt_rd(v)), pen);
                }
            }
            if (a.rho > 0.f && t < H) {
                if (ahead) {
                    const float q = live && lane >= s && lane < s + k ? sq_min_rd(ul[i], uh[i]) : 0.f;
                    vu = __shfl_sync(0xFFFFFFFFu, q, lane + s);
                    vu = lane < k ? __fadd_rd(0.f, vu) : 0.f;
                } else if (live)
                    for (int j = lane; j < k; j += 32)
                        vu = __fadd_rd(vu, sq_min_rd(a.lo[(size_t)box * d + t * k + j], a.hi[(size_t)box * d + t * k + j]));
                vu = warp_sum_rd(vu);
            }
            if (lane == 0) {
                float lb = lbacc[r];
                if (t > 0) lb = __fadd_rd(lb, v);
                if (a.rho > 0.f && t < H) lb = __fadd_rd(lb, __fmul_rd(a.rho, vu));
                lbacc[r] = lb;
                if (a.cost.kind == 1 && live && t < H) {
                    // the pusher after u_t (read at x_{t+1}'s cost)
                    const float *ul = a.lo + (size_t)box * d + t * k, *uh = a.hi + (size_t)box * d + t * k;
                    pbx[4 * r] = __fadd_rd(pbx[4 * r], ul[0]);
                    pbx[4 * r + 1] = __fadd_rd(pbx[4 * r + 1], ul[1]);
                    pbx[4 * r + 2] = __fadd_ru(pbx[4 * r + 2], uh[0]);
                    pbx[4 * r + 3] = __fadd_ru(pbx[4 * r + 3], uh[1]);
                }
            }
        }
        if (t == H) break;
        if (ahead) load_u(t + 1);
        int any = group_or(grp, TG, safe | (int)bad);
        cur = 0;
        for (int l = 1; l <= L; ++l) {
            const int Kp = pad4(N.dims[l - 1]), Np = pad4(N.dims[l]);
            IbpSink o;
            const size_t base = (size_t)box0 * H + t;
            o.pre_lo = a.pre_lo + base * sumh + (l < L ? N.hoff[l] : 0);
            o.pre_hi = a.pre_hi + base * sumh + (l < L ? N.hoff[l] : 0);
            o.S = a.S ? a.S + base * (sumh + s) + (l < L ? N.hoff[l] : sumh) : nullptr;
            o.rstride_h = (size_t)H * sumh;
            o.rstride_s = (size_t)H * (sumh + s);
            o.dl = N.dims[l];
            o.nrows = nlive - box0;
            o.hidden = l < L;
            o.vec_h = (vec_h >> l) & 1;
            o.vec_s = (vec_s >> l) & 1;
            o.full = (rb * Np) % 512 == 0;
            // the input's masks, the output's, and the ones to clear for the next layer (read before the last barrier)
            const uint32_t *mk = masks + (size_t)mcur * 8 * rb;
            mcur = mcur == 2 ? 0 : mcur + 1;
            o.mask = masks + (size_t)mcur * 8 * rb;
            {
                uint32_t *clear = masks + (size_t)(mcur == 2 ? 0 : mcur + 1) * 8 * rb;
                for (int i = tid; i < 8 * rb; i += TG) clear[i] = 0u;
            }
            const float *in_l = buf_lo(cur), *in_h = buf_hi(cur), *Wt = img + N.fwd_w[l], *bias = img + N.fwd_b[l];
            float *zl = buf_lo(cur ^ 1), *zh = buf_hi(cur ^ 1);
            if (any) {
                bad = ibp_dense_any(tid, TG, l == 1, in_l, in_h, ld, rb, Wt, bias, Kp, Np, zl, zh, o);
            } else if (!STREAM && l > 1 && rb * Np <= 2 * TG && Np < 64) {
                bad = ibp_dense_narrow(tid, TG, in_l, in_h, ld, rb, Wt, bias, Kp, Np, zl, zh, o);
            } else if (STREAM) {
                // the largest tile whose items still cover the threads: 32 rows of 256, 128 or 32 columns, and half the
                // rows a thread for each halving of the rows
#define IBP_STREAM(TR, TN, F) ibp_dense_stream<TR, TN, F>(in_l, in_h, mk, ld, ring, Wt, bias, Kp, Np, ROWS ? ROWS : rb, zl, zh, o)
                if (ROWS) {
                    if (l == 1) {
                        if (Np > 128) bad = IBP_STREAM(4, 4, true);
                        else if (Np > 32) bad = IBP_STREAM(2, 4, true);
                        else bad = IBP_STREAM(1, 2, true);
                    } else {
                        if (Np > 128) bad = IBP_STREAM(4, 4, false);
                        else if (Np > 32) bad = IBP_STREAM(2, 4, false);
                        else bad = IBP_STREAM(1, 2, false);
                    }
                } else {
                    const int tr = Np > 128 ? (rb > 16 ? 4 : rb > 8 ? 2 : 1) : Np > 32 ? (rb > 16 ? 2 : 1) : 0;
                    if (l == 1) {
                        if (tr == 4) bad = IBP_STREAM(4, 4, true);
                        else if (tr == 2) bad = IBP_STREAM(2, 4, true);
                        else if (tr == 1) bad = IBP_STREAM(1, 4, true);
                        else bad = IBP_STREAM(1, 2, true);
                    } else {
                        if (tr == 4) bad = IBP_STREAM(4, 4, false);
                        else if (tr == 2) bad = IBP_STREAM(2, 4, false);
                        else if (tr == 1) bad = IBP_STREAM(1, 4, false);
                        else bad = IBP_STREAM(1, 2, false);
                    }
                }
#undef IBP_STREAM
            } else {
                switch ((l == 1 ? 4 : 0) + ((tiles >> (2 * l)) & 3)) {
                    case 0: bad = ibp_dense<4, 4, false>(tid, in_l, in_h, mk, ld, rb, Wt, bias, Kp, Np, zl, zh, o); break;
                    case 1: bad = ibp_dense<2, 4, false>(tid, in_l, in_h, mk, ld, rb, Wt, bias, Kp, Np, zl, zh, o); break;
                    case 2: bad = ibp_dense<1, 4, false>(tid, in_l, in_h, mk, ld, rb, Wt, bias, Kp, Np, zl, zh, o); break;
                    case 3: bad = ibp_dense<1, 2, false>(tid, in_l, in_h, mk, ld, rb, Wt, bias, Kp, Np, zl, zh, o); break;
                    case 4:
                    case 5: bad = ibp_dense<2, 4, true>(tid, in_l, in_h, mk, ld, rb, Wt, bias, Kp, Np, zl, zh, o); break;
                    case 6: bad = ibp_dense<1, 4, true>(tid, in_l, in_h, mk, ld, rb, Wt, bias, Kp, Np, zl, zh, o); break;
                    default: bad = ibp_dense<1, 2, true>(tid, in_l, in_h, mk, ld, rb, Wt, bias, Kp, Np, zl, zh, o); break;
                }
            }
            any = group_or(grp, TG, safe | (int)bad);
            cur ^= 1;
        }
    }
    __syncwarp();
    if (a.lb_ibp && lane == 0)
        for (int r = warp; r < rb; r += TG / 32)
            if (box0 + r < nlive) a.lb_ibp[box0 + r] = lbacc[r];
}

// ---------------------------------------------------------------------------
// CROWN and its adjoint over a tile of rows.  The per-box arrays are reached
// through a RowsView whose pointers start at the tile's first box, so the same
// code runs on the global arrays (k_rows) and on copies held in
// shared memory for a whole alpha optimisation (k_alpha_fused).
// ---------------------------------------------------------------------------
struct RowsView {
    const float *lo, *hi;            // [rows][d]
    const float *pre_lo, *pre_hi;    // [rows][H][sumh]
    const float *x_lo, *x_hi;        // [rows][H+1][s]
    const float *S;                  // [rows][H][sumh + s]
    float *alpha;                    // [rows][H][sumh] (nullable: adaptive slopes)
    float *A_pre;                    // [rows][H][sumh] (nullable)
    float *ustar, *lin_coef;         // [rows][d] (nullable)
    float *lb, *margin, *lin_const, *lb_best;  // [rows] (lb required, the rest nullable)
    float *grad;                     // [rows][H][sumh]: adjoint output (nullable when Adam is fused)
    float *adam_m, *adam_v;          // [rows][H][sumh]: fused Adam moments (nullable)
};

__device__ __forceinline__ RowsView global_view(const BoundArgs &a, int box0)
{
    const size_t b = (size_t)box0, hs = (size_t)a.H * a.net.sumh;
    RowsView v;
    v.lo = a.lo + b * a.d;
    v.hi = a.hi + b * a.d;
    v.pre_lo = a.pre_lo + b * hs;
    v.pre_hi = a.pre_hi + b * hs;
    v.x_lo = a.x_lo + b * (a.H + 1) * a.net.s;
    v.x_hi = a.x_hi + b * (a.H + 1) * a.net.s;
    v.S = a.S + b * a.H * (a.net.sumh + a.net.s);
    v.alpha = a.alpha ? const_cast<float *>(a.alpha) + b * hs : nullptr;
    v.A_pre = a.A_pre ? a.A_pre + b * hs : nullptr;
    v.ustar = a.ustar ? a.ustar + b * a.d : nullptr;
    v.lin_coef = a.lin_coef ? a.lin_coef + b * a.d : nullptr;
    v.lb = a.lb + b;
    v.margin = a.margin ? a.margin + b : nullptr;
    v.lin_const = a.lin_const ? a.lin_const + b : nullptr;
    v.lb_best = a.lb_best ? a.lb_best + b : nullptr;
    v.grad = a.grad_alpha ? a.grad_alpha + b * hs : nullptr;
    v.adam_m = v.adam_v = nullptr;
    return v;
}

// shared-memory floats of crown_rows / fwd_rows scratch
__host__ __device__ inline size_t crown_rows_floats(const NetDesc &N, int rb, int d)
{
    return 2 * (size_t)rb * N.maxw_p + (size_t)rb * pad4(N.s) + (size_t)rb * pad4(d) + 2 * rb + 4 * rb;
}
__host__ __device__ inline size_t fwd_rows_floats(const NetDesc &N, int rb)
{
    return 2 * (size_t)rb * N.maxw_p + (size_t)rb * pad4(N.s);
}

// A layer's product over RBT rows by NTT threads: dense_rows_auto's tiles, but 4 x 4 outputs a thread where 4 x 8 would
// leave half of the threads idle (coefficients of 9728 boxes, H = 5: two 256-wide layers 947 -> 651 us, four of them, the
// image read through L2, 2348 -> 1470).
template <int RBT, int NTT>
__device__ __forceinline__ void rows_product(const float *in, int ldi, const float *B, const float *bias, int Kp, int Np,
                                             float *out, int ldo, int tid)
{
    if (RBT == 8 && NTT == 128 && Np > 128)
        dense_rows<RBT, NTT, (RBT == 8 ? 4 : 1), 4>(in, ldi, B, bias, Kp, Np, out, ldo, false, tid);
    else
        dense_rows_auto<RBT, NTT>(in, ldi, B, bias, Kp, Np, out, ldo, false, tid);
}

// Theorem 1 backward propagation of the tangent-linearised cost through all H
// steps, then Theorem 2 in box form, for rows 0 .. nrows-1 of the view (rows
// nrows .. RBT-1 are padding), by NTT consecutive threads of the CTA (group grp
// of them).  img: backward image; p: crown_rows_floats of shared memory.
template <int RBT, int NTT>
__device__ void crown_rows(const BoundArgs &a, const float *img, float *p, const RowsView &v, int nrows, int grp = 0)
{
    const int tid = threadIdx.x % NTT;
    const NetDesc &N = a.net;
    const int s = N.s, k = N.k, L = N.L, d = a.d, H = a.H, sumh = N.sumh, sw = sumh + s;
    const int ld = N.maxw_p, s4 = pad4(s), d4 = pad4(d);
    float *Ab[2];
    Ab[0] = p; p += RBT * ld;
    Ab[1] = p; p += RBT * ld;
    float *lam = p; p += RBT * s4;
    float *mu = p; p += RBT * d4;
    float *Pu = p; p += 4 * RBT;  // obstacle cost: per row the pusher coefficient of the actions (2) and its |sum| (2)
    const int lane = tid & 31, warp = tid >> 5;
    const bool obst = a.cost.kind == 1;
    const bool has_alpha = v.alpha != nullptr;
    const int ts = a.t_stop;              // early stop: propagate back to x_ts only
    const bool with_margin = v.S != nullptr;
    // A warp's rows (warp, warp + NTT / 32, ..): a row's constant (rounded down; the same on every lane), summed over the
    // lanes in every layer, and each lane's own margin terms (rounded up, all nonnegative), added over the lanes once at
    // the end.  (The constant's terms have both signs: kept per lane too, 32 larger sums rounded in every layer, it came
    // out up to 1.2 times further from the exact one.)
    constexpr int NW = NTT / 32, RW = (RBT + NW - 1) / NW;
    float cl[RW], ml[RW];
#pragma unroll
    for (int i = 0; i < RW; ++i) cl[i] = ml[i] = 0.f;

    // early stop: the cost terms at steps 1 .. ts on their intervals, no coefficient of u before ts
    if (ts > 0) {
        for (int i = tid; i < RBT * d4; i += NTT) mu[i] = 0.f;
#pragma unroll
        for (int ri = 0; ri < RW; ++ri) {
            const int r = warp + ri * NW;
            if (r >= nrows) break;
            float c = 0.f;
            for (int q = lane; q < ts * s; q += 32) {
                const int t = 1 + q / s, i = q % s;
                const float g = a.goal[i];
                const size_t xi = ((size_t)r * (H + 1) + t) * s + i;
                c = __fadd_rd(c, sq_min_rd(__fsub_rd(v.x_lo[xi], g), __fsub_ru(v.x_hi[xi], g)));
            }
            cl[ri] = warp_sum_rd(c);
        }
    }
    // tangent of ||x_H - g||^2: coefficient 2m, constant -(2 m g + m^2)
#pragma unroll
    for (int ri = 0; ri < RW; ++ri) {
        const int r = warp + ri * NW;
        if (r >= RBT) break;
        if (obst) {
            // the obstacle cost at step H: its linear lower bound on x_H, and the pusher penalties at H
            float aa = 0.f, c = 0.f;
            if (r < nrows && H > ts) {
                const size_t xi = ((size_t)r * (H + 1) + H) * s;
                c = obstacle_state_lin(a.cost, H, s, v.x_lo + xi, v.x_hi + xi, a.goal, lane, aa);
            }
            if (lane < s) lam[r * s4 + lane] = aa;
            if (lane == 0) {
                Pu[4 * r] = Pu[4 * r + 1] = Pu[4 * r + 2] = Pu[4 * r + 3] = 0.f;
                if (r < nrows) c = __fadd_rd(c, pusher_lin(a.cost, H, k, v.lo + (size_t)r * d, v.hi + (size_t)r * d,
                                                           Pu + 4 * r, Pu + 4 * r + 2));
            }
            cl[ri] = __shfl_sync(0xFFFFFFFFu, c, 0);
            continue;
        }
        float c = 0.f;
        for (int i = lane; i < s; i += 32) {
            float aa = 0.f;
            if (r < nrows && H > ts) {
                const float g = a.goal[i];
                const size_t xi = ((size_t)r * (H + 1) + H) * s + i;
                const float Ls = __fsub_rd(v.x_lo[xi], g), Us = __fsub_ru(v.x_hi[xi], g);
                const float m = 0.5f * (Ls + Us);
                aa = 2.f * m;
                c = __fadd_rd(c, __fmaf_rd(-aa, g, -__fmul_ru(m, m)));
            }
            lam[r * s4 + i] = aa;
        }
        c = warp_sum_rd(c);
        cl[ri] = ts > 0 ? __fadd_rd(cl[ri], c) : c;
    }
    group_barrier(grp, NTT);

    for (int t = H - 1; t >= ts; --t) {
        // last layer: A = lam on z_L (rows of W_L), constant lam . b_L
        {
            const int NpL = pad4(N.dims[L]);
            const float *bL = img + N.bwd_b[L];
#pragma unroll
            for (int ri = 0; ri < RW; ++ri) {
                const int r = warp + ri * NW;
                if (r >= RBT) break;
                float c = 0.f, e = 0.f;
                for (int q = lane; q < NpL; q += 32) {
                    const float A = q < s ? lam[r * s4 + q] : 0.f;
                    Ab[0][r * ld + q] = A;
                    if (q < s && r < nrows) {
                        c = __fmaf_rd(A, bL[q], c);
                        if (with_margin) e = __fmaf_ru(fabsf(A), v.S[((size_t)r * H + t) * sw + sumh + q], e);
                    }
                }
                cl[ri] = __fadd_rd(cl[ri], warp_sum_rd(c));
                ml[ri] = __fmaf_ru(N.gam[L], e, ml[ri]);
            }
            group_barrier(grp, NTT);
            rows_product<RBT, NTT>(Ab[0], ld, img + N.bwd_w[L], nullptr, NpL, pad4(N.dims[L - 1]), Ab[1], ld, tid);
            group_barrier(grp, NTT);
        }
        int cur = 1;
        for (int l = L - 1; l >= 1; --l) {
            const int dl = N.dims[l], Npl = pad4(dl);
            const float *bl = img + N.bwd_b[l];
#pragma unroll
            for (int ri = 0; ri < RW; ++ri) {
                const int r = warp + ri * NW;
                if (r >= RBT) break;
                if (r >= nrows) {
                    for (int q = lane; q < dl; q += 32) Ab[cur][r * ld + q] = 0.f;
                    continue;
                }
                const size_t base = ((size_t)r * H + t), row = base * sumh + N.hoff[l], srow = base * sw + N.hoff[l];
                float c = 0.f, eg = 0.f, er = 0.f;
                // four of the lane's neurons at a time: their intervals, margin helpers and slopes loaded together
                for (int q0 = lane; q0 < dl; q0 += 128) {
                    float zl[4], zu[4], sv[4], al[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int q = q0 + 32 * e;
                        const bool in = q < dl;
                        zl[e] = in ? v.pre_lo[row + q] : 0.f;
                        zu[e] = in ? v.pre_hi[row + q] : 0.f;
                        sv[e] = in && with_margin ? v.S[srow + q] : 0.f;
                        al[e] = in && has_alpha ? v.alpha[row + q] : 0.f;
                    }
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int q = q0 + 32 * e;
                        if (q >= dl) break;
                        const float A = Ab[cur][r * ld + q];
                        if (v.A_pre) v.A_pre[row + q] = A;
                        float D, ci;
                        relax_select(zl[e], zu[e], A, al[e], has_alpha, D, ci);
                        const float Ap = A * D;
                        Ab[cur][r * ld + q] = Ap;
                        c = __fmaf_rd(A, ci, c);
                        c = __fmaf_rd(Ap, bl[q], c);
                        if (with_margin) {
                            eg = __fmaf_ru(fabsf(Ap), sv[e], eg);
                            if (D != 0.f && D != 1.f) er = __fmaf_ru(fabsf(Ap), fmaxf(-zl[e], zu[e]), er);
                        }
                    }
                }
                cl[ri] = __fadd_rd(cl[ri], warp_sum_rd(c));
                ml[ri] = __fadd_ru(ml[ri], __fmaf_ru(N.gam[l], eg, __fmul_ru(kTwoU, er)));
            }
            group_barrier(grp, NTT);
            rows_product<RBT, NTT>(Ab[cur], ld, img + N.bwd_w[l], nullptr, Npl, pad4(N.dims[l - 1]), Ab[cur ^ 1], ld, tid);
            group_barrier(grp, NTT);
            cur ^= 1;
        }
        // A is on [x_t | u_t]: mu_t = A_u; lam <- lam + A_x (+ tangent of ||x_t - g||^2 for t >= 1)
#pragma unroll
        for (int ri = 0; ri < RW; ++ri) {
            const int r = warp + ri * NW;
            if (r >= RBT) break;
            float e = 0.f;
            if (obst) {
                // mu_t = A_u + the pusher coefficient of the later steps; its rounding (H additions) in the margin
                const float *lo_r = v.lo + (size_t)r * d, *hi_r = v.hi + (size_t)r * d;
                for (int j = lane; j < k; j += 32) {
                    const float Au = Ab[cur][r * ld + s + j];
                    const float Pj = j < 2 ? Pu[4 * r + j] : 0.f, Pa = j < 2 ? Pu[4 * r + 2 + j] : 0.f;
                    mu[r * d4 + t * k + j] = Au + Pj;
                    if (with_margin && r < nrows) {
                        const float um = fmaxf(fabsf(lo_r[t * k + j]), fabsf(hi_r[t * k + j]));
                        e = __fmaf_ru(__fmul_ru(__fmul_ru((float)(H + 2), kTwoU), __fadd_ru(fabsf(Au), Pa)), um, e);
                    }
                }
                float aa = 0.f, c = 0.f;
                if (t > ts && t >= 1 && r < nrows) {
                    const size_t xi = ((size_t)r * (H + 1) + t) * s;
                    c = obstacle_state_lin(a.cost, t, s, v.x_lo + xi, v.x_hi + xi, a.goal, lane, aa);
                }
                if (lane < s) {
                    const float Ax = Ab[cur][r * ld + lane];
                    const float lo_ = lam[r * s4 + lane];
                    const size_t xi = ((size_t)r * (H + 1) + t) * s + lane;
                    const float B = (t >= 1 && r < nrows) ? fmaxf(fabsf(v.x_lo[xi]), fabsf(v.x_hi[xi])) : fabsf(a.x0[lane]);
                    lam[r * s4 + lane] = (lo_ + Ax) + aa;
                    const float mag = __fadd_ru(__fadd_ru(fabsf(lo_), fabsf(Ax)), fabsf(aa));
                    if (with_margin) e = __fmaf_ru(__fmul_ru(kTwoU, mag), B, e);
                }
                if (lane == 0 && t >= 1 && r < nrows)
                    c = __fadd_rd(c, pusher_lin(a.cost, t, k, lo_r, hi_r, Pu + 4 * r, Pu + 4 * r + 2));
                cl[ri] = __fadd_rd(cl[ri], __shfl_sync(0xFFFFFFFFu, c, 0));
                ml[ri] = __fadd_ru(ml[ri], e);
                __syncwarp();
                continue;
            }
            for (int j = lane; j < k; j += 32) mu[r * d4 + t * k + j] = Ab[cur][r * ld + s + j];
            float c = 0.f;
            for (int i = lane; i < s; i += 32) {
                const float Ax = Ab[cur][r * ld + i];
                const float lo_ = lam[r * s4 + i];
                float aa = 0.f, B = fabsf(a.x0[i]);
                if (t >= 1 && r < nrows) {
                    // the updated coefficient multiplies x_t (concretized on its interval at an early stop)
                    const size_t xi = ((size_t)r * (H + 1) + t) * s + i;
                    const float xl = v.x_lo[xi], xu = v.x_hi[xi];
                    B = fmaxf(fabsf(xl), fabsf(xu));
                    if (t > ts) {
                        const float g = a.goal[i];
                        const float Ls = __fsub_rd(xl, g), Us = __fsub_ru(xu, g);
                        const float m = 0.5f * (Ls + Us);
                        aa = 2.f * m;
                        c = __fadd_rd(c, __fmaf_rd(-aa, g, -__fmul_ru(m, m)));
                    }
                }
                const float ln = (lo_ + Ax) + aa;
                lam[r * s4 + i] = ln;
                const float mag = __fadd_ru(__fadd_ru(fabsf(lo_), fabsf(Ax)), fabsf(aa));
                if (with_margin) e = __fmaf_ru(__fmul_ru(kTwoU, mag), B, e);
            }
            cl[ri] = __fadd_rd(cl[ri], warp_sum_rd(c));
            ml[ri] = __fadd_ru(ml[ri], e);
        }
        group_barrier(grp, NTT);
    }

    // lam . x0, then Theorem 2 in box form: sum_j min_{u in [lo, hi]} mu_j u + rho u^2
#pragma unroll
    for (int ri = 0; ri < RW; ++ri) {
        const int r = warp + ri * NW;
        if (r >= nrows) break;
        float c = 0.f, val = 0.f, e = ml[ri];
        if (ts == 0) {
            for (int i = lane; i < s; i += 32) c = __fmaf_rd(lam[r * s4 + i], a.x0[i], c);
        } else {
            // early stop: the coefficient of x_ts on that state's interval (Theorem 2, box form)
            for (int i = lane; i < s; i += 32) {
                const size_t xi = ((size_t)r * (H + 1) + ts) * s + i;
                const float li = lam[r * s4 + i];
                c = __fadd_rd(c, fminf(__fmul_rd(li, v.x_lo[xi]), __fmul_rd(li, v.x_hi[xi])));
            }
        }
        c = __fadd_rd(cl[ri], warp_sum_rd(c));
        for (int j = lane; j < d; j += 32) {
            const float m_ = mu[r * d4 + j];
            const float lo = v.lo[(size_t)r * d + j], hi = v.hi[(size_t)r * d + j];
            float us, vj;
            if (a.rho > 0.f) {
                const float uc = -m_ / (2.f * a.rho);
                if (uc >= lo && uc <= hi) {
                    us = uc;
                    vj = __fdiv_rd(-__fmul_ru(m_, m_), 4.f * a.rho);
                } else {
                    us = uc < lo ? lo : hi;
                    vj = __fmaf_rd(m_, us, __fmul_rd(a.rho, __fmul_rd(us, us)));
                    // the face choice can be off only when uc is within rounding of the face:
                    // the minimum then lies below q(us) by at most rho (2u uc)^2
                    const float du = __fmul_ru(kTwoU, fabsf(uc));
                    e = __fmaf_ru(__fmul_ru(a.rho, du), du, e);
                }
            } else {
                us = m_ >= 0.f ? lo : hi;
                vj = __fmul_rd(m_, us);
            }
            val = __fadd_rd(val, vj);
            if (v.ustar) v.ustar[(size_t)r * d + j] = us;
            if (v.lin_coef) v.lin_coef[(size_t)r * d + j] = m_;
        }
        val = warp_sum_rd(val);
        e = warp_sum_ru(e);
        if (lane == 0) {
            const float raw = __fadd_rd(c, val);
            const float lbv = __fsub_rd(raw, e);
            v.lb[r] = lbv;
            if (v.margin) v.margin[r] = e;
            if (v.lin_const) v.lin_const[r] = c;
            if (v.lb_best) v.lb_best[r] = fmaxf(v.lb_best[r], lbv);
        }
    }
}

// alpha gradient: forward pass of the relaxed network from x_0 and u*;
// dLB/dalpha_j = A_j z~_j for an unstable neuron whose coefficient A_j >= 0
// selects the lower line, 0 otherwise.  With `adam` the projected Adam step is
// applied to each slope as soon as its gradient is known (its own slope is
// not needed again in this pass); otherwise the gradient goes to v.grad.
template <int RBT, int NTT>
__device__ void fwd_rows(const BoundArgs &a, const float *img, float *p, const RowsView &v, int nrows,
                         const AdamStep *adam, int grp = 0)
{
    const int tid = threadIdx.x % NTT;
    const NetDesc &N = a.net;
    const int s = N.s, k = N.k, L = N.L, d = a.d, H = a.H, sumh = N.sumh;
    const int ld = N.maxw_p, s4 = pad4(s);
    float *Z[2];
    Z[0] = p; p += RBT * ld;
    Z[1] = p; p += RBT * ld;
    float *xs = p; p += RBT * s4;
    const bool has_alpha = v.alpha != nullptr;
    const int Kp1 = pad4(s + k);
    for (int i = tid; i < RBT * s; i += NTT) xs[(i / s) * s4 + i % s] = a.x0[i % s];
    group_barrier(grp, NTT);
    for (int t = 0; t < H; ++t) {
        for (int i = tid; i < RBT * Kp1; i += NTT) {
            const int r = i / Kp1, c = i % Kp1;
            float val = 0.f;
            if (c < s) val = xs[r * s4 + c];
            else if (c < s + k && r < nrows) val = v.ustar[(size_t)r * d + t * k + (c - s)];
            Z[0][r * ld + c] = val;
        }
        group_barrier(grp, NTT);
        int cur = 0;
        for (int l = 1; l <= L; ++l) {
            rows_product<RBT, NTT>(Z[cur], ld, img + N.fwd_w[l], img + N.fwd_b[l], pad4(N.dims[l - 1]), pad4(N.dims[l]),
                                   Z[cur ^ 1], ld, tid);
            group_barrier(grp, NTT);
            cur ^= 1;
            if (l < L) {
                const int dl = N.dims[l];
                // four neurons at a time, their loads together
                for (int i0 = tid; i0 < nrows * dl; i0 += 4 * NTT) {
                    float zl[4], zu[4], A[4], al[4];
                    size_t idx[4];
                    int at[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int i = i0 + e * NTT, r = i / dl, q = i - r * dl;
                        idx[e] = ((size_t)r * H + t) * sumh + N.hoff[l] + q;
                        at[e] = i < nrows * dl ? r * ld + q : -1;
                        const bool in = at[e] >= 0;
                        zl[e] = in ? v.pre_lo[idx[e]] : 0.f;
                        zu[e] = in ? v.pre_hi[idx[e]] : 0.f;
                        A[e] = in ? v.A_pre[idx[e]] : 0.f;
                        al[e] = in && has_alpha ? v.alpha[idx[e]] : 0.f;
                    }
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        if (at[e] < 0) break;
                        const float z = Z[cur][at[e]];
                        float D, c;
                        relax_select(zl[e], zu[e], A[e], al[e], has_alpha, D, c);
                        const bool unstable = zl[e] < 0.f && zu[e] > 0.f;
                        const float g = (unstable && A[e] >= 0.f) ? A[e] * z : 0.f;
                        if (adam) adam_update(v.alpha[idx[e]], v.adam_m[idx[e]], v.adam_v[idx[e]], g, *adam);
                        else v.grad[idx[e]] = g;
                        Z[cur][at[e]] = fmaf(D, z, c);
                    }
                }
                group_barrier(grp, NTT);
            }
        }
        for (int i = tid; i < RBT * s; i += NTT) {
            const int r = i / s, c = i % s;
            xs[r * s4 + c] += Z[cur][r * ld + c];
        }
        group_barrier(grp, NTT);
    }
}

// CROWN (FWD: the forward pass of its adjoint) over RBT boxes per group of warps: the image in shared memory (WSMEM,
// else read through L2) is shared by kRowGroups groups with their own buffers and barriers, so that one group's interval
// loads and row reductions run under another's products.
constexpr int kRowGroups = 4, kRowGroupThreads = NT / kRowGroups;

template <int RBT, bool WSMEM, bool FWD>
__global__ void __launch_bounds__(NT, 1) k_rows(BoundArgs a, int stride)
{
    extern __shared__ float4 smem4[];
    float *sm = reinterpret_cast<float *>(smem4);
    const NetDesc &N = a.net;
    const int nlive = live_count(a.n, a.d_n, a.row0);
    if ((int)blockIdx.x * kRowGroups * RBT >= nlive) return;
    const float *img = FWD ? a.fwd : a.bwd;
    float *p = sm;
    if (WSMEM) {
        for (int i = threadIdx.x; i < N.img_floats / 4; i += NT) smem4[i] = reinterpret_cast<const float4 *>(img)[i];
        img = sm;
        p += N.img_floats;
        __syncthreads();
    }
    const int grp = threadIdx.x / kRowGroupThreads;
    const int box0 = ((int)blockIdx.x * kRowGroups + grp) * RBT;
    if (box0 >= nlive) return;
    const int nrows = min(RBT, nlive - box0);
    p += (size_t)grp * stride;
    if (FWD) fwd_rows<RBT, kRowGroupThreads>(a, img, p, global_view(a, box0), nrows, nullptr, grp);
    else crown_rows<RBT, kRowGroupThreads>(a, img, p, global_view(a, box0), nrows, grp);
}

// ---------------------------------------------------------------------------
// Fused alpha-CROWN: the whole optimisation of a tile of RBT boxes in one CTA.
// Both network images and every per-box array (interval bounds, margin
// helpers, slopes, Adam moments, coefficients before relaxation, u*) stay in
// shared memory for all `steps` (bound, adjoint + Adam) rounds; only the best
// bound (and the final slopes, when asked for) go back to global memory.  The
// arithmetic is that of k_rows and k_adam, step for step.
// ---------------------------------------------------------------------------
__host__ __device__ inline size_t fused_box_floats(const NetDesc &N, int H, int d)
{
    const size_t hs = (size_t)H * N.sumh;
    return 6 * hs + (size_t)H * (N.sumh + N.s) + 2 * (size_t)(H + 1) * N.s + 3 * (size_t)d + 2;
}

template <int RBT, int NTT>
__global__ void __launch_bounds__(NTT) k_alpha_fused(BoundArgs a, int steps, float lr, float *alpha_out,
                                                     const AdamTable tab)
{
    __shared__ float bc_sh[2];
    extern __shared__ float4 smem4[];
    float *sm = reinterpret_cast<float *>(smem4);
    const NetDesc &N = a.net;
    const int H = a.H, d = a.d, s = N.s;
    const size_t hs = (size_t)H * N.sumh, hw = (size_t)H * (N.sumh + s), xs_ = (size_t)(H + 1) * s;
    const int nlive = live_count(a.n, a.d_n, a.row0);
    const int box0 = blockIdx.x * RBT;
    if (box0 >= nlive) return;
    const int nrows = min(RBT, nlive - box0);

    float *p = sm;
    const float *fwd = p;
    for (int i = threadIdx.x; i < N.img_floats / 4; i += NTT) smem4[i] = reinterpret_cast<const float4 *>(a.fwd)[i];
    p += N.img_floats;
    const float *bwd = p;
    for (int i = threadIdx.x; i < N.img_floats / 4; i += NTT)
        reinterpret_cast<float4 *>(p)[i] = reinterpret_cast<const float4 *>(a.bwd)[i];
    p += N.img_floats;
    RowsView v;
    float *pl = p; p += RBT * hs;
    float *ph = p; p += RBT * hs;
    v.alpha = p; p += RBT * hs;
    v.adam_m = p; p += RBT * hs;
    v.adam_v = p; p += RBT * hs;
    v.A_pre = p; p += RBT * hs;
    float *Sv = p; p += RBT * hw;
    float *xl = p; p += RBT * xs_;
    float *xu = p; p += RBT * xs_;
    float *blo = p; p += (size_t)RBT * d;
    float *bhi = p; p += (size_t)RBT * d;
    v.ustar = p; p += (size_t)RBT * d;
    v.lb = p; p += RBT;
    v.lb_best = p; p += RBT;
    float *scratch = sm + ((p - sm + 3) & ~(ptrdiff_t)3);  // float4-aligned for dense_rows
    v.pre_lo = pl;
    v.pre_hi = ph;
    v.S = Sv;
    v.x_lo = xl;
    v.x_hi = xu;
    v.lo = blo;
    v.hi = bhi;
    v.lin_coef = nullptr;
    v.margin = v.lin_const = nullptr;
    v.grad = nullptr;

    const size_t b = (size_t)box0;
    for (size_t i = threadIdx.x; i < (size_t)nrows * hs; i += NTT) {
        const float zl = a.pre_lo[b * hs + i], zu = a.pre_hi[b * hs + i];
        pl[i] = zl;
        ph[i] = zu;
        v.alpha[i] = (zu >= -zl) ? 1.f : 0.f;  // adaptive initial slopes
        v.adam_m[i] = 0.f;
        v.adam_v[i] = 0.f;
    }
    for (size_t i = threadIdx.x; i < (size_t)nrows * hw; i += NTT) Sv[i] = a.S[b * hw + i];
    for (size_t i = threadIdx.x; i < (size_t)nrows * xs_; i += NTT) {
        xl[i] = a.x_lo[b * xs_ + i];
        xu[i] = a.x_hi[b * xs_ + i];
    }
    for (size_t i = threadIdx.x; i < (size_t)nrows * d; i += NTT) {
        blo[i] = a.lo[b * d + i];
        bhi[i] = a.hi[b * d + i];
    }
    for (int r = threadIdx.x; r < RBT; r += NTT) v.lb_best[r] = -INFINITY;
    __syncthreads();

    for (int step = 1; step <= steps; ++step) {
        crown_rows<RBT, NTT>(a, bwd, scratch, v, nrows);
        __syncthreads();
        AdamStep st;
        st.lr = lr;
        if (step <= kAdamTable) {
            st.bc1 = tab.bc1[step - 1];
            st.bc2 = tab.bc2[step - 1];
        } else {
            // beyond the table: one thread forms the constants (FP64 is slow on this part)
            if (threadIdx.x == 0) {
                bc_sh[0] = (float)(1.0 - pow(0.9, (double)step));
                bc_sh[1] = (float)(1.0 - pow(0.999, (double)step));
            }
            __syncthreads();
            st.bc1 = bc_sh[0];
            st.bc2 = bc_sh[1];
        }
        fwd_rows<RBT, NTT>(a, fwd, scratch, v, nrows, &st);
        __syncthreads();
    }
    for (int r = threadIdx.x; r < nrows; r += NTT) a.lb_best[box0 + r] = v.lb_best[r];
    if (alpha_out)
        for (size_t i = threadIdx.x; i < (size_t)nrows * hs; i += NTT) alpha_out[b * hs + i] = v.alpha[i];
}

__global__ void k_alpha_init(BoundArgs a)
{
    const int nlive = live_count(a.n, a.d_n, a.row0);
    const long long total = (long long)nlive * a.H * a.net.sumh;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x)
        const_cast<float *>(a.alpha)[i] = (a.pre_hi[i] >= -a.pre_lo[i]) ? 1.f : 0.f;
}

__global__ void k_adam(float *alpha, float *m, float *v, const float *g, long long count, float lr, float bc1, float bc2)
{
    AdamStep st;
    st.lr = lr;
    st.bc1 = bc1;
    st.bc2 = bc2;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count; i += (long long)gridDim.x * blockDim.x) {
        float al = alpha[i], mi = m[i], vi = v[i];
        adam_update(al, mi, vi, g[i], st);
        alpha[i] = al;
        m[i] = mi;
        v[i] = vi;
    }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
static int max_optin_smem()
{
    int dev, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    return v - 1024;
}

// Cycles one input of a layer takes a scheduler of k_ibp with groups of rb rows, and the tile (0: 4 x 4, 1: 2 x 4,
// 2: 1 x 4, 3: 1 x 2 outputs a thread) that takes the fewest: the FMAs of the tile, the sign split of its weights (the
// ALU pipe has half the FMA pipe's width) and its loads, times the warps' passes; a tile that leaves a group fewer
// than four warps leaves schedulers without one.
static int ibp_tile(int rb, int Np, int &tile)
{
    static const int tr[4] = {4, 2, 1, 1}, tn[4] = {4, 4, 4, 2}, cost[4] = {50, 30, 22, 13};
    int best = -1;
    for (int i = 0; i < 4; ++i) {
        if (rb % tr[i]) continue;
        const int warps = ((rb / tr[i]) * (Np / tn[i]) + 31) / 32;
        const int c = (warps > 4 ? (warps + 3) / 4 : 1) * cost[i] * kIbpGroups * (warps < 4 ? 3 : 4) / 4;
        if (best < 0 || c < best) {
            best = c;
            tile = i;
        }
    }
    return best;
}

// Boxes per group of k_ibp over n boxes: the count up to `most` whose waves of tiles take the least time (per layer
// its inputs' cycles plus about 700 for the barrier, the stores and the step's share of the rest, as measured on 128-wide
// layers; networks of layers up to 64 wide go to k_ibp_warp).
static int ibp_rows(const NetDesc &N, int n, int num_sms, int most, int &tiles)
{
    int best = most;
    long long best_cost = -1;
    for (int rb = most; rb >= 1; --rb) {
        const int per = rb * kIbpGroups;
        const long long waves = ((n + per - 1) / per + num_sms - 1) / num_sms;
        long long c = 0;
        int code = 0;
        for (int l = 1; l <= N.L; ++l) {
            int tile;
            c += 700 + 16 * rb + (long long)pad4(N.dims[l - 1]) * ibp_tile(rb, pad4(N.dims[l]), tile);
            code |= tile << (2 * l);
        }
        if (best_cost < 0 || waves * c < best_cost) {
            best_cost = waves * c;
            best = rb;
            tiles = code;
        }
    }
    return best;
}

static int sm_count()
{
    int dev, v = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    return v;
}

// Which layers' columns can be stored four at a time: bit l for layer l of the [n][H][sumh] arrays (vec_h) and of S
// (vec_s).
static void ibp_vec(const BoundArgs &a, int &vec_h, int &vec_s)
{
    const NetDesc &N = a.net;
    auto al = [](const void *p) { return ((uintptr_t)p & 15) == 0; };
    vec_h = vec_s = 0;
    for (int l = 1; l <= N.L; ++l) {
        const int off = l < N.L ? N.hoff[l] : N.sumh;
        if (N.sumh % 4 == 0 && off % 4 == 0 && al(a.pre_lo) && al(a.pre_hi)) vec_h |= 1 << l;
        if ((N.sumh + N.s) % 4 == 0 && off % 4 == 0 && al(a.S)) vec_s |= 1 << l;
    }
}

cudaError_t launch_ibp(const BoundArgs &a, int num_sms, cudaStream_t st)
{
    if (a.n <= 0) return cudaSuccess;
    if (ibp_warp_takes(a)) return launch_ibp_warp(a, st);
    const NetDesc &N = a.net;
    const int budget = max_optin_smem();
    if (num_sms <= 0) num_sms = sm_count();
    int vec_h, vec_s;
    ibp_vec(a, vec_h, vec_s);
    const size_t img = N.img_floats;
    int most = 8;
    while (most >= 1 && (img + kIbpGroups * ibp_rest_floats(N, most)) * 4 > (size_t)budget) --most;
    if (most >= 4) {
        int tiles = 0;
        const int rb = ibp_rows(N, a.n, num_sms, most, tiles), per = rb * kIbpGroups;
        const size_t smem = (img + kIbpGroups * ibp_rest_floats(N, rb)) * 4;
        cudaError_t e = cudaFuncSetAttribute(k_ibp<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        k_ibp<false><<<(a.n + per - 1) / per, kIbpNT, smem, st>>>(a, rb, tiles, vec_h, vec_s, a.unchecked, 0);
    } else {
        // Whole waves of full tiles, then one wave of tiles with as few rows as hold the rest: a tile of the object-
        // manipulation network (H = 40) takes 5.1 ms with 32 rows, 4.9 with 24, 3.3 with 12 or 16, 2.5 with 8, 1.9
        // with 4.  32 rows throughout -> this: 16 boxes 6.3 -> 1.9 ms, 1200 6.3 -> 2.5, 6000 11.3 -> 7.6, 16384
        // 20.1 -> 18.5, whole waves as before.  A full tile has kIbpStreamRows rows, or the most that fit beside the
        // ring (28 or 24 of the widest layers from 113 states on).
        auto bytes = [&](int rb) { return ((size_t)kIbpStages * kIbpSpan * kMaxWidth + ibp_rest_floats(N, rb)) * 4; };
        int rows = kIbpStreamRows;
        while (rows > 4 && bytes(rows) > (size_t)budget) rows -= 4;
        if (bytes(rows) > (size_t)budget) return cudaErrorInvalidConfiguration;
        const int wave = rows * num_sms, full = a.n / wave * wave, left = a.n - full;
        auto run = [&](auto kern, int rb, int first, int boxes) {
            cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes(rb));
            if (e != cudaSuccess) return e;
            kern<<<(boxes + rb - 1) / rb, kIbpNT, bytes(rb), st>>>(a, rb, 0, vec_h, vec_s, a.unchecked, first);
            return cudaGetLastError();
        };
        const int tail = ((left + num_sms - 1) / num_sms + 3) & ~3;
        cudaError_t e = cudaSuccess;
        if (full > 0)
            e = rows == kIbpStreamRows ? run(k_ibp<true, kIbpStreamRows>, rows, 0, full) : run(k_ibp<true>, rows, 0, full);
        if (e == cudaSuccess && left > 0)
            e = run(k_ibp<true>, tail, full, left);
        if (e != cudaSuccess) return e;
    }
    return cudaGetLastError();
}

// The same call for the boxes from `row` on.
static BoundArgs from_row(BoundArgs a, int row)
{
    const size_t r = (size_t)row, hs = r * a.H * a.net.sumh, xs = r * (a.H + 1) * a.net.s;
    auto move = [](auto *&p, size_t by) {
        if (p) p += by;
    };
    a.row0 += row;
    a.n -= row;
    move(a.lo, r * a.d);
    move(a.hi, r * a.d);
    move(a.pre_lo, hs);
    move(a.pre_hi, hs);
    move(a.x_lo, xs);
    move(a.x_hi, xs);
    move(a.S, r * a.H * (a.net.sumh + a.net.s));
    move(a.lb_ibp, r);
    move(a.alpha, hs);
    move(a.lb, r);
    move(a.margin, r);
    move(a.lin_const, r);
    move(a.lb_best, r);
    move(a.lin_coef, r * a.d);
    move(a.ustar, r * a.d);
    move(a.A_pre, hs);
    move(a.grad_alpha, hs);
    return a;
}

// Rows per group of k_rows: the smallest of 1, 2, 4, 8 with which one wave of CTAs holds all boxes (a step takes a group
// about the same time with one row as with two), at most what fits in shared memory; beyond one wave, whole waves of the
// most rows and then one wave of what is left (16384 boxes of four 256-wide layers, H = 5, the gradient call 10.6 -> 10.2
// ms; two 32-wide layers, H = 40, the coefficients 1553 -> 1439 us).
template <bool FWD>
static cudaError_t launch_rows(const BoundArgs &a, int num_sms, cudaStream_t st)
{
    if (a.n <= 0) return cudaSuccess;
    const NetDesc &N = a.net;
    const size_t budget = (size_t)max_optin_smem(), img = (size_t)N.img_floats * 4;
    auto floats = [&](int rb) { return FWD ? fwd_rows_floats(N, rb) : crown_rows_floats(N, rb, a.d); };
    auto group = [&](int rb) { return ((floats(rb) + 3) & ~size_t(3)) * 4; };
    if (floats(RB) * 4 > budget) return cudaErrorInvalidConfiguration;  // (the working set of a tile of RB boxes)
    if (num_sms <= 0) num_sms = sm_count();
    // (fewer rows rather than the image out of shared memory)
    const size_t beside = img + kRowGroups * group(1) <= budget ? img : 0;
    int most = 8;
    while (most > 1 && beside + kRowGroups * group(most) > budget) most /= 2;
    auto run = [&](int rb, const BoundArgs &b, int boxes) {
        const bool wsmem = img + kRowGroups * group(rb) <= budget;
        const size_t smem = (wsmem ? img : 0) + kRowGroups * group(rb);
        auto go = [&](auto kern) {
            cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
            const int per = kRowGroups * rb;
            kern<<<(boxes + per - 1) / per, NT, smem, st>>>(b, (int)(group(rb) / 4));
            return cudaGetLastError();
        };
        switch (rb) {
            case 1: return wsmem ? go(k_rows<1, true, FWD>) : go(k_rows<1, false, FWD>);
            case 2: return wsmem ? go(k_rows<2, true, FWD>) : go(k_rows<2, false, FWD>);
            case 4: return wsmem ? go(k_rows<4, true, FWD>) : go(k_rows<4, false, FWD>);
            default: return wsmem ? go(k_rows<8, true, FWD>) : go(k_rows<8, false, FWD>);
        }
    };
    auto fit = [&](int boxes) {
        int rb = 1;
        while (rb < most && (long long)num_sms * kRowGroups * rb < boxes) rb *= 2;
        return rb;
    };
    const int wave = num_sms * kRowGroups * most, left = a.n % wave;
    int full = a.n - left;
    // (one launch where the rest would take the most rows all the same)
    if (fit(left) == most) full = a.n;
    if (full > 0) {
        BoundArgs b = a;
        b.n = full;
        const cudaError_t e = run(most, b, full);
        if (e != cudaSuccess || full == a.n) return e;
    }
    return run(fit(left), full > 0 ? from_row(a, full) : a, left);
}

cudaError_t launch_crown(const BoundArgs &a, int num_sms, cudaStream_t st) { return launch_rows<false>(a, num_sms, st); }

cudaError_t preload_ibp_crown()
{
    cudaFuncAttributes fa;
    const void *kerns[] = {(const void *)k_ibp<true>, (const void *)k_ibp<true, kIbpStreamRows>, (const void *)k_ibp<false>,
                           (const void *)k_rows<1, true, false>, (const void *)k_rows<1, false, false>,
                           (const void *)k_rows<2, true, false>, (const void *)k_rows<2, false, false>,
                           (const void *)k_rows<4, true, false>, (const void *)k_rows<4, false, false>,
                           (const void *)k_rows<8, true, false>, (const void *)k_rows<8, false, false>};
    for (const void *k : kerns) {
        cudaError_t e = cudaFuncGetAttributes(&fa, k);
        if (e != cudaSuccess) return e;
    }
    return preload_ibp_warp();
}

cudaError_t launch_alpha_fwd(const BoundArgs &a, int num_sms, cudaStream_t st) { return launch_rows<true>(a, num_sms, st); }

static size_t fused_smem(const NetDesc &N, int rb, int H, int d)
{
    const size_t rows = crown_rows_floats(N, rb, d), fw = fwd_rows_floats(N, rb);
    return (2 * (size_t)N.img_floats + (size_t)rb * fused_box_floats(N, H, d) + 4 + (rows > fw ? rows : fw)) *
           sizeof(float);
}

template <int RBT, int NTT>
static cudaError_t launch_fused_variant(const BoundArgs &a, int steps, float lr, float *alpha_out, cudaStream_t st)
{
    const size_t smem = fused_smem(a.net, RBT, a.H, a.d);
    if (smem > (size_t)max_optin_smem()) return cudaErrorInvalidConfiguration;
    cudaError_t e = cudaFuncSetAttribute(k_alpha_fused<RBT, NTT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    AdamTable tab;
    fill_adam_table(tab);
    k_alpha_fused<RBT, NTT><<<(a.n + RBT - 1) / RBT, NTT, smem, st>>>(a, steps, lr, alpha_out, tab);
    return cudaGetLastError();
}

int alpha_fused_variants() { return 3; }

bool alpha_fused_fits(const NetDesc &N, int H, int d)
{
    return fused_smem(N, 2, H, d) <= (size_t)max_optin_smem();
}

// variant 0: 2 boxes x 64 threads per CTA; 1: 4 x 128; 2: 8 x 256; < 0: the most boxes that fit in shared memory,
// at most 4.  Returns cudaErrorInvalidConfiguration when the tile does not fit.
cudaError_t launch_alpha_fused(const BoundArgs &a, int steps, float lr, float *alpha_out, int variant, cudaStream_t st)
{
    if (a.n <= 0) return cudaSuccess;
    if (variant < 0) variant = fused_smem(a.net, 4, a.H, a.d) <= (size_t)max_optin_smem() ? 1 : 0;
    switch (variant) {
        case 0: return launch_fused_variant<2, 64>(a, steps, lr, alpha_out, st);
        case 1: return launch_fused_variant<4, 128>(a, steps, lr, alpha_out, st);
        default: return launch_fused_variant<8, 256>(a, steps, lr, alpha_out, st);
    }
}

__global__ void k_fill_f32(float *p, int n, float v)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) p[i] = v;
}

cudaError_t launch_fill(float *p, int n, float v, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    k_fill_f32<<<(n + 255) / 256 < 1024 ? (n + 255) / 256 : 1024, 256, 0, st>>>(p, n, v);
    return cudaGetLastError();
}

cudaError_t launch_alpha_init(const BoundArgs &a, cudaStream_t st)
{
    if (a.n <= 0) return cudaSuccess;
    k_alpha_init<<<1024, 256, 0, st>>>(a);
    return cudaGetLastError();
}

void fill_adam_table(AdamTable &tab)
{
    for (int i = 0; i < kAdamTable; ++i) {
        tab.bc1[i] = (float)(1.0 - std::pow(0.9, i + 1));
        tab.bc2[i] = (float)(1.0 - std::pow(0.999, i + 1));
    }
}

cudaError_t launch_adam(float *alpha, float *m, float *v, const float *grad, long long count, float lr, float bc1,
                        float bc2, cudaStream_t st)
{
    if (count <= 0) return cudaSuccess;
    long long blocks = (count + 255) / 256;
    k_adam<<<(int)(blocks < 4096 ? blocks : 4096), 256, 0, st>>>(alpha, m, v, grad, count, lr, bc1, bc2);
    return cudaGetLastError();
}

}  // namespace bab
