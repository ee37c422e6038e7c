// Fused inference on groups of eight rows that stay in shared memory (sm_100a).
//
// Algorithm 2 without PCA: label_i = argmin_k ||y_i - c_k||^2, out_i = gamma_l * y_i + beta_l, for K <= 128.
//
// A row crosses the SM once: it is copied into shared memory (bulk copies of whole rows, so any row
// length goes: eight rows are a multiple of 16 bytes), scored, decided -- exactly, in the same kernel --
// and corrected from there.  With so few rows per group tcgen05 has nothing to work on (its tile
// has 64 rows at least), but the contraction is small here: mma.sync m16n8k16 with the centroids as the
// 16-row operand and the eight rows as the other wastes nothing and needs no operand staging.
//
//   team      TW warps (4 for rows of 1000) work on a group: each scores a part of the columns,
//             the partial scores meet in shared memory, then each warp decides and corrects 8 / TW rows
//   CTA       T teams around one fp16 copy of the centroids; one CTA per SM, the teams' phases
//             overlap (copy, scoring, loads of gamma and beta from L2, stores)
//
// What bounds it: latency and instruction issue -- a group's way through its phases takes about 7 us, and
// shared memory holds five groups of rows of 1000 columns per SM.  Measured against the kernels that read
// a row twice (64-row tiles with a separate exact pass; padded copies where D % 4 != 0): 1024 x 1000, K = 8
// 18 us against 62; 50 000 x 1000, K = 16 113 against 158, K = 32 142 against 262; 50 000 x 1001, K = 50 250
// against 342; 1 000 000 x 768, K = 32 1.47 ms against 2.39.
//
// Scores.  t_k = ||c_k||^2 - ||m||^2 - 2 y.(c_k - m) with m the mean of the centroids: m changes all
// scores of a row alike, and the operand c_k - m is smaller than c_k, which tightens the error bound.
// Rows are scaled by a power of two from the largest magnitude of the 64 columns at hand (no overflow,
// whatever comes later), centroids by one of their own.  The rounding errors dy, dc of the fp16 operands
// are not bounded but measured while they are made (their norms), so
//   |t - exact| <= e = 1.0625 * 2 (||dy|| c + ||y|| (1 + 2^-10) d + q ||y|| c) + 8 u a,
// c = max ||c_k - m||, d = max ||dc_k||, a = max | ||c_k||^2 - ||m||^2 |, q = (W + TW + 2) 2^-22 for the fp32
// additions of W columns per warp and of the TW warps' parts.  Centroids within 2 e of the best are
// candidates; one candidate is the label.  Several: direct-form fp32 sums of squares, a lane's D / 32 terms
// first, then a tree (relative error at most (D / 32 + 12) 2^-24), and among what these leave within that
// error direct-form fp64, lowest index on equality.
//
// Algorithm 2 with PCA (label_i = argmin_k ||z_i - c_k||^2, z_i = fp32 of V (y_i - mean)) is the same kernel: with
// w_k = V'(c_k - m) in place of c_k - m and y - mean in place of y, t_k = ||c_k||^2 - ||m||^2 - 2 (y - mean).w_k.  The
// projection is never formed for a row that its scores decide; its rounding to fp32 and that of y - mean enter the bound,
//   e += 2^-24 ||y - mean|| (||w|| + ||V||_F max ||c_k - m||).
// Several candidates: the same dot products in fp32 from w_k in fp32; for the rows that these leave (one in a thousand) a kernel
// behind this one forms the projection in fp64 and the distances in the reduced space.  50 000 x 1000, 50 components, K = 64: the projection in fp64, the assignment of
// the reduced rows and the correction took 377 us, this takes 235.
#include "cat_half.cuh"

#include <cuda_bf16.h>

namespace cat {

namespace {

constexpr int RR = 8;                    // rows of a group
constexpr int RES_MAX_THREADS = 640;     // (96 registers a thread)
constexpr int RES_MAX_TEAMS = RES_MAX_THREADS / 32;
constexpr int PREP_THREADS = 512;
constexpr int KS = 4;                    // 16-column steps that share a scale; fragments are padded to whole blocks of them
constexpr size_t RES_SMEM = 227 * 1024;

// byte offsets in dynamic shared memory
struct ResLayout {
    uint32_t bs, ak, coef, mean, part, stat, slots, bars, total;
    uint32_t part_team, slot_bytes;
};

ResLayout res_layout(int MT, int ldy, int nk, int TW, int T, int S, bool bg, bool pca)
{
    ResLayout L{};
    size_t o = 0;
    const int KP = MT * 16 + 4;
    L.bs = 0;
    o += bg ? 0 : (size_t)nk * MT * 512;
    const size_t slot_bytes = (size_t)RR * ldy * 4, part_team = (size_t)S * TW * RR * KP * 4;
    L.slot_bytes = (uint32_t)slot_bytes;
    L.part_team = (uint32_t)part_team;
    L.slots = (uint32_t)o;
    o += (size_t)T * S * slot_bytes;
    L.ak = (uint32_t)o;
    o += (size_t)MT * 16 * 4;
    L.coef = (uint32_t)o;
    o += (size_t)MT * 16 * 4;
    L.mean = (uint32_t)o;
    o += pca ? (size_t)nk * 64 : 0;
    L.part = (uint32_t)o;
    o += (size_t)T * part_team;
    L.stat = (uint32_t)o;
    o += (size_t)T * S * TW * RR * 8;   // (norm and rounding error of a row, squared)
    o = (o + 7) & ~(size_t)7;
    L.bars = (uint32_t)o;
    o += (size_t)(T * S + 1) * 8;
    L.total = o < 0x7fffffff ? (uint32_t)o : 0x7fffffffu;
    return L;
}

// What the preparation leaves for the main kernel: fragments [nk][MT][32] x 16 bytes, then per centroid
// (MT * 16 of them) ||c||^2 - ||m||^2, -2 / scale, ||c - m||^2 and the norm of its rounding error.
// With PCA also the norm of each c - m in the reduced space, the squared Frobenius norm of the components, and
// behind these the w_k in fp32.
__host__ __device__ constexpr size_t lift_offset(int MT, int nk) { return (size_t)nk * MT * 512 + ((size_t)MT * 16 * 5 + 4) * sizeof(float); }
size_t prep_bytes(int MT, int nk) { return (size_t)nk * MT * 512 + (size_t)MT * 16 * 4 * sizeof(float); }
size_t prep_bytes_pca(int MT, int nk, int D, int K) { return lift_offset(MT, nk) + (size_t)K * D * sizeof(float); }

struct ResParams {
    const float *Y, *C, *gamma, *beta;
    const unsigned char *prep;
    void *out;
    int32_t *labels;
    Control *ctl;
    int64_t N;
    int D, K;
    int ldy;       // row stride in shared memory (floats)
    int nk;        // 16-column steps of a row, a multiple of KS
    int T, S;      // teams, row slots per team
    int out_bf16;
    const float *mean;   // PCA: [D]
    uint4 *open_rows;    // PCA: [N] {row, candidates, whether their scores are the same} that fp32 has not decided
    int p;
    ResLayout L;
};

__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src),
                 "r"(bytes), "r"(bar)
                 : "memory");
}

__device__ __forceinline__ float warp_sum_f(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Two consecutive columns' fp16 roundings and what they leave, squared.
__device__ __forceinline__ uint32_t round2(f32x2 v, f32x2 &left2)
{
    const float2 x = unpack2(v);
    const __half2 h = __floats2half2_rn(x.x, x.y);
    const float2 f = __half22float2(h);
    const f32x2 d = fma2(pack2(f.x, f.y), pack2(-1.f, -1.f), v);   // (exact)
    left2 = fma2(d, d, left2);
    return *reinterpret_cast<const uint32_t *>(&h);
}

__device__ __forceinline__ float sq_diff(float y, float c, float s)
{
    const float d = y - c;
    return fmaf(d, d, s);
}

// Sum of squared differences of a row (shared memory) and two centroids, fp32, in every lane.
template <bool VEC>
__device__ __forceinline__ void distances2(const float *y, const float *c0, const float *c1, int D, int lane, float &s0, float &s1)
{
    s0 = s1 = 0.f;
    if (VEC) {
        const int D4 = D >> 2;
#pragma unroll 4
        for (int j = lane; j < D4; j += 32) {
            const float4 a = __ldg(reinterpret_cast<const float4 *>(c0) + j), b = __ldg(reinterpret_cast<const float4 *>(c1) + j);
            const float4 v = reinterpret_cast<const float4 *>(y)[j];
            s0 = sq_diff(v.x, a.x, sq_diff(v.y, a.y, sq_diff(v.z, a.z, sq_diff(v.w, a.w, s0))));
            s1 = sq_diff(v.x, b.x, sq_diff(v.y, b.y, sq_diff(v.z, b.z, sq_diff(v.w, b.w, s1))));
        }
    } else {
#pragma unroll 8
        for (int j = lane; j < D; j += 32) {
            const float a = __ldg(c0 + j), b = __ldg(c1 + j), v = y[j];
            s0 = sq_diff(v, a, s0);
            s1 = sq_diff(v, b, s1);
        }
    }
    s0 = warp_sum_f(s0);
    s1 = warp_sum_f(s1);
}

__device__ __forceinline__ double distance64(const float *y, const float *c, int D, int lane)
{
    double s = 0.0;
#pragma unroll 4
    for (int j = lane; j < D; j += 32) {
        const double d = (double)y[j] - (double)__ldg(c + j);
        s = fma(d, d, s);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

// Exact label among the candidates (bit k & 31 of word k >> 5 of the mask).  Not inlined: few rows come
// here, and its loads in flight would take registers from every row's path.
template <bool VEC>
__device__ __noinline__ int settle(const float *y, const float *C, int D, uint4 mask4, int lane)
{
    uint32_t mask[4] = {mask4.x, mask4.y, mask4.z, mask4.w};
    float dist[4];   // of candidate lane + 32 i
    float best = CUDART_INF_F;
    int first = -1, held = -1;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        dist[i] = CUDART_INF_F;
        uint32_t m = mask[i];
        while (m) {
            const int ka = 32 * i + __ffs(m) - 1;
            m &= m - 1;
            const int kb = m ? 32 * i + __ffs(m) - 1 : ka;
            m &= m ? m - 1 : 0u;
            float s0, s1;
            distances2<VEC>(y, C + (size_t)ka * D, C + (size_t)kb * D, D, lane, s0, s1);
            if (lane == (ka & 31)) dist[i] = s0;
            if (lane == (kb & 31)) dist[i] = s1;
            best = fminf(best, fminf(s0, s1));
            if (first < 0) first = ka;
        }
    }
    const float lim = fp32_sum_limit(best, D);
    int left = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        mask[i] &= __ballot_sync(0xffffffffu, !(dist[i] > lim));
        left += __popc(mask[i]);
        if (mask[i] && held < 0) held = 32 * i + __ffs(mask[i]) - 1;
    }
    if (left == 1) return held;
    double b64 = CUDART_INF;
    int l = first < 0 ? 0 : first;   // (when every distance is NaN)
#pragma unroll
    for (int i = 0; i < 4; ++i)
        for (uint32_t m = mask[i]; m; m &= m - 1) {
            const int k = 32 * i + __ffs(m) - 1;
            const double d = distance64(y, C + (size_t)k * D, D, lane);
            if (d < b64) {
                b64 = d;
                l = k;
            }
        }
    return l;
}

// (y - mean) . w for two of the w_k, fp32, in every lane; y and mean in shared memory
template <bool VEC>
__device__ __forceinline__ void dots2(const float *y, const float *mean, const float *w0, const float *w1, int D, int lane, float &s0,
                                      float &s1)
{
    s0 = s1 = 0.f;
    if (VEC) {
#pragma unroll 4
        for (int j = lane; j < (D >> 2); j += 32) {
            const float4 a = reinterpret_cast<const float4 *>(w0)[j], b = reinterpret_cast<const float4 *>(w1)[j];
            const float4 v = reinterpret_cast<const float4 *>(y)[j], m = reinterpret_cast<const float4 *>(mean)[j];
            const float4 d = make_float4(v.x - m.x, v.y - m.y, v.z - m.z, v.w - m.w);
            s0 = fmaf(d.x, a.x, fmaf(d.y, a.y, fmaf(d.z, a.z, fmaf(d.w, a.w, s0))));
            s1 = fmaf(d.x, b.x, fmaf(d.y, b.y, fmaf(d.z, b.z, fmaf(d.w, b.w, s1))));
        }
    } else {
#pragma unroll 8
        for (int j = lane; j < D; j += 32) {
            const float d = y[j] - mean[j];
            s0 = fmaf(d, w0[j], s0);
            s1 = fmaf(d, w1[j], s1);
        }
    }
    s0 = warp_sum_f(s0);
    s1 = warp_sum_f(s1);
}

// Label among the candidates (K <= 64) by the same dot products in fp32; where that does not decide, those left go to *rest and
// the result is whether their scores are all the same (those of equal centroids are).
// noise: bound on the error of a fp32 score here, the rounding of the projected row included.
template <bool VEC>
__device__ __noinline__ int settle_pca(const float *y, const float *mean, const float *lift, const float *ak, int D, uint2 mask2, float noise,
                                       int lane, uint2 *rest)
{
    uint32_t mask[2] = {mask2.x, mask2.y};
    float sc[2];   // of candidate lane + 32 i
    float best = CUDART_INF_F;
    int held = -1;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        sc[i] = CUDART_INF_F;
        uint32_t m = mask[i];
        while (m) {
            const int ka = 32 * i + __ffs(m) - 1;
            m &= m - 1;
            const int kb = m ? 32 * i + __ffs(m) - 1 : ka;
            m &= m ? m - 1 : 0u;
            float s0, s1;
            dots2<VEC>(y, mean, lift + (size_t)ka * D, lift + (size_t)kb * D, D, lane, s0, s1);
            s0 = fmaf(-2.f, s0, ak[ka]);
            s1 = fmaf(-2.f, s1, ak[kb]);
            if (lane == (ka & 31)) sc[i] = s0;
            if (lane == (kb & 31)) sc[i] = s1;
            best = fminf(best, fminf(s0, s1));
        }
    }
    const float lim = fmaxf(best, -3.4028235e38f) + 2.f * noise;
    int left = 0;
    uint32_t others = 0u;   // candidates whose score is not the smallest, bit for bit
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        mask[i] &= __ballot_sync(0xffffffffu, !(sc[i] > lim));
        others |= mask[i] & __ballot_sync(0xffffffffu, sc[i] != best);
        left += __popc(mask[i]);
        if (mask[i] && held < 0) held = 32 * i + __ffs(mask[i]) - 1;
    }
    *rest = left == 1 ? make_uint2(0u, 0u) : make_uint2(mask[0], mask[1]);
    return left > 1 ? others == 0u : (held < 0 ? 0 : held);
}

template <int TW>
__device__ __forceinline__ void team_sync(int team)
{
    if (TW == 1) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "r"(TW * 32) : "memory");
}

// rows [row0, row0 + 8) of Y into a slot (one thread)
template <bool VEC>
__device__ __forceinline__ void load_group(const ResParams &p, int64_t row0, float *slot, uint64_t *bar)
{
    const int nr = p.N - row0 < RR ? (int)(p.N - row0) : RR;
    const float *src = p.Y + (size_t)row0 * p.D;
    const uint32_t dst = smem_u32(slot), b = smem_u32(bar);
    if (VEC) {
        mbar_arrive_expect_tx(b, (uint32_t)(nr * p.D * 4));
        for (int r = 0; r < nr; ++r) bulk_load(dst + (uint32_t)(r * p.ldy * 4), src + (size_t)r * p.D, (uint32_t)(p.D * 4), b);
    } else {
        // contiguous; the last group's length need not be a multiple of 16 bytes
        const uint32_t n = (uint32_t)(nr * p.D), whole = n & ~3u;
        for (uint32_t e = whole; e < n; ++e) slot[e] = src[e];
        mbar_arrive_expect_tx(b, whole * 4);
        if (whole) bulk_load(dst, src, whole * 4, b);
    }
}

// What a lane handles at a time: four columns where rows are 16-byte aligned, else one.
template <bool VEC>
struct Unit {
    typedef float4 T;
    static constexpr int N = 4;
};
template <>
struct Unit<false> {
    typedef float T;
    static constexpr int N = 1;
};

// gamma * y + beta, y in shared memory, `e` the place in the output
__device__ __forceinline__ void correct(const ResParams &p, size_t e, const float *y, const float4 g, const float4 b)
{
    const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(y);
    const f32x2 lo = fma2(pack2(g.x, g.y), v.x, pack2(b.x, b.y)), hi = fma2(pack2(g.z, g.w), v.y, pack2(b.z, b.w));
    const float2 l = unpack2(lo), h = unpack2(hi);
    if (p.out_bf16) {
        const __nv_bfloat162 bl = __floats2bfloat162_rn(l.x, l.y), bh = __floats2bfloat162_rn(h.x, h.y);
        __stcs(reinterpret_cast<uint2 *>(reinterpret_cast<__nv_bfloat16 *>(p.out) + e),
               make_uint2(*reinterpret_cast<const uint32_t *>(&bl), *reinterpret_cast<const uint32_t *>(&bh)));
    } else
        __stcs(reinterpret_cast<float4 *>(reinterpret_cast<float *>(p.out) + e), make_float4(l.x, l.y, h.x, h.y));
}
__device__ __forceinline__ void correct(const ResParams &p, size_t e, const float *y, float g, float b)
{
    const float o = fmaf(g, y[0], b);
    if (p.out_bf16) reinterpret_cast<__nv_bfloat16 *>(p.out)[e] = __float2bfloat16_rn(o);
    else reinterpret_cast<float *>(p.out)[e] = o;
}

// One CTA per centroid (MT * 16 of them): the mean of all centroids, c - m, its norm, scale, fp16 fragments
// and what rounding left.  Also resets the control block.  A launch of its own because the columns' sums
// over all centroids are latency that every CTA of the main kernel would pay (9 us there, 4 here).
// With PCA (p > 0) the centroids are [K][p] and what becomes fragments is V'(c - m), formed in fp64.
template <bool PCA>
__global__ void __launch_bounds__(PREP_THREADS) centroid_fragments_kernel(const float *__restrict__ C, int D, int K, int MT, int nk,
                                                                          unsigned char *__restrict__ prep, Control *ctl,
                                                                          const float *__restrict__ V, int p)
{
    pdl_enter();
    extern __shared__ float4 diff4[];   // [16 nk] c - m, zero beyond D
    __shared__ float rmax[PREP_THREADS / 32], rn2[PREP_THREADS / 32], rleft[PREP_THREADS / 32];
    __shared__ double ra[PREP_THREADS / 32];
    float *diff = reinterpret_cast<float *>(diff4);
    const int k = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (k == 0 && tid == 0) {
        ctl->refine_count = 0;
        ctl->cand_count = 0;
        ctl->device_status = CAT_OK;
        ctl->refined_total = 0;
        ctl->refined_last = 0;
        ctl->grid_bar = 0;
    }
    const bool live = k < K;
    float mx = 0.f, n2 = 0.f;
    double a = 0.0;
    double *cred = reinterpret_cast<double *>(diff + 16 * nk);   // PCA: [p] c - m
    float nred = 0.f, vf2 = 0.f;
    if constexpr (PCA) {
        for (int r = tid; r < p; r += PREP_THREADS) {
            double s = 0.0;
#pragma unroll 16
            for (int q = 0; q < K; ++q) s += (double)__ldg(C + (size_t)q * p + r);
            const double m = s / (double)K, c = live ? (double)__ldg(C + (size_t)k * p + r) : m;
            cred[r] = c - m;
            nred = fmaf((float)(c - m), (float)(c - m), nred);
            a = fma(c - m, c + m, a);
        }
        __syncthreads();
    }
    for (int j = tid; j < 16 * nk; j += PREP_THREADS) {
        float d = 0.f;
        if (PCA) {
            if (live && j < D) {
                double s = 0.0;
#pragma unroll 8
                for (int r = 0; r < p; ++r) {
                    const float v = __ldg(V + (size_t)r * D + j);
                    s = fma(cred[r], (double)v, s);
                    if (k == 0) vf2 = fmaf(v, v, vf2);
                }
                d = (float)s;
                mx = fmaxf(mx, fabsf(d));
                n2 = fmaf(d, d, n2);
                reinterpret_cast<float *>(prep + lift_offset(MT, nk))[(size_t)k * D + j] = d;
            }
        } else if (live && j < D) {
            float s = 0.f;
#pragma unroll 16
            for (int q = 0; q < K; ++q) s += __ldg(C + (size_t)q * D + j);
            const float m = s / (float)K, c = __ldg(C + (size_t)k * D + j);
            d = c - m;
            mx = fmaxf(mx, fabsf(d));
            n2 = fmaf(d, d, n2);
            a = fma((double)c - (double)m, (double)c + (double)m, a);
        }
        diff[j] = d;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        n2 += __shfl_xor_sync(0xffffffffu, n2, o);
        a += __shfl_xor_sync(0xffffffffu, a, o);
        if (PCA) {
            nred += __shfl_xor_sync(0xffffffffu, nred, o);
            vf2 += __shfl_xor_sync(0xffffffffu, vf2, o);
        }
    }
    __shared__ float2 rp[PREP_THREADS / 32];
    if (lane == 0) {
        rmax[warp] = mx;
        rn2[warp] = n2;
        ra[warp] = a;
        if (PCA) rp[warp] = make_float2(nred, vf2);
    }
    __syncthreads();
    mx = 0.f;
    for (int w = 0; w < PREP_THREADS / 32; ++w) mx = fmaxf(mx, rmax[w]);
    const int sh = half_shift(mx);
    const float sc = pow2i(sh), inv = pow2i(-sh);
    uint2 *dst = reinterpret_cast<uint2 *>(prep) + ((k >> 4) * 32 + (k & 7) * 4) * 2 + ((k >> 3) & 1);
    f32x2 left = 0;
    for (int c4 = tid; c4 < nk * 4; c4 += PREP_THREADS) {
        const float4 v = diff4[c4];
        const uint32_t lo = round2(pack2(v.x * sc, v.y * sc), left), hi = round2(pack2(v.z * sc, v.w * sc), left);
        dst[((size_t)(c4 >> 2) * MT * 32 + (c4 & 3)) * 2] = make_uint2(lo, hi);
    }
    float left2 = unpack2(left).x + unpack2(left).y;
    left2 = warp_sum_f(left2);
    if (lane == 0) rleft[warp] = left2;
    __syncthreads();
    if (tid == 0) {
        n2 = left2 = 0.f;
        a = 0.0;
        for (int w = 0; w < PREP_THREADS / 32; ++w) {
            n2 += rn2[w];
            left2 += rleft[w];
            a += ra[w];
        }
        float *cw = reinterpret_cast<float *>(prep + (size_t)nk * MT * 512);
        cw[k] = (float)a;
        cw[MT * 16 + k] = -2.f * inv;
        cw[2 * MT * 16 + k] = n2;
        cw[3 * MT * 16 + k] = sqrtf(left2) * inv;
        if (PCA) {
            nred = vf2 = 0.f;
            for (int w = 0; w < PREP_THREADS / 32; ++w) {
                nred += rp[w].x;
                vf2 += rp[w].y;
            }
            cw[4 * MT * 16 + k] = sqrtf(nred);
            if (k == 0) cw[5 * MT * 16] = vf2;
        }
    }
}

// MT: groups of 16 centroids; VEC: D % 4 == 0; TW: warps per team; BG: the fragments stay in global memory (L2).
// PCA: the scores are those of the projected rows.  WIDE: see wide_steps.
template <int MT, bool VEC, int TW, bool BG, bool PCA, bool WIDE>
__global__ void __launch_bounds__(RES_MAX_THREADS, 1) apply_rows_kernel(ResParams p)
{
    pdl_enter();
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ int fail[RES_MAX_TEAMS][2];
    constexpr int KP = MT * 16 + 4;           // (2 KP = 8 mod 32: no bank conflicts among a fragment's stores)
    constexpr int LPR = 4 * TW;               // lanes that decide a row
    constexpr int KI = (MT * 16 + LPR - 1) / LPR;   // scores per lane
    constexpr int RPW = RR / TW;              // rows a warp decides and corrects
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = lane >> 2, t = lane & 3;
    const int team = warp / TW, tw = warp % TW;
    const ResLayout &L = p.L;
    const uint4 *bs = reinterpret_cast<const uint4 *>(BG ? p.prep : smem + L.bs) + lane;
    float *ak = reinterpret_cast<float *>(smem + L.ak), *coef = reinterpret_cast<float *>(smem + L.coef);
    float *slots = reinterpret_cast<float *>(smem + L.slots + team * p.S * L.slot_bytes);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + L.bars) + team * p.S;
    const int groups = (int)((p.N + RR - 1) / RR);
    // (the first groups go to different CTAs: a small batch spreads over the SMs)
    const int g_first = team * (int)gridDim.x + (int)blockIdx.x, g_step = (int)gridDim.x * p.T;
    const int slot_floats = RR * p.ldy;

    if (tid < p.T) fail[tid][0] = fail[tid][1] = 0;
    if (lane == 0 && tw == 0) {
        for (int s = 0; s < p.S; ++s) mbar_init(smem_u32(bars + s), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        if (g_first < groups) load_group<VEC>(p, (int64_t)g_first * RR, slots, bars);
    }
    // fragments of the centroids, their constants and the maxima behind the error bound
    uint64_t *prep_bar = reinterpret_cast<uint64_t *>(smem + L.bars) + p.T * p.S;
    const uint32_t frag_bytes = (uint32_t)p.nk * MT * 512;
    if (!BG && tid == 0) {
        mbar_init(smem_u32(prep_bar), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_arrive_expect_tx(smem_u32(prep_bar), frag_bytes);
        for (uint32_t o = 0; o < frag_bytes; o += 16384)
            bulk_load(smem_u32(smem + L.bs) + o, p.prep + o, frag_bytes - o < 16384 ? frag_bytes - o : 16384, smem_u32(prep_bar));
    }
    const float *cw = reinterpret_cast<const float *>(p.prep + frag_bytes);
    for (int k = tid; k < MT * 16; k += blockDim.x) {
        ak[k] = __ldg(cw + k);
        coef[k] = __ldg(cw + MT * 16 + k);
    }
    float *mean = reinterpret_cast<float *>(smem + L.mean);   // PCA: zero beyond D
    if (PCA)
        for (int j = tid; j < 16 * p.nk; j += blockDim.x) mean[j] = j < p.D ? __ldg(p.mean + j) : 0.f;
    float cmax2 = 0.f, amax = 0.f, dc = 0.f, cred = 0.f;
    for (int k = lane; k < p.K; k += 32) {
        // (a centroid that is not finite has scores that decide nothing, whatever the bound)
        amax = fmaxf(amax, fabsf(__ldg(cw + k)));
        cmax2 = fmaxf(cmax2, __ldg(cw + 2 * MT * 16 + k));
        dc = fmaxf(dc, __ldg(cw + 3 * MT * 16 + k));
        if (PCA) cred = fmaxf(cred, __ldg(cw + 4 * MT * 16 + k));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
        cmax2 = fmaxf(cmax2, __shfl_xor_sync(0xffffffffu, cmax2, o));
        dc = fmaxf(dc, __shfl_xor_sync(0xffffffffu, dc, o));
        if (PCA) cred = fmaxf(cred, __shfl_xor_sync(0xffffffffu, cred, o));
    }
    __syncthreads();
    if (!BG && !mbar_wait_warp(smem_u32(prep_bar), 0, &fail[team][0], p.ctl)) fail[team][0] = 1;

    const int nb = p.nk / KS, kb0 = tw * nb / TW, kb1 = (tw + 1) * nb / TW;   // this warp's blocks of columns
    const float slack = 1.0001f + (float)p.D * 6.0e-8f;   // covers the rounding of the running sums of squares
    const float cnorm = sqrtf(cmax2 * slack);
    // (c_k - m is rounded to fp32 before it is scaled: 2^-24 of c beside dc)
    // PCA: y - mean, and the projected row, are rounded to fp32
    const float e_z = PCA ? 5.9604645e-8f * (1.001f * cnorm + sqrtf(__ldg(cw + 5 * MT * 16) * (slack + (float)p.p * 6.0e-8f)) * cred * 1.01f) : 0.f;
    const float e_y = 1.001f * (dc * slack + 5.9604645e-8f * cnorm) +
                      (float)(16 * KS * ((nb + TW - 1) / TW) + TW + 2) * 2.3841858e-7f * cnorm + e_z;
    const float e_abs = 8.f * 5.9604645e-8f * amax + 1e-30f;   // (squares below that may have underflowed)

    int undecided = 0;
    int it = 0;
    for (int grp = g_first; grp < groups; grp += g_step, ++it) {
        const int slot = p.S == 2 ? it & 1 : 0;
        const uint32_t phase = (uint32_t)(p.S == 2 ? it >> 1 : it) & 1u;
        const int64_t row0 = (int64_t)grp * RR;
        const float *rows = slots + slot * slot_floats;
        float *part = reinterpret_cast<float *>(smem + L.part + team * L.part_team) + slot * TW * RR * KP;
        float2 *stat = reinterpret_cast<float2 *>(smem + L.stat) + (team * p.S + slot) * TW * RR;

        if (!mbar_wait_warp(smem_u32(bars + slot), phase, &fail[team][it & 1], p.ctl)) fail[team][it & 1] = 1;

        // ---- this warp's columns, 64 at a time: largest magnitude of each row, then partial scores
        {
            const float *y = rows + g * p.ldy + 4 * t;
            f32x2 n2 = 0;
            float left2 = 0.f;
            float tot[MT][4];
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int q = 0; q < 4; ++q) tot[m][q] = 0.f;
#pragma unroll 1
            for (int kb = kb0; kb < kb1; ++kb) {
                f32x2 v[KS][2];
                const float *yb = y + kb * (16 * KS);
                if ((kb + 1) * (16 * KS) <= p.D) {
#pragma unroll
                    for (int u = 0; u < KS; ++u) {
                        if (VEC) {
                            const ulonglong2 w = *reinterpret_cast<const ulonglong2 *>(yb + u * 16);
                            v[u][0] = w.x;
                            v[u][1] = w.y;
                        } else {
                            v[u][0] = pack2(yb[u * 16], yb[u * 16 + 1]);
                            v[u][1] = pack2(yb[u * 16 + 2], yb[u * 16 + 3]);
                        }
                    }
                } else {
                    const int rem = p.D - kb * (16 * KS) - 4 * t;   // columns left from this lane's first
#pragma unroll
                    for (int u = 0; u < KS; ++u) {
                        v[u][0] = pack2(u * 16 < rem ? yb[u * 16] : 0.f, u * 16 + 1 < rem ? yb[u * 16 + 1] : 0.f);
                        v[u][1] = pack2(u * 16 + 2 < rem ? yb[u * 16 + 2] : 0.f, u * 16 + 3 < rem ? yb[u * 16 + 3] : 0.f);
                    }
                }
                if (PCA) {
#pragma unroll
                    for (int u = 0; u < KS; ++u) {
                        const ulonglong2 m = *reinterpret_cast<const ulonglong2 *>(mean + kb * (16 * KS) + u * 16 + 4 * t);
                        v[u][0] = fma2(m.x, pack2(-1.f, -1.f), v[u][0]);
                        v[u][1] = fma2(m.y, pack2(-1.f, -1.f), v[u][1]);
                    }
                }
                float mx = 0.f;
#pragma unroll
                for (int u = 0; u < KS; ++u) {
                    const float2 a = unpack2(v[u][0]), c = unpack2(v[u][1]);
                    mx = fmaxf(fmaxf(mx, fmaxf(fabsf(a.x), fabsf(a.y))), fmaxf(fabsf(c.x), fabsf(c.y)));
                    n2 = fma2(v[u][0], v[u][0], n2);
                    n2 = fma2(v[u][1], v[u][1], n2);
                }
                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
                const int sh = half_shift(mx);
                const float sc = pow2i(sh), inv = pow2i(-sh);
                const f32x2 sc2 = pack2(sc, sc);
                float acc[MT][4];
                f32x2 l2 = 0;
#pragma unroll
                for (int m = 0; m < MT; ++m)
#pragma unroll
                    for (int q = 0; q < 4; ++q) acc[m][q] = 0.f;
#pragma unroll
                for (int u = 0; u < KS; ++u) {
                    const uint32_t b0 = round2(mul2(v[u][0], sc2), l2), b1 = round2(mul2(v[u][1], sc2), l2);
#pragma unroll
                    for (int m = 0; m < MT; ++m) {
                        // fragment order of a 16 x 16 operand: rows g and g + 8, columns 4 t ... 4 t + 3 in both operands
                        const uint4 f = BG ? __ldg(bs + ((kb * KS + u) * MT + m) * 32) : bs[((kb * KS + u) * MT + m) * 32];
                        mma_16816(acc[m], make_uint4(f.x, f.z, f.y, f.w), b0, b1);
                    }
                }
                left2 = fmaf((unpack2(l2).x + unpack2(l2).y) * inv, inv, left2);
                const float i0 = __shfl_sync(0xffffffffu, inv, 8 * t), i1 = __shfl_sync(0xffffffffu, inv, 8 * t + 4);
#pragma unroll
                for (int m = 0; m < MT; ++m)
#pragma unroll
                    for (int q = 0; q < 4; ++q) tot[m][q] = fmaf(acc[m][q], q & 1 ? i1 : i0, tot[m][q]);
            }
            float *pw = part + tw * RR * KP + 2 * t * KP + g;
#pragma unroll
            for (int m = 0; m < MT; ++m) {
                pw[m * 16] = tot[m][0];
                pw[m * 16 + KP] = tot[m][1];
                pw[m * 16 + 8] = tot[m][2];
                pw[m * 16 + KP + 8] = tot[m][3];
            }
            float nn = unpack2(n2).x + unpack2(n2).y;
            nn += __shfl_xor_sync(0xffffffffu, nn, 1);
            left2 += __shfl_xor_sync(0xffffffffu, left2, 1);
            nn += __shfl_xor_sync(0xffffffffu, nn, 2);
            left2 += __shfl_xor_sync(0xffffffffu, left2, 2);
            if (t == 0) stat[tw * RR + g] = make_float2(nn, left2);
        }
        team_sync<TW>(team);
        if (fail[team][it & 1]) break;   // the same for the whole team: written before the barrier only
        // every warp of the team is through with the group before this one: its slot is free
        if (p.S == 2 && lane == 0 && tw == 0 && grp + g_step < groups)
            load_group<VEC>(p, (int64_t)(grp + g_step) * RR, slots + (slot ^ 1) * slot_floats, bars + (slot ^ 1));

        // ---- decide this warp's rows, LPR lanes each
        int label;   // of row tw + (lane / LPR) TW; -1: beyond the matrix, or left to the kernel behind this one
        {
            const int r = tw + (lane / LPR) * TW, l = lane % LPR;
            const uint32_t mine = LPR == 32 ? 0xffffffffu : ((1u << (LPR & 31)) - 1u) << (lane / LPR * LPR);
            const bool live = row0 + r < p.N;
            float yn2 = 0.f, left2 = 0.f;
#pragma unroll
            for (int w = 0; w < TW; ++w) {
                const float2 s = stat[w * RR + r];
                yn2 += s.x;
                left2 += s.y;
            }
            float sc[KI];
            float best = CUDART_INF_F;
            int bk = 0;
#pragma unroll
            for (int i = 0; i < KI; ++i) {
                const int k = l + LPR * i;
                float s = 0.f;
#pragma unroll
                for (int w = 0; w < TW; ++w) s += part[(w * RR + r) * KP + k];
                sc[i] = k < p.K ? fmaf(coef[k], s, ak[k]) : CUDART_INF_F;
                if (sc[i] < best) {
                    best = sc[i];
                    bk = k;
                }
            }
            const float own = best;
#pragma unroll
            for (int o = LPR / 2; o > 0; o >>= 1) best = fminf(best, __shfl_xor_sync(0xffffffffu, best, o));
            const float e = 1.0625f * 2.f * (sqrt_approx(left2 * slack) * cnorm + sqrt_approx(yn2 * slack) * e_y) + e_abs;
            // (a score that overflowed downwards is no lower than the lowest finite one as far as the bound goes)
            const float lim = fmaxf(best, -3.4028235e38f) + 2.f * e;
            int cands = 0;
#pragma unroll
            for (int i = 0; i < KI; ++i) cands += __popc(__ballot_sync(0xffffffffu, l + LPR * i < p.K && !(sc[i] > lim)) & mine);
            const uint32_t won = __ballot_sync(0xffffffffu, own == best) & mine;
            label = __shfl_sync(0xffffffffu, bk, won ? __ffs(won) - 1 : lane);
            uint32_t open = __ballot_sync(0xffffffffu, cands != 1 && live && l == 0);
            undecided += __popc(open);
            while (open) {
                // rows with several candidates, one after the other
                const int src = __ffs(open) - 1, ro = tw + (src / LPR) * TW;
                open &= open - 1;
                const float lm = __shfl_sync(0xffffffffu, lim, src);
                uint32_t mask[4] = {0u, 0u, 0u, 0u};
#pragma unroll
                for (int i = 0; i < KI; ++i) {
                    const uint32_t bl = __ballot_sync(0xffffffffu, l + LPR * i < p.K && !(sc[i] > lm));
                    mask[i * LPR / 32] |= (bl >> src & (LPR == 32 ? 0xffffffffu : (1u << (LPR & 31)) - 1u)) << (i * LPR % 32);
                }
                int exact;
                if constexpr (PCA) {
                    // (fp32 sums of D / 32 terms a lane, then a tree; w_k rounded to fp32)
                    const float yn = __shfl_sync(0xffffffffu, sqrt_approx(yn2 * slack), src);
                    const float noise = 1.0625f * 2.f * yn * (((float)p.D * 0.03125f + 13.f) * 5.9604645e-8f * cnorm + e_z) + e_abs;
                    uint2 rest;
                    exact = settle_pca<VEC>(rows + ro * p.ldy, mean, reinterpret_cast<const float *>(p.prep + lift_offset(MT, p.nk)), ak, p.D,
                                            make_uint2(mask[0], mask[1]), noise, lane, &rest);
                    if ((rest.x | rest.y) != 0u) {
                        // (left as it is: the kernel behind this one reads the row again, and Y may be the output)
                        if (lane == 0) p.open_rows[atomicAdd(&p.ctl->refine_count, 1)] = make_uint4((uint32_t)(row0 + ro), rest.x, rest.y, (uint32_t)exact);
                        exact = -1;
                    }
                } else
                    exact = settle<VEC>(rows + ro * p.ldy, p.C, p.D, make_uint4(mask[0], mask[1], mask[2], mask[3]), lane);
                if (lane / LPR == src / LPR) label = exact;
            }
            if (l == 0 && live && (!PCA || label >= 0)) p.labels[row0 + r] = label;
            if (!live) label = -1;
        }

        // ---- correct them, several loads of gamma and of beta per lane in flight
        typedef typename Unit<VEC>::T UT;
        constexpr int V = Unit<VEC>::N;
        const int DV = p.D / V;
        if (TW >= 4) {
            // column steps at a time, for each of the warp's rows
            constexpr int U = VEC ? (TW == 8 ? 4 : 2) : (TW == 8 || WIDE ? 8 : 4);
            int lq[RPW];
#pragma unroll
            for (int q = 0; q < RPW; ++q) lq[q] = __shfl_sync(0xffffffffu, label, q * LPR);
#pragma unroll 1
            for (int j0 = lane; j0 < DV; j0 += 32 * U) {
                UT gv[RPW][U], bv[RPW][U];
#pragma unroll
                for (int q = 0; q < RPW; ++q) {
                    const size_t o = (size_t)(lq[q] < 0 ? 0 : lq[q]) * p.D + (size_t)j0 * V;
                    const UT *ga = reinterpret_cast<const UT *>(p.gamma + o), *be = reinterpret_cast<const UT *>(p.beta + o);
#pragma unroll
                    for (int u = 0; u < U; ++u)
                        if (j0 + 32 * u < DV) {
                            gv[q][u] = __ldg(ga + 32 * u);
                            bv[q][u] = __ldg(be + 32 * u);
                        }
                }
#pragma unroll
                for (int q = 0; q < RPW; ++q) {
                    if (lq[q] < 0) continue;
                    const int r = tw + q * TW;
                    const float *y = rows + r * p.ldy + j0 * V;
                    const size_t o = (size_t)(row0 + r) * p.D + (size_t)j0 * V;
#pragma unroll
                    for (int u = 0; u < U; ++u)
                        if (j0 + 32 * u < DV) correct(p, o + 32 * u * V, y + 32 * u * V, gv[q][u], bv[q][u]);
                }
            }
        } else {
            // several short rows per warp, as one list of elements so that loads of all rows are in flight
            constexpr int U = VEC ? 3 : 6;
            const int n = RPW * DV;
#pragma unroll 1
            for (int base = 0; base < n; base += 32 * U) {
                UT gv[U], bv[U];
                int yo[U];   // place in shared memory, -1: nothing
                size_t eo[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int e = base + lane + 32 * u;
                    const int q = e < n ? e / DV : 0;
                    const int j = (e - q * DV) * V, r = tw + q * TW;
                    const int lb = __shfl_sync(0xffffffffu, label, q * LPR);
                    yo[u] = e < n && lb >= 0 ? r * p.ldy + j : -1;
                    eo[u] = (size_t)(row0 + r) * p.D + (size_t)j;
                    if (yo[u] >= 0) {
                        const size_t o = (size_t)lb * p.D + (size_t)j;
                        gv[u] = __ldg(reinterpret_cast<const UT *>(p.gamma + o));
                        bv[u] = __ldg(reinterpret_cast<const UT *>(p.beta + o));
                    }
                }
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (yo[u] >= 0) correct(p, eo[u], rows + yo[u], gv[u], bv[u]);
            }
        }
        if (p.S == 1) {
            // one slot: it is free once the whole team has read its rows
            team_sync<TW>(team);
            if (lane == 0 && tw == 0 && grp + g_step < groups) load_group<VEC>(p, (int64_t)(grp + g_step) * RR, slots, bars);
        }
    }
    if (lane == 0 && undecided) {
        atomicAdd(reinterpret_cast<unsigned long long *>(&p.ctl->refined_last), (unsigned long long)undecided);
        atomicAdd(reinterpret_cast<unsigned long long *>(&p.ctl->refined_total), (unsigned long long)undecided);
    }
}

// The rows that fp32 has not decided, a CTA each: the projection in fp64, rounded to fp32, and the candidates' distances to it
// in fp64, lowest index on equality; then the correction.  Candidates that are equal to the first one have its distance, so a row
// that has no others needs no projection (50 000 x 1000, 50 components, K = 64 in 32 pairs, which leaves every row to this
// kernel: 2310 us a call with projections, 541 without).  (Y may be `out`: a row is read before it is written, by the thread
// that writes it.)  A launch of its own: a warp of the kernel above
// would be at one such row for as long as it takes its team to go through three groups of rows.
constexpr int OPEN_THREADS = 256;
constexpr int OPEN_MAX_D = 1024;
__global__ void __launch_bounds__(OPEN_THREADS) open_rows_kernel(const float *Y, const float *__restrict__ C, int D, int K, int p,
                                                                 const float *__restrict__ mean, const float *__restrict__ comps,
                                                                 const float *__restrict__ gamma, const float *__restrict__ beta,
                                                                 float *out, int32_t *__restrict__ labels,
                                                                 const uint4 *__restrict__ open_rows, const Control *ctl)
{
    pdl_enter();
    extern __shared__ double xs[];   // [D] y - mean, then [p] the projected row
    __shared__ double s_dist[64];
    __shared__ int s_label;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float *z = reinterpret_cast<float *>(xs + D);
    constexpr int PER = OPEN_MAX_D / OPEN_THREADS;   // columns a thread has
    const int n = ctl->refine_count;
    for (int i = blockIdx.x; i < n; i += gridDim.x) {
        const uint4 e = open_rows[i];
        const float *y = Y + (size_t)e.x * D;
        const int first = e.y ? __ffs(e.y) - 1 : 31 + __ffs(e.z);
        float yv[PER], mv[PER];   // (read here and stored from here: a load behind a store that may be to the same place would wait for it)
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const int j = tid + u * OPEN_THREADS;
            yv[u] = j < D ? y[j] : 0.f;
            mv[u] = j < D ? __ldg(mean + j) : 0.f;
        }
        bool same = e.w != 0u;
        if (same)
            for (unsigned long long left = (unsigned long long)e.z << 32 | e.y; left &= left - 1;) {
                const float *c = C + (size_t)(__ffsll((long long)left) - 1) * p, *c0 = C + (size_t)first * p;
                for (int r = tid; r < p; r += OPEN_THREADS) same &= __ldg(c + r) == __ldg(c0 + r);
            }
#pragma unroll
        for (int u = 0; u < PER; ++u)
            if (tid + u * OPEN_THREADS < D) xs[tid + u * OPEN_THREADS] = (double)yv[u] - (double)mv[u];
        const bool one = __syncthreads_and(same);
        if (!one) {
            // (eight components of a warp side by side, 32 loads in flight per lane)
            for (int r0 = warp * 8; r0 < p; r0 += OPEN_THREADS / 32 * 8) {
                double s[8];
                const float *v[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    s[q] = 0.0;
                    v[q] = comps + (size_t)(r0 + q < p ? r0 + q : r0) * D;
                }
                for (int j0 = lane; j0 < D; j0 += 128) {
                    float c[4][8];
#pragma unroll
                    for (int u = 0; u < 4; ++u)
#pragma unroll
                        for (int q = 0; q < 8; ++q) c[u][q] = j0 + 32 * u < D ? __ldg(v[q] + j0 + 32 * u) : 0.f;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const double x = j0 + 32 * u < D ? xs[j0 + 32 * u] : 0.0;
#pragma unroll
                        for (int q = 0; q < 8; ++q) s[q] = fma(x, (double)c[u][q], s[q]);
                    }
                }
#pragma unroll
                for (int q = 0; q < 8; ++q) {
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) s[q] += __shfl_xor_sync(0xffffffffu, s[q], o);
                    if (lane == 0 && r0 + q < p) z[r0 + q] = (float)s[q];
                }
            }
            __syncthreads();
            for (int k = warp; k < K; k += OPEN_THREADS / 32) {
                if (!((k < 32 ? e.y >> k : e.z >> (k - 32)) & 1u)) continue;
                double s = 0.0;
                for (int r = lane; r < p; r += 32) {
                    const double d = (double)z[r] - (double)__ldg(C + (size_t)k * p + r);
                    s = fma(d, d, s);
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                if (lane == 0) s_dist[k] = s;
            }
            __syncthreads();
        }
        if (tid == 0) {
            double best = CUDART_INF;
            int l = first;   // (also when every distance is infinite or NaN)
            if (!one)
                for (unsigned long long left = (unsigned long long)e.z << 32 | e.y; left; left &= left - 1) {
                    const int k = __ffsll((long long)left) - 1;
                    if (s_dist[k] < best) {
                        best = s_dist[k];
                        l = k;
                    }
                }
            s_label = l;
            labels[e.x] = l;
        }
        __syncthreads();
        const size_t o = (size_t)s_label * D;
        float gv[PER], bv[PER];
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const int j = tid + u * OPEN_THREADS;
            gv[u] = j < D ? __ldg(gamma + o + j) : 0.f;
            bv[u] = j < D ? __ldg(beta + o + j) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < PER; ++u)
            if (tid + u * OPEN_THREADS < D) out[(size_t)e.x * D + tid + u * OPEN_THREADS] = fmaf(gv[u], yv[u], bv[u]);
        __syncthreads();
    }
}

struct ResPlan {
    int MT, ldy, nk, TW, T, S;
    bool bg;
    ResLayout L;
};

// Teams, warps per team and where the fragments live, for a shape; false where two groups of rows do not fit.
//   warps per team   a warp's part of a row is 128 to 256 columns; shorter parts pay more for the exchange of
//                    the partial scores (50 000 x 1000, K = 16: 113 us with 4 warps per team, 131 with 8)
//   teams            as many as fit (same shape: 132, 125, 113 us with 3, 4, 5 teams)
//   fragments        in shared memory as long as that leaves sixteen warps, else in L2: 50 000 x 600, K = 64
//                    takes 112 us from shared memory (5 teams) and 135 from L2; 50 000 x 1000, K = 60 270 us (2 teams)
//                    and 205 (5 teams), 20 000 x 2047, K = 64 237 us from L2 where shared memory has no room
bool res_plan(int64_t N, int D, int K, ResPlan *pl, bool pca = false)
{
    if (N < 1 || D < 1 || K < 2 || K > 128) return false;
    const int m16 = (K + 15) / 16;
    pl->MT = m16 <= 4 ? m16 : 8;
    pl->nk = (D + 16 * KS - 1) / (16 * KS) * KS;
    pl->TW = D > 1024 ? 8 : (D > 256 ? 4 : (D > 128 ? 2 : 1));
    // rows 16 floats off a multiple of the 32 banks: a fragment's 128-bit reads of two rows touch all banks
    pl->ldy = D % 4 == 0 ? (D + 15) / 32 * 32 + 16 : D;
    for (int bg = 0; bg < 2; ++bg)
        for (int T = RES_MAX_THREADS / 32 / pl->TW; T >= 2 && (bg || T * pl->TW >= 16); --T)
            for (int S = 2; S >= 1; --S) {
                pl->L = res_layout(pl->MT, pl->ldy, pl->nk, pl->TW, T, S, bg != 0, pca);
                if (pl->L.total + 1024 <= RES_SMEM) {
                    pl->T = T;
                    pl->S = S;
                    pl->bg = bg != 0;
                    return true;
                }
            }
    return false;
}

// Eight column steps of gamma and beta in flight in place of four, for scalar rows of 257 to 1024 columns: half as many waits for
// L2, but registers that spill, in the scores' loops too.  Which weighs more was measured (49 999 rows, us with four / eight):
//   K to 16     long rows with many centroids gain: 1001, K = 12 143 / 138, K = 16 141 / 134 (15 000 rows, K = 10 63 / 60); 1001,
//               K = 4 114 / 118; 513, K = 16 76 / 78; 301, K = 16 45 / 50
//   K to 32     none: 1001, K = 32 153 / 164; 301 53 / 60
//   K to 48     777, K = 40 183 / 145; 423 86 / 85; 301 63 / 65
//   K to 64     1001, K = 64 258 / 238; 777 199 / 188; 641 147 / 158
//   above       short rows gain: 301, K = 72 114 / 109; 423 182 / 194; 1001, K = 128 394 / 425
//   with PCA    none: 2 to 18 % longer with eight
template <int MT>
bool wide_steps(int D, int K)
{
    switch (MT) {
    case 1: return K > 8 && D > 700;
    case 2: return false;
    case 3: return D > 400;
    case 4: return D > 700;
    default: return D <= 384;
    }
}

template <int MT, bool VEC, int TW, bool BG, bool PCA = false, bool WIDE = false>
cudaError_t launch_rows(const ResPlan &pl, const ResParams &p, cudaStream_t s)
{
    if constexpr (!VEC && TW == 4 && MT != 2 && !PCA && !WIDE)
        if (wide_steps<MT>(p.D, p.K)) return launch_rows<MT, VEC, TW, BG, PCA, true>(pl, p, s);
    auto kern = apply_rows_kernel<MT, VEC, TW, BG, PCA, WIDE>;
    // (the same value whatever the shape: several threads may be launching)
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(RES_SMEM - 1024));
    if (e != cudaSuccess) return e;
    const int64_t groups = (p.N + RR - 1) / RR;
    const int64_t grid = groups < tc_sm_count() ? groups : tc_sm_count();
    e = launch_pdl(kern, dim3((unsigned)grid), dim3((unsigned)(pl.T * TW * 32)), pl.L.total, s, p);
    count_launch();
    return e;
}

template <bool VEC, int TW>
cudaError_t launch_rows_mt(const ResPlan &pl, const ResParams &p, cudaStream_t s)
{
    if constexpr (TW >= 4)   // (shorter rows always leave room)
        if (pl.bg) switch (pl.MT) {
            case 1: return launch_rows<1, VEC, TW, true>(pl, p, s);
            case 2: return launch_rows<2, VEC, TW, true>(pl, p, s);
            case 3: return launch_rows<3, VEC, TW, true>(pl, p, s);
            case 4: return launch_rows<4, VEC, TW, true>(pl, p, s);
            default: return launch_rows<8, VEC, TW, true>(pl, p, s);
            }
    if (pl.bg) return cudaErrorInvalidValue;
    switch (pl.MT) {
    case 1: return launch_rows<1, VEC, TW, false>(pl, p, s);
    case 2: return launch_rows<2, VEC, TW, false>(pl, p, s);
    case 3: return launch_rows<3, VEC, TW, false>(pl, p, s);
    case 4: return launch_rows<4, VEC, TW, false>(pl, p, s);
    default: return launch_rows<8, VEC, TW, false>(pl, p, s);
    }
}

template <bool VEC>
cudaError_t launch_rows_tw(const ResPlan &pl, const ResParams &p, cudaStream_t s)
{
    switch (pl.TW) {
    case 1: return launch_rows_mt<VEC, 1>(pl, p, s);
    case 2: return launch_rows_mt<VEC, 2>(pl, p, s);
    case 4: return launch_rows_mt<VEC, 4>(pl, p, s);
    default: return launch_rows_mt<VEC, 8>(pl, p, s);
    }
}

}  // namespace

bool apply_rows_supported(int64_t N, int D, int K)
{
    ResPlan pl;
    return res_plan(N, D, K, &pl);
}

size_t apply_rows_prep_bytes(int64_t N, int D, int K)
{
    ResPlan pl;
    return res_plan(N, D, K, &pl) ? prep_bytes(pl.MT, pl.nk) : 0;
}

cudaError_t launch_apply_rows(const float *Y, int64_t N, int D, int K, const float *C, const float *gamma, const float *beta,
                              void *out, bool out_bf16, int32_t *labels, Control *ctl, void *prep, cudaStream_t s)
{
    ResPlan pl;
    if (!res_plan(N, D, K, &pl)) return cudaErrorInvalidValue;
    cudaError_t e = launch_pdl(centroid_fragments_kernel<false>, dim3((unsigned)pl.MT * 16), dim3(PREP_THREADS), (size_t)pl.nk * 64, s, C, D, K,
                               pl.MT, pl.nk, reinterpret_cast<unsigned char *>(prep), ctl, nullptr, 0);
    if (e != cudaSuccess) return e;
    count_launch();
    ResParams p{Y, C, gamma, beta, reinterpret_cast<const unsigned char *>(prep), out, labels, ctl, N, D, K, pl.ldy, pl.nk, pl.T, pl.S,
                out_bf16 ? 1 : 0, nullptr, nullptr, 0, pl.L};
    return D % 4 == 0 ? launch_rows_tw<true>(pl, p, s) : launch_rows_tw<false>(pl, p, s);
}

bool apply_rows_pca_supported(int64_t N, int D, int K)
{
    ResPlan pl;
    return D <= OPEN_MAX_D && K <= 64 && res_plan(N, D, K, &pl, true);
}

size_t apply_rows_pca_prep_bytes(int64_t N, int D, int K)
{
    ResPlan pl;
    return apply_rows_pca_supported(N, D, K) && res_plan(N, D, K, &pl, true) ? prep_bytes_pca(pl.MT, pl.nk, D, K) : 0;
}

template <bool VEC, int TW>
static cudaError_t launch_rows_pca(const ResPlan &pl, const ResParams &p, cudaStream_t s)
{
    if constexpr (TW >= 4)
        if (pl.bg) switch (pl.MT) {
            case 1: return launch_rows<1, VEC, TW, true, true>(pl, p, s);
            case 2: return launch_rows<2, VEC, TW, true, true>(pl, p, s);
            case 3: return launch_rows<3, VEC, TW, true, true>(pl, p, s);
            default: return launch_rows<4, VEC, TW, true, true>(pl, p, s);
            }
    if (pl.bg) return cudaErrorInvalidValue;
    switch (pl.MT) {
    case 1: return launch_rows<1, VEC, TW, false, true>(pl, p, s);
    case 2: return launch_rows<2, VEC, TW, false, true>(pl, p, s);
    case 3: return launch_rows<3, VEC, TW, false, true>(pl, p, s);
    default: return launch_rows<4, VEC, TW, false, true>(pl, p, s);
    }
}

cudaError_t launch_apply_rows_pca(const float *Y, int64_t N, int D, int K, int p, const float *mean, const float *comps, const float *C,
                                  const float *gamma, const float *beta, float *out, int32_t *labels, Control *ctl, void *prep,
                                  void *open_rows, cudaStream_t s)
{
    ResPlan pl;
    if (!apply_rows_pca_supported(N, D, K) || !res_plan(N, D, K, &pl, true)) return cudaErrorInvalidValue;
    cudaError_t e = launch_pdl(centroid_fragments_kernel<true>, dim3((unsigned)pl.MT * 16), dim3(PREP_THREADS),
                               (size_t)pl.nk * 64 + (size_t)p * sizeof(double), s, C, D, K, pl.MT, pl.nk,
                               reinterpret_cast<unsigned char *>(prep), ctl, comps, p);
    if (e != cudaSuccess) return e;
    count_launch();
    ResParams q{Y, C, gamma, beta, reinterpret_cast<const unsigned char *>(prep), out, labels, ctl, N, D, K, pl.ldy, pl.nk, pl.T, pl.S, 0,
                mean, reinterpret_cast<uint4 *>(open_rows), p, pl.L};
    const bool vec = D % 4 == 0;
    switch (pl.TW) {
    case 1: e = vec ? launch_rows_pca<true, 1>(pl, q, s) : launch_rows_pca<false, 1>(pl, q, s); break;
    case 2: e = vec ? launch_rows_pca<true, 2>(pl, q, s) : launch_rows_pca<false, 2>(pl, q, s); break;
    case 4: e = vec ? launch_rows_pca<true, 4>(pl, q, s) : launch_rows_pca<false, 4>(pl, q, s); break;
    default: return cudaErrorInvalidValue;
    }
    if (e != cudaSuccess) return e;
    e = launch_pdl(open_rows_kernel, dim3((unsigned)tc_sm_count() * 4), dim3(OPEN_THREADS), (size_t)D * sizeof(double) + (size_t)p * sizeof(float), s, Y, C,
                   D, K, p, mean, comps, gamma, beta, out, labels, reinterpret_cast<const uint4 *>(open_rows), ctl);
    count_launch();
    return e;
}

}  // namespace cat
