// Inference on short rows, a warp at a time (sm_100a).
//
// Algorithm 2 without PCA: label_i = argmin_k ||y_i - c_k||^2, out_i = gamma_l * y_i + beta_l, for rows of 32 to 128
// columns in whole steps of sixteen.  A warp takes sixteen rows from the load to the store by itself: they stay in its
// registers in the layout of the A operand of mma.sync m16n8k16 (lane (g, t): columns 4 t ... 4 t + 3 of every step, rows g
// and g + 8), so that scores, decision, exact settlement and correction need no hand-over.  The centroids (fp32, and
// fp16 fragments of them) and gamma and beta sit in shared memory.
//
// The kernel this takes such calls from (csrc/cat_small.cu) passes a tile of 128 rows through five warp roles, whose
// hand-overs bounded it.  tcgen05 would bring them back: its accumulators are read by other warps than those that
// wait for its operands; the contraction is small here (K <= 128, D <= 128).
// Only the tiles of sixteen centroids that exist are formed (all eight from K = 65 on before: 80 000 x 64, K = 80 30.6 us, 26.0 so, 28.1
// in the persistent kernel; 80 000 x 32, K = 70 22.0, 18.5 and 20.3).
// The next group's rows are on their way into shared memory (cp.async, every lane what it will read itself) while this one's
// are worked on.
//   bound: instruction issue, about 700 instructions a group; 11 us are start, centroids and end.  200 704 x 64, K = 64 (floor
//   16 us): 48 - 53 us in the persistent kernel, 36.7 without the rows fetched ahead and with labels beside the scores, 35.1 now.
//   Sixteen rows a warp: the A operand's height; thirty-two do not fit into the registers beside the scores.
//
// Scores and error bound as in csrc/cat_apply_rows.cu: t_k = ||c_k||^2 - ||m||^2 - 2 y.(c_k - m), m the centroids' mean; the
// rounding errors of the fp16 operands are measured.  Rows with several centroids within the bound are settled by the
// quad of lanes that has the row: direct-form fp32 sums of squares, a lane's D / 4 terms first, and what these leave
// within their error in fp64, lowest index on equality.
#include "cat_half.cuh"

#include <cuda_bf16.h>

namespace cat {

namespace {

constexpr size_t SH_SMEM = 220 * 1024;

struct ShortParams {
    const float *Y, *C, *gamma, *beta;
    void *out;
    int32_t *labels;
    Control *ctl;
    int64_t N;
    int K, nt;         // nt: tiles of sixteen centroids
};

// threads by steps of columns: what a row's registers allow
__host__ __device__ constexpr int short_threads(int nks) { return nks <= 4 ? 512 : (nks <= 6 ? 384 : 320); }
// row stride of what is read by label: 64 bytes off a multiple of 128, so that two rows in a phase collide half as often
__host__ __device__ constexpr int short_ld(int D) { return D % 32 == 0 ? D + 16 : D; }
size_t short_smem(int D, int K, bool ahead)
{
    const size_t nt = (K + 15) / 16;
    const size_t rows = ahead ? (size_t)short_threads(D / 16) / 32 * 16 * D * 4 : 0;
    return rows + (size_t)3 * K * short_ld(D) * 4 + nt * 16 * D * 2 + nt * 16 * 2 * 4 + (size_t)D * 4;
}

__device__ __forceinline__ float dist4(float4 y, float4 c, float s)
{
    const float a = y.x - c.x, b = y.y - c.y, d = y.z - c.z, e = y.w - c.w;
    return fmaf(e, e, fmaf(d, d, fmaf(b, b, fmaf(a, a, s))));
}
__device__ __forceinline__ double dist4(float4 y, float4 c, double s)
{
    const double a = (double)y.x - (double)c.x, b = (double)y.y - (double)c.y, d = (double)y.z - (double)c.z, e = (double)y.w - (double)c.w;
    return fma(e, e, fma(d, d, fma(b, b, fma(a, a, s))));
}

// The label of each quad's row among the candidates of its mask (none: `label` stands).  The whole warp calls it.
template <int NKS, int W>
__device__ __forceinline__ int settle_quads(const float4 (&y)[NKS], const uint32_t (&all)[W], const float *cs, int ld, int t, int label)
{
    constexpr int D = 16 * NKS;
    uint32_t m[W], any = 0;
#pragma unroll
    for (int i = 0; i < W; ++i) {
        m[i] = all[i];
        any |= all[i];
    }
    float f1 = CUDART_INF_F, f2 = CUDART_INF_F;
    int k1 = -1;
    for (;;) {
        const int k = pop_bit(m);
        if (!__any_sync(0xffffffffu, k >= 0)) break;
        const float *c = cs + (k < 0 ? 0 : k) * ld + 4 * t;
        float s = 0.f;
#pragma unroll
        for (int ks = 0; ks < NKS; ++ks) s = dist4(y[ks], *reinterpret_cast<const float4 *>(c + 16 * ks), s);
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        if (k >= 0) {
            if (s < f1) { f2 = f1; f1 = s; k1 = k; }
            else f2 = s < f2 || s != s ? s : f2;
        }
    }
    // (a lane adds D / 4 terms: the limit of sums eight times as long)
    const bool again = any && !(f2 > fp32_sum_limit(f1, 8 * D));
    if (__any_sync(0xffffffffu, again)) {
        double best = CUDART_INF;
        int kd = -1;
#pragma unroll
        for (int i = 0; i < W; ++i) m[i] = again ? all[i] : 0u;
        for (;;) {
            const int k = pop_bit(m);
            if (!__any_sync(0xffffffffu, k >= 0)) break;
            const float *c = cs + (k < 0 ? 0 : k) * ld + 4 * t;
            double s = 0.0;
#pragma unroll
            for (int ks = 0; ks < NKS; ++ks) s = dist4(y[ks], *reinterpret_cast<const float4 *>(c + 16 * ks), s);
            s += __shfl_xor_sync(0xffffffffu, s, 1);
            s += __shfl_xor_sync(0xffffffffu, s, 2);
            if (k >= 0 && s < best) {
                best = s;
                kd = k;
            }
        }
        if (again) k1 = kd;
    }
    return any ? (k1 < 0 ? 0 : k1) : label;   // (-1: every distance infinite or NaN)
}

template <bool BF16>
__device__ __forceinline__ void put4(void *out, size_t at, float4 y, float4 g, float4 b)
{
    const float4 v = make_float4(fmaf(g.x, y.x, b.x), fmaf(g.y, y.y, b.y), fmaf(g.z, y.z, b.z), fmaf(g.w, y.w, b.w));
    if (BF16) {
        const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
        __stcs(reinterpret_cast<uint2 *>(reinterpret_cast<__nv_bfloat16 *>(out) + at),
               make_uint2(*reinterpret_cast<const unsigned int *>(&lo), *reinterpret_cast<const unsigned int *>(&hi)));
    } else
        __stcs(reinterpret_cast<float4 *>(reinterpret_cast<float *>(out) + at), v);
}

__device__ __forceinline__ void copy_async16(float4 *dst, const float4 *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

// NKS: steps of sixteen columns; NC: chunks of 64 centroids; AHEAD: rows come through shared memory (where it has room).
template <int NKS, int NC, bool BF16, bool AHEAD>
__global__ void __launch_bounds__(short_threads(NKS), 1) apply_short_kernel(ShortParams p)
{
    pdl_enter();
    extern __shared__ __align__(128) unsigned char smem[];
    constexpr int D = 16 * NKS, LD = short_ld(D), TH = short_threads(NKS), NW = TH / 32, W = 2 * NC;
    __shared__ float s_max[3][NW];
    const int K = p.K, nt = p.nt;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
    float4 *ahead = reinterpret_cast<float4 *>(smem) + (size_t)warp * NKS * 64 + lane;   // [2 NKS][32] of this warp
    float *cs = reinterpret_cast<float *>(smem + (AHEAD ? (size_t)NW * NKS * 1024 : 0)), *gs = cs + K * LD, *bs = gs + K * LD;
    uint4 *bfrag = reinterpret_cast<uint4 *>(bs + K * LD);
    float *ak = reinterpret_cast<float *>(bfrag + (size_t)NKS * nt * 32), *coef = ak + nt * 16, *mean = coef + nt * 16;

    const int64_t groups = (p.N + 15) / 16;
    // (neighbouring groups on different SMs: a small call spreads over the device)
    const int64_t first = (int64_t)warp * gridDim.x + blockIdx.x, step = (int64_t)gridDim.x * NW;
    auto row_of = [&](int64_t row) { return reinterpret_cast<const float4 *>(p.Y + (size_t)(row < p.N ? row : 0) * D) + t; };
    auto request = [&](int64_t grp) {
        const float4 *pa = row_of(grp * 16 + g), *pb = row_of(grp * 16 + g + 8);
#pragma unroll
        for (int ks = 0; ks < NKS; ++ks) {
            copy_async16(ahead + (2 * ks) * 32, pa + 4 * ks);
            copy_async16(ahead + (2 * ks + 1) * 32, pb + 4 * ks);
        }
    };
    if (AHEAD && first < groups) request(first);

    // ---- centroids: copy, mean, fragments of c - m
    for (int e = tid; e < K * (D / 4); e += TH) {
        const int k = e / (D / 4), c = e - k * (D / 4);
        *reinterpret_cast<float4 *>(cs + k * LD + 4 * c) = __ldg(reinterpret_cast<const float4 *>(p.C) + e);
        *reinterpret_cast<float4 *>(gs + k * LD + 4 * c) = __ldg(reinterpret_cast<const float4 *>(p.gamma) + e);
        *reinterpret_cast<float4 *>(bs + k * LD + 4 * c) = __ldg(reinterpret_cast<const float4 *>(p.beta) + e);
    }
    __syncthreads();
    for (int j = tid; j < D; j += TH) {
        float s = 0.f;
        for (int k = 0; k < K; ++k) s += cs[k * LD + j];
        mean[j] = s / (float)K;
    }
    __syncthreads();
    const float slack = 1.0001f + (float)D * 6.0e-8f;   // covers the rounding of the running sums of squares
    {
        float cm = 0.f, am = 0.f, dm = 0.f;
        for (int k = warp; k < nt * 16; k += NW) {
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            double a = 0.0;
            if (k < K && lane < D / 4) {
                const float4 c = *reinterpret_cast<const float4 *>(cs + k * LD + 4 * lane), m = *reinterpret_cast<const float4 *>(mean + 4 * lane);
                v = make_float4(c.x - m.x, c.y - m.y, c.z - m.z, c.w - m.w);
                a = ((double)c.x - (double)m.x) * ((double)c.x + (double)m.x);
                a = fma((double)c.y - (double)m.y, (double)c.y + (double)m.y, a);
                a = fma((double)c.z - (double)m.z, (double)c.z + (double)m.z, a);
                a = fma((double)c.w - (double)m.w, (double)c.w + (double)m.w, a);
            }
            float mx = max4(v, 0.f), n2 = fmaf(v.x, v.x, fmaf(v.y, v.y, fmaf(v.z, v.z, v.w * v.w)));
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
                n2 += __shfl_xor_sync(0xffffffffu, n2, o);
                a += __shfl_xor_sync(0xffffffffu, a, o);
            }
            const int sh = half_shift(mx);
            const float sc = pow2i(sh);
            float left2 = 0.f;
            const uint32_t lo = round_pair(v.x * sc, v.y * sc, left2), hi = round_pair(v.z * sc, v.w * sc, left2);
            uint2 *dst = reinterpret_cast<uint2 *>(bfrag) + (((k >> 4) * 32 + (k & 7) * 4) * 2 + ((k >> 3) & 1));
            if (lane < D / 4) dst[((size_t)(lane >> 2) * nt * 32 + (lane & 3)) * 2] = make_uint2(lo, hi);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) left2 += __shfl_xor_sync(0xffffffffu, left2, o);
            if (lane == 0) {
                ak[k] = k < K ? (float)a : TC_KEY_INIT;
                coef[k] = -2.f * pow2i(-sh);
            }
            if (k < K) {   // (NaN stays out: a centroid that is not finite has scores that decide nothing)
                cm = fmaxf(cm, n2);
                am = fmaxf(am, fabsf((float)a));
                dm = fmaxf(dm, sqrtf(left2 * slack) * pow2i(-sh));
            }
        }
        if (lane == 0) {
            s_max[0][warp] = cm;
            s_max[1][warp] = am;
            s_max[2][warp] = dm;
        }
    }
    __syncthreads();
    float cmax2 = 0.f, amax = 0.f, dc = 0.f;
    for (int w = 0; w < NW; ++w) {
        cmax2 = fmaxf(cmax2, s_max[0][w]);
        amax = fmaxf(amax, s_max[1][w]);
        dc = fmaxf(dc, s_max[2][w]);
    }
    const float cnorm = sqrtf(cmax2 * slack);
    // e = 1.0625 * 2 (|dy| c + |y| e_y) + e_abs (c - m is rounded to fp32 before it is scaled: 2^-24 of c beside dc)
    // and 2^-16 of a score for the index in its low seven bits
    const float e_y = 1.001f * (dc + 5.9604645e-8f * cnorm) + ((float)(D + 2) * 2.3841858e-7f + 1.5258789e-5f) * cnorm;
    const float e_abs = (8.f * 5.9604645e-8f + 1.5258789e-5f) * amax + 1e-30f;   // (squares below that may have underflowed)

    int undecided = 0;
    for (int64_t grp = first; grp < groups; grp += step) {
        const int64_t ra = grp * 16 + g, rb = ra + 8;
        const bool ina = ra < p.N, inb = rb < p.N;
        float4 ya[NKS], yb[NKS];
        if constexpr (AHEAD) {
            asm volatile("cp.async.wait_all;" ::: "memory");
#pragma unroll
            for (int ks = 0; ks < NKS; ++ks) {
                ya[ks] = ahead[(2 * ks) * 32];
                yb[ks] = ahead[(2 * ks + 1) * 32];
            }
            if (grp + step < groups) request(grp + step);   // (this lane's pieces are in its registers)
        } else {
            const float4 *pa = row_of(ra), *pb = row_of(rb);
#pragma unroll
            for (int ks = 0; ks < NKS; ++ks) {
                ya[ks] = __ldcs(pa + 4 * ks);
                yb[ks] = __ldcs(pb + 4 * ks);
            }
        }
        float ma = 0.f, mb = 0.f, na = 0.f, nb = 0.f, la = 0.f, lb = 0.f;
#pragma unroll
        for (int ks = 0; ks < NKS; ++ks) {
            ma = max4(ya[ks], ma);
            mb = max4(yb[ks], mb);
            na = fmaf(ya[ks].x, ya[ks].x, fmaf(ya[ks].y, ya[ks].y, fmaf(ya[ks].z, ya[ks].z, fmaf(ya[ks].w, ya[ks].w, na))));
            nb = fmaf(yb[ks].x, yb[ks].x, fmaf(yb[ks].y, yb[ks].y, fmaf(yb[ks].z, yb[ks].z, fmaf(yb[ks].w, yb[ks].w, nb))));
        }
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            ma = fmaxf(ma, __shfl_xor_sync(0xffffffffu, ma, o));
            mb = fmaxf(mb, __shfl_xor_sync(0xffffffffu, mb, o));
        }
        const int sha = half_shift(ma), shb = half_shift(mb);
        const float sa = pow2i(sha), sb = pow2i(shb), ia = pow2i(-sha), ib = pow2i(-shb);
        uint4 fr[NKS];
#pragma unroll
        for (int ks = 0; ks < NKS; ++ks) {
            fr[ks].x = round_pair(ya[ks].x * sa, ya[ks].y * sa, la);
            fr[ks].y = round_pair(yb[ks].x * sb, yb[ks].y * sb, lb);
            fr[ks].z = round_pair(ya[ks].z * sa, ya[ks].w * sa, la);
            fr[ks].w = round_pair(yb[ks].z * sb, yb[ks].w * sb, lb);
        }
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            na += __shfl_xor_sync(0xffffffffu, na, o);
            nb += __shfl_xor_sync(0xffffffffu, nb, o);
            la += __shfl_xor_sync(0xffffffffu, la, o);
            lb += __shfl_xor_sync(0xffffffffu, lb, o);
        }
        // twice the bound on a score's error (NaN where the row is not finite)
        const float wa = 2.f * (1.0625f * 2.f * (sqrt_approx(la * slack) * ia * cnorm + sqrt_approx(na * slack) * e_y) + e_abs);
        const float wb = 2.f * (1.0625f * 2.f * (sqrt_approx(lb * slack) * ib * cnorm + sqrt_approx(nb * slack) * e_y) + e_abs);

        float acc[8][4];
        float a1 = TC_KEY_INIT, a2 = TC_KEY_INIT, c1 = TC_KEY_INIT, c2 = TC_KEY_INIT;   // smallest two keys of rows ra and rb
        auto contract = [&](int ch) {
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[i][q] = 0.f;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (ch * 4 + q >= nt) break;
#pragma unroll
                for (int ks = 0; ks < NKS; ++ks) {
                    const uint4 b = bfrag[(size_t)(ks * nt + ch * 4 + q) * 32 + lane];
                    mma_16816(acc[2 * q], fr[ks], b.x, b.y);
                    mma_16816(acc[2 * q + 1], fr[ks], b.z, b.w);
                }
            }
        };
        const f32x2 ia2 = pack2(ia, ia), ib2 = pack2(ib, ib);
#pragma unroll 1
        for (int ch = 0; ch < NC; ++ch) {
            contract(ch);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                if (ch * 4 + (i >> 1) >= nt) break;
                const int k = ch * 64 + i * 8 + 2 * t;
                const f32x2 n = *reinterpret_cast<const f32x2 *>(ak + k), f = *reinterpret_cast<const f32x2 *>(coef + k);
                const float2 ua = unpack2(fma2(f, mul2(pack2(acc[i][0], acc[i][1]), ia2), n));
                const float2 ub = unpack2(fma2(f, mul2(pack2(acc[i][2], acc[i][3]), ib2), n));
                take_key(ua.x, k, a1, a2);
                take_key(ua.y, k + 1, a1, a2);
                take_key(ub.x, k, c1, c2);
                take_key(ub.y, k + 1, c1, c2);
            }
        }
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            merge_keys(o, a1, a2);
            merge_keys(o, c1, c2);
        }
        int ka = (int)(__float_as_uint(a1) & 0x7Fu), kb = (int)(__float_as_uint(c1) & 0x7Fu);
        if (ka >= K) ka = 0;
        if (kb >= K) kb = 0;
        // (scores of a bound below 1e33 have not overflowed)
        const bool ua = ina && !(a2 - a1 > wa && wa < 2e33f), ub = inb && !(c2 - c1 > wb && wb < 2e33f);
        if (__any_sync(0xffffffffu, ua || ub)) {
            // all centroids within reach, one bit each
            undecided += __popc(__ballot_sync(0xffffffffu, ua && t == 0)) + __popc(__ballot_sync(0xffffffffu, ub && t == 0));
            uint32_t xa[W], xb[W];
            const float ta = wa < 2e33f ? a1 + wa : CUDART_INF_F, tb = wb < 2e33f ? c1 + wb : CUDART_INF_F;
#pragma unroll
            for (int i = 0; i < W; ++i) xa[i] = xb[i] = 0u;
#pragma unroll
            for (int ch = 0; ch < NC; ++ch) {
                if (NC > 1) contract(ch);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    if (ch * 4 + (i >> 1) >= nt) break;
                    const int k = ch * 64 + i * 8 + 2 * t, wd = 2 * ch + (i >> 2), at = (i & 3) * 8 + 2 * t;
                    const float2 n = *reinterpret_cast<const float2 *>(ak + k), f = *reinterpret_cast<const float2 *>(coef + k);
                    const uint32_t in0 = k < K ? 1u : 0u, in1 = k + 1 < K ? 2u : 0u;
                    xa[wd] |= ((fmaf(f.x, acc[i][0] * ia, n.x) > ta ? 0u : in0) | (fmaf(f.y, acc[i][1] * ia, n.y) > ta ? 0u : in1)) << at;
                    xb[wd] |= ((fmaf(f.x, acc[i][2] * ib, n.x) > tb ? 0u : in0) | (fmaf(f.y, acc[i][3] * ib, n.y) > tb ? 0u : in1)) << at;
                }
            }
#pragma unroll
            for (int i = 0; i < W; ++i) {
#pragma unroll
                for (int o = 1; o < 4; o <<= 1) {
                    xa[i] |= __shfl_xor_sync(0xffffffffu, xa[i], o);
                    xb[i] |= __shfl_xor_sync(0xffffffffu, xb[i], o);
                }
                if (!ua) xa[i] = 0u;
                if (!ub) xb[i] = 0u;
            }
            if (__any_sync(0xffffffffu, ua)) ka = settle_quads<NKS, W>(ya, xa, cs, LD, t, ka);
            if (__any_sync(0xffffffffu, ub)) kb = settle_quads<NKS, W>(yb, xb, cs, LD, t, kb);
        }
        if (ina) {
            const float *ga = gs + ka * LD + 4 * t, *ba = bs + ka * LD + 4 * t;
#pragma unroll
            for (int ks = 0; ks < NKS; ++ks)
                put4<BF16>(p.out, (size_t)ra * D + 16 * ks + 4 * t, ya[ks], *reinterpret_cast<const float4 *>(ga + 16 * ks),
                           *reinterpret_cast<const float4 *>(ba + 16 * ks));
            if (t == 0) p.labels[ra] = ka;
        }
        if (inb) {
            const float *gb = gs + kb * LD + 4 * t, *bb = bs + kb * LD + 4 * t;
#pragma unroll
            for (int ks = 0; ks < NKS; ++ks)
                put4<BF16>(p.out, (size_t)rb * D + 16 * ks + 4 * t, yb[ks], *reinterpret_cast<const float4 *>(gb + 16 * ks),
                           *reinterpret_cast<const float4 *>(bb + 16 * ks));
            if (t == 0) p.labels[rb] = kb;
        }
    }
    if (lane == 0 && undecided) {
        atomicAdd(reinterpret_cast<unsigned long long *>(&p.ctl->refined_last), (unsigned long long)undecided);
        atomicAdd(reinterpret_cast<unsigned long long *>(&p.ctl->refined_total), (unsigned long long)undecided);
    }
}

template <int NKS, int NC, bool BF16, bool AHEAD>
cudaError_t launch_short(const ShortParams &p, cudaStream_t s)
{
    auto kern = apply_short_kernel<NKS, NC, BF16, AHEAD>;
    // (the same value whatever the shape: several threads may be launching)
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SH_SMEM);
    if (e != cudaSuccess) return e;
    const int64_t groups = (p.N + 15) / 16;
    const int64_t grid = groups < tc_sm_count() ? groups : tc_sm_count();
    e = launch_pdl(kern, dim3((unsigned)grid), dim3(short_threads(NKS)), short_smem(16 * NKS, p.K, AHEAD), s, p);
    count_launch();
    return e;
}
template <int NKS, bool BF16>
cudaError_t launch_short_nks(const ShortParams &p, cudaStream_t s)
{
    const bool ahead = short_smem(16 * NKS, p.K, true) <= SH_SMEM;
    if (p.nt > 4) return ahead ? launch_short<NKS, 2, BF16, true>(p, s) : launch_short<NKS, 2, BF16, false>(p, s);
    return ahead ? launch_short<NKS, 1, BF16, true>(p, s) : launch_short<NKS, 1, BF16, false>(p, s);
}
template <bool BF16>
cudaError_t launch_short_d(int D, const ShortParams &p, cudaStream_t s)
{
    switch (D / 16) {
    case 2: return launch_short_nks<2, BF16>(p, s);
    case 3: return launch_short_nks<3, BF16>(p, s);
    case 4: return launch_short_nks<4, BF16>(p, s);
    case 5: return launch_short_nks<5, BF16>(p, s);
    case 6: return launch_short_nks<6, BF16>(p, s);
    case 7: return launch_short_nks<7, BF16>(p, s);
    default: return launch_short_nks<8, BF16>(p, s);
    }
}

}  // namespace

bool apply_short_supported(int64_t N, int D, int K)
{
    return N >= 1 && K >= 2 && K <= 128 && D >= 32 && D <= 128 && D % 16 == 0 && short_smem(D, K, false) <= SH_SMEM;
}

cudaError_t launch_apply_short(const float *Y, int64_t N, int D, int K, const float *C, const float *gamma, const float *beta, void *out,
                               bool out_bf16, int32_t *labels, Control *ctl, cudaStream_t s)
{
    if (!apply_short_supported(N, D, K)) return cudaErrorInvalidValue;
    const int nt = (K + 15) / 16;
    const ShortParams p{Y, C, gamma, beta, out, labels, ctl, N, K, nt};
    return out_bf16 ? launch_short_d<true>(D, p, s) : launch_short_d<false>(D, p, s);
}

}  // namespace cat
