// The Lloyd rounds of a fit in one cooperative launch for many rows of few columns (Algorithm 1 step 2 with K-Means).
//
// Every CTA keeps its rows in shared memory for the whole fit, as fp16 operand fragments of mma.sync, so that a round
// reads nothing but the rows that are undecided or have moved; a warp takes sixteen rows from scores to labels by itself.
// tcgen05 is not used: its accumulators would have to pass from one warp role to the next, and these hand-overs
// were what bounded such rounds (csrc/cat_small.cu: 50 us a round on 200 704 x 64, K = 64), while the contraction is
// small (3 us of mma.sync there).  A round:
//
//   centroids   fp16 fragments of c - m, their norms and rounding errors (m: a point among the rows)
//   score       t_k = ||c_k - m||^2 - 2 (y - m).(c_k - m), the two smallest of each row, certainty test with the measured
//               rounding errors; a row that fails it goes to its warp's queue with all centroids within reach
//   settle      four queued rows at a time, eight lanes each: direct-form fp32 sums of squares from the rows and centroids
//               themselves, and fp64 where these are within their own error of one another, lowest index on equality
//   move        rows whose label changed, in row order, enter and leave the CTA's fp64 sums per cluster; a thread
//               owns a column of some clusters, so nothing is added in a varying order
//   barrier, the CTAs' sums added up in CTA order, barrier
//
//   bound, 200 704 x 64, K = 64 (cycles a round): scores 21 000 (issue), moves 23 000 on average (latency of the moved rows, more in the
//   first rounds), barriers 12 000, combination 7 000, centroids 5 000, settlement 2 500.  25 rounds take 1030 us, 1390 in the
//   persistent kernel.  Moves by groups of lanes with four columns each: 1090 (the scores' registers spill).
//
// A round in which no label changes leaves everything as it is, and so would all behind it: the rounds end there.  Sums
// that follow moves keep what a far larger row rounded off after it has left; where the largest row's exponent is more than
// X_SPREAD above the rows' average every round adds up all rows afresh (and none ends early).
#include "cat_half.cuh"

namespace cat {

namespace {

constexpr int XT = 512;
constexpr int XW = XT / 32;
constexpr int X_QUEUE = 16;           // undecided rows a warp holds
constexpr int X_SPREAD = 16;          // (2^16 of the 2^53 that fp64 resolves)
constexpr int X_PART_PAD = 48;        // doubles between the CTAs' planes of sums (no power-of-two stride)
constexpr size_t X_SMEM = 227 * 1024 - 1024;
constexpr uint32_t X_NONE = 0xFFu;    // no label yet

struct TilesLayout {
    uint32_t b, plane, cn, coef, list, queue, dcnt, dirty, meta, shift, lab, fresh, total;
};

// groups: sixteen rows each; nk: 16-column steps; nt: 16-centroid tiles
TilesLayout tiles_layout(int64_t groups, int nk, int nt, int D, int K)
{
    TilesLayout L{};
    size_t o = (size_t)groups * nk * 512;
    auto take = [&](size_t bytes) {
        o = (o + 15) & ~(size_t)15;
        const size_t at = o;
        o += bytes;
        return (uint32_t)(at < 0x7fffffff ? at : 0x7fffffff);
    };
    const int words = nt > 4 ? 4 : 2;   // of a candidate mask
    L.b = take((size_t)nk * nt * 512);
    L.plane = take((size_t)K * D * 8);
    L.cn = take((size_t)nt * 16 * 4);
    L.coef = take((size_t)nt * 16 * 4);
    L.list = take((size_t)XT * 4);
    L.queue = take((size_t)XW * X_QUEUE * (1 + words) * 4);
    L.dcnt = take((size_t)K * 4);
    L.dirty = take((size_t)K);
    L.meta = take((size_t)groups * 16 * 4);
    L.shift = take((size_t)groups * 16);
    L.lab = take((size_t)groups * 16);
    L.fresh = take((size_t)groups * 16);
    L.total = o < 0x7fffffff ? (uint32_t)o : 0x7fffffffu;
    return L;
}

struct TilesParams {
    const float *Y;
    float *C;                // [K, D] in: start, out: final centroids
    const float *mean;       // [D] what operands are taken relative to
    int32_t *labels;         // [N] out
    double *part;            // [G][K D + X_PART_PAD] the CTAs' sums
    int32_t *size;           // [K] cluster sizes; then rows moved in even and odd passes, and of the rows' largest magnitudes
                             // the sum of exponents, the number above zero, the largest exponent; all zero at launch
    double *sums;            // [K, D] out
    int64_t *counts;         // [K] out
    Control *ctl;
    int64_t N;
    int D, K, passes;
    int rpc;                 // rows per CTA, a multiple of 16
    int nk, nt;
    TilesLayout L;
};

// upper half of a float that is not below x >= 0
__device__ __forceinline__ uint32_t ceil_bf16(float x) { return x < CUDART_INF_F ? (__float_as_uint(x) + 0xFFFFu) >> 16 : 0x7F80u; }

// columns j ... j + 3 of a row of D (zero beyond); CG: past L1, for what other CTAs write during the launch
template <bool VEC, bool CG>
__device__ __forceinline__ float4 load4(const float *row, int j, int D)
{
    if constexpr (VEC) {
        if (j >= D) return make_float4(0.f, 0.f, 0.f, 0.f);
        return CG ? __ldcg(reinterpret_cast<const float4 *>(row + j)) : __ldg(reinterpret_cast<const float4 *>(row + j));
    } else {
        float v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = j + q < D ? (CG ? __ldcg(row + j + q) : __ldg(row + j + q)) : 0.f;
        return make_float4(v[0], v[1], v[2], v[3]);
    }
}
__device__ __forceinline__ float4 sub4(float4 a, float4 b) { return make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w); }
__device__ __forceinline__ float sq4(float4 a, float s) { return fmaf(a.x, a.x, fmaf(a.y, a.y, fmaf(a.z, a.z, fmaf(a.w, a.w, s)))); }
__device__ __forceinline__ double sq4(float4 y, float4 c, double s)
{
    const double a = (double)y.x - (double)c.x, b = (double)y.y - (double)c.y, d = (double)y.z - (double)c.z, e = (double)y.w - (double)c.w;
    return fma(e, e, fma(d, d, fma(b, b, fma(a, a, s))));
}

// Labels of n <= 4 queued rows, eight lanes a row.
template <bool VEC, int W>
__device__ __noinline__ void settle_four(const float *Y, const float *C, int D, const uint32_t *queue, int n, int64_t row0, unsigned char *fresh,
                                         int lane)
{
    const int e = lane >> 3, sub = lane & 7;
    const bool live = e < n;
    const uint32_t *q = queue + (live ? e : 0) * (1 + W);
    const int r = (int)q[0];
    const float *y = Y + (size_t)(row0 + r) * D;
    uint32_t all[W], m[W];
#pragma unroll
    for (int i = 0; i < W; ++i) m[i] = all[i] = live ? q[1 + i] : 0u;
    float f1 = CUDART_INF_F, f2 = CUDART_INF_F;
    int k1 = -1;
    for (;;) {
        const int ka = pop_bit(m), kb = pop_bit(m);
        if (!__any_sync(0xffffffffu, ka >= 0)) break;
        const float *ca = C + (size_t)(ka < 0 ? 0 : ka) * D, *cb = C + (size_t)(kb < 0 ? (ka < 0 ? 0 : ka) : kb) * D;
        float sa = 0.f, sb = 0.f;
#pragma unroll 2
        for (int j = sub * 4; j < D; j += 32) {
            const float4 yv = load4<VEC, false>(y, j, D), av = load4<VEC, true>(ca, j, D), bv = load4<VEC, true>(cb, j, D);
            sa = sq4(sub4(yv, av), sa);
            sb = sq4(sub4(yv, bv), sb);
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
            sa += __shfl_xor_sync(0xffffffffu, sa, o);
            sb += __shfl_xor_sync(0xffffffffu, sb, o);
        }
        if (ka >= 0) {
            if (sa < f1) { f2 = f1; f1 = sa; k1 = ka; }
            else f2 = sa < f2 || sa != sa ? sa : f2;
        }
        if (kb >= 0) {
            if (sb < f1) { f2 = f1; f1 = sb; k1 = kb; }
            else f2 = sb < f2 || sb != sb ? sb : f2;
        }
    }
    // (a lane adds D / 8 terms: the limit of sums four times as long)
    const bool again = live && !(f2 > fp32_sum_limit(f1, 4 * D));
    if (__any_sync(0xffffffffu, again)) {
        double best = CUDART_INF;
        int kd = -1;
#pragma unroll
        for (int i = 0; i < W; ++i) m[i] = again ? all[i] : 0u;
        for (;;) {
            const int k = pop_bit(m);
            if (!__any_sync(0xffffffffu, k >= 0)) break;
            const float *c = C + (size_t)(k < 0 ? 0 : k) * D;
            double s = 0.0;
            for (int j = sub * 4; j < D; j += 32) s = sq4(load4<VEC, false>(y, j, D), load4<VEC, true>(c, j, D), s);
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (k >= 0 && s < best) {
                best = s;
                kd = k;
            }
        }
        if (again) k1 = kd;
    }
    if (live && sub == 0) fresh[r] = (unsigned char)(k1 < 0 ? 0 : k1);   // (-1: every distance infinite or NaN)
}

// NC: chunks of 64 centroids; NV: float4 units of a row per lane, 128 columns each.
template <bool VEC, int NC, int NV>
__global__ void __launch_bounds__(XT, 1) fit_tiles_kernel(TilesParams p)
{
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ int s_warp[XW], s_ex[3];
    __shared__ float s_cmax2, s_dc;
    constexpr int W = 2 * NC;   // words of a candidate mask
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
    const int D = p.D, K = p.K, G = gridDim.x, nk = p.nk, nt = p.nt, KD = K * D;
    const TilesLayout &L = p.L;
    uint4 *frag = reinterpret_cast<uint4 *>(smem);
    uint4 *bfrag = reinterpret_cast<uint4 *>(smem + L.b);
    double *plane = reinterpret_cast<double *>(smem + L.plane);
    float *cn = reinterpret_cast<float *>(smem + L.cn), *coef = reinterpret_cast<float *>(smem + L.coef);
    uint32_t *list = reinterpret_cast<uint32_t *>(smem + L.list);
    static_assert(NC == 1 || NC == 2, "the layout has two or four words a mask");
    uint32_t *queue = reinterpret_cast<uint32_t *>(smem + L.queue) + warp * X_QUEUE * (1 + W);
    int *dcnt = reinterpret_cast<int *>(smem + L.dcnt);
    unsigned char *dirty = smem + L.dirty;
    uint32_t *meta = reinterpret_cast<uint32_t *>(smem + L.meta);   // norm of y - m, and of its rounding error, as bf16 not below them
    signed char *shift = reinterpret_cast<signed char *>(smem + L.shift);
    unsigned char *lab = smem + L.lab, *fresh = smem + L.fresh;
    const int64_t row0 = (int64_t)blockIdx.x * p.rpc;
    const int nrows = (int)(p.N - row0 < p.rpc ? p.N - row0 : p.rpc), groups = (nrows + 15) / 16;
    int32_t *moved = p.size + K, *spread = moved + 2;
    const float slack = 1.0001f + (float)D * 6.0e-8f;   // covers the rounding of the running sums of squares

    // ---- rows to fragments: lane (g, t) has columns 4 t ... 4 t + 3 of a step, of rows g and g + 8
    if (tid < 3) s_ex[tid] = 0;
    for (int e = tid; e < KD; e += XT) plane[e] = 0.0;
    for (int k = tid; k < K; k += XT) {
        dcnt[k] = 0;
        dirty[k] = 1;   // (the first pass leaves every cluster's sums)
    }
    __syncthreads();
    {
        int esum = 0, enum_ = 0, emax = 0;
        for (int grp = warp; grp < groups; grp += XW) {
            const int ra = grp * 16 + g, rb = ra + 8;
            const float *ya = p.Y + (size_t)(row0 + (ra < nrows ? ra : 0)) * D, *yb = p.Y + (size_t)(row0 + (rb < nrows ? rb : 0)) * D;
            float ma = 0.f, mb = 0.f, wa = 0.f, wb = 0.f;
#pragma unroll 4
            for (int ks = 0; ks < nk; ++ks) {
                const int j = ks * 16 + 4 * t;
                const float4 m = load4<VEC, false>(p.mean, j, D), a = load4<VEC, false>(ya, j, D), b = load4<VEC, false>(yb, j, D);
                ma = max4(sub4(a, m), ma);
                mb = max4(sub4(b, m), mb);
                wa = max4(a, wa);
                wb = max4(b, wb);
            }
#pragma unroll
            for (int o = 1; o < 4; o <<= 1) {
                ma = fmaxf(ma, __shfl_xor_sync(0xffffffffu, ma, o));
                mb = fmaxf(mb, __shfl_xor_sync(0xffffffffu, mb, o));
                wa = fmaxf(wa, __shfl_xor_sync(0xffffffffu, wa, o));
                wb = fmaxf(wb, __shfl_xor_sync(0xffffffffu, wb, o));
            }
            const int sha = half_shift(ma), shb = half_shift(mb);
            const float sa = pow2i(sha), sb = pow2i(shb);
            float na = 0.f, nb = 0.f, la = 0.f, lb = 0.f;
#pragma unroll 4
            for (int ks = 0; ks < nk; ++ks) {
                const int j = ks * 16 + 4 * t;
                const float4 m = load4<VEC, false>(p.mean, j, D);
                float4 a = sub4(load4<VEC, false>(ya, j, D), m), b = sub4(load4<VEC, false>(yb, j, D), m);
                if (ra >= nrows) a = make_float4(0.f, 0.f, 0.f, 0.f);
                if (rb >= nrows) b = make_float4(0.f, 0.f, 0.f, 0.f);
                na = sq4(a, na);
                nb = sq4(b, nb);
                uint4 f;
                f.x = round_pair(a.x * sa, a.y * sa, la);
                f.y = round_pair(b.x * sb, b.y * sb, lb);
                f.z = round_pair(a.z * sa, a.w * sa, la);
                f.w = round_pair(b.z * sb, b.w * sb, lb);
                frag[(size_t)(grp * nk + ks) * 32 + lane] = f;
            }
#pragma unroll
            for (int o = 1; o < 4; o <<= 1) {
                na += __shfl_xor_sync(0xffffffffu, na, o);
                nb += __shfl_xor_sync(0xffffffffu, nb, o);
                la += __shfl_xor_sync(0xffffffffu, la, o);
                lb += __shfl_xor_sync(0xffffffffu, lb, o);
            }
            if (t == 0) {
                // (NaN becomes infinity: such a row decides nothing by its scores)
                meta[ra] = ceil_bf16(sqrtf(na * slack)) << 16 | ceil_bf16(sqrtf(la * slack) * pow2i(-sha));
                meta[rb] = ceil_bf16(sqrtf(nb * slack)) << 16 | ceil_bf16(sqrtf(lb * slack) * pow2i(-shb));
                shift[ra] = (signed char)sha;
                shift[rb] = (signed char)shb;
                lab[ra] = lab[rb] = (unsigned char)X_NONE;
                const int ea = ra < nrows ? (int)(__float_as_uint(wa) >> 23) : 0, eb = rb < nrows ? (int)(__float_as_uint(wb) >> 23) : 0;
                esum += ea + eb;
                enum_ += (ea > 0) + (eb > 0);
                emax = max(emax, max(ea, eb));
            }
        }
        esum = __reduce_add_sync(0xffffffffu, esum);
        enum_ = __reduce_add_sync(0xffffffffu, enum_);
        emax = __reduce_max_sync(0xffffffffu, emax);
        if (lane == 0) {
            atomicAdd(&s_ex[0], esum);
            atomicAdd(&s_ex[1], enum_);
            atomicMax(&s_ex[2], emax);
        }
    }
    __syncthreads();
    if (tid == 0) {
        atomicAdd(spread, s_ex[0]);
        atomicAdd(spread + 1, s_ex[1]);
        atomicMax(spread + 2, s_ex[2]);
    }

    // this thread's column and clusters in the update: a warp has one set of clusters
    const int Dp = (D + 31) & ~31;
    int ng = 1;
    while (2 * ng * Dp <= XT) ng *= 2;
    const int ucol = tid % Dp, ugrp = tid / Dp;
    const bool uactive = ugrp < ng;   // (of whole warps)

    uint32_t bar = 0;
    bool afresh = false, alive = true;
    // The sums follow the list: a warp picks the entries of its clusters out of it, 32 at a time, into its queue and fetches
    // sixteen rows together.  (Where all rows are added afresh only what enters counts.)
    auto follow = [&](int n) {
        int held = 0;
        for (int e0 = 0; e0 < n || held > 0;) {
            while (e0 < n && held < 16) {
                const uint32_t en = e0 + lane < n ? list[e0 + lane] : 0u;
                const int ln = (int)(en >> 16 & 0xFFu), lo = (int)(en >> 24);
                const bool hit = e0 + lane < n && ((ln & (ng - 1)) == ugrp || (lo != (int)X_NONE && !afresh && (lo & (ng - 1)) == ugrp));
                const uint32_t m = __ballot_sync(0xffffffffu, hit);
                if (hit) queue[held + __popc(m & ((1u << lane) - 1u))] = en;
                held += __popc(m);
                e0 += 32;
            }
            __syncwarp();
            const int nb = held < 16 ? held : 16;
            float y[16];
#pragma unroll
            for (int u = 0; u < 16; ++u) y[u] = u < nb && ucol < D ? __ldg(p.Y + (size_t)(row0 + (queue[u] & 0xFFFFu)) * D + ucol) : 0.f;
#pragma unroll
            for (int u = 0; u < 16; ++u) {
                if (u >= nb) break;
                const uint32_t en = queue[u];
                const int ln = (int)(en >> 16 & 0xFFu), lo = (int)(en >> 24);
                if ((ln & (ng - 1)) == ugrp && ucol < D) plane[ln * D + ucol] += (double)y[u];
                if (lo != (int)X_NONE && !afresh && (lo & (ng - 1)) == ugrp && ucol < D) plane[lo * D + ucol] -= (double)y[u];
            }
            const uint32_t rest = 16 + lane < held ? queue[16 + lane] : 0u;   // (31 at most)
            __syncwarp();
            held = held > 16 ? held - 16 : 0;
            if (lane < held) queue[lane] = rest;
            __syncwarp();
        }
    };
    long long refined = 0;
    int refined_pass = 0;
    for (int pass = 0; pass < p.passes; ++pass) {
        // ---- centroids: four at a time a warp, all their loads in flight
        for (int k0 = warp * 4; k0 < nt * 16; k0 += XW * 4) {
            float4 v[4][NV];
            float mx[4], left[4], n2[4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int u = 0; u < NV; ++u)
                    v[i][u] = k0 + i < K ? load4<VEC, true>(p.C + (size_t)(k0 + i) * D, 4 * (lane + 32 * u), D) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                mx[i] = left[i] = 0.f;
                n2[i] = 0.f;
#pragma unroll
                for (int u = 0; u < NV; ++u) {
                    if (k0 + i < K) v[i][u] = sub4(v[i][u], load4<VEC, false>(p.mean, 4 * (lane + 32 * u), D));
                    const float4 c = v[i][u];
                    mx[i] = max4(c, mx[i]);
                    n2[i] = sq4(c, n2[i]);
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    mx[i] = fmaxf(mx[i], __shfl_xor_sync(0xffffffffu, mx[i], o));
                    n2[i] += __shfl_xor_sync(0xffffffffu, n2[i], o);
                }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int k = k0 + i, sh = half_shift(mx[i]);
                const float sc = pow2i(sh);
                uint2 *dst = reinterpret_cast<uint2 *>(bfrag) + (((k >> 4) * 32 + (k & 7) * 4) * 2 + ((k >> 3) & 1));
#pragma unroll
                for (int u = 0; u < NV; ++u) {
                    const int c4 = lane + 32 * u;
                    const float4 c = v[i][u];
                    const uint32_t lo = round_pair(c.x * sc, c.y * sc, left[i]), hi = round_pair(c.z * sc, c.w * sc, left[i]);
                    if (c4 < nk * 4) dst[((size_t)(c4 >> 2) * nt * 32 + (c4 & 3)) * 2] = make_uint2(lo, hi);
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) left[i] += __shfl_xor_sync(0xffffffffu, left[i], o);
                if (lane == 0) {
                    cn[k] = k < K ? n2[i] : TC_KEY_INIT;
                    coef[k] = -2.f * pow2i(-sh);
                    // (the rounding errors' norms pass through the candidates' list, which is not in use yet)
                    if (k < K) reinterpret_cast<float *>(list)[k] = sqrtf(left[i] * slack) * pow2i(-sh);
                }
            }
        }
        __syncthreads();
        if (warp == 0) {
            float m = 0.f, d = 0.f;
            for (int k = lane; k < K; k += 32) {
                // (NaN stays out: a centroid that is not finite has scores that decide nothing)
                m = fmaxf(m, cn[k]);
                d = fmaxf(d, reinterpret_cast<float *>(list)[k]);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
                d = fmaxf(d, __shfl_xor_sync(0xffffffffu, d, o));
            }
            if (lane == 0) {
                s_cmax2 = m;
                s_dc = d;
            }
        }
        __syncthreads();
        const float cnorm = sqrtf(s_cmax2) * 1.0001f;
        // e = 1.0625 * 2 (|dy| c + |y| e_y) + e_abs: fp16 operands' measured errors, y - m and c - m rounded to fp32, D additions
        // and 2^-16 of a score for the index in its low seven bits
        const float e_y = 1.001f * (s_dc + 2.f * 5.9604645e-8f * cnorm) + ((float)(16 * nk + 2) * 2.3841858e-7f + 1.5258789e-5f) * cnorm;
        const float e_abs = (24.f * 5.9604645e-8f + 1.5258789e-5f) * s_cmax2 + 1e-30f;   // (squares below that may have underflowed)

        // ---- labels of this warp's groups
        refined_pass = 0;
        int held = 0;   // queued rows
        for (int grp = warp; grp < groups; grp += XW) {
            const uint4 *fa = frag + (size_t)grp * nk * 32 + lane;
            const int ra = grp * 16 + g, rb = ra + 8;
            const float ia = pow2i(-(int)shift[ra]), ib = pow2i(-(int)shift[rb]);
            float acc[8][4];
            float a1 = TC_KEY_INIT, a2 = TC_KEY_INIT, c1 = TC_KEY_INIT, c2 = TC_KEY_INIT;   // smallest two keys of rows ra and rb
            auto contract = [&](int ch) {
#pragma unroll
                for (int i = 0; i < 8; ++i)
#pragma unroll
                    for (int q = 0; q < 4; ++q) acc[i][q] = 0.f;
                for (int ks = 0; ks < nk; ++ks) {
                    const uint4 a = fa[ks * 32];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        if (ch * 4 + q >= nt) break;
                        const uint4 b = bfrag[(size_t)(ks * nt + ch * 4 + q) * 32 + lane];
                        mma_16816(acc[2 * q], a, b.x, b.y);
                        mma_16816(acc[2 * q + 1], a, b.z, b.w);
                    }
                }
            };
            const f32x2 ia2 = pack2(ia, ia), ib2 = pack2(ib, ib);
#pragma unroll 1
            for (int ch = 0; ch < NC; ++ch) {
                if (ch * 4 >= nt) break;
                contract(ch);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    if (ch * 4 + (i >> 1) >= nt) break;
                    const int k = ch * 64 + i * 8 + 2 * t;
                    const f32x2 n = *reinterpret_cast<const f32x2 *>(cn + k), f = *reinterpret_cast<const f32x2 *>(coef + k);
                    const float2 sa = unpack2(fma2(f, mul2(pack2(acc[i][0], acc[i][1]), ia2), n));
                    const float2 sb = unpack2(fma2(f, mul2(pack2(acc[i][2], acc[i][3]), ib2), n));
                    take_key(sa.x, k, a1, a2);
                    take_key(sa.y, k + 1, a1, a2);
                    take_key(sb.x, k, c1, c2);
                    take_key(sb.y, k + 1, c1, c2);
                }
            }
#pragma unroll
            for (int o = 1; o < 4; o <<= 1) {
                merge_keys(o, a1, a2);
                merge_keys(o, c1, c2);
            }
            const int ka = (int)(__float_as_uint(a1) & 0x7Fu) < K ? (int)(__float_as_uint(a1) & 0x7Fu) : 0;
            const int kb = (int)(__float_as_uint(c1) & 0x7Fu) < K ? (int)(__float_as_uint(c1) & 0x7Fu) : 0;
            const uint32_t mta = meta[ra], mtb = meta[rb];
            auto bound = [&](uint32_t mt) {
                return 1.0625f * 2.f * (__uint_as_float(mt << 16) * cnorm + __uint_as_float(mt & 0xFFFF0000u) * e_y) + e_abs;
            };
            const float la = 2.f * bound(mta), lb = 2.f * bound(mtb);
            // (scores of a bound below 1e33 have not overflowed)
            const bool ua = ra < nrows && !(a2 - a1 > la && la < 2e33f), ub = rb < nrows && !(c2 - c1 > lb && lb < 2e33f);
            if (t == 0) {
                fresh[ra] = (unsigned char)ka;
                fresh[rb] = (unsigned char)kb;
            }
            const uint32_t oa = __ballot_sync(0xffffffffu, ua && t == 0), ob = __ballot_sync(0xffffffffu, ub && t == 0);
            const int more = __popc(oa) + __popc(ob);
            if (more == 0) continue;
            refined_pass += more;
            // all centroids within reach, one bit each
            uint32_t xa[W], xb[W];
            const float ta = la < 2e33f ? a1 + la : CUDART_INF_F, tb = lb < 2e33f ? c1 + lb : CUDART_INF_F;
#pragma unroll
            for (int i = 0; i < W; ++i) xa[i] = xb[i] = 0u;
#pragma unroll
            for (int ch = 0; ch < NC; ++ch) {
                if (ch * 4 >= nt) break;
                if (NC > 1) contract(ch);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    if (ch * 4 + (i >> 1) >= nt) break;
                    const int k = ch * 64 + i * 8 + 2 * t, wd = 2 * ch + (i >> 2), at = (i & 3) * 8 + 2 * t;
                    const float2 n = *reinterpret_cast<const float2 *>(cn + k), f = *reinterpret_cast<const float2 *>(coef + k);
                    const uint32_t in0 = k < K ? 1u : 0u, in1 = k + 1 < K ? 2u : 0u;
                    xa[wd] |= ((fmaf(f.x, acc[i][0] * ia, n.x) > ta ? 0u : in0) | (fmaf(f.y, acc[i][1] * ia, n.y) > ta ? 0u : in1)) << at;
                    xb[wd] |= ((fmaf(f.x, acc[i][2] * ib, n.x) > tb ? 0u : in0) | (fmaf(f.y, acc[i][3] * ib, n.y) > tb ? 0u : in1)) << at;
                }
            }
#pragma unroll
            for (int i = 0; i < W; ++i)
#pragma unroll
                for (int o = 1; o < 4; o <<= 1) {
                    xa[i] |= __shfl_xor_sync(0xffffffffu, xa[i], o);
                    xb[i] |= __shfl_xor_sync(0xffffffffu, xb[i], o);
                }
            if (held + more > X_QUEUE) {
                __syncwarp();
                for (int q = 0; q < held; q += 4)
                    settle_four<VEC, W>(p.Y, p.C, D, queue + q * (1 + W), held - q < 4 ? held - q : 4, row0, fresh, lane);
                __syncwarp();
                held = 0;
            }
            const uint32_t before = (1u << lane) - 1u;
            if (ua && t == 0) {
                uint32_t *q = queue + (held + __popc(oa & before)) * (1 + W);
                q[0] = (uint32_t)ra;
#pragma unroll
                for (int i = 0; i < W; ++i) q[1 + i] = xa[i];
            }
            if (ub && t == 0) {
                uint32_t *q = queue + (held + __popc(oa) + __popc(ob & before)) * (1 + W);
                q[0] = (uint32_t)rb;
#pragma unroll
                for (int i = 0; i < W; ++i) q[1 + i] = xb[i];
            }
            held += more;
        }
        __syncwarp();
        for (int q = 0; q < held; q += 4)
            settle_four<VEC, W>(p.Y, p.C, D, queue + q * (1 + W), held - q < 4 ? held - q : 4, row0, fresh, lane);
        if (lane == 0) refined += refined_pass;
        if (afresh) {
            for (int e = tid; e < KD; e += XT) plane[e] = 0.0;
            for (int k = tid; k < K; k += XT) {
                dirty[k] = 1;
                dcnt[k] = 0;
            }
        }
        __syncthreads();

        // ---- moves: rows whose label changed, in row order; the sums follow when the list is full, and at the end
        int total = 0, listed = 0;
        for (int base = 0; base < nrows; base += XT) {
            const int r = base + tid;
            const uint32_t l = r < nrows ? fresh[r] : 0u, was = r < nrows ? lab[r] : 0u;
            const bool mv = r < nrows && (afresh || l != was);
            const uint32_t m = __ballot_sync(0xffffffffu, mv);
            if (lane == 0) s_warp[warp] = __popc(m);
            __syncthreads();   // (the sums have followed the list before, too)
            int first = 0, n = 0;
#pragma unroll
            for (int w = 0; w < XW; ++w) {
                const int c = s_warp[w];
                if (w < warp) first += c;
                n += c;
            }
            if (listed + n > XT) {   // (the same in every thread)
                if (uactive) follow(listed);
                listed = 0;
                __syncthreads();
            }
            if (mv) {
                list[listed + first + __popc(m & ((1u << lane) - 1u))] = (uint32_t)r | l << 16 | was << 24;
                lab[r] = (unsigned char)l;
                // (sizes are integers: any order will do)
                atomicAdd(dcnt + l, 1);
                dirty[l] = 1;
                if (was != X_NONE && !afresh) {
                    atomicSub(dcnt + was, 1);
                    dirty[was] = 1;
                }
            }
            listed += n;
            total += n;
            __syncthreads();
        }
        if (uactive && listed) follow(listed);
        __syncthreads();
        for (int e = tid; e < KD; e += XT)
            if (dirty[e / D]) __stcg(p.part + (size_t)blockIdx.x * (KD + X_PART_PAD) + e, plane[e]);
        __syncthreads();
        for (int k = tid; k < K; k += XT) {
            if (dcnt[k]) atomicAdd(p.size + k, dcnt[k]);
            dcnt[k] = 0;
            dirty[k] = 0;
        }
        if (tid == 0 && total) atomicAdd(moved + (pass & 1), total);
        if (!grid_barrier(&p.ctl->grid_bar, ++bar, p.ctl)) { alive = false; break; }
        if (__ldcg(moved + (pass & 1)) == 0) {   // nothing moved: nothing would from here on, and every assignment left would settle these rows
            if (lane == 0) refined += (long long)refined_pass * (p.passes - 1 - pass);
            break;
        }
        // (the first pass has added all rows in either case; the same decision in every CTA)
        afresh = (__ldcg(spread + 2) - X_SPREAD) * (long long)__ldcg(spread + 1) > (long long)__ldcg(spread);

        // ---- the CTAs' sums, in CTA order: a warp per four neighbouring entries, lane (g8, c) takes entry c of CTAs
        // g8, g8 + 8, ..., and a fixed tree adds the eight parts
        const bool last = pass + 1 == p.passes;
        static_assert(SMALL_MAX_GRID <= 8 * 20, "a lane holds at most twenty CTAs' parts");
        for (int e4 = warp * G + (int)blockIdx.x; 4 * e4 < KD; e4 += G * XW) {
            const int e = 4 * e4 + (lane & 3);
            double v[20];
#pragma unroll
            for (int q = 0; q < 20; ++q) {
                const int c = (lane >> 2) + 8 * q;
                v[q] = c < G && e < KD ? __ldcg(p.part + (size_t)c * (KD + X_PART_PAD) + e) : 0.0;
            }
            const int k = e < KD ? e / D : 0;
            const long long n = __ldcg(p.size + k);
            double s = v[0];
#pragma unroll
            for (int q = 1; q < 20; ++q)
                if ((lane >> 2) + 8 * q < G) s += v[q];
#pragma unroll
            for (int o = 4; o < 32; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane < 4 && e < KD) {
                p.sums[e] = s;
                if (e == k * D) p.counts[k] = n;
                if (!last && n > 0) __stcg(p.C + e, (float)(s / (double)n));
            }
        }
        // the other count of moves is the next pass's: nobody adds to it before the barrier below
        if (blockIdx.x == 0 && tid == 0) moved[(pass & 1) ^ 1] = 0;
        if (last) break;
        if (!grid_barrier(&p.ctl->grid_bar, ++bar, p.ctl)) { alive = false; break; }
        if (afresh && blockIdx.x == 0) {
            // sizes are counted anew too (all have read the old ones before the barrier above)
            for (int k = tid; k < K; k += XT) p.size[k] = 0;
        }
        if (afresh && !grid_barrier(&p.ctl->grid_bar, ++bar, p.ctl)) { alive = false; break; }
    }
    if (!alive) return;
    __syncthreads();
    for (int r = tid; r < nrows; r += XT) p.labels[row0 + r] = (int32_t)lab[r];
    if (lane == 0 && refined) atomicAdd(reinterpret_cast<unsigned long long *>(&p.ctl->refined_total), (unsigned long long)refined);
    if (lane == 0 && refined_pass) atomicAdd(reinterpret_cast<unsigned long long *>(&p.ctl->refined_last), (unsigned long long)refined_pass);
}

struct TilesPlan {
    int grid, rpc, nk, nt;
    TilesLayout L;
};

bool tiles_shape(int D, int K) { return D >= 4 && D <= 256 && K >= 2 && K <= 128 && K * D <= 8192; }

bool tiles_plan(int64_t N, int D, int K, TilesPlan *pl)
{
    if (!tiles_shape(D, K) || N < K || N > ((int64_t)1 << 23)) return false;
    int grid = tc_sm_count();
    if (grid > SMALL_MAX_GRID) grid = SMALL_MAX_GRID;
    const int64_t g16 = (N + 15) / 16;
    const int64_t per = (g16 + grid - 1) / grid;   // groups per CTA
    pl->rpc = (int)(per * 16);
    pl->grid = (int)((g16 + per - 1) / per);
    pl->nk = (D + 15) / 16;
    pl->nt = (K + 15) / 16;
    pl->nt = pl->nt <= 4 ? pl->nt : 8;
    pl->L = tiles_layout(per, pl->nk, pl->nt, D, K);
    return pl->rpc <= 65520 && pl->L.total <= X_SMEM;
}

template <bool VEC, int NC, int NV>
cudaError_t launch_tiles(const TilesPlan &pl, const TilesParams &p, cudaStream_t s)
{
    auto kern = fit_tiles_kernel<VEC, NC, NV>;
    // (the same value whatever the shape: several threads may be launching)
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)X_SMEM);
    if (e != cudaSuccess) return e;
    void *args[] = {(void *)&p};
    e = cudaLaunchCooperativeKernel((const void *)kern, dim3((unsigned)pl.grid), dim3(XT), args, pl.L.total, s);
    count_launch();
    return e;
}

}  // namespace

bool fit_tiles_supported(int64_t N, int D, int K)
{
    TilesPlan pl;
    return tiles_plan(N, D, K, &pl);
}
size_t fit_tiles_part_doubles(int D, int K) { return tiles_shape(D, K) ? (size_t)SMALL_MAX_GRID * ((size_t)K * D + X_PART_PAD) : 0; }
size_t fit_tiles_counts(int K) { return (size_t)K + 5; }

cudaError_t launch_fit_tiles(const float *Y, int64_t N, int D, int K, float *C, const float *mean, int passes, int32_t *labels, double *part,
                             int32_t *part_counts, double *sums, int64_t *counts, Control *ctl, cudaStream_t s)
{
    TilesPlan pl;
    if (!tiles_plan(N, D, K, &pl) || passes < 1) return cudaErrorInvalidValue;
    const cudaError_t e = cudaMemsetAsync(part_counts, 0, fit_tiles_counts(K) * sizeof(int32_t), s);
    if (e != cudaSuccess) return e;
    TilesParams p{Y, C, mean, labels, part, part_counts, sums, counts, ctl, N, D, K, passes, pl.rpc, pl.nk, pl.nt, pl.L};
    const bool vec = D % 4 == 0;
    const int form = (pl.nt > 4 ? 2 : 0) + (D > 128 ? 1 : 0);
    switch (form) {
    case 0: return vec ? launch_tiles<true, 1, 1>(pl, p, s) : launch_tiles<false, 1, 1>(pl, p, s);
    case 1: return vec ? launch_tiles<true, 1, 2>(pl, p, s) : launch_tiles<false, 1, 2>(pl, p, s);
    case 2: return vec ? launch_tiles<true, 2, 1>(pl, p, s) : launch_tiles<false, 2, 1>(pl, p, s);
    default: return cudaErrorInvalidValue;   // (128 columns and more than 64 centroids are beyond K D = 8192)
    }
}

}  // namespace cat
