// The Lloyd rounds of a fit in one cooperative launch, for calibration sets whose rows fit into the SMs'
// shared memory (Algorithm 1 step 2 with K-Means; any row length).
//
// The general path takes seven launches a round, 38 us for 1024 rows of 1000 columns of which the
// arithmetic needs less than one.  Here every CTA keeps its rows in shared memory for the whole fit, and a
// round is two grid barriers:
//
//   assign    distances of the CTA's rows to all centroids (staged in chunks), direct form in fp32: a sum of
//             squares, so its relative error is at most (D / 32 + 12) 2^-24 (a lane adds D / 32 terms, then a
//             tree).  Centroids within that error of the smallest distance are settled in fp64, lowest
//             index on equality.  Rows whose label changed go to a list, in row order.
//   barrier
//   update    a team of warps owns eight columns of a range of clusters: their fp64 sums live in shared memory
//             and follow the list -- each warp takes its part of it, four rows at a time into four partial
//             sums, added up in a fixed order (results do not vary from run to run) -- then the team writes its
//             part of the new centroids
//   barrier
//
// A round in which no label changes leaves the centroids as they are, bit for bit, and so do all that would
// follow: the rounds end there.  The last pass assigns against the final centroids and leaves them alone;
// its sums and sizes feed the closed form.
//
// Sums that follow a list keep what the addition of a row rounded off after that row has left.  That is harmless as long
// as no row is far larger than the others; where the largest row's exponent is more than F_SPREAD above the rows'
// average, every round adds up all rows afresh instead (and none ends early).
//   bound: latency (barriers, staging the centroids, the list's row fetches) for small sets -- 1024 x 1000,
//   K = 16: 7 us a round --, staging and fp32 issue for the largest that are taken (4096 x 1000, K = 32: 36 us).
#include "cat_tc.cuh"

namespace cat {

namespace {

constexpr int FT = 512;
constexpr int FW = FT / 32;
constexpr int F_LIST = 2048;          // list entries staged at a time
constexpr int F_QUEUE = 64;           // hits a warp holds before it fetches their rows
constexpr int F_MAX_GRID = 160;
constexpr int F_SPREAD = 16;          // (2^16 of the 2^53 that fp64 resolves)
constexpr size_t F_SMEM = 225 * 1024;

struct FitRowsParams {
    const float *Y;
    float *C;                // [K, D] in: start, out: final centroids
    float *Cp;               // [K][ldy] scratch: the same in rows of ldy, for the bulk copies
    int32_t *labels;         // [N] out
    double *sums;            // [K, D] out
    int64_t *counts;         // [K] out
    uint2 *list;             // [G][rpc] {row, new label | old label << 16}
    int4 *list_count;        // [G] {entries; first pass, of the rows' largest magnitudes: sum of exponents, number above zero, largest exponent}
    Control *ctl;
    int64_t N;
    int D, K, passes;
    int ldy;                 // row stride in shared memory (floats, multiple of 4, zero beyond D)
    int rpc;                 // rows per CTA
    int chunk;               // centroids staged at a time (multiple of 4)
    int span;                // clusters per team of the update
    int tu;                  // warps per team
    int parts;               // partial sums per warp: 4 (8-lane groups side by side), or 1 where they would not fit
    uint32_t o_c, o_dist, o_sum, o_cnt, o_part, o_pcnt, o_list, o_queue, o_lab, o_pref;   // shared memory (rows first)
};

__device__ __forceinline__ double exact_distance(const float *y, const float *c, int D, int lane)
{
    double s = 0.0;
#pragma unroll 4
    for (int j = lane; j < D; j += 32) {
        const double d = (double)y[j] - (double)__ldcg(c + j);
        s = fma(d, d, s);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

// one list entry's value into the sums of the clusters [k0, k1) that its row entered and left
__device__ __forceinline__ void add_entry(uint32_t w, float v, int k0, int k1, int c, double *sums, int *counts)
{
    const int ln = (int)(w & 0xFFFFu), lo = (int)(w >> 16);
    if (ln >= k0 && ln < k1) {
        sums[(ln - k0) * 8] += (double)v;
        if (c == 0) ++counts[ln - k0];
    }
    if (lo >= k0 && lo < k1) {
        sums[(lo - k0) * 8] -= (double)v;
        if (c == 0) --counts[lo - k0];
    }
}

__global__ void __launch_bounds__(FT, 1) fit_rows_kernel(FitRowsParams p)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_total, s_fail, s_afresh;
    __shared__ int3 s_exp[FW];
    __shared__ __align__(8) uint64_t s_bar;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int D = p.D, K = p.K, G = gridDim.x;
    float *ys = reinterpret_cast<float *>(smem);
    float *cs = reinterpret_cast<float *>(smem + p.o_c);
    float *dist = reinterpret_cast<float *>(smem + p.o_dist);
    const int team = warp / p.tu, tw = warp % p.tu;
    double *sum = reinterpret_cast<double *>(smem + p.o_sum) + (size_t)team * p.span * 8;        // the team's sums
    int *cnt = reinterpret_cast<int *>(smem + p.o_cnt) + team * p.span;
    double *part = reinterpret_cast<double *>(smem + p.o_part) + (size_t)warp * p.parts * p.span * 8;   // this round's, [parts][span][8]
    int *pcnt = reinterpret_cast<int *>(smem + p.o_pcnt) + warp * p.parts * p.span;
    uint2 *list = reinterpret_cast<uint2 *>(smem + p.o_list);
    uint2 *queue = reinterpret_cast<uint2 *>(smem + p.o_queue) + warp * F_QUEUE;
    int *lab = reinterpret_cast<int *>(smem + p.o_lab), *prev = lab + p.rpc;
    int *pref = reinterpret_cast<int *>(smem + p.o_pref);   // [G + 1]
    const int64_t row0 = (int64_t)blockIdx.x * p.rpc;
    const int nrows = (int)(p.N - row0 < p.rpc ? p.N - row0 : p.rpc);

    // this team's part of the update: columns [col0, col0 + 8) of clusters [k0, k1)
    const int units = (K + p.span - 1) / p.span, u = team * G + (int)blockIdx.x;
    const int col0 = u / units * 8, k0 = u % units * p.span, k1 = k0 + p.span < K ? k0 + p.span : K;
    const bool owner = col0 < D;

    // rows, zero-padded to whole groups of four rows and columns
    const int n4 = (nrows + 3) & ~3, ld4 = p.ldy >> 2;
    int3 ex = make_int3(0, 0, 0);
    for (int r = warp; r < n4; r += FW) {
        float m = 0.f;
        for (int j = lane; j < p.ldy; j += 32) {
            const float v = r < nrows && j < D ? __ldg(p.Y + (size_t)(row0 + r) * D + j) : 0.f;
            ys[(size_t)r * p.ldy + j] = v;
            m = fmaxf(m, fabsf(v));
        }
        const uint32_t bits = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
        if (bits) ex = make_int3(ex.x + (int)(bits >> 23), ex.y + 1, max(ex.z, (int)(bits >> 23)));
    }
    if (lane == 0) s_exp[warp] = ex;
    for (int r = tid; r < p.rpc; r += FT) prev[r] = -1;
    if (tw == 0) {
        for (int e = lane; e < p.span * 8; e += 32) sum[e] = 0.0;
        for (int e = lane; e < p.span; e += 32) cnt[e] = 0;
    }
    if (tid == 0) {
        mbar_init(smem_u32(&s_bar), 1);
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async;" ::: "memory");
    }
    uint32_t copies = 0;

    int refined = 0, refined_pass = 0;
    uint32_t bar = 0;
    bool afresh = false;
    for (int pass = 0; pass < p.passes; ++pass) {
        // ---- distances to all centroids, a chunk of them at a time
        for (int c0 = 0; c0 < K; c0 += p.chunk) {
            const int nc = K - c0 < p.chunk ? K - c0 : p.chunk, nc4 = (nc + 3) & ~3;
            __syncthreads();
            if (pass == 0) {
                for (int r = warp; r < nc4; r += FW)
#pragma unroll 8
                    for (int j = lane; j < p.ldy; j += 32)
                        cs[(size_t)r * p.ldy + j] = r < nc && j < D ? __ldcg(p.C + (size_t)(c0 + r) * D + j) : 0.f;
                __syncthreads();
            } else {
                if (tid == 0) {
                    // (the other CTAs' stores, seen through the grid barrier, and this copy use different proxies)
                    asm volatile("fence.proxy.async;" ::: "memory");
                    const uint32_t bytes = (uint32_t)nc * p.ldy * 4, dst = smem_u32(cs), b = smem_u32(&s_bar);
                    const unsigned char *src = reinterpret_cast<const unsigned char *>(p.Cp + (size_t)c0 * p.ldy);
                    mbar_arrive_expect_tx(b, bytes);
                    for (uint32_t o = 0; o < bytes; o += 8192) {
                        const uint32_t n = bytes - o < 8192 ? bytes - o : 8192;
                        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst + o),
                                     "l"(src + o), "r"(n), "r"(b)
                                     : "memory");
                    }
                }
                if (!mbar_wait(smem_u32(&s_bar), copies & 1u, &s_fail, p.ctl)) s_fail = 1;
                ++copies;
                if (__syncthreads_or(*(volatile int *)&s_fail)) return;
            }
            const int tiles_c = nc4 >> 2, tiles = (n4 >> 2) * tiles_c;
            for (int tile = warp; tile < tiles; tile += FW) {
                const int r = tile / tiles_c * 4, c = tile % tiles_c * 4;
                const float4 *y4 = reinterpret_cast<const float4 *>(ys + (size_t)r * p.ldy);
                const float4 *c4 = reinterpret_cast<const float4 *>(cs + (size_t)c * p.ldy);
                float acc[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) acc[i] = 0.f;
                for (int j = lane; j < ld4; j += 32) {
                    float4 yv[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) yv[i] = y4[i * ld4 + j];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float4 cv = c4[q * ld4 + j];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            float a = acc[i * 4 + q], d;
                            d = yv[i].x - cv.x; a = fmaf(d, d, a);
                            d = yv[i].y - cv.y; a = fmaf(d, d, a);
                            d = yv[i].z - cv.z; a = fmaf(d, d, a);
                            d = yv[i].w - cv.w; a = fmaf(d, d, a);
                            acc[i * 4 + q] = a;
                        }
                    }
                }
                const float s = warp_sum16(acc, lane);
                const int i = lane >> 3, q = (lane >> 1) & 3;
                if ((lane & 1) == 0 && r + i < nrows && c + q < nc) dist[(size_t)(r + i) * K + c0 + c + q] = s;
            }
        }
        __syncthreads();
        // ---- labels
        refined_pass = 0;
        for (int r = warp; r < nrows; r += FW) {
            const float *d = dist + (size_t)r * K;
            float best = CUDART_INF_F;
            for (int k = lane; k < K; k += 32) best = fminf(best, d[k]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) best = fminf(best, __shfl_xor_sync(0xffffffffu, best, o));
            const float lim = fp32_sum_limit(best, D);
            int n = 0, l = -1;
            for (int b = 0; b < K; b += 32) {
                const uint32_t m = __ballot_sync(0xffffffffu, b + lane < K && !(d[b + lane < K ? b + lane : 0] > lim));
                if (m && l < 0) l = b + __ffs(m) - 1;
                n += __popc(m);
            }
            if (n != 1) {
                ++refined_pass;
                double b64 = CUDART_INF;
                if (l < 0) l = 0;   // (NaN distances only)
                for (int b = 0; b < K; b += 32)
                    for (uint32_t m = __ballot_sync(0xffffffffu, b + lane < K && !(d[b + lane < K ? b + lane : 0] > lim)); m; m &= m - 1) {
                        const int k = b + __ffs(m) - 1;
                        const double e = exact_distance(ys + (size_t)r * p.ldy, p.C + (size_t)k * D, D, lane);
                        if (e < b64) {
                            b64 = e;
                            l = k;
                        }
                    }
            }
            if (lane == 0) lab[r] = l;
        }
        refined += refined_pass;
        __syncthreads();
        // ---- rows that changed (or all of them), in row order
        if (warp == 0) {
            int n = 0;
            for (int b = 0; b < nrows; b += 32) {
                const int r = b + lane;
                const int l = r < nrows ? lab[r] : 0, o = r < nrows ? prev[r] : 0;
                const bool moved = r < nrows && (afresh || l != o);
                const uint32_t m = __ballot_sync(0xffffffffu, moved);
                if (moved) {
                    p.list[(size_t)row0 + n + __popc(m & ((1u << lane) - 1u))] =
                        make_uint2((uint32_t)(row0 + r), (uint32_t)l | ((uint32_t)(o < 0 || afresh ? 0xFFFF : o) << 16));
                    prev[r] = l;
                }
                n += __popc(m);
            }
            if (lane == 0) {
                int4 w = make_int4(n, 0, 0, 0);
                for (int q = 0; pass == 0 && q < FW; ++q) {
                    w.y += s_exp[q].x;
                    w.z += s_exp[q].y;
                    w.w = max(w.w, s_exp[q].z);
                }
                p.list_count[blockIdx.x] = w;
            }
        }
        if (!grid_barrier(&p.ctl->grid_bar, ++bar, p.ctl)) return;
        if (warp == 0) {
            int run = 0, esum = 0, rows = 0, emax = 0;
            for (int b = 0; b < G; b += 32) {
                const int4 w = b + lane < G ? __ldcg(p.list_count + b + lane) : make_int4(0, 0, 0, 0);
                const int v = w.x;
                esum += w.y;
                rows += w.z;
                emax = max(emax, w.w);
                int incl = v;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int t = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += t;
                }
                if (b + lane < G) pref[b + lane] = run + incl - v;
                run += __shfl_sync(0xffffffffu, incl, 31);
            }
            if (lane == 0) {
                pref[G] = run;
                s_total = run;
            }
            if (pass == 0) {
                esum = __reduce_add_sync(0xffffffffu, esum);
                rows = __reduce_add_sync(0xffffffffu, rows);
                emax = __reduce_max_sync(0xffffffffu, emax);
                if (lane == 0) s_afresh = (emax - F_SPREAD) * rows > esum;
            }
        }
        __syncthreads();
        const int M = s_total;
        const bool last = pass + 1 == p.passes;
        if (M == 0) break;   // nothing moved: nothing would from here on
        // (the first list has all rows in either case; the same decision in every CTA)
        const bool carried = !afresh;
        afresh = s_afresh != 0;

        // ---- the sums follow the list
        if (owner) {
            for (int e = lane; e < p.parts * p.span * 8; e += 32) part[e] = 0.0;
            for (int e = lane; e < p.parts * p.span; e += 32) pcnt[e] = 0;
        }
        for (int b = 0; b < M; b += F_LIST) {
            const int nb = M - b < F_LIST ? M - b : F_LIST;
            __syncthreads();
            for (int c = warp; c < G; c += FW) {
                const int a0 = pref[c], a1 = pref[c + 1];
                for (int e = (a0 > b ? a0 : b) + lane; e < a1 && e < b + nb; e += 32)
                    list[e - b] = __ldcg(p.list + (size_t)c * p.rpc + (e - a0));
            }
            __syncthreads();
            if (!owner) continue;
            const int g = lane >> 3, c = lane & 7;
            const bool col = col0 + c < D;
            const int share = (nb / 32 + p.tu) / p.tu * 32;          // this warp's part of the block
            const int e1 = (tw + 1) * share < nb ? (tw + 1) * share : nb;
            int held = 0;
            for (int e0 = tw * share; e0 < e1;) {
                // fill the queue with entries that touch this team's clusters
                while (e0 < e1 && held + 32 <= F_QUEUE) {
                    const uint2 en = e0 + lane < e1 ? list[e0 + lane] : make_uint2(0u, 0xFFFFFFFFu);
                    const int ln = (int)(en.y & 0xFFFFu), lo = (int)(en.y >> 16);
                    const bool hit = e0 + lane < e1 && ((ln >= k0 && ln < k1) || (lo >= k0 && lo < k1));
                    const uint32_t m = __ballot_sync(0xffffffffu, hit);
                    if (hit) queue[held + __popc(m & ((1u << lane) - 1u))] = en;
                    held += __popc(m);
                    e0 += 32;
                }
                __syncwarp();
                // their rows, sixteen in flight, then the additions
                for (int h0 = 0; h0 < held; h0 += 16) {
                    float v[4];
                    uint32_t w[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int h = h0 + 4 * i + g;
                        w[i] = h < held ? queue[h].y : 0xFFFFFFFFu;
                        v[i] = h < held && col ? __ldg(p.Y + (size_t)queue[h].x * D + col0 + c) : 0.f;
                    }
                    if (p.parts == 4) {
                        double *mine = part + (size_t)g * p.span * 8 + c;
                        int *minc = pcnt + g * p.span;
#pragma unroll
                        for (int i = 0; i < 4; ++i) add_entry(w[i], v[i], k0, k1, c, mine, minc);
                    } else {
#pragma unroll
                        for (int i = 0; i < 4; ++i)
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                if (g == q) add_entry(w[i], v[i], k0, k1, c, part + c, pcnt);
                                __syncwarp();
                            }
                    }
                }
                held = 0;
                __syncwarp();
            }
        }
        __syncthreads();
        if (owner && tw == 0) {
            for (int e = lane; e < (k1 - k0) * 8; e += 32) {
                double a = carried ? sum[e] : 0.0;
                for (int w = 0; w < p.tu; ++w) {
                    const double *q = part + (size_t)w * p.parts * p.span * 8 + e;
                    const int st = p.span * 8;
                    a += p.parts == 4 ? (q[0] + q[st]) + (q[2 * st] + q[3 * st]) : q[0];
                }
                sum[e] = a;
            }
            for (int e = lane; e < k1 - k0; e += 32) {
                int n = carried ? cnt[e] : 0;
                for (int w = 0; w < p.tu * p.parts; ++w) n += pcnt[w * p.span + e];
                cnt[e] = n;
            }
            __syncwarp();
        }
        if (last) break;
        if (owner && tw == 0) {
            for (int e = lane; e < (k1 - k0) * 8; e += 32) {
                const int k = e >> 3, j = col0 + (e & 7), n = cnt[k];
                const size_t o = (size_t)(k0 + k) * D + j;
                if (j < D) {
                    // (an empty cluster keeps its centroid)
                    const float v = n > 0 ? (float)(sum[e] / (double)n) : __ldcg(p.C + o);
                    p.C[o] = v;
                    p.Cp[(size_t)(k0 + k) * p.ldy + j] = v;
                } else if (j < p.ldy)
                    p.Cp[(size_t)(k0 + k) * p.ldy + j] = 0.f;
            }
            asm volatile("fence.proxy.async;" ::: "memory");
        }
        if (!grid_barrier(&p.ctl->grid_bar, ++bar, p.ctl)) return;
    }
    for (int r = tid; r < nrows; r += FT) p.labels[row0 + r] = lab[r];
    if (owner && tw == 0)
        for (int e = lane; e < (k1 - k0) * 8; e += 32) {
            const int k = e >> 3, j = col0 + (e & 7);
            if (j < D) p.sums[(size_t)(k0 + k) * D + j] = sum[e];
            if (j == 0) p.counts[k0 + k] = cnt[k];
        }
    if (lane == 0 && refined) atomicAdd(reinterpret_cast<unsigned long long *>(&p.ctl->refined_total), (unsigned long long)refined);
    if (lane == 0 && refined_pass) atomicAdd(reinterpret_cast<unsigned long long *>(&p.ctl->refined_last), (unsigned long long)refined_pass);
}

// Geometry; false where the kernel does not go.
bool fit_rows_plan(int64_t N, int D, int K, FitRowsParams *p, int *grid, size_t *smem)
{
    // The distances cost N K D / (148 SMs * 64 per clock), short rows as much as 256 columns; the lists and the
    // update a latency per changed row.  25 rounds against the general rounds: 1024 x 1000, K = 16 0.24 ms and 0.96,
    // 4096 x 1000, K = 64 1.15 and 1.76, 8192 x 50, K = 32 0.57 and 0.82, 3000 x 300, K = 256 0.57 and 2.0; past the lines
    // drawn here 7000 x 400, K = 90 1.47 and 1.40, 8000 x 16, K = 256 1.50 and 0.88, 20 000 x 50, K = 64 1.25 and 1.19.
    // From 256 columns on the line comes down with the rows a CTA holds (logits, whose labels change in every round; well
    // separated clusters reach their fixed point early and gain throughout): up to 32 rows 4500 x 768, K = 48 1.01 and 1.08;
    // up to 48 6144 x 256, K = 96 0.86 and 0.88, past it K = 128 1.09 and 0.89; above 8192 x 256, K = 32 0.80 and 0.86, past it
    // K = 64 1.08 and 0.93.
    if (D < 4 || K < 2 || K > CAT_MAX_K || N < K || N > 8192) return false;
    const int shift = D < 256 ? N > 6144 : (N > 148 * 48 ? 2 : N > 148 * 32);
    if (N * (int64_t)K * (D < 256 ? 256 : D) > ((int64_t)1 << 28) >> shift) return false;
    const int sms = 148;
    int64_t rpc = (N + sms - 1) / sms;
    if (rpc < 4) rpc = 4;
    rpc = (rpc + 3) & ~(int64_t)3;
    const int G = (int)((N + rpc - 1) / rpc);
    if (G > F_MAX_GRID) return false;
    p->ldy = (D + 3) & ~3;
    p->rpc = (int)rpc;
    // teams of the update: as few clusters each as there are warps for, then several warps each
    const int64_t slices = (D + 7) / 8, warps = (int64_t)G * FW;
    int span = 1, tu = 1;
    while (span < K && slices * ((K + span - 1) / span) > warps) ++span;
    if (slices * ((K + span - 1) / span) > warps) return false;
    while (tu < FW && slices * ((K + span - 1) / span) * (2 * tu) <= warps) tu *= 2;
    p->span = span;
    p->tu = tu;
    p->parts = span <= 8 ? 4 : 1;
    size_t o = (size_t)rpc * p->ldy * 4;
    const size_t fixed = (size_t)rpc * K * 4 + (size_t)(FW / tu) * span * (64 + 4) + (size_t)FW * p->parts * span * (64 + 4) +
                         (size_t)F_LIST * 8 + (size_t)FW * F_QUEUE * 8 + (size_t)rpc * 8 + (F_MAX_GRID + 1) * 4 + 256;
    if (o + fixed + (size_t)4 * p->ldy * 4 > F_SMEM) return false;
    int64_t chunk = (int64_t)((F_SMEM - o - fixed) / ((size_t)p->ldy * 4)) & ~(int64_t)3;
    const int k4 = (K + 3) & ~3;
    if (chunk > k4) chunk = k4;
    p->chunk = (int)chunk;
    auto place = [&](size_t bytes) {
        const size_t at = align_up(o, 16);
        o = at + bytes;
        return (uint32_t)at;
    };
    p->o_c = place((size_t)chunk * p->ldy * 4);
    p->o_sum = place((size_t)(FW / tu) * span * 64);
    p->o_part = place((size_t)FW * p->parts * span * 64);
    p->o_list = place((size_t)F_LIST * 8);
    p->o_queue = place((size_t)FW * F_QUEUE * 8);
    p->o_dist = place((size_t)rpc * K * 4);
    p->o_cnt = place((size_t)(FW / tu) * span * 4);
    p->o_pcnt = place((size_t)FW * p->parts * span * 4);
    p->o_lab = place((size_t)rpc * 8);
    p->o_pref = place((F_MAX_GRID + 1) * 4);
    *grid = G;
    *smem = o;
    return o <= F_SMEM;
}

}  // namespace

bool fit_rows_supported(int64_t N, int D, int K)
{
    FitRowsParams p{};
    int grid;
    size_t smem;
    return fit_rows_plan(N, D, K, &p, &grid, &smem) && grid <= tc_sm_count();   // (all CTAs resident)
}

cudaError_t launch_fit_rows(const float *Y, int64_t N, int D, int K, float *C, int passes, int32_t *labels, double *sums,
                            int64_t *counts, void *list, void *list_count, float *padded, Control *ctl, cudaStream_t s)
{
    FitRowsParams p{};
    int grid;
    size_t smem;
    if (!fit_rows_plan(N, D, K, &p, &grid, &smem) || grid > tc_sm_count()) return cudaErrorInvalidValue;
    p.Y = Y;
    p.C = C;
    p.Cp = padded;
    p.labels = labels;
    p.sums = sums;
    p.counts = counts;
    p.list = reinterpret_cast<uint2 *>(list);
    p.list_count = reinterpret_cast<int4 *>(list_count);
    p.ctl = ctl;
    p.N = N;
    p.D = D;
    p.K = K;
    p.passes = passes;
    // (the same value whatever the shape: several threads may be launching)
    cudaError_t e = cudaFuncSetAttribute(fit_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)F_SMEM);
    if (e != cudaSuccess) return e;
    void *args[] = {&p};
    e = cudaLaunchCooperativeKernel((const void *)fit_rows_kernel, dim3((unsigned)grid), dim3(FT), args, smem, s);
    count_launch();
    return e;
}

}  // namespace cat
