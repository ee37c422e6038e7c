// Segmented (per-cluster) sums through a stable sort of the rows by label.
//
//   label_hist_kernel     per-block key histograms (1024 entries per block)
//   label_scan_blocks_kernel  per-block offsets and key totals
//                         (key offsets, segment table and cluster sizes: scan_keys, inside the scatter kernel)
//   label_scatter_kernel  stable scatter of the row indices: order[] lists the rows of
//                         key 0 in ascending row order, then key 1, ...
//
// Two modes.  Full: every row is an entry with key = its label (K keys).  Delta (the Lloyd
// rounds of cat_fit): only rows whose label differs from the previous round's are entries,
// each twice -- under key `new label` (its values enter that cluster's sum) and under key
// K + `old label` (they leave that one) -- so 2K keys over 2N virtual entries, nearly all of
// them empty once the clustering settles.  The running sums S_k += sum(in) - sum(out) are the
// same per-cluster sums up to fp64 rounding, at the cost of the rows that moved.
//   segment_sums_kernel   one CTA per segment (<= seg_rows consecutive entries of order[], all of
//                         one cluster): streams those rows with 128-bit loads and keeps the
//                         column sums in fp64 registers -- no atomics, no shared accumulators,
//                         fixed summation order -- and writes one partial row per segment
//   segment_combine_kernel  adds a cluster's segment partials in order; optionally turns the
//                         sums into centroids
//
// Three reductions use the same machinery: column sums of one matrix (a Lloyd round), of
// two matrices (the final pass: sums of Yq and Yfp), and the centred second moments
// sum (q - muQ)^2, sum (q - muQ)(f - muF) with the cluster means held in registers.
#include "cat_internal.cuh"

#include <cuda_fp16.h>

namespace cat {

namespace {

constexpr int SORT_BLOCK = 1024;     // rows per histogram / scatter block
constexpr int SEG_THREADS = 256;
constexpr int COMB_THREADS = 512;

// Key of virtual entry e: entries [0, N) are the rows under their current label; in delta
// mode (prev != NULL) a row whose label did not change has no entry, and entries [N, 2N)
// are the changed rows under K + previous label.  -1 = no entry.
__device__ __forceinline__ int entry_key(const int32_t *__restrict__ cur, const int32_t *__restrict__ prev,
                                         int64_t N, int K, int64_t e)
{
    if (e < N) {
        const int l = cur[e], was = prev ? prev[e] : -1;   // (both on their way together)
        if (l < 0 || l >= K) return -1;
        if (prev && was == l) return -1;
        return l;
    }
    if (!prev || e >= 2 * N) return -1;
    const int64_t r = e - N;
    const int o = prev[r], now = cur[r];
    if (o < 0 || o >= K || o == now) return -1;
    return K + o;
}

__global__ void __launch_bounds__(SORT_BLOCK) label_hist_kernel(const int32_t *__restrict__ cur,
                                                                 const int32_t *__restrict__ prev, int64_t N, int K,
                                                                 int KK, uint32_t *__restrict__ blk_hist,
                                                                 const int32_t *settled)
{
    extern __shared__ uint32_t hist[];   // [KK]
    for (int k = threadIdx.x; k < KK; k += SORT_BLOCK) hist[k] = 0;
    pdl_enter();
    const int over = settled ? *settled : 0;
    const int64_t e = (int64_t)blockIdx.x * SORT_BLOCK + threadIdx.x;
    const int l = entry_key(cur, prev, N, K, e);
    if (over) return;
    __syncthreads();
    if (l >= 0) atomicAdd(&hist[l], 1u);
    __syncthreads();
    for (int k = threadIdx.x; k < KK; k += SORT_BLOCK) blk_hist[(size_t)k * gridDim.x + blockIdx.x] = hist[k];   // [key][block]
}

// One warp per key: blk_hist[k][b] becomes the number of entries of key k in blocks before
// b, key_total[k] their total.
__global__ void __launch_bounds__(256) label_scan_blocks_kernel(uint32_t *__restrict__ blk_hist, int nblk, int KK,
                                                                 uint32_t *__restrict__ key_total, const int32_t *settled)
{
    pdl_enter();
    const int over = settled ? *settled : 0;
    const int k = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (k >= KK) return;
    uint32_t carry = 0, next = lane < nblk ? blk_hist[(size_t)k * nblk + lane] : 0u;
    if (over) return;
    for (int b0 = 0; b0 < nblk; b0 += 32) {
        const int b = b0 + lane;
        const uint32_t v = next;
        next = b + 32 < nblk ? blk_hist[(size_t)k * nblk + b + 32] : 0u;
        uint32_t incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (b < nblk) blk_hist[(size_t)k * nblk + b] = carry + incl - v;
        carry += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (lane == 0) key_total[k] = carry;
}

// Exclusive scan over the 1024 threads of the CTA (one value per thread); returns the exclusive
// prefix of the calling thread and, through `total`, the sum of all values.
__device__ __forceinline__ uint32_t cta_exclusive_scan(uint32_t v, uint32_t *wsum /*[33] shared*/, uint32_t &total)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    __syncthreads();   // wsum may still be read from an earlier scan
    if (lane == 31) wsum[w] = incl;
    __syncthreads();
    if (w == 0) {
        const uint32_t a = wsum[lane];
        uint32_t x = a;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += t;
        }
        wsum[lane] = x - a;   // exclusive
        if (lane == 31) wsum[32] = x;
    }
    __syncthreads();
    total = wsum[32];
    return wsum[w] + incl - v;
}

// One CTA of 1024 threads (KK <= 1024): exclusive scan of the key totals (cluster_start, KK + 1
// entries), the segment length for this sort, the exclusive scan of the segment counts
// ceil(total / length) (seg_start, KK + 1 entries, followed by the length itself), and the cluster
// sizes: full mode counts[k] = total[k]; delta mode counts[k] += total[k] - total[K + k].
// The segment length shrinks with the number of entries M actually present (a delta sort of a
// settled clustering holds a handful): length = seg_rows_max * M / NE rounded up to 16, at least 16,
// so that short lists still spread over many CTAs and the segment count stays within
// NE / seg_rows_max + KK.
// Runs in every CTA of the scatter kernel (each needs the key offsets for its own entries); the CTA
// with `publish` set also writes the tables and updates the cluster sizes.  Returns this thread's
// key offset (thread k < KK).
__device__ __forceinline__ uint32_t scan_keys(const uint32_t *__restrict__ key_total, int K, int KK, int seg_rows_max,
                                              int64_t NE, int delta, bool publish, int64_t *__restrict__ counts,
                                              int32_t *__restrict__ cluster_start, int32_t *__restrict__ seg_start,
                                              int32_t *settled, uint32_t *wsum /*[33] shared*/)
{
    const int k = threadIdx.x;
    const uint32_t tot = (k < KK) ? key_total[k] : 0u;
    uint32_t M = 0;
    const uint32_t ea = cta_exclusive_scan(tot, wsum, M);
    if (!publish) return ea;
    int64_t sr = ((int64_t)seg_rows_max * (int64_t)M + NE - 1) / NE;
    sr = (sr + 15) / 16 * 16;
    if (sr < 16) sr = 16;
    if (sr > seg_rows_max) sr = seg_rows_max;
    const uint32_t sg = (tot + (uint32_t)sr - 1) / (uint32_t)sr;
    uint32_t nseg = 0;
    const uint32_t es = cta_exclusive_scan(sg, wsum, nseg);
    if (k < KK) {
        cluster_start[k] = (int32_t)ea;
        seg_start[k] = (int32_t)es;
    }
    if (k == 0) {
        cluster_start[KK] = (int32_t)M;
        seg_start[KK] = (int32_t)nseg;
        seg_start[KK + 1] = (int32_t)sr;
        if (settled && M == 0) *settled = 1;   // (read by later launches; a CTA of this one that sees it has no entry to place)
    }
    if (k < K) {
        if (delta) counts[k] += (int64_t)tot - (int64_t)key_total[K + k];
        else counts[k] = (int64_t)tot;
    }
    return ea;
}

// Stable scatter.  Within a block, an entry's rank among the entries of its key is
// (entries of that key in earlier warps) + (entries of that key in earlier lanes).
__global__ void __launch_bounds__(SORT_BLOCK) label_scatter_kernel(const int32_t *__restrict__ cur,
                                                                    const int32_t *__restrict__ prev, int64_t N, int K,
                                                                    int KK, const uint32_t *__restrict__ blk_hist,
                                                                    const uint32_t *__restrict__ key_total,
                                                                    int seg_rows_max, int64_t NE, int delta,
                                                                    int64_t *__restrict__ counts,
                                                                    int32_t *__restrict__ cluster_start,
                                                                    int32_t *__restrict__ seg_start,
                                                                    int32_t *__restrict__ order, int32_t *settled)
{
    extern __shared__ uint32_t scatter_smem[];   // [KK] key offsets, then [32][KK] 16-bit warp histograms
    __shared__ uint32_t wsum[33];
    uint32_t *key_off = scatter_smem;
    uint16_t *warp_hist = reinterpret_cast<uint16_t *>(scatter_smem + KK);
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    for (int e = tid; e < 32 * KK; e += SORT_BLOCK) warp_hist[e] = 0;
    pdl_enter();
    const int64_t e = (int64_t)blockIdx.x * SORT_BLOCK + tid;
    const bool over = settled && tid == 0 && *(volatile int32_t *)settled;
    const int l = entry_key(cur, prev, N, K, e);
    // (one read per CTA: CTA 0 may set the word while others of this launch are here)
    if (settled && __syncthreads_or(over)) return;
    {
        const uint32_t ea = scan_keys(key_total, K, KK, seg_rows_max, NE, delta, blockIdx.x == 0, counts, cluster_start,
                                      seg_start, settled, wsum);
        if (tid < KK) key_off[tid] = ea;
    }
    __syncthreads();
    const unsigned peers = __match_any_sync(0xffffffffu, l);
    const int rank_in_warp = __popc(peers & ((1u << lane) - 1u));
    if (l >= 0 && rank_in_warp == 0) warp_hist[w * KK + l] = (uint16_t)__popc(peers);
    __syncthreads();
    for (int k = tid; k < KK; k += SORT_BLOCK) {
        uint16_t run = 0;
        for (int q = 0; q < 32; ++q) {
            const uint16_t v = warp_hist[q * KK + k];
            warp_hist[q * KK + k] = run;
            run = (uint16_t)(run + v);
        }
    }
    __syncthreads();
    if (l >= 0) {
        const uint32_t pos = key_off[l] + blk_hist[(size_t)l * gridDim.x + blockIdx.x] +
                             warp_hist[w * KK + l] + (uint32_t)rank_in_warp;
        order[pos] = (int32_t)(e < N ? e : e - N);
    }
}

struct SegParams {
    const float *Yq;
    const float *Yf;            // second matrix (modes 1, 2)
    const int32_t *order;
    const int32_t *cluster_start;
    const int32_t *seg_start;
    const double *meanQ;        // mode 2
    const double *meanF;
    double *part;               // [maxsegs][2][D]
    int D;
    int K;
    int seg_rows;
    int tpr;                    // threads per row (power of two <= 256)
    const int32_t *settled;
};

__device__ __forceinline__ void add4(double (&a)[4], const float4 v)
{
    a[0] += (double)v.x;
    a[1] += (double)v.y;
    a[2] += (double)v.z;
    a[3] += (double)v.w;
}

// One row's contribution (VEC columns) to the accumulators of a segment.
template <int MODE, int VEC>
__device__ __forceinline__ void seg_accumulate(double (&a0)[4], double (&a1)[4], double (&a2)[4], const double (&mq)[4],
                                               const double (&mf)[4], const float4 q4, const float4 f4)
{
    if (MODE == 0) {
        add4(a0, q4);
    } else if (MODE == 1) {
        add4(a0, q4);
        add4(a1, f4);
    } else {
        const float qv[4] = {q4.x, q4.y, q4.z, q4.w};
        const float fv[4] = {f4.x, f4.y, f4.z, f4.w};
#pragma unroll
        for (int q = 0; q < VEC; ++q) {
            const double dq = (double)qv[q] - mq[q];
            const double df = (double)fv[q] - mf[q];
            a0[q] = fma(dq, dq, a0[q]);
            a1[q] = fma(dq, df, a1[q]);
            if (MODE == 3) a2[q] += (double)fv[q];
        }
    }
}

// MODE 0: sums of Yq -> plane 0.  MODE 1: sums of Yq, Yf -> planes 0, 1.
// MODE 2: centred moments -> plane 0 = sum (q-muQ)^2, plane 1 = sum (q-muQ)(f-muF).
// MODE 3: the final pass of cat_fit in one sweep, with the cluster mean muQ known beforehand:
//         plane 0 = sum (q-muQ)^2, plane 1 = sum (q-muQ)(f-muQ), plane 2 = sum f (three planes
//         per segment).  Since sum (q-muQ) = 0, plane 1 is the centred cross moment whatever
//         constant is subtracted from f; muQ keeps the products small.
// VEC: 4 = 128-bit loads (D % 4 == 0), 1 = scalar loads.
template <int MODE, int VEC>
__global__ void __launch_bounds__(SEG_THREADS) segment_sums_kernel(SegParams p)
{
    pdl_enter();
    __shared__ int32_t rows_s[128];
    __shared__ double red_s[SEG_THREADS * VEC];
    const int over = p.settled ? *p.settled : 0, nseg_total = p.seg_start[p.K];
    if (over) return;
    for (int seg = blockIdx.x; seg < nseg_total; seg += gridDim.x) {
    // cluster of this segment: last k with seg_start[k] <= seg
    int lo = 0, hi = p.K;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (p.seg_start[mid] <= seg) lo = mid; else hi = mid;
    }
    const int k = lo;
    const int seg_rows = p.seg_start[p.K + 1];   // length chosen by the sort for this list
    const int first = p.cluster_start[k] + (seg - p.seg_start[k]) * seg_rows;
    int nrows = p.cluster_start[k + 1] - first;
    if (nrows > seg_rows) nrows = seg_rows;

    const int tid = threadIdx.x;
    const int tpr = p.tpr;
    const int c = tid & (tpr - 1);      // column unit within the block of columns
    const int g = tid / tpr;            // row group
    const int G = SEG_THREADS / tpr;
    const int units = (p.D + VEC - 1) / VEC;          // column units per row
    const int col0 = blockIdx.y * SEG_THREADS;        // first unit of this column block
    const int unit = col0 + c;
    const bool active = (c < SEG_THREADS) && (unit < units);
    const int col = unit * VEC;

    double a0[4] = {0, 0, 0, 0}, a1[4] = {0, 0, 0, 0}, a2[4] = {0, 0, 0, 0};
    double mq[4] = {0, 0, 0, 0}, mf[4] = {0, 0, 0, 0};
    if (MODE >= 2 && active) {
#pragma unroll
        for (int q = 0; q < VEC; ++q) {
            mq[q] = p.meanQ[(size_t)k * p.D + col + q];
            mf[q] = (MODE == 2) ? p.meanF[(size_t)k * p.D + col + q] : mq[q];
        }
    }

    for (int base = 0; base < nrows; base += 128) {
        const int nb = (nrows - base < 128) ? (nrows - base) : 128;
        __syncthreads();
        if (tid < nb) rows_s[tid] = p.order[first + base + tid];
        __syncthreads();
        if (!active) continue;
        int r = g;
        // four rows in flight per thread
        for (; r + 3 * G < nb; r += 4 * G) {
            float4 q4[4], f4[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const size_t o = (size_t)rows_s[r + u * G] * p.D + col;
                if (VEC == 4) {
                    q4[u] = __ldg(reinterpret_cast<const float4 *>(p.Yq + o));
                    if (MODE != 0) f4[u] = __ldg(reinterpret_cast<const float4 *>(p.Yf + o));
                } else {
                    q4[u] = make_float4(__ldg(p.Yq + o), 0.f, 0.f, 0.f);
                    if (MODE != 0) f4[u] = make_float4(__ldg(p.Yf + o), 0.f, 0.f, 0.f);
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) seg_accumulate<MODE, VEC>(a0, a1, a2, mq, mf, q4[u], f4[u]);
        }
        for (; r < nb; r += G) {
            const size_t o = (size_t)rows_s[r] * p.D + col;
            float4 q4, f4 = make_float4(0.f, 0.f, 0.f, 0.f);
            if (VEC == 4) {
                q4 = __ldg(reinterpret_cast<const float4 *>(p.Yq + o));
                if (MODE != 0) f4 = __ldg(reinterpret_cast<const float4 *>(p.Yf + o));
            } else {
                q4 = make_float4(__ldg(p.Yq + o), 0.f, 0.f, 0.f);
                if (MODE != 0) f4 = make_float4(__ldg(p.Yf + o), 0.f, 0.f, 0.f);
            }
            seg_accumulate<MODE, VEC>(a0, a1, a2, mq, mf, q4, f4);
        }
    }

    // add the row groups in a fixed order and publish the segment's partial row
    constexpr int NPLANES = (MODE == 0) ? 1 : (MODE == 3 ? 3 : 2);
    constexpr int PSTRIDE = (MODE == 3) ? 3 : 2;   // planes per segment in `part`
#pragma unroll
    for (int pl = 0; pl < NPLANES; ++pl) {
        __syncthreads();
#pragma unroll
        for (int q = 0; q < VEC; ++q) red_s[tid * VEC + q] = (pl == 0) ? a0[q] : (pl == 1 ? a1[q] : a2[q]);
        __syncthreads();
        if (g == 0 && active) {
            double *dst = p.part + ((size_t)seg * PSTRIDE + pl) * p.D + col;
#pragma unroll
            for (int q = 0; q < VEC; ++q) {
                double s = 0.0;
                for (int gg = 0; gg < G; ++gg) s += red_s[(gg * tpr + c) * VEC + q];
                dst[q] = s;
            }
        }
    }
    __syncthreads();   // red_s and rows_s are reused by the next segment
    }
}

// out0/out1[k*D+j] = sum over the segments of key k of plane 0/1 (out1 may be NULL); in
// delta mode out0[k*D+j] += (segments of key k) - (segments of key K + k).  With C != NULL
// also C[k*D+j] = float(out0 / n_k) where n_k > 0.
__global__ void segment_combine_kernel(const double *__restrict__ part, const int32_t *__restrict__ seg_start,
                                       const int64_t *__restrict__ counts, int D, int K, size_t KD, int delta,
                                       double *__restrict__ out0, double *__restrict__ out1,
                                       float *__restrict__ C)
{
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= KD) return;
    const int k = (int)(e / D);
    const int j = (int)(e - (size_t)k * D);
    const int s0 = seg_start[k], s1 = seg_start[k + 1];
    double a = 0.0, b = 0.0;
    for (int sgm = s0; sgm < s1; ++sgm) {
        a += part[((size_t)sgm * 2) * D + j];
        if (out1) b += part[((size_t)sgm * 2 + 1) * D + j];
    }
    if (delta) {
        double m = 0.0;
        for (int sgm = seg_start[K + k]; sgm < seg_start[K + k + 1]; ++sgm) m += part[((size_t)sgm * 2) * D + j];
        a = out0[e] + (a - m);
    }
    out0[e] = a;
    if (out1) out1[e] = b;
    if (C) {
        const int64_t n = counts[k];
        if (n > 0) C[e] = (float)(a / (double)n);
    }
}

// The kernels that add up a cluster's segments: a CTA takes `cols` columns of a cluster, G = threads / cols threads
// a column, thread g of them the segments first + g, first + g + G, ..., whose sums are then added
// in that order.  (One thread per column is a chain of loads as long as the cluster has segments: with K = 2 and
// 100 000 rows 224 us for the three planes and 19 us a Lloyd round.  More threads than segments are a longer
// exchange for nothing: 8192 x 64, K = 200 takes 8.6 us a round with 16 of them, 6.3 with two and whole rows.)
// P planes of a segment lie `plane` apart; four segments' loads are in flight together
template <int P>
__device__ __forceinline__ void sum_segments(const double *__restrict__ p, int s0, int s1, int step, size_t stride, size_t plane,
                                             double (&out)[P])
{
    double a[P][4];
#pragma unroll
    for (int q = 0; q < P; ++q)
#pragma unroll
        for (int u = 0; u < 4; ++u) a[q][u] = 0.0;
    for (int s = s0; s < s1; s += 4 * step) {
        double v[P][4];
#pragma unroll
        for (int q = 0; q < P; ++q)
#pragma unroll
            for (int u = 0; u < 4; ++u) v[q][u] = s + u * step < s1 ? __ldg(p + (size_t)(s + u * step) * stride + q * plane) : 0.0;
#pragma unroll
        for (int q = 0; q < P; ++q)
#pragma unroll
            for (int u = 0; u < 4; ++u) a[q][u] += v[q][u];
    }
#pragma unroll
    for (int q = 0; q < P; ++q) out[q] = (a[q][0] + a[q][1]) + (a[q][2] + a[q][3]);
}

// every thread of a column gets the sum of its threads' values; red: [COMB_THREADS]
__device__ __forceinline__ double sum_column(double v, int cols, double *red)
{
    if (cols == (int)blockDim.x) return v;
    __syncthreads();
    red[threadIdx.x] = v;
    __syncthreads();
    double t = 0.0;
    for (int g = threadIdx.x & (cols - 1); g < (int)blockDim.x; g += cols) t += red[g];
    return t;
}

// Columns and threads of a CTA: as many CTAs as the device holds a few times over, no more; as many threads a column as
// a cluster has segments on average; whole rows where they fit then.
struct CombGeom {
    int cols, threads;
};
CombGeom comb_geometry(int D, int K, int max_segs)
{
    int cols = 32, G = 1;
    while (cols < COMB_THREADS && (int64_t)K * ((D + cols - 1) / cols) > 4 * 148) cols *= 2;
    while (cols * G < COMB_THREADS && 2 * G * (int64_t)K <= max_segs) G *= 2;
    int whole = 32;
    while (whole < D && whole < COMB_THREADS) whole *= 2;
    if (whole >= D && whole > cols) {
        const int Gw = G < COMB_THREADS / whole ? G : COMB_THREADS / whole;
        if (max_segs <= (int64_t)K * Gw * 8) {   // (two batches of loads a thread at most)
            cols = whole;
            G = Gw;
        }
    }
    return {cols, cols * G};
}

// Three-plane partials (MODE 3) added up per cluster.
__global__ void __launch_bounds__(COMB_THREADS) segment_combine3_kernel(const double *__restrict__ part,
                                                                        const int32_t *__restrict__ seg_start, int D, int cols,
                                                                        double *__restrict__ out0, double *__restrict__ out1,
                                                                        double *__restrict__ out2)
{
    pdl_enter();
    __shared__ double red[COMB_THREADS];
    const int k = blockIdx.x, g = threadIdx.x / cols, G = (int)blockDim.x / cols;
    const int j = (int)blockIdx.y * cols + (threadIdx.x & (cols - 1));
    const int s0 = seg_start[k], s1 = seg_start[k + 1];
    double v[3] = {0.0, 0.0, 0.0};
    if (j < D) sum_segments<3>(part + j, s0 + g, s1, G, (size_t)3 * D, (size_t)D, v);
#pragma unroll
    for (int q = 0; q < 3; ++q) v[q] = sum_column(v[q], cols, red);
    if (g == 0 && j < D) {
        const size_t e = (size_t)k * D + j;
        out0[e] = v[0];
        out1[e] = v[1];
        out2[e] = v[2];
    }
}

// What a Lloyd round does with a cluster once the change d of its sums is known: S_k += d; c_k = float(S_k / n_k) where
// n_k > 0; and for the next assignment the squared norm of c_k (fp64, rounded up), optionally the fp16 copy
// fp16(c_k * scale[0]) with the norm of its rounding error -- both of c_k less `mean` if that is given.  The CTAs
// (k, 0 ... gridDim.y - 1) of a cluster have `cols` columns each, thread j of the first `cols` the j-th; they leave their
// parts of the two norms in `norm_part`, and the last one to arrive (`arrivals`, which wraps back to zero) adds them up, in an
// order that does not depend on who came when.
struct FinishParams {
    double *sums;
    float *C;
    float *cnorm;
    const float *scale;
    __half *Ch;
    const float *mean;
    float *cerr;
    double2 *norm_part;
    unsigned int *arrivals;
    int64_t *counts_out;   // the cluster's size is left here by whoever finishes last (or null)
    int D, cols;
};

__device__ __forceinline__ void finish_centroid(const FinishParams &f, double d, int64_t n, double *red, float *red_err, int *s_last)
{
    const int D = f.D, cols = f.cols;
    const int k = blockIdx.x, cb = blockIdx.y, j = cb * cols + (int)threadIdx.x;
    const float sc = f.Ch ? f.scale[0] : 1.f;
    double nrm = 0.0;
    float left2 = 0.f;
    if ((int)threadIdx.x < cols && j < D) {
        const size_t e = (size_t)k * D + j;
        const double sum = f.sums[e] + d;
        f.sums[e] = sum;
        float c = f.C[e];
        if (n > 0) {
            c = (float)(sum / (double)n);
            f.C[e] = c;
        }
        if (f.mean) c -= __ldg(f.mean + j);
        nrm = (double)c * (double)c;
        if (f.Ch) {
            const __half h = __float2half_rn(c * sc);
            f.Ch[(size_t)k * half_ld(D) + j] = h;
            const float l = c * sc - __half2float(h);
            left2 = l * l;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        nrm += __shfl_xor_sync(0xffffffffu, nrm, o);
        left2 += __shfl_xor_sync(0xffffffffu, left2, o);
    }
    __syncthreads();
    if ((threadIdx.x & 31) == 0) {
        red[threadIdx.x >> 5] = nrm;
        red_err[threadIdx.x >> 5] = left2;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0, l = 0.0;
        for (int w = 0; w < cols / 32; ++w) {
            t += red[w];
            l += (double)red_err[w];
        }
        if (gridDim.y == 1) {
            f.cnorm[k] = __double2float_ru(t);
            if (f.Ch) f.cerr[k] = sqrtf((float)l) / sc * 1.001f;
            if (f.counts_out) f.counts_out[k] = n;
        } else {
            f.norm_part[(size_t)k * gridDim.y + cb] = make_double2(t, l);
            __threadfence();
            *s_last = atomicInc(f.arrivals + k, gridDim.y - 1) == gridDim.y - 1;
        }
    }
    if (gridDim.y == 1) return;
    __syncthreads();
    if (*s_last && threadIdx.x < 32) {
        __threadfence();
        double t = 0.0, l = 0.0;
        for (int q = threadIdx.x; q < (int)gridDim.y; q += 32) {
            const double2 v = __ldcg(f.norm_part + (size_t)k * gridDim.y + q);
            t += v.x;
            l += v.y;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            t += __shfl_xor_sync(0xffffffffu, t, o);
            l += __shfl_xor_sync(0xffffffffu, l, o);
        }
        if (threadIdx.x != 0) return;
        f.cnorm[k] = __double2float_ru(t);
        if (f.Ch) f.cerr[k] = sqrtf((float)l) / sc * 1.001f;
        if (f.counts_out) f.counts_out[k] = n;
    }
}

// Delta-mode centroid update from the segments' partial sums: the change of a cluster's sums is (partials of key k) -
// (partials of key K + k).  Also resets the exact-pass queues.
// (32 registers a thread: four CTAs per SM, so that the 592 CTAs of the geometry above are one wave)
__global__ void __launch_bounds__(COMB_THREADS, 4) centroid_update_kernel(const double *__restrict__ part,
                                                              const int32_t *__restrict__ seg_start,
                                                              const int64_t *__restrict__ counts, int K, FinishParams f,
                                                              Control *ctl, const int32_t *settled)
{
    pdl_enter();
    __shared__ double red[COMB_THREADS];
    __shared__ float red_err[COMB_THREADS / 32];
    __shared__ int s_last;
    const int D = f.D, cols = f.cols;
    const int k = blockIdx.x, cb = blockIdx.y, g = threadIdx.x / cols, G = (int)blockDim.x / cols;
    if (k == 0 && cb == 0 && threadIdx.x == 0) {
        ctl->refine_count = 0;
        ctl->cand_count = 0;
    }
    const int over = settled ? *settled : 0;
    const int j = cb * cols + (threadIdx.x & (cols - 1));
    const int64_t n = counts[k];
    if (over) return;
    double in[1] = {0.0}, gone[1] = {0.0};
    if (j < D) {
        sum_segments<1>(part + j, seg_start[k] + g, seg_start[k + 1], G, (size_t)2 * D, 0, in);
        sum_segments<1>(part + j, seg_start[K + k] + g, seg_start[K + k + 1], G, (size_t)2 * D, 0, gone);
    }
    finish_centroid(f, sum_column(in[0] - gone[0], cols, red), n, red, red_err, &s_last);
}

// ---- rounds in which few rows move: two launches in place of five
//
// The sort, its tables and the segments cost 25 to 45 us a round whatever moves (histograms of 2 K keys for every 1024
// rows of two label buffers; five launches).  Once the clustering has found its shape a hundredth of the rows moves: those are
// listed, by cluster within each CTA's rows, and a cluster's CTAs read its pieces of the list.  (A list in row order, of which a
// cluster's CTAs read all and picked theirs, lost where a tenth of the rows keeps moving: 25 rounds on a cloud of 1 048 576 x 64, K = 256
// 9.21 ms sorted, 9.77 with it, 8.13 so; on logits of 262 144 x 512, K = 128 4.31, 4.49 and 3.90.)

constexpr int MOVE_THREADS = 512;
constexpr int MOVE_WARPS = MOVE_THREADS / 32;
constexpr int MOVE_GRID = 148;
constexpr int MOVE_TILE = 4 * MOVE_THREADS;
constexpr int MOVE_CHUNK = 2048;

__device__ __forceinline__ void load_labels(const int32_t *__restrict__ l, int64_t r, int64_t end, int (&v)[4])
{
    if (r + 4 <= end) {
        const int4 x = __ldg(reinterpret_cast<const int4 *>(l + r));
        v[0] = x.x, v[1] = x.y, v[2] = x.z, v[3] = x.w;
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = r + q < end ? __ldg(l + r + q) : -1;
    }
}

// Lists the rows whose label changed, once under either label: a CTA has `per` consecutive rows and leaves its entries (row,
// bit 31: it leaves) in list[2 per b ...], those of cluster k from table[k][b] up to table[k + 1][b].  Sets *settled if no row of
// any CTA has moved (*state, CTAs arrived << 32 | rows moved, is zero before and after).  Entries of a cluster are in an order
// that does not depend on timing: by tiles of 2048 rows, the tile's warps, the four rows of a lane, entering before leaving, lanes.
// (K <= MOVE_THREADS; labels outside [0, K) are left out.)
__global__ void __launch_bounds__(MOVE_THREADS) moved_list_kernel(const int32_t *__restrict__ cur, const int32_t *__restrict__ prev, int64_t N,
                                                                  int K, int per, uint32_t *__restrict__ list, uint32_t *__restrict__ table,
                                                                  unsigned long long *state, int32_t *settled)
{
    __shared__ uint32_t base[MOVE_THREADS];     // where the next entry of a cluster goes
    __shared__ uint32_t s_warp[MOVE_WARPS];
    __shared__ int s_moved;
    __shared__ uint16_t cnt[MOVE_WARPS * MOVE_THREADS];   // [warp][K] entries of a tile
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, G = gridDim.x;
    base[tid] = 0u;
    for (int e = tid; e < MOVE_WARPS * K; e += MOVE_THREADS) cnt[e] = 0;
    if (tid == 0) s_moved = 0;
    pdl_enter();
    if (*(volatile int32_t *)settled) return;   // (set by the last CTA to arrive below: every thread of the launch has been here by then)
    const int64_t row0 = (int64_t)blockIdx.x * per, end = row0 + per < N ? row0 + per : N;
    auto key_ok = [&](int k) { return (unsigned)k < (unsigned)K; };
    int c[4], p[4];
    uint32_t rank[8], run = 0;   // run: of thread k, entries of cluster k in the tile
    auto load = [&](int64_t r) {
        load_labels(cur, r, end, c);
        load_labels(prev, r, end, p);
        return c[0] != p[0] || c[1] != p[1] || c[2] != p[2] || c[3] != p[3];
    };
    // place of each of this thread's entries among its warp's of the same cluster
    auto rank_tile = [&]() {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int q = i >> 1, key = c[q] != p[q] ? (i & 1 ? p[q] : c[q]) : -1;
            const bool ok = key_ok(key);
            rank[i] = 0u;
            if (!__any_sync(0xffffffffu, ok)) continue;
            const unsigned peers = __match_any_sync(0xffffffffu, ok ? key : -1);
            const uint32_t had = ok ? cnt[warp * K + key] : 0u;
            __syncwarp();
            if (ok && lane == __ffs(peers) - 1) cnt[warp * K + key] = (uint16_t)(had + __popc(peers));
            __syncwarp();
            rank[i] = had + __popc(peers & ((1u << lane) - 1u));
        }
    };
    // the warps' numbers to places ahead of each warp's
    auto scan_warps = [&]() {
        run = 0;
        if (tid < K)
#pragma unroll 4
            for (int w = 0; w < MOVE_WARPS; ++w) {
                const uint32_t v = cnt[w * K + tid];
                cnt[w * K + tid] = (uint16_t)run;
                run += v;
            }
    };
    const bool one = per == MOVE_TILE;   // the usual case: labels are read once
    bool some = load(row0 + 4 * tid);
    __syncthreads();
    int moved = 0;
    if (one) {
#pragma unroll
        for (int q = 0; q < 4; ++q) moved += c[q] != p[q];
        if (__any_sync(0xffffffffu, some)) rank_tile();
    } else
        for (int64_t r = row0 + 4 * tid; r < end; r += MOVE_TILE) {
            load(r);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (c[q] != p[q]) {
                    ++moved;
                    if (key_ok(c[q])) atomicAdd(base + c[q], 1u);
                    if (key_ok(p[q])) atomicAdd(base + p[q], 1u);
                }
        }
    moved = __reduce_add_sync(0xffffffffu, moved);
    if (lane == 0 && moved) atomicAdd(&s_moved, moved);
    __syncthreads();
    unsigned long long before_me = 0ull;   // (asked for here and looked at last)
    if (tid == 0) before_me = atomicAdd(state, 1ull << 32 | (unsigned long long)(unsigned)s_moved);
    {
        if (one) scan_warps();
        const uint32_t v = one ? run : base[tid];
        uint32_t incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) s_warp[warp] = incl;
        __syncthreads();
        uint32_t before = 0;
#pragma unroll
        for (int w = 0; w < MOVE_WARPS; ++w) before += w < warp ? s_warp[w] : 0u;
        base[tid] = before + incl - v;
        if (tid < K) {
            table[(size_t)tid * G + blockIdx.x] = before + incl - v;
            if (tid == K - 1) table[(size_t)K * G + blockIdx.x] = before + incl;
        }
    }
    if (s_moved != 0) {
        uint32_t *out = list + 2 * row0;
        auto put_tile = [&](int64_t r) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int q = i >> 1, key = c[q] != p[q] ? (i & 1 ? p[q] : c[q]) : -1;
                if (key_ok(key)) out[base[key] + cnt[warp * K + key] + rank[i]] = (uint32_t)(r + q) | (i & 1 ? 0x80000000u : 0u);
            }
        };
        __syncthreads();
        if (one) {
            if (some) put_tile(row0 + 4 * tid);
        } else
            for (int64_t t0 = row0; t0 < end; t0 += MOVE_TILE) {
                some = load(t0 + 4 * tid);
                if (!__syncthreads_or(some)) continue;   // (also: the tile before is through)
                if (__any_sync(0xffffffffu, some)) rank_tile();
                __syncthreads();
                scan_warps();
                __syncthreads();
                if (some) put_tile(t0 + 4 * tid);
                __syncthreads();
                if (tid < K) {
                    base[tid] += run;
                    for (int w = 0; w < MOVE_WARPS; ++w) cnt[w * K + tid] = 0;
                }
            }
    }
    if (tid == 0 && (unsigned)(before_me >> 32) == (unsigned)G - 1u) {
        if ((uint32_t)before_me + (uint32_t)s_moved == 0u) *settled = 1;
        *state = 0ull;
    }
}

// A CTA per `cols` columns of a cluster: its entries of the list, in order, entering and leaving, then as above.  tpr threads
// (of VEC columns) have a row, 256 / tpr rows at a time, each group of threads into sums of its own.
template <int VEC>
__global__ void __launch_bounds__(SEG_THREADS) cluster_move_kernel(const float *__restrict__ Y, const uint32_t *__restrict__ list,
                                                                   const uint32_t *__restrict__ table, int sources, int per,
                                                                   const int64_t *__restrict__ counts, int tpr, FinishParams f, Control *ctl,
                                                                   const int32_t *settled)
{
    pdl_enter();
    __shared__ double red[SEG_THREADS * VEC];
    __shared__ float red_err[SEG_THREADS / 32];
    __shared__ uint32_t sel[MOVE_CHUNK];
    __shared__ uint32_t pos[MOVE_GRID + 1], from[MOVE_GRID];   // entries ahead of a source's first, and where that one is
    __shared__ int s_cnt[SEG_THREADS / 32], s_last;
    static_assert(MOVE_GRID < SEG_THREADS, "a thread per source");
    const int k = blockIdx.x, cb = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (k == 0 && cb == 0 && tid == 0) {
        ctl->refine_count = 0;
        ctl->cand_count = 0;
    }
    if (*settled) return;
    const int D = f.D, g = tid / tpr, G = SEG_THREADS / tpr, col = cb * f.cols + (tid & (tpr - 1)) * VEC;
    int64_t n = counts[k];
    {
        uint32_t at = 0u, len = 0u;
        if (tid < sources) {
            at = __ldg(table + (size_t)k * sources + tid);
            len = __ldg(table + (size_t)(k + 1) * sources + tid) - at;
        }
        uint32_t incl = len;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) s_cnt[warp] = (int)incl;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < SEG_THREADS / 32; ++w) incl += w < warp ? (uint32_t)s_cnt[w] : 0u;
        if (tid < sources) {
            pos[tid] = incl - len;
            from[tid] = 2u * (uint32_t)tid * (uint32_t)per + at;
            if (tid == sources - 1) pos[sources] = incl;
        }
        __syncthreads();
    }
    double acc[VEC];
#pragma unroll
    for (int q = 0; q < VEC; ++q) acc[q] = 0.0;
    const uint32_t total = pos[sources];
    int dn = 0;
    for (uint32_t h0 = 0; h0 < total; h0 += MOVE_CHUNK) {
        const int hits = (int)(total - h0 < (uint32_t)MOVE_CHUNK ? total - h0 : (uint32_t)MOVE_CHUNK);
        __syncthreads();   // (the rows of the chunk before are through)
        for (int i = tid; i < hits; i += SEG_THREADS) {
            // the last source with no more than h0 + i entries ahead of it has the entry
            int lo = 0, hi = sources;
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (pos[mid] <= h0 + i) lo = mid;
                else hi = mid;
            }
            const uint32_t en = __ldg(list + from[lo] + (h0 + i - pos[lo]));
            sel[i] = en;
            dn += en >> 31 ? -1 : 1;
        }
        __syncthreads();
        for (int e = g; e < hits; e += 4 * G) {
            float4 y[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = e + u * G;
                y[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (i < hits && col < D) {
                    const float *src = Y + (size_t)(sel[i] & 0x7FFFFFFFu) * D + col;
                    if (VEC == 4) y[u] = __ldg(reinterpret_cast<const float4 *>(src));
                    else y[u].x = __ldg(src);
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = e + u * G;
                if (i >= hits) break;
                const float v[4] = {y[u].x, y[u].y, y[u].z, y[u].w};
                const bool leaves = sel[i] >> 31;
#pragma unroll
                for (int q = 0; q < VEC; ++q) acc[q] += leaves ? -(double)v[q] : (double)v[q];
            }
        }
    }
    // the change of the cluster's size (integers: any order will do)
    dn = __reduce_add_sync(0xffffffffu, dn);
    __syncthreads();
    if (lane == 0) s_cnt[warp] = dn;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < SEG_THREADS / 32; ++q) n += s_cnt[q];
    __syncthreads();
#pragma unroll
    for (int q = 0; q < VEC; ++q) red[tid * VEC + q] = acc[q];
    __syncthreads();
    double d = 0.0;
    if (tid < f.cols)
        for (int q = 0; q < G; ++q) d += red[q * f.cols + tid];   // (thread tid of a group's tpr has columns VEC tid ... )
    __syncthreads();
    finish_centroid(f, d, n, red, red_err, &s_last);
}

// ---- the closed form of a small set in one launch
//
// A CTA has `cols` columns of a cluster: it picks the cluster's rows out of the labels, in row order, and goes through them
// for the moments (for the means too, where the sums are not known yet) -- tpr threads (of VEC columns) a row, 256 / tpr rows
// at a time, each group of threads into fp64 sums of its own -- and solves.  The general way sorts the rows, makes
// segments, adds those up and solves, in seven launches: 29 us of a fit of 1024 x 1000 rows with K = 16.
constexpr int MOM_MAX_ROWS = 8192;

template <int VEC>
__global__ void __launch_bounds__(SEG_THREADS) cluster_moments_kernel(const float *__restrict__ Yq, const float *__restrict__ Yf,
                                                                      const int32_t *__restrict__ labels, int N, int D, int cols, int tpr,
                                                                      const double *__restrict__ sumQ, float *__restrict__ gamma,
                                                                      float *__restrict__ beta)
{
    pdl_enter();
    __shared__ double red[SEG_THREADS * VEC];
    __shared__ uint16_t sel[MOM_MAX_ROWS];
    __shared__ int s_cnt[SEG_THREADS / 32];
    const int k = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = tid / tpr, G = SEG_THREADS / tpr, col = (int)blockIdx.y * cols + (tid & (tpr - 1)) * VEC;
    // a thread looks at 32 consecutive rows
    const int r0 = tid * (MOM_MAX_ROWS / SEG_THREADS);
    uint32_t mine = 0;
#pragma unroll
    for (int q = 0; q < MOM_MAX_ROWS / SEG_THREADS; q += 4) {
        const int r = r0 + q;
        if (r + 4 <= N) {
            const int4 l = __ldg(reinterpret_cast<const int4 *>(labels + r));
            mine |= (uint32_t)((l.x == k) | (l.y == k) << 1 | (l.z == k) << 2 | (l.w == k) << 3) << q;
        } else
            for (int u = 0; u < 4 && r + u < N; ++u) mine |= (uint32_t)(__ldg(labels + r + u) == k) << (q + u);
    }
    const int c = __popc(mine);
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) s_cnt[warp] = incl;
    __syncthreads();
    int at = incl - c, n = 0;
#pragma unroll
    for (int w = 0; w < SEG_THREADS / 32; ++w) {
        if (w < warp) at += s_cnt[w];
        n += s_cnt[w];
    }
    for (; mine; mine &= mine - 1) sel[at++] = (uint16_t)(r0 + __ffs(mine) - 1);
    __syncthreads();
    const double dn = (double)n;
    double mu[VEC];
#pragma unroll
    for (int q = 0; q < VEC; ++q) mu[q] = 0.0;
    // adds the groups' values of a plane up, in order; thread j of the first `cols` gets column j
    auto combine = [&](const double (&v)[VEC]) {
        __syncthreads();
#pragma unroll
        for (int q = 0; q < VEC; ++q) red[tid * VEC + q] = v[q];
        __syncthreads();
        double s = 0.0;
        if (tid < cols)
            for (int q = 0; q < G; ++q) s += red[q * cols + tid];
        return s;
    };
    auto row4 = [&](const float *Y, int e) {
        float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
        if (e < n && col < D) {
            const float *src = Y + (size_t)sel[e] * D + col;
            if constexpr (VEC == 4) y = __ldg(reinterpret_cast<const float4 *>(src));
            else y.x = __ldg(src);
        }
        return y;
    };
    const int j = (int)blockIdx.y * cols + tid;   // the column this thread finishes
    double mean = 0.0;
    if (sumQ) {
        if (n > 0) {
#pragma unroll
            for (int q = 0; q < VEC; ++q)
                if (col + q < D) mu[q] = sumQ[(size_t)k * D + col + q] / dn;
            if (tid < cols && j < D) mean = sumQ[(size_t)k * D + j] / dn;
        }
    } else {
        double a[VEC] = {};
        for (int e = g; e < n; e += 8 * G) {
            float4 y[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) y[u] = row4(Yq, e + u * G);
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const float v[4] = {y[u].x, y[u].y, y[u].z, y[u].w};
#pragma unroll
                for (int q = 0; q < VEC; ++q) a[q] += (double)v[q];   // (beyond the last row: + 0)
            }
        }
        mean = n > 0 ? combine(a) / dn : 0.0;
        __syncthreads();
        if (tid < cols) red[tid] = mean;
        __syncthreads();
#pragma unroll
        for (int q = 0; q < VEC; ++q) mu[q] = red[(tid & (tpr - 1)) * VEC + q];
    }
    double var[VEC] = {}, cov[VEC] = {}, sf[VEC] = {};
    for (int e = g; e < n; e += 4 * G) {
        float4 y[4], f[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            y[u] = row4(Yq, e + u * G);
            f[u] = row4(Yf, e + u * G);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (e + u * G >= n) break;
            const float yv[4] = {y[u].x, y[u].y, y[u].z, y[u].w}, fv[4] = {f[u].x, f[u].y, f[u].z, f[u].w};
#pragma unroll
            for (int q = 0; q < VEC; ++q) {
                // (sum (q - mu) = 0: the cross moment is the centred one whatever is taken off f)
                const double dq = (double)yv[q] - mu[q], df = (double)fv[q] - mu[q];
                var[q] = fma(dq, dq, var[q]);
                cov[q] = fma(dq, df, cov[q]);
                sf[q] += (double)fv[q];
            }
        }
    }
    const double v = combine(var), w = combine(cov), s = combine(sf);
    if (tid >= cols || j >= D) return;
    const size_t e = (size_t)k * D + j;
    if (n == 0) {
        gamma[e] = 1.f;
        beta[e] = 0.f;
        return;
    }
    double vv = v / dn;
    if (vv < 1e-8) vv = 1e-8;
    const double gm = (w / dn) / vv;
    gamma[e] = (float)gm;
    beta[e] = (float)(s / dn - gm * mean);
}

int tpr_for(int units)
{
    int t = 1;
    while (t < units && t < SEG_THREADS) t <<= 1;
    return t;
}

}  // namespace

// Geometry for NE virtual entries over KK keys.
SegGeom seg_geometry(int64_t NE, int D, int KK)
{
    SegGeom g{};
    g.nblk = (int)((NE + SORT_BLOCK - 1) / SORT_BLOCK);
    // About 2048 segments of at least 128 rows; a short list has sixteen-row segments, which spread it over the SMs
    // (the moments of 1024 x 1000 rows take 8 us instead of 35; from 50 000 rows on such segments cost 2 %).
    int64_t sr = (NE + 2047) / 2048;
    if (sr < 128) sr = 128;
    sr = NE <= 8192 ? 16 : (sr + 127) / 128 * 128;
    g.seg_rows = (int)sr;
    g.max_segs = (int)((NE + sr - 1) / sr) + KK;
    (void)D;
    return g;
}

// Room for the segments of any list of up to NE entries (never less for a longer list: a workspace for more rows
// serves fewer).
int seg_capacity(int64_t NE, int KK)
{
    int64_t n = (NE + 15) / 16;
    if (NE > 8192) {
        n = (NE + 127) / 128;
        n = n < 512 ? 512 : (n < 2048 ? n : 2048);
    }
    return (int)n + KK;
}

cudaError_t launch_label_sort(const int32_t *labels, const int32_t *prev, int64_t N, int K, const SegGeom &g,
                              uint32_t *blk_hist, uint32_t *key_total, int64_t *counts, int32_t *cluster_start,
                              int32_t *seg_start, int32_t *order, cudaStream_t s, int32_t *settled)
{
    const int KK = prev ? 2 * K : K;
    launch_pdl(label_hist_kernel, dim3(g.nblk), dim3(SORT_BLOCK), (size_t)KK * sizeof(uint32_t), s, labels, prev, N, K, KK, blk_hist,
               settled);
    launch_pdl(label_scan_blocks_kernel, dim3((KK * 32 + 255) / 256), dim3(256), 0, s, blk_hist, g.nblk, KK, key_total,
               settled);
    // (the scan over the keys -- key offsets, segment table, cluster sizes -- runs inside the scatter
    // kernel: every CTA needs the offsets, CTA 0 publishes the tables)
    const size_t sc_smem = (size_t)KK * sizeof(uint32_t) + (size_t)32 * KK * sizeof(uint16_t);
    if (sc_smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(label_scatter_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)sc_smem);
        if (e != cudaSuccess) return e;
    }
    launch_pdl(label_scatter_kernel, dim3(g.nblk), dim3(SORT_BLOCK), sc_smem, s, labels, prev, N, K, KK, blk_hist, key_total,
               g.seg_rows, prev ? 2 * N : N, prev ? 1 : 0, counts, cluster_start, seg_start, order, settled);
    count_launch(3);
    return cudaGetLastError();
}

template <int MODE>
static cudaError_t launch_segment_sums_mode(const SegParams &p, const SegGeom &g, cudaStream_t s)
{
    const bool vec = (p.D % 4 == 0);
    const int units = vec ? p.D / 4 : p.D;
    // a CTA walks segments blockIdx.x, blockIdx.x + gridDim.x, ...: in delta mode most of the
    // max_segs slots are empty, so the grid stays at a few CTAs per SM
    const unsigned gx = (unsigned)(g.max_segs < 1184 ? g.max_segs : 1184);
    dim3 grid(gx, (unsigned)((units + SEG_THREADS - 1) / SEG_THREADS));
    if (vec)
        launch_pdl(segment_sums_kernel<MODE, 4>, grid, dim3(SEG_THREADS), 0, s, p);
    else
        launch_pdl(segment_sums_kernel<MODE, 1>, grid, dim3(SEG_THREADS), 0, s, p);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_segment_sums(int mode, const float *Yq, const float *Yf, const int32_t *order,
                                const int32_t *cluster_start, const int32_t *seg_start, const double *meanQ,
                                const double *meanF, int D, int K, const SegGeom &g, double *part,
                                cudaStream_t s, const int32_t *settled)
{
    SegParams p{};
    p.Yq = Yq;
    p.Yf = Yf;
    p.order = order;
    p.cluster_start = cluster_start;
    p.seg_start = seg_start;
    p.meanQ = meanQ;
    p.meanF = meanF;
    p.part = part;
    p.D = D;
    p.K = K;
    p.seg_rows = g.seg_rows;
    p.settled = settled;
    const int units = (D % 4 == 0) ? D / 4 : D;
    p.tpr = tpr_for(units);
    switch (mode) {
    case 0: return launch_segment_sums_mode<0>(p, g, s);
    case 1: return launch_segment_sums_mode<1>(p, g, s);
    case 2: return launch_segment_sums_mode<2>(p, g, s);
    default: return launch_segment_sums_mode<3>(p, g, s);
    }
}

cudaError_t launch_segment_combine(const double *part, const int32_t *seg_start, const int64_t *counts, int D,
                                   int K, bool delta, double *out0, double *out1, float *C, cudaStream_t s)
{
    const size_t KD = (size_t)K * D;
    const int threads = 256;
    const unsigned blocks = (unsigned)((KD + threads - 1) / threads);
    segment_combine_kernel<<<blocks, threads, 0, s>>>(part, seg_start, counts, D, K, KD, delta ? 1 : 0, out0, out1, C);
    count_launch();
    return cudaGetLastError();
}

cudaError_t launch_segment_combine3(const double *part, const int32_t *seg_start, int D, int K, int max_segs, double *out0,
                                    double *out1, double *out2, cudaStream_t s)
{
    const CombGeom cg = comb_geometry(D, K, max_segs);
    const int cols = cg.cols;
    const cudaError_t e = launch_pdl(segment_combine3_kernel, dim3((unsigned)K, (unsigned)((D + cols - 1) / cols)), dim3((unsigned)cg.threads), 0, s,
                                     part, seg_start, D, cols, out0, out1, out2);
    count_launch();
    return e;
}

size_t centroid_update_scratch_bytes(int D, int K) { return (size_t)K * ((D + 31) / 32) * sizeof(double2); }

cudaError_t launch_centroid_update(const double *part, const int32_t *seg_start, const int64_t *counts, int D,
                                   int K, int max_segs, double *sums, float *C, float *cnorm, const float *scale, void *Ch,
                                   const float *mean, float *cerr, void *norm_part, uint32_t *arrivals, Control *ctl,
                                   cudaStream_t s, const int32_t *settled)
{
    const CombGeom cg = comb_geometry(D, K, max_segs);
    const int cols = cg.cols;
    const FinishParams f{sums, C, cnorm, scale, reinterpret_cast<__half *>(Ch), mean, cerr, reinterpret_cast<double2 *>(norm_part), arrivals,
                         nullptr, D, cols};
    const cudaError_t e = launch_pdl(centroid_update_kernel, dim3((unsigned)K, (unsigned)((D + cols - 1) / cols)), dim3((unsigned)cg.threads), 0, s,
                                     part, seg_start, counts, K, f, ctl, settled);
    count_launch();
    return e;
}

// 32 columns per CTA, so that 32 rows (8 where rows are not aligned) are in work side by side: a cluster that has all of the
// set's rows takes 64 steps of four rows then, some 0.7 us each.  Few clusters go the general way (6481 x 1000, K = 4: a fit of
// 788 us against 772), and so do shapes of more than 4096 CTAs, whose looking the labels over costs more than the sort.
constexpr int MOM_COLS = 32;
bool closed_form_supported(int64_t N, int D, int K)
{
    return N <= (D % 4 == 0 ? MOM_MAX_ROWS : MOM_MAX_ROWS / 4) && (int64_t)K * ((D + MOM_COLS - 1) / MOM_COLS) <= 4096 &&
           N <= 512 * (int64_t)K;
}

cudaError_t launch_closed_form(const float *Yq, const float *Yf, const int32_t *labels, int64_t N, int D, int K, const double *sumQ,
                               float *gamma, float *beta, cudaStream_t s)
{
    if (!closed_form_supported(N, D, K)) return cudaErrorInvalidValue;
    const int vec = D % 4 == 0 ? 4 : 1;
    const cudaError_t e = launch_pdl(vec == 4 ? cluster_moments_kernel<4> : cluster_moments_kernel<1>,
                                     dim3((unsigned)K, (unsigned)((D + MOM_COLS - 1) / MOM_COLS)), dim3(SEG_THREADS), 0, s, Yq, Yf, labels,
                                     (int)N, D, MOM_COLS, MOM_COLS / vec, sumQ, gamma, beta);
    count_launch();
    return e;
}

// One centroid update from the rows whose label changed, for rounds in which few do.
cudaError_t launch_moved_update(const float *Y, const int32_t *cur, const int32_t *prev, int64_t N, int D, int K, void *list, void *table,
                                void *state, int64_t *counts, double *sums, float *C, float *cnorm, const float *scale, void *Ch,
                                const float *mean, float *cerr, void *norm_part, uint32_t *arrivals, Control *ctl, int32_t *settled,
                                cudaStream_t s)
{
    if (K > MOVE_THREADS) return cudaErrorInvalidValue;
    const int64_t per = ((N + MOVE_GRID - 1) / MOVE_GRID + MOVE_TILE - 1) / MOVE_TILE * MOVE_TILE;
    const unsigned grid = (unsigned)((N + per - 1) / per);
    cudaError_t e = launch_pdl(moved_list_kernel, dim3(grid), dim3(MOVE_THREADS), 0, s, cur, prev, N, K, (int)per,
                               reinterpret_cast<uint32_t *>(list), reinterpret_cast<uint32_t *>(table), reinterpret_cast<unsigned long long *>(state),
                               settled);
    if (e != cudaSuccess) return e;
    // columns per CTA: as many CTAs as there are SMs, no fewer columns than a warp has
    const int vec = D % 4 == 0 ? 4 : 1;
    int cols = 256;
    while (cols > 32 && (int64_t)K * ((D + cols - 1) / cols) < 2 * 148) cols >>= 1;
    while (cols > 32 && cols / 2 >= D) cols >>= 1;
    const FinishParams f{sums, C, cnorm, scale, reinterpret_cast<__half *>(Ch), mean, cerr, reinterpret_cast<double2 *>(norm_part), arrivals,
                         counts, D, cols};
    const dim3 blocks((unsigned)K, (unsigned)((D + cols - 1) / cols));
    e = launch_pdl(vec == 4 ? cluster_move_kernel<4> : cluster_move_kernel<1>, blocks, dim3(SEG_THREADS), 0, s, Y,
                   reinterpret_cast<const uint32_t *>(list), reinterpret_cast<const uint32_t *>(table), (int)grid, (int)per, counts, cols / vec, f,
                   ctl, settled);
    count_launch(2);
    return e;
}

}  // namespace cat
