// Leading eigenpairs of a symmetric positive semi-definite D x D matrix in fp64, for the PCA of
// Section 3.1 (the projection that Algorithm 1 step 1 fits).
//
// Only the p largest of D pairs are wanted (p is 50 of 1000 in the method's setting), so the matrix
// is reduced to tridiagonal form once (Householder reflections, 4/3 D^3 operations) and the pairs
// are taken from the tridiagonal matrix: eigenvalues by bisection on the Sturm sequence, vectors by
// inverse iteration with orthogonalisation against all larger pairs, then the reflections are
// applied to the p vectors.  (Golub & Van Loan, Matrix Computations, ch. 8.)  One-sided Jacobi
// rotations over all pairs of columns, the earlier form, took 155 ms for D = 1000: about ten sweeps
// of 999 dependent launches.  This takes 3.2 ms there with p = 50 (2.5 the reduction, bound by the fp64 latency of its sweeps and one
// exchange between CTAs a step; 0.7 the eigenvectors); with two exchanges a step and branches in the sweep it took 5.1.
//
// Both kernels are cooperative launches; every wait is bounded by TC_TIMEOUT_NS and reports
// CAT_ERR_DEVICE_TIMEOUT in the control block.  Every sum has a fixed order: results do not vary
// from run to run.
#include "cat_internal.cuh"
#include "cat_tc.cuh"

namespace cat {

namespace {

constexpr int ET = 256;              // threads of a CTA
constexpr int EW = ET / 32;
constexpr int MAX_ROWS = 32;         // rows of the matrix per CTA: ceil(CAT_PCA_MAX_D / 128)
constexpr int MAX_VECS = 4;          // vectors per CTA of the second kernel: CAT_PCA_MAX_P over at least 128 CTAs
constexpr size_t DYN_SMEM_LIMIT = 219 * 1024;   // 227 KB less the static arrays

// Values that pass between CTAs without a barrier: each is its own flag.  The buffers start as all ones,
// every word is written once per launch, and a reader polls the word until it is something else -- 64-bit
// accesses are whole, so no fence is needed.
constexpr unsigned long long UNSET = ~0ull;
__device__ __forceinline__ void publish(double *p, double v)
{
    unsigned long long b = (unsigned long long)__double_as_longlong(v);
    if (b == UNSET) b = 0x7FF8000000000000ull;   // (a NaN stays a NaN)
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(b) : "memory");
}
__device__ __forceinline__ unsigned long long peek(const double *p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
// bookkeeping of a poll that found something missing: false when the time limit is over or another CTA has given up
__device__ __forceinline__ bool still_waiting(uint32_t it, uint64_t &t0, Control *ctl)
{
    if ((it & 255u) != 255u) return true;
    if (*(volatile int *)&ctl->device_status != (int)CAT_OK) return false;
    const uint64_t now = global_timer();
    if (t0 == 0) t0 = now;
    else if (now - t0 > TC_TIMEOUT_NS) {
        atomicExch(&ctl->device_status, (int)CAT_ERR_DEVICE_TIMEOUT);
        return false;
    }
    return true;
}
// out[c] = p[k0 + c * ET] for the columns in [lo, D), 0 elsewhere; false when the time limit is over
template <int C>
__device__ __forceinline__ bool collect(const double *p, int lo, int D, double (&out)[C], Control *ctl)
{
    unsigned long long b[C];
    uint64_t t0 = 0;
    for (uint32_t it = 0;; ++it) {
        bool all = true;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const int k = threadIdx.x + c * ET;
            b[c] = k >= lo && k < D ? peek(p + k) : 0ull;
        }
#pragma unroll
        for (int c = 0; c < C; ++c) all = all && b[c] != UNSET;
        if (all) break;
        if (!still_waiting(it, t0, ctl)) return false;
    }
#pragma unroll
    for (int c = 0; c < C; ++c) out[c] = __longlong_as_double((long long)b[c]);
    return true;
}
// The same for one word that every thread reads.
__device__ __forceinline__ bool collect_word(const double *p, double &out, Control *ctl)
{
    uint64_t t0 = 0;
    unsigned long long b;
    for (uint32_t it = 0; (b = peek(p)) == UNSET; ++it)
        if (!still_waiting(it, t0, ctl)) return false;
    out = __longlong_as_double((long long)b);
    return true;
}
// Products prod[k] and row entries next[k] of this thread's columns k > j, 0 elsewhere; edge = {prod[j + 1], prod[j + 2],
// next[j + 2]} (0 beyond the matrix).  Words that have arrived are not asked for again.
template <int C>
__device__ __forceinline__ bool collect_step(const double *prod, const double *next, int j, int D, double (&wp)[C], double (&a)[C],
                                             double (&edge)[3], Control *ctl)
{
    unsigned long long b[2 * C + 3];
    const int j2 = j + 2 < D ? j + 2 : j + 1;
#pragma unroll
    for (int i = 0; i < 2 * C + 3; ++i) b[i] = UNSET;
    uint64_t t0 = 0;
    for (uint32_t it = 0;; ++it) {
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const int k = threadIdx.x + c * ET;
            const bool in = k > j && k < D;
            if (b[c] == UNSET) b[c] = in ? peek(prod + k) : 0ull;
            if (b[C + c] == UNSET) b[C + c] = in ? peek(next + k) : 0ull;
        }
        if (b[2 * C] == UNSET) b[2 * C] = peek(prod + j + 1);
        if (b[2 * C + 1] == UNSET) b[2 * C + 1] = peek(prod + j2);
        if (b[2 * C + 2] == UNSET) b[2 * C + 2] = peek(next + j2);
        bool all = true;
#pragma unroll
        for (int i = 0; i < 2 * C + 3; ++i) all = all && b[i] != UNSET;
        if (all) break;
        if (!still_waiting(it, t0, ctl)) return false;
    }
#pragma unroll
    for (int c = 0; c < C; ++c) {
        wp[c] = __longlong_as_double((long long)b[c]);
        a[c] = __longlong_as_double((long long)b[C + c]);
    }
    edge[0] = __longlong_as_double((long long)b[2 * C]);
    edge[1] = j + 2 < D ? __longlong_as_double((long long)b[2 * C + 1]) : 0.0;
    edge[2] = j + 2 < D ? __longlong_as_double((long long)b[2 * C + 2]) : 0.0;
    return true;
}

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ double tree8(const double *r)
{
    static_assert(EW == 8, "sum of the warps' parts");
    return ((r[0] + r[1]) + (r[2] + r[3])) + ((r[4] + r[5]) + (r[6] + r[7]));
}

// every thread gets the CTA's sum; `red` must not be in use from an earlier call (callers alternate two)
__device__ __forceinline__ double block_sum(double v, double *red)
{
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    return tree8(red);
}
// the same; `ok` becomes false in every thread if it was in one
__device__ __forceinline__ double block_sum(double v, double *red, bool &ok)
{
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    ok = __syncthreads_and(ok);
    return tree8(red);
}

// Sums of 8 values over the warp: each exchange halves how many values a lane still carries, 9
// exchanges in place of 40.  Lanes 4 i ... 4 i + 3 end with the sum of acc[i].
__device__ __forceinline__ double warp_sum8(double (&acc)[8], int lane)
{
#pragma unroll
    for (int h = 4, o = 16; h > 0; h >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (i < h) {
                const double send = up ? acc[i] : acc[i + h];
                const double keep = up ? acc[i + h] : acc[i];
                acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
    }
    double s = acc[0];
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    return s;
}

// Sums of 4 values over the warp; lanes 8 i ... 8 i + 7 end with the sum of acc[i].
__device__ __forceinline__ double warp_sum4(double (&acc)[4], int lane)
{
#pragma unroll
    for (int h = 2, o = 16; h > 0; h >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < 2; ++i)
            if (i < h) {
                const double send = up ? acc[i] : acc[i + h];
                const double keep = up ? acc[i + h] : acc[i];
                acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
    }
    double s = acc[0];
    s += __shfl_xor_sync(0xffffffffu, s, 4);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    return s;
}

// power of two that brings the largest diagonal entry (the largest entry of a semi-definite matrix)
// into [1, 2), so that squares of entries neither overflow nor vanish
__device__ double diagonal_scale(const double *diag, int D, double *red)
{
    double m = 0.0;
    for (int k = threadIdx.x; k < D; k += ET) m = fmax(m, diag[k]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < EW; ++w) m = fmax(m, red[w]);
    __syncthreads();
    if (!(m > 0.0) || !isfinite(m)) return 1.0;
    int e = ilogb(m);
    e = e < -1000 ? -1000 : e;
    return scalbn(1.0, -e);
}

struct TridiagParams {
    double *A;            // [D][D] symmetric, full
    const double *diag;   // [D] its diagonal
    double *refl;         // [D][D] reflection j: entries k > j of row j
    double *d, *e, *tau;  // [D]
    double *prod;         // [D][D] row j: products of step j; all ones at launch
    double *next;         // [D][D] row j: row j of the matrix after update j - 2; all ones at launch
    Control *ctl;
    int D;
    int resident;         // (rows not in registers) the CTA's rows live in shared memory
};

// Householder reduction to tridiagonal form, D <= 1024.  A row of the matrix belongs to one CTA and stays in its
// registers: rows 8 me ... 8 me + 7, column k with thread k mod 256 (8 MB over 125 SMs at D = 1000); a CTA's
// products are one 64-byte store and it leaves when its rows are done.  Step j: every CTA has row j (which its owner
// has published up to update j - 2) up to date, so it knows reflection j, applies update j - 1 to its own rows and in
// the same sweep multiplies them with the reflection; it publishes its products and collects everybody's, and row
// j + 1 with them, word by word, without a barrier.
//   A reflection is H = I - tau u u' with u = x - off e_1 as it stands (tau = 2 / u'u): its division passes during the sweep.
//   The sums of a step -- u'Au for the update, the squares of the next row for the next reflection -- are taken together,
//   before the first of them is known: with w0 = tau A u, h = tau u'w0 / 2, the next row is x = y + 2 h u_1 u where
//   y = a - u_1 w0 - w0_1 u needs no sum, so |x|^2 = |y|^2 + 4 h u_1 y'u + 4 h^2 u_1^2 u'u.  Where these cancel by more than
//   16, the squares are added up in a second exchange.  (u'u is added up with the others: carried over from the step before,
//   as |x|^2 less one entry, its error would grow by up to 16 a step.)  The mean of the diagonal is taken off the matrix and put back
//   on the tridiagonal one, which makes h smaller: without it nearly every step of a covariance would cancel, with it those whose spectrum
//   is far from one value still do in most steps (a second summation stays within the CTA).
//   bound: latency.  A step moves 2 D values between CTAs and does 6 (D - j)^2 / G operations per CTA.
template <int C>
__global__ void __launch_bounds__(ET) tridiag_regs_kernel(TridiagParams P)
{
    __shared__ double red0[EW], red[4][EW], red_x[EW], red_rows[EW][8], s_prod[8], su[2][C * ET];
    const int D = P.D, me = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int i0 = me * 8, R = D - i0 < 8 ? D - i0 : 8;   // own rows: i0 ... i0 + R - 1
    const double scale = diagonal_scale(P.diag, D, red0);
    double mu = 0.0;
    for (int k = tid; k < D; k += ET) mu += P.diag[k] * scale;
    mu = block_sum(mu, red_x) / (double)D;
    if (!isfinite(mu)) mu = 0.0;
    double ar[8][C];
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const int i = i0 + r, k = tid + c * ET;
            ar[r][c] = i < D && k < D ? fma(P.A[(size_t)i * D + k], scale, i == k ? -mu : 0.0) : 0.0;
            if (i == 0 && k < D) publish(P.next + k, ar[r][c]);
        }
    for (int k = tid; k < 2 * C * ET; k += ET) (&su[0][0])[k] = 0.0;
    if (tid < 8) s_prod[tid] = 0.0;

    double x[C], uo[C], wo[C], one[1], ss = 0.0, x1, tau = 0.0, h = 0.0;
#pragma unroll
    for (int c = 0; c < C; ++c) uo[c] = wo[c] = 0.0;
    bool ok = collect<C>(P.next, 0, D, x, P.ctl);
    ok = collect_word(P.next + (D > 1 ? 1 : 0), one[0], P.ctl) && ok;
    x1 = one[0];
#pragma unroll
    for (int c = 0; c < C; ++c)
        if (tid + c * ET > 1) ss = fma(x[c], x[c], ss);
    __syncthreads();
    ss = block_sum(ss, red0, ok);
    if (!ok) return;

    for (int j = 0;; ++j) {
        // the CTA of row j + 1 (or the last one) records step j
        const bool lead = me == (j + 1 < D ? j + 1 : j) / 8;
        if (lead)
#pragma unroll
            for (int c = 0; c < C; ++c)
                if (tid + c * ET == j) P.d[j] = x[c] + mu;
        if (j == D - 1 || i0 + R <= j + 1) break;
        const double *u_old = su[(j & 1) ^ 1];
        double *u_new = su[j & 1];
        // (a row whose squares have vanished is as good as reduced: what is dropped is below 1e-125 of the matrix)
        const bool reflect = ss > 1e-250;
        const double tt = fma(x1, x1, ss), nrm = sqrt(tt);
        const double off = reflect ? (x1 >= 0.0 ? -nrm : nrm) : x1;
        const double u1 = reflect ? x1 - off : 0.0;
        double un[C];
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const int k = tid + c * ET;
            un[c] = k == j + 1 ? u1 : (reflect && k > j + 1 ? x[c] : 0.0);
            u_new[k] = un[c];
            if (lead && k > j && k < D) P.refl[(size_t)j * D + k] = un[c];
        }
        // update j - 1 of the own rows and their products with the new reflection
        // (rows that are done with go along: a branch per row would leave one row's chain of dependent operations after the
        // other, 1750 cycles of a step's 5900 where the eight together take a third of that)
        double acc[8], ui[8], wi[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            acc[r] = 0.0;
            ui[r] = -u_old[i0 + r];
            wi[r] = -fma(h, ui[r], tau * s_prod[r]);
        }
#pragma unroll
        for (int c = 0; c < C; ++c)
            if (warp * 32 + 31 + c * ET > j) {   // (columns up to j are done with)
#pragma unroll
                for (int r = 0; r < 8; ++r) ar[r][c] = fma(wi[r], uo[c], fma(ui[r], wo[c], ar[r][c]));
#pragma unroll
                for (int r = 0; r < 8; ++r) acc[r] = fma(ar[r][c], un[c], acc[r]);
            }
#pragma unroll
        for (int r = 0; r < 8; ++r)
            if (i0 + r == j + 1) {
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    const int k = tid + c * ET;
                    if (k > j && k < D) publish(P.next + (size_t)(j + 1) * D + k, ar[r][c]);
                }
            }
        const double s = warp_sum8(acc, lane);
        if ((lane & 3) == 0) red_rows[warp][lane >> 2] = s;
        tau = reflect ? 1.0 / fma(fabs(x1), nrm, tt) : 0.0;
        if (lead && tid == 0) {
            P.e[j] = off;
            P.tau[j] = tau;
        }
        __syncthreads();
        if (tid < R && i0 + tid > j) {
            double part[EW];
#pragma unroll
            for (int w = 0; w < EW; ++w) part[w] = red_rows[w][tid];
            const double prod = tree8(part);
            publish(P.prod + (size_t)j * D + i0 + tid, prod);
            s_prod[tid] = prod;
        }
        // the products, row j + 1, and of both the words that every thread needs
        double a[C], edge[3];
        ok = collect_step<C>(P.prod + (size_t)j * D, P.next + (size_t)(j + 1) * D, j, D, wo, a, edge, P.ctl);
        const double u2 = u_new[j + 2 < D ? j + 2 : 0], w01 = tau * edge[0];
        double sums[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const int k = tid + c * ET;
            wo[c] *= tau;
            sums[0] = fma(wo[c], un[c], sums[0]);
            if (k > j + 2) {
                const double y = fma(-u1, wo[c], fma(-w01, un[c], a[c]));
                sums[1] = fma(y, y, sums[1]);
                sums[2] = fma(y, un[c], sums[2]);
                sums[3] = fma(un[c], un[c], sums[3]);
            }
        }
        {
            const double v = warp_sum4(sums, lane);
            if ((lane & 7) == 0) red[lane >> 3][warp] = v;
        }
        ok = __syncthreads_and(ok);
        if (!ok) break;
        h = 0.5 * tau * tree8(red[0]);
        const double y2 = tree8(red[1]), yu = tree8(red[2]), q = 2.0 * h * u1;
        const double uu = q * q * tree8(red[3]);
        const double w1 = fma(-h, u1, w01), w2 = fma(-h, u2, tau * edge[1]);
        x1 = fma(-u1, w2, fma(-w1, u2, edge[2]));
#pragma unroll
        for (int c = 0; c < C; ++c) {
            uo[c] = un[c];
            wo[c] = fma(-h, un[c], wo[c]);
            x[c] = fma(-u1, wo[c], fma(-w1, un[c], a[c]));
        }
        ss = fma(2.0 * q, yu, y2 + uu);
        if (!(ss > 0.0625 * fmax(y2, uu))) {   // (the same numbers in every thread)
            ss = 0.0;
#pragma unroll
            for (int c = 0; c < C; ++c)
                if (tid + c * ET > j + 2) ss = fma(x[c], x[c], ss);
            ss = block_sum(ss, red_x);
        }
    }
}

// The same for rows that registers do not hold: a CTA's rows (me, me + G, ...) lie in shared or global memory; there
// the work per step counts, and the two sums of a step are taken one after the other.
//   H = I - tau v v' with v_1 = 1.
template <int C>
__global__ void __launch_bounds__(ET) tridiag_kernel(TridiagParams P)
{
    extern __shared__ double sm[];
    __shared__ double red[2][EW], red_rows[EW][MAX_ROWS];
    // Each is written before a step's barrier and read behind it, and written again only behind another barrier of
    // the step: s_x1 around the sum of squares, s_w1 around v'Av.  (One word for both would be written by a warp that
    // is a step ahead while another has yet to read it.)
    __shared__ double s_x1, s_w1;
    const int D = P.D, G = gridDim.x, me = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int R = (D - me + G - 1) / G;   // own rows: me + r G
    double *sv = sm, *sw = sm + D, *rows = sm + 2 * D;
    const double scale = diagonal_scale(P.diag, D, red[0]);
    for (int k = tid; k < 2 * D; k += ET) sm[k] = 0.0;
    for (int r = 0; r < R; ++r) {
        double *src = P.A + (size_t)(me + r * G) * D;
        double *dst = P.resident ? rows + (size_t)r * D : src;
        for (int k = tid; k < D; k += ET) {
            const double a = src[k] * scale;
            dst[k] = a;
            if (me + r * G == 0) publish(P.next + k, a);
        }
    }
    double vo[C], wo[C];
#pragma unroll
    for (int c = 0; c < C; ++c) vo[c] = wo[c] = 0.0;
    double v1 = 0.0, w1 = 0.0;   // the previous update's v, w at index j
    __syncthreads();

    for (int j = 0; j < D; ++j) {
        const bool lead = me == j % G;   // records step j
        // row j after update j - 1, and the sum of squares behind its first off-diagonal entry
        double x[C];
        bool ok = collect<C>(P.next + (size_t)j * D, j, D, x, P.ctl);
        double ss = 0.0;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const int k = tid + c * ET;
            x[c] = fma(-v1, wo[c], fma(-w1, vo[c], x[c]));   // (v, w are zero up to index j - 1)
            if (k == j && lead) P.d[j] = x[c];
            if (k == j + 1) s_x1 = x[c];
            if (k > j + 1) ss = fma(x[c], x[c], ss);
        }
        ss = block_sum(ss, red[0], ok);
        if (!ok || j == D - 1) break;
        const double x1 = s_x1;
        double tau = 0.0, inv = 0.0, off = x1;
        if (ss > 0.0) {
            const double nrm = sqrt(fma(x1, x1, ss));
            off = x1 >= 0.0 ? -nrm : nrm;
            tau = (off - x1) / off;
            inv = 1.0 / (x1 - off);
        }
        double vn[C];
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const int k = tid + c * ET;
            vn[c] = k == j + 1 ? (ss > 0.0 ? 1.0 : 0.0) : (k > j + 1 ? x[c] * inv : 0.0);
            if (lead && k > j && k < D) P.refl[(size_t)j * D + k] = vn[c];
        }
        if (lead && tid == 0) {
            P.e[j] = off;
            P.tau[j] = tau;
        }
        // update j - 1 of the own rows and their products with the new reflection
        const int r_first = j + 1 <= me ? 0 : (j + 1 - me + G - 1) / G;   // first own row with index > j
        for (int r0 = r_first; r0 < R; r0 += 8) {
            double acc[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                acc[u] = 0.0;
                const int r = r0 + u, i = me + r * G;
                if (r < R) {
                    double *a_row = P.resident ? rows + (size_t)r * D : P.A + (size_t)i * D;
                    const double vi = -sv[i], wi = -sw[i];
#pragma unroll
                    for (int c = 0; c < C; ++c) {
                        const int k = tid + c * ET;
                        if (k > j && k < D) {
                            const double a = fma(wi, vo[c], fma(vi, wo[c], a_row[k]));
                            a_row[k] = a;
                            acc[u] = fma(a, vn[c], acc[u]);
                            if (i == j + 1) publish(P.next + (size_t)(j + 1) * D + k, a);
                        }
                    }
                }
            }
            const double s = warp_sum8(acc, lane);
            if ((lane & 3) == 0 && r0 + (lane >> 2) < R) red_rows[warp][r0 + (lane >> 2)] = s;
        }
        __syncthreads();
        if (tid >= r_first && tid < R) {
            double part[EW];
#pragma unroll
            for (int w = 0; w < EW; ++w) part[w] = red_rows[w][tid];
            publish(P.prod + (size_t)j * D + me + tid * G, tree8(part));
        }
        // w = tau A v - (tau / 2)(tau v'Av) v
        ok = collect<C>(P.prod + (size_t)j * D, j + 1, D, wo, P.ctl);
        double pv = 0.0;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            wo[c] *= tau;
            pv = fma(wo[c], vn[c], pv);
            if (tid + c * ET == j + 1) s_w1 = wo[c];
        }
        const double half = 0.5 * tau * block_sum(pv, red[1], ok);
        if (!ok) break;
        v1 = ss > 0.0 ? 1.0 : 0.0;
        w1 = s_w1 - half * v1;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const int k = tid + c * ET;
            vo[c] = vn[c];
            wo[c] -= half * vn[c];
            if (k < D) {
                sv[k] = vo[c];
                sw[k] = wo[c];
            }
        }
    }
}

struct EigvecParams {
    const double *diag;               // [D] diagonal of the unreduced matrix (for its scale)
    const double *d, *e, *refl;
    const double *wy;                 // blocks of reflections: see refl_block_kernel
    double *Z;                        // [p][D] vectors
    double *words;                    // [4][p][D] the vectors that leave each orthogonalisation; all ones at launch
    float *comps;                     // [p][D] out
    double *eig_out;                  // [p] out or null
    Control *ctl;
    int D, p;
};

// Eigenvalues of the tridiagonal matrix below each of two points: sign changes of the leading minors p_i = (d_i - x) p_{i-1} -
// e_{i-1}^2 p_{i-2} (Givens' form of the Sturm sequence; the products' rounding amounts to relative changes of d - x and
// e^2 by a few units, as in the form with quotients, and a step is one dependent operation where a division was some
// twenty).  Every eight steps the pair is scaled by a power of two: entries are below 2^14 and above 2^-65 of the norm, so that
// eight steps stay within fp64's range.  de[i] = {d_i, e_{i-1}^2}; two points keep the fp64 pipe and its latency in balance.
__device__ __forceinline__ void count_below(const double2 *de, int D, const double (&x)[2], int (&n)[2])
{
    double p0[2], p1[2];
    const double d0 = de[0].x;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        p0[q] = 1.0;
        p1[q] = d0 - x[q];
        n[q] = (int)((unsigned)__double2hiint(p1[q]) >> 31);
    }
    auto step = [&](double2 v) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const double t = fma(v.x - x[q], p1[q], -(v.y * p0[q]));
            n[q] += (int)((unsigned)(__double2hiint(t) ^ __double2hiint(p1[q])) >> 31);
            p0[q] = p1[q];
            p1[q] = t;
        }
    };
    int i = 1;
    for (; i + 8 <= D; i += 8) {
        double2 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = de[i + u];
#pragma unroll
        for (int u = 0; u < 8; ++u) step(v[u]);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int ea = __double2hiint(p0[q]) & 0x7FF00000, eb = __double2hiint(p1[q]) & 0x7FF00000;
            const double f = __hiloint2double(0x7FE00000 - (ea > eb ? ea : eb), 0);
            p0[q] *= f;
            p1[q] *= f;
        }
    }
    for (; i < D; ++i) step(de[i]);
}

// Reflections are applied RB at a time: H_j H_{j+1} ... H_{j+RB-1} z = z - U' (M (U z)), rows of U the vectors u, M upper
// triangular from their products with one another (the compact form of Schreiber and Van Loan).  M_kk = tau_k,
// M_ik = -tau_i sum_{i < l <= k} (u_i . u_l) M_lk.  A CTA per block.
template <int RB>
__global__ void __launch_bounds__(ET) refl_block_kernel(const double *__restrict__ refl, const double *__restrict__ tau, int D,
                                                        double *__restrict__ wy)
{
    __shared__ double g[RB][RB], m[RB][RB];
    const int j0 = blockIdx.x * RB, nref = D - 2, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int e = warp; e < RB * RB; e += EW) {
        const int i = e / RB, l = e % RB;
        if (i >= l || j0 + l >= nref) continue;
        const double *a = refl + (size_t)(j0 + i) * D, *b = refl + (size_t)(j0 + l) * D;
        double s = 0.0;
#pragma unroll 8
        for (int k = j0 + l + 1 + lane; k < D; k += 32) s = fma(a[k], b[k], s);
        s = warp_sum(s);
        if (lane == 0) g[i][l] = s;
    }
    __syncthreads();
    const int k = threadIdx.x;
    if (k < RB) {
        for (int i = RB - 1; i >= 0; --i) {
            double v = 0.0;
            if (j0 + k < nref && i <= k) {
                const double t = tau[j0 + i];
                v = t;
                if (i < k) {
                    double s = 0.0;
                    for (int l = i + 1; l <= k; ++l) s = fma(g[i][l], m[l][k], s);
                    v = -t * s;
                }
            }
            m[i][k] = v;
            wy[(size_t)blockIdx.x * RB * RB + i * RB + k] = v;
        }
    }
}

// The p largest eigenpairs.  CTA b has the vectors b, b + G, ...; all of them go through
//   bisection      512 points of the interval at a time, 9 bits of the eigenvalue per pass over the matrix
//   solve          (T - lambda) z = z by Gaussian elimination with partial pivoting (one thread:
//                  a chain of D dependent steps; the vectors run beside each other)
//   orthogonalise  modified Gram-Schmidt in order of decreasing eigenvalue: a CTA takes each earlier vector out of its
//                  own as it arrives, word by word.  Clustered or equal eigenvalues get different starts, so their vectors
//                  span the eigenspace.
//   back           the reflections in reverse order, RB at a time, then sign, fp32 store
// Three rounds of solve and orthogonalise, the last one orthogonalised twice.  Every pass leaves its vectors in words of
// its own, so no pass waits for the one before it: the first vectors are a round ahead of the last ones.
//   bound: latency of the serial chains.
template <int C, int RB>
__global__ void __launch_bounds__(ET) eigvec_kernel(EigvecParams P)
{
    extern __shared__ __align__(16) double sm[];
    __shared__ double red[2][EW], lam[MAX_VECS], red_b[EW][RB], s_blk[RB];
    __shared__ int s_idx[EW];
    const int D = P.D, p = P.p, G = gridDim.x, me = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int NV = (p - me + G - 1) / G;
    double *sd = sm, *u0 = sm + D, *u1 = sm + 2 * D, *u2 = sm + 3 * D, *l = sm + 4 * D;
    unsigned char *swapped = reinterpret_cast<unsigned char *>(sm + 5 * D);
    const double scale = diagonal_scale(P.diag, D, red[0]);
    int par = 0;

    // ---- bisection between the Gershgorin bounds
    double2 *de = reinterpret_cast<double2 *>(sm);
    double lo0 = INFINITY, hi0 = -INFINITY;
    for (int k = tid; k < D; k += ET) {
        const double el = k > 0 ? fabs(P.e[k - 1]) : 0.0, er = k + 1 < D ? fabs(P.e[k]) : 0.0;
        lo0 = fmin(lo0, P.d[k] - el - er);
        hi0 = fmax(hi0, P.d[k] + el + er);
    }
    double b2[2] = {-lo0, hi0};
#pragma unroll
    for (int q = 0; q < 2; ++q) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) b2[q] = fmax(b2[q], __shfl_xor_sync(0xffffffffu, b2[q], o));
        __syncthreads();
        if (lane == 0) red[0][warp] = b2[q];
        __syncthreads();
        for (int w = 0; w < EW; ++w) b2[q] = fmax(b2[q], red[0][w]);
    }
    const double tnorm = fmax(fmax(fabs(b2[0]), fabs(b2[1])), 1e-290);
    const double margin = 4.0 * (double)D * 2.3e-16 * tnorm;
    const double e_min = tnorm * 2.7e-20;   // (2^-65: far below what the reduction has rounded off)
    for (int k = tid; k < D; k += ET) {
        const double el = k > 0 ? fmax(fabs(P.e[k - 1]), e_min) : 0.0;
        de[k] = make_double2(P.d[k], el * el);
    }
    __syncthreads();
    for (int q = 0; q < NV; ++q) {
        const int want = D - 1 - (me + q * G);   // index of the eigenvalue in ascending order
        double lo = -b2[0] - margin, hi = b2[1] + margin;
        for (int pass = 0; pass < 8 && hi - lo > 2.3e-16 * tnorm; ++pass) {
            const double step = (hi - lo) / (double)(2 * ET + 1);
            const double x[2] = {lo + step * (double)(2 * tid + 1), lo + step * (double)(2 * tid + 2)};
            int n[2];
            count_below(de, D, x, n);
            const int below = __syncthreads_count(n[0] <= want) + __syncthreads_count(n[1] <= want);
            const double nlo = below > 0 ? lo + step * (double)below : lo;
            const double nhi = below < 2 * ET ? lo + step * (double)(below + 1) : hi;
            if (!(nhi - nlo < hi - lo)) break;
            lo = nlo;
            hi = nhi;
        }
        if (tid == 0) lam[q] = 0.5 * (lo + hi);
    }

    // ---- inverse iteration
    const double tiny = 2.3e-16 * tnorm;
    for (int round = 0; round < 3; ++round) {
        for (int q = 0; q < NV; ++q) {
            const int m = me + q * G;
            __syncthreads();
            // (a CTA with one vector keeps its factors over the rounds)
            const bool factor = round == 0 || NV > 1;
            if (factor) {
                for (int k = tid; k < D; k += ET) sd[k] = P.d[k];
                for (int k = tid; k + 1 < D; k += ET) l[k] = P.e[k];
            }
            __syncthreads();
            if (factor && tid == 0) {
                // P L U = T - lambda: u0 (inverted), u1, u2 the rows of U; l overwrites the off-diagonal.  (What a
                // block of steps reads is read before its first step: the stores in between would hold it up.)
                const double lm = lam[q];
                double a = sd[0] - lm, b = D > 1 ? l[0] : 0.0;
                auto eliminate = [&](int i, double sub, double dg, double sup) {
                    const bool keep = fabs(a) >= fabs(sub);
                    double pv = keep ? a : sub;
                    if (fabs(pv) < tiny) pv = pv < 0.0 ? -tiny : tiny;
                    const double r = 1.0 / pv, f = (keep ? sub : a) * r;
                    u0[i] = r;
                    u1[i] = keep ? b : dg;
                    u2[i] = keep ? 0.0 : sup;
                    l[i] = f;
                    swapped[i] = keep ? 0 : 1;
                    a = keep ? fma(-f, b, dg) : fma(-f, dg, b);
                    b = keep ? sup : -f * sup;
                };
                int i = 0;
                for (; i + 9 < D; i += 8) {
                    double sub[9], dg[8];
#pragma unroll
                    for (int u = 0; u < 9; ++u) sub[u] = l[i + u];
#pragma unroll
                    for (int u = 0; u < 8; ++u) dg[u] = sd[i + 1 + u] - lm;
#pragma unroll
                    for (int u = 0; u < 8; ++u) eliminate(i + u, sub[u], dg[u], sub[u + 1]);
                }
                for (; i + 1 < D; ++i) eliminate(i, l[i], sd[i + 1] - lm, i + 2 < D ? l[i + 1] : 0.0);
                if (fabs(a) < tiny) a = a < 0.0 ? -tiny : tiny;
                u0[D - 1] = 1.0 / a;
            }
            __syncthreads();
            double *x = sd, *z = P.Z + (size_t)m * D;
            for (int k = tid; k < D; k += ET) {
                double v = 0.0;
                if (round == 0) {
                    uint32_t h = (uint32_t)m * 0x9E3779B9u + (uint32_t)k * 0x85EBCA6Bu + 1u;   // a different start for each vector (Wellons' lowbias32 mixer)
                    h ^= h >> 16;
                    h *= 0x7FEB352Du;
                    h ^= h >> 15;
                    h *= 0x846CA68Bu;
                    h ^= h >> 16;
                    v = ((double)h + 0.5) * (1.0 / 2147483648.0) - 1.0;
                } else
                    v = z[k];
                x[k] = v;
            }
            __syncthreads();
            if (tid == 0) {
                double cur = x[0];
                auto forward = [&](int i, double nx, double f, bool sw) {
                    x[i] = sw ? nx : cur;
                    cur = fma(-f, sw ? nx : cur, sw ? cur : nx);
                };
                int i = 0;
                for (; i + 8 < D; i += 8) {
                    double nx[8], f[8];
                    bool sw[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        nx[u] = x[i + 1 + u];
                        f[u] = l[i + u];
                        sw[u] = swapped[i + u];
                    }
#pragma unroll
                    for (int u = 0; u < 8; ++u) forward(i + u, nx[u], f[u], sw[u]);
                }
                for (; i + 1 < D; ++i) forward(i, x[i + 1], l[i], swapped[i]);
                double z1 = cur * u0[D - 1], z2 = 0.0;
                x[D - 1] = z1;
                auto backward = [&](int at, double xv, double r, double c1, double c2) {
                    const double t = fma(-c1, z1, fma(-c2, z2, xv)) * r;
                    x[at] = t;
                    z2 = z1;
                    z1 = t;
                };
                i = D - 2;
                for (; i >= 7; i -= 8) {
                    double xv[8], r[8], c1[8], c2[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        xv[u] = x[i - u];
                        r[u] = u0[i - u];
                        c1[u] = u1[i - u];
                        c2[u] = u2[i - u];
                    }
#pragma unroll
                    for (int u = 0; u < 8; ++u) backward(i - u, xv[u], r[u], c1[u], c2[u]);
                }
                for (; i >= 0; --i) backward(i, x[i], u0[i], u1[i], u2[i]);
            }
            __syncthreads();
            double ss = 0.0;
            for (int k = tid; k < D; k += ET) ss = fma(x[k], x[k], ss);
            ss = block_sum(ss, red[par ^= 1]);
            const double inv = ss > 0.0 && isfinite(ss) ? 1.0 / sqrt(ss) : 0.0;
            for (int k = tid; k < D; k += ET) z[k] = inv > 0.0 ? x[k] * inv : (k == m ? 1.0 : 0.0);
        }
        // Gram-Schmidt passes
        for (int pass = 0; pass < (round == 2 ? 2 : 1); ++pass) {
            double *words = P.words + (size_t)(round + pass) * p * D;
            double z[MAX_VECS][C];
#pragma unroll
            for (int q = 0; q < MAX_VECS; ++q)
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    const int k = tid + c * ET;
                    z[q][c] = q < NV && k < D ? P.Z[(size_t)(me + q * G) * D + k] : 0.0;
                }
            const int last = me + (NV - 1) * G;
            unsigned long long ahead[C];   // the next vector's words, if they are there already
#pragma unroll
            for (int c = 0; c < C; ++c) ahead[c] = UNSET;
            for (int i = 0; i <= last; ++i) {
                if (i % G == me) {
                    double ss = 0.0;
#pragma unroll
                    for (int q = 0; q < MAX_VECS; ++q)
                        if (me + q * G == i)
#pragma unroll
                            for (int c = 0; c < C; ++c) ss = fma(z[q][c], z[q][c], ss);
                    ss = block_sum(ss, red[par ^= 1]);
                    const double inv = ss > 0.0 ? 1.0 / sqrt(ss) : 0.0;
#pragma unroll
                    for (int q = 0; q < MAX_VECS; ++q)
                        if (me + q * G == i)
#pragma unroll
                            for (int c = 0; c < C; ++c) {
                                const int k = tid + c * ET;
                                z[q][c] *= inv;
                                if (k < D) {
                                    publish(words + (size_t)i * D + k, z[q][c]);
                                    P.Z[(size_t)i * D + k] = z[q][c];
                                }
                            }
                }
                if (i == last) break;
                bool there = true, ok = true;
#pragma unroll
                for (int c = 0; c < C; ++c) there = there && ahead[c] != UNSET;
                double zi[C], dot[MAX_VECS];
#pragma unroll
                for (int c = 0; c < C; ++c) zi[c] = __longlong_as_double((long long)ahead[c]);
                if (!there) ok = collect<C>(words + (size_t)i * D, 0, D, zi, P.ctl);
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    const int k = tid + c * ET;
                    ahead[c] = k < D ? (i + 1 < last ? peek(words + (size_t)(i + 1) * D + k) : UNSET) : 0ull;
                }
#pragma unroll
                for (int q = 0; q < MAX_VECS; ++q) {
                    if (q >= NV || me + q * G <= i) continue;
                    dot[q] = 0.0;
#pragma unroll
                    for (int c = 0; c < C; ++c) dot[q] = fma(zi[c], z[q][c], dot[q]);
                    dot[q] = block_sum(dot[q], red[par ^= 1], ok);
                    if (!ok) return;   // (the same in every thread)
#pragma unroll
                    for (int c = 0; c < C; ++c) z[q][c] = fma(-dot[q], zi[c], z[q][c]);
                }
            }
        }
    }

    // ---- back transformation: z <- H_0 H_1 ... H_{D-3} z, then sign and store
    const int nref = D - 2, nblk = D > 2 ? (nref + RB - 1) / RB : 0;
    for (int q = 0; q < NV; ++q) {
        const int m = me + q * G;
        double z[C], u[RB][C], mm;
        __syncthreads();
        auto fetch = [&](int blk, double (&v)[RB][C], double &w) {
#pragma unroll
            for (int i = 0; i < RB; ++i)
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    const int j = blk * RB + i, k = tid + c * ET;
                    v[i][c] = blk >= 0 && j < nref && k > j && k < D ? P.refl[(size_t)j * D + k] : 0.0;
                }
            w = blk >= 0 && warp < RB ? P.wy[((size_t)blk * RB + warp) * RB + (lane & (RB - 1))] : 0.0;
        };
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const int k = tid + c * ET;
            z[c] = k < D ? P.Z[(size_t)m * D + k] : 0.0;
        }
        fetch(nblk - 1, u, mm);
        for (int blk = nblk - 1; blk >= 0; --blk) {
            double un[RB][C], mn, acc[RB];
            fetch(blk - 1, un, mn);
#pragma unroll
            for (int i = 0; i < RB; ++i) {
                acc[i] = 0.0;
#pragma unroll
                for (int c = 0; c < C; ++c) acc[i] = fma(u[i][c], z[c], acc[i]);
            }
            if constexpr (RB == 8) {
                const double s = warp_sum8(acc, lane);
                if ((lane & 3) == 0) red_b[warp][lane >> 2] = s;
            } else {
#pragma unroll
                for (int i = 0; i < RB; ++i) {
                    const double s = warp_sum(acc[i]);
                    if (lane == 0) red_b[warp][i] = s;
                }
            }
            __syncthreads();
            if (warp < RB) {
                // a warp per entry of M (U z)
                double t = 0.0;
                for (int w = lane / RB; w < EW; w += 32 / RB) t += red_b[w][lane & (RB - 1)];
#pragma unroll
                for (int o = RB; o < 32; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
                t *= mm;
#pragma unroll
                for (int o = RB >> 1; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
                if (lane == 0) s_blk[warp] = t;
            }
            __syncthreads();
            // (in pairs, then a tree: dependent additions are what a block's time is made of)
#pragma unroll
            for (int c = 0; c < C; ++c) {
                double part[RB / 2];
#pragma unroll
                for (int i = 0; i < RB / 2; ++i) part[i] = fma(s_blk[2 * i], u[2 * i][c], s_blk[2 * i + 1] * u[2 * i + 1][c]);
#pragma unroll
                for (int o = RB / 4; o > 0; o >>= 1)
#pragma unroll
                    for (int i = 0; i < o; ++i) part[i] += part[i + o];
                z[c] -= part[0];
            }
#pragma unroll
            for (int i = 0; i < RB; ++i)
#pragma unroll
                for (int c = 0; c < C; ++c) u[i][c] = un[i][c];
            mm = mn;
        }
        // the entry of largest magnitude (lowest index among equals) is made positive
        double best = -1.0, val = 0.0;
        int bi = D;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const int k = tid + c * ET;
            if (k < D && fabs(z[c]) > best) {
                best = fabs(z[c]);
                bi = k;
                val = z[c];
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double ob = __shfl_xor_sync(0xffffffffu, best, o), ov = __shfl_xor_sync(0xffffffffu, val, o);
            const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
            if (ob > best || (ob == best && oi < bi)) {
                best = ob;
                bi = oi;
                val = ov;
            }
        }
        __syncthreads();
        if (lane == 0) {
            red[0][warp] = best;
            red[1][warp] = val;
            s_idx[warp] = bi;
        }
        __syncthreads();
        best = red[0][0];
        val = red[1][0];
        bi = s_idx[0];
        for (int w = 1; w < EW; ++w)
            if (red[0][w] > best || (red[0][w] == best && s_idx[w] < bi)) {
                best = red[0][w];
                bi = s_idx[w];
                val = red[1][w];
            }
        const double sign = val < 0.0 ? -1.0 : 1.0;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const int k = tid + c * ET;
            if (k < D) P.comps[(size_t)m * D + k] = (float)(sign * z[c]);
        }
        // (an eigenvalue of a semi-definite matrix that rounding has left below zero is zero)
        if (tid == 0 && P.eig_out) P.eig_out[m] = fmax(lam[q], 0.0) / scale;
    }
}

struct EigWs {
    double *Z, *d, *e, *tau, *wy, *prod, *next, *words;
    size_t bytes;
};

constexpr int REFL_BLOCK = 8;   // reflections applied together (two where rows are longer than 1024)

size_t eig_words(int D, int p) { return 2 * (size_t)D * D + 4 * (size_t)p * D; }

EigWs carve_eig(void *base, int D, int p)
{
    unsigned char *b = reinterpret_cast<unsigned char *>(base);
    size_t off = 0;
    auto take = [&](size_t bytes) {
        off = align_up(off, 256);
        void *q = b ? b + off : nullptr;
        off += bytes;
        return q;
    };
    EigWs w{};
    const size_t row = (size_t)D * sizeof(double);
    w.Z = (double *)take((size_t)p * row);
    w.d = (double *)take(row);
    w.e = (double *)take(row);
    w.tau = (double *)take(row);
    w.wy = (double *)take((size_t)(D + REFL_BLOCK) * REFL_BLOCK * sizeof(double));
    // (one piece: all ones at launch)
    w.prod = (double *)take(eig_words(D, p) * sizeof(double));
    w.next = b ? w.prod + (size_t)D * D : nullptr;
    w.words = b ? w.next + (size_t)D * D : nullptr;
    w.bytes = align_up(off, 256);
    return w;
}

template <typename P>
cudaError_t launch_coop(void (*kern)(P), int grid, size_t smem, P &params, cudaStream_t s)
{
    // (always the same value: another thread may be launching the same kernel with another size)
    cudaError_t err = smem == 0 ? cudaSuccess : cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DYN_SMEM_LIMIT);
    if (err != cudaSuccess) return err;
    void *args[] = {&params};
    err = cudaLaunchCooperativeKernel((const void *)kern, dim3((unsigned)grid), dim3(ET), args, smem, s);
    count_launch();
    return err;
}

}  // namespace

size_t sym_eig_workspace_bytes(int D, int p) { return carve_eig(nullptr, D, p).bytes; }

cudaError_t launch_sym_eig(double *A, const double *diag, double *refl, int D, int p, float *comps, double *eig_out,
                           Control *ctl, void *workspace, cudaStream_t s)
{
    EigWs w = carve_eig(workspace, D, p);
    cudaError_t err = cudaMemsetAsync(w.prod, 0xFF, eig_words(D, p) * sizeof(double), s);
    if (err != cudaSuccess) return err;
    int sms = 0, dev = 0;
    if ((err = cudaGetDevice(&dev)) != cudaSuccess) return err;
    if ((err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return err;
    // eight rows per CTA (what a thread's registers hold for D <= 1024), more where the SMs run out
    int G = (D + 7) / 8;
    if (G > sms) G = sms;
    const int R = (D + G - 1) / G;
    if (R > MAX_ROWS || (p + sms - 1) / sms > MAX_VECS) return cudaErrorInvalidValue;
    TridiagParams T{A, diag, refl, w.d, w.e, w.tau, w.prod, w.next, ctl, D, 0};
    const bool regs = D <= 1024 && R <= 8;
    size_t smem = (size_t)(2 + R) * D * sizeof(double);
    T.resident = !regs && smem <= DYN_SMEM_LIMIT;   // D up to about 1850
    if (!T.resident) smem = (size_t)2 * D * sizeof(double);
    const int C = (D + ET - 1) / ET;
    if (regs && C <= 1) err = launch_coop(tridiag_regs_kernel<1>, G, 0, T, s);
    else if (regs && C <= 2) err = launch_coop(tridiag_regs_kernel<2>, G, 0, T, s);
    else if (regs) err = launch_coop(tridiag_regs_kernel<4>, G, 0, T, s);
    else if (C <= 8) err = launch_coop(tridiag_kernel<8>, G, smem, T, s);
    else err = launch_coop(tridiag_kernel<16>, G, smem, T, s);
    if (err != cudaSuccess) return err;
    if (D > 2) {
        const int rb = C <= 4 ? REFL_BLOCK : 2, nblk = (D - 2 + rb - 1) / rb;
        if (C <= 4) refl_block_kernel<REFL_BLOCK><<<nblk, ET, 0, s>>>(refl, w.tau, D, w.wy);
        else refl_block_kernel<2><<<nblk, ET, 0, s>>>(refl, w.tau, D, w.wy);
        count_launch();
        if ((err = cudaGetLastError()) != cudaSuccess) return err;
    }
    EigvecParams V{diag, w.d, w.e, refl, w.wy, w.Z, w.words, comps, eig_out, ctl, D, p};
    const int GV = p < sms ? p : sms;
    const size_t smem_v = (size_t)5 * D * sizeof(double) + (size_t)D;
    if (C <= 1) return launch_coop(eigvec_kernel<1, REFL_BLOCK>, GV, smem_v, V, s);
    if (C <= 2) return launch_coop(eigvec_kernel<2, REFL_BLOCK>, GV, smem_v, V, s);
    if (C <= 4) return launch_coop(eigvec_kernel<4, REFL_BLOCK>, GV, smem_v, V, s);
    return launch_coop(eigvec_kernel<16, 2>, GV, smem_v, V, s);
}

}  // namespace cat
