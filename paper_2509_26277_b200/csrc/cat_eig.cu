// Leading eigenpairs of a symmetric positive semi-definite D x D matrix in fp64, for the PCA of
// Section 3.1 (the projection that Algorithm 1 step 1 fits).
//
// Only the p largest of D pairs are wanted (p is 50 of 1000 in the method's setting), so the matrix
// is reduced to tridiagonal form once (Householder reflections, 4/3 D^3 operations) and the pairs
// are taken from the tridiagonal matrix: eigenvalues by bisection on the Sturm sequence, vectors by
// inverse iteration with orthogonalisation against all larger pairs, then the reflections are
// applied to the p vectors.  (Golub & Van Loan, Matrix Computations, ch. 8.)  One-sided Jacobi
// rotations over all pairs of columns, the earlier form, took 155 ms for D = 1000: about ten sweeps
// of 999 dependent launches.  This takes 5.1 ms there with p = 50.
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

__device__ __forceinline__ void store_flag(uint32_t *p, uint32_t v)
{
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

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
        if ((it & 255u) == 255u) {
            if (*(volatile int *)&ctl->device_status != (int)CAT_OK) return false;
            const uint64_t now = global_timer();
            if (t0 == 0) t0 = now;
            else if (now - t0 > TC_TIMEOUT_NS) {
                atomicExch(&ctl->device_status, (int)CAT_ERR_DEVICE_TIMEOUT);
                return false;
            }
        }
    }
#pragma unroll
    for (int c = 0; c < C; ++c) out[c] = __longlong_as_double((long long)b[c]);
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

// Householder reduction to tridiagonal form.  A row of the matrix belongs to one CTA and stays with it: for
// D <= 1024 in registers (REGS: rows 8 me ... 8 me + 7, column k with thread k mod 256; 8 MB over 125 SMs at
// D = 1000; a CTA's products are one 64-byte store and it leaves when its rows are done), beyond that in
// shared or global memory (rows me, me + G, ...: there the work per step counts).  Step j: every CTA forms reflection j from
// row j (which its owner has published up to update j - 2) and the vectors v, w of update j - 1, applies
// that update to its own rows and in the same sweep multiplies them with the new reflection; each CTA
// publishes its products and collects everybody's, word by word, without a barrier.
//   bound: latency.  A step moves 2 D values between CTAs and does 6 (D - j)^2 / G operations per CTA;
//   the exchange, three block-wide sums and a square root and two divisions in fp64 make it 3.1 us (D = 1000; 3.7 with 512 threads).
//   With a grid barrier (a flag per CTA, polled by all) in place of the self-validating words the exchange alone
//   took 6 of 9 us.
template <int C, bool REGS>
__global__ void __launch_bounds__(ET) tridiag_kernel(TridiagParams P)
{
    extern __shared__ double sm[];
    __shared__ double red[2][EW], red_rows[EW][MAX_ROWS];
    // Each is written before a step's barrier and read behind it, and written again only behind another barrier of
    // the step: s_x1 around the sum of squares, s_w1 around v'Av.  (One word for both would be written by a warp that
    // is a step ahead while another has yet to read it.)
    __shared__ double s_x1, s_w1;
    constexpr int RR = REGS ? 8 : 1;
    const int D = P.D, G = gridDim.x, me = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int R = REGS ? (D - me * 8 < 8 ? D - me * 8 : 8) : (D - me + G - 1) / G;
    const int i0 = REGS ? me * 8 : me, di = REGS ? 1 : G;   // own rows: i0 + r di
    double *sv = sm, *sw = sm + D, *rows = sm + 2 * D;
    const double scale = diagonal_scale(P.diag, D, red[0]);
    for (int k = tid; k < 2 * D; k += ET) sm[k] = 0.0;
    double ar[RR][C];
    if (REGS) {
#pragma unroll
        for (int r = 0; r < RR; ++r)
#pragma unroll
            for (int c = 0; c < C; ++c) {
                const int i = i0 + r * di, k = tid + c * ET;
                ar[r][c] = i < D && k < D ? P.A[(size_t)i * D + k] * scale : 0.0;
                if (i == 0 && k < D) publish(P.next + k, ar[r][c]);
            }
    } else {
        for (int r = 0; r < R; ++r) {
            double *src = P.A + (size_t)(me + r * G) * D;
            double *dst = P.resident ? rows + (size_t)r * D : src;
            for (int k = tid; k < D; k += ET) {
                const double a = src[k] * scale;
                dst[k] = a;
                if (me + r * G == 0) publish(P.next + k, a);
            }
        }
    }
    double vo[C], wo[C];
#pragma unroll
    for (int c = 0; c < C; ++c) vo[c] = wo[c] = 0.0;
    double v1 = 0.0, w1 = 0.0;   // the previous update's v, w at index j
    __syncthreads();

    for (int j = 0; j < D; ++j) {
        // the CTA of row j + 1 (or the last one) records step j; in registers' form a CTA leaves with its last row
        const bool lead = REGS ? me == (j + 1 < D ? j + 1 : j) / 8 : me == j % G;
        if (REGS && i0 + R <= j) break;
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
        const int r_first = j + 1 <= i0 ? 0 : (j + 1 - i0 + di - 1) / di;   // first own row with index > j
        if (REGS) {
            double acc[8];
#pragma unroll
            for (int r = 0; r < RR; ++r) {
                acc[r] = 0.0;
                const int i = i0 + r;
                if (i > j && i < D) {
                    const double vi = -sv[i], wi = -sw[i];
#pragma unroll
                    for (int c = 0; c < C; ++c)
                        if (warp * 32 + 31 + c * ET > j) {   // (columns up to j are done with)
                            ar[r][c] = fma(wi, vo[c], fma(vi, wo[c], ar[r][c]));
                            acc[r] = fma(ar[r][c], vn[c], acc[r]);
                        }
                    if (i == j + 1) {
#pragma unroll
                        for (int c = 0; c < C; ++c) {
                            const int k = tid + c * ET;
                            if (k > j && k < D) publish(P.next + (size_t)(j + 1) * D + k, ar[r][c]);
                        }
                    }
                }
            }
            const double s = warp_sum8(acc, lane);
            if ((lane & 3) == 0) red_rows[warp][lane >> 2] = s;
        } else {
            for (int r0 = r_first; r0 < R; r0 += 8) {
                double acc[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    acc[u] = 0.0;
                    const int r = r0 + u, i = i0 + r * di;
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
        }
        __syncthreads();
        if (tid >= r_first && tid < R) {
            double part[EW];
#pragma unroll
            for (int w = 0; w < EW; ++w) part[w] = red_rows[w][tid];
            publish(P.prod + (size_t)j * D + i0 + tid * di, tree8(part));
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
    const double *d, *e, *tau, *refl;
    double *Z;                        // [p][D] vectors
    uint32_t *flags;                  // barrier counter, then [p] published vectors; zero at launch
    float *comps;                     // [p][D] out
    double *eig_out;                  // [p] out or null
    Control *ctl;
    int D, p;
};

// eigenvalues of the tridiagonal matrix below x (Sturm sequence)
__device__ __forceinline__ int count_below(const double *d, const double *e2, int D, double x, double pivmin)
{
    int n = 0;
    double q = d[0] - x;
    for (int i = 0;;) {
        if (fabs(q) < pivmin) q = -pivmin;
        n += q < 0.0;
        if (++i == D) return n;
        q = d[i] - x - e2[i - 1] / q;
    }
}

// The p largest eigenpairs.  CTA b has the vectors b, b + G, ...; all of them go through
//   bisection      256 points of the interval at a time, 8 bits of the eigenvalue per pass over the matrix
//   solve          (T - lambda) z = z by Gaussian elimination with partial pivoting (one thread:
//                  a chain of D dependent steps; the vectors run beside each other)
//   orthogonalise  modified Gram-Schmidt in order of decreasing eigenvalue: a CTA waits for each
//                  earlier vector and takes it out of its own.  Clustered or equal eigenvalues get
//                  different starts, so their vectors span the eigenspace.
//   back           the reflections in reverse order, then sign, fp32 store
// Three rounds of solve and orthogonalise, the last one orthogonalised twice.
//   bound: latency of the serial chains (D = 1000, p = 50: 1.7 ms in all).
template <int C>
__global__ void __launch_bounds__(ET) eigvec_kernel(EigvecParams P)
{
    extern __shared__ double sm[];
    __shared__ double red[2][EW], lam[MAX_VECS];
    __shared__ int s_idx[EW];
    __shared__ int ok_flag;
    const int D = P.D, p = P.p, G = gridDim.x, me = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int NV = (p - me + G - 1) / G;
    uint32_t *vec_flag = P.flags + 1;
    double *sd = sm, *u0 = sm + D, *u1 = sm + 2 * D, *u2 = sm + 3 * D, *l = sm + 4 * D;
    unsigned char *swapped = reinterpret_cast<unsigned char *>(sm + 5 * D);
    const double scale = diagonal_scale(P.diag, D, red[0]);
    int par = 0;

    // ---- bisection between the Gershgorin bounds
    double lo0 = INFINITY, hi0 = -INFINITY, emax = 0.0;
    for (int k = tid; k < D; k += ET) {
        const double el = k > 0 ? fabs(P.e[k - 1]) : 0.0, er = k + 1 < D ? fabs(P.e[k]) : 0.0;
        sd[k] = P.d[k];
        if (k + 1 < D) u0[k] = er * er;
        emax = fmax(emax, er * er);
        lo0 = fmin(lo0, P.d[k] - el - er);
        hi0 = fmax(hi0, P.d[k] + el + er);
    }
    double b3[3] = {-lo0, hi0, emax};
#pragma unroll
    for (int q = 0; q < 3; ++q) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) b3[q] = fmax(b3[q], __shfl_xor_sync(0xffffffffu, b3[q], o));
        __syncthreads();
        if (lane == 0) red[0][warp] = b3[q];
        __syncthreads();
        for (int w = 0; w < EW; ++w) b3[q] = fmax(b3[q], red[0][w]);
    }
    const double tnorm = fmax(fmax(fabs(b3[0]), fabs(b3[1])), 1e-290);
    const double margin = 4.0 * (double)D * 2.3e-16 * tnorm;
    const double pivmin = 1e-300 * fmax(1.0, b3[2]);
    for (int q = 0; q < NV; ++q) {
        const int want = D - 1 - (me + q * G);   // index of the eigenvalue in ascending order
        double lo = -b3[0] - margin, hi = b3[1] + margin;
        for (int pass = 0; pass < 8; ++pass) {
            const double step = (hi - lo) / (double)(ET + 1);
            const double x = lo + step * (double)(tid + 1);
            const int below = __syncthreads_count(count_below(sd, u0, D, x, pivmin) <= want);
            const double nlo = below > 0 ? lo + step * (double)below : lo;
            const double nhi = below < ET ? lo + step * (double)(below + 1) : hi;
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
                // P L U = T - lambda: u0 (inverted), u1, u2 the rows of U; l overwrites the off-diagonal
                const double lm = lam[q];
                double a = sd[0] - lm, b = D > 1 ? l[0] : 0.0;
                for (int i = 0; i + 1 < D; ++i) {
                    const double sub = l[i], dg = sd[i + 1] - lm, sup = i + 2 < D ? l[i + 1] : 0.0;
                    if (fabs(a) >= fabs(sub)) {
                        if (fabs(a) < tiny) a = a < 0.0 ? -tiny : tiny;
                        const double r = 1.0 / a, f = sub * r;
                        u0[i] = r;
                        u1[i] = b;
                        u2[i] = 0.0;
                        l[i] = f;
                        swapped[i] = 0;
                        a = fma(-f, b, dg);
                        b = sup;
                    } else {
                        double pv = sub;
                        if (fabs(pv) < tiny) pv = pv < 0.0 ? -tiny : tiny;
                        const double r = 1.0 / pv, f = a * r;
                        u0[i] = r;
                        u1[i] = dg;
                        u2[i] = sup;
                        l[i] = f;
                        swapped[i] = 1;
                        a = fma(-f, dg, b);
                        b = -f * sup;
                    }
                }
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
                for (int i = 0; i + 1 < D; ++i) {
                    const double nx = x[i + 1], f = l[i];
                    if (swapped[i]) {
                        x[i] = nx;
                        cur = fma(-f, nx, cur);
                    } else {
                        x[i] = cur;
                        cur = fma(-f, cur, nx);
                    }
                }
                double z1 = cur * u0[D - 1], z2 = 0.0;
                x[D - 1] = z1;
                for (int i = D - 2; i >= 0; --i) {
                    const double t = fma(-u1[i], z1, fma(-u2[i], z2, x[i])) * u0[i];
                    x[i] = t;
                    z2 = z1;
                    z1 = t;
                }
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
            const uint32_t gen = (uint32_t)(round + pass + 1);
            double z[MAX_VECS][C];
#pragma unroll
            for (int q = 0; q < MAX_VECS; ++q)
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    const int k = tid + c * ET;
                    z[q][c] = q < NV && k < D ? P.Z[(size_t)(me + q * G) * D + k] : 0.0;
                }
            const int last = me + (NV - 1) * G;
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
                                if (k < D) P.Z[(size_t)i * D + k] = z[q][c];
                            }
                    __syncthreads();
                    if (tid == 0) {
                        __threadfence();
                        store_flag(vec_flag + i, gen);
                    }
                }
                if (i == last) break;
                if (tid == 0) ok_flag = wait_flag(vec_flag + i, gen, P.ctl);
                __syncthreads();
                if (!ok_flag) return;
                double zi[C], dot[MAX_VECS];
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    const int k = tid + c * ET;
                    zi[c] = k < D ? __ldcg(P.Z + (size_t)i * D + k) : 0.0;
                }
#pragma unroll
                for (int q = 0; q < MAX_VECS; ++q) {
                    if (q >= NV || me + q * G <= i) continue;
                    dot[q] = 0.0;
#pragma unroll
                    for (int c = 0; c < C; ++c) dot[q] = fma(zi[c], z[q][c], dot[q]);
                    dot[q] = block_sum(dot[q], red[par ^= 1]);
#pragma unroll
                    for (int c = 0; c < C; ++c) z[q][c] = fma(-dot[q], zi[c], z[q][c]);
                }
            }
            // every CTA has read what this pass published before anything rewrites it
            if (!grid_barrier(P.flags, gen, P.ctl)) return;
        }
    }

    // ---- back transformation: z <- H_0 H_1 ... H_{D-3} z, then sign and store
    for (int q = 0; q < NV; ++q) {
        const int m = me + q * G;
        double z[C], v[C];
        __syncthreads();
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const int k = tid + c * ET;
            z[c] = k < D ? P.Z[(size_t)m * D + k] : 0.0;
            v[c] = D >= 3 && k > D - 3 && k < D ? P.refl[(size_t)(D - 3) * D + k] : 0.0;
        }
        for (int j = D - 3; j >= 0; --j) {
            double vnext[C];
#pragma unroll
            for (int c = 0; c < C; ++c) {
                const int k = tid + c * ET;
                vnext[c] = j > 0 && k > j - 1 && k < D ? P.refl[(size_t)(j - 1) * D + k] : 0.0;
            }
            double s = 0.0;
#pragma unroll
            for (int c = 0; c < C; ++c) s = fma(v[c], z[c], s);
            s = -P.tau[j] * block_sum(s, red[par ^= 1]);
#pragma unroll
            for (int c = 0; c < C; ++c) {
                z[c] = fma(s, v[c], z[c]);
                v[c] = vnext[c];
            }
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
    double *Z, *d, *e, *tau, *prod, *next;
    uint32_t *flags;
    size_t bytes;
};

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
    w.flags = (uint32_t *)take((size_t)(1 + p) * sizeof(uint32_t));
    w.prod = (double *)take(2 * (size_t)D * row);
    w.next = b ? w.prod + (size_t)D * D : nullptr;
    w.bytes = align_up(off, 256);
    return w;
}

template <typename P>
cudaError_t launch_coop(void (*kern)(P), int grid, size_t smem, P &params, cudaStream_t s)
{
    // (always the same value: another thread may be launching the same kernel with another size)
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DYN_SMEM_LIMIT);
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
    cudaError_t err = cudaMemsetAsync(w.flags, 0, (size_t)(1 + p) * sizeof(uint32_t), s);
    if (err == cudaSuccess) err = cudaMemsetAsync(w.prod, 0xFF, 2 * (size_t)D * D * sizeof(double), s);
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
    if (regs && C <= 1) err = launch_coop(tridiag_kernel<1, true>, G, smem, T, s);
    else if (regs && C <= 2) err = launch_coop(tridiag_kernel<2, true>, G, smem, T, s);
    else if (regs) err = launch_coop(tridiag_kernel<4, true>, G, smem, T, s);
    else if (C <= 8) err = launch_coop(tridiag_kernel<8, false>, G, smem, T, s);
    else err = launch_coop(tridiag_kernel<16, false>, G, smem, T, s);
    if (err != cudaSuccess) return err;
    EigvecParams V{diag, w.d, w.e, w.tau, refl, w.Z, w.flags, comps, eig_out, ctl, D, p};
    const int GV = p < sms ? p : sms;
    const size_t smem_v = (size_t)5 * D * sizeof(double) + (size_t)D;
    if (C <= 1) return launch_coop(eigvec_kernel<1>, GV, smem_v, V, s);
    if (C <= 2) return launch_coop(eigvec_kernel<2>, GV, smem_v, V, s);
    if (C <= 4) return launch_coop(eigvec_kernel<4>, GV, smem_v, V, s);
    return launch_coop(eigvec_kernel<16>, GV, smem_v, V, s);
}

}  // namespace cat
