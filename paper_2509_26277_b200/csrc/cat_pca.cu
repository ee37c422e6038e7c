// PCA front-end of CAT (Section 3.1: the LQ outputs are reduced with PCA before clustering, and
// "PCA is only used to obtain clusters"; Algorithm 1 step 1, Algorithm 2 step 1).
//
//   column means            fp64 partial sums per row chunk, added in a fixed order
//   covariance              D x D, fp64 mma on 64 x 64 tiles over the centred rows
//                           (upper-triangular tiles, mirrored); 1 / (N - 1) normalisation
//   eigen-decomposition     the p largest pairs by tridiagonal reduction, bisection and inverse
//                           iteration in fp64 (cat_eig.cu); a component's sign is fixed so that its
//                           entry of largest magnitude is positive, stored as fp32 rows
//   projection              Z = (Y - mean) V_p^T, fp64 accumulation, fp32 result
//   affine with labels      out_i = gamma_l * y_i + beta_l for given cluster ids (Algorithm 2 steps 4-8)
//
// Everything is deterministic: no floating-point atomics, fixed summation orders.
#include "cat_internal.cuh"

#include <cuda_bf16.h>

namespace cat {

namespace {

constexpr int PT = 64;          // tile edge of the fp64 contractions
constexpr int PK = 16;          // depth of a shared-memory step
constexpr int P_THREADS = 128;  // 2 x 2 warps, 32 x 32 outputs each
constexpr int MEAN_CHUNKS = 64;

// ---------------------------------------------------------------- column means
__global__ void __launch_bounds__(128) col_partial_kernel(const float *__restrict__ Y, int64_t N, int D,
                                                          double *__restrict__ part)
{
    const int col = blockIdx.x * 128 + threadIdx.x;
    const int64_t per = (N + gridDim.y - 1) / gridDim.y;
    const int64_t r0 = (int64_t)blockIdx.y * per;
    const int64_t r1 = r0 + per < N ? r0 + per : N;
    if (col >= D) return;
    double s = 0.0;
    for (int64_t r = r0; r < r1; ++r) s += (double)Y[(size_t)r * D + col];
    part[(size_t)blockIdx.y * D + col] = s;
}

__global__ void col_mean_kernel(const double *__restrict__ part, int chunks, int64_t N, int D,
                                double *__restrict__ mean64, float *__restrict__ mean32)
{
    const int col = blockIdx.x * blockDim.x + threadIdx.x;
    if (col >= D) return;
    double s = 0.0;
    for (int c = 0; c < chunks; ++c) s += part[(size_t)c * D + col];
    s /= (double)N;
    mean64[col] = s;
    if (mean32) mean32[col] = (float)s;
}

// ---------------------------------------------------------------- 64 x 64 fp64 tile product
// Four warps, 32 x 32 each, as 4 x 4 tiles of mma.m8n8k4 in fp64: 16 multiply-adds per operand element
// read from shared memory, where the 4 x 4 register tiles of scalar FMAs this replaces had two.  Operands
// sit in shared memory with strides of 4 mod 16 doubles, which spreads a fragment's half-warp reads over
// all banks.
__device__ __forceinline__ void mma_f64(double (&c)[2], double a, double b)
{
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};"
                 : "+d"(c[0]), "+d"(c[1])
                 : "d"(a), "d"(b));
}

// Covariance tile (bi, bj), bj >= bi, over the rows of split blockIdx.z:
// part[z][a][b] = sum_i (y_ia - mean_a)(y_ib - mean_b)
//   bound: fp64 multiply-adds (4096 x 1000: 2.2 GFMA over the upper tiles, 0.13 ms at 64 per clock and SM).
__global__ void __launch_bounds__(P_THREADS) cov_kernel(const float *__restrict__ Y, int64_t N, int D,
                                                        const double *__restrict__ mean, double *__restrict__ part)
{
    constexpr int LD = PT + 4;
    __shared__ double As[2][PK][LD], Bs[2][PK][LD];
    const int bi = blockIdx.y, bj = blockIdx.x;
    if (bj < bi) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int m0 = (warp >> 1) * 32, n0 = (warp & 1) * 32, g = lane >> 2, t = lane & 3;
    const int64_t per = (N + gridDim.z - 1) / gridDim.z;
    const int64_t r0 = (int64_t)blockIdx.z * per;
    const int64_t r1 = r0 + per < N ? r0 + per : N;
    // a thread always fetches the same column of each operand, rows k0, k0 + 2, ...
    const int c = tid & 63, k0 = tid >> 6;
    const int ca = bi * PT + c, cb = bj * PT + c;
    const double ma = ca < D ? mean[ca] : 0.0, mb = cb < D ? mean[cb] : 0.0;
    float fa[PK / 2], fb[PK / 2];
    auto fetch = [&](int64_t r) {
#pragma unroll
        for (int q = 0; q < PK / 2; ++q) {
            const int64_t row = r + k0 + 2 * q;
            fa[q] = row < r1 && ca < D ? __ldg(Y + (size_t)row * D + ca) : 0.f;
            fb[q] = row < r1 && cb < D ? __ldg(Y + (size_t)row * D + cb) : 0.f;
        }
    };
    auto put = [&](int64_t r, int buf) {
#pragma unroll
        for (int q = 0; q < PK / 2; ++q) {
            const bool in = r + k0 + 2 * q < r1;
            As[buf][k0 + 2 * q][c] = in && ca < D ? (double)fa[q] - ma : 0.0;
            Bs[buf][k0 + 2 * q][c] = in && cb < D ? (double)fb[q] - mb : 0.0;
        }
    };
    double acc[4][4][2] = {};
    fetch(r0);
    put(r0, 0);
    int buf = 0;
    for (int64_t r = r0; r < r1; r += PK, buf ^= 1) {
        __syncthreads();
        const bool more = r + PK < r1;
        if (more) fetch(r + PK);
#pragma unroll
        for (int k = 0; k < PK; k += 4) {
            double a[4], b[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                a[i] = As[buf][k + t][m0 + 8 * i + g];
                b[i] = Bs[buf][k + t][n0 + 8 * i + g];
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) mma_f64(acc[i][j], a[i], b[j]);
        }
        if (more) put(r + PK, buf ^ 1);
    }
    double *out = part + (size_t)blockIdx.z * D * D;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int a = bi * PT + m0 + 8 * i + g, b = bj * PT + n0 + 8 * j + 2 * t + q;
                if (a < D && b < D) out[(size_t)a * D + b] = acc[i][j][q];
            }
}

// G = (sum of the splits' upper triangles, mirrored) / (N - 1), and its diagonal once more
__global__ void cov_finish_kernel(const double *__restrict__ part, int splits, int D, int64_t N,
                                  double *__restrict__ G, double *__restrict__ diag)
{
    const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (size_t)D * D) return;
    const int a = (int)(e / D), b = (int)(e % D);
    const int lo = a < b ? a : b, hi = a < b ? b : a;
    double s = 0.0;
    for (int z = 0; z < splits; ++z) s += part[(size_t)z * D * D + (size_t)lo * D + hi];
    s /= (double)(N > 1 ? N - 1 : 1);
    G[e] = s;
    if (a == b) diag[a] = s;
}

// ---------------------------------------------------------------- projection
// Z[i, r] = sum_j (Y[i, j] - mean[j]) * comps[r, j], fp64 accumulation: one CTA per 64 rows x 64 components.
//   bound: the fp64 tensor pipe, 73 % busy (50 000 x 1000, p = 50: 2.8 GFMA with p rounded up to 56, 0.15 ms at 64
//   per clock and SM; takes 0.27; tiles of 32 rows, for a fuller last wave, 0.30).
__global__ void __launch_bounds__(P_THREADS) project_kernel(const float *__restrict__ Y, int64_t N, int D, int p,
                                                            const float *__restrict__ mean, const float *__restrict__ comps,
                                                            float *__restrict__ Z)
{
    pdl_enter();
    constexpr int LD = PK + 4;
    __shared__ double As[2][PT][LD], Bs[2][PT][LD];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int m0 = (warp >> 1) * 32, n0 = (warp & 1) * 32, g = lane >> 2, t = lane & 3;
    const int64_t row0 = (int64_t)blockIdx.x * PT;
    const int c0 = blockIdx.y * PT;
    const int tiles = p - c0 - n0 >= 32 ? 4 : (p - c0 - n0 + 7) / 8;   // component tiles of this warp that hold anything
    // a thread always fetches the same column of a step, rows / components m, m + 8, ...
    const int k = tid & 15, mb = tid >> 4;
    float fa[8], fb[8], fm = 0.f;
    auto fetch = [&](int j0) {
        const int j = j0 + k;
        fm = j < D ? __ldg(mean + j) : 0.f;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int64_t row = row0 + mb + 8 * q;
            const int r = c0 + mb + 8 * q;
            fa[q] = row < N && j < D ? __ldg(Y + (size_t)row * D + j) : 0.f;
            fb[q] = r < p && j < D ? __ldg(comps + (size_t)r * D + j) : 0.f;
        }
    };
    auto put = [&](int j0, int buf) {
        const bool in = j0 + k < D;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            As[buf][mb + 8 * q][k] = in ? (double)fa[q] - (double)fm : 0.0;
            Bs[buf][mb + 8 * q][k] = (double)fb[q];
        }
    };
    double acc[4][4][2] = {};
    fetch(0);
    put(0, 0);
    int buf = 0;
    for (int j0 = 0; j0 < D; j0 += PK, buf ^= 1) {
        __syncthreads();
        const bool more = j0 + PK < D;
        if (more) fetch(j0 + PK);
#pragma unroll
        for (int kk = 0; kk < PK; kk += 4) {
            double a[4], b[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                a[i] = As[buf][m0 + 8 * i + g][kk + t];
                b[i] = Bs[buf][n0 + 8 * i + g][kk + t];
            }
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (j < tiles)
#pragma unroll
                    for (int i = 0; i < 4; ++i) mma_f64(acc[i][j], a[i], b[j]);
        }
        if (more) put(j0 + PK, buf ^ 1);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int64_t row = row0 + m0 + 8 * i + g;
                const int r = c0 + n0 + 8 * j + 2 * t + q;
                if (row < N && r < p) Z[(size_t)row * p + r] = (float)acc[i][j][q];
            }
}

// ---------------------------------------------------------------- affine map for given cluster ids
// one warp per row: out = fma(gamma_l, y, beta_l); a label outside [0, K) leaves the row as it is.
// All loads of a step (eight per lane and operand) are in flight together.
template <int VEC>
__global__ void __launch_bounds__(256) affine_labels_kernel(const float *__restrict__ Y, int64_t N, int D, int K,
                                                            const int32_t *__restrict__ labels,
                                                            const float *__restrict__ gamma, const float *__restrict__ beta,
                                                            float *__restrict__ out)
{
    pdl_enter();
    const int lane = threadIdx.x & 31;
    for (int64_t row = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5); row < N; row += (int64_t)gridDim.x * 8) {
        const int l = labels[row];
        const bool ok = l >= 0 && l < K;
        const float *y = Y + (size_t)row * D;
        const float *g = gamma + (size_t)(ok ? l : 0) * D;
        const float *b = beta + (size_t)(ok ? l : 0) * D;
        float *o = out + (size_t)row * D;
        if (VEC == 4) {
            const int D4 = D >> 2;
            for (int j0 = lane; j0 < D4; j0 += 128) {
                float4 yv[4], gv[4], bv[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int j = j0 + 32 * u;
                    if (j < D4) {
                        yv[u] = __ldcs(reinterpret_cast<const float4 *>(y) + j);
                        gv[u] = __ldg(reinterpret_cast<const float4 *>(g) + j);
                        bv[u] = __ldg(reinterpret_cast<const float4 *>(b) + j);
                    }
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int j = j0 + 32 * u;
                    if (j >= D4) continue;
                    float4 v = yv[u];
                    if (ok)
                        v = make_float4(fmaf(gv[u].x, v.x, bv[u].x), fmaf(gv[u].y, v.y, bv[u].y), fmaf(gv[u].z, v.z, bv[u].z),
                                        fmaf(gv[u].w, v.w, bv[u].w));
                    __stcs(reinterpret_cast<float4 *>(o) + j, v);
                }
            }
        } else {
            for (int j0 = lane; j0 < D; j0 += 256) {
                float yv[8], gv[8], bv[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int j = j0 + 32 * u;
                    if (j < D) {
                        yv[u] = __ldg(y + j);
                        gv[u] = __ldg(g + j);
                        bv[u] = __ldg(b + j);
                    }
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int j = j0 + 32 * u;
                    if (j < D) o[j] = ok ? fmaf(gv[u], yv[u], bv[u]) : yv[u];
                }
            }
        }
    }
}

// The same with a bf16 result (round to nearest even of the fp32 fused multiply-add), for all rows or
// for the rows of the two exact-pass queues (whose lengths are read from ctl).
__global__ void __launch_bounds__(256) affine_bf16_kernel(const float *__restrict__ Y, int64_t N, int D, int K,
                                                          const int32_t *__restrict__ labels,
                                                          const float *__restrict__ gamma, const float *__restrict__ beta,
                                                          __nv_bfloat16 *__restrict__ out,
                                                          const int32_t *__restrict__ refine_rows,
                                                          const int32_t *__restrict__ cand_rows, const Control *ctl)
{
    const int lane = threadIdx.x & 31;
    const bool listed = ctl != nullptr;
    int64_t nref = 0, total = N;
    if (listed) {
        nref = ctl->refine_count < N ? ctl->refine_count : N;
        const int64_t nc = ctl->cand_count < N ? ctl->cand_count : N;
        total = nref + nc;
    }
    const bool vec4 = (D & 3) == 0;
    for (int64_t q = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5); q < total; q += (int64_t)gridDim.x * 8) {
        const int64_t row = listed ? (int64_t)(q < nref ? refine_rows[q] : cand_rows[q - nref]) : q;
        if (row < 0 || row >= N) continue;
        const int l = labels[row];
        const bool ok = l >= 0 && l < K;
        const float *y = Y + (size_t)row * D;
        const float *g = gamma + (size_t)(ok ? l : 0) * D;
        const float *b = beta + (size_t)(ok ? l : 0) * D;
        __nv_bfloat16 *o = out + (size_t)row * D;
        if (vec4) {
            for (int j = lane; j < (D >> 2); j += 32) {
                const float4 yv = __ldcs(reinterpret_cast<const float4 *>(y) + j);
                float4 v = yv;
                if (ok) {
                    const float4 gv = __ldg(reinterpret_cast<const float4 *>(g) + j);
                    const float4 bv = __ldg(reinterpret_cast<const float4 *>(b) + j);
                    v = make_float4(fmaf(gv.x, yv.x, bv.x), fmaf(gv.y, yv.y, bv.y), fmaf(gv.z, yv.z, bv.z),
                                    fmaf(gv.w, yv.w, bv.w));
                }
                const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
                uint2 w2;
                w2.x = *reinterpret_cast<const unsigned int *>(&lo);
                w2.y = *reinterpret_cast<const unsigned int *>(&hi);
                reinterpret_cast<uint2 *>(o)[j] = w2;
            }
        } else {
            for (int j = lane; j < D; j += 32) o[j] = __float2bfloat16_rn(ok ? fmaf(g[j], y[j], b[j]) : y[j]);
        }
    }
}

// row splits of the covariance: enough CTAs for four per SM
int cov_splits(int D)
{
    const int T = (D + PT - 1) / PT;
    const int tiles = T * (T + 1) / 2;
    const int s = (4 * 148 + tiles - 1) / tiles;
    return s > 32 ? 32 : s;
}

struct PcaWs {
    Control *ctl;        // (first: cat_workspace_report reads the status of the bounded waits here)
    double *mean_part;   // [MEAN_CHUNKS][D]
    double *mean64;      // [D]
    double *diag;        // [D]
    double *G;           // [D][D] covariance
    double *refl;        // [D][D] reflections of the tridiagonal reduction
    double *cov_part;    // [splits][D][D]
    void *eig;
    size_t bytes;
};

PcaWs carve_pca(void *base, int D, int p)
{
    unsigned char *b = reinterpret_cast<unsigned char *>(base);
    size_t off = 0;
    auto take = [&](size_t bytes) {
        off = align_up(off, 256);
        void *q = b ? b + off : nullptr;
        off += bytes;
        return q;
    };
    PcaWs w{};
    const size_t DD = (size_t)D * D;
    w.ctl = (Control *)take(sizeof(Control));
    w.mean_part = (double *)take((size_t)MEAN_CHUNKS * D * sizeof(double));
    w.mean64 = (double *)take((size_t)D * sizeof(double));
    w.diag = (double *)take((size_t)D * sizeof(double));
    w.G = (double *)take(DD * sizeof(double));
    w.refl = (double *)take(DD * sizeof(double));
    w.cov_part = (double *)take((size_t)cov_splits(D) * DD * sizeof(double));
    w.eig = take(sym_eig_workspace_bytes(D, p));
    w.bytes = align_up(off, 256);
    return w;
}

inline bool al16(const void *q) { return (reinterpret_cast<uintptr_t>(q) & 15u) == 0; }

}  // namespace

cudaError_t launch_affine_labels(const float *Y, int64_t N, int D, int K, const int32_t *labels, const float *gamma,
                                 const float *beta, float *out, cudaStream_t s)
{
    int64_t blocks = (N + 7) / 8;
    if (blocks > 148 * 16) blocks = 148 * 16;
    const cudaError_t e = launch_pdl(D % 4 == 0 ? affine_labels_kernel<4> : affine_labels_kernel<1>, dim3((unsigned)blocks), dim3(256),
                                     0, s, Y, N, D, K, labels, gamma, beta, out);
    count_launch();
    return e;
}

cudaError_t launch_affine_bf16(const float *Y, int64_t N, int D, int K, const int32_t *labels, const float *gamma,
                               const float *beta, void *out_bf16, const int32_t *refine_rows, const int32_t *cand_rows,
                               const Control *ctl, cudaStream_t s)
{
    int64_t blocks = (N + 7) / 8;
    if (blocks > 148 * 16) blocks = 148 * 16;
    affine_bf16_kernel<<<(unsigned)blocks, 256, 0, s>>>(Y, N, D, K, labels, gamma, beta,
                                                        reinterpret_cast<__nv_bfloat16 *>(out_bf16), refine_rows, cand_rows, ctl);
    count_launch();
    return cudaGetLastError();
}

}  // namespace cat

using namespace cat;

#define CAT_CUDA(expr)                                  \
    do {                                                \
        if (!cuda_ok((expr))) return CAT_ERR_CUDA;      \
    } while (0)

static cat_status_t pca_shape(int64_t N, int32_t D, int32_t p)
{
    if (N < 2 || D < 1 || p < 1 || p > D) return CAT_ERR_SHAPE;
    if (D > CAT_PCA_MAX_D || p > CAT_PCA_MAX_P || N >= ((int64_t)1 << 31)) return CAT_ERR_UNSUPPORTED;
    return CAT_OK;
}

extern "C" {

size_t cat_pca_workspace_bytes(int64_t N, int32_t D, int32_t p)
{
    if (pca_shape(N, D, p) != CAT_OK) return 0;
    return carve_pca(nullptr, D, p).bytes;
}

cat_status_t cat_pca_fit(const float *Yq, int64_t N, int32_t D, int32_t p, float *mean_out,
                         float *components_out, double *eigenvalues_out, void *workspace,
                         size_t workspace_bytes, void *stream)
{
    if (!Yq || !mean_out || !components_out) return CAT_ERR_NULL;
    cat_status_t st = pca_shape(N, D, p);
    if (st != CAT_OK) return st;
    if (!al16(Yq) || !al16(mean_out) || !al16(components_out) || (eigenvalues_out && !al16(eigenvalues_out)))
        return CAT_ERR_ALIGN;
    if (!workspace || !al16(workspace) || workspace_bytes < cat_pca_workspace_bytes(N, D, p)) return CAT_ERR_WORKSPACE;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    PcaWs w = carve_pca(workspace, D, p);
    CAT_CUDA(launch_reset_control(w.ctl, s));

    int chunks = (int)(N < MEAN_CHUNKS ? N : MEAN_CHUNKS);
    col_partial_kernel<<<dim3((D + 127) / 128, chunks), 128, 0, s>>>(Yq, N, D, w.mean_part);
    col_mean_kernel<<<(D + 255) / 256, 256, 0, s>>>(w.mean_part, chunks, N, D, w.mean64, mean_out);
    const int T = (D + PT - 1) / PT;
    int splits = cov_splits(D);
    if ((int64_t)splits > N) splits = (int)N;
    cov_kernel<<<dim3(T, T, splits), P_THREADS, 0, s>>>(Yq, N, D, w.mean64, w.cov_part);
    const size_t DD = (size_t)D * D;
    cov_finish_kernel<<<(unsigned)((DD + 255) / 256), 256, 0, s>>>(w.cov_part, splits, D, N, w.G, w.diag);
    count_launch(4);
    CAT_CUDA(cudaGetLastError());
    CAT_CUDA(launch_sym_eig(w.G, w.diag, w.refl, D, p, components_out, eigenvalues_out, w.ctl, w.eig, s));
    return CAT_OK;
}

cat_status_t cat_pca_project(const float *Y, int64_t N, int32_t D, int32_t p, const float *mean,
                             const float *components, float *Z_out, void *stream)
{
    if (!Y || !mean || !components || !Z_out) return CAT_ERR_NULL;
    if (N < 1 || D < 1 || p < 1 || p > D) return CAT_ERR_SHAPE;
    if (D > CAT_PCA_MAX_D || p > CAT_PCA_MAX_P || N >= ((int64_t)1 << 31)) return CAT_ERR_UNSUPPORTED;
    if (!al16(Y) || !al16(mean) || !al16(components) || !al16(Z_out)) return CAT_ERR_ALIGN;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    CAT_CUDA(launch_pdl(project_kernel, dim3((unsigned)((N + PT - 1) / PT), (p + PT - 1) / PT), dim3(P_THREADS), 0, s, Y, N, D, p, mean,
                        components, Z_out));
    count_launch();
    return CAT_OK;
}

cat_status_t cat_affine_with_labels(const float *Yq, int64_t N, int32_t D, int32_t K, const int32_t *labels,
                                    const float *gamma, const float *beta, float *Y_out, void *stream)
{
    if (!Yq || !labels || !gamma || !beta || !Y_out) return CAT_ERR_NULL;
    if (N < 1 || D < 1 || K < 1) return CAT_ERR_SHAPE;
    if (K > CAT_MAX_K || D > CAT_MAX_D || N >= ((int64_t)1 << 31)) return CAT_ERR_UNSUPPORTED;
    if (!al16(Yq) || !al16(labels) || !al16(gamma) || !al16(beta) || !al16(Y_out)) return CAT_ERR_ALIGN;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    CAT_CUDA(launch_affine_labels(Yq, N, D, K, labels, gamma, beta, Y_out, s));
    return CAT_OK;
}

// ---- Algorithm 1 and Algorithm 2 with the PCA step, composed from the calls above and the
//      clustering / closed-form entry points

namespace {
struct FitPcaWs {
    void *pca;  size_t pca_bytes;   // (first: its control block speaks for the whole call)
    float *Z;                       // [N, p]
    int32_t *labels;                // [N]
    void *fit;  size_t fit_bytes;   // cat_fit workspace for (N, p, K), then for (N, D, K)
    size_t bytes;
};
FitPcaWs carve_fit_pca(void *base, int64_t N, int D, int K, int p)
{
    unsigned char *b = reinterpret_cast<unsigned char *>(base);
    size_t off = 0;
    auto take = [&](size_t bytes) {
        off = align_up(off, 256);
        void *q = b ? b + off : nullptr;
        off += bytes;
        return q;
    };
    FitPcaWs w{};
    w.pca_bytes = cat_pca_workspace_bytes(N, D, p);
    w.pca = take(w.pca_bytes);
    w.Z = (float *)take((size_t)N * p * sizeof(float));
    w.labels = (int32_t *)take((size_t)N * sizeof(int32_t));
    const size_t a = cat_fit_workspace_bytes(N, p, K), c = cat_fit_workspace_bytes(N, D, K);
    w.fit_bytes = a > c ? a : c;
    w.fit = take(w.fit_bytes);
    w.bytes = align_up(off, 256);
    return w;
}
}  // namespace

size_t cat_fit_pca_workspace_bytes(int64_t N, int32_t D, int32_t K, int32_t p)
{
    if (pca_shape(N, D, p) != CAT_OK || cat_fit_workspace_bytes(N, D, K) == 0 || cat_fit_workspace_bytes(N, p, K) == 0)
        return 0;
    return carve_fit_pca(nullptr, N, D, K, p).bytes;
}

cat_status_t cat_fit_pca(const float *Yq, const float *Yfp, int64_t N, int32_t D, int32_t K, int32_t iters,
                         int32_t p, float *mean_out, float *components_out, float *centroids_out,
                         float *gamma_out, float *beta_out, int32_t *labels_out, void *workspace,
                         size_t workspace_bytes, void *stream)
{
    if (!Yq || !Yfp || !mean_out || !components_out || !centroids_out || !gamma_out || !beta_out) return CAT_ERR_NULL;
    cat_status_t st = pca_shape(N, D, p);
    if (st != CAT_OK) return st;
    if (K < 1 || N < K || iters < 0) return CAT_ERR_SHAPE;
    const size_t need = cat_fit_pca_workspace_bytes(N, D, K, p);
    if (need == 0) return CAT_ERR_UNSUPPORTED;
    if (!workspace || !al16(workspace) || workspace_bytes < need) return CAT_ERR_WORKSPACE;
    // (gamma and beta are written word by word: any address does)
    if (!al16(Yq) || !al16(Yfp) || !al16(mean_out) || !al16(components_out) || !al16(centroids_out) || (labels_out && !al16(labels_out)))
        return CAT_ERR_ALIGN;
    FitPcaWs w = carve_fit_pca(workspace, N, D, K, p);
    int32_t *labels = labels_out ? labels_out : w.labels;
    // Algorithm 1 step 1: the projection; step 2: K-Means on the reduced rows
    if ((st = cat_pca_fit(Yq, N, D, p, mean_out, components_out, nullptr, w.pca, w.pca_bytes, stream)) != CAT_OK) return st;
    if ((st = cat_pca_project(Yq, N, D, p, mean_out, components_out, w.Z, stream)) != CAT_OK) return st;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    if ((st = fit_clusters(w.Z, N, p, K, iters, centroids_out, labels, w.fit, w.fit_bytes, s)) != CAT_OK) return st;
    CAT_CUDA(launch_absorb_control(reinterpret_cast<Control *>(w.pca), reinterpret_cast<const Control *>(w.fit), s));
    // the loop over the clusters: moments and the closed form in the original space
    return fit_closed_form(Yq, Yfp, N, D, K, labels, gamma_out, beta_out, w.fit, s);
}

size_t cat_apply_pca_workspace_bytes(int64_t N, int32_t D, int32_t K, int32_t p)
{
    if (N < 1 || D < 1 || p < 1 || p > D || D > CAT_PCA_MAX_D || p > CAT_PCA_MAX_P) return 0;
    const size_t a = cat_apply_workspace_bytes(N, p, K);
    if (a == 0) return 0;
    const size_t three = align_up(a, 256) + align_up((size_t)N * p * sizeof(float), 256) + align_up((size_t)N * sizeof(int32_t), 256);
    const size_t rows = 256 + align_up(apply_rows_pca_prep_bytes(N, D, K), 256) + align_up((size_t)N * 16, 256) + align_up((size_t)N * sizeof(int32_t), 256);
    return three > rows ? three : rows;
}

// One kernel that keeps rows in shared memory, where it takes the shape (the selector of cat_apply's kernel of that kind
// holds here too): against the three steps, 8000 x 777, K = 16, 8 components 30 us and 123, 50 000 x 1000, K = 64, 50
// components 235 and 372, 50 000 x 100, K = 40 42 and 81, and at the line 656 x 100, K = 2 25 and 31, with 256 components 66 x 1000, K = 16 45
// and 83.  (Less than a few hundred rows leave either idle.)
static bool use_apply_rows_pca(int64_t N, int D, int K)
{
    return N * D >= 65536 && (cat_get_small_problem_kernels() & 1) && get_apply_column_split() == 0 && apply_rows_pca_supported(N, D, K);
}

cat_status_t cat_apply_pca(const float *Yq, int64_t N, int32_t D, int32_t K, int32_t p, const float *mean,
                           const float *components, const float *centroids, const float *gamma,
                           const float *beta, float *Y_out, int32_t *labels_out, void *workspace,
                           size_t workspace_bytes, void *stream)
{
    if (!Yq || !mean || !components || !centroids || !gamma || !beta || !Y_out) return CAT_ERR_NULL;
    const size_t need = cat_apply_pca_workspace_bytes(N, D, K, p);
    if (need == 0) return (N < 1 || D < 1 || p < 1 || p > D || K < 1) ? CAT_ERR_SHAPE : CAT_ERR_UNSUPPORTED;
    if (!workspace || !al16(workspace) || workspace_bytes < need) return CAT_ERR_WORKSPACE;
    // (the assignment's part first: its control block is where cat_workspace_report looks)
    unsigned char *b = reinterpret_cast<unsigned char *>(workspace);
    if (use_apply_rows_pca(N, D, K)) {
        if (!al16(Yq) || !al16(mean) || !al16(components) || !al16(centroids) || !al16(gamma) || !al16(beta) || !al16(Y_out) ||
            (labels_out && !al16(labels_out)))
            return CAT_ERR_ALIGN;
        unsigned char *open_rows = b + 256 + align_up(apply_rows_pca_prep_bytes(N, D, K), 256);
        int32_t *labels = labels_out ? labels_out : reinterpret_cast<int32_t *>(open_rows + align_up((size_t)N * 16, 256));
        CAT_CUDA(launch_apply_rows_pca(Yq, N, D, K, p, mean, components, centroids, gamma, beta, Y_out, labels,
                                       reinterpret_cast<Control *>(b), b + 256, open_rows, reinterpret_cast<cudaStream_t>(stream)));
        return CAT_OK;
    }
    const size_t assign_bytes = align_up(cat_apply_workspace_bytes(N, p, K), 256);
    float *Z = reinterpret_cast<float *>(b + assign_bytes);
    int32_t *labels =
        labels_out ? labels_out : reinterpret_cast<int32_t *>(b + assign_bytes + align_up((size_t)N * p * sizeof(float), 256));
    cat_status_t st;
    // Algorithm 2 step 1: project; step 2: predict the cluster; steps 4-8: correct in the original space
    if ((st = cat_pca_project(Yq, N, D, p, mean, components, Z, stream)) != CAT_OK) return st;
    if ((st = cat_assign(Z, N, p, K, centroids, labels, b, assign_bytes, stream)) != CAT_OK) return st;
    return cat_affine_with_labels(Yq, N, D, K, labels, gamma, beta, Y_out, stream);
}

}  // extern "C"
