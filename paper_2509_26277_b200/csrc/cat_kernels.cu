// CUDA kernels of the CAT hot path (sm_100a), general fp32 path.
//
//   centroid_norms_kernel   ||c_k||^2 for the expanded-form scores
//   assign_kernel           nearest-centroid scores on the fp32 pipes + certainty test
//                           (+ fused per-cluster affine epilogue for inference)
//   refine_kernel           exact fp64 direct-form decision for the rows the fast
//                           scores cannot separate
//   small element-wise kernels for centroid update, means and the gamma/beta solve
//
// Label decision rule.  The K-Means assignment step needs argmin_k ||y - c_k||^2
// (lowest k on ties).  The fast pass evaluates t_k = ||c_k||^2 - 2 y.c_k in fp32,
// whose error is bounded by
//     e <= u * ((2D + 4) * ||y|| * cmax + 4 * cmax^2),  u = 2^-24, cmax = max_k ||c_k||
// (D-term FMA chain, rounding of the stored norm, the final FMA).  If the two smallest
// scores are further apart than 2e the fast argmin is the exact argmin.  Otherwise the
// row is queued and decided by direct-form fp64 distances, scanning k upwards with a
// strict '<' -- the same arithmetic a straightforward double-precision K-Means uses.
#include "cat_internal.cuh"

#include <math_constants.h>

namespace cat {

constexpr int kMaxDevices = 64;

// ======================================================================================
// small helpers
// ======================================================================================

__device__ __forceinline__ void cp_async16(void *smem_dst, const void *gmem_src, int src_bytes)
{
    unsigned s = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(s), "l"(gmem_src),
                 "r"(src_bytes)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait()
{
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// ======================================================================================
// centroid norms
// ======================================================================================

__global__ void centroid_norms_kernel(const float *__restrict__ C, int D, int K,
                                      float *__restrict__ cnorm, Control *ctl, int reset_all)
{
    int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int lane = threadIdx.x & 31;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        ctl->refine_count = 0;
        ctl->cand_count = 0;
        if (reset_all) {
            ctl->device_status = CAT_OK;
            ctl->refined_total = 0;
            ctl->refined_last = 0;
            ctl->settled = 0;
        }
    }
    if (warp >= K) return;
    const float *c = C + (size_t)warp * D;
    double s = 0.0;
    for (int j = lane; j < D; j += 32) {
        double v = (double)c[j];
        s += v * v;
    }
    s = warp_sum(s);
    // round up so that the stored norm never under-states the true one
    if (lane == 0) cnorm[warp] = __double2float_ru(s);
}

cudaError_t launch_centroid_norms(const float *C, int D, int K, float *cnorm, Control *ctl,
                                  cudaStream_t s, bool reset_all)
{
    int threads = 128;
    int blocks = (K * 32 + threads - 1) / threads;
    centroid_norms_kernel<<<blocks, threads, 0, s>>>(C, D, K, cnorm, ctl, reset_all ? 1 : 0);
    count_launch();
    return cudaGetLastError();
}

// ======================================================================================
// assignment (fast fp32 scores)
// ======================================================================================

constexpr int A_BM = 128;       // rows per CTA
constexpr int A_BK = 16;        // D-slab per pipeline stage
constexpr int A_LD = A_BK + 4;  // padded row stride in floats (5 x 16 B: conflict-free 128-bit reads)
constexpr int A_STAGES = 3;
constexpr int A_THREADS = 128;

struct AssignParams {
    const float *Y;
    const float *C;
    const float *cnorm;
    int32_t *labels;
    int32_t *refine_rows;
    Control *ctl;
    const float *gamma;
    const float *beta;
    float *out;
    int64_t N;
    int D;
    int K;
    FastOut fast;
    const int32_t *settled;   // nothing to do once this is set (or null)
};

template <int BN>
struct AssignSmem {
    float a[A_STAGES][A_BM * A_LD];
    float b[A_STAGES][BN * A_LD];
    float red[4];
    float best[A_BM];
    float second[A_BM];
    int idx[A_BM];
    int lab[A_BM];
};

template <int BN, bool VEC4>
__device__ __forceinline__ void assign_load_tile(AssignSmem<BN> &sm, int stage, const AssignParams &p,
                                                 int64_t row0, int chunk, int k0, int tid)
{
    float *As = sm.a[stage];
    float *Bs = sm.b[stage];
    if (VEC4) {
#pragma unroll
        for (int q = 0; q < (A_BM * A_BK / 4) / A_THREADS; ++q) {
            int e = tid + q * A_THREADS;
            int r = e >> 2, c4 = e & 3;
            int col = k0 + c4 * 4;
            int64_t row = row0 + r;
            bool ok = (row < p.N) && (col < p.D);
            const float *src = ok ? (p.Y + (size_t)row * p.D + col) : p.Y;
            cp_async16(As + r * A_LD + c4 * 4, src, ok ? 16 : 0);
        }
        for (int e = tid; e < BN * A_BK / 4; e += A_THREADS) {
            int n = e >> 2, c4 = e & 3;
            int col = k0 + c4 * 4;
            int k = chunk * BN + n;
            bool ok = (k < p.K) && (col < p.D);
            const float *src = ok ? (p.C + (size_t)k * p.D + col) : p.C;
            cp_async16(Bs + n * A_LD + c4 * 4, src, ok ? 16 : 0);
        }
    } else {
        for (int e = tid; e < A_BM * A_BK; e += A_THREADS) {
            int r = e / A_BK, c = e % A_BK;
            int col = k0 + c;
            int64_t row = row0 + r;
            As[r * A_LD + c] = (row < p.N && col < p.D) ? p.Y[(size_t)row * p.D + col] : 0.f;
        }
        for (int e = tid; e < BN * A_BK; e += A_THREADS) {
            int n = e / A_BK, c = e % A_BK;
            int col = k0 + c;
            int k = chunk * BN + n;
            Bs[n * A_LD + c] = (k < p.K && col < p.D) ? p.C[(size_t)k * p.D + col] : 0.f;
        }
    }
}

// BN centroids per chunk, 8 per thread; TX = BN/8 threads share a row; each thread owns
// TM = TX rows (row = ty + TY*i) so that a CTA always covers 128 rows.
template <int BN, bool VEC4, bool AFFINE>
__global__ void __launch_bounds__(A_THREADS) assign_kernel(AssignParams p)
{
    const int over = p.settled ? *p.settled : 0;
    constexpr int TX = BN / 8;
    constexpr int TY = A_THREADS / TX;
    constexpr int TM = A_BM / TY;
    static_assert(TM == TX, "tile shape");

    extern __shared__ __align__(16) unsigned char smem_raw[];
    AssignSmem<BN> &sm = *reinterpret_cast<AssignSmem<BN> *>(smem_raw);

    const int tid = threadIdx.x;
    const int tx = tid % TX;
    const int ty = tid / TX;
    const int64_t row0 = (int64_t)blockIdx.x * A_BM;

    // cmax^2 = max_k ||c_k||^2
    {
        float m = 0.f;
        for (int k = tid; k < p.K; k += A_THREADS) m = fmaxf(m, p.cnorm[k]);
        if (over) return;   // (the word and the norms on their way together)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        if ((tid & 31) == 0) sm.red[tid >> 5] = m;
    }

    const int ktiles = (p.D + A_BK - 1) / A_BK;
    const int nchunks = (p.K + BN - 1) / BN;
    const int T = ktiles * nchunks;

    for (int s = 0; s < A_STAGES - 1; ++s) {
        if (s < T) assign_load_tile<BN, VEC4>(sm, s, p, row0, s / ktiles, (s % ktiles) * A_BK, tid);
        cp_async_commit();
    }

    float acc[TM][8];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;

    float rb1[TM], rb2[TM];
    int ridx[TM];
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        rb1[i] = CUDART_INF_F;
        rb2[i] = CUDART_INF_F;
        ridx[i] = 0;
    }
    float ysq = 0.f;  // ||y_row||^2 of row `tid`, accumulated during the first chunk

    int chunk = 0, kt = 0;
    for (int t = 0; t < T; ++t) {
        cp_async_wait<A_STAGES - 2>();
        __syncthreads();
        {
            int tn = t + A_STAGES - 1;
            if (tn < T)
                assign_load_tile<BN, VEC4>(sm, tn % A_STAGES, p, row0, tn / ktiles,
                                           (tn % ktiles) * A_BK, tid);
            cp_async_commit();
        }
        const float *As = sm.a[t % A_STAGES];
        const float *Bs = sm.b[t % A_STAGES];

        if (chunk == 0) {
#pragma unroll
            for (int kk = 0; kk < A_BK; kk += 4) {
                float4 v = *reinterpret_cast<const float4 *>(As + tid * A_LD + kk);
                ysq = fmaf(v.x, v.x, ysq);
                ysq = fmaf(v.y, v.y, ysq);
                ysq = fmaf(v.z, v.z, ysq);
                ysq = fmaf(v.w, v.w, ysq);
            }
        }

#pragma unroll
        for (int kk = 0; kk < A_BK; kk += 4) {
            float4 a[TM];
#pragma unroll
            for (int i = 0; i < TM; ++i)
                a[i] = *reinterpret_cast<const float4 *>(As + (ty + TY * i) * A_LD + kk);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                float4 b = *reinterpret_cast<const float4 *>(Bs + (tx + TX * j) * A_LD + kk);
#pragma unroll
                for (int i = 0; i < TM; ++i) {
                    acc[i][j] = fmaf(a[i].x, b.x, acc[i][j]);
                    acc[i][j] = fmaf(a[i].y, b.y, acc[i][j]);
                    acc[i][j] = fmaf(a[i].z, b.z, acc[i][j]);
                    acc[i][j] = fmaf(a[i].w, b.w, acc[i][j]);
                }
            }
        }

        if (++kt == ktiles) {
            // scores of this chunk of centroids: t = ||c||^2 - 2 y.c
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                int n = chunk * BN + tx + TX * j;
                float cn = (n < p.K) ? p.cnorm[n] : CUDART_INF_F;
#pragma unroll
                for (int i = 0; i < TM; ++i) {
                    float sc = (n < p.K) ? fmaf(-2.f, acc[i][j], cn) : CUDART_INF_F;
                    if (sc < rb1[i]) {
                        rb2[i] = rb1[i];
                        rb1[i] = sc;
                        ridx[i] = n;
                    } else if (sc < rb2[i]) {
                        rb2[i] = sc;
                    }
                    acc[i][j] = 0.f;
                }
            }
            kt = 0;
            ++chunk;
        }
    }
    cp_async_wait<0>();

    // merge the TX threads that share a row
#pragma unroll
    for (int i = 0; i < TM; ++i) {
#pragma unroll
        for (int o = 1; o < TX; o <<= 1) {
            float ob1 = __shfl_xor_sync(0xffffffffu, rb1[i], o);
            float ob2 = __shfl_xor_sync(0xffffffffu, rb2[i], o);
            int oidx = __shfl_xor_sync(0xffffffffu, ridx[i], o);
            bool take = (ob1 < rb1[i]) || (ob1 == rb1[i] && oidx < ridx[i]);
            float hi = take ? rb1[i] : ob1;  // the larger of the two bests
            rb2[i] = fminf(fminf(rb2[i], ob2), hi);
            if (take) {
                rb1[i] = ob1;
                ridx[i] = oidx;
            }
        }
        if (tx == 0) {
            int r = ty + TY * i;
            sm.best[r] = rb1[i];
            sm.second[r] = rb2[i];
            sm.idx[r] = ridx[i];
        }
    }
    __syncthreads();

    {
        const float cmax2 = fmaxf(fmaxf(sm.red[0], sm.red[1]), fmaxf(sm.red[2], sm.red[3]));
        const int64_t row = row0 + tid;
        int lab = -1;
        if (row < p.N) {
            const float u = 5.9604645e-8f;  // 2^-24
            float e = 1.0625f * u *
                      ((2.f * (float)p.D + 4.f) * sqrtf(ysq) * sqrtf(cmax2) + 4.f * cmax2);
            float gap = sm.second[tid] - sm.best[tid];
            int k = sm.idx[tid];
            bool certain = (p.K == 1) || (gap > 2.f * e);
            p.labels[row] = k;
            if (p.fast.best) p.fast.best[row] = sm.best[tid];
            if (p.fast.second) p.fast.second[row] = sm.second[tid];
            if (p.fast.bound) p.fast.bound[row] = e;
            if (p.fast.label) p.fast.label[row] = k;
            if (certain) {
                lab = k;
            } else {
                int slot = atomicAdd(&p.ctl->refine_count, 1);
                p.refine_rows[slot] = (int32_t)row;
            }
        }
        sm.lab[tid] = lab;
    }

    if (AFFINE) {
        __syncthreads();
        if (VEC4) {
            const int D4 = p.D >> 2;
            const float4 *Y4 = reinterpret_cast<const float4 *>(p.Y);
            const float4 *G4 = reinterpret_cast<const float4 *>(p.gamma);
            const float4 *B4 = reinterpret_cast<const float4 *>(p.beta);
            float4 *O4 = reinterpret_cast<float4 *>(p.out);
            for (int r = 0; r < A_BM; r += 4) {
                for (int c = tid; c < D4; c += A_THREADS) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        int l = sm.lab[r + q];
                        if (l < 0) continue;
                        size_t o = (size_t)(row0 + r + q) * D4 + c;
                        float4 y = __ldcs(Y4 + o);
                        float4 g = __ldg(G4 + (size_t)l * D4 + c);
                        float4 b = __ldg(B4 + (size_t)l * D4 + c);
                        float4 v;
                        v.x = fmaf(g.x, y.x, b.x);
                        v.y = fmaf(g.y, y.y, b.y);
                        v.z = fmaf(g.z, y.z, b.z);
                        v.w = fmaf(g.w, y.w, b.w);
                        __stcs(O4 + o, v);
                    }
                }
            }
        } else {
            for (int r = 0; r < A_BM; ++r) {
                int l = sm.lab[r];
                if (l < 0) continue;
                size_t o = (size_t)(row0 + r) * p.D;
                for (int c = tid; c < p.D; c += A_THREADS)
                    p.out[o + c] = fmaf(p.gamma[(size_t)l * p.D + c], p.Y[o + c],
                                        p.beta[(size_t)l * p.D + c]);
            }
        }
    }
}

template <int BN, bool VEC4, bool AFFINE>
static cudaError_t launch_assign_t(const AssignParams &p, cudaStream_t s)
{
    auto kern = assign_kernel<BN, VEC4, AFFINE>;
    size_t smem = sizeof(AssignSmem<BN>);
    static bool configured[kMaxDevices] = {};  // the attribute is kept per device
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) dev = -1;
    if (dev < 0 || !configured[dev]) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
        if (e != cudaSuccess) return e;
        if (dev >= 0) configured[dev] = true;
    }
    unsigned blocks = (unsigned)((p.N + A_BM - 1) / A_BM);
    kern<<<blocks, A_THREADS, smem, s>>>(p);
    count_launch();
    return cudaGetLastError();
}

template <bool VEC4, bool AFFINE>
static cudaError_t launch_assign_bn(const AssignParams &p, cudaStream_t s)
{
    if (p.K <= 8) return launch_assign_t<8, VEC4, AFFINE>(p, s);
    if (p.K <= 16) return launch_assign_t<16, VEC4, AFFINE>(p, s);
    if (p.K <= 32) return launch_assign_t<32, VEC4, AFFINE>(p, s);
    return launch_assign_t<64, VEC4, AFFINE>(p, s);
}

cudaError_t launch_assign(const float *Y, int64_t N, int D, int K, const float *C,
                          const float *cnorm, int32_t *labels, int32_t *refine_rows, Control *ctl,
                          const float *gamma, const float *beta, float *out, cudaStream_t s,
                          const FastOut *fast, const int32_t *settled)
{
    AssignParams p{Y, C, cnorm, labels, refine_rows, ctl, gamma, beta, out, N, D, K, fast ? *fast : FastOut{}, settled};
    const bool vec = (D % 4 == 0);
    const bool affine = (out != nullptr);
    if (vec) return affine ? launch_assign_bn<true, true>(p, s) : launch_assign_bn<true, false>(p, s);
    return affine ? launch_assign_bn<false, true>(p, s) : launch_assign_bn<false, false>(p, s);
}

// ======================================================================================
// exact decision for queued rows
// ======================================================================================

constexpr int R_THREADS = 256;
constexpr int R_WARPS = R_THREADS / 32;

__device__ __forceinline__ double exact_distance(const float *y, const float *__restrict__ c, int D, int lane)
{
    double s0 = 0.0, s1 = 0.0;
    int j = lane;
#pragma unroll 2
    for (; j + 32 < D; j += 64) {
        const double d0 = (double)y[j] - (double)c[j], d1 = (double)y[j + 32] - (double)c[j + 32];
        s0 = fma(d0, d0, s0);
        s1 = fma(d1, d1, s1);
    }
    if (j < D) {
        const double d0 = (double)y[j] - (double)c[j];
        s0 = fma(d0, d0, s0);
    }
    return warp_sum(s0 + s1);
}

// Scan of all K centroids for RG queued rows per CTA at a time.  The rows sit in shared memory; a warp forms
// the fp32 direct-form distances of eight rows to four centroids together (12 operand loads for 32 sums, all of
// a step's centroid loads in flight), then a warp per row takes the smallest and settles what lies within the
// sums' error of it in fp64, lowest index on equality.  (All distances in fp64, the earlier form, was bound by
// the fp32 to fp64 conversions: this pass took 43 us of a Lloyd round on 50 000 x 1000 logits, K = 32, and
// takes 21 now, with a quarter of the rows left undecided that were before.)
constexpr int RG = 8;
constexpr int RG_MAX_D = 1536;
constexpr size_t RG_MAX_SMEM = (size_t)RG * RG_MAX_D * 4 + (size_t)RG * CAT_MAX_K * 4;

// RT: rows a warp takes at a time; fewer where K alone does not occupy the warps
template <bool VEC, int RT>
__device__ __forceinline__ void refine_distances(const float *ys_all, int ld, const float *__restrict__ C, int D, int K, float *dist_all)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int unit = w; unit < (K + 3) / 4 * (RG / RT); unit += R_WARPS) {
        const int k0 = unit / (RG / RT) * 4, r0 = unit % (RG / RT) * RT;
        const float *ys = ys_all + r0 * ld;
        float *dist = dist_all + r0 * K;
        float acc[RT * 4];
#pragma unroll
        for (int i = 0; i < RT * 4; ++i) acc[i] = 0.f;
        const float *cp[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) cp[q] = C + (size_t)(k0 + q < K ? k0 + q : k0) * D;
        if (VEC) {
#pragma unroll 2
            for (int j = lane; j < (D >> 2); j += 32) {
                float4 cv[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) cv[q] = reinterpret_cast<const float4 *>(cp[q])[j];
#pragma unroll
                for (int r = 0; r < RT; ++r) {
                    const float4 y = reinterpret_cast<const float4 *>(ys + r * ld)[j];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        float a = acc[r * 4 + q], d;
                        d = y.x - cv[q].x; a = fmaf(d, d, a);
                        d = y.y - cv[q].y; a = fmaf(d, d, a);
                        d = y.z - cv[q].z; a = fmaf(d, d, a);
                        d = y.w - cv[q].w; a = fmaf(d, d, a);
                        acc[r * 4 + q] = a;
                    }
                }
            }
        } else {
#pragma unroll 4
            for (int j = lane; j < D; j += 32) {
                float cv[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) cv[q] = cp[q][j];
#pragma unroll
                for (int r = 0; r < RT; ++r) {
                    const float y = ys[r * ld + j];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float d = y - cv[q];
                        acc[r * 4 + q] = fmaf(d, d, acc[r * 4 + q]);
                    }
                }
            }
        }
        if constexpr (RT == 8) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float s = warp_sum16(acc + 16 * h, lane);
                const int r = 4 * h + (lane >> 3), q = (lane >> 1) & 3;
                if ((lane & 1) == 0 && k0 + q < K) dist[r * K + k0 + q] = s;
            }
        } else {
#pragma unroll
            for (int i = 0; i < RT * 4; ++i) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], o);
                if (lane == 0 && k0 + (i & 3) < K) dist[(i >> 2) * K + k0 + (i & 3)] = acc[i];
            }
        }
    }
}

template <bool VEC>
__device__ __forceinline__ void refine_distances(const float *ys, int ld, const float *__restrict__ C, int D, int K, float *dist)
{
    if (K > 16) refine_distances<VEC, 8>(ys, ld, C, D, K, dist);
    else if (K > 4) refine_distances<VEC, 2>(ys, ld, C, D, K, dist);
    else refine_distances<VEC, 1>(ys, ld, C, D, K, dist);
}

// The counters behind an assignment that has queued `count` rows for the full exact pass (the candidate pass, if any, has
// already added its rows).  (Behind a fixed point nothing
// runs: the assignments there would have queued the rows of the one before them.)
__device__ __forceinline__ void count_refined(Control *ctl, int count)
{
    const bool over = ctl->settled;
    const int64_t last = ctl->refined_last, total = ctl->refined_total;
    ctl->refined_total = total + (over ? last : count);
    if (!over) ctl->refined_last = count + ctl->cand_count;
}

template <bool AFFINE>
__device__ __forceinline__ void refine_body_grouped(const float *__restrict__ Y, int64_t N, int D, int K,
                                                    const float *__restrict__ C, int32_t *labels,
                                                    const int32_t *__restrict__ refine_rows, Control *ctl,
                                                    const float *gamma, const float *beta, float *out, float *ys)
{
    int count = ctl->refine_count;
    if ((int64_t)count > N) count = (int)N;
    if (blockIdx.x == 0 && threadIdx.x == 0) count_refined(ctl, count);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int ld = (D + 3) & ~3;
    float *dist = ys + RG * ld;   // [RG][K]
    const bool vec4 = (D & 3) == 0 && ((reinterpret_cast<uintptr_t>(Y) | reinterpret_cast<uintptr_t>(C)) & 15u) == 0;
    static_assert(RG == R_WARPS, "a warp per row of the group");
    for (int base = blockIdx.x * RG; base < count; base += gridDim.x * RG) {
        // this warp's row
        int64_t row = base + w < count ? (int64_t)refine_rows[base + w] : -1;
        if (row >= N) row = -1;
        float *y = ys + w * ld;
        if (vec4) {
#pragma unroll 4
            for (int j = lane; j < (D >> 2); j += 32)
                reinterpret_cast<float4 *>(y)[j] =
                    row >= 0 ? __ldg(reinterpret_cast<const float4 *>(Y + (size_t)row * D) + j) : make_float4(0.f, 0.f, 0.f, 0.f);
        } else {
#pragma unroll 8
            for (int j = lane; j < D; j += 32) y[j] = row >= 0 ? __ldg(Y + (size_t)row * D + j) : 0.f;
        }
        __syncthreads();
        if (vec4) refine_distances<true>(ys, ld, C, D, K, dist);
        else refine_distances<false>(ys, ld, C, D, K, dist);
        __syncthreads();
        if (row >= 0) {
            const float *d = dist + w * K;
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
                double b64 = CUDART_INF;
                if (l < 0) l = 0;   // only when every distance is NaN
                for (int b = 0; b < K; b += 32)
                    for (uint32_t m = __ballot_sync(0xffffffffu, b + lane < K && !(d[b + lane < K ? b + lane : 0] > lim)); m; m &= m - 1) {
                        const int k = b + __ffs(m) - 1;
                        const double v = exact_distance(y, C + (size_t)k * D, D, lane);
                        if (v < b64) {
                            b64 = v;
                            l = k;
                        }
                    }
            }
            if (lane == 0) labels[row] = l;
            if (AFFINE) {
                const float *g = gamma + (size_t)l * D;
                const float *bb = beta + (size_t)l * D;
                float *o = out + (size_t)row * D;
#pragma unroll 4
                for (int j = lane; j < D; j += 32) o[j] = fmaf(g[j], y[j], bb[j]);
            }
        }
        __syncthreads();
    }
}

// One CTA per queued row (rows too long for the form above): warp w evaluates centroids w, w + 8, ... in
// direct form with fp64 accumulation; the CTA then takes the smallest distance, lowest index on equality.
template <bool AFFINE>
__device__ __forceinline__ void refine_body(const float *__restrict__ Y, int64_t N, int D, int K,
                                            const float *__restrict__ C, int32_t *labels,
                                            const int32_t *__restrict__ refine_rows, Control *ctl,
                                            const float *gamma, const float *beta, float *out)
{
    __shared__ double s_best[R_WARPS];
    __shared__ int s_idx[R_WARPS];
    __shared__ int s_label;
    int count = ctl->refine_count;
    if ((int64_t)count > N) count = (int)N;
    if (blockIdx.x == 0 && threadIdx.x == 0) count_refined(ctl, count);
    const int lane = threadIdx.x & 31;
    const int w = threadIdx.x >> 5;
    for (int it = blockIdx.x; it < count; it += gridDim.x) {
        int64_t row = refine_rows[it];
        if (row < 0 || row >= N) continue;  // uniform across the CTA
        const float *y = Y + (size_t)row * D;
        double best = CUDART_INF;
        int bk = K;  // "none": loses every comparison below
        for (int k = w; k < K; k += R_WARPS) {
            const float *c = C + (size_t)k * D;
            double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
            int j = lane;
            for (; j + 96 < D; j += 128) {
                double d0 = (double)y[j] - (double)c[j];
                double d1 = (double)y[j + 32] - (double)c[j + 32];
                double d2 = (double)y[j + 64] - (double)c[j + 64];
                double d3 = (double)y[j + 96] - (double)c[j + 96];
                s0 = fma(d0, d0, s0);
                s1 = fma(d1, d1, s1);
                s2 = fma(d2, d2, s2);
                s3 = fma(d3, d3, s3);
            }
            for (; j < D; j += 32) {
                double d0 = (double)y[j] - (double)c[j];
                s0 = fma(d0, d0, s0);
            }
            double s = warp_sum((s0 + s1) + (s2 + s3));
            if (s < best) {
                best = s;
                bk = k;
            }
        }
        if (lane == 0) {
            s_best[w] = best;
            s_idx[w] = bk;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            double b = s_best[0];
            int k = s_idx[0];
#pragma unroll
            for (int q = 1; q < R_WARPS; ++q) {
                if (s_best[q] < b || (s_best[q] == b && s_idx[q] < k)) {
                    b = s_best[q];
                    k = s_idx[q];
                }
            }
            if (k >= K) k = 0;  // only when every distance is NaN
            labels[row] = k;
            s_label = k;
        }
        __syncthreads();
        if (AFFINE) {
            const int l = s_label;
            const float *g = gamma + (size_t)l * D;
            const float *bb = beta + (size_t)l * D;
            float *o = out + (size_t)row * D;
            for (int j = threadIdx.x; j < D; j += R_THREADS) o[j] = fmaf(g[j], y[j], bb[j]);
        }
        __syncthreads();
    }
}

// GROUPED: rows of at most RG_MAX_D columns.  (A kernel of its own for longer ones: the grouped form's 128 registers
// a thread would leave two CTAs per SM where the other fits five, and its scan lives on loads in flight.)
template <bool AFFINE, bool GROUPED>
__global__ void __launch_bounds__(R_THREADS) refine_kernel(const float *__restrict__ Y, int64_t N,
                                                           int D, int K, const float *__restrict__ C,
                                                           int32_t *labels,
                                                           const int32_t *__restrict__ refine_rows,
                                                           Control *ctl, const float *gamma,
                                                           const float *beta, float *out)
{
    extern __shared__ __align__(16) float refine_rows_f32[];
    if constexpr (GROUPED) refine_body_grouped<AFFINE>(Y, N, D, K, C, labels, refine_rows, ctl, gamma, beta, out, refine_rows_f32);
    else refine_body<AFFINE>(Y, N, D, K, C, labels, refine_rows, ctl, gamma, beta, out);
}

// dynamic shared memory of the full-K exact pass: RG rows and their distances where the grouped form applies
static size_t refine_smem_bytes(int D, int K) { return D <= RG_MAX_D ? (size_t)RG * ((D + 3) & ~3) * 4 + (size_t)RG * K * 4 : 0; }

template <typename Kern>
static cudaError_t refine_config(Kern kern, size_t smem)   // (the same value whatever the shape: several threads may be launching)
{
    if (smem <= 48 * 1024) return cudaSuccess;   // (what any kernel may have; the call costs the host a microsecond)
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RG_MAX_SMEM);
}

cudaError_t launch_refine(const float *Y, int64_t N, int D, int K, const float *C,
                          int32_t *labels, const int32_t *refine_rows, Control *ctl,
                          const float *gamma, const float *beta, float *out, cudaStream_t s)
{
    const bool grouped = D <= RG_MAX_D;
    const int blocks = (int)(N < 1184 ? N : 1184);
    const auto kern = out ? (grouped ? refine_kernel<true, true> : refine_kernel<true, false>)
                          : (grouped ? refine_kernel<false, true> : refine_kernel<false, false>);
    const size_t smem = refine_smem_bytes(D, K);
    const cudaError_t e = refine_config(kern, smem);
    if (e != cudaSuccess) return e;
    kern<<<blocks, R_THREADS, smem, s>>>(Y, N, D, K, C, labels, refine_rows, ctl, gamma, beta, out);
    count_launch();
    return cudaGetLastError();
}

// Exact decision among at most four listed candidates: one warp per queued row, the
// candidates' fp64 direct-form distances formed together (the row is read once).
constexpr int RC_THREADS = 256;

template <bool AFFINE>
__device__ __forceinline__ void refine_candidates_body(
    const float *__restrict__ Y, int64_t N, int D, int K, const float *__restrict__ C, int32_t *labels,
    const int32_t *__restrict__ cand_rows, const uint64_t *__restrict__ cand_list, Control *ctl,
    const float *gamma, const float *beta, float *out, bool fast_output_valid)
{
    int count = ctl->cand_count;
    if ((int64_t)count > N) count = (int)N;
    if (blockIdx.x == 0 && threadIdx.x == 0) ctl->refined_total += count;
    const int lane = threadIdx.x & 31;
    const bool vec4 = (D & 3) == 0 && ((reinterpret_cast<uintptr_t>(Y) | reinterpret_cast<uintptr_t>(C)) & 15u) == 0 &&
                      (!AFFINE || ((reinterpret_cast<uintptr_t>(gamma) | reinterpret_cast<uintptr_t>(beta) |
                                    reinterpret_cast<uintptr_t>(out)) & 15u) == 0);
    const int gw = blockIdx.x * (RC_THREADS / 32) + (threadIdx.x >> 5);
    const int nw = gridDim.x * (RC_THREADS / 32);
    // A warp walks its rows one after the other, and each row is a chain of dependent loads (queue
    // entry -> row and centroids -> label): the queue entry of the warp's next row is fetched while
    // this row is worked on, and the row's fast label is requested together with its data.
    int64_t next_row = (gw < count) ? (int64_t)cand_rows[gw] : -1;
    uint64_t next_packed = (gw < count) ? cand_list[gw] : 0;
    for (int it = gw; it < count; it += nw) {
        const int64_t row = next_row;
        const uint64_t packed = next_packed;
        if (it + nw < count) {
            next_row = cand_rows[it + nw];
            next_packed = cand_list[it + nw];
        }
        if (row < 0 || row >= N) continue;
        const int fast = labels[row];
        int cand[4];
        const float *cp[4];
        int ncand = 0;   // the list is filled from the front: unused slots are at the end
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            int k = (int)((packed >> (16 * q)) & 0xFFFFu);
            cand[q] = (k < K) ? k : -1;
            cp[q] = C + (size_t)(k < K ? k : 0) * D;
            if (k < K) ncand = q + 1;
        }
        const float *y = Y + (size_t)row * D;
        float s[4] = {0.f, 0.f, 0.f, 0.f};
        if (vec4) {
            // rows and centroids as 128-bit loads (D a multiple of 4, bases 16-byte aligned)
            const float4 *y4 = reinterpret_cast<const float4 *>(y);
            const int D4 = D >> 2;
            if (ncand <= 2) {
                const float4 *c0 = reinterpret_cast<const float4 *>(cp[0]);
                const float4 *c1 = reinterpret_cast<const float4 *>(cp[1]);
                // (unrolled so that the loads of several steps are in flight together: one warp walks
                // its row alone, and a step that waited for its own loads cost a memory latency each)
#pragma unroll 8
                for (int j = lane; j < D4; j += 32) {
                    const float4 yv = y4[j], a = c0[j], b = c1[j];
                    float d;
                    d = yv.x - a.x; s[0] = fmaf(d, d, s[0]);
                    d = yv.y - a.y; s[0] = fmaf(d, d, s[0]);
                    d = yv.z - a.z; s[0] = fmaf(d, d, s[0]);
                    d = yv.w - a.w; s[0] = fmaf(d, d, s[0]);
                    d = yv.x - b.x; s[1] = fmaf(d, d, s[1]);
                    d = yv.y - b.y; s[1] = fmaf(d, d, s[1]);
                    d = yv.z - b.z; s[1] = fmaf(d, d, s[1]);
                    d = yv.w - b.w; s[1] = fmaf(d, d, s[1]);
                }
            } else {
#pragma unroll 4
                for (int j = lane; j < D4; j += 32) {
                    const float4 yv = y4[j];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float4 c = reinterpret_cast<const float4 *>(cp[q])[j];
                        float d;
                        d = yv.x - c.x; s[q] = fmaf(d, d, s[q]);
                        d = yv.y - c.y; s[q] = fmaf(d, d, s[q]);
                        d = yv.z - c.z; s[q] = fmaf(d, d, s[q]);
                        d = yv.w - c.w; s[q] = fmaf(d, d, s[q]);
                    }
                }
            }
        } else {
#pragma unroll 8
            for (int j = lane; j < D; j += 32) {
                const float yv = y[j];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float d = yv - cp[q][j];
                    s[q] = fmaf(d, d, s[q]);
                }
            }
        }
        // fp32 sums first; what lies within their error of the smallest is settled in fp64
        float fbest = CUDART_INF_F;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s[q] += __shfl_xor_sync(0xffffffffu, s[q], o);
            if (cand[q] >= 0) fbest = fminf(fbest, s[q]);
        }
        const float lim = fp32_sum_limit(fbest, D);
        int left = 0, bk = K;
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (cand[q] >= 0 && !(s[q] > lim)) {
                ++left;
                bk = cand[q];
            }
        if (left != 1) {
            double best = CUDART_INF;
            bk = K;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (cand[q] < 0 || s[q] > lim) continue;
                const double v = exact_distance(y, cp[q], D, lane);
                if (v < best || (v == best && cand[q] < bk)) {
                    best = v;
                    bk = cand[q];
                }
            }
        }
        if (bk >= K) bk = (cand[0] >= 0) ? cand[0] : 0;   // only when every distance is NaN
        // The fast pass has already written this row's output with the label it left in
        // labels[row] (read above); the row is rewritten only when the exact label differs.
        __syncwarp();
        if (lane == 0) labels[row] = bk;
        if (AFFINE && (bk != fast || !fast_output_valid)) {
            const float *g = gamma + (size_t)bk * D;
            const float *bb = beta + (size_t)bk * D;
            float *o = out + (size_t)row * D;
            if (vec4) {
                for (int j = lane; j < (D >> 2); j += 32) {
                    const float4 yv = reinterpret_cast<const float4 *>(y)[j];
                    const float4 gv = reinterpret_cast<const float4 *>(g)[j];
                    const float4 bv = reinterpret_cast<const float4 *>(bb)[j];
                    reinterpret_cast<float4 *>(o)[j] = make_float4(fmaf(gv.x, yv.x, bv.x), fmaf(gv.y, yv.y, bv.y),
                                                                   fmaf(gv.z, yv.z, bv.z), fmaf(gv.w, yv.w, bv.w));
                }
            } else {
                for (int j = lane; j < D; j += 32) o[j] = fmaf(g[j], y[j], bb[j]);
            }
        }
    }
}

// Both exact passes in one launch: the rows queued with their candidates (a warp each), then the
// rows queued for a scan of all K (a CTA each).  A row is in one queue only.
static_assert(RC_THREADS == R_THREADS, "the fused exact pass runs both bodies with one block size");
template <bool AFFINE, bool GROUPED>
__global__ void __launch_bounds__(R_THREADS) refine_both_kernel(
    const float *__restrict__ Y, int64_t N, int D, int K, const float *__restrict__ C, int32_t *labels,
    const int32_t *__restrict__ cand_rows, const uint64_t *__restrict__ cand_list,
    const int32_t *__restrict__ refine_rows, Control *ctl, const float *gamma, const float *beta, float *out)
{
    pdl_enter();
    refine_candidates_body<AFFINE>(Y, N, D, K, C, labels, cand_rows, cand_list, ctl, gamma, beta, out, AFFINE);
    __syncthreads();   // (block 0's thread 0 updates the counters in both bodies, in this order)
    extern __shared__ __align__(16) float refine_rows_f32[];
    if constexpr (GROUPED) refine_body_grouped<AFFINE>(Y, N, D, K, C, labels, refine_rows, ctl, gamma, beta, out, refine_rows_f32);
    else refine_body<AFFINE>(Y, N, D, K, C, labels, refine_rows, ctl, gamma, beta, out);
}

cudaError_t launch_refine_both(const float *Y, int64_t N, int D, int K, const float *C, int32_t *labels,
                               const int32_t *cand_rows, const uint64_t *cand_list, const int32_t *refine_rows,
                               Control *ctl, const float *gamma, const float *beta, float *out, cudaStream_t s)
{
    int64_t want = (N + (RC_THREADS / 32) - 1) / (RC_THREADS / 32);
    const bool grouped = D <= RG_MAX_D;
    const int blocks = (int)(want < 1184 ? want : 1184);
    const auto kern = out ? (grouped ? refine_both_kernel<true, true> : refine_both_kernel<true, false>)
                          : (grouped ? refine_both_kernel<false, true> : refine_both_kernel<false, false>);
    const size_t smem = refine_smem_bytes(D, K);
    cudaError_t e = refine_config(kern, smem);
    if (e != cudaSuccess) return e;
    e = launch_pdl(kern, dim3(blocks), dim3(R_THREADS), smem, s, Y, N, D, K, C, labels, cand_rows, cand_list, refine_rows, ctl, gamma, beta,
                   out);
    if (e != cudaSuccess) return e;
    count_launch();
    return cudaGetLastError();
}

// ======================================================================================
// element-wise kernels
// ======================================================================================

__global__ void centroids_from_sums_kernel(const double *__restrict__ sums,
                                           const int64_t *__restrict__ counts, int D, size_t KD,
                                           float *__restrict__ C)
{
    size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= KD) return;
    int64_t n = counts[e / D];
    if (n > 0) C[e] = (float)(sums[e] / (double)n);
}

cudaError_t launch_centroids_from_sums(const double *sums, const int64_t *counts, int D, int K,
                                       float *C, cudaStream_t s)
{
    size_t KD = (size_t)K * D;
    int threads = 256;
    unsigned blocks = (unsigned)((KD + threads - 1) / threads);
    centroids_from_sums_kernel<<<blocks, threads, 0, s>>>(sums, counts, D, KD, C);
    count_launch();
    return cudaGetLastError();
}

// one block per cluster: the cluster's size first (by thread 0, before anyone reads it), then its columns
__global__ void shard_update_kernel(const double *__restrict__ dsums, const int64_t *__restrict__ dcounts, int D,
                                    double *__restrict__ sums, int64_t *__restrict__ counts, float *__restrict__ C)
{
    __shared__ long long n_s;
    const int k = blockIdx.x;
    if (threadIdx.x == 0) {
        const long long n = (long long)counts[k] + (long long)dcounts[k];
        counts[k] = n;
        n_s = n;
    }
    __syncthreads();
    const long long n = n_s;
    for (int j = threadIdx.x; j < D; j += blockDim.x) {
        const size_t e = (size_t)k * D + j;
        const double a = sums[e] + dsums[e];
        sums[e] = a;
        if (n > 0) C[e] = (float)(a / (double)n);
    }
}

cudaError_t launch_shard_update(const double *delta_sums, const int64_t *delta_counts, int D, int K, double *sums,
                                int64_t *counts, float *C, cudaStream_t s)
{
    shard_update_kernel<<<K, 256, 0, s>>>(delta_sums, delta_counts, D, sums, counts, C);
    count_launch();
    return cudaGetLastError();
}

__global__ void means_from_sums_kernel(const double *__restrict__ sums,
                                       const int64_t *__restrict__ counts, int D, size_t KD,
                                       double *__restrict__ mean)
{
    size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= KD) return;
    int64_t n = counts[e / D];
    mean[e] = (n > 0) ? sums[e] / (double)n : 0.0;
}

cudaError_t launch_means_from_sums(const double *sums, const int64_t *counts, int D, int K,
                                   double *mean, cudaStream_t s)
{
    size_t KD = (size_t)K * D;
    int threads = 256;
    unsigned blocks = (unsigned)((KD + threads - 1) / threads);
    means_from_sums_kernel<<<blocks, threads, 0, s>>>(sums, counts, D, KD, mean);
    count_launch();
    return cudaGetLastError();
}

// gamma = (cov/n) / max(var/n, 1e-8), beta = muF - gamma*muQ; empty cluster -> (1, 0).
__global__ void solve_kernel(const double *__restrict__ sumQ, const double *__restrict__ sumF,
                             const double *__restrict__ var, const double *__restrict__ cov,
                             const int64_t *__restrict__ counts, int D, size_t KD,
                             float *__restrict__ gamma, float *__restrict__ beta)
{
    size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= KD) return;
    int64_t n = counts[e / D];
    if (n <= 0) {
        gamma[e] = 1.f;
        beta[e] = 0.f;
        return;
    }
    double dn = (double)n;
    double v = var[e] / dn;
    double c = cov[e] / dn;
    if (v < 1e-8) v = 1e-8;
    double g = c / v;
    double b = sumF[e] / dn - g * (sumQ[e] / dn);
    gamma[e] = (float)g;
    beta[e] = (float)b;
}

cudaError_t launch_solve(const double *sumQ, const double *sumF, const double *var,
                         const double *cov, const int64_t *counts, int D, int K, float *gamma,
                         float *beta, cudaStream_t s)
{
    size_t KD = (size_t)K * D;
    int threads = 256;
    unsigned blocks = (unsigned)((KD + threads - 1) / threads);
    solve_kernel<<<blocks, threads, 0, s>>>(sumQ, sumF, var, cov, counts, D, KD, gamma, beta);
    count_launch();
    return cudaGetLastError();
}

// gamma' = 1 + alpha (gamma - 1), beta' = alpha beta  (so that gamma' y + beta' is the blend)
__global__ void blend_params_kernel(const float *__restrict__ gamma, const float *__restrict__ beta,
                                    double alpha, size_t KD, float *__restrict__ gb,
                                    float *__restrict__ bb)
{
    size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= KD) return;
    gb[e] = (float)(1.0 + alpha * ((double)gamma[e] - 1.0));
    bb[e] = (float)(alpha * (double)beta[e]);
}

cudaError_t launch_blend_params(const float *gamma, const float *beta, float alpha, int64_t KD,
                                float *gamma_b, float *beta_b, cudaStream_t s)
{
    int threads = 256;
    unsigned blocks = (unsigned)((KD + threads - 1) / threads);
    blend_params_kernel<<<blocks, threads, 0, s>>>(gamma, beta, (double)alpha, (size_t)KD, gamma_b,
                                                   beta_b);
    count_launch();
    return cudaGetLastError();
}

__global__ void fit_diag_kernel(const Control *ctl, const int64_t *counts, int K,
                                cat_fit_diag_t *diag)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    int64_t empty = 0;
    for (int k = 0; k < K; ++k) empty += (counts[k] == 0);
    diag->refined_rows_total = ctl->refined_total;
    diag->refined_rows_final = ctl->refined_last;
    diag->empty_clusters_final = empty;
    diag->device_status = ctl->device_status;
}

cudaError_t launch_fit_diag(const Control *ctl, const int64_t *counts, int K, cat_fit_diag_t *diag,
                            cudaStream_t s)
{
    fit_diag_kernel<<<1, 32, 0, s>>>(ctl, counts, K, diag);
    count_launch();
    return cudaGetLastError();
}

// ---- per-assignment diagnostics (only when the caller asks for them)

// objective += sum over rows of ||y - c_label||^2 (fp64, one warp per row, one atomic per block)
__global__ void __launch_bounds__(256) diag_objective_kernel(const float *__restrict__ Y, int64_t N, int D,
                                                             const float *__restrict__ C,
                                                             const int32_t *__restrict__ labels, double *objective)
{
    __shared__ double part[8];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    double acc = 0.0;
    for (int64_t row = (int64_t)blockIdx.x * 8 + w; row < N; row += (int64_t)gridDim.x * 8) {
        const float *y = Y + (size_t)row * D;
        const float *c = C + (size_t)labels[row] * D;
        double s = 0.0;
        for (int j = lane; j < D; j += 32) {
            const double d = (double)y[j] - (double)c[j];
            s = fma(d, d, s);
        }
        acc += warp_sum(s);
    }
    if (lane == 0) part[w] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int q = 0; q < 8; ++q) t += part[q];
        atomicAdd(objective, t);
    }
}

// Rows of the two exact-pass queues whose two nearest centroids are within 1e-6 relative of each
// other in squared distance (fp64 direct form over all K): one warp per queued row.
__global__ void __launch_bounds__(256) diag_near_kernel(const float *__restrict__ Y, int64_t N, int D, int K,
                                                        const float *__restrict__ C,
                                                        const int32_t *__restrict__ refine_rows,
                                                        const int32_t *__restrict__ cand_rows, const Control *ctl,
                                                        long long *near_out)
{
    const int lane = threadIdx.x & 31;
    int nref = ctl->refine_count, ncand = ctl->cand_count;
    if ((int64_t)nref > N) nref = (int)N;
    if ((int64_t)ncand > N) ncand = (int)N;
    const int total = nref + ncand;
    int found = 0;
    for (int q = blockIdx.x * 8 + (threadIdx.x >> 5); q < total; q += gridDim.x * 8) {
        const int64_t row = q < nref ? refine_rows[q] : cand_rows[q - nref];
        if (row < 0 || row >= N) continue;
        const float *y = Y + (size_t)row * D;
        double best = CUDART_INF, second = CUDART_INF;
        for (int k = 0; k < K; ++k) {
            const float *c = C + (size_t)k * D;
            double s = 0.0;
            for (int j = lane; j < D; j += 32) {
                const double d = (double)y[j] - (double)c[j];
                s = fma(d, d, s);
            }
            s = warp_sum(s);
            if (s < best) {
                second = best;
                best = s;
            } else if (s < second) {
                second = s;
            }
        }
        if (K > 1 && (second - best) <= 1e-6 * second) ++found;
    }
    if (lane == 0 && found) atomicAdd(reinterpret_cast<unsigned long long *>(near_out), (unsigned long long)found);
}

__global__ void diag_round_begin_kernel(const Control *ctl, int64_t N, cat_fit_diag_t *diag, int slot, int recorded)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    int64_t q = (int64_t)ctl->refine_count + (int64_t)ctl->cand_count;
    diag->undecided_rows[slot] = q < N ? q : N;
    diag->near_tie_rows[slot] = 0;
    diag->objective[slot] = 0.0;
    diag->assignments_recorded = recorded;
}

cudaError_t launch_fit_diag_round(const float *Y, int64_t N, int D, int K, const float *C, const int32_t *labels,
                                  const int32_t *refine_rows, const int32_t *cand_rows, const Control *ctl,
                                  cat_fit_diag_t *diag, int slot, int recorded, cudaStream_t s)
{
    diag_round_begin_kernel<<<1, 32, 0, s>>>(ctl, N, diag, slot, recorded);
    int64_t blocks = (N + 7) / 8;
    if (blocks > 1184) blocks = 1184;
    diag_objective_kernel<<<(unsigned)blocks, 256, 0, s>>>(Y, N, D, C, labels, &diag->objective[slot]);
    diag_near_kernel<<<(unsigned)blocks, 256, 0, s>>>(Y, N, D, K, C, refine_rows, cand_rows, ctl,
                                                      reinterpret_cast<long long *>(&diag->near_tie_rows[slot]));
    count_launch(3);
    return cudaGetLastError();
}

__global__ void reset_control_kernel(Control *ctl)
{
    pdl_enter();
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        ctl->refine_count = 0;
        ctl->cand_count = 0;
        ctl->device_status = CAT_OK;
        ctl->refined_total = 0;
        ctl->refined_last = 0;
        ctl->grid_bar = 0;
        ctl->settled = 0;
    }
}

__global__ void absorb_control_kernel(Control *ctl, const Control *from)
{
    pdl_enter();
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        if (ctl->device_status == CAT_OK) ctl->device_status = from->device_status;
        ctl->refined_total += from->refined_total;
        ctl->refined_last = from->refined_last;
    }
}

cudaError_t launch_absorb_control(Control *ctl, const Control *from, cudaStream_t s)
{
    const cudaError_t e = launch_pdl(absorb_control_kernel, dim3(1), dim3(32), 0, s, ctl, from);
    count_launch();
    return e;
}

cudaError_t launch_reset_control(Control *ctl, cudaStream_t s)
{
    const cudaError_t e = launch_pdl(reset_control_kernel, dim3(1), dim3(32), 0, s, ctl);
    count_launch();
    return e;
}

}  // namespace cat
