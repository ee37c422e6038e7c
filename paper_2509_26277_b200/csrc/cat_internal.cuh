// Internal declarations shared by the translation units of libcat.so.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "cat.h"

namespace cat {

// ---------------------------------------------------------------- launch bookkeeping
extern thread_local int g_last_cuda_error;
void count_launch(int n = 1);

inline bool cuda_ok(cudaError_t e)
{
    if (e != cudaSuccess) {
        g_last_cuda_error = (int)e;
        return false;
    }
    return true;
}

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Programmatic dependent launch for the chains of short kernels (a Lloyd round is seven of them):
// a kernel launched with launch_pdl may be scheduled while the previous kernel of its stream is
// still running, which hides its launch latency.  Such a kernel calls pdl_enter() before anything
// else: it lets its own dependents be scheduled early, then waits until the previous grid has
// completed and its writes are visible -- so the kernels still run in stream order.  Both
// instructions do nothing in a kernel that was launched the ordinary way.
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_enter()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args &&...args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}

// Direct-form fp32 sums of squares whose lanes add D / 32 terms each before a tree adds the lanes have a relative error of
// at most eta = (D / 32 + 12) 2^-24.  Sums above this limit are in the order of the exact ones against `best`; what lies
// within it is settled in fp64.  Sums below 1e-30 may have lost squares to underflow: whatever is that small stays a
// candidate.  (Every exact decision of the library goes by this line.)
__device__ __forceinline__ float fp32_sum_limit(float best, int D)
{
    const float eta = 1.0625f * ((float)D * 0.03125f + 12.f) * 5.9604645e-8f;
    return fmaxf(best, 1e-30f) * (1.f + 2.25f * eta);
}

// Sums of 16 values over the warp, 16 exchanges in place of 80; lanes 2 i and 2 i + 1 end with the sum of acc[i].
__device__ __forceinline__ float warp_sum16(float *acc, int lane)
{
#pragma unroll
    for (int h = 8, o = 16; h > 0; h >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (i < h) {
                const float send = up ? acc[i] : acc[i + h];
                const float keep = up ? acc[i + h] : acc[i];
                acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
    }
    return acc[0] + __shfl_xor_sync(0xffffffffu, acc[0], 1);
}
#endif

// ---------------------------------------------------------------- workspace layouts
// Optional outputs of the fast pass (device pointers, each may be null): see cat_fast_scores_t.
struct FastOut {
    float *best = nullptr;
    float *second = nullptr;
    float *bound = nullptr;
    int32_t *label = nullptr;
};

// Control block at the start of every workspace (device memory).
struct Control {
    int32_t refine_count;        // rows queued for the exact fp64 pass by the current assignment
    int32_t device_status;       // CAT_OK or CAT_ERR_DEVICE_TIMEOUT
    int64_t refined_total;       // running total over assignments
    int64_t refined_last;        // rows of the latest finished assignment that took an exact pass
    int32_t cand_count;          // rows queued with a short candidate list by the current assignment
    uint32_t grid_bar;           // arrival counter of the grid-wide barrier of the persistent small-problem kernel
    int32_t settled;             // a Lloyd round of cat_fit moved no row: the rounds behind it have nothing to do
    int32_t pad32;
    int64_t pad[3];
};

// Geometry of the sort-based segmented sums for NE entries over KK keys (full mode: N rows,
// K labels; delta mode: 2N virtual entries, 2K keys): identical in the workspace query and
// at launch time.
struct SegGeom {
    int nblk;       // 1024-entry blocks of the sort
    int seg_rows;   // largest rows per segment (multiple of 16); a sort may choose shorter segments
    int max_segs;   // upper bound on the number of segments: ceil(NE / seg_rows) + KK
};
SegGeom seg_geometry(int64_t NE, int D, int KK);
int seg_capacity(int64_t NE, int KK);

struct AssignWs {          // what assign/apply need
    Control *ctl;
    float *cnorm;          // [K] squared centroid norms, fp32
    int32_t *refine_rows;  // [N]
    int32_t *labels;       // [N] (used when the caller passes no labels_out)
    float *gamma_b;        // [K*D] blended gamma (alpha != 1)
    float *beta_b;         // [K*D]
    float *ynorm2;         // [N] squared row norms (tensor-core labels-only path)
    int32_t *cand_rows;    // [N] rows queued with candidates
    uint64_t *cand_list;   // [N] their candidates, 4 x 16 bit
    float *cmax;           // [K] largest magnitude of each centroid
    float *cerr;           // [K] norms of the rounding errors of the fp16 centroids
    float *mean;           // [D] what rows and centroids are taken relative to on fp16 operands
    float *cconst;         // [K] squared norms less that of the mean (inference on 64-row tiles)
    void *ch;              // [K][half_ld(D)] fp16 copy of the centroids (inference on fp16 operands)
    float *hscale;         // [4] scale of that copy: {s_c, -2 / s_c, 2^-25 / s_c, -}; with yh followed by [slab] inverse row scales and [slab] rounding errors
    void *prep;            // prepared centroids of the inference kernel that keeps rows in shared memory (or null)
    void *yh;              // [slab][half_ld(D)] fp16 copy of a slab of rows (inference with D % 4 != 0), else null
    size_t bytes;
};
AssignWs carve_assign(void *base, int64_t N, int D, int K);

struct FitWs {
    AssignWs a;
    // sized for delta mode (2N virtual entries, 2K keys)
    uint32_t *blk_hist;    // [nblk][2K] key histogram / offsets of the sort
    uint32_t *key_total;   // [2K] entries per key
    int32_t *cluster_start; // [2K+1] first position of each key in `order`
    int32_t *seg_start;    // [2K+2] first segment of each key, total, segment length of the current sort
    int32_t *order;        // [2N] row indices sorted by key (stable)
    int32_t *labels_prev;  // [N] labels of the previous Lloyd round
    double *segpart;       // [max_segs][2][D] per-segment partial sums
    void *yh;              // [N][half_ld(D)] fp16 copy of Yq (tensor-core fits)
    void *ch;              // [K][half_ld(D)] fp16 copy of the centroids
    float *hscale;         // [4 + 2N] scale of the fp16 centroids, the inverse row scales, the rows' rounding errors
    double *sumQ, *sumF, *var, *cov;   // [K*D] each
    double *meanQ, *meanF;             // [K*D] each
    int64_t *counts;       // [K]
    void *norm_part;       // parts of the centroid norms (centroid update)
    uint32_t *arrivals;    // [K] CTAs of a cluster that have left theirs
    uint64_t *moved_state; // what passes between the CTAs that list moved rows
    double *small_part;    // per-CTA sums of the single-launch fits that keep them in planes (or null)
    int32_t *small_counts; // ... and their counters
    size_t bytes;
};
FitWs carve_fit(void *base, int64_t N, int D, int K);

// K-Means as cat_fit runs it, without the closed form (workspace of cat_fit); and the closed form for given labels (a
// workspace of cat_fit for this shape).
cat_status_t fit_clusters(const float *Y, int64_t N, int D, int K, int iters, float *centroids_out, int32_t *labels_out, void *workspace,
                          size_t workspace_bytes, cudaStream_t s);
cat_status_t fit_closed_form(const float *Yq, const float *Yfp, int64_t N, int D, int K, const int32_t *labels, float *gamma_out,
                             float *beta_out, void *workspace, cudaStream_t s);

// ---------------------------------------------------------------- kernel launchers (cat_kernels.cu)
// All return a cudaError_t from the launch; none synchronises.

// cnorm[k] = ||c_k||^2 (fp64 accumulate, rounded up to fp32); also resets ctl->refine_count,
// and with reset_all the status word and the counters (start of a top-level call).
cudaError_t launch_centroid_norms(const float *C, int D, int K, float *cnorm, Control *ctl,
                                  cudaStream_t s, bool reset_all = false);

// Fast fp32 scores + certainty test; optional fused affine epilogue.
cudaError_t launch_assign(const float *Y, int64_t N, int D, int K, const float *C,
                          const float *cnorm, int32_t *labels, int32_t *refine_rows, Control *ctl,
                          const float *gamma, const float *beta, float *out, cudaStream_t s,
                          const FastOut *fast = nullptr, const int32_t *settled = nullptr);

// Exact fp64 direct-form labels for the queued rows; optional affine output.
cudaError_t launch_refine(const float *Y, int64_t N, int D, int K, const float *C,
                          int32_t *labels, const int32_t *refine_rows, Control *ctl,
                          const float *gamma, const float *beta, float *out, cudaStream_t s);

// Persistent single-launch kernels for small problems (D in {32, 64, 128}, K <= 128): a run of
// Lloyd rounds with the per-cluster sums in registers and a grid-wide combine, and inference.
constexpr int SMALL_MAX_GRID = 160;   // CTAs the partial-sum planes are sized for
bool small_fit_supported(int64_t N, int D, int K);
bool small_apply_supported(int64_t N, int D, int K);
size_t small_part_doubles(int D, int K);
size_t small_part_counts(int K);
cudaError_t launch_small_fit(const float *Y, int64_t N, int D, int K, float *C, int passes, bool update_last,
                             int32_t *labels, double *part, int32_t *part_counts, double *sums, int64_t *counts,
                             Control *ctl, unsigned int *bar_count, cudaStream_t s);
cudaError_t launch_small_apply(const float *Y, int64_t N, int D, int K, const float *C, const float *gamma,
                               const float *beta, float *out, int32_t *labels, Control *ctl, cudaStream_t s);

// The Lloyd rounds of a fit and its final assignment in one cooperative launch, the rows in shared memory
// (cat_fit_rows.cu); ctl must have been reset.  passes = rounds + 1.  list: N 8-byte entries, list_count: 16
// bytes per CTA (four rows of one at least), padded: [K][D rounded up to 4].  Leaves final labels, per-cluster sums and sizes.
bool fit_rows_supported(int64_t N, int D, int K);
cudaError_t launch_fit_rows(const float *Y, int64_t N, int D, int K, float *C, int passes, int32_t *labels, double *sums,
                            int64_t *counts, void *list, void *list_count, float *padded, Control *ctl, cudaStream_t s);

// The same for many rows of few columns, held as fp16 operand fragments (cat_fit_tiles.cu); ctl must have been reset, mean
// is a point among the rows (launch_sample_mean).  part: fit_tiles_part_doubles, part_counts: fit_tiles_counts.
bool fit_tiles_supported(int64_t N, int D, int K);
size_t fit_tiles_part_doubles(int D, int K);   // (0: no such shape whatever N is)
size_t fit_tiles_counts(int K);
cudaError_t launch_fit_tiles(const float *Y, int64_t N, int D, int K, float *C, const float *mean, int passes, int32_t *labels, double *part,
                             int32_t *part_counts, double *sums, int64_t *counts, Control *ctl, cudaStream_t s);

// Inference on rows of 32 to 128 columns that stay in a warp's registers, exact decisions included
// (cat_apply_short.cu); ctl must have been reset.  out_bf16: `out` is a [N, D] bf16 matrix.
bool apply_short_supported(int64_t N, int D, int K);
cudaError_t launch_apply_short(const float *Y, int64_t N, int D, int K, const float *C, const float *gamma, const float *beta, void *out,
                               bool out_bf16, int32_t *labels, Control *ctl, cudaStream_t s);

// Inference on groups of eight rows held in shared memory, exact decisions included (cat_apply_rows.cu).
// Resets ctl.  out_bf16: `out` is a [N, D] bf16 matrix; prep: apply_rows_prep_bytes of scratch.
bool apply_rows_supported(int64_t N, int D, int K);
size_t apply_rows_prep_bytes(int64_t N, int D, int K);
cudaError_t launch_apply_rows(const float *Y, int64_t N, int D, int K, const float *C, const float *gamma, const float *beta,
                              void *out, bool out_bf16, int32_t *labels, Control *ctl, void *prep, cudaStream_t s);

// The same for clusters in a reduced space: C [K][p], labels by z = fp32 of comps (y - mean) (D <= 1024, K <= 64).  open_rows: N
// 16-byte entries of scratch.
bool apply_rows_pca_supported(int64_t N, int D, int K);
size_t apply_rows_pca_prep_bytes(int64_t N, int D, int K);
cudaError_t launch_apply_rows_pca(const float *Y, int64_t N, int D, int K, int p, const float *mean, const float *comps, const float *C,
                                  const float *gamma, const float *beta, float *out, int32_t *labels, Control *ctl, void *prep,
                                  void *open_rows, cudaStream_t s);

// Tensor-core (tcgen05, TF32) variant of launch_assign; ynorm2 is needed when out == nullptr.
bool tc_supported(int64_t N, int D, int K);
// Form of the fused inference kernel on the tensor path: 0 = chosen by shape, 1 = TF32 row tiles
// (128 rows per CTA), 2 / 4 = column split over that many CTAs where it applies, 64 = 64-row tiles
// on fp16 operands made on the fly where that applies.
void set_apply_column_split(int cs);
int get_apply_column_split();
int choose_apply_form(int64_t N, int D, int K);   // 1, 2, 4 or 64 for this shape under the current setting
// 64-row-tile inference kernel on fp16 operands (cat_apply64.cu).  Ch = fp16((C - m) * scale[0]),
// scale = {s_c, -2 / s_c, 2^-25 / s_c, -}, cnorm, cerr and cconst come from launch_centroid_half with m.
bool apply_h64_supported(int64_t N, int D, int K);
cudaError_t launch_half_scale(float *scale, cudaStream_t s);                           // bits of the maximum -> the three scale words
cudaError_t launch_apply_h64(const float *Y, int64_t N, int D, int K, const void *Ch, const float *scale,
                             const float *cnorm, const float *cerr, const float *cconst, int32_t *labels, int32_t *refine_rows,
                             int32_t *cand_rows, uint64_t *cand_list, Control *ctl, const float *gamma, const float *beta, float *out,
                             cudaStream_t s, bool out_bf16 = false);   // out_bf16: `out` is a [N, D] bf16 matrix
// out_bf16[row] = bf16(gamma_l * y + beta_l), l = labels[row]: for all rows (rows == nullptr, n_rows = N) or
// for the listed rows (two lists, lengths read from ctl: the exact-pass queues).
cudaError_t launch_affine_bf16(const float *Y, int64_t N, int D, int K, const int32_t *labels, const float *gamma,
                               const float *beta, void *out_bf16, const int32_t *refine_rows, const int32_t *cand_rows,
                               const Control *ctl, cudaStream_t s);
cudaError_t launch_row_norms(const float *Y, int64_t N, int D, float *out, cudaStream_t s);
// With Yh / Ch / scale (labels only): the fp16 copies of the rows and centroids are the MMA operands.
cudaError_t launch_assign_tc(const float *Y, int64_t N, int D, int K, const float *C, const float *cnorm,
                             const float *ynorm2, int32_t *labels, int32_t *refine_rows,
                             int32_t *cand_rows, uint64_t *cand_list, Control *ctl,
                             const float *gamma, const float *beta, float *out, cudaStream_t s,
                             const void *Yh = nullptr, const void *Ch = nullptr, const float *scale = nullptr,
                             const float *cerr = nullptr, const FastOut *fast = nullptr, int64_t row_base = 0,
                             const int32_t *settled = nullptr);

// One warp waits (at most limit_ms, clamped to 1 .. 1000) on a barrier that is never completed.
cudaError_t launch_wait_selftest(Control *ctl, int limit_ms, cudaStream_t s);

// fp16 copy of a matrix for repeated assignments, made in one sweep, of the rows less `mean` (null: as they
// are): squared row norms, per-row power-of-two scales, Yh[i] = fp16((Y[i] - mean) * scale_i), and
// scale[4 + 2 N] = {centroid scale s_c from the largest magnitude of Y, -2 / s_c, 2^-25 / s_c, unused, then
// 1 / scale_i for every row, then the norm of every row's rounding error}.  Rows of the copies (of the centroids
// too) are half_ld(D) elements apart, so that any row length suits the tensor maps.
__host__ __device__ constexpr int half_ld(int D) { return (D + 7) & ~7; }
constexpr int TC_HALF_MIN_D = 8;
bool tc_half_supported(int64_t N, int D, int K);
// finish_scale = false leaves the bits of the largest magnitude in scale[0] (launch_half_scale turns them
// into the three scale words later, e.g. once the maximum over several shards is known); want_amax = false leaves
// those words alone.
cudaError_t launch_half_shadow(const float *Y, int64_t N, int D, const float *mean, float *ynorm2, float *scale, void *Yh,
                               cudaStream_t s, bool want_amax = true, bool finish_scale = true);
// A point among the rows to take them relative to, from the first 128 (any finite point will do; one that a few stray
// rows do not move keeps the operands small).
cudaError_t launch_sample_mean(const float *Y, int64_t N, int D, float *mean, cudaStream_t s);
// Everything an assignment on fp16 operands needs of the centroids less `mean` (null: as they are): norms,
// the fp16 copy, the norms cerr of its rounding errors, and with own_scale the scale words from their largest
// magnitude (cmax: [K] scratch).  With aconst they are taken less a point m among them instead, which goes to
// `mean`, and aconst is ||c||^2 - ||m||^2.  Empties the exact-pass queues as launch_centroid_norms does.
cudaError_t launch_centroid_half(const float *C, int D, int K, float *mean, float *cnorm, float *cmax, float *cerr, float *scale,
                                 void *Ch, Control *ctl, cudaStream_t s, bool reset_all, bool own_scale = true, float *aconst = nullptr);

// Exact fp64 decision among the listed candidates of each queued row; optional affine output.
cudaError_t launch_refine_both(const float *Y, int64_t N, int D, int K, const float *C, int32_t *labels,
                               const int32_t *cand_rows, const uint64_t *cand_list, const int32_t *refine_rows,
                               Control *ctl, const float *gamma, const float *beta, float *out, cudaStream_t s);

// Stable sort of the row indices by key.  prev == NULL (full mode): key = label, counts[k] = size of
// cluster k.  prev != NULL (delta mode): entries only for rows with labels[i] != prev[i], under keys
// labels[i] and K + prev[i]; counts[k] += (rows that entered k) - (rows that left k).  Tables have one
// entry per key (+1).  Labels outside [0, K) are left out.
// settled (delta mode, here and in the launchers below and of the assignments; may be null): the sort of a round in
// which no label changed sets it, and once it is set the kernels return at once.  Such a round leaves sums, centroids
// and labels as they are, bit for bit, and so do all that would follow.  262 144 x 1024 rows in 256 far-apart clusters
// stand still after about seventeen of 25 rounds.
cudaError_t launch_label_sort(const int32_t *labels, const int32_t *prev, int64_t N, int K, const SegGeom &g,
                              uint32_t *blk_hist, uint32_t *key_total, int64_t *counts, int32_t *cluster_start,
                              int32_t *seg_start, int32_t *order, cudaStream_t s, int32_t *settled = nullptr);

// Per-segment partial sums over KK keys.  mode 0: column sums of Yq (plane 0); mode 1: of Yq and Yf
// (planes 0, 1); mode 2 (full mode only): centred moments sum (q-muQ)^2 (plane 0) and
// sum (q-muQ)(f-muF) (plane 1); mode 3 (full mode only, three planes per segment): sum (q-muQ)^2,
// sum (q-muQ)(f-muQ), sum f.
cudaError_t launch_segment_sums(int mode, const float *Yq, const float *Yf, const int32_t *order,
                                const int32_t *cluster_start, const int32_t *seg_start, const double *meanQ,
                                const double *meanF, int D, int KK, const SegGeom &g, double *part,
                                cudaStream_t s, const int32_t *settled = nullptr);

// gamma and beta of a small set for given labels (sumQ: the clusters' sums of Yq, or null).
bool closed_form_supported(int64_t N, int D, int K);
cudaError_t launch_closed_form(const float *Yq, const float *Yf, const int32_t *labels, int64_t N, int D, int K, const double *sumQ,
                               float *gamma, float *beta, cudaStream_t s);

// Adds each cluster's segment partials in order into out0 (and out1 if not NULL); in delta mode
// out0[k] += (partials of key k) - (partials of key K + k).  With C also writes the centroid
// float(out0 / n_k) for clusters with n_k > 0.
cudaError_t launch_segment_combine(const double *part, const int32_t *seg_start, const int64_t *counts, int D,
                                   int K, bool delta, double *out0, double *out1, float *C, cudaStream_t s);

// Sums of the three planes of mode 3 per cluster: out0 = sum (q-muQ)^2, out1 = sum (q-muQ)(f-muQ), out2 = sum f.
cudaError_t launch_segment_combine3(const double *part, const int32_t *seg_start, int D, int K, int max_segs, double *out0,
                                    double *out1, double *out2, cudaStream_t s);

// Delta-mode centroid update fused with what the next assignment needs: running sums, centroids,
// their squared norms, (with Ch) their fp16 copy with its rounding errors' norms -- norms and copy of the
// centroids less `mean` if that is given -- and the reset of the exact-pass queues.  norm_part: scratch;
// arrivals: [K], zero before the first call (left at zero).
cudaError_t launch_centroid_update(const double *part, const int32_t *seg_start, const int64_t *counts, int D,
                                   int K, int max_segs, double *sums, float *C, float *cnorm, const float *scale, void *Ch,
                                   const float *mean, float *cerr, void *norm_part, uint32_t *arrivals, Control *ctl,
                                   cudaStream_t s, const int32_t *settled = nullptr);
size_t centroid_update_scratch_bytes(int D, int K);
// The same, counts included, straight from two label buffers: for rounds in which few rows move.  list: N 8-byte entries; table:
// 4 (K + 1) bytes for every 2048 rows; state: an 8-byte word, zero before the first call.
cudaError_t launch_moved_update(const float *Y, const int32_t *cur, const int32_t *prev, int64_t N, int D, int K, void *list, void *table,
                                void *state, int64_t *counts, double *sums, float *C, float *cnorm, const float *scale, void *Ch,
                                const float *mean, float *cerr, void *norm_part, uint32_t *arrivals, Control *ctl, int32_t *settled,
                                cudaStream_t s);

cudaError_t launch_centroids_from_sums(const double *sums, const int64_t *counts, int D, int K,
                                       float *C, cudaStream_t s);
// sums += delta_sums, counts += delta_counts, C = float(sums / counts) where counts > 0
cudaError_t launch_shard_update(const double *delta_sums, const int64_t *delta_counts, int D, int K, double *sums,
                                int64_t *counts, float *C, cudaStream_t s);
cudaError_t launch_means_from_sums(const double *sums, const int64_t *counts, int D, int K,
                                   double *mean, cudaStream_t s);
cudaError_t launch_solve(const double *sumQ, const double *sumF, const double *var,
                         const double *cov, const int64_t *counts, int D, int K, float *gamma,
                         float *beta, cudaStream_t s);
cudaError_t launch_blend_params(const float *gamma, const float *beta, float alpha, int64_t KD,
                                float *gamma_b, float *beta_b, cudaStream_t s);
cudaError_t launch_fit_diag(const Control *ctl, const int64_t *counts, int K, cat_fit_diag_t *diag,
                            cudaStream_t s);
// Record of one assignment in diag (slot): objective against C for the given labels, rows that were
// queued for the exact pass (the queues of the workspace as the exact pass left them), and how many
// of those have their two nearest centroids within 1e-6 relative.  An extra pass over Y.
cudaError_t launch_fit_diag_round(const float *Y, int64_t N, int D, int K, const float *C, const int32_t *labels,
                                  const int32_t *refine_rows, const int32_t *cand_rows, const Control *ctl,
                                  cat_fit_diag_t *diag, int slot, int recorded, cudaStream_t s);
cudaError_t launch_reset_control(Control *ctl, cudaStream_t s);
// Adds the counters of a step that ran on a workspace of its own to ctl; its status too, unless ctl has one already.
cudaError_t launch_absorb_control(Control *ctl, const Control *from, cudaStream_t s);

// Y_out_i = gamma_l * Y_i + beta_l, l = labels[i]; a label outside [0, K) copies the row
cudaError_t launch_affine_labels(const float *Y, int64_t N, int D, int K, const int32_t *labels, const float *gamma,
                                 const float *beta, float *out, cudaStream_t s);

// The p largest eigenpairs of the symmetric positive semi-definite matrix A [D, D] (full, fp64; overwritten),
// whose diagonal is also given: unit vectors -> comps [p, D] (fp32 rows, decreasing eigenvalue, entry of largest
// magnitude positive), eigenvalues -> eig_out [p] (may be null).  refl: [D, D] scratch.  D <= CAT_PCA_MAX_D.
size_t sym_eig_workspace_bytes(int D, int p);
cudaError_t launch_sym_eig(double *A, const double *diag, double *refl, int D, int p, float *comps, double *eig_out,
                           Control *ctl, void *workspace, cudaStream_t s);

}  // namespace cat
