// model.cu -- model-level operations over all Gaussians (Sec. 3.2, Sec. 3.3):
//   * the two simplification passes on the importance score s: Pass 1 keeps k
//     Gaussians by importance-weighted sampling without replacement (as
//     exponential clocks: Gaussian i fires at e_i / s_i with e_i ~ Exp(1)
//     given, the k earliest are kept), Pass 2 keeps the smallest prefix by
//     descending s carrying a fraction `mass` of the total;
//   * order-preserving compaction of the model by a keep bit array;
//   * density control: the averaged view-space positional gradient, reweighted
//     by phi_i = c^vis_i / (c^rad_i + eps), selects Gaussians; small ones are
//     cloned, large ones split into two children (LOD: a clone keeps its
//     parent's level, a split child takes the next finer one), low-opacity
//     ones removed; the new model is written in parent order.
// Keep decisions are integer results of FP32 arithmetic done identically on
// every call (no transcendental functions), and the selections use the
// stable radix sort, so results are deterministic.
#include <math.h>
#include <string.h>

#include "gs_internal.cuh"

namespace gs {

cudaError_t launch_radix_sort_scratch(cudaStream_t st, uint32_t *keys[2], uint32_t *vals[2],
                                      const unsigned long long *count, unsigned long long cap, int bits,
                                      bool vals_identity, uint32_t *status, uint32_t *hist, DevCounters *ctr,
                                      int &out_buf);
cudaError_t launch_mass_scan(cudaStream_t st, const uint32_t *sorted, const float *w, double *bsum, double *cum,
                             const DevCounters *ctr, unsigned long long cap);

// ---- selections ------------------------------------------------------------------

// Pass 1 keys: FP32 bits of e_i / s_i (positive, so the bits order as the
// values); s_i = 0 gives +inf and fires after every Gaussian with s > 0.
__global__ void sample_keys_kernel(const float *s, const float *expo, long long n, uint32_t *keys, DevCounters *ctr)
{
    griddep_wait(); // programmatic dependent launch: the previous kernel is complete
    const long long i = (long long)blockIdx.x * 256 + threadIdx.x;
    if (i == 0) {
        ctr->n_records = (unsigned long long)n;
        ctr->error = 0;
    }
    if (i >= n) return;
    const float si = s[i];
    keys[i] = si > 0.f ? __float_as_uint(__fdiv_rn(expo[i], si)) : 0x7f800000u;
}

// Pass 2 keys: bit-complement of the FP32 bits of s (s >= 0), so ascending
// keys are descending s and s = 0 sorts last.
__global__ void mass_keys_kernel(const float *s, long long n, uint32_t *keys, DevCounters *ctr)
{
    griddep_wait(); // programmatic dependent launch: the previous kernel is complete
    const long long i = (long long)blockIdx.x * 256 + threadIdx.x;
    if (i == 0) {
        ctr->n_records = (unsigned long long)n;
        ctr->error = 0;
    }
    if (i < n) keys[i] = ~__float_as_uint(s[i]);
}

__global__ void clear_bits_kernel(uint32_t *bits, long long words)
{
    griddep_wait(); // programmatic dependent launch: the previous kernel is complete
    const long long k = (long long)blockIdx.x * 256 + threadIdx.x;
    if (k < words) bits[k] = 0u;
}

__global__ void keep_first_kernel(const uint32_t *sorted, long long n, long long k, uint32_t *keep)
{
    griddep_wait(); // programmatic dependent launch: the previous kernel is complete
    const long long j = (long long)blockIdx.x * 256 + threadIdx.x;
    if (j >= n || j >= k) return;
    const uint32_t g = sorted[j];
    atomicOr(&keep[g >> 5], 1u << (g & 31));
}

__global__ void keep_mass_kernel(const uint32_t *sorted, const float *s, const double *cum, long long n, float mass,
                                 uint32_t *keep)
{
    griddep_wait(); // programmatic dependent launch: the previous kernel is complete
    const long long j = (long long)blockIdx.x * 256 + threadIdx.x;
    if (j >= n) return;
    const uint32_t g = sorted[j];
    if (!(s[g] > 0.f)) return;
    const double excl = j > 0 ? cum[j - 1] : 0.0;
    if (excl < (double)mass * cum[n - 1]) atomicOr(&keep[g >> 5], 1u << (g & 31));
}

// ---- compaction and density control ------------------------------------------------

struct ModelRows {
    float *p[5];        // mean [n][3], log-scale [n][3], quat [n][4], opacity [n], SH [n][48]
    float *m[5], *v[5]; // Adam moments in the same layout (NULL: not carried)
    uint8_t *lod;       // may be NULL
};

struct ScatterArgs {
    ModelRows src, dst;
    long long n;
    long long dst_cap;
    const uint32_t *keep; // compaction; NULL: density control
    // density control
    const float *absgrad;
    const uint32_t *denom, *cvis, *crad;
    const float *noise;   // [n][2][3]
    float tau, eps, logit_min, log_dense, log_shrink;
    int max_level;
    unsigned long long *lb_status;
    long long *n_out;     // device
    // the output rows, in order: source Gaussian (the first list_n in list0, the
    // rest, of density control, in list1) and how the row is made (RowHow)
    uint32_t *list0, *list1;
    long long list_n;
    uint8_t *how;
    DevCounters *ctr;
};

// How an output row is made from its source: a copy with its moments, a copy
// whose moments start from zero (a clone), a split child (its mean and scales
// written already, moments from zero), or not written (it lies past dst_cap).
enum RowHow { kRowCopy = 0, kRowClone = 1, kRowChild = 2, kRowNone = 3 };

// 0 removed, 1 kept, 2 cloned, 3 split: FP32 quantities formed as the oracle
// forms them (its decision instance mirrors these operations).
__device__ __forceinline__ int densify_kind(const ScatterArgs &a, long long i)
{
    if (a.src.p[3][i] < a.logit_min) return 0;
    const uint32_t d = a.denom[i];
    const float grad = d > 0 ? __fdiv_rn(a.absgrad[i], (float)d) : 0.f;
    const float phi = __fdiv_rn((float)a.cvis[i], __fadd_rn((float)a.crad[i], a.eps));
    if (!(__fmul_rn(grad, phi) >= a.tau)) return 1;
    const float *ls = a.src.p[1] + 3 * i;
    return fmaxf(ls[0], fmaxf(ls[1], ls[2])) <= a.log_dense ? 2 : 3;
}

__device__ __forceinline__ void put_row(const ScatterArgs &a, long long o, long long i, RowHow how)
{
    (o < a.list_n ? a.list0 : a.list1 - a.list_n)[o] = (uint32_t)i;
    a.how[o] = (uint8_t)how;
}

// The mean and scales of one split child: mu + R(q) (s * z), log-scale - log(1.6).
__device__ __forceinline__ void write_child(const ScatterArgs &a, long long i, long long o, int c)
{
    const float *q = a.src.p[2] + 4 * i;
    const float qn = sqrtf(q[0] * q[0] + q[1] * q[1] + q[2] * q[2] + q[3] * q[3]);
    const float w = q[0] / qn, x = q[1] / qn, y = q[2] / qn, z = q[3] / qn;
    const float R[3][3] = {{1.f - 2.f * (y * y + z * z), 2.f * (x * y - w * z), 2.f * (x * z + w * y)},
                           {2.f * (x * y + w * z), 1.f - 2.f * (x * x + z * z), 2.f * (y * z - w * x)},
                           {2.f * (x * z - w * y), 2.f * (y * z + w * x), 1.f - 2.f * (x * x + y * y)}};
    const float *ls = a.src.p[1] + 3 * i;
    const float *zz = a.noise + 6 * i + 3 * c;
    const float l[3] = {expf(ls[0]) * zz[0], expf(ls[1]) * zz[1], expf(ls[2]) * zz[2]};
    for (int r = 0; r < 3; r++) {
        a.dst.p[0][3 * o + r] = a.src.p[0][3 * i + r] + (R[r][0] * l[0] + R[r][1] * l[1] + R[r][2] * l[2]);
        a.dst.p[1][3 * o + r] = ls[r] - a.log_shrink;
    }
}

// The list of output rows.  Ticket-ordered blocks of kListGauss Gaussians (four
// consecutive ones per thread): each block counts its outputs, finds its offset
// by decoupled look-back and writes its rows' sources in parent order, with the
// levels and the split children's mean and scales; model_rows_kernel then
// copies the rows.
constexpr int kListItems = 4, kListGauss = 256 * kListItems;
__global__ void __launch_bounds__(256) model_scatter_kernel(ScatterArgs a)
{
    griddep_wait(); // programmatic dependent launch: the previous kernel is complete
    __shared__ unsigned s_bid;
    __shared__ unsigned long long s_warp[8];
    __shared__ unsigned long long s_base;
    if (threadIdx.x == 0) s_bid = atomicAdd((unsigned *)a.lb_status, 1u);
    __syncthreads();
    const unsigned bid = s_bid;
    const long long i0 = (long long)bid * kListGauss + threadIdx.x * kListItems;
    int kind[kListItems];
    unsigned long long mine = 0;
    const uint32_t bits = a.keep && i0 < a.n ? a.keep[i0 >> 5] >> (i0 & 31) : 0u;
#pragma unroll
    for (int q = 0; q < kListItems; q++) {
        kind[q] = i0 + q >= a.n ? 0 : a.keep ? (int)((bits >> q) & 1u) : densify_kind(a, i0 + q);
        mine += kind[q] == 0 ? 0 : (kind[q] == 1 ? 1 : 2);
    }
    unsigned long long total;
    const unsigned long long excl = block_exclusive_scan_256<unsigned long long>(mine, s_warp, total);
    if (threadIdx.x < 32) {
        const unsigned long long b = lookback_exclusive(a.lb_status + 1, bid, total, a.ctr, kSiteModel);
        if (threadIdx.x == 0) s_base = b;
    }
    __syncthreads();
    unsigned long long o = s_base + excl;
    if (i0 < a.n && i0 + kListItems >= a.n) *a.n_out = (long long)(o + mine); // the last Gaussian's thread
#pragma unroll
    for (int q = 0; q < kListItems; q++) {
        const long long i = i0 + q, r = (long long)o;
        const unsigned cnt = kind[q] == 0 ? 0 : (kind[q] == 1 ? 1 : 2);
        o += cnt;
        if (cnt == 0) continue;
        if (r + (long long)cnt > a.dst_cap) {
            set_error(a.ctr, GS_ERR_CAPACITY, kSiteModel);
            if (r < a.dst_cap) put_row(a, r, i, kRowNone); // the first of two rows
            continue;
        }
        if (kind[q] == 3) {
            for (int c = 0; c < 2; c++) {
                put_row(a, r + c, i, kRowChild);
                write_child(a, i, r + c, c);
            }
        } else {
            put_row(a, r, i, kRowCopy);
            if (kind[q] == 2) put_row(a, r + 1, i, kRowClone);
        }
        if (a.dst.lod) {
            int lv = a.src.lod ? (int)a.src.lod[i] : 0;
            if (kind[q] == 3) lv = min(lv + 1, a.max_level); // the next finer level
            a.dst.lod[r] = (uint8_t)lv;
            if (cnt == 2) a.dst.lod[r + 1] = (uint8_t)lv;
        }
    }
}

// A warp's 32 output rows of one array, LEN floats each, from row base on; lane
// r holds row r's source Gaussian i.  Consecutive lanes move consecutive
// elements (float4 where the rows are whole float4s of aligned arrays), up to
// four loads of a lane in flight.  Rows of `write` are written, those of `read`
// with the source's values, the others (and all without a source array) with
// zeros.
template <int LEN, bool VEC>
__device__ __forceinline__ void copy_rows(const float *__restrict__ src, float *__restrict__ dst, long long base,
                                          uint32_t i, unsigned write, unsigned read)
{
    if (!dst) return;
    constexpr int W = VEC && LEN % 4 == 0 ? 4 : 1, kPer = LEN / W; // elements moved at once, moves per row
    constexpr int kIn = kPer < 4 ? kPer : 4;                       // loads in flight
    static_assert(kPer % kIn == 0, "whole groups of loads");
    const int lane = threadIdx.x & 31;
    if (!src) read = 0u;
#pragma unroll 1
    for (int g = 0; g < kPer; g += kIn) {
        float4 v[kIn];
#pragma unroll
        for (int q = 0; q < kIn; q++) {
            const int e = (g + q) * 32 + lane, row = e / kPer;
            const size_t from = (size_t)__shfl_sync(0xffffffffu, i, row) * LEN + (e % kPer) * W;
            v[q] = make_float4(0.f, 0.f, 0.f, 0.f);
            if ((read >> row) & 1u) {
                if (W == 4) v[q] = __ldcs(reinterpret_cast<const float4 *>(src + from));
                else v[q].x = __ldcs(src + from);
            }
        }
#pragma unroll
        for (int q = 0; q < kIn; q++) {
            const int e = (g + q) * 32 + lane, row = e / kPer;
            if ((write >> row) & 1u) {
                float *to = dst + (size_t)base * LEN + (size_t)e * W;
                if (W == 4) __stcs(reinterpret_cast<float4 *>(to), v[q]);
                else __stcs(to, v[q].x);
            }
        }
    }
}

// The rows of the list, 32 per warp, array by array.  Bound by HBM (708 bytes
// read and written per row of a model with moments).  One thread per Gaussian
// copying its 177 floats one after another, as the list kernel once did, touched
// a sector per float: the mass cut and compaction of 3M Gaussians with moments
// took 2.52 ms and takes 0.98, the density control of 1.5M 2.32 and 0.67 (array by
// array over the whole model, 62 registers: 1.14 and 0.82; the 32 registers of eight
// blocks per SM spill 48 B).  (A list entry left unset by a look-back that gave up is
// not followed: i < n.)
template <bool VEC> __global__ void __launch_bounds__(256, 8) model_rows_kernel(ScatterArgs a)
{
    griddep_wait(); // programmatic dependent launch: the previous kernel is complete
    const long long rows = min(*a.n_out, a.dst_cap);
    const int lane = threadIdx.x & 31;
    for (long long base = ((long long)blockIdx.x * 8 + (threadIdx.x >> 5)) * 32; base < rows;
         base += (long long)gridDim.x * 256) {
        const long long o = base + lane;
        uint32_t i = 0;
        int how = kRowNone;
        if (o < rows) {
            i = (o < a.list_n ? a.list0 : a.list1 - a.list_n)[o];
            how = (long long)i < a.n ? a.how[o] : kRowNone;
            if (how == kRowNone) i = 0;
        }
        const unsigned put = __ballot_sync(0xffffffffu, how != kRowNone);
        const unsigned whole = __ballot_sync(0xffffffffu, how == kRowCopy); // rows that keep their moments
        const unsigned geom = __ballot_sync(0xffffffffu, how != kRowNone && how != kRowChild);
        copy_rows<48, VEC>(a.src.p[4], a.dst.p[4], base, i, put, put);
        copy_rows<48, VEC>(a.src.m[4], a.dst.m[4], base, i, put, whole);
        copy_rows<48, VEC>(a.src.v[4], a.dst.v[4], base, i, put, whole);
        copy_rows<4, VEC>(a.src.p[2], a.dst.p[2], base, i, put, put);
        copy_rows<4, VEC>(a.src.m[2], a.dst.m[2], base, i, put, whole);
        copy_rows<4, VEC>(a.src.v[2], a.dst.v[2], base, i, put, whole);
#pragma unroll
        for (int k = 0; k < 2; k++) { // mean, log-scale: a split child's are in place already
            copy_rows<3, VEC>(a.src.p[k], a.dst.p[k], base, i, geom, geom);
            copy_rows<3, VEC>(a.src.m[k], a.dst.m[k], base, i, put, whole);
            copy_rows<3, VEC>(a.src.v[k], a.dst.v[k], base, i, put, whole);
        }
        copy_rows<1, VEC>(a.src.p[3], a.dst.p[3], base, i, put, put);
        copy_rows<1, VEC>(a.src.m[3], a.dst.m[3], base, i, put, whole);
        copy_rows<1, VEC>(a.src.v[3], a.dst.v[3], base, i, put, whole);
    }
}

// Views in which each Gaussian has a record (+= per Gaussian; records of a
// Gaussian are contiguous).
__global__ void count_views_kernel(const uint32_t *rec_g, const float4 *rd2, const DevCounters *ctr, uint32_t *counts)
{
    griddep_wait(); // programmatic dependent launch: the previous kernel is complete
    const unsigned long long r = (unsigned long long)blockIdx.x * 256 + threadIdx.x;
    const unsigned long long nrec = ctr->n_records;
    if (r >= nrec || (r > 0 && rec_g[r - 1] == rec_g[r])) return;
    uint32_t views = 0;
    for (unsigned long long e = r; e < nrec && rec_g[e] == rec_g[r]; e++)
        views += rd2[e].w != 0.f ? 0u : 1u; // records marked culled (GS_CULL_MARK) are not rendered
    counts[rec_g[r]] += views;
}

// ---- launchers ------------------------------------------------------------------------

static cudaError_t sort_model_keys(gs_workspace *ws, cudaStream_t st, long long n, int &ob)
{
    return launch_radix_sort_scratch(st, ws->mkey, ws->mval, &ws->mctr->n_records, (unsigned long long)n, 32, true,
                                     ws->mrx_status, ws->mhist, ws->mctr, ob);
}

cudaError_t launch_prune_sample(gs_workspace *ws, cudaStream_t st, const float *s, const float *expo, long long n,
                                long long k, uint32_t *keep)
{
    const unsigned blocks = (unsigned)((n + 255) / 256);
    const long long words = (n + 31) / 32;
    launch_pdl(sample_keys_kernel, blocks, 256, 0, st, s, expo, n, ws->mkey[0], ws->mctr);
    note_launch();
    launch_pdl(clear_bits_kernel, (unsigned)((words + 255) / 256), 256, 0, st, keep, words);
    note_launch();
    int ob = 0;
    cudaError_t e = sort_model_keys(ws, st, n, ob);
    if (e != cudaSuccess) return e;
    launch_pdl(keep_first_kernel, blocks, 256, 0, st, ws->mval[ob], n, k, keep);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_prune_mass(gs_workspace *ws, cudaStream_t st, const float *s, long long n, float mass,
                              uint32_t *keep)
{
    const unsigned blocks = (unsigned)((n + 255) / 256);
    const long long words = (n + 31) / 32;
    launch_pdl(mass_keys_kernel, blocks, 256, 0, st, s, n, ws->mkey[0], ws->mctr);
    note_launch();
    launch_pdl(clear_bits_kernel, (unsigned)((words + 255) / 256), 256, 0, st, keep, words);
    note_launch();
    int ob = 0;
    cudaError_t e = sort_model_keys(ws, st, n, ob);
    if (e != cudaSuccess) return e;
    if ((e = launch_mass_scan(st, ws->mval[ob], s, ws->mbsum, ws->mcum, ws->mctr, (unsigned long long)n)) !=
        cudaSuccess)
        return e;
    launch_pdl(keep_mass_kernel, blocks, 256, 0, st, ws->mval[ob], s, ws->mcum, n, mass, keep);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_model_scatter(gs_workspace *ws, cudaStream_t st, ScatterArgs &a)
{
    const unsigned long long blocks = ((unsigned long long)a.n + kListGauss - 1) / kListGauss;
    cudaError_t e;
    if ((e = cudaMemsetAsync(ws->mlb, 0, (blocks + 1) * sizeof(unsigned long long), st)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(a.n_out, 0, sizeof(long long), st)) != cudaSuccess) return e;
    a.lb_status = ws->mlb;
    a.ctr = ws->mctr;
    if (blocks == 0) return cudaSuccess;
    // the row list in the sort scratch of the selections (their keys and values
    // are read by now): up to two rows per Gaussian, one byte each for how
    a.list0 = ws->mkey[0];
    a.list1 = ws->mkey[1];
    a.list_n = ws->cap.max_gaussians;
    a.how = reinterpret_cast<uint8_t *>(ws->mval[0]);
    launch_pdl(model_scatter_kernel, (unsigned)blocks, 256, 0, st, a);
    note_launch();
    // the SH and quaternion rows move as float4 where every such array is 16-byte aligned
    bool vec = true;
    for (const ModelRows *r : {&a.src, &a.dst})
        for (int k : {2, 4})
            for (const float *p : {r->p[k], r->m[k], r->v[k]}) vec = vec && ((uintptr_t)p & 15u) == 0;
    launch_pdl(vec ? model_rows_kernel<true> : model_rows_kernel<false>, 8u * (unsigned)ws->sm_count, 256, 0, st, a);
    note_launch();
    return cudaGetLastError();
}

static ModelRows rows_of(const gs_model &m)
{
    ModelRows r;
    r.p[0] = m.mean; r.p[1] = m.log_scale; r.p[2] = m.quat; r.p[3] = m.opacity_logit; r.p[4] = m.sh;
    float *mm[5] = {m.m.mean, m.m.log_scale, m.m.quat, m.m.opacity_logit, m.m.sh};
    float *vv[5] = {m.v.mean, m.v.log_scale, m.v.quat, m.v.opacity_logit, m.v.sh};
    for (int k = 0; k < 5; k++) { r.m[k] = mm[k]; r.v[k] = vv[k]; }
    r.lod = m.lod;
    return r;
}

cudaError_t launch_compact(gs_workspace *ws, cudaStream_t st, const gs_model &src, const uint32_t *keep,
                           const gs_model &dst, long long dst_cap, long long *n_out)
{
    ScatterArgs a;
    memset(&a, 0, sizeof(a));
    a.src = rows_of(src);
    a.dst = rows_of(dst);
    a.n = src.n;
    a.dst_cap = dst_cap;
    a.keep = keep;
    a.n_out = n_out;
    return launch_model_scatter(ws, st, a);
}

cudaError_t launch_densify(gs_workspace *ws, cudaStream_t st, const gs_model &src, const float *absgrad,
                           const uint32_t *denom, const uint32_t *cvis, const uint32_t *crad, const float *noise,
                           const gs_densify_params &p, const gs_model &dst, long long dst_cap, long long *n_out)
{
    ScatterArgs a;
    memset(&a, 0, sizeof(a));
    a.src = rows_of(src);
    a.dst = rows_of(dst);
    a.n = src.n;
    a.dst_cap = dst_cap;
    a.keep = nullptr;
    a.absgrad = absgrad; a.denom = denom; a.cvis = cvis; a.crad = crad; a.noise = noise;
    // thresholds in the form the kernel compares, from FP64 (the oracle rounds them the same way)
    a.tau = p.grad_threshold;
    a.eps = p.eps;
    a.logit_min = (float)log((double)p.min_opacity / (1.0 - (double)p.min_opacity));
    a.log_dense = (float)log((double)p.dense_scale);
    a.log_shrink = (float)log((double)p.split_shrink);
    a.max_level = p.n_levels - 1;
    a.n_out = n_out;
    return launch_model_scatter(ws, st, a);
}

cudaError_t launch_count_views(gs_workspace *ws, cudaStream_t st, uint32_t *counts)
{
    const unsigned blocks = (unsigned)((ws->cap.max_records + 255) / 256);
    if (blocks == 0) return cudaSuccess;
    launch_pdl(count_views_kernel, blocks, 256, 0, st, ws->rec_g, ws->rd2, ws->ctr, counts);
    note_launch();
    return cudaGetLastError();
}

} // namespace gs
