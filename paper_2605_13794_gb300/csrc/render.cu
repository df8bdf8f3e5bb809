// render.cu -- per-tile compositing (App. A, Eq. for C(p) and T_i), its
// adjoint, and the instrumented colourless sweep of the importance pass
// (Sec. 3.2, Fig. 2).
//
// One block per tile; each warp owns an 8 x 8 pixel square of it (lane l the
// horizontal pixel pair (2 (l % 4), l / 4), packed FP32x2).  The block stages the
// tile's depth-ordered list in rounds, an entry per thread, and each warp visits
// those entries of a round that can reach alpha_min in its square (the adjoint:
// those that composited there).
// Per-Gaussian quantities are warp reductions (recursive halving for the
// adjoint's nine values), then the warps' partials summed in warp order,
// rather than per-pixel global atomics.  The backward and the importance
// sweep write one gradient/score slot per (record, tile) -- slot index = the
// record's first instance + the tile's position inside the record's rectangle
// -- and a later per-record pass sums a record's slots in a fixed order, so
// results are bit-reproducible run to run.
#include "gs_internal.cuh"

namespace gs {

// Compositing works in tile-local pixel coordinates: pixel centres are exact
// small floats, and each staged entry's mean is moved to the tile's origin
// once, from its double-length form u + u_lo, so px - u keeps its full
// precision however far the tile lies from the image origin.

// ---- packed pair arithmetic (Blackwell FP32x2) ----------------------------------
// A lane's two pixels are one float2, so the exponent, alpha, transmittance
// and colour updates are packed FP32x2 operations.  The exponent is evaluated from the conic's form
// power = -1/2 (A (dx + k dy)^2 + D dy^2), with A and D pre-scaled at staging so
// it comes out in base 2: G = exp(power) = 2^(log2(e) power).  Every kernel
// that takes skip decisions (forward, backward, importance) stages and
// evaluates through these same functions.
constexpr float kNegHalfLog2e = -0.72134752044448170f; // -log2(e) / 2

// A staged entry: e0 = (u, v) tile-local, A and k; e1.x = D (A, D scaled to base 2)
__device__ __forceinline__ float4 stage_e0_at(float4 r0, float4 r2, float ox, float oy)
{
    return make_float4(__fadd_rn(__fsub_rn(r0.x, ox), r2.y), __fadd_rn(__fsub_rn(r0.y, oy), r2.z),
                       __fmul_rn(r0.z, kNegHalfLog2e), r0.w);
}
__device__ __forceinline__ float stage_D(float4 r1) { return __fmul_rn(r1.x, kNegHalfLog2e); }

__device__ __forceinline__ float ex2_approx(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }

// alpha = min(alpha_max, o 2^p) of a pixel pair
__device__ __forceinline__ float2 pair_alpha(float2 p, float o, float amax, float2 &G)
{
    G = make_float2(ex2_approx(p.x), ex2_approx(p.y));
    const float2 og = __fmul2_rn(f2(o), G);
    return make_float2(fminf(amax, og.x), fminf(amax, og.y));
}

// Whether an entry can composite anywhere in a warp's square, the box
// [bx0, bx0 + 7] x [by0, by0 + 7] of its pixel centres (tile-local; (u, v) the
// entry's tile-local mean).  alpha >= alpha_min needs o G >= alpha_min, i.e.
// q = A (dx + k dy)^2 + D dy^2 <= tau, tau = 2 ln(o / alpha_min).  The test
// compares tau with the minimum of q over the box.  q is convex with its
// minimum 0 at the mean, so on the way from any point of the box towards the
// mean it falls: the minimum lies where that way leaves the box, on the
// vertical side nearest the mean (x = xe: least q at dy = -A k xe / (A k^2 + D),
// clamped to the side) or the horizontal one (y = ye: at dx = -k ye); where the
// box reaches across the mean in x or y, xe or ye is 0 and the smaller of the
// two is the minimum all the same.
// Widened (tau by 0.2 % + 2e-3, the box by 1/32 px) far beyond the FP32 error
// of the exponent the kernels evaluate and of the approximate logarithm and
// reciprocal here (a few units in the last place), so no pixel of a square that
// fails can reach alpha_min in them; it always fails when o is below alpha_min.
// A warp skips an entry that fails: it composites nowhere in the warp, so
// skipping it changes nothing.  (The bounding box of the ellipse and a looser
// bound of q, before, took as many instructions and dropped fewer entries; the
// whole passes are alike within what their repeats differ by.)
struct SquareTest {
    float A, k, D, tau, slope, u, v;
    __device__ __forceinline__ SquareTest(float4 r0, float D_, float o, float alpha_min, float u_, float v_)
        : A(r0.z), k(r0.w), D(D_), u(u_), v(v_)
    {
        tau = fmaf(2.f * __logf(__fdividef(o, alpha_min)), 1.002f, 2e-3f);
        slope = -A * k * rcp_approx(fmaf(A * k, k, D));
    }
    __device__ __forceinline__ bool meets(float bx0, float by0) const
    {
        const float dx0 = bx0 - 0.03125f - u, dx1 = bx0 + 7.03125f - u;
        const float dy0 = by0 - 0.03125f - v, dy1 = by0 + 7.03125f - v;
        const float xe = fminf(fmaxf(0.f, dx0), dx1), ye = fminf(fmaxf(0.f, dy0), dy1);
        const float y1 = fminf(fmaxf(slope * xe, dy0), dy1);
        const float s1 = fmaf(k, y1, xe);
        const float x2 = fminf(fmaxf(-k * ye, dx0), dx1);
        const float s2 = fmaf(k, ye, x2);
        const float q = fminf(fmaf(A * s1, s1, D * y1 * y1), fmaf(A * s2, s2, D * ye * ye));
        return tau > 0.f && !(q > tau);
    }
};

__device__ __forceinline__ float warp_sum_f(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sums the 9 slot values over the warp by recursive halving (a reduce-scatter):
// at each of the first four levels a lane keeps half of its values and trades
// the other half with its partner, so 5 + 3 + 2 + 1 + 1 = 12 shuffles replace
// the 45 of nine butterfly sums.  Lane l ends with the full sum of value
// red9_index(l), valid when red9_owner(l).
__device__ __forceinline__ float warp_reduce9(const float (&v)[kSlotFloats], int lane)
{
    static_assert(kSlotFloats == 9, "the halving schedule is laid out for 9 values");
    const bool h1 = lane & 16, h2 = lane & 8, h3 = lane & 4, h4 = lane & 2;
    float a[5], b[3], c[2];
#pragma unroll
    for (int i = 0; i < 5; i++) {
        const float lo = v[i], hi = i + 5 < 9 ? v[i + 5] : 0.f;
        a[i] = (h1 ? hi : lo) + __shfl_xor_sync(0xffffffffu, h1 ? lo : hi, 16);
    }
#pragma unroll
    for (int i = 0; i < 3; i++) {
        const float lo = a[i], hi = i + 3 < 5 ? a[i + 3] : 0.f;
        b[i] = (h2 ? hi : lo) + __shfl_xor_sync(0xffffffffu, h2 ? lo : hi, 8);
    }
#pragma unroll
    for (int i = 0; i < 2; i++) {
        const float lo = b[i], hi = i + 2 < 3 ? b[i + 2] : 0.f;
        c[i] = (h3 ? hi : lo) + __shfl_xor_sync(0xffffffffu, h3 ? lo : hi, 4);
    }
    const float d = (h4 ? c[1] : c[0]) + __shfl_xor_sync(0xffffffffu, h4 ? c[0] : c[1], 2);
    return d + __shfl_xor_sync(0xffffffffu, d, 1);
}
// value held by lane l after warp_reduce9: lane bit 4 picks 0-4 / 5-8, bits 3, 2
// and 1 pick within the halves (padding positions hold no value)
__device__ __forceinline__ int red9_index(int lane)
{
    return 5 * ((lane >> 4) & 1) + 3 * ((lane >> 3) & 1) + 2 * ((lane >> 2) & 1) + ((lane >> 1) & 1);
}
__device__ __forceinline__ bool red9_owner(int lane)
{
    const int h1 = (lane >> 4) & 1, h2 = (lane >> 3) & 1, h3 = (lane >> 2) & 1, h4 = (lane >> 1) & 1;
    const int ai = 3 * h2 + 2 * h3 + h4;
    return (lane & 1) == 0 && (h2 ? h3 == 0 : 2 * h3 + h4 <= 2) && ai < (h1 ? 4 : 5);
}

// Slot of (record r, tile (tx, ty)): first instance of r + position of the
// tile inside r's rectangle (row-major, the order of emission).
__device__ __forceinline__ unsigned long long slot_of(const uint32_t *inst_off, const uint2 *rect, uint32_t r, int tx,
                                                      int ty)
{
    int x0, y0, x1, y1;
    unpack_rect(rect[r], x0, y0, x1, y1);
    return (unsigned long long)inst_off[r] + (unsigned long long)((ty - y0) * (x1 - x0) + (tx - x0));
}

// ---- warp squares ------------------------------------------------------------
//
// Every walk gives each warp an 8 x 8 pixel square of the tile: lane l holds the
// horizontal pixel pair (2 (l % 4), l / 4) of it, as FP32x2.  A batch is 32
// consecutive entries of the tile's list, staged by one warp for the whole block
// (lane i the i-th); the staging lane tests its entry against every square
// (SquareTest), and one ballot per square gives the entries of the batch that its
// warp visits.

template <int TW, int TH> struct SquareShape {
    static_assert(TW % 8 == 0 && TH % 8 == 0, "the tile splits into 8 x 8 pixel squares");
    static constexpr int wx = TW / 8;
    static constexpr int warps = (TW / 8) * (TH / 8);
    static constexpr int threads = 32 * warps;
    // the adjoint's register budget: at least six resident blocks of 128 threads per
    // SM, which ptxas meets with 64 registers (so eight fit); on the 16 x 16 tile
    // 10-15 % faster than both its own choice (86 registers, five blocks) and tighter
    // budgets (56-57 registers); both measured when each warp staged for itself
    static constexpr int bwd_min_blocks = 768 / threads;
    // the importance walk's: eight blocks of 128 threads (64 registers; the fused walk
    // with the training image measured 8 % faster than with the compiler's 60, when each
    // warp staged for itself)
    static constexpr int imp_min_blocks = 1024 / threads;
};

// Tile, camera and pixel geometry of one warp square.
struct SquareGeom {
    const CamInfo *ci;
    int tx, ty;            // tile coordinates in its camera
    float ox, oy;          // pixel origin of the tile
    int lx, ly;            // tile-local pixel of the lane's pair (left pixel)
    float2 pxc;            // its two pixel-centre x, tile-local
    float pyc;             // its pixel-centre y, tile-local
    float bx0, by0;        // the square's first pixel centre, tile-local
};

template <int TW, int TH> __device__ __forceinline__ SquareGeom square_geom(const CamTable &ct, int tile, int warp,
                                                                            int lane)
{
    SquareGeom q;
    q.ci = &ct.c[camera_of_tile(ct, tile)];
    const int lt = tile - q.ci->tile_base;
    q.tx = lt % q.ci->tiles_x;
    q.ty = lt / q.ci->tiles_x;
    q.ox = (float)(q.tx * TW);
    q.oy = (float)(q.ty * TH);
    const int sx = 8 * (warp % SquareShape<TW, TH>::wx), sy = 8 * (warp / SquareShape<TW, TH>::wx);
    q.lx = sx + 2 * (lane & 3);
    q.ly = sy + (lane >> 2);
    q.pxc = make_float2((float)q.lx + 0.5f, (float)q.lx + 1.5f);
    q.pyc = (float)q.ly + 0.5f;
    q.bx0 = (float)sx + 0.5f;
    q.by0 = (float)sy + 0.5f;
    return q;
}

// Base-2 exponent of a staged entry (e0 = (u, v, A, k), Ds = scaled D) at the
// lane's pixel pair; every kernel evaluates it through this function, so all
// take the same decisions.  e returns dx + k dy.
__device__ __forceinline__ float2 pair_power(float4 e0, float Ds, float2 pxc, float pyc, float2 &dx, float &dy,
                                             float2 &e)
{
    dx = __fadd2_rn(pxc, f2(-e0.x));
    dy = __fadd_rn(pyc, -e0.y);
    const float kdy = __fmul_rn(e0.w, dy);
    const float ddy = __fmul_rn(__fmul_rn(Ds, dy), dy);
    e = __fadd2_rn(dx, f2(kdy));
    return __ffma2_rn(f2(e0.z), __fmul2_rn(e, e), f2(ddy));
}

// The entries of a batch (list positions b .. b + 31 of the tile whose list
// starts at start) that composite in a warp's square, one bit each, left by the
// forward for the adjoint.  Tiles' batches follow one another, each tile's from
// start / 32 + its index.
template <int WARPS> __device__ __forceinline__ size_t visits_at(int start, int b, int warp)
{
    return ((size_t)(start / 32) + blockIdx.x + (unsigned)(b - start) / 32u) * WARPS + warp;
}
template <int WARPS>
__device__ __forceinline__ void put_visits(uint32_t *visits, int start, int b, int warp, unsigned comp)
{
    comp = __reduce_or_sync(0xffffffffu, comp);
    if ((threadIdx.x & 31) == 0) visits[visits_at<WARPS>(start, b, warp)] = comp;
}

// ---- forward --------------------------------------------------------------
//
// The block goes through the tile's list front to back in rounds of 32 entries
// per warp: each warp stages 32 of them, one per lane, tests each against every
// square of the tile and leaves a bit mask per square; then every warp walks
// the round's entries of its own square.  The staged entries are double
// buffered, so one block barrier per round is enough: a warp that is done
// with a round stages the next while others still walk.  So every entry is
// gathered once per tile, and a warp waits for a gather once per round.
// (Each warp staging every batch for itself, with no barrier, gathered each
// entry once per warp: 24 mixed views, whole pass, 2.80 ms, this 2.59; the
// 1080p view of the 5M city 218 and 212 us.)
// A warp stops walking once all of its pixels have stopped (T would drop below
// T_min), which it asks once per batch: a vote after every entry cost more than
// the entries it saved (24 mixed views, whole pass: 2.84 ms with it, 2.79
// without), as did a vote to skip the entries that reach no live pixel (3.06).
// Where every pixel stops within the first entries of a long list the walk alone is
// slower than with batches staged per warp, by the round staged in vain (200k opaque
// Gaussians of 45M instances at 720p: 37 and 54 us, their binning 7.8 and 4.5 ms);
// asking before a round is staged whether any warp goes on does not help, the warps
// of a tile finish together, and costs the other scenes 2 %.

// VISITS: note the entries that composite in each square for the adjoint (not in
// a forward-only workspace: the bookkeeping costs the walk 6 %).
template <int TW, int TH, bool VISITS>
__global__ void __launch_bounds__(SquareShape<TW, TH>::threads)
    render_fwd_kernel(const uint2 *__restrict__ ranges, const uint32_t *__restrict__ vals,
                      const float4 *__restrict__ rd0, const float4 *__restrict__ rd1, const float4 *__restrict__ rd2,
                      const CamTable *__restrict__ ctp, RenderConsts rc, float *__restrict__ rgb_out,
                      float *__restrict__ T_out, float *__restrict__ T_ws, uint32_t *__restrict__ n_contrib,
                      uint32_t *__restrict__ tile_last, uint32_t *__restrict__ visits)
{
    griddep_wait(); // programmatic dependent launch: the previous kernel is complete
    constexpr int kWarps = SquareShape<TW, TH>::warps;
    constexpr int kRound = 32 * kWarps; // entries per round
    __shared__ float4 s0[2][kRound];
    __shared__ float4 s1[2][kRound];
    __shared__ float s2[2][kRound];
    __shared__ unsigned s_mask[2][kWarps][kWarps]; // [square][batch of the round]
    const CamTable &ct = *ctp;
    if ((int)blockIdx.x >= ct.total_tiles) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const SquareGeom q = square_geom<TW, TH>(ct, blockIdx.x, warp, lane);
    const CamInfo &cam = *q.ci;
    const uint2 rg = ranges[blockIdx.x];
    const int start = (int)rg.x, end = (int)rg.y;
    const int px = q.tx * TW + q.lx, py = q.ty * TH + q.ly;
    float2 T = f2(1.f), Cr = f2(0.f), Cg = f2(0.f), Cb = f2(0.f);
    uint32_t last0 = 0, last1 = 0;
    bool dn0 = px >= cam.width || py >= cam.height, dn1 = px + 1 >= cam.width || py >= cam.height;
    int buf = 0;
    for (int first = start; first < end; first += kRound, buf ^= 1) {
        {
            const int at = 32 * warp + lane;
            unsigned meets = 0; // squares the entry may composite in
            if (first + at < end) {
                const uint32_t r = vals[first + at];
                const float4 r0 = rd0[r], r1 = rd1[r], r2 = rd2[r];
                const float op = r2.w != 0.f ? 0.f : r1.y; // a record marked culled composites nowhere
                const float4 e0 = stage_e0_at(r0, r2, q.ox, q.oy);
                s0[buf][at] = e0;
                s1[buf][at] = make_float4(stage_D(r1), op, r1.z, r1.w);
                s2[buf][at] = r2.x;
                const SquareTest test(r0, r1.x, op, rc.alpha_min, e0.x, e0.y);
#pragma unroll
                for (int k = 0; k < kWarps; k++)
                    meets |= test.meets(8.f * (k % SquareShape<TW, TH>::wx) + 0.5f, 8.f * (k / SquareShape<TW, TH>::wx) + 0.5f) ? 1u << k : 0u;
            }
#pragma unroll
            for (int k = 0; k < kWarps; k++) {
                const unsigned m = __ballot_sync(0xffffffffu, (meets >> k) & 1u);
                if (lane == k) s_mask[buf][k][warp] = m;
            }
        }
        if (__syncthreads_and(dn0 && dn1)) break; // the round is staged; every pixel of the tile has stopped
        for (int sub = 0, b = first; sub < kWarps && b < end; sub++, b += 32) {
            if (__all_sync(0xffffffffu, dn0 && dn1)) break;
            unsigned m = s_mask[buf][warp][sub];
            const float4 *e0s = s0[buf] + 32 * sub, *e1s = s1[buf] + 32 * sub;
            const float *e2s = s2[buf] + 32 * sub;
            unsigned comp = 0; // entries that composite in the lane's pixels
            while (m != 0u) {
                const int jj = __ffs(m) - 1; // front to back
                m &= m - 1u;
                const float4 p0 = e0s[jj];
                const float4 p1 = e1s[jj];
                const uint32_t pos = (uint32_t)(b - start + jj + 1);
                float2 dx, e;
                float dy;
                const float2 pw = pair_power(p0, p1.x, q.pxc, q.pyc, dx, dy, e);
                float2 G;
                const float2 al = pair_alpha(pw, p1.y, rc.alpha_max, G);
                const float2 tT = __ffma2_rn(make_float2(-T.x, -T.y), al, T); // T (1 - alpha)
                const bool ok0 = !dn0 && al.x >= rc.alpha_min, ok1 = !dn1 && al.y >= rc.alpha_min;
                const bool st0 = ok0 && tT.x < rc.T_min, st1 = ok1 && tT.y < rc.T_min;
                const bool c0 = ok0 && !st0, c1 = ok1 && !st1;
                dn0 = dn0 || st0;
                dn1 = dn1 || st1;
                if (VISITS && (c0 || c1)) comp |= 1u << jj;
                const float2 ae = make_float2(c0 ? al.x : 0.f, c1 ? al.y : 0.f); // skipped fragments add nothing
                const float2 w = __fmul2_rn(ae, T);
                Cr = __ffma2_rn(w, f2(p1.z), Cr);
                Cg = __ffma2_rn(w, f2(p1.w), Cg);
                Cb = __ffma2_rn(w, f2(e2s[jj]), Cb);
                T = __ffma2_rn(make_float2(-T.x, -T.y), ae, T);
                last0 = c0 ? pos : last0;
                last1 = c1 ? pos : last1;
            }
            if (VISITS) put_visits<kWarps>(visits, start, b, warp, comp);
        }
    }
    const long long np = (long long)cam.width * cam.height;
    float *img = rgb_out + 3 * cam.pix_base;
#pragma unroll
    for (int h = 0; h < 2; h++) {
        if (px + h >= cam.width || py >= cam.height) continue;
        const float Tk = h ? T.y : T.x;
        const long long pix = (long long)py * cam.width + px + h;
        img[pix] = (h ? Cr.y : Cr.x) + Tk * rc.bg[0];
        img[np + pix] = (h ? Cg.y : Cg.x) + Tk * rc.bg[1];
        img[2 * np + pix] = (h ? Cb.y : Cb.x) + Tk * rc.bg[2];
        const long long gp = cam.pix_base + pix;
        if (T_out) T_out[gp] = Tk;
        T_ws[gp] = Tk;
        n_contrib[gp] = h ? last1 : last0;
    }
    // the tile's largest n_contrib, where the adjoint's reverse walk starts
    const unsigned wl = __reduce_max_sync(0xffffffffu, max(last0, last1));
    if (lane == 0 && wl != 0u) atomicMax(&tile_last[blockIdx.x], wl);
}

template <int TW, int TH> static void fwd_launch(gs_workspace *ws, cudaStream_t st, float *rgb, float *T_out)
{
    const auto kernel = ws->visits ? render_fwd_kernel<TW, TH, true> : render_fwd_kernel<TW, TH, false>;
    launch_pdl(kernel, ws->cams.total_tiles, SquareShape<TW, TH>::threads, 0, st,
        ws->ranges, ws->sval, ws->rd0, ws->rd1, ws->rd2, ws->d_cams, ws->rc, rgb, T_out, ws->T_final,
        ws->n_contrib, ws->tile_last, ws->visits);
}

cudaError_t launch_render_fwd(gs_workspace *ws, cudaStream_t st, float *rgb, float *T_out)
{
    if (ws->cams.total_tiles == 0) return cudaSuccess;
    kt_begin(ws, GS_KT_RENDER_FWD, st);
    switch (tile_shape_id(ws->cams.tile_w, ws->cams.tile_h)) {
    case 0: fwd_launch<16, 16>(ws, st, rgb, T_out); break;
    case 1: fwd_launch<32, 8>(ws, st, rgb, T_out); break;
    case 2: fwd_launch<8, 32>(ws, st, rgb, T_out); break;
    case 3: fwd_launch<32, 16>(ws, st, rgb, T_out); break;
    case 4: fwd_launch<16, 8>(ws, st, rgb, T_out); break;
    case 5: fwd_launch<8, 16>(ws, st, rgb, T_out); break;
    default: return cudaErrorInvalidValue;
    }
    kt_end(ws, GS_KT_RENDER_FWD, st);
    note_launch();
    return cudaGetLastError();
}

// ---- backward ---------------------------------------------------------------
//
// Each warp owns an 8 x 8 pixel square of the tile -- lane l the horizontal
// pixel pair (2 (l % 4), l / 4) of it, packed as FP32x2 -- and walks the
// tile's list back to front, starting with the forward's batch of the tile's
// last contribution (the forward's largest n_contrib of the tile) and
// recovering T by T / (1 - alpha) from the final transmittance.  It visits
// exactly the entries that composite in its square, which the forward noted
// (visits), so it tests no footprint and needs no vote per visit.  The block
// goes in rounds of up to kBwdRound entries: a thread per entry gathers its
// record if any square visits it; then each warp walks its own entries, the
// nine slot values of each one warp reduction into shared memory; then the
// entry's thread adds the warps' partials in warp order and writes the entry's
// slot.  Two block barriers per round (staged, walked).  (Warps staging for
// themselves and meeting at arrival counters: the single-view training step on
// 5M Gaussians 756 us, this 748; the eight-view step on 8M 7.37 and 7.32 ms.)

constexpr int kBwdRound = 128; // entries per round, at most one per thread

struct BwdRenderArgs {
    const uint2 *ranges;
    const uint32_t *vals;
    const float4 *rd0, *rd1, *rd2;
    const uint32_t *inst_off;
    const uint2 *rect;
    const float *T_final;
    const uint32_t *n_contrib;
    const uint32_t *tile_last; // largest n_contrib of each tile (the forward's)
    const uint32_t *visits;    // entries of each batch that composite in each warp's square (the forward's)
    const float *dL_drgb;
    float *slots;
    DevCounters *ctr; // fragments += sum of the tile's n_contrib; composited += composited pairs
};

template <int TW, int TH>
__global__ void __launch_bounds__(SquareShape<TW, TH>::threads, SquareShape<TW, TH>::bwd_min_blocks)
    render_bwd_kernel(BwdRenderArgs a, const CamTable *__restrict__ ctp, RenderConsts rc)
{
    griddep_wait(); // programmatic dependent launch: the previous kernel is complete
    constexpr int kWarps = SquareShape<TW, TH>::warps, kRT = SquareShape<TW, TH>::threads;
    constexpr int kRound = kBwdRound < kRT ? kBwdRound : kRT, kSubs = kRound / 32; // batches of the forward per round
    __shared__ float4 s0[kRound];
    __shared__ float4 s1[kRound];
    __shared__ float s2[kRound];
    __shared__ float s_part[kWarps][kRound][kSlotFloats];
    __shared__ unsigned s_mask[kWarps][kSubs]; // [square][batch of the round]
    __shared__ int s_wmax[kWarps];             // each square's last contribution
    const CamTable &ct = *ctp;
    if ((int)blockIdx.x >= ct.total_tiles) return;
    const int tile = blockIdx.x;
    const CamInfo &ci = ct.c[camera_of_tile(ct, tile)];
    const int lt = tile - ci.tile_base;
    const int tx = lt % ci.tiles_x, ty = lt / ci.tiles_x;
    const float ox = (float)(tx * TW), oy = (float)(ty * TH);
    const uint2 rg = a.ranges[blockIdx.x];
    const int start = (int)rg.x, end = (int)rg.y;
    // the reverse walk starts with the batch of the tile's last contribution
    // (the forward's largest n_contrib); entries behind it carry zero gradient
    const int batches = (min((int)a.tile_last[blockIdx.x], end - start) + 31) / 32;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool red_own = red9_owner(lane);
    const int red_q = red9_index(lane);
    // the warp's square and the lane's pixel pair (tile-local)
    const int sx = 8 * (warp % SquareShape<TW, TH>::wx), sy = 8 * (warp / SquareShape<TW, TH>::wx);
    const int lx = sx + 2 * (lane & 3), ly = sy + (lane >> 2);
    const float2 pxc = make_float2((float)lx + 0.5f, (float)lx + 1.5f);
    const float pyc = (float)ly + 0.5f;

    // per-pixel state of the pair: dL/dC (g), T (from T_final back to each
    // fragment's own), S = colour composited behind the current fragment plus
    // the background seen through T_final
    float2 T = f2(1.f), g0 = f2(0.f), g1 = f2(0.f), g2 = f2(0.f);
    int nc0 = 0, nc1 = 0;
    {
        const long long np = (long long)ci.width * ci.height;
        const float *gimg = a.dL_drgb + 3 * ci.pix_base;
        const int px = tx * TW + lx, py = ty * TH + ly;
        float t[2] = {1.f, 1.f}, c0[2] = {0.f, 0.f}, c1[2] = {0.f, 0.f}, c2[2] = {0.f, 0.f};
        int n[2] = {0, 0};
#pragma unroll
        for (int h = 0; h < 2; h++) {
            if (px + h < ci.width && py < ci.height) {
                const long long pix = (long long)py * ci.width + px + h;
                c0[h] = gimg[pix]; c1[h] = gimg[np + pix]; c2[h] = gimg[2 * np + pix];
                t[h] = a.T_final[ci.pix_base + pix];
                n[h] = (int)a.n_contrib[ci.pix_base + pix];
            }
        }
        T = make_float2(t[0], t[1]);
        g0 = make_float2(c0[0], c0[1]); g1 = make_float2(c1[0], c1[1]); g2 = make_float2(c2[0], c2[1]);
        nc0 = n[0]; nc1 = n[1];
    }
    float2 S0 = __fmul2_rn(T, f2(rc.bg[0])), S1 = __fmul2_rn(T, f2(rc.bg[1])), S2 = __fmul2_rn(T, f2(rc.bg[2]));
    const int wmax = __reduce_max_sync(0xffffffffu, max(nc0, nc1));
    {
        const unsigned f = __reduce_add_sync(0xffffffffu, (unsigned)(nc0 + nc1));
        if (lane == 0 && f) atomicAdd(&a.ctr->fragments, (unsigned long long)f);
    }
    if (lane == 0) s_wmax[warp] = wmax;
    __syncthreads();
    int ncomp = 0;
    // rounds from the last batch down: batches [hi - kSubs, hi) of the forward
    for (int hi = batches; hi > 0; hi -= kSubs) {
        const int b0 = max(hi - kSubs, 0), first = start + 32 * b0; // the round's first batch and entry
        const int count = min(32 * (hi - b0), end - first);
        const int at = threadIdx.x;
        unsigned visited = 0; // squares that visit the thread's entry
        uint32_t slot = 0;
        if (warp < hi - b0) {
#pragma unroll
            for (int k = 0; k < kWarps; k++) {
                // (a batch behind a square's own last contribution may not have been walked by the forward)
                const int lo = first + 32 * warp;
                const unsigned m = lo - start < s_wmax[k] ? a.visits[visits_at<kWarps>(start, lo, k)] : 0u;
                if (lane == k) s_mask[k][warp] = m;
                visited |= ((m >> lane) & 1u) << k;
            }
            if (at < count) {
                const uint32_t r = a.vals[first + at];
                slot = (uint32_t)slot_of(a.inst_off, a.rect, r, tx, ty);
                if (visited) {
                    const float4 r0 = a.rd0[r], r1 = a.rd1[r], r2 = a.rd2[r];
                    s0[at] = stage_e0_at(r0, r2, ox, oy);
                    s1[at] = make_float4(stage_D(r1), r1.y, r1.z, r1.w);
                    s2[at] = r2.x;
                }
            }
        }
        __syncthreads(); // the round is staged
        for (int sub = hi - b0 - 1; sub >= 0; sub--) {
        for (unsigned m = s_mask[warp][sub]; m != 0u;) {
            const int bit = 31 - __clz(m); // back to front
            m ^= 1u << bit;
            const int jj = 32 * sub + bit;      // the entry's place in the round
            const int j = first + jj - start;   // position in the tile list
            const float4 p0 = s0[jj];
            const float4 p1 = s1[jj];
            // the forward's own exponent and alpha (the same operations, the same bits)
            float2 dx, e;
            float dy;
            const float2 pw = pair_power(p0, p1.x, pxc, pyc, dx, dy, e);
            float2 G;
            const float2 al = pair_alpha(pw, p1.y, rc.alpha_max, G);
            // composited pixels: in front of the pixel's last contribution, alpha >= alpha_min
            const bool m0 = j < nc0 && al.x >= rc.alpha_min;
            const bool m1 = j < nc1 && al.y >= rc.alpha_min;
            // Every lane runs the adjoint (no divergent branch): a pixel that does not
            // composite here has aT = dG = 0, so it adds exact zeros and keeps its T and S
            // (all terms stay finite: alpha <= alpha_max < 1).
            ncomp += (int)m0 + (int)m1;
            const float cb = s2[jj];
            const float2 inv = make_float2(rcp_approx(1.f - al.x), rcp_approx(1.f - al.y));
            const float2 Tj = __fmul2_rn(T, inv); // transmittance in front of this fragment
            const float2 aTf = __fmul2_rn(al, Tj);
            const float2 aT = make_float2(m0 ? aTf.x : 0.f, m1 ? aTf.y : 0.f);
            // dL/dalpha = Tj (g . c) - (g . S) / (1 - alpha)
            const float2 gc = __ffma2_rn(g2, f2(cb), __ffma2_rn(g1, f2(p1.w), __fmul2_rn(g0, f2(p1.z))));
            const float2 gS = __ffma2_rn(g2, S2, __ffma2_rn(g1, S1, __fmul2_rn(g0, S0)));
            const float2 dal = __ffma2_rn(make_float2(-inv.x, -inv.y), gS, __fmul2_rn(Tj, gc));
            S0 = __ffma2_rn(aT, f2(p1.z), S0);
            S1 = __ffma2_rn(aT, f2(p1.w), S1);
            S2 = __ffma2_rn(aT, f2(cb), S2);
            T = make_float2(m0 ? Tj.x : T.x, m1 ? Tj.y : T.y);
            // dL/do of the pixel = G dL/dalpha, zero where alpha is clamped at alpha_max;
            // dL/dpower = o times it
            const float2 dGf = __fmul2_rn(G, dal);
            const float2 dG = make_float2(m0 && al.x < rc.alpha_max ? dGf.x : 0.f,
                                          m1 && al.y < rc.alpha_max ? dGf.y : 0.f);
            // The slot takes dG-weighted moments of the pixel offsets: the record's
            // opacity and conic factors of the mean and conic gradients are applied
            // once per record, when its slots are summed (slot_grads_from_moments).
            float v[kSlotFloats];
            const float sG = dG.x + dG.y;
            const float2 gx = __fmul2_rn(dG, dx);
            v[0] = fmaf(dG.y, e.y, dG.x * e.x);   // sum dG e,  e = dx + k dy
            v[1] = sG * dy;                       // sum dG dy
            v[2] = fmaf(gx.y, dx.y, gx.x * dx.x); // sum dG dx^2
            v[3] = (gx.x + gx.y) * dy;            // sum dG dx dy
            v[4] = v[1] * dy;                     // sum dG dy^2
            v[5] = sG;                            // dL/do = sum dG
            v[6] = fmaf(aT.y, g0.y, aT.x * g0.x); // dL/dc = sum alpha T dL/dC
            v[7] = fmaf(aT.y, g1.y, aT.x * g1.x);
            v[8] = fmaf(aT.y, g2.y, aT.x * g2.x);
            const float sum = warp_reduce9(v, lane);
            if (red_own) s_part[warp][jj][red_q] = sum;
        }
        }
        __syncthreads(); // the round is walked
        if (at < count) {
            float sum[kSlotFloats];
#pragma unroll
            for (int q = 0; q < kSlotFloats; q++) sum[q] = 0.f;
#pragma unroll
            for (int w = 0; w < kWarps; w++) {
                if ((visited >> w) & 1u) {
#pragma unroll
                    for (int q = 0; q < kSlotFloats; q++) sum[q] += s_part[w][at][q];
                }
            }
            float *dst = a.slots + (size_t)slot * kSlotFloats;
#pragma unroll
            for (int q = 0; q < kSlotFloats; q++) dst[q] = sum[q];
        }
    }
    // entries after the batch of the tile's last contribution carry zero gradient
    for (int s = start + 32 * batches + threadIdx.x; s < end; s += kRT) {
        float *dst = a.slots + slot_of(a.inst_off, a.rect, a.vals[s], tx, ty) * kSlotFloats;
#pragma unroll
        for (int k = 0; k < kSlotFloats; k++) dst[k] = 0.f;
    }
    const unsigned f = __reduce_add_sync(0xffffffffu, (unsigned)ncomp);
    if (lane == 0 && f) atomicAdd(&a.ctr->composited, (unsigned long long)f);
}

cudaError_t launch_render_bwd(gs_workspace *ws, cudaStream_t st, const float *dL_drgb)
{
    if (ws->cams.total_tiles == 0) return cudaSuccess;
    BwdRenderArgs a;
    a.ranges = ws->ranges; a.vals = ws->sval; a.rd0 = ws->rd0; a.rd1 = ws->rd1; a.rd2 = ws->rd2;
    a.inst_off = ws->inst_off; a.rect = ws->rect; a.T_final = ws->T_final; a.n_contrib = ws->n_contrib;
    a.tile_last = ws->tile_last;
    a.visits = ws->visits;
    a.dL_drgb = dL_drgb; a.slots = ws->slots; a.ctr = ws->ctr;
    const unsigned grid = (unsigned)ws->cams.total_tiles;
    kt_begin(ws, GS_KT_RENDER_BWD, st);
    switch (tile_shape_id(ws->cams.tile_w, ws->cams.tile_h)) {
    case 0: launch_pdl(render_bwd_kernel<16, 16>, grid, SquareShape<16, 16>::threads, 0, st, a, ws->d_cams, ws->rc); break;
    case 1: launch_pdl(render_bwd_kernel<32, 8>, grid, SquareShape<32, 8>::threads, 0, st, a, ws->d_cams, ws->rc); break;
    case 2: launch_pdl(render_bwd_kernel<8, 32>, grid, SquareShape<8, 32>::threads, 0, st, a, ws->d_cams, ws->rc); break;
    case 3: launch_pdl(render_bwd_kernel<32, 16>, grid, SquareShape<32, 16>::threads, 0, st, a, ws->d_cams, ws->rc); break;
    case 4: launch_pdl(render_bwd_kernel<16, 8>, grid, SquareShape<16, 8>::threads, 0, st, a, ws->d_cams, ws->rc); break;
    case 5: launch_pdl(render_bwd_kernel<8, 16>, grid, SquareShape<8, 16>::threads, 0, st, a, ws->d_cams, ws->rc); break;
    default: return cudaErrorInvalidValue;
    }
    kt_end(ws, GS_KT_RENDER_BWD, st);
    note_launch();
    return cudaGetLastError();
}

// ---- importance sweep (colourless forward), alone or fused with the forward ----
//
// The walk of render_fwd_kernel with every record at its own opacity (the
// importance sweep never applies the Cull column it recomputes), in the same
// rounds: per visited entry the warp sums alpha T and the count of composited
// pixels over its lanes into shared memory; after the round the thread that
// staged an entry adds the warps' partials in warp order and writes the
// entry's importance slot.  Two block barriers per round (staged, walked).
// Once every pixel of the tile has stopped the remaining slots are zero.  With
// FWD the same walk also composites the training image (records marked culled
// composite nowhere in it): one evaluation of each entry's alpha serves both,
// the image, T and n_contrib equal render_fwd_kernel's and the slots this
// kernel's alone, bit for bit.  (Warps staging for themselves and meeting at
// arrival counters took 1.15 ms for the sweep of eight 1080p views of 3M
// Gaussians, whole pass, this 1.04.  The fused walk of the 5M view is no faster than
// it was, 148 and 147 us: the rounds pay for the visits that it notes besides.)

struct ImpArgs {
    const uint2 *ranges;
    const uint32_t *vals;
    const float4 *rd0, *rd1, *rd2;
    const uint32_t *inst_off;
    const uint2 *rect;
    float2 *slots;         // [I]: alpha-weight (float), composited pixels (uint32 bits)
    DevCounters *ctr;
    // FWD only
    float *rgb_out, *T_out, *T_ws;
    uint32_t *n_contrib;
    uint32_t *tile_last;   // the tile's largest n_contrib (atomic max; zeroed by the binning)
    uint32_t *visits;      // as render_fwd_kernel's, or NULL
};

template <int TW, int TH, bool FWD>
__global__ void __launch_bounds__(SquareShape<TW, TH>::threads, SquareShape<TW, TH>::imp_min_blocks)
    importance_raster_kernel(ImpArgs a, const CamTable *__restrict__ ctp, RenderConsts rc)
{
    griddep_wait(); // programmatic dependent launch: the previous kernel is complete
    constexpr int kWarps = SquareShape<TW, TH>::warps;
    constexpr int kRound = 32 * kWarps; // entries per round
    __shared__ float4 s0[kRound];
    __shared__ float4 s1[kRound];           // (D scaled, own opacity, training opacity, blue)
    __shared__ float2 s3[FWD ? kRound : 1]; // (red, green) of the training image
    __shared__ float2 s_part[kWarps][kRound];
    __shared__ unsigned s_mask[kWarps][kWarps]; // [square][batch of the round]
    const CamTable &ct = *ctp;
    if ((int)blockIdx.x >= ct.total_tiles) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const SquareGeom q = square_geom<TW, TH>(ct, blockIdx.x, warp, lane);
    const CamInfo &cam = *q.ci;
    const uint2 rg = a.ranges[blockIdx.x];
    const int start = (int)rg.x, end = (int)rg.y;
    const int px = q.tx * TW + q.lx, py = q.ty * TH + q.ly;
    const bool out0 = px >= cam.width || py >= cam.height, out1 = px + 1 >= cam.width || py >= cam.height;
    float2 Ti = f2(1.f);             // importance transmittance
    bool di0 = out0, di1 = out1;     // importance walk stopped
    float2 T = f2(1.f), Cr = f2(0.f), Cg = f2(0.f), Cb = f2(0.f); // training image (FWD)
    uint32_t last0 = 0, last1 = 0;
    bool dn0 = out0, dn1 = out1;
    int first = start;
    for (; first < end; first += kRound) {
        const int at = threadIdx.x; // the thread's entry of the round
        unsigned meets = 0;         // squares it may composite in
        uint32_t slot = 0;
        if (first + at < end) {
            const uint32_t r = a.vals[first + at];
            const float4 r0 = a.rd0[r], r1 = a.rd1[r], r2 = a.rd2[r];
            slot = (uint32_t)slot_of(a.inst_off, a.rect, r, q.tx, q.ty);
            const float4 e0 = stage_e0_at(r0, r2, q.ox, q.oy);
            s0[at] = e0;
            s1[at] = make_float4(stage_D(r1), r1.y, r2.w != 0.f ? 0.f : r1.y, r2.x);
            if (FWD) s3[FWD ? at : 0] = make_float2(r1.z, r1.w);
            // the record's own opacity: the training opacity is the same or 0
            const SquareTest test(r0, r1.x, r1.y, rc.alpha_min, e0.x, e0.y);
#pragma unroll
            for (int k = 0; k < kWarps; k++)
                meets |= test.meets(8.f * (k % SquareShape<TW, TH>::wx) + 0.5f, 8.f * (k / SquareShape<TW, TH>::wx) + 0.5f) ? 1u << k : 0u;
        }
#pragma unroll
        for (int k = 0; k < kWarps; k++) {
            const unsigned m = __ballot_sync(0xffffffffu, (meets >> k) & 1u);
            if (lane == k) s_mask[k][warp] = m;
        }
        if (__syncthreads_and(di0 && di1 && (!FWD || (dn0 && dn1)))) break; // staged; every pixel has stopped
        for (int sub = 0, b = first; sub < kWarps && b < end; sub++, b += 32) {
            if (__all_sync(0xffffffffu, di0 && di1 && (!FWD || (dn0 && dn1)))) { // the warp's pixels have stopped
                s_part[warp][32 * sub + lane] = make_float2(0.f, __uint_as_float(0u));
                continue;
            }
            unsigned comp = 0; // FWD: entries that composite in the lane's pixels of the image
            for (unsigned m = s_mask[warp][sub]; m != 0u;) {
                const int jj = __ffs(m) - 1; // front to back
                m &= m - 1u;
                const float4 p0 = s0[32 * sub + jj];
                const float4 p1 = s1[32 * sub + jj];
                float2 dx, e;
                float dy;
                const float2 pw = pair_power(p0, p1.x, q.pxc, q.pyc, dx, dy, e);
                float2 G;
                const float2 al = pair_alpha(pw, p1.y, rc.alpha_max, G);
                if (FWD && p1.z != 0.f) { // the training image: render_fwd_kernel's update
                    const uint32_t pos = (uint32_t)(b - start + jj + 1);
                    const float2 tT = __ffma2_rn(make_float2(-T.x, -T.y), al, T);
                    const bool ok0 = !dn0 && al.x >= rc.alpha_min, ok1 = !dn1 && al.y >= rc.alpha_min;
                    const bool st0 = ok0 && tT.x < rc.T_min, st1 = ok1 && tT.y < rc.T_min;
                    const bool c0 = ok0 && !st0, c1 = ok1 && !st1;
                    dn0 = dn0 || st0;
                    dn1 = dn1 || st1;
                    if (c0 || c1) comp |= 1u << jj;
                    const float2 ae = make_float2(c0 ? al.x : 0.f, c1 ? al.y : 0.f);
                    const float2 w = __fmul2_rn(ae, T);
                    const float2 rgc = s3[FWD ? 32 * sub + jj : 0];
                    Cr = __ffma2_rn(w, f2(rgc.x), Cr);
                    Cg = __ffma2_rn(w, f2(rgc.y), Cg);
                    Cb = __ffma2_rn(w, f2(p1.w), Cb);
                    T = __ffma2_rn(make_float2(-T.x, -T.y), ae, T);
                    last0 = c0 ? pos : last0;
                    last1 = c1 ? pos : last1;
                }
                // the importance sweep
                const float2 tT = __ffma2_rn(make_float2(-Ti.x, -Ti.y), al, Ti);
                const bool ok0 = !di0 && al.x >= rc.alpha_min, ok1 = !di1 && al.y >= rc.alpha_min;
                const bool st0 = ok0 && tT.x < rc.T_min, st1 = ok1 && tT.y < rc.T_min;
                const bool c0 = ok0 && !st0, c1 = ok1 && !st1;
                di0 = di0 || st0;
                di1 = di1 || st1;
                const float2 ae = make_float2(c0 ? al.x : 0.f, c1 ? al.y : 0.f);
                const float2 w = __fmul2_rn(ae, Ti);
                float wv = w.x + w.y;
                uint32_t av = (uint32_t)c0 + (uint32_t)c1;
                Ti = __ffma2_rn(make_float2(-Ti.x, -Ti.y), ae, Ti);
                if (__any_sync(0xffffffffu, av != 0)) {
                    wv = warp_sum_f(wv);
                    av = __reduce_add_sync(0xffffffffu, av);
                }
                if (lane == 0) s_part[warp][32 * sub + jj] = make_float2(wv, __uint_as_float(av));
            }
            if (FWD && a.visits) put_visits<kWarps>(a.visits, start, b, warp, comp);
        }
        __syncthreads(); // the round is walked
        if (first + at < end) {
            float ws = 0.f;
            uint32_t as = 0;
#pragma unroll
            for (int w = 0; w < kWarps; w++)
                if ((meets >> w) & 1u) {
                    const float2 pv = s_part[w][at];
                    ws += pv.x;
                    as += __float_as_uint(pv.y);
                }
            a.slots[slot] = make_float2(ws, __uint_as_float(as));
        }
    }
    for (int at = first + (int)threadIdx.x; at < end; at += kRound) // entries behind the last pixel's stop
        a.slots[slot_of(a.inst_off, a.rect, a.vals[at], q.tx, q.ty)] = make_float2(0.f, __uint_as_float(0u));
    if (FWD) {
        const long long np = (long long)cam.width * cam.height;
        float *img = a.rgb_out + 3 * cam.pix_base;
#pragma unroll
        for (int h = 0; h < 2; h++) {
            if (px + h >= cam.width || py >= cam.height) continue;
            const float Tk = h ? T.y : T.x;
            const long long pix = (long long)py * cam.width + px + h;
            img[pix] = (h ? Cr.y : Cr.x) + Tk * rc.bg[0];
            img[np + pix] = (h ? Cg.y : Cg.x) + Tk * rc.bg[1];
            img[2 * np + pix] = (h ? Cb.y : Cb.x) + Tk * rc.bg[2];
            const long long gp = cam.pix_base + pix;
            if (a.T_out) a.T_out[gp] = Tk;
            a.T_ws[gp] = Tk;
            a.n_contrib[gp] = h ? last1 : last0;
        }
        const unsigned wl = __reduce_max_sync(0xffffffffu, max(last0, last1));
        if (lane == 0 && wl != 0u) atomicMax(&a.tile_last[blockIdx.x], wl);
    }
}

template <bool FWD> static cudaError_t importance_launch(gs_workspace *ws, cudaStream_t st, const ImpArgs &a)
{
    const unsigned grid = (unsigned)ws->cams.total_tiles;
    switch (tile_shape_id(ws->cams.tile_w, ws->cams.tile_h)) {
    case 0: launch_pdl(importance_raster_kernel<16, 16, FWD>, grid, SquareShape<16, 16>::threads, 0, st, a, ws->d_cams, ws->rc); break;
    case 1: launch_pdl(importance_raster_kernel<32, 8, FWD>, grid, SquareShape<32, 8>::threads, 0, st, a, ws->d_cams, ws->rc); break;
    case 2: launch_pdl(importance_raster_kernel<8, 32, FWD>, grid, SquareShape<8, 32>::threads, 0, st, a, ws->d_cams, ws->rc); break;
    case 3: launch_pdl(importance_raster_kernel<32, 16, FWD>, grid, SquareShape<32, 16>::threads, 0, st, a, ws->d_cams, ws->rc); break;
    case 4: launch_pdl(importance_raster_kernel<16, 8, FWD>, grid, SquareShape<16, 8>::threads, 0, st, a, ws->d_cams, ws->rc); break;
    case 5: launch_pdl(importance_raster_kernel<8, 16, FWD>, grid, SquareShape<8, 16>::threads, 0, st, a, ws->d_cams, ws->rc); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaSuccess;
}

static ImpArgs importance_args(gs_workspace *ws)
{
    ImpArgs a{};
    a.ranges = ws->ranges; a.vals = ws->sval; a.rd0 = ws->rd0; a.rd1 = ws->rd1; a.rd2 = ws->rd2;
    a.inst_off = ws->inst_off; a.rect = ws->rect; a.slots = ws->imp_slots; a.ctr = ws->ctr;
    return a;
}

cudaError_t launch_importance_raster(gs_workspace *ws, cudaStream_t st)
{
    if (ws->cams.total_tiles == 0) return cudaSuccess;
    kt_begin(ws, GS_KT_IMPORTANCE, st);
    cudaError_t e = importance_launch<false>(ws, st, importance_args(ws));
    if (e != cudaSuccess) return e;
    kt_end(ws, GS_KT_IMPORTANCE, st);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_render_fwd_importance(gs_workspace *ws, cudaStream_t st, float *rgb, float *T_out)
{
    if (ws->cams.total_tiles == 0) return cudaSuccess;
    ImpArgs a = importance_args(ws);
    a.rgb_out = rgb; a.T_out = T_out; a.T_ws = ws->T_final; a.n_contrib = ws->n_contrib; a.tile_last = ws->tile_last;
    a.visits = ws->visits;
    kt_begin(ws, GS_KT_RENDER_FWD, st);
    cudaError_t e = importance_launch<true>(ws, st, a);
    if (e != cudaSuccess) return e;
    kt_end(ws, GS_KT_RENDER_FWD, st);
    note_launch();
    return cudaGetLastError();
}

} // namespace gs
