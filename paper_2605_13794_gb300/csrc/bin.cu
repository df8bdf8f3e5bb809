// bin.cu -- the tile lists of a binning (App. A: tile-based rasterisation of
// depth-ordered projected Gaussians), built by tile first and sorted by depth
// inside each tile.
//
// Order of the work:
//   1. count: every instance adds one to its tile's count and keeps the count
//      it found, its rank in the tile (in whatever order they came).  The
//      projection numbers the instances in record order ((Gaussian, camera)
//      order, inst_off, the base of the gradient slots); blocks take equal
//      chunks of them, so a record of thousands of tiles is spread over many;
//   2. tile scan: exclusive scan of the tile counts (decoupled look-back over
//      blocks of tiles) gives each tile's range;
//   3. scatter: every instance writes its (depth key, record) pair at its
//      tile's start plus its rank;
//   4. per-tile sort of the (depth bits, record) pairs -- unique keys, so the
//      order is the same in any scatter order -- in registers (bitonic
//      networks over shuffles): up to kWarpSort entries in one warp, up to
//      kBlockSort in the four warps of a block, which then rank their runs
//      against each other, longer lists in sorted chunks merged through a
//      scratch copy in global memory.
// Bound by the latency of atomics and scattered stores.  Dealing out records
// (32 to a warp or block) left whole SMs waiting for the blocks that held
// records of hundreds of tiles: the count and scatter of the 1.14M instances
// of the 5M city at 1080p took 17 + 24 us and take 13 + 11 in equal chunks of
// instances, the 11.2M of 24 mixed views 78 + 233 us and 95 + 147.
// The final order of a tile's list is (depth bits, record): depth ties go to
// the lower record, i.e. the lower Gaussian index.  Counts stay on the
// device; nothing here synchronises with the host.
#include <algorithm>

#include "gs_internal.cuh"

namespace gs {

constexpr int kBinThreads = 128;       // threads per block of the count and scatter passes
constexpr int kBinItems = kBinChunk / kBinThreads; // instances per thread
constexpr int kTileScanItems = 4;      // tiles per thread of the tile scan (1024 per block)
constexpr int kSortWarps = 4;          // warps (and tiles) per block of the per-tile sort
constexpr int kWarpSort = 256;         // entries one warp sorts alone (8 per lane)
constexpr int kBlockSort = 2048;       // entries a block sorts in shared memory (16 per lane)

struct BinArgs {
    const uint32_t *tt;
    const uint2 *rect;
    const uint16_t *rec_cam;
    const uint32_t *dkey;          // FP32 bits of each record's camera depth
    const uint32_t *inst_off;      // first instance of each record (record order)
    const uint32_t *chunk_rec;     // record of each chunk's first instance
    uint32_t *rank;                // [instances] rank of each instance among those of its tile
    uint32_t *tile_cnt;            // [tiles] instances per tile (zero before the count)
    uint32_t *tile_last;           // [tiles] the forward's largest n_contrib per tile: zeroed here
    uint2 *ranges;                 // [tiles] [start, end) of each tile's list
    uint2 *pairs;                  // [instances] scattered (depth key, record) pairs
    uint32_t *sval;                // [instances] the sorted records
    uint2 *scratch;                // [instances] scratch of the merges of long lists
    unsigned long long *lb_tiles;  // look-back of the tile scan (ticket at word 0)
    DevCounters *ctr;
    unsigned long long max_instances;
    int total_tiles;
};

// The records of one chunk of kBinChunk consecutive instances, in shared memory.
struct BinRecs {
    uint32_t off[kBinChunk + 1];   // first instance
    uint2 rect[kBinChunk + 1];
    int tile_base[kBinChunk + 1], tiles_x[kBinChunk + 1];
};

// Instances of the tile lists: those of the records there are, at most the
// capacity (more is an error, which the count pass reports).  Past the record
// capacity (an error already) only the kept records' count.
__device__ __forceinline__ unsigned long long bin_instances(const BinArgs &a, unsigned long long nrec,
                                                            unsigned long long &needed)
{
    needed = a.ctr->inst_total;
    if (a.ctr->records_needed > nrec) needed = nrec ? (unsigned long long)a.inst_off[nrec - 1] + a.tt[nrec - 1] : 0ull;
    return needed < a.max_instances ? needed : a.max_instances;
}

// Loads the records of chunk b (ninst instances in all); returns the first.
// (Whatever a projection that gave up left behind, records stay below nrec.)
__device__ __forceinline__ uint32_t bin_load(const BinArgs &a, const CamTable &ct, BinRecs &s, unsigned long long b,
                                             unsigned long long ninst, uint32_t nrec, uint32_t &count)
{
    const uint32_t r0 = min(a.chunk_rec[b], nrec - 1u);
    const uint32_t r1 = (b + 1) * kBinChunk < ninst ? max(r0, min(a.chunk_rec[b + 1], nrec - 1u)) : nrec - 1u;
    count = min(r1 - r0 + 1u, (uint32_t)kBinChunk + 1u);
    for (uint32_t i = threadIdx.x; i < count; i += kBinThreads) {
        const uint32_t r = r0 + i;
        const int cam = a.rec_cam[r];
        s.off[i] = a.inst_off[r];
        s.rect[i] = a.rect[r];
        s.tile_base[i] = ct.c[cam].tile_base;
        s.tiles_x[i] = ct.c[cam].tiles_x;
    }
    __syncthreads();
    return r0;
}

// Instance j: its record (as its slot among the chunk's) and its global tile id.
__device__ __forceinline__ uint32_t bin_instance(const BinRecs &s, uint32_t count, uint32_t j, uint32_t &slot)
{
    uint32_t lo = 0, hi = count - 1; // the last record whose first instance is at most j
    while (lo < hi) {
        const uint32_t mid = (lo + hi + 1) >> 1;
        if (s.off[mid] <= j) lo = mid; else hi = mid - 1;
    }
    slot = lo;
    const uint32_t local = j - s.off[lo];
    int x0, y0, x1, y1;
    unpack_rect(s.rect[lo], x0, y0, x1, y1);
    const uint32_t w = (uint32_t)(x1 - x0);
    // local / w: below 2^20 the rounded quotient of local + 1/2 cannot reach the
    // next integer (its error, 2^-22 of at most 2^20 / w, is below 1 / (2 w))
    const uint32_t q = local < (1u << 20) ? (uint32_t)__fdividef((float)local + 0.5f, (float)w) : local / w;
    return (uint32_t)(s.tile_base[lo] + (y0 + (int)q) * s.tiles_x[lo] + x0 + (int)(local - q * w));
}

// 1. Count: every tile's count and every instance's rank in its tile.  Blocks
// stride over the chunks there are (not as many as the capacity could hold).
__global__ void __launch_bounds__(kBinThreads) bin_count_kernel(BinArgs a, const CamTable *__restrict__ ctp)
{
    griddep_wait(); // programmatic dependent launch: the previous kernel is complete
    __shared__ BinRecs s;
    const unsigned long long nrec = a.ctr->n_records;
    unsigned long long needed;
    const unsigned long long ninst = bin_instances(a, nrec, needed);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.ctr->instances_needed = needed;
        a.ctr->n_instances = ninst;
        if (needed > a.max_instances) set_error(a.ctr, GS_ERR_CAPACITY, kSiteEmit);
    }
    for (unsigned long long b = blockIdx.x; b * kBinChunk < ninst; b += gridDim.x) {
        uint32_t count;
        bin_load(a, *ctp, s, b, ninst, (uint32_t)nrec, count);
        uint32_t rank[kBinItems];
#pragma unroll
        for (int q = 0; q < kBinItems; q++) { // the atomics in flight together
            const unsigned long long j = b * kBinChunk + q * kBinThreads + threadIdx.x;
            if (j >= ninst) continue;
            uint32_t slot;
            const uint32_t t = bin_instance(s, count, (uint32_t)j, slot);
            rank[q] = t < (uint32_t)a.total_tiles ? atomicAdd(&a.tile_cnt[t], 1u) : 0u;
        }
#pragma unroll
        for (int q = 0; q < kBinItems; q++) {
            const unsigned long long j = b * kBinChunk + q * kBinThreads + threadIdx.x;
            if (j < ninst) a.rank[j] = rank[q];
        }
        __syncthreads(); // every thread is done with the chunk's records
    }
}

// 2. Tile scan: exclusive scan of the tile counts; ranges clamped to the
// instance capacity (an overflow is already an error); the tile counts and the
// forward's per-tile maxima of n_contrib cleared.
__global__ void __launch_bounds__(256) tile_scan_kernel(BinArgs a)
{
    griddep_wait(); // programmatic dependent launch: the previous kernel is complete
    __shared__ unsigned long long s_warp[8];
    __shared__ unsigned s_bid;
    __shared__ unsigned long long s_base;
    if (threadIdx.x == 0) s_bid = atomicAdd((unsigned *)a.lb_tiles, 1u);
    __syncthreads();
    const unsigned bid = s_bid;
    const long long t0 = ((long long)bid * 256 + threadIdx.x) * kTileScanItems;
    if ((long long)bid * 256 * kTileScanItems >= a.total_tiles) return;
    uint32_t cnt[kTileScanItems];
    unsigned long long sum = 0;
#pragma unroll
    for (int q = 0; q < kTileScanItems; q++) {
        cnt[q] = t0 + q < a.total_tiles ? a.tile_cnt[t0 + q] : 0u;
        sum += cnt[q];
    }
    unsigned long long total;
    const unsigned long long excl = block_exclusive_scan_256<unsigned long long>(sum, s_warp, total);
    if (threadIdx.x < 32) {
        const unsigned long long b = lookback_exclusive(a.lb_tiles + 1, bid, total, a.ctr, kSiteEmit);
        if (threadIdx.x == 0) s_base = b;
    }
    __syncthreads();
    unsigned long long off = s_base + excl;
#pragma unroll
    for (int q = 0; q < kTileScanItems; q++) {
        if (t0 + q >= a.total_tiles) break;
        const unsigned long long e = off + cnt[q];
        a.ranges[t0 + q] = make_uint2((uint32_t)min(off, a.max_instances), (uint32_t)min(e, a.max_instances));
        a.tile_last[t0 + q] = 0u;
        a.tile_cnt[t0 + q] = 0u; // for the next binning
        off = e;
    }
}

// 3. Scatter: every instance's pair to its place, one store of eight bytes.
__global__ void __launch_bounds__(kBinThreads) bin_scatter_kernel(BinArgs a, const CamTable *__restrict__ ctp)
{
    griddep_wait(); // programmatic dependent launch: the previous kernel is complete
    __shared__ BinRecs s;
    const unsigned long long nrec = a.ctr->n_records;
    unsigned long long needed;
    const unsigned long long ninst = bin_instances(a, nrec, needed);
    for (unsigned long long b = blockIdx.x; b * kBinChunk < ninst; b += gridDim.x) {
        uint32_t rank[kBinItems];
#pragma unroll
        for (int q = 0; q < kBinItems; q++) {
            const unsigned long long j = b * kBinChunk + q * kBinThreads + threadIdx.x;
            rank[q] = j < ninst ? a.rank[j] : 0u;
        }
        uint32_t count;
        const uint32_t r0 = bin_load(a, *ctp, s, b, ninst, (uint32_t)nrec, count);
#pragma unroll
        for (int q = 0; q < kBinItems; q++) {
            const unsigned long long j = b * kBinChunk + q * kBinThreads + threadIdx.x;
            if (j >= ninst) continue;
            uint32_t slot;
            const uint32_t t = bin_instance(s, count, (uint32_t)j, slot);
            if (t >= (uint32_t)a.total_tiles) continue;
            const unsigned long long pos = (unsigned long long)a.ranges[t].x + rank[q];
            if (pos < a.max_instances) a.pairs[pos] = make_uint2(a.dkey[r0 + slot], r0 + slot);
        }
        __syncthreads(); // every thread is done with the chunk's records
    }
}

// Ascending bitonic sort of the warp's 32 * E keys held in registers: key
// x[e] of lane l is element g = E l + e.  A stage of stride s < E pairs
// registers of one lane (e, e ^ s); a stage of stride s >= E pairs lanes
// (l, l ^ s / E) by a shuffle.  The network is fixed, so the result is the
// sorted order of the keys (all distinct) whatever order they came in.
template <int E> __device__ __forceinline__ void warp_sort_regs(unsigned long long (&x)[E])
{
    // the loops over sizes and lane strides stay loops (a short kernel body
    // for the instruction cache); the registers' indices are unrolled
    const int lane = threadIdx.x & 31;
    for (int size = 2; size <= 32 * E; size <<= 1) {
        for (int stride = size >> 1; stride >= E; stride >>= 1) {
            const int ls = stride / E;
            const bool lower = (lane & ls) == 0;
#pragma unroll
            for (int e = 0; e < E; e++) {
                const unsigned long long u = x[e];
                const unsigned lo = __shfl_xor_sync(0xffffffffu, (unsigned)u, ls);
                const unsigned hi = __shfl_xor_sync(0xffffffffu, (unsigned)(u >> 32), ls);
                const unsigned long long v = ((unsigned long long)hi << 32) | lo;
                const bool up = ((lane * E + e) & size) == 0;
                x[e] = (u < v) == (lower == up) ? u : v;
            }
        }
#pragma unroll
        for (int stride = E / 2; stride > 0; stride >>= 1) {
            if (stride >= size) continue;
#pragma unroll
            for (int e = 0; e < E; e++) {
                if (e & stride) continue; // the lower element of each pair
                const bool up = ((lane * E + e) & size) == 0;
                const unsigned long long u = x[e], v = x[e ^ stride];
                const bool swap = (u > v) == up;
                x[e] = swap ? v : u;
                x[e ^ stride] = swap ? u : v;
            }
        }
    }
}

__device__ __forceinline__ unsigned long long key_of(uint2 p) { return ((unsigned long long)p.x << 32) | p.y; }

// Number of the first d outputs of the merge of X (nx) and Y (ny) that come
// from X (merge path; keys unique).
__device__ __forceinline__ uint32_t merge_split(const uint2 *x, uint32_t nx, const uint2 *y, uint32_t ny, uint32_t d)
{
    uint32_t lo = d > ny ? d - ny : 0u, hi = d < nx ? d : nx;
    while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (key_of(x[mid]) < key_of(y[d - 1 - mid])) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// The same network on 32-bit keys: a shuffle and a minimum or maximum per element
// and stage, against two shuffles, a 64-bit compare and two selects.  Within runs
// shorter than E the direction is the register's, known to the compiler, and from
// there on the lane's alone, one flag per stage (computed per element, as above,
// it cost as much as the exchange: 28 us for 24 in the 5M city at 1080p).
template <int E> __device__ __forceinline__ void warp_sort_regs(unsigned (&x)[E])
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int size = 2; size < E; size <<= 1) {
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
#pragma unroll
            for (int e = 0; e < E; e++) {
                if (e & stride) continue; // the lower element of each pair
                const unsigned u = x[e], v = x[e ^ stride];
                x[e] = e & size ? max(u, v) : min(u, v);
                x[e ^ stride] = e & size ? min(u, v) : max(u, v);
            }
        }
    }
    for (int run = E > 1 ? 1 : 2; run <= 32; run <<= 1) { // runs of E * run elements
        const bool up = (lane & run) == 0;
        for (int ls = run >> 1; ls > 0; ls >>= 1) {
            const bool least = ((lane & ls) == 0) == up;
#pragma unroll
            for (int e = 0; e < E; e++) {
                const unsigned v = __shfl_xor_sync(0xffffffffu, x[e], ls);
                x[e] = least ? min(x[e], v) : max(x[e], v);
            }
        }
#pragma unroll
        for (int stride = E / 2; stride > 0; stride >>= 1) {
#pragma unroll
            for (int e = 0; e < E; e++) {
                if (e & stride) continue;
                const unsigned u = x[e], v = x[e ^ stride];
                x[e] = up ? min(u, v) : max(u, v);
                x[e ^ stride] = up ? max(u, v) : min(u, v);
            }
        }
    }
}

// The warp's n <= 32 * E keys at p in order: y[e] of lane l is key E l + e, the
// places past n hold the largest key.  The keys are ordered by 32 bits, the
// depth above the list's least one in as many bits as the place in the list
// leaves (all of them in a list whose depths lie within one binade or so) and
// that place, which fetches the key from its copy in shared memory (stage, 32 E
// of the warp's own).  Two keys that agree in those depth bits (equal depths,
// above all) are in no order: then the 64-bit network sorts the list.
// kWarpSort is 256: with 128, the lists of 129 to 256 entries go to the block, which
// makes no difference beyond the repeats' (importance pass of eight views).
template <int E>
__device__ __forceinline__ void sort_keys(const uint2 *p, uint32_t n, unsigned long long *stage,
                                          unsigned long long (&y)[E])
{
    constexpr int kBits = E == 1 ? 5 : E == 2 ? 6 : E == 4 ? 7 : E == 8 ? 8 : 9; // log2(32 E)
    const int lane = threadIdx.x & 31;
    unsigned x[E], least = ~0u, most = 0u;
#pragma unroll
    for (int e = 0; e < E; e++) {
        const uint32_t g = (uint32_t)(e * 32 + lane);
        const uint2 q = g < n ? p[g] : make_uint2(~0u, ~0u);
        stage[g] = key_of(q);
        x[e] = q.x;
        least = min(least, q.x);
        most = max(most, g < n ? q.x : 0u);
    }
    least = __reduce_min_sync(0xffffffffu, least);
    most = __reduce_max_sync(0xffffffffu, most);
    const int shift = max(0, 32 - __clz(most - least) + kBits - 32);
#pragma unroll
    for (int e = 0; e < E; e++) {
        const uint32_t g = (uint32_t)(e * 32 + lane);
        x[e] = g < n ? ((x[e] - least) >> shift) << kBits | g : ~0u;
    }
    warp_sort_regs<E>(x);
    __syncwarp(); // the staged keys are in place
    bool clash = false;
    const unsigned next = __shfl_down_sync(0xffffffffu, x[0], 1);
#pragma unroll
    for (int e = 0; e < E; e++) {
        const unsigned after = e + 1 < E ? x[e + 1 < E ? e + 1 : 0] : next;
        clash = clash || ((x[e] ^ after) >> kBits == 0u && (uint32_t)(lane * E + e + 1) < n);
        y[e] = stage[x[e] & (32u * E - 1u)];
    }
    if (__any_sync(0xffffffffu, clash)) {
#pragma unroll
        for (int e = 0; e < E; e++) y[e] = stage[e * 32 + lane];
        warp_sort_regs<E>(y);
    }
    __syncwarp(); // the staged keys are read
}

// One warp sorts the n <= 32 * E keys at p and writes the records in order.
template <int E>
__device__ __forceinline__ void warp_sort(const uint2 *p, uint32_t n, unsigned long long *stage, uint32_t *out)
{
    const int lane = threadIdx.x & 31;
    unsigned long long y[E];
    sort_keys<E>(p, n, stage, y);
#pragma unroll
    for (int e = 0; e < E; e++)
        if ((uint32_t)(lane * E + e) < n) out[lane * E + e] = (uint32_t)y[e];
}

// The block sorts the n <= 32 * E * kSortWarps keys at p: each warp a run of a
// quarter of them, in registers, into shared memory; then every key's place is
// its place in its run plus the keys below it in each other run (a binary
// search; keys unique).  Writes the records to out, or the keys to outk.
template <int E>
__device__ __forceinline__ void block_sort(const uint2 *p, uint32_t n, unsigned long long (*s)[kBlockSort / kSortWarps],
                                           uint32_t *out, uint2 *outk)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t run = (n + kSortWarps - 1) / kSortWarps;
    const uint32_t first = min(warp * run, n), len = min(run, n - first);
    {
        unsigned long long y[E];
        sort_keys<E>(p + first, len, s[warp], y);
#pragma unroll
        for (int e = 0; e < E; e++) s[warp][lane * E + e] = y[e];
    }
    __syncthreads();
    for (uint32_t i = lane; i < len; i += 32) {
        const unsigned long long key = s[warp][i];
        uint32_t place = i;
#pragma unroll
        for (int o = 1; o < kSortWarps; o++) {
            const int r = (warp + o) % kSortWarps;
            uint32_t lo = 0; // keys of run r below this one (the padding is above every key)
#pragma unroll
            for (uint32_t step = 16 * E; step > 0; step >>= 1) lo += s[r][lo + step - 1] < key ? step : 0;
            lo += s[r][lo] < key ? 1u : 0u;
            place += lo;
        }
        if (outk) outk[place] = make_uint2((uint32_t)(key >> 32), (uint32_t)key);
        else out[place] = (uint32_t)key;
    }
    __syncthreads(); // the runs are read
}

__device__ __forceinline__ void block_sort_any(const uint2 *p, uint32_t n,
                                               unsigned long long (*s)[kBlockSort / kSortWarps], uint32_t *out,
                                               uint2 *outk)
{
    constexpr uint32_t kRun = 32 * kSortWarps;
    if (n <= 2 * kRun) block_sort<2>(p, n, s, out, outk);
    else if (n <= 4 * kRun) block_sort<4>(p, n, s, out, outk);
    else if (n <= 8 * kRun) block_sort<8>(p, n, s, out, outk);
    else block_sort<16>(p, n, s, out, outk);
}

// 4. Per-tile sort of the scattered pairs; the sorted records end in sval.  A
// block has per_block <= kSortWarps tiles: each warp sorts its own if it is
// short, then the whole block the longer ones, one after the other, so that a
// view of few tiles with long lists does not wait for one warp's chain of
// stages.
__global__ void __launch_bounds__(32 * kSortWarps, 8) tile_sort_kernel(BinArgs a, int per_block)
{
    griddep_wait(); // programmatic dependent launch: the previous kernel is complete
    __shared__ unsigned long long s_run[kSortWarps][kBlockSort / kSortWarps];
    __shared__ uint2 s_rg[kSortWarps];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long t = (long long)blockIdx.x * per_block + warp;
    uint2 rg = make_uint2(0u, 0u);
    if (warp < per_block && t < a.total_tiles) {
        rg = a.ranges[t];
        if (lane == 0 && t % (256 * kTileScanItems) == 0) { // the tile scan's look-back words, for the next binning
            a.lb_tiles[1 + t / (256 * kTileScanItems)] = 0ull;
            if (t == 0) a.lb_tiles[0] = 0ull;
        }
    }
    const uint32_t mine = rg.y - rg.x;
    if (lane == 0) s_rg[warp] = rg;
    if (mine > 0 && mine <= (uint32_t)kWarpSort) {
        const uint2 *p = a.pairs + rg.x;
        uint32_t *out = a.sval + rg.x;
        unsigned long long *stage = s_run[warp];
        if (mine <= 32) warp_sort<1>(p, mine, stage, out);
        else if (mine <= 64) warp_sort<2>(p, mine, stage, out);
        else if (mine <= 128) warp_sort<4>(p, mine, stage, out);
        else warp_sort<8>(p, mine, stage, out);
    }
    if (!__syncthreads_or(mine > (uint32_t)kWarpSort)) return;
    for (int w = 0; w < kSortWarps; w++) {
        const uint32_t start = s_rg[w].x, n = s_rg[w].y - start;
        if (n <= (uint32_t)kWarpSort) continue; // the same for the whole block
        uint2 *pairs = a.pairs + start, *scratch = a.scratch + start;
        if (n <= (uint32_t)kBlockSort) {
            block_sort_any(pairs, n, s_run, a.sval + start, nullptr);
            continue;
        }
        // a longer list: sorted chunks of kBlockSort into the scratch, then
        // pairwise merges of runs, the threads on equal shares of each merge
        for (uint32_t c0 = 0; c0 < n; c0 += kBlockSort)
            block_sort_any(pairs + c0, min((uint32_t)kBlockSort, n - c0), s_run, nullptr, scratch + c0);
        const uint2 *src = scratch;
        uint2 *dst = pairs;
        constexpr uint32_t kThreads = 32 * kSortWarps;
        for (uint32_t width = kBlockSort; width < n; width <<= 1) {
            __syncthreads(); // the previous level's writes, before this level reads them
            for (uint32_t p = 0; p < n; p += 2 * width) {
                const uint32_t nx = min(width, n - p), ny = p + width < n ? min(width, n - p - width) : 0u;
                const uint2 *x = src + p, *y = src + p + nx;
                const uint32_t L = nx + ny, d0 = (uint32_t)(((unsigned long long)L * threadIdx.x) / kThreads),
                               d1 = (uint32_t)(((unsigned long long)L * (threadIdx.x + 1)) / kThreads);
                uint32_t i = merge_split(x, nx, y, ny, d0), j = d0 - i;
                for (uint32_t d = d0; d < d1; d++) {
                    const bool take_x = j >= ny || (i < nx && key_of(x[i]) < key_of(y[j]));
                    dst[p + d] = take_x ? x[i] : y[j];
                    if (take_x) i++;
                    else j++;
                }
            }
            uint2 *was = const_cast<uint2 *>(src);
            src = dst;
            dst = was;
        }
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < n; i += kThreads) a.sval[start + i] = src[i].y;
    }
}

// The tile lists of the records of the last preprocess: ranges and
// ws->sval (records sorted by (tile, depth bits, record)), the
// instance counters.  Scratch: tile_cnt, bin_lb, pairs, inst_rank, and the
// importance slots (for merges; they are written only after the binning).
// tile_cnt and bin_lb are zero between calls: the pass after the last reader
// clears them, so a binning needs no memset.
cudaError_t launch_bin(gs_workspace *ws, cudaStream_t st)
{
    const int tiles = ws->cams.total_tiles;
    const unsigned sblocks = (unsigned)((tiles + 256 * kTileScanItems - 1) / (256 * kTileScanItems));
    if ((size_t)sblocks + 1 > ws->bin_lb_words) return cudaErrorInvalidValue; // sized at creation
    BinArgs a;
    a.tt = ws->tt; a.rect = ws->rect; a.rec_cam = ws->rec_cam; a.dkey = ws->dkey;
    a.inst_off = ws->inst_off; a.chunk_rec = ws->chunk_rec; a.rank = ws->inst_rank; a.tile_cnt = ws->tile_cnt; a.ranges = ws->ranges;
    a.tile_last = ws->tile_last;
    a.pairs = ws->pairs; a.sval = ws->sval; a.scratch = reinterpret_cast<uint2 *>(ws->imp_slots);
    a.lb_tiles = ws->bin_lb;
    a.ctr = ws->ctr; a.max_instances = (unsigned long long)ws->cap.max_instances; a.total_tiles = tiles;
    // as many blocks as stay resident, striding over the chunks
    const unsigned long long chunks = (a.max_instances + kBinChunk - 1) / kBinChunk;
    const unsigned rblocks = (unsigned)std::max(1ull, std::min(chunks, 16ull * ws->sm_count));
    kt_begin(ws, GS_KT_BIN_COUNT, st);
    launch_pdl(bin_count_kernel, rblocks, kBinThreads, 0, st, a, ws->d_cams);
    kt_end(ws, GS_KT_BIN_COUNT, st);
    note_launch();
    kt_begin(ws, GS_KT_BIN_SORT, st);
    if (tiles > 0) {
        launch_pdl(tile_scan_kernel, sblocks, 256, 0, st, a);
        note_launch();
    }
    launch_pdl(bin_scatter_kernel, rblocks, kBinThreads, 0, st, a, ws->d_cams);
    note_launch();
    if (tiles > 0) {
        // one tile per block while all the blocks are resident at once (eight per SM): the long lists of a
        // small view then sort side by side, not four to a block one after the other (384 tiles of 300
        // entries: 28 us with four, 9 with one)
        const int per_block = tiles <= 8 * ws->sm_count ? 1 : kSortWarps;
        launch_pdl(tile_sort_kernel, (unsigned)((tiles + per_block - 1) / per_block), 32 * kSortWarps, 0, st, a, per_block);
        note_launch();
    }
    kt_end(ws, GS_KT_BIN_SORT, st);
    return cudaGetLastError();
}

} // namespace gs
