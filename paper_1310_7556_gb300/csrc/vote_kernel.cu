// Stage-1 vote (Sec. 4, first step; the A[B[i]] += 1 scatter of Sec. 8), accumulator flush and
// the peak search over row bands (Sec. 4, second step).
//
// Two ways to fill the accumulator, the second in two forms:
//
// 1. Gather (layers whose hits share one radius; every configured workload).  On row i every
//    hit of such a layer votes at J - I_i - (f < g_i): its own bin coordinate J + f shifted by the
//    table's Nphi asin(x_i) / (2 pi) = I_i + g_i.  So layer l's bit of cell (i, j) is set exactly
//    when bucket J' = (j + I_i) mod Nphi holds a hit with f >= g_i, or bucket J' + 1 holds one with
//    f < g_i -- a test of the buckets' largest and smallest f, which the staging recorded.  The
//    gather kernel evaluates that test for every (cell, layer) of a tile: no atomics, each
//    accumulator word written once with a coalesced 16-byte store.  Same FP32 comparisons as the
//    per-vote form, so the same accumulator bit for bit.
//
// 2. Scatter (the paper's remedy, Sec. 6.1: shared-memory atomics instead of global ones).  One CTA
//    per (event, tile of tile_qpt rows x tile_phi columns) in shared memory.  The CTA reads only the
//    hits that can vote into its tile -- per layer one or two contiguous ranges of the
//    (layer, phi bin)-sorted hits -- lane by lane, and loops over the tile's rows in lockstep, so a
//    warp's 32 same-layer, azimuth-sorted hits update neighbouring words of one row; a lane whose
//    (word, bit) equals its left neighbour's skips its atomicOr.  With the count accumulator the
//    tile holds a 32-bit counter per cell instead: each run of lanes voting into the same cell
//    adds its length with one atomicAdd from its first lane, and the flush saturates every counter
//    to 16 bits -- the literal A[B[i]] += 1 of Sec. 8.  Table layers vote at
//    J - I - (f < g); other layers take FP32 asinf per vote, and a vote within `refine_eps` of an
//    edge (or with |x| > kRefineXLim) is recomputed in FP64 in the definition's order.  It handles
//    every layer and stores its tile: the vote in scatter mode and of counts in either mode.  After
//    the gather of layer masks general_kernel adds the layers whose radii differ.
//
// Peaks: candidates of each band of band_rows rows (one row by default) go to a band list in
// raster order; a scan of the band counts and a copy then concatenate the band lists of all events
// into one list.
// With a d0 axis a band lies in one slice and its cells take the 3 x 3 x 3 rule (peaks_mask_kernel<true>, peaks3_count_kernel).
#include <algorithm>
#include <atomic>
#include <climits>
#include <type_traits>

#include "hough_internal.cuh"

namespace hough {

namespace {

struct VoteParams {
    Axes ax;
    Workspace w;
    int R, W, n_spans, tiles_per_event;
    float s32;          // Nphi / (2 pi) in FP32
    float refine_eps;
};

constexpr int kMaxRanges = 2 * HOUGH_MAX_LAYERS;
constexpr int kRefineQueue = 64;   // a warp's queue of votes decided in FP64 (see scatter_kernel)
constexpr int kCompactThreads = 1024;

// Layers of the batch: bit l of *uniform_out is set when layer l takes the table path; bit l of
// *general_out when it has hits at more than one radius.  Called by warp 0.
__device__ __forceinline__ void layer_masks(const Workspace &w, int L, unsigned *uniform_out, unsigned *general_out)
{
    const int l = threadIdx.x;
    LayerInfo li;
    li.present = 0;
    li.uniform = 1;
    if (l < L) li = w.info[l];
    *uniform_out = __ballot_sync(0xFFFFFFFFu, l < L && li.uniform);
    *general_out = __ballot_sync(0xFFFFFFFFu, l < L && li.present && !li.uniform);
}

// Shared tile of the scatter kernel, column-major: cell (row rr, column jt) of a tile of R rows
// lives in word jt * pitch + rr (CELL 1: a layer mask a word; CELL 2: a 32-bit counter a word) or,
// when that tile does not fit in shared memory, word (jt >> 1) * pitch + rr (CELL 0: two 16-bit layer
// masks a word).  The lanes of a warp vote for 32 consecutive rows, so their 32 atomics fall in 32
// different banks whatever columns the votes land in.
__host__ __device__ inline int tile_row_pitch(int R) { return R <= 32 ? R : (R + 31) & ~31; }
// Margin columns on each side of the tile: a table layer's vote j - J0 lies within its window's
// spread of I beyond the tile's columns, so when that spread fits the margin every vote of the
// layer is cast where it falls -- into the tile or into a margin, which the flush ignores --
// without a test, a clamp or a select (even, so two-mask words keep their pairing).
constexpr int kTileMargin = 64;
__host__ __device__ inline int scatter_tile_words(int R, int W, bool wide)
{
    return (wide ? W + 2 * kTileMargin : (W + 2 * kTileMargin) >> 1) * tile_row_pitch(R);
}
// Byte offset of the per-warp hit buffers in the scatter kernel's dynamic shared memory.
__host__ __device__ inline size_t scatter_hit_offset(int R, int W, int L, bool wide)
{
    return ((size_t)scatter_tile_words(R, W, wide) * 4 + (size_t)L * R * sizeof(TabEntry) + (size_t)R * 4 + 15) &
           ~(size_t)15;
}

// One shared atomic update of cell (rr, jt) of the tile: the layer bit (masks) or one vote (counts).
template <int CELL>
__device__ __forceinline__ void tile_vote(uint32_t *tile, int pitch, int rr, int jt, uint32_t lbit)
{
    if (CELL == 2) atomicAdd(&tile[jt * pitch + rr], 1u);
    else if (CELL == 1) atomicOr(&tile[jt * pitch + rr], lbit);
    else atomicOr(&tile[(jt >> 1) * pitch + rr], lbit << ((jt & 1) << 4));
}

// A vote cast where it falls, at column jt of the lane's row (base: the row's word of column 0 as a
// shared-memory address, s4: the column stride in bytes, 0 for a lane whose votes all go to a
// word of its own).  jt may lie in a margin.
template <int CELL>
__device__ __forceinline__ void tile_vote_at(unsigned base, int s4, int jt, uint32_t lbit)
{
    if (CELL == 2) asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(base + jt * s4) : "memory");
    else if (CELL == 1) asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(base + jt * s4), "r"(lbit) : "memory");
    else asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(base + (jt >> 1) * s4), "r"(lbit << ((jt & 1) << 4)) : "memory");
}

// The votes of hits k0..k1-1 of the warp's buffer (f, byte offset of the column) for one row and
// one layer of one mask a word: the vote of hit k goes to rowbase + offset_k - (f_k < g) s4b.  PRED:
// some lane's row casts nothing (valid false), its atomics predicated off.
template <int CELL, bool PRED>
__device__ __forceinline__ void vote_run(const uint2 *hb2, int k0, int k1, float g, unsigned rowbase, unsigned s4b,
                                         uint32_t lbit, bool valid)
{
    const unsigned vflag = valid ? 1u : 0u;
    auto one = [&](uint2 h) {
        const unsigned a = rowbase + h.y - (__uint_as_float(h.x) < g ? s4b : 0u);
        if (PRED) {
            if (CELL == 2)
                asm volatile("{ .reg .pred p; setp.ne.u32 p, %1, 0; @p red.shared.add.u32 [%0], 1; }" ::"r"(a), "r"(vflag)
                             : "memory");
            else
                asm volatile("{ .reg .pred p; setp.ne.u32 p, %2, 0; @p red.shared.or.b32 [%0], %1; }" ::"r"(a), "r"(lbit),
                             "r"(vflag) : "memory");
        } else {
            if (CELL == 2) asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(a) : "memory");
            else asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(a), "r"(lbit) : "memory");
        }
    };
    int k = k0;
    for (; k + 8 <= k1; k += 8) {
        uint2 h[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) h[u] = hb2[2 * (k + u)];
#pragma unroll
        for (int u = 0; u < 8; ++u) one(h[u]);
    }
    for (; k < k1; ++k) one(hb2[2 * k]);
}

// The same for a vote that may miss the tile (in false): every lane issues its atomic, a missing
// vote adding nothing to a cell of its own row, so that no branch surrounds the atomic.  rowp,
// stride: the lane's row of the tile and the column stride (pitch), or for a lane without a row of
// the tile a word of its own with stride 0.
template <int CELL>
__device__ __forceinline__ void tile_vote_if(uint32_t *rowp, int stride, int jt, int W, bool in, uint32_t lbit)
{
    const int jc = (int)min((unsigned)jt, (unsigned)(W - 1));   // a column of the tile
    if (CELL == 2) atomicAdd(&rowp[jc * stride], in ? 1u : 0u);
    else if (CELL == 1) atomicOr(&rowp[jc * stride], in ? lbit : 0u);
    else atomicOr(&rowp[(jc >> 1) * stride], in ? lbit << ((jc & 1) << 4) : 0u);
}

template <int TPB, int CELL>
__global__ void __launch_bounds__(TPB) scatter_kernel(VoteParams p)
{
    constexpr bool COUNTS = CELL == 2;
    pdl_enter();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_start[kMaxRanges], s_off[kMaxRanges];
    __shared__ int s_pre[kMaxRanges + 1];
    __shared__ unsigned long long s_refined;
    __shared__ unsigned s_umask;
    __shared__ unsigned s_fast;   // table layers whose spread of I fits the tile's margins

    const Axes &ax = p.ax;
    const int R = p.R, W = p.W, L = ax.n_layers, nphi = ax.n_phi;
    const int pitch = tile_row_pitch(R);
    uint32_t *tile_all = reinterpret_cast<uint32_t *>(smem_raw);
    const int tile_words = scatter_tile_words(R, W, CELL != 0);
    uint32_t *tile = tile_all + (CELL != 0 ? kTileMargin : kTileMargin / 2) * pitch;   // column 0
    TabEntry *tab = reinterpret_cast<TabEntry *>(tile_all + tile_words);
    float *kq = reinterpret_cast<float *>(tab + L * R);
    // the warp's 32 staged hits: f (bits), J (shifted into the window for a table layer), c (bits), rows
    uint4 *hitbuf = reinterpret_cast<uint4 *>(smem_raw + scatter_hit_offset(R, W, L, CELL != 0)) + 32 * (threadIdx.x >> 5);
    // the warp's queue of votes to be decided in FP64: (staged position, row | layer << 16)
    uint2 *rq = reinterpret_cast<uint2 *>(smem_raw + scatter_hit_offset(R, W, L, CELL != 0) + (size_t)TPB * sizeof(uint4)) +
                kRefineQueue * (threadIdx.x >> 5);
    // 32 words that the atomics of lanes without a row of the tile go to (adding nothing)
    uint32_t *spare = reinterpret_cast<uint32_t *>(smem_raw + scatter_hit_offset(R, W, L, CELL != 0) +
                                                   (size_t)TPB * sizeof(uint4) + (size_t)(TPB / 32) * kRefineQueue * sizeof(uint2));

    const int e = blockIdx.x / p.tiles_per_event;
    const int t = blockIdx.x - e * p.tiles_per_event;
    const int slab = t / p.n_spans, span = t - slab * p.n_spans;
    const int i0 = slab * R;
    const int nrows = min(R, ax.n_qpt - i0);
    const int J0 = span * W;
    const int nkeys = L * nphi;
    const int64_t hstart = p.w.hit_start[e];
    const HotHit *hot = p.w.hot + hstart;
    const ColdHit *cold = p.w.cold + hstart;
    const int32_t *offs = p.w.offs + (int64_t)e * (nkeys + 1);

    if (threadIdx.x < 32) {
        unsigned u, g;
        layer_masks(p.w, L, &u, &g);
        if (threadIdx.x == 0) {
            s_umask = u;   // layers treated with the table
            s_refined = 0ull;
            s_fast = 0u;
        }
    }
    __syncthreads();
    const unsigned umask = s_umask;

    // clear the tile; stage this slab's table rows and FP32 q/pT centres
    uint4 *tile4 = reinterpret_cast<uint4 *>(tile_all);
    for (int q = threadIdx.x; q < tile_words >> 2; q += TPB) tile4[q] = make_uint4(0u, 0u, 0u, 0u);
    for (int q = threadIdx.x; q < L * R; q += TPB) {
        const int l = q / R, rr = q - l * R;
        TabEntry te;
        te.I = kNoVote;
        te.g = 0.f;
        if (rr < nrows && ((umask >> l) & 1u)) te = p.w.tab[l * ax.n_qpt + i0 + rr];
        tab[q] = te;
    }
    for (int q = threadIdx.x; q < R; q += TPB) kq[q] = q < nrows ? p.w.kq32[i0 + q] : 0.f;
    __syncthreads();

    // Per layer, the hits that can vote into this tile: a cyclic window [ja, jb] of phi bins J,
    // as one or two ranges of the sorted hits.  s_off[q] is the shift that takes the J of range q's
    // hits into the window's unwrapped coordinates (J + s_off in [ja, jb]).
    if (threadIdx.x < HOUGH_MAX_LAYERS) {
        const int l = threadIdx.x;
        int nr = 0, st[2] = {0, 0}, ln[2] = {0, 0}, of[2] = {0, 0};
        if (l < L) {
            const int lstart = offs[l * nphi], lend = offs[(l + 1) * nphi];
            int ja = 0, jb = -1;   // inclusive J window, possibly beyond [0, nphi)
            bool none = lend == lstart;
            if (!none && ((umask >> l) & 1u)) {
                // vote bin J - I - (f < g) lies in [J0, J0 + W) only for J in
                // [J0 + min I, J0 + W + max I] over the slab's voting rows
                int imin = INT_MAX, imax = INT_MIN;
                for (int rr = 0; rr < nrows; ++rr) {
                    const int I = tab[l * R + rr].I;
                    if (I != kNoVote) {
                        imin = min(imin, I);
                        imax = max(imax, I);
                    }
                }
                if (imin > imax) {
                    none = true;
                } else {
                    ja = J0 + imin;
                    jb = J0 + W + imax;
                    // votes of this window fall in [imin - imax - 1, W + imax - imin] of the tile
                    if (imax - imin + 1 <= kTileMargin) atomicOr(&s_fast, 1u << l);
                }
            } else if (!none && ax.n_d0) {
                ja = 0;   // per-vote layer on a grid with a d0 axis: every hit of the layer
                jb = nphi;
            } else if (!none) {
                // per-vote layer: bound asin(c k) over the layer's radius range and the slab's rows
                const float c_lo = 0.15f * (float)ax.b / 100.f * __uint_as_float(p.w.radii->rmin[l]);
                const float c_hi = 0.15f * (float)ax.b / 100.f * __uint_as_float(p.w.radii->rmax[l]);
                const float k_a = p.w.kq32[i0], k_b = p.w.kq32[i0 + nrows - 1];
                float amin = 2.f, amax = -2.f;
                const float cs[2] = {c_lo * 0.999f, c_hi * 1.001f};
                const float ks[2] = {k_a, k_b};
#pragma unroll
                for (int u = 0; u < 2; ++u)
#pragma unroll
                    for (int v = 0; v < 2; ++v) {
                        const float a = asinf(fminf(fmaxf(cs[u] * ks[v], -1.f), 1.f));
                        amin = fminf(amin, a);
                        amax = fmaxf(amax, a);
                    }
                ja = (int)floorf(J0 + p.s32 * amin) - 2;
                jb = (int)floorf(J0 + W + p.s32 * amax) + 2;
            }
            if (!none) {
                if (jb - ja + 1 >= nphi) {
                    nr = 1;
                    st[0] = lstart;
                    ln[0] = lend - lstart;
                } else {
                    const int a = ((ja % nphi) + nphi) % nphi;
                    const int b = ((jb % nphi) + nphi) % nphi;
                    of[0] = ja - a;
                    if (a <= b) {
                        nr = 1;
                        st[0] = offs[l * nphi + a];
                        ln[0] = offs[l * nphi + b + 1] - st[0];
                    } else {
                        nr = 2;
                        st[0] = offs[l * nphi + a];
                        ln[0] = lend - st[0];
                        st[1] = lstart;
                        ln[1] = offs[l * nphi + b + 1] - lstart;
                        of[1] = ja - a + nphi;
                    }
                }
            }
        }
        s_start[2 * l] = st[0];
        s_start[2 * l + 1] = st[1];
        s_off[2 * l] = of[0];
        s_off[2 * l + 1] = of[1];
        s_pre[2 * l] = nr >= 1 ? ln[0] : 0;       // lengths for now
        s_pre[2 * l + 1] = nr >= 2 ? ln[1] : 0;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int acc = 0;
        for (int q = 0; q < kMaxRanges; ++q) {
            const int len = s_pre[q];
            s_pre[q] = acc;
            acc += len;
        }
        s_pre[kMaxRanges] = acc;
    }
    __syncthreads();

    // A warp votes for 32 consecutive rows of the tile, a lane per row, taking the tile's hits 32
    // at a time: the 32 are staged in the warp's buffer and broadcast one by one to all lanes.  For
    // a table layer the lane's vote is j = J - I_row - (f < g_row): with the table entry in
    // registers, a compare, an add and the atomic.  When the tile is at most a quarter of the row,
    // the window of a layer's J is shorter than a row less the tile, so the vote lands in the tile
    // exactly when (J + s_off) - (I + J0) - (f < g) lies in [0, W), with no reduction modulo Nphi.
    const int total = s_pre[kMaxRanges];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int NW = TPB / 32;
    const int NG = (R + 31) >> 5;           // groups of 32 rows
    const int HS = max(1, NW / NG);         // warps sharing a row group's hits
    const bool wrap = W > (nphi >> 2);
    unsigned long long refined = 0;
    // Votes of the per-vote path within the refine window are not decided in the loop below: a
    // warp would run the FP64 arcsine for one lane.  They wait in the warp's queue, and every 32 of
    // them are decided together, a lane each (and cast: the atomics commute).
    int qn = 0;   // queued votes (the same in every lane)
    auto flush_refines = [&]() {
        __syncwarp();
        for (int t = lane; t < qn; t += 32) {
            const uint2 q = rq[t];
            const int row = (int)(q.y & 0xFFFFu);
            const ColdHit ch = cold[q.x];
            const double x64 = __dmul_rn(sagitta_coef(ax, (double)ch.r), qpt_centre(ax, i0 + row));
            const int jt = exact_bin(ax, (double)ch.phi, x64) - J0;
            if ((unsigned)jt < (unsigned)W) tile_vote<CELL>(tile, pitch, row, jt, 1u << (q.y >> 16));
        }
        __syncwarp();
        qn = 0;
    };
    for (int task = warp; task < NG * HS; task += NW) {
        const int rr = (task % NG) * 32 + lane;
        const int hs = task / NG;
        const bool rowok = rr < nrows;
        const int i = i0 + rr;
        const float kqr = rowok ? kq[rr] : 0.f;
        uint32_t *rowp = rowok ? tile + rr : spare + lane;
        const int stride = rowok ? pitch : 0;
        // hit v's staged position, window shift and record (empty past the last hit); the next
        // chunk's record is requested before this chunk votes, so its load overlaps the votes
        auto fetch_hit = [&](int v, int &pos, int &off, HotHit &hh) {
            hh.f = 0.f;
            hh.c = 0.f;
            hh.jl = 16u << 16;   // layer 16: none
            hh.rows = 1u;        // rows [1, 0]: none
            pos = 0;
            off = 0;
            if (v < total) {
                int q = 0;   // the range holding v: the last q with s_pre[q] <= v
#pragma unroll
                for (int step = 16; step > 0; step >>= 1)
                    if (s_pre[q + step] <= v) q += step;
                pos = s_start[q] + (v - s_pre[q]);
                off = s_off[q];
                hh = hot[pos];
            }
        };
        int pos_n, off_n;
        HotHit hh_n;
        fetch_hit(hs * 32 + lane, pos_n, off_n, hh_n);
        for (int cb = hs * 32; cb < total; cb += HS * 32) {
            const int nvalid = min(32, total - cb);
            const int pos = pos_n, off = off_n;
            const HotHit hh = hh_n;
            if (cb + HS * 32 < total) fetch_hit(cb + HS * 32 + lane, pos_n, off_n, hh_n);
            const int l = (int)((hh.jl >> 16) & 0x1Fu);
            const int J = (int)(hh.jl & 0xFFFFu);
            const bool table_hit = l < 16 && ((umask >> l) & 1u);
            // a table layer whose votes fall within the margins, one mask a word: the byte offset
            // of its column in a row of the tile (the vote then subtracts the row's shift in bytes)
            const bool fast_hit = CELL != 0 && !wrap && table_hit && ((s_fast >> l) & 1u);
            hitbuf[lane] = make_uint4(__float_as_uint(hh.f),
                                      fast_hit ? (uint32_t)((J + off) * 4 * pitch)
                                               : (uint32_t)(wrap || !table_hit ? J : J + off),
                                      __float_as_uint(hh.c), hh.rows);
            __syncwarp();
            // runs of hits of one layer (the ranges are in layer order)
            const int lprev = __shfl_up_sync(0xFFFFFFFFu, l, 1);
            unsigned heads = __ballot_sync(0xFFFFFFFFu, lane < nvalid && (lane == 0 || l != lprev));
            while (heads) {
                const int k0 = __ffs(heads) - 1;
                heads &= heads - 1u;
                const int k1 = heads ? __ffs(heads) - 1 : nvalid;
                const int lr = __shfl_sync(0xFFFFFFFFu, l, k0);
                const uint32_t lbit = 1u << lr;
                if ((umask >> lr) & 1u) {
                    const TabEntry te = tab[lr * R + (rowok ? rr : 0)];
                    const bool valid = rowok && te.I != kNoVote;
                    const float g = te.g;
                    if (CELL != 0 && !wrap && ((s_fast >> lr) & 1u)) {
                        // every vote where it falls: the word of column (J + off) - K - (f < g) of the
                        // lane's row, its byte offset from the staged column offset; a lane of an
                        // invalid row (or none) casts nothing
                        const unsigned s4b = 4u * (unsigned)pitch;
                        const unsigned rowbase = smem_u32(tile + rr) - (unsigned)(te.I + J0) * s4b;
                        const uint2 *hb2 = reinterpret_cast<const uint2 *>(hitbuf);   // (f, column bytes) of hit k at 2 k
                        if (__all_sync(0xFFFFFFFFu, valid))
                            vote_run<CELL, false>(hb2, k0, k1, g, rowbase, s4b, lbit, true);
                        else
                            vote_run<CELL, true>(hb2, k0, k1, g, rowbase, s4b, lbit, valid);
                    } else if (!wrap && ((s_fast >> lr) & 1u)) {
                        // the same with two masks a word: the vote's column from its J
                        const unsigned base = valid ? smem_u32(tile + rr) : smem_u32(spare + lane);
                        const int s4 = valid ? 4 * pitch : 0;
                        const int K = te.I + J0;
                        int k = k0;
                        const uint2 *hb2 = reinterpret_cast<const uint2 *>(hitbuf);   // (f, J) of hit k at 2 k
                        for (; k + 8 <= k1; k += 8) {
                            uint2 h[8];
#pragma unroll
                            for (int u = 0; u < 8; ++u) h[u] = hb2[2 * (k + u)];
#pragma unroll
                            for (int u = 0; u < 8; ++u)
                                tile_vote_at<CELL>(base, s4, (int)h[u].y - K - (__uint_as_float(h[u].x) < g ? 1 : 0), lbit);
                        }
                        for (; k < k1; ++k) {
                            const uint2 h = hb2[2 * k];
                            tile_vote_at<CELL>(base, s4, (int)h.y - K - (__uint_as_float(h.x) < g ? 1 : 0), lbit);
                        }
                    } else if (!wrap) {
                        const int K = valid ? te.I + J0 : -(1 << 30);   // an invalid row's votes all miss
                        // four hits at a time: their loads issue together, then their atomics
                        int k = k0;
                        const uint2 *hb2 = reinterpret_cast<const uint2 *>(hitbuf);   // (f, J) of hit k at 2 k
                        for (; k + 4 <= k1; k += 4) {
                            uint2 h[4];
#pragma unroll
                            for (int u = 0; u < 4; ++u) h[u] = hb2[2 * (k + u)];
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                const int jt = (int)h[u].y - K - (__uint_as_float(h[u].x) < g ? 1 : 0);
                                tile_vote_if<CELL>(rowp, stride, jt, W, (unsigned)jt < (unsigned)W, lbit);
                            }
                        }
                        for (; k < k1; ++k) {
                            const uint2 h = hb2[2 * k];
                            const int jt = (int)h.y - K - (__uint_as_float(h.x) < g ? 1 : 0);
                            tile_vote_if<CELL>(rowp, stride, jt, W, (unsigned)jt < (unsigned)W, lbit);
                        }
                    } else {
                        for (int k = k0; k < k1; ++k) {
                            const uint4 h = hitbuf[k];
                            int j = (int)h.y - te.I - (__uint_as_float(h.x) < g ? 1 : 0);
                            j += j < 0 ? nphi : 0;
                            j -= j >= nphi ? nphi : 0;
                            const int jt = j - J0;
                            tile_vote_if<CELL>(rowp, stride, jt, W, valid && (unsigned)jt < (unsigned)W, lbit);
                        }
                    }
                    continue;
                }
                // a layer whose hits lie at several radii: every vote evaluated per hit
                for (int k = k0; k < k1; ++k) {
                    const uint4 h = hitbuf[k];
                    const float c = __uint_as_float(h.z), fk = __uint_as_float(h.x);
                    const uint32_t rows = h.w;
                    const int Jk = (int)h.y;
                    bool act = rowok && i >= (int)(rows & 0xFFFFu) && i <= (int)(rows >> 16);
                    int j = 0;
                    if (ax.n_d0) {
                        // a grid with a d0 axis: every vote of a per-vote layer in FP64, in the definition's order
                        const int pk = __shfl_sync(0xFFFFFFFFu, pos, k);
                        if (act) {
                            const ColdHit ch = cold[pk];
                            act = exact_vote(ax, (double)ch.r, (double)ch.phi, i, &j);
                        }
                    } else {
                        const float x = fminf(fmaxf(c * kqr, -1.f), 1.f);
                        const float vq = fmaf(-asinf(x), p.s32, fk);
                        const float fl = floorf(vq);
                        const float d = vq - fl;
                        j = Jk + (int)fl;
                        const bool need = act && (d < p.refine_eps || d > 1.f - p.refine_eps || fabsf(x) > kRefineXLim);
                        if (__any_sync(0xFFFFFFFFu, need)) {   // rare: queue them
                            const int pk = __shfl_sync(0xFFFFFFFFu, pos, k);
                            const unsigned rb = __ballot_sync(0xFFFFFFFFu, need);
                            if (need) rq[qn + __popc(rb & ((1u << lane) - 1u))] = make_uint2((uint32_t)pk, (uint32_t)rr | ((uint32_t)lr << 16));
                            qn += __popc(rb);
                            if (lane == 0) refined += __popc(rb);
                            act = act && !need;
                        }
                    }
                    j += j < 0 ? nphi : 0;
                    j -= j >= nphi ? nphi : 0;
                    const int jt = j - J0;
                    tile_vote_if<CELL>(rowp, stride, jt, W, act && (unsigned)jt < (unsigned)W, lbit);
                    if (qn >= 32) flush_refines();   // at most 63 queued
                }
            }
            __syncwarp();   // the buffer is read before the next chunk overwrites it
        }
    }
    if (qn) flush_refines();
    if (refined) atomicAdd(&s_refined, refined);
    __syncthreads();

    // flush the tile: 8 cells of a row per thread, consecutive threads on consecutive rows (one
    // bank each in the column-major tile), one 16-byte store
    uint16_t *M = p.w.M + (int64_t)e * ax.n_qpt * nphi;
    const int v8 = W >> 3;
    for (int q = threadIdx.x; q < nrows * v8; q += TPB) {
        const int c8 = q / nrows, rr = q - c8 * nrows;
        uint4 *dst = reinterpret_cast<uint4 *>(M + (int64_t)(i0 + rr) * nphi + J0 + c8 * 8);
        if (COUNTS) {
            uint32_t cnt[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) cnt[k] = tile[(c8 * 8 + k) * pitch + rr];
            auto pack = [](uint32_t lo, uint32_t hi) { return min(lo, 65535u) | (min(hi, 65535u) << 16); };
            *dst = make_uint4(pack(cnt[0], cnt[1]), pack(cnt[2], cnt[3]), pack(cnt[4], cnt[5]), pack(cnt[6], cnt[7]));
            continue;
        }
        uint4 v;
        if (CELL == 1) {   // a mask a word: pairs of cells into one word
            uint32_t m[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) m[k] = tile[(c8 * 8 + k) * pitch + rr];
            v = make_uint4(m[0] | (m[1] << 16), m[2] | (m[3] << 16), m[4] | (m[5] << 16), m[6] | (m[7] << 16));
        } else {
            v = make_uint4(tile[(c8 * 4) * pitch + rr], tile[(c8 * 4 + 1) * pitch + rr], tile[(c8 * 4 + 2) * pitch + rr],
                           tile[(c8 * 4 + 3) * pitch + rr]);
        }
        *dst = v;
    }
    if (threadIdx.x == 0 && s_refined) atomicAdd(&p.w.stats[e].refined_votes, s_refined);
}

// The vote of layers whose hits lie at several radii, after the gather of layer masks: ORed into the
// gathered accumulator.  A CTA takes tiles of kGenRows rows x kGenCols columns, a lane a row, the tile's hits 32
// at a time a warp, each broadcast to all lanes.  The detectors that need this have their modules near
// a common radius, so instead of an arcsine per vote the lane holds, for its row and the layer, the
// cubic of T(r) = Nphi asin(c(r) k) / (2 pi) around the layer's middle radius r0 (T(r0) in FP64, split
// into a whole number and a fraction): a vote is three multiply-adds and a floor.  A (layer, row) takes
// the cubic when its error over the layer's radii stays below kCubicErr bins (the fourth derivative of
// asin, (9 x + 6 x^3) / (1 - x^2)^(7/2), at the largest x, bounds the remainder) and T moves by at most
// kCubicSpan bins; r - r0 is exact, so with the roundings of f and of the sums a vote is known to
// kCubicEps bins, and only votes closer than that to a bin edge are redone in FP64, 32 of a warp's queue
// at a time.  Rows with |x| above kNearLimit on which the cubic will not do take the arcsine from its end,
// asin|x| = pi/2 - 2 asin(sqrt((1 - |x|) / 2)), with 1 - |x| and the square root in two-float arithmetic
// and the series of asin to the eleventh power: known to the same window (deciding the votes of |x| > 0.99
// in FP64 instead put 60,000 of them on the 16 tiles of the largest |q/pT|, 260 us).  What is left (radii
// far apart) evaluates asinf per vote with the wider window refine_eps.  Measured on the 100k-hit event
// with radii +-0.5 cm: 511 us with asinf per vote and a CTA of eight warps a tile.  With no such layer it returns at once: a grid of at most one CTA per
// SM strides over the tiles, so that an empty launch costs the same for one event and for a batch.
constexpr int kGenRows = 32, kGenCols = 256, kGenThreads = 1024;
constexpr double kCubicErr = 2e-5, kCubicSpan = 32.0;
constexpr float kCubicEps = 2e-4f, kNearLimit = 0.85f;

struct GeneralParams {
    Axes ax;
    Workspace w;
    int n_spans, tiles_per_event;
    float s32, refine_eps;
};

// Per (layer, row) of a tile: the negated cubic's fraction and coefficients, and I with the row's kind in
// its low two bits (0: the layer's hits cannot vote, 1: cubic, 2: asinf per vote, 3: the arcsine from its
// end, the row's |x| / r as two floats in the first two coefficients).
struct GeneralSmem {
    uint32_t tile[kGenCols * kGenRows];
    uint4 hits[kGenThreads];                           // per warp: f, r - r0, column of J in the tile, staged position
    uint2 queue[kGenThreads / 32 * kRefineQueue];      // per warp: staged position, row | layer << 16
    float4 co[HOUGH_MAX_LAYERS * kGenRows];
    int I[HOUGH_MAX_LAYERS * kGenRows];
    float kq[kGenRows];
};

__global__ void __launch_bounds__(kGenThreads) general_kernel(GeneralParams p)
{
    // Nothing the predecessor (the gather) writes is read until a tile is flushed: the layer records,
    // bucket offsets and sorted hits come from kernels that finished before the gather could launch.  So
    // the votes are cast first, and the wait comes before the first flush.
    extern __shared__ __align__(16) unsigned char general_smem[];
    GeneralSmem &S = *reinterpret_cast<GeneralSmem *>(general_smem);
    __shared__ int s_start[kMaxRanges], s_off[kMaxRanges], s_pre[kMaxRanges + 1];
    __shared__ unsigned s_wrap;
    __shared__ unsigned long long s_refined;
    const Axes &ax = p.ax;
    const int L = ax.n_layers, nphi = ax.n_phi, nkeys = L * nphi;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    LayerInfo li{};
    if (lane < L) li = p.w.info[lane];
    const unsigned gmask = __ballot_sync(0xFFFFFFFFu, lane < L && li.present && !li.uniform);
    if (!gmask) {
        pdl_enter();
        return;
    }
    bool waited = false;
    uint4 *hitbuf = S.hits + 32 * warp;
    uint2 *rq = S.queue + kRefineQueue * warp;
    const unsigned rowaddr = smem_u32(S.tile + lane);
    for (int tile = blockIdx.x; tile < p.w.n_events * p.tiles_per_event; tile += gridDim.x) {
        const int e = tile / p.tiles_per_event, t = tile - e * p.tiles_per_event;
        const int slab = t / p.n_spans, span = t - slab * p.n_spans;
        const int i0 = slab * kGenRows, nrows = min(kGenRows, ax.n_qpt - i0);
        const int J0 = span * kGenCols, W = min(kGenCols, nphi - J0);
        const int64_t hstart = p.w.hit_start[e];
        const HotHit *hot = p.w.hot + hstart;
        const ColdHit *cold = p.w.cold + hstart;
        const int32_t *offs = p.w.offs + (int64_t)e * (nkeys + 1);
        if (threadIdx.x == 0) {
            s_wrap = 0u;
            s_refined = 0ull;
        }
        __syncthreads();
        for (int q = threadIdx.x; q < kGenCols * kGenRows / 4; q += kGenThreads)
            reinterpret_cast<uint4 *>(S.tile)[q] = make_uint4(0u, 0u, 0u, 0u);
        if (threadIdx.x < kGenRows) S.kq[threadIdx.x] = threadIdx.x < nrows ? p.w.kq32[i0 + threadIdx.x] : 0.f;
        for (int q = threadIdx.x; q < L * kGenRows; q += kGenThreads) {
            const int l = q / kGenRows, rr = q - l * kGenRows;
            float4 co = make_float4(0.f, 0.f, 0.f, 0.f);
            int kind = 0, I = 0;
            if (((gmask >> l) & 1u) && rr < nrows) {
                kind = 2;
                const float rmin = __uint_as_float(p.w.radii->rmin[l]), rmax = __uint_as_float(p.w.radii->rmax[l]);
                const float r0 = 0.5f * (rmin + rmax);
                if (!ax.n_d0) {
                    const double k = qpt_centre(ax, i0 + rr), ck = sagitta_coef(ax, 1.0) * k;   // x = ck r
                    const double xm = fabs(ck) * (double)rmax;
                    if (fabs(ck) * (double)rmin > 1.0 + 1e-9) {
                        kind = 0;
                    } else if (xm <= 0.97 && rmin >= 0.5f * r0 && rmax <= 2.f * r0) {
                        const double s = (double)ax.n_phi * kInvTwoPi, x = ck * (double)r0;
                        const double y = 1.0 - x * x, rs = rsqrt(y), dx = ck * 0.5 * (double)(rmax - rmin) * 1.0001;
                        const float ym = (float)(1.0 - xm * xm), xf = (float)xm;
                        const float d4 = (9.f * xf + 6.f * xf * xf * xf) * rsqrtf(ym) / (ym * ym * ym);
                        const float dx2 = (float)(dx * dx);
                        const double d1 = s * ck * rs;
                        if ((float)s * dx2 * dx2 * d4 * (1.01f / 24.f) <= (float)kCubicErr &&
                            s * fabs(dx) * rsqrtf(ym) <= kCubicSpan) {
                            const double T = s * asin(x), fI = floor(T);
                            kind = 1;
                            I = (int)fI;
                            co.x = -(float)(T - fI);
                            co.y = -(float)d1;
                            co.z = -(float)(0.5 * s * ck * ck * x * rs * rs * rs);
                            co.w = -(float)(s * ck * ck * ck * (1.0 + 2.0 * x * x) * rs * rs * rs * rs * rs * (1.0 / 6.0));
                        }
                    }
                    if (kind == 2 && fabs(ck) * (double)rmin >= (double)kNearLimit) {
                        kind = 3;
                        I = k < 0.0 ? -1 : 1;
                        co.x = (float)fabs(ck);
                        co.y = (float)(fabs(ck) - (double)co.x);
                    }
                }
            }
            S.co[q] = co;
            S.I[q] = I * 4 + kind;
        }
        // per layer, the hits that can vote into this tile: a cyclic window [ja, jb] of phi bins J, as one
        // or two ranges of the sorted hits; s_off[q] takes the J of range q's hits to columns of the tile
        if (threadIdx.x < HOUGH_MAX_LAYERS) {
            const int l = threadIdx.x;
            int nr = 0, st[2] = {0, 0}, ln[2] = {0, 0}, of[2] = {0, 0};
            if ((gmask >> l) & 1u) {
                const int lstart = offs[l * nphi], lend = offs[(l + 1) * nphi];
                int ja = 0, jb = nphi;   // a grid with a d0 axis: every hit of the layer
                if (!ax.n_d0) {
                    // bound asin(c k) over the layer's radius range and the slab's rows
                    const float c_lo = 0.15f * (float)ax.b / 100.f * __uint_as_float(p.w.radii->rmin[l]) * 0.999f;
                    const float c_hi = 0.15f * (float)ax.b / 100.f * __uint_as_float(p.w.radii->rmax[l]) * 1.001f;
                    const float k_a = p.w.kq32[i0], k_b = p.w.kq32[i0 + nrows - 1];
                    const float xs[4] = {c_lo * k_a, c_lo * k_b, c_hi * k_a, c_hi * k_b};
                    float amin = 2.f, amax = -2.f;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const float a = asinf(fminf(fmaxf(xs[u], -1.f), 1.f));
                        amin = fminf(amin, a);
                        amax = fmaxf(amax, a);
                    }
                    ja = (int)floorf(J0 + p.s32 * amin) - 2;
                    jb = (int)floorf(J0 + W + p.s32 * amax) + 2;
                }
                if (lend > lstart && jb - ja + 1 >= nphi) {
                    nr = 1;
                    st[0] = lstart;
                    ln[0] = lend - lstart;
                    of[0] = -J0;
                    atomicOr(&s_wrap, 1u << l);
                } else if (lend > lstart) {
                    const int a = ((ja % nphi) + nphi) % nphi, b = ((jb % nphi) + nphi) % nphi;
                    of[0] = ja - a - J0;
                    st[0] = offs[l * nphi + a];
                    if (a <= b) {
                        nr = 1;
                        ln[0] = offs[l * nphi + b + 1] - st[0];
                    } else {
                        nr = 2;
                        ln[0] = lend - st[0];
                        st[1] = lstart;
                        ln[1] = offs[l * nphi + b + 1] - lstart;
                        of[1] = ja - a + nphi - J0;
                    }
                }
            }
            s_start[2 * l] = st[0];
            s_start[2 * l + 1] = st[1];
            s_off[2 * l] = of[0];
            s_off[2 * l + 1] = of[1];
            s_pre[2 * l] = nr >= 1 ? ln[0] : 0;   // lengths for now
            s_pre[2 * l + 1] = nr >= 2 ? ln[1] : 0;
        }
        __syncthreads();
        if (warp == 0) {   // (kMaxRanges is a warp's lanes)
            const int len = s_pre[lane];
            int incl = len;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int v = __shfl_up_sync(0xFFFFFFFFu, incl, d);
                if (lane >= d) incl += v;
            }
            s_pre[lane] = incl - len;
            if (lane == 31) s_pre[kMaxRanges] = incl;
        }
        __syncthreads();
        const int total = s_pre[kMaxRanges];
        const unsigned wrapm = s_wrap;
        const bool rowok = lane < nrows;
        const int i = i0 + lane;
        const float kqr = S.kq[lane];
        unsigned refined = 0;
        int qn = 0;   // the warp's queued votes (the same in every lane)
        auto cast = [&](int jt, unsigned lbit) {
            asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(rowaddr + (unsigned)jt * (4u * kGenRows)), "r"(lbit) : "memory");
        };
        auto flush_queue = [&]() {
            __syncwarp();
            for (int u = lane; u < qn; u += 32) {
                const uint2 q = rq[u];
                const int row = (int)(q.y & 0xFFFFu);
                const ColdHit ch = cold[q.x];
                const double x64 = __dmul_rn(sagitta_coef(ax, (double)ch.r), qpt_centre(ax, i0 + row));
                const int jt = exact_bin(ax, (double)ch.phi, x64) - J0;
                if ((unsigned)jt < (unsigned)W) atomicOr(&S.tile[jt * kGenRows + row], 1u << (q.y >> 16));
            }
            __syncwarp();
            qn = 0;
        };
        // a vote too close to a bin edge waits in the queue
        auto enqueue = [&](bool need, unsigned pos, int l) {
            const unsigned rb = __ballot_sync(0xFFFFFFFFu, need);
            if (need) rq[qn + __popc(rb & ((1u << lane) - 1u))] = make_uint2(pos, (uint32_t)lane | ((uint32_t)l << 16));
            qn += __popc(rb);
            refined += (unsigned)__popc(rb);
            if (qn >= 32) flush_queue();   // at most 63 queued
        };
        for (int cb = warp * 32; cb < total; cb += kGenThreads) {
            const int nvalid = min(32, total - cb);
            int l = HOUGH_MAX_LAYERS, pos = 0;
            HotHit hh{0.f, 0.f, 0u, 1u};
            if (lane < nvalid) {
                const int v = cb + lane;
                int q = 0;   // the range holding v: the last q with s_pre[q] <= v
#pragma unroll
                for (int step = 16; step > 0; step >>= 1)
                    if (s_pre[q + step] <= v) q += step;
                pos = s_start[q] + (v - s_pre[q]);
                hh = hot[pos];
                const float r = cold[pos].r;
                l = (int)((hh.jl >> 16) & 0xFu);
                const float r0 = 0.5f * (__uint_as_float(p.w.radii->rmin[l]) + __uint_as_float(p.w.radii->rmax[l]));
                hitbuf[lane] = make_uint4(__float_as_uint(hh.f), __float_as_uint(r - r0),
                                          (uint32_t)((int)(hh.jl & 0xFFFFu) + s_off[q]), (uint32_t)pos);
            }
            __syncwarp();
            // runs of hits of one layer (the ranges are in layer order)
            const int lprev = __shfl_up_sync(0xFFFFFFFFu, l, 1);
            unsigned heads = __ballot_sync(0xFFFFFFFFu, lane < nvalid && (lane == 0 || l != lprev));
            while (heads) {
                const int k0 = __ffs(heads) - 1;
                heads &= heads - 1u;
                const int k1 = heads ? __ffs(heads) - 1 : nvalid;
                const int lr = __shfl_sync(0xFFFFFFFFu, l, k0);
                const unsigned lbit = 1u << lr;
                const bool wrap = (wrapm >> lr) & 1u;
                const float4 co = S.co[lr * kGenRows + lane];
                const int Ik = S.I[lr * kGenRows + lane];
                const int kind = rowok ? Ik & 3 : 0, I = Ik >> 2;
                if (__any_sync(0xFFFFFFFFu, kind == 1)) {
                    // a lane of another kind has its votes fall far outside the tile
                    const int shift = (kind == 1 ? -I : -(1 << 28)) - 0x4B400000;
                    const float half_less = 0.5f - kCubicEps;
                    // four hits at a time without a branch: a vote outside the tile or too close to an edge is
                    // predicated off, and the four are looked at again when one of them was close
                    auto four = [&](auto wrap_type, const int k, const int n) {
                        constexpr bool wraps = decltype(wrap_type)::value;
                        uint4 h[4];
                        float dist[4];
                        int jt[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) h[u] = hitbuf[k + min(u, n - 1)];
                        float far = 0.f;
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const float x = __uint_as_float(h[u].y);
                            const float v = fmaf(x, fmaf(x, fmaf(x, co.w, co.z), co.y), __uint_as_float(h[u].x)) + co.x;
                            const float fl = __fadd_rd(v, 12582912.f);   // 1.5 * 2^23: the sum's low bits are floor(v)
                            dist[u] = fabsf((v - (fl - 12582912.f)) - 0.5f);
                            far = fmaxf(far, dist[u]);
                            jt[u] = (int)h[u].z + __float_as_int(fl) + shift;
                            if (wraps) {   // every hit of the layer: the column modulo Nphi
                                jt[u] += jt[u] + J0 < 0 ? nphi : 0;
                                jt[u] -= jt[u] + J0 >= nphi ? nphi : 0;
                            }
                            if (u >= n) jt[u] = -1;   // (n: the same for the whole warp)
                            const unsigned addr = rowaddr + (unsigned)jt[u] * (4u * kGenRows);
                            asm volatile("{\n\t.reg .pred p, q;\n\tsetp.gt.f32 q, %1, %2;\n\t"
                                         "setp.lt.and.u32 p, %3, %4, !q;\n\t@p red.shared.or.b32 [%0], %5;\n\t}"
                                         ::"r"(addr), "f"(dist[u]), "f"(half_less), "r"(jt[u]), "r"(W), "r"(lbit) : "memory");
                        }
                        if (!__any_sync(0xFFFFFFFFu, far > half_less)) return;
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            enqueue(u < n && kind == 1 && dist[u] > half_less &&
                                        (wraps || (unsigned)(jt[u] + 1) <= (unsigned)(W + 1)), h[u].w, lr);
                    };
                    if (wrap) {
                        for (int k = k0; k < k1; k += 4) four(std::true_type{}, k, min(4, k1 - k));
                    } else {
                        int k = k0;
                        for (; k + 4 <= k1; k += 4) four(std::false_type{}, k, 4);
                        if (k < k1) four(std::false_type{}, k, k1 - k);
                    }
                }
                if (__any_sync(0xFFFFFFFFu, kind == 3)) {
                    const float r0 = 0.5f * (__uint_as_float(p.w.radii->rmin[lr]) + __uint_as_float(p.w.radii->rmax[lr]));
                    const float s2h = 2.f * ax.u_hi, s2l = 2.f * ax.u_lo, sg = (float)I;
                    for (int k = k0; k < k1; ++k) {
                        const uint4 h = hitbuf[k];
                        const uint32_t rows = __shfl_sync(0xFFFFFFFFu, hh.rows, k);
                        const bool act = kind == 3 && i >= (int)(rows & 0xFFFFu) && i <= (int)(rows >> 16);
                        const float r = r0 + __uint_as_float(h.y);   // exact: the difference was
                        // |x| = xp.x + xp.y, then w = (1 - |x|) / 2 = wv.x + wv.y
                        float2 xp = two_prod(r, co.x);
                        xp.y = fmaf(r, co.y, xp.y);
                        float2 wv = two_sum(1.f - xp.x, -xp.y);
                        wv.x = fmaxf(0.5f * wv.x, 1e-30f);
                        wv.y *= 0.5f;
                        const float rs = rsqrtf(wv.x), tt = wv.x * rs;   // tt + tl = sqrt(w)
                        const float tl = 0.5f * rs * (fmaf(-tt, tt, wv.x) + wv.y);
                        float z = fmaf(wv.x, 945.f / 42240.f, 105.f / 3456.f);
                        z = fmaf(wv.x, z, 15.f / 336.f);
                        z = fmaf(wv.x, z, 3.f / 40.f);
                        z = fmaf(wv.x, z, 1.f / 6.f);
                        const float small = fmaf(tt * wv.x, z, tl);      // asin(sqrt(w)) = tt + small
                        // Q = Nphi / (2 pi) 2 asin(sqrt(w)); T = +-(Nphi / 4 - Q)
                        float2 Q = two_prod(tt, s2h);
                        Q.y += fmaf(tt, s2l, small * s2h);
                        const float fq = floorf(Q.x);
                        const float v = fmaf(sg, (Q.x - fq) + Q.y, __uint_as_float(h.x));
                        const float fl = floorf(v);
                        const float d = v - fl;
                        int jt = (int)h.z + I * ((int)fq - (nphi >> 2)) + (int)fl;
                        if (wrap) {
                            jt += jt + J0 < 0 ? nphi : 0;
                            jt -= jt + J0 >= nphi ? nphi : 0;
                        }
                        const bool near = act && fabsf(d - 0.5f) > 0.5f - kCubicEps &&
                                          (wrap || (unsigned)(jt + 1) <= (unsigned)(W + 1));
                        if (act && !near && (unsigned)jt < (unsigned)W) cast(jt, lbit);
                        if (__any_sync(0xFFFFFFFFu, near)) enqueue(near, h.w, lr);
                    }
                }
                if (!__any_sync(0xFFFFFFFFu, kind == 2)) continue;
                for (int k = k0; k < k1; ++k) {
                    const uint4 h = hitbuf[k];
                    const float c = __shfl_sync(0xFFFFFFFFu, hh.c, k);
                    const uint32_t rows = __shfl_sync(0xFFFFFFFFu, hh.rows, k);
                    bool act = kind == 2 && i >= (int)(rows & 0xFFFFu) && i <= (int)(rows >> 16);
                    int jt = 0;
                    if (ax.n_d0) {
                        // a grid with a d0 axis: every vote in FP64, in the definition's order
                        if (act) {
                            const ColdHit ch = cold[h.w];
                            int j;
                            act = exact_vote(ax, (double)ch.r, (double)ch.phi, i, &j);
                            jt = j - J0;
                        }
                    } else {
                        const float x = fminf(fmaxf(c * kqr, -1.f), 1.f);
                        const float vq = fmaf(-asinf(x), p.s32, __uint_as_float(h.x));
                        const float fl = floorf(vq);
                        const float d = vq - fl;
                        jt = (int)h.z + (int)fl;
                        if (wrap) {
                            jt += jt + J0 < 0 ? nphi : 0;
                            jt -= jt + J0 >= nphi ? nphi : 0;
                        }
                        const bool need = act && (d < p.refine_eps || d > 1.f - p.refine_eps || fabsf(x) > kRefineXLim);
                        if (__any_sync(0xFFFFFFFFu, need)) enqueue(need, h.w, lr);
                        act = act && !need;
                    }
                    if (act && (unsigned)jt < (unsigned)W) cast(jt, lbit);
                }
            }
            __syncwarp();   // the buffer is read before the next chunk overwrites it
        }
        if (qn) flush_queue();
        if (lane == 0 && refined) atomicAdd(&s_refined, (unsigned long long)refined);
        if (!waited) pdl_enter();   // the gathered accumulator is complete
        waited = true;
        __syncthreads();
        // flush the tile: 8 cells of a row per thread, consecutive threads on consecutive rows
        uint16_t *M = p.w.M + (int64_t)e * ax.n_qpt * nphi;
        if (total)
            for (int q = threadIdx.x; q < (W >> 3) * kGenRows; q += kGenThreads) {
                const int c8 = q / kGenRows, rr = q - c8 * kGenRows;
                if (rr >= nrows) continue;
                uint32_t m[8], any = 0u;
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    m[k] = S.tile[(c8 * 8 + k) * kGenRows + rr];
                    any |= m[k];
                }
                if (!any) continue;
                uint4 *dst = reinterpret_cast<uint4 *>(M + (int64_t)(i0 + rr) * nphi + J0 + c8 * 8);
                const uint4 old = *dst;
                const uint32_t ow[4] = {old.x, old.y, old.z, old.w};
                uint32_t v[4];
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    v[k] = ow[k] | m[2 * k] | m[2 * k + 1] << 16;
                *dst = make_uint4(v[0], v[1], v[2], v[3]);
            }
        if (threadIdx.x == 0 && s_refined) atomicAdd(&p.w.stats[e].refined_votes, s_refined);
        __syncthreads();   // the tile and the windows are free
    }
    if (!waited) pdl_enter();
}

// Gather: one tile of `rows` rows x `cols` columns of the accumulator from the per-bucket f
// extrema and the table.  On row i a layer's cells read the bucket entries shifted by I_i, which
// grows with i, so the tile reads one contiguous window of each layer's entries:
// [c0 + min_i I_i, c0 + cols + 2 + max_i I_i).  Thread 0 copies every layer's window into shared
// memory with bulk asynchronous copies (one or two pieces, the second when the window wraps
// around phi) completing on one mbarrier, while the other threads wait; a layer whose window does
// not fit its slot reads global memory instead.  A warp then takes a strip of up to 256 cells of a
// row, 8 per lane at a stride of 32; the staging put bucket J+1's smallest fraction beside bucket
// J's largest, so a layer's bit of cell j reads the one 8-byte entry j + I: conflict-free shared
// loads, one per (cell, voting layer), the layer's shift and threshold read once per 8 cells.
struct GatherParams {
    Axes ax;
    Workspace w;
    int rows, cols, col_tiles, tiles_per_event;
    int cap;   // entries of a layer's staging slot (even)
};

constexpr int kGatherRowsMax = 32;
constexpr long long kCopyWaitCycles = 2000000000LL;   // about a second: bulk copies take microseconds

// The first bound on the wait for a CTA's bulk copies: about a second, or none at all when a test of
// the error path asked for it (Workspace::copy_wait < 0).  On expiry the CTA reports
// HOUGH_DEVERR_TIMEOUT and waits once more, with the full bound, for its copies to land, so that it
// leaves no copy writing into shared memory after it has exited (unless that wait expires too).
__device__ __forceinline__ bool first_copy_wait(const Workspace &w, uint64_t *bar)
{
    if (w.copy_wait < 0) return false;
    return mbar_wait_bounded(bar, 0, kCopyWaitCycles);
}

template <int NL, int TPB>
__global__ void __launch_bounds__(TPB, 1) gather_kernel(GatherParams p)
{
    pdl_enter();
    extern __shared__ __align__(16) unsigned char gather_smem[];
    __shared__ int rowI[kGatherRowsMax * 16];
    __shared__ unsigned rowG[kGatherRowsMax * 16];
    __shared__ unsigned rowMask[kGatherRowsMax];
    __shared__ int s_wbase[16], s_wlen[16];
    __shared__ unsigned s_staged;
    __shared__ __align__(8) uint64_t s_bar;
    const Axes &ax = p.ax;
    const Workspace &w = p.w;
    const int e = blockIdx.x / p.tiles_per_event;
    const int t = blockIdx.x - e * p.tiles_per_event;
    const int rt = t / p.col_tiles, ct = t - rt * p.col_tiles;
    const int i0 = rt * p.rows, c0 = ct * p.cols;
    const int nrows = min(p.rows, ax.n_qpt - i0);
    const int L = ax.n_layers, nphi = ax.n_phi;

    // per (row, layer): the table entry and whether the layer votes on that row by the gather
    // (whole warps, so that the ballot sees full warps; TPB is a multiple of 32)
    for (int q = threadIdx.x; q < ((p.rows * 16 + 31) & ~31); q += TPB) {
        const int rr = q >> 4, l = q & 15, i = i0 + rr;
        int I = 0;
        unsigned gb = 0u, valid = 0u;
        if (l < L && rr < nrows) {
            const LayerInfo li = w.info[l];
            const TabEntry te = w.tab[l * ax.n_qpt + i];   // requested with the layer record: one round trip
            if (li.present && li.uniform && i >= li.lo && i <= li.hi) {
                if (te.I != kNoVote) {
                    I = te.I;
                    gb = __float_as_uint(te.g);
                    valid = 1u;
                }
            }
        }
        const unsigned m = __ballot_sync(0xFFFFFFFFu, valid) >> (threadIdx.x & 16);
        rowI[q] = I;
        rowG[q] = gb;
        if ((threadIdx.x & 15) == 0) rowMask[rr] = m & 0xFFFFu;
    }
    __syncthreads();
    // each layer's window of bucket entries (unwrapped indices, start even)
    if (threadIdx.x < 32) {
        const int l = threadIdx.x;
        bool staged = false;
        if (l < L) {
            int lo = INT_MAX, hi = INT_MIN;
            for (int rr = 0; rr < nrows; ++rr)
                if ((rowMask[rr] >> l) & 1u) {
                    lo = min(lo, rowI[rr * 16 + l]);
                    hi = max(hi, rowI[rr * 16 + l]);
                }
            if (lo <= hi) {
                const int ws = (c0 + lo) - ((c0 + lo) & 1);
                int len = c0 + p.cols + 2 + hi - ws;
                len += len & 1;
                staged = len <= p.cap && len <= nphi;
                s_wbase[l] = ws;
                s_wlen[l] = len;
            }
        }
        const unsigned sm = __ballot_sync(0xFFFFFFFFu, staged);
        if (l == 0) {
            s_staged = sm;
            if (sm) mbar_init(&s_bar, 1);
        }
    }
    __syncthreads();
    const unsigned staged = s_staged;
    const uint2 *prof = w.prof + (int64_t)e * prof_event_entries(ax);
    const int pstride = prof_stride(ax);
    uint2 *win = reinterpret_cast<uint2 *>(gather_smem);
    if (staged) {
        if (threadIdx.x == 0) {
            unsigned bytes = 0;
            for (int l = 0; l < L; ++l)
                if ((staged >> l) & 1u) bytes += 8u * (unsigned)s_wlen[l];
            mbar_arrive_expect(&s_bar, bytes);
            for (int l = 0; l < L; ++l) {
                if (!((staged >> l) & 1u)) continue;
                const int len = s_wlen[l];
                const int a = ((s_wbase[l] % nphi) + nphi) % nphi;   // even, as nphi is
                const uint2 *src = prof + (int64_t)l * pstride;
                uint2 *dst = win + (int64_t)l * p.cap;
                const int first = min(len, nphi - a);
                bulk_copy_g2s(dst, src + a, 8u * (unsigned)first, &s_bar);
                if (first < len) bulk_copy_g2s(dst + first, src, 8u * (unsigned)(len - first), &s_bar);
            }
        }
        const bool ok = first_copy_wait(w, &s_bar);
        if (!__syncthreads_and(ok)) {
            // the copies did not land in time: report it, give them one more bound, write nothing
            if (threadIdx.x == 0) atomicOr(&w.stats[e].device_error, HOUGH_DEVERR_TIMEOUT);
            mbar_wait_bounded(&s_bar, 0, kCopyWaitCycles);
            return;
        }
    }
    // one warp per strip of up to 256 cells of a row, lane t taking cells t, t + 32, ...: a layer's
    // bit of cell j is the comparison of bucket entry j + I alone, so each of the lane's loads is
    // one 8-byte entry and a warp's loads cover consecutive entries
    constexpr int kCells = 8;
    uint16_t *M = w.M + (int64_t)e * ax.n_qpt * nphi;
    const int kc = min(kCells, p.cols >> 5);   // cells per lane (cols is a multiple of 64)
    const int strip = kc * 32;
    const int per_row = p.cols / strip;
    const int nstrips = nrows * per_row;
    const int lane = threadIdx.x & 31;
    for (int sidx = threadIdx.x >> 5; sidx < nstrips; sidx += TPB / 32) {
        const int rr = sidx / per_row;
        const int jb = c0 + (sidx - rr * per_row) * strip + lane;
        const unsigned vm = rowMask[rr];
        const int *rI = rowI + rr * 16;
        const unsigned *rG = rowG + rr * 16;
        unsigned mask[kCells];
#pragma unroll
        for (int c = 0; c < kCells; ++c) mask[c] = 0u;
#pragma unroll
        for (int l = 0; l < NL; ++l) {
            if (!((vm >> l) & 1u)) continue;   // the same for the whole warp: the row's layers
            const int I = rI[l];
            const unsigned gb = rG[l], ngb = ~gb;
            if ((staged >> l) & 1u) {
                const uint2 *src = win + (int64_t)l * p.cap + (jb + I - s_wbase[l]);   // inside the window
#pragma unroll
                for (int c = 0; c < kCells; ++c)
                    if (c < kc) {
                        const uint2 v = src[32 * c];
                        mask[c] |= (unsigned)((v.x > gb) | (v.y > ngb)) << l;
                    }
            } else {
                const uint2 *src = prof + (int64_t)l * pstride;
#pragma unroll
                for (int c = 0; c < kCells; ++c)
                    if (c < kc) {
                        const uint2 v = __ldg(&src[wrap_col(jb + 32 * c + I, nphi)]);
                        mask[c] |= (unsigned)((v.x > gb) | (v.y > ngb)) << l;
                    }
            }
        }
        uint16_t *row = M + (int64_t)(i0 + rr) * nphi + jb;
#pragma unroll
        for (int c = 0; c < kCells; ++c)
            if (c < kc) row[32 * c] = (uint16_t)mask[c];
    }
}


// The gather in rank form (see kRankRows in hough_internal.cuh).  A (cell, layer) costs one 4-byte
// shared load, one saturating half-pair addition -- 1 in either half says that the bucket, or the one
// after it, votes -- and one half-pair multiply-add that puts the layer's bit into the cell's two masks
// (one for each bucket, whole numbers below 1024, exact in halves), which are ORed at the end.  Why
// halves: gather_kernel's two integer comparisons, selects and ORs per (cell, layer), and likewise a
// packed 16-bit maximum, run in the half-rate integer pipe and bound the kernel there (11.9
// instructions per 32 (cell, layer)s, 6.5 of them in that pipe), while half arithmetic runs in the
// multiply-add pipe; what is left to bind is the shared loads.  The windows' copies are issued a layer
// a lane.
constexpr int kRankPad = 128;   // window entries beyond the tile's columns held in a layer's slot

__device__ __forceinline__ __half2 pair_of(uint32_t bits)
{
    return __halves2half2(__ushort_as_half((unsigned short)bits), __ushort_as_half((unsigned short)(bits >> 16)));
}

// The OR of a pair of masks below 1024: 1024 added, a mask is the significand's bits.
__device__ __forceinline__ uint32_t pair_mask(__half2 m)
{
    const __half2 s = __hadd2(m, __float2half2_rn(1024.f));
    const uint32_t u = (uint32_t)__half_as_ushort(__low2half(s)) | (uint32_t)__half_as_ushort(__high2half(s)) << 16;
    return (u | u >> 16) & 0x3FFu;
}

// A strip of 32 kc cells of a row: lane t's cells are columns jb, jb + 32, ... of the tile, jb holding the
// lane.  rowQ: per layer, the entry of column 0 in `win` and the threshold (kNoRank: no vote, or a layer
// whose window is not staged); slow: the layers of that kind, read from global memory (src, columns
// c0 + jb on, shift and threshold in rowS).  KC: cells a lane takes, when all strips are full (else 0).
template <int NL, int KC>
__device__ __forceinline__ void rank_strip(const uint32_t *win, const int2 *rowQ, unsigned slow, const int2 *rowS,
                                           const uint32_t *prof, int pstride, int nphi, int c0, int jb, int kc,
                                           uint16_t *row)
{
    constexpr int kCells = 8;
    // a mask pair holds ten layers; with more than ten, eight and the rest
    constexpr int kSplit = NL <= 10 ? NL : 8;
    __half2 mask[kCells], more[NL <= 10 ? 1 : kCells];
#pragma unroll
    for (int c = 0; c < kCells; ++c) mask[c] = __half2half2(__ushort_as_half(0));
#pragma unroll
    for (int c = 0; c < (NL <= 10 ? 1 : kCells); ++c) more[c] = __half2half2(__ushort_as_half(0));
    auto vote = [&](int l, int c, uint32_t entry, uint32_t th) {
        const __half2 bit = __float2half2_rn((float)(1 << (l < kSplit ? l : l - kSplit)));
        __half2 &m = l < kSplit ? mask[c] : more[NL <= 10 ? 0 : c];
        m = __hfma2(__hadd2_sat(pair_of(entry), pair_of(th)), bit, m);
    };
#pragma unroll
    for (int l = 0; l < NL; ++l) {
        const int2 q = rowQ[l];
        if ((uint32_t)q.y == kNoRank) continue;   // the same for the whole warp
        const uint32_t *src = win + q.x + jb;     // inside the window
        uint32_t v[kCells];
#pragma unroll
        for (int c = 0; c < kCells; ++c) v[c] = KC == kCells || c < kc ? src[32 * c] : 0u;
#pragma unroll
        for (int c = 0; c < kCells; ++c) vote(l, c, v[c], (uint32_t)q.y);
    }
    if (slow) {
#pragma unroll
        for (int l = 0; l < NL; ++l) {
            if (!((slow >> l) & 1u) || (uint32_t)rowS[l].y == kNoRank) continue;
            const uint32_t *src = prof + (int64_t)l * pstride;
#pragma unroll
            for (int c = 0; c < kCells; ++c)
                if (c < kc) vote(l, c, __ldg(&src[wrap_col(c0 + jb + 32 * c + rowS[l].x, nphi)]), (uint32_t)rowS[l].y);
        }
    }
#pragma unroll
    for (int c = 0; c < kCells; ++c)
        if (KC == kCells || c < kc) {
            uint32_t m = pair_mask(mask[c]);
            if (NL > 10) m |= pair_mask(more[NL <= 10 ? 0 : c]) << kSplit;
            row[32 * c] = (uint16_t)m;
        }
}

template <int NL, int TPB>
__global__ void __launch_bounds__(TPB) gather_rank_kernel(GatherParams p)
{
    pdl_enter();
    extern __shared__ __align__(16) unsigned char gather_smem[];
    __shared__ int2 rowS[kGatherRowsMax * 16];   // per (row, layer): I and threshold
    __shared__ int2 rowQ[kGatherRowsMax * 16];   // the same with I as the entry of the tile's column 0 in its window
    __shared__ unsigned s_staged, s_used;
    __shared__ __align__(8) uint64_t s_bar;
    const Axes &ax = p.ax;
    const Workspace &w = p.w;
    const int e = blockIdx.x / p.tiles_per_event;
    const int t = blockIdx.x - e * p.tiles_per_event;
    const int rt = t / p.col_tiles, ct = t - rt * p.col_tiles;
    const int i0 = rt * p.rows, c0 = ct * p.cols;
    const int nrows = min(p.rows, ax.n_qpt - i0);
    const int L = ax.n_layers, nphi = ax.n_phi;
    if (threadIdx.x == 0) mbar_init(&s_bar, 1);
    for (int q = threadIdx.x; q < nrows * 16; q += TPB) {
        const int rr = q >> 4, l = q & 15, i = i0 + rr;
        int2 v = make_int2(0, (int)kNoRank);
        if (l < L) {
            const LayerInfo li = w.info[l];
            const TabEntry te = w.tab[l * ax.n_qpt + i];   // all requested together: one round trip
            const uint32_t tr = w.rankt[l * ax.n_qpt + i];
            if (li.present && li.uniform && te.I != kNoVote) v = make_int2(te.I, (int)tr);
        }
        rowS[q] = v;
    }
    __syncthreads();
    const uint32_t *prof = w.prank + (int64_t)e * prof_event_entries(ax);
    const int pstride = prof_stride(ax);
    uint32_t *win = reinterpret_cast<uint32_t *>(gather_smem);
    if (threadIdx.x < 32) {
        // lane l: layer l's window of entries [c0 + min I, c0 + cols + max I) (unwrapped, rounded out to
        // 16 bytes), copied in pieces that end at the axis' seam; a window may hold more than the whole axis
        const int l = threadIdx.x;
        int lo = INT_MAX, hi = INT_MIN;
        if (l < L)
            for (int rr = 0; rr < nrows; ++rr) {
                const int2 v = rowS[rr * 16 + l];
                if ((uint32_t)v.y != kNoRank) {
                    lo = min(lo, v.x);
                    hi = max(hi, v.x);
                }
            }
        int ws = 0, len = 0;
        if (lo <= hi) {
            ws = (c0 + lo) & ~3;
            len = (c0 + p.cols + hi - ws + 3) & ~3;
        }
        const bool staged = len > 0 && len <= p.cap;
        const unsigned sm = __ballot_sync(0xFFFFFFFFu, staged), used = __ballot_sync(0xFFFFFFFFu, len > 0);
        const unsigned bytes = __reduce_add_sync(0xFFFFFFFFu, staged ? 4u * (unsigned)len : 0u);
        if (l == 0) {
            s_staged = sm;
            s_used = used;
            if (sm) mbar_arrive_expect(&s_bar, bytes);
        }
        __syncwarp();
        if (staged) {
            const uint32_t *src = prof + (int64_t)l * pstride;
            int a = ws % nphi;
            a += a < 0 ? nphi : 0;   // a multiple of 4, as nphi is
            for (int at = 0; at < len;) {
                const int n = min(len - at, nphi - a);
                bulk_copy_g2s(win + l * p.cap + at, src + a, 4u * (unsigned)n, &s_bar);
                at += n;
                a = 0;
            }
        }
        if (l < 16)
            for (int rr = 0; rr < nrows; ++rr) {
                const int2 v = rowS[rr * 16 + l];
                rowQ[rr * 16 + l] = make_int2(l * p.cap + c0 + v.x - ws, staged ? v.y : (int)kNoRank);
            }
    }
    __syncthreads();
    const unsigned staged = s_staged, slow = s_used & ~staged;
    if (staged) {
        const bool ok = first_copy_wait(w, &s_bar);
        if (!__syncthreads_and(ok)) {
            // the copies did not land in time: report it, give them one more bound, write nothing
            if (threadIdx.x == 0) atomicOr(&w.stats[e].device_error, HOUGH_DEVERR_TIMEOUT);
            mbar_wait_bounded(&s_bar, 0, kCopyWaitCycles);
            return;
        }
    }
    // one warp per strip of up to 256 cells of a row
    uint16_t *M = w.M + (int64_t)e * ax.n_qpt * nphi;
    const int kc = min(8, p.cols >> 5);   // cells per lane (cols is a multiple of 64)
    const int strip = kc * 32;
    // Known fault, the same as in gather_kernel: a tile more than 256 columns wide whose width is not a
    // multiple of 256 (320, 384, 448) loses the columns past its last whole strip; their cells keep the
    // zeros they were created with.
    const int per_row = p.cols / strip;
    const int nstrips = nrows * per_row;
    const int lane = threadIdx.x & 31;
    for (int sidx = threadIdx.x >> 5; sidx < nstrips; sidx += TPB / 32) {
        const int rr = sidx / per_row;
        const int jb = (sidx - rr * per_row) * strip + lane;   // column within the tile
        uint16_t *row = M + (int64_t)(i0 + rr) * nphi + c0 + jb;
        if (kc == 8)
            rank_strip<NL, 8>(win, rowQ + rr * 16, slow, rowS + rr * 16, prof, pstride, nphi, c0, jb, 8, row);
        else
            rank_strip<NL, 0>(win, rowQ + rr * 16, slow, rowS + rr * 16, prof, pstride, nphi, c0, jb, kc, row);
    }
}

// Fused vote and peak search (vote_mode HOUGH_VOTE_FUSED): a CTA per band of band_rows full rows.
// A cell of a layer of one radius is a function of its row's table entry and two bucket-profile
// entries alone, so the CTA computes the band's masks and those of the row above and below it
// (the 3 x 3 neighbourhoods; phi wraps within the full rows) into shared memory, searches the
// band for peaks there and writes the band's candidate list and count as the peak kernel does --
// the accumulator never goes to device memory.  Full rows read every bucket of a layer, so when
// they fit (STAGE) the voting layers' whole profiles are first copied into shared memory with
// bulk asynchronous copies; otherwise they are read through the cache.  When a present layer's
// hits lie at several radii the scatter kernel adds that layer's votes afterwards: the CTA then
// writes the band's rows to the accumulator instead, and the peak kernel searches it.

__device__ __forceinline__ bool all_layers_uniform(const Axes &ax, const Workspace &w)
{
    for (int l = 0; l < ax.n_layers; ++l) {
        const LayerInfo li = w.info[l];
        if (li.present && !li.uniform) return false;
    }
    return true;
}

template <int NL, int TPB, bool STAGE>
__global__ void __launch_bounds__(TPB) fused_kernel(GatherParams p)
{
    pdl_enter();
    extern __shared__ __align__(16) unsigned char fused_smem[];
    __shared__ int rowI[kGatherRowsMax * 16];
    __shared__ unsigned rowG[kGatherRowsMax * 16];
    __shared__ unsigned rowMask[kGatherRowsMax];
    __shared__ __align__(8) uint64_t s_bar;
    const Axes &ax = p.ax;
    const Workspace &w = p.w;
    const int nb = p.tiles_per_event;
    const int e = blockIdx.x / nb, band = blockIdx.x - e * nb;
    const int R = p.rows, i0 = band * R;
    const int nrows = min(R, ax.n_qpt - i0);
    const int L = ax.n_layers, nphi = ax.n_phi;
    const bool search = all_layers_uniform(ax, w);
    // computed rows: i0 - 1 .. i0 + nrows (halo included) when searching, else the band's own
    const int first = search ? i0 - 1 : i0;
    const int S = search ? nrows + 2 : nrows;
    for (int q = threadIdx.x; q < ((S * 16 + 31) & ~31); q += TPB) {
        const int s = q >> 4, l = q & 15, i = first + s;
        int I = 0;
        unsigned gb = 0u, valid = 0u;
        if (l < L && s < S && i >= 0 && i < ax.n_qpt) {   // rows outside the grid hold no votes
            const LayerInfo li = w.info[l];
            const TabEntry te = w.tab[l * ax.n_qpt + i];   // requested with the layer record: one round trip
            if (li.present && li.uniform && i >= li.lo && i <= li.hi) {
                if (te.I != kNoVote) {
                    I = te.I;
                    gb = __float_as_uint(te.g);
                    valid = 1u;
                }
            }
        }
        const unsigned m = __ballot_sync(0xFFFFFFFFu, valid) >> (threadIdx.x & 16);
        rowI[q] = I;
        rowG[q] = gb;
        if ((threadIdx.x & 15) == 0) rowMask[s] = m & 0xFFFFu;
    }
    __syncthreads();
    constexpr bool stage = STAGE;
    const uint2 *prof = w.prof + (int64_t)e * prof_event_entries(ax);
    const int pstride = prof_stride(ax);
    uint2 *win = reinterpret_cast<uint2 *>(fused_smem);   // staged: layer l's profile at l * n_phi
    uint16_t *tm = reinterpret_cast<uint16_t *>(fused_smem + (stage ? (size_t)L * nphi * sizeof(uint2) : 0));
    unsigned used = 0u;   // layers voting on any computed row
    for (int q = 0; q < S; ++q) used |= rowMask[q];
    if (stage && used) {
        if (threadIdx.x == 0) mbar_init(&s_bar, 1);
        __syncthreads();
        if (threadIdx.x == 0) {
            mbar_arrive_expect(&s_bar, (unsigned)__popc(used) * (unsigned)nphi * 8u);
            for (int l = 0; l < L; ++l)
                if ((used >> l) & 1u)
                    bulk_copy_g2s(win + (int64_t)l * nphi, prof + (int64_t)l * pstride, 8u * (unsigned)nphi, &s_bar);
        }
        const bool ok = first_copy_wait(w, &s_bar);
        if (!__syncthreads_and(ok)) {
            // the copies did not land in time: report it, give them one more bound, find nothing
            if (threadIdx.x == 0) {
                atomicOr(&w.stats[e].device_error, HOUGH_DEVERR_TIMEOUT);
                if (search) w.band_counts[(int64_t)e * nb + band] = 0;
            }
            mbar_wait_bounded(&s_bar, 0, kCopyWaitCycles);
            return;
        }
    }
    // a warp per strip of 256 cells of a row (the last strip of a row may be shorter: n_phi is a
    // multiple of 64), lane t taking cells t, t + 32, ...; a layer's bit of cell j compares the
    // profile entry j + I of that layer
    constexpr int kCells = 8;
    const int per_row = (nphi + 32 * kCells - 1) / (32 * kCells);
    const int lane = threadIdx.x & 31;
    for (int sidx = threadIdx.x >> 5; sidx < S * per_row; sidx += TPB / 32) {
        const int s = sidx / per_row;
        const int jb = (sidx - s * per_row) * 32 * kCells + lane;
        const unsigned vm = rowMask[s];
        unsigned mask[kCells];
#pragma unroll
        for (int c = 0; c < kCells; ++c) mask[c] = 0u;
#pragma unroll
        for (int l = 0; l < NL; ++l) {
            if (!((vm >> l) & 1u)) continue;   // the same for the whole warp: the row's layers
            const int I = rowI[s * 16 + l];
            const unsigned gb = rowG[s * 16 + l], ngb = ~gb;
            if (stage) {
                const uint2 *src = win + (int64_t)l * nphi;
#pragma unroll
                for (int c = 0; c < kCells; ++c)
                    if (jb + 32 * c < nphi) {
                        const uint2 v = src[wrap_col(jb + 32 * c + I, nphi)];
                        mask[c] |= (unsigned)((v.x > gb) | (v.y > ngb)) << l;
                    }
            } else {
                const uint2 *src = prof + (int64_t)l * pstride;
#pragma unroll
                for (int c = 0; c < kCells; ++c)
                    if (jb + 32 * c < nphi) {
                        const uint2 v = __ldg(&src[wrap_col(jb + 32 * c + I, nphi)]);
                        mask[c] |= (unsigned)((v.x > gb) | (v.y > ngb)) << l;
                    }
            }
        }
#pragma unroll
        for (int c = 0; c < kCells; ++c)
            if (jb + 32 * c < nphi) tm[s * nphi + jb + 32 * c] = (uint16_t)mask[c];
    }
    __syncthreads();
    if (!search) {
        // the scatter adds the other layers' votes: hand the band's rows to the peak kernel
        uint16_t *M = w.M + (int64_t)e * ax.n_qpt * nphi;
        const int v8 = nphi >> 3;
        for (int q = threadIdx.x; q < nrows * v8; q += TPB) {
            const int rr = q / v8, c8 = q - rr * v8;
            *reinterpret_cast<uint4 *>(M + (int64_t)(i0 + rr) * nphi + c8 * 8) =
                *reinterpret_cast<const uint4 *>(tm + rr * nphi + c8 * 8);
        }
        return;
    }
    uint2 *out = w.band_cands + ((int64_t)e * nb + band) * w.band_cap;
    const int cnt = band_peak_search<TPB, uint16_t, false, true>(tm, nrows, i0, nphi, ax.threshold, nullptr, out,
                                                                 w.band_cap);
    if (threadIdx.x == 0) w.band_counts[(int64_t)e * nb + band] = cnt;
}

// A context's bucket profile is read for the last time by the vote, which the peak search follows:
// zero it here for the next event (Workspace::recycle).
__device__ __forceinline__ void recycle_profile(const Axes &ax, const Workspace &w)
{
    if (!w.recycle || !w.prof || w.use_ranks) return;   // (with ranks the hit sort has zeroed it)
    uint4 *p4 = reinterpret_cast<uint4 *>(w.prof);
    const int64_t n4 = (int64_t)w.n_events * prof_event_entries(ax) / 2;   // two entries a vector
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n4; q += (int64_t)gridDim.x * blockDim.x)
        p4[q] = make_uint4(0u, 0u, 0u, 0u);
}

// Eight cells' layer counts of one row held by a lane, two to a word, with those of the columns to their
// left and right, and the three columns' maxima.
struct PeakRow {
    unsigned p[4], left[4], right[4], h[4];
};

// The row's masks v (eight cells) and, for the first and the last lane of a segment, the mask `halo` of the
// column before or after it: their layer counts.  `last`: the segment's last lane.
__device__ __forceinline__ PeakRow peak_row(const uint4 v, const unsigned halo, const int lane, const int last)
{
    PeakRow r;
    const unsigned m[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) r.p[k] = (unsigned)__popc(m[k] & 0xFFFFu) | (unsigned)__popc(m[k] >> 16) << 16;
    const unsigned hp = (unsigned)__popc(halo);
    unsigned before = __shfl_up_sync(0xFFFFFFFFu, r.p[3], 1), after = __shfl_down_sync(0xFFFFFFFFu, r.p[0], 1);
    if (lane == 0) before = hp << 16;
    if (lane == last) after = hp;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        r.left[k] = __byte_perm(k ? r.p[k - 1] : before, r.p[k], 0x5432);    // the columns one to the left
        r.right[k] = __byte_perm(r.p[k], k < 3 ? r.p[k + 1] : after, 0x5432);
        r.h[k] = __vmaxu2(__vmaxu2(r.left[k], r.p[k]), r.right[k]);
    }
    return r;
}

// Peak search of one band of band_rows rows of layer masks.  A warp takes segments of 256 columns, eight a
// lane, and walks down the band's rows and their halo: a row's masks are loaded and counted once, its
// neighbours to the left and right come from the next lanes, and a cell with count p is a candidate when p
// reaches the threshold, exceeds the maximum of the row above and of its left neighbour, and is not below
// those of the row below and of its right neighbour -- halfwise maxima of two cells a word.  The cells'
// flags, eight a byte, and each segment's number go to shared memory; once the band is searched, a scan of
// the segments in raster order places every candidate, and the warps write them out.  Bound by the
// counting (eight population counts a lane and row) and the halfwise maxima; with counts staged a byte a
// cell in shared memory and a thread comparing nine bytes a cell, 256 events took 739 us.
constexpr int kSegCols = 256;

__host__ __device__ inline int peak_segments(int nphi) { return (nphi + kSegCols - 1) / kSegCols; }
// Dynamic shared memory: the flags, then a count per (row, segment).
__host__ __device__ inline size_t peak_smem_bytes(int band_rows, int nphi)
{
    return (size_t)band_rows * peak_segments(nphi) * (32 + sizeof(int));
}

// D3: a grid with a d0 axis.  A band is band_rows q/pT rows of one slice m, and a cell's 3 x 3 x 3 block adds
// the maxima of its nine neighbours in slice m - 1, which precede it in raster order (strictly lower), and in
// slice m + 1 (not higher); rows outside the slice and slices outside the grid are empty.
template <bool D3>
__global__ void __launch_bounds__(kPeakThreads) peaks_mask_kernel(Axes ax, Workspace w)
{
    pdl_enter();
    recycle_profile(ax, w);
    if (!D3 && w.fused && all_layers_uniform(ax, w)) return;   // the fused vote searched the bands
    extern __shared__ __align__(16) unsigned char pc[];
    __shared__ int s_warp[kPeakThreads / 32];
    const int R = w.band_rows, nphi = ax.n_phi;
    const int nb = n_bands(ax, R), nseg = peak_segments(nphi);
    const int e = blockIdx.x / nb, band = blockIdx.x - e * nb;
    const int Q = ax.q_rows;                                     // rows of a slice
    const int bps = (Q + R - 1) / R, m = D3 ? band / bps : 0;    // bands of a slice, the band's slice
    const int i0 = (band - m * bps) * R, nrows = min(R, Q - i0);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int NW = kPeakThreads / 32;
    const uint16_t *M = w.M + ((int64_t)e * ax.n_qpt + (int64_t)m * Q) * nphi;   // the band's slice
    unsigned char *flags = pc;                                   // [row][segment][lane]
    int *seg_n = reinterpret_cast<int *>(pc + (size_t)R * nseg * 32);   // [row][segment]
    const unsigned thr = (unsigned)ax.threshold | (unsigned)ax.threshold << 16;
    for (int s = warp; s < nseg; s += NW) {
        const int j0 = s * kSegCols + lane * 8;
        const bool on = j0 < nphi;                               // n_phi is a multiple of 64
        const int last = min(31, ((nphi - s * kSegCols) >> 3) - 1);
        // the column before the first lane's, or after the last lane's (phi wraps)
        const int jh = lane == 0 ? (j0 ? j0 - 1 : nphi - 1) : (j0 + 8 < nphi ? j0 + 8 : 0);
        const bool halo_lane = lane == 0 || lane == last;
        auto load = [&](int i, uint4 &v, unsigned &halo, int slice = 0) {   // slice: -1, 0, 1 of the band's
            v = make_uint4(0u, 0u, 0u, 0u);
            halo = 0u;
            if (i >= 0 && i < Q && (!D3 || (m + slice >= 0 && m + slice < ax.n_d0))) {
                const uint16_t *row = M + (int64_t)(i + slice * Q) * nphi;
                if (on) v = *reinterpret_cast<const uint4 *>(row + j0);
                if (halo_lane) halo = row[jh];
            }
        };
        uint4 v[3];
        unsigned halo[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) load(i0 - 1 + q, v[q], halo[q]);
        unsigned up[4];   // the row above: maxima of three columns
        {
            const PeakRow r = peak_row(v[0], halo[0], lane, last);
#pragma unroll
            for (int k = 0; k < 4; ++k) up[k] = r.h[k];
        }
        PeakRow cur = peak_row(v[1], halo[1], lane, last);
        uint4 vn = v[2];
        unsigned hn = halo[2];
        // the slices before and after: their rows' maxima of three columns, the last two rows
        unsigned before[2][4], after[2][4];
        uint4 vb, va;
        unsigned hb, ha;
        if (D3) {
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                load(i0 - 1 + q, vb, hb, -1);
                load(i0 - 1 + q, va, ha, 1);
                const PeakRow rb = peak_row(vb, hb, lane, last), ra = peak_row(va, ha, lane, last);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    before[q][k] = rb.h[k];
                    after[q][k] = ra.h[k];
                }
            }
            load(i0 + 1, vb, hb, -1);
            load(i0 + 1, va, ha, 1);
        }
        for (int r = 0; r < nrows; ++r) {
            const PeakRow dn = peak_row(vn, hn, lane, last);
            if (r + 1 < nrows) load(i0 + r + 2, vn, hn);
            PeakRow rb, ra;
            if (D3) {
                rb = peak_row(vb, hb, lane, last);
                ra = peak_row(va, ha, lane, last);
                if (r + 1 < nrows) {
                    load(i0 + r + 2, vb, hb, -1);
                    load(i0 + r + 2, va, ha, 1);
                }
            }
            unsigned f = 0u;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                // counts are at most 16: no carry between the halves
                unsigned lower = __vmaxu2(up[k], cur.left[k]), upper = __vmaxu2(dn.h[k], cur.right[k]);
                if (D3) {
                    lower = __vmaxu2(lower, __vmaxu2(__vmaxu2(before[0][k], before[1][k]), rb.h[k]));
                    upper = __vmaxu2(upper, __vmaxu2(__vmaxu2(after[0][k], after[1][k]), ra.h[k]));
                    before[0][k] = before[1][k];
                    before[1][k] = rb.h[k];
                    after[0][k] = after[1][k];
                    after[1][k] = ra.h[k];
                }
                const unsigned need = __vmaxu2(__vmaxu2(lower + 0x00010001u, thr), upper);
                const unsigned ge = ((cur.p[k] | 0x80008000u) - need) & 0x80008000u;   // p >= need, by halves
                f |= (ge >> 15 & 1u) << (2 * k) | (ge >> 31) << (2 * k + 1);
            }
            if (!on) f = 0u;
            flags[(r * nseg + s) * 32 + lane] = (unsigned char)f;
            const int n = (int)__reduce_add_sync(0xFFFFFFFFu, (unsigned)__popc(f));
            if (lane == 0) seg_n[r * nseg + s] = n;
#pragma unroll
            for (int k = 0; k < 4; ++k) up[k] = cur.h[k];
            cur = dn;
        }
    }
    __syncthreads();
    // exclusive scan of the segments' numbers, in raster order, in place; each thread takes a run of them
    const int ns = nrows * nseg, per = (ns + kPeakThreads - 1) / kPeakThreads;
    const int q0 = min(ns, (int)threadIdx.x * per), q1 = min(ns, q0 + per);
    int sum = 0;
    for (int q = q0; q < q1; ++q) sum += seg_n[q];
    int incl = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int x = __shfl_up_sync(0xFFFFFFFFu, incl, d);
        if (lane >= d) incl += x;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    int base = 0, all = 0;
#pragma unroll
    for (int k = 0; k < NW; ++k) {
        base += k < warp ? s_warp[k] : 0;
        all += s_warp[k];
    }
    int run = base + incl - sum;
    for (int q = q0; q < q1; ++q) {
        const int n = seg_n[q];
        seg_n[q] = run;
        run += n;
    }
    if (threadIdx.x == 0) w.band_counts[(int64_t)e * nb + band] = all;
    if (!all) return;
    __syncthreads();
    uint2 *out = w.band_cands + ((int64_t)e * nb + band) * w.band_cap;
    for (int q = warp; q < ns; q += NW) {
        const int at0 = seg_n[q], end = q + 1 < ns ? seg_n[q + 1] : all;
        if (at0 == end) continue;
        unsigned f = flags[q * 32 + lane];
        const int n = __popc(f);
        int at = n;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int x = __shfl_up_sync(0xFFFFFFFFu, at, d);
            if (lane >= d) at += x;
        }
        at += at0 - n;
        const int r = q / nseg, i = i0 + r, j0 = (q - r * nseg) * kSegCols + lane * 8;
        while (f) {
            const int c = __ffs(f) - 1;
            f &= f - 1u;
            if (at < w.band_cap)
                out[at] = make_uint2((unsigned)(m * Q + i) << 16 | (unsigned)(j0 + c), M[(int64_t)i * nphi + j0 + c]);
            ++at;
        }
    }
}

// Peak search of one band of band_rows rows of vote counts, staged as they are (2 bytes each) with a halo
// row on each side.
__global__ void __launch_bounds__(kPeakThreads) peaks_count_kernel(Axes ax, Workspace w)
{
    pdl_enter();
    recycle_profile(ax, w);
    extern __shared__ __align__(16) unsigned char pc[];
    const int R = w.band_rows;
    const int nb = n_bands(ax, R);
    const int e = blockIdx.x / nb, band = blockIdx.x - e * nb;
    const int nphi = ax.n_phi;
    const int i0 = band * R;
    const int nrows = min(R, ax.n_qpt - i0);
    const uint16_t *M = w.M + (int64_t)e * ax.n_qpt * nphi;
    const int v8 = nphi >> 3;
    uint2 *out = w.band_cands + ((int64_t)e * nb + band) * w.band_cap;
    uint16_t *pv = reinterpret_cast<uint16_t *>(pc);
    for (int q = threadIdx.x; q < (nrows + 2) * v8; q += kPeakThreads) {
        const int rr = q / v8, c8 = q - rr * v8;
        const int i = i0 - 1 + rr;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (i >= 0 && i < ax.n_qpt) v = *reinterpret_cast<const uint4 *>(M + (int64_t)i * nphi + c8 * 8);
        *reinterpret_cast<uint4 *>(pv + rr * nphi + c8 * 8) = v;
    }
    __syncthreads();
    const int cnt = band_peak_search<kPeakThreads>(pv, nrows, i0, nphi, ax.threshold, M, out, w.band_cap);
    if (threadIdx.x == 0) w.band_counts[(int64_t)e * nb + band] = cnt;
}

// Peak search of one band of band_rows q/pT rows of one d0 slice m of a grid of vote counts with a d0 axis:
// the rows of its cells' 3 x 3 x 3 blocks -- rows i0 - 1 .. i0 + nrows of slices m - 1, m, m + 1 -- are staged
// as they are, rows outside the slice and slices outside the grid as empty.  Bands never cross a slice, so
// the band lists concatenate in raster order.
__global__ void __launch_bounds__(kPeakThreads) peaks3_count_kernel(Axes ax, Workspace w)
{
    pdl_enter();
    recycle_profile(ax, w);
    extern __shared__ __align__(16) unsigned char pc[];
    uint16_t *pv = reinterpret_cast<uint16_t *>(pc);
    const int R = w.band_rows, Q = ax.q_rows;
    const int bps = (Q + R - 1) / R;   // bands per slice
    const int nb = n_bands(ax, R);
    const int e = blockIdx.x / nb, band = blockIdx.x - e * nb;
    const int m = band / bps, i0 = (band - m * bps) * R;
    const int nrows = min(R, Q - i0);
    const int S = nrows + 2;
    const int nphi = ax.n_phi;
    const uint16_t *M = w.M + (int64_t)e * ax.n_qpt * nphi;
    const int v8 = nphi >> 3;
    for (int q = threadIdx.x; q < 3 * S * v8; q += kPeakThreads) {
        const int sidx = q / v8, c8 = q - sidx * v8;
        const int slice = sidx / S;
        const int mm = m + slice - 1, ii = i0 - 1 + (sidx - slice * S);
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (mm >= 0 && mm < ax.n_d0 && ii >= 0 && ii < Q)
            v = *reinterpret_cast<const uint4 *>(M + (int64_t)(mm * Q + ii) * nphi + c8 * 8);
        *reinterpret_cast<uint4 *>(pv + sidx * nphi + c8 * 8) = v;
    }
    __syncthreads();
    uint2 *out = w.band_cands + ((int64_t)e * nb + band) * w.band_cap;
    const int cnt = band_peak_search<kPeakThreads, uint16_t, true>(pv, nrows, m * Q + i0, nphi, ax.threshold, M, out, w.band_cap);
    if (threadIdx.x == 0) w.band_counts[(int64_t)e * nb + band] = cnt;
}

// Exclusive scan over the CTA (kCompactThreads threads); *total receives the sum.  Every thread takes part.
__device__ __forceinline__ int block_excl(int v, int *total)
{
    __shared__ int s_warp[kCompactThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int t = __shfl_up_sync(0xFFFFFFFFu, incl, d);
        if (lane >= d) incl += t;
    }
    __syncthreads();   // the last call's readers are done
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    int wi = s_warp[lane];
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int t = __shfl_up_sync(0xFFFFFFFFu, wi, d);
        if (lane >= d) wi += t;
    }
    *total = __shfl_sync(0xFFFFFFFFu, wi, 31);
    return incl - v + (warp > 0 ? __shfl_sync(0xFFFFFFFFu, wi, warp - 1) : 0);
}

// Compaction, first launch, one CTA per event: the exclusive scan of its band counts (band_offs) and
// its number of candidates; the CTA that finishes last adds up the kept candidates of the events
// before each one (cand_base), so that later kernels can spread all events' candidates over the
// whole device.
__global__ void __launch_bounds__(kCompactThreads) band_scan_kernel(Axes ax, Workspace w)
{
    pdl_enter();
    __shared__ int s_last;
    const int e = blockIdx.x, nb = n_bands(ax, w.band_rows);
    const int32_t *counts = w.band_counts + (int64_t)e * nb;
    int32_t *offs = w.band_offs + (int64_t)e * nb;
    int carry = 0;
    for (int b0 = 0; b0 < nb; b0 += kCompactThreads) {
        const int b = b0 + threadIdx.x;
        int sum;
        const int excl = block_excl(b < nb ? counts[b] : 0, &sum);
        if (b < nb) offs[b] = carry + excl;
        carry += sum;
    }
    if (threadIdx.x == 0) {
        w.stats[e].n_candidates = (unsigned)carry;
        if (carry > w.max_cand) atomicOr(&w.stats[e].device_error, HOUGH_DEVERR_CAND);
        __threadfence();
        s_last = atomicAdd(&w.counters->scans_done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    int base = 0;
    for (int e0 = 0; e0 < w.n_events; e0 += kCompactThreads) {
        const int ev = e0 + threadIdx.x;
        int sum;
        const int kept = ev < w.n_events ? (int)min((unsigned)w.max_cand, __ldcg(&w.stats[ev].n_candidates)) : 0;
        const int excl = block_excl(kept, &sum);
        if (ev < w.n_events) w.cand_base[ev] = base + excl;
        base += sum;
    }
    if (threadIdx.x == 0) {
        w.cand_base[w.n_events] = base;
        w.counters->total_cands = (unsigned)base;
        w.counters->scans_done = 0u;   // ready for the next event
    }
}

// Compaction, second launch: a warp per band copies its list to the flattened one (and, with
// `records`, to candidate records whose stage-2 fields are empty).  Bound by the 16-byte entries it
// writes; a CTA per part of an event that searched the bands of each candidate and wrote 32-byte
// records took 310 us for the 7.5M candidates of a 256-event batch.
__global__ void __launch_bounds__(256) band_copy_kernel(Axes ax, Workspace w, int records)
{
    pdl_enter();
    const int nb = n_bands(ax, w.band_rows);
    const int lane = threadIdx.x & 31;
    const int64_t bands = (int64_t)w.n_events * nb, nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t q = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); q < bands; q += nwarps) {
        const int n = w.band_counts[q];
        if (!n) continue;
        const int e = (int)(q / nb), o = w.band_offs[q], base = w.cand_base[e];
        const unsigned hstart = (unsigned)w.hit_start[e];
        const uint2 *list = w.band_cands + q * w.band_cap;
        for (int k = lane; k < min(n, w.max_cand - o); k += 32) {
            const uint2 v = list[k];
            w.cand_list[base + o + k] = make_uint4(v.x, v.y, (unsigned)e, hstart);
            if (records) {
                uint4 *cd = reinterpret_cast<uint4 *>(w.cands + base + o + k);
                cd[0] = make_uint4(v.x >> 16, v.x & 0xFFFFu, v.y, 0u);
                cd[1] = make_uint4(0u, 0u, 0u, 0u);
            }
        }
    }
}

// The first `limit` candidate records of all events to `out`, 16 bytes a thread.
__global__ void copy_candidates_kernel(Workspace w, hough_candidate *out, long long limit)
{
    pdl_enter();
    static_assert(sizeof(hough_candidate) == 32, "a record is two 16-byte vectors");
    const long long n = 2 * min((long long)w.cand_base[w.n_events], limit);
    const uint4 *src = reinterpret_cast<const uint4 *>(w.cands);
    uint4 *dst = reinterpret_cast<uint4 *>(out);
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x)
        dst[q] = src[q];
}

template <int TPB, int CELL>
cudaError_t launch_scatter(const VoteParams &p, size_t smem, int grid, cudaStream_t stream)
{
    cudaError_t err = cudaFuncSetAttribute(scatter_kernel<TPB, CELL>,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err) return err;
    return launch_chained(scatter_kernel<TPB, CELL>, dim3(grid), dim3(TPB), smem, stream, p);
}

template <int CELL>
cudaError_t launch_scatter_tpb(const VoteParams &p, int threads, size_t smem, int grid, cudaStream_t stream)
{
    switch (threads) {
    case 128: return launch_scatter<128, CELL>(p, smem, grid, stream);
    case 256: return launch_scatter<256, CELL>(p, smem, grid, stream);
    case 512: return launch_scatter<512, CELL>(p, smem, grid, stream);
    case 1024: return launch_scatter<1024, CELL>(p, smem, grid, stream);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace

// Shared memory of the scatter kernel: the column-major tile, the slab's table rows and q/pT centres,
// then a 32-hit buffer and a queue of FP64 votes per warp.  wide: a 32-bit word a cell.
static size_t scatter_smem_bytes(const Axes &ax, const Tiling &t, bool wide)
{
    return scatter_hit_offset(t.tile_qpt, t.tile_phi, ax.n_layers, wide) + (size_t)t.threads * sizeof(uint4) +
           (size_t)(t.threads / 32) * kRefineQueue * sizeof(uint2) + 32 * sizeof(uint32_t);
}

// The smallest form the tile can take: two 16-bit masks a word, or 32-bit counters.
size_t vote_smem_bytes(const Axes &ax, const Tiling &t) { return scatter_smem_bytes(ax, t, ax.counts != 0); }


static VoteParams vote_params(const Axes &ax, const Workspace &w, const Tiling &t, float refine_eps)
{
    VoteParams p;
    p.ax = ax;
    p.w = w;
    p.R = t.tile_qpt;
    p.W = t.tile_phi;
    p.n_spans = ax.n_phi / t.tile_phi;
    p.tiles_per_event = ((ax.n_qpt + t.tile_qpt - 1) / t.tile_qpt) * p.n_spans;
    p.s32 = (float)(ax.n_phi * kInvTwoPi);
    p.refine_eps = refine_eps;
    return p;
}

template <int NL>
cudaError_t launch_gather_nl(const GatherParams &p, int threads, size_t smem, int blocks, cudaStream_t stream)
{
    cudaError_t err;
    switch (threads) {
    case 256:
        if ((err = cudaFuncSetAttribute(gather_kernel<NL, 256>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)))
            return err;
        return launch_chained(gather_kernel<NL, 256>, dim3(blocks), dim3(256), smem, stream, p);
    case 1024:
        if ((err = cudaFuncSetAttribute(gather_kernel<NL, 1024>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)))
            return err;
        return launch_chained(gather_kernel<NL, 1024>, dim3(blocks), dim3(1024), smem, stream, p);
    default:
        if ((err = cudaFuncSetAttribute(gather_kernel<NL, 512>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)))
            return err;
        return launch_chained(gather_kernel<NL, 512>, dim3(blocks), dim3(512), smem, stream, p);
    }
}

size_t fused_smem_bytes(const Axes &ax, int band_rows)
{
    return (size_t)(band_rows + 2) * ax.n_phi * sizeof(uint16_t);
}

// Whether the fused kernel's CTA also holds every layer's whole bucket profile (8 bytes a bucket)
// beside its masks and row tables.
bool fused_stages_profiles(const Axes &ax, int band_rows)
{
    static std::atomic<int> optin{0};
    int m = optin.load(std::memory_order_relaxed);
    if (!m) {
        int dev = 0;
        cudaGetDevice(&dev);
        if (cudaDeviceGetAttribute(&m, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) return false;
        optin.store(m, std::memory_order_relaxed);
    }
    return fused_smem_bytes(ax, band_rows) + (size_t)ax.n_layers * ax.n_phi * sizeof(uint2) + 6144 + 1024 <= (size_t)m;
}

size_t gather_smem_bytes(const Axes &ax, const Tiling &t)
{
    return (size_t)ax.n_layers * (size_t)(t.gather_cols + 64) * sizeof(uint2);
}

template <int NL>
cudaError_t launch_gather_rank_nl(const GatherParams &p, int threads, size_t smem, int blocks, cudaStream_t stream)
{
    auto kernel = threads == 256 ? gather_rank_kernel<NL, 256> : threads == 1024 ? gather_rank_kernel<NL, 1024>
                                                                                 : gather_rank_kernel<NL, 512>;
    cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err) return err;
    return launch_chained(kernel, dim3(blocks), dim3(threads), smem, stream, p);
}

static cudaError_t launch_gather_tiled(const Axes &ax, const Workspace &w, const Tiling &t, cudaStream_t stream)
{
    GatherParams p;
    p.ax = ax;
    p.w = w;
    p.rows = t.gather_rows;
    p.cols = t.gather_cols;
    p.col_tiles = ax.n_phi / p.cols;
    p.tiles_per_event = ((ax.n_qpt + p.rows - 1) / p.rows) * p.col_tiles;
    const int blocks = w.n_events * p.tiles_per_event;
    if (w.use_ranks) {
        p.cap = t.gather_cols + kRankPad;
        const size_t smem = (size_t)ax.n_layers * p.cap * sizeof(uint32_t);
        // layer loops unrolled
        if (ax.n_layers <= 4) return launch_gather_rank_nl<4>(p, t.gather_threads, smem, blocks, stream);
        if (ax.n_layers <= 8) return launch_gather_rank_nl<8>(p, t.gather_threads, smem, blocks, stream);
        if (ax.n_layers <= 10) return launch_gather_rank_nl<10>(p, t.gather_threads, smem, blocks, stream);
        return launch_gather_rank_nl<16>(p, t.gather_threads, smem, blocks, stream);
    }
    p.cap = t.gather_cols + 64;
    const size_t smem = gather_smem_bytes(ax, t);
    // layer loops unrolled to the next multiple of four
    if (ax.n_layers <= 4) return launch_gather_nl<4>(p, t.gather_threads, smem, blocks, stream);
    if (ax.n_layers <= 8) return launch_gather_nl<8>(p, t.gather_threads, smem, blocks, stream);
    if (ax.n_layers <= 12) return launch_gather_nl<12>(p, t.gather_threads, smem, blocks, stream);
    return launch_gather_nl<16>(p, t.gather_threads, smem, blocks, stream);
}

template <int NL, int TPB>
cudaError_t launch_fused_tpb(const GatherParams &p, size_t smem, int blocks, cudaStream_t stream)
{
    auto kernel = p.cap ? fused_kernel<NL, TPB, true> : fused_kernel<NL, TPB, false>;
    cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err) return err;
    return launch_chained(kernel, dim3(blocks), dim3(TPB), smem, stream, p);
}

template <int NL>
cudaError_t launch_fused_nl(const GatherParams &p, int threads, size_t smem, int blocks, cudaStream_t stream)
{
    switch (threads) {
    case 256: return launch_fused_tpb<NL, 256>(p, smem, blocks, stream);
    case 1024: return launch_fused_tpb<NL, 1024>(p, smem, blocks, stream);
    default: return launch_fused_tpb<NL, 512>(p, smem, blocks, stream);
    }
}

// One CTA per band of the peak search (w.band_rows full rows).
static cudaError_t launch_fused(const Axes &ax, const Workspace &w, const Tiling &t, cudaStream_t stream)
{
    GatherParams p;
    p.ax = ax;
    p.w = w;
    p.rows = w.band_rows;
    p.cols = ax.n_phi;
    p.cap = fused_stages_profiles(ax, w.band_rows) ? 1 : 0;
    p.col_tiles = 1;
    p.tiles_per_event = n_bands(ax, w.band_rows);
    const int blocks = w.n_events * p.tiles_per_event;
    const size_t smem = fused_smem_bytes(ax, w.band_rows) + (p.cap ? (size_t)ax.n_layers * ax.n_phi * sizeof(uint2) : 0);
    if (ax.n_layers <= 4) return launch_fused_nl<4>(p, t.gather_threads, smem, blocks, stream);
    if (ax.n_layers <= 8) return launch_fused_nl<8>(p, t.gather_threads, smem, blocks, stream);
    if (ax.n_layers <= 12) return launch_fused_nl<12>(p, t.gather_threads, smem, blocks, stream);
    return launch_fused_nl<16>(p, t.gather_threads, smem, blocks, stream);
}

// The tile of the shared-atomic vote where the caller's tiling does not choose it (counts in gather mode,
// the allocation-free vote): 32 rows, a lane each, and as many warps as make the chip busy -- 32 when the
// tiles do not outnumber the SMs (one 100k-hit event, 128 tiles: 37 us against 45 and 65 us with 16 and 8
// warps), 8 when there are many, mostly empty ones (16 x 256 x 2048 cells, 1,024 tiles: 33 us against 53
// us with 32 warps).
Tiling scatter_tiling(const Axes &ax, int n_events, Tiling t)
{
    t.tile_phi = std::min(ax.n_phi, 256);
    while (ax.n_phi % t.tile_phi) t.tile_phi -= 64;
    t.tile_qpt = std::min(ax.n_qpt, 32);
    const int64_t tiles = (int64_t)n_events * ((ax.n_qpt + t.tile_qpt - 1) / t.tile_qpt) * (ax.n_phi / t.tile_phi);
    t.threads = tiles <= 152 ? 1024 : tiles <= 608 ? 512 : 256;
    return t;
}

cudaError_t launch_gather(const Axes &ax, const Workspace &w, const Tiling &t, cudaStream_t stream)
{
    if (t.vote_mode == HOUGH_VOTE_FUSED) return launch_fused(ax, w, t, stream);
    if (!ax.counts) return launch_gather_tiled(ax, w, t, stream);
    // Counts are scattered in either mode: a cell's count depends on every hit of its buckets, not on two
    // extrema, and listing them cell by cell took three to fifteen times the scatter's time (100k-hit event
    // 186 us against 37, 16 x 256 x 2048 cells 628 against 33, 2048 x 2048 with 5,000 hits 342 against 26).
    return launch_scatter(ax, w, scatter_tiling(ax, w.n_events, t), refine_eps_for(ax), false, stream);
}

static cudaError_t launch_general(const Axes &ax, const Workspace &w, float refine_eps, cudaStream_t stream)
{
    GeneralParams p;
    p.ax = ax;
    p.w = w;
    p.n_spans = (ax.n_phi + kGenCols - 1) / kGenCols;
    p.tiles_per_event = ((ax.n_qpt + kGenRows - 1) / kGenRows) * p.n_spans;
    p.s32 = (float)(ax.n_phi * kInvTwoPi);
    p.refine_eps = refine_eps;
    cudaError_t err = cudaFuncSetAttribute(general_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(GeneralSmem));
    if (err) return err;
    const int grid = (int)std::min<int64_t>((int64_t)w.n_events * p.tiles_per_event, 152);
    return launch_chained(general_kernel, dim3(grid), dim3(kGenThreads), sizeof(GeneralSmem), stream, p);
}

cudaError_t launch_scatter(const Axes &ax, const Workspace &w, const Tiling &t, float refine_eps, bool general_only,
                           cudaStream_t stream)
{
    if (general_only) return ax.counts ? cudaSuccess : launch_general(ax, w, refine_eps, stream);   // (counts: every layer is voted)
    const VoteParams p = vote_params(ax, w, t, refine_eps);
    const int grid = w.n_events * p.tiles_per_event;
    if (ax.counts) {
        const size_t smem = scatter_smem_bytes(ax, t, true);
        return launch_scatter_tpb<2>(p, t.threads, smem, grid, stream);
    }
    // a mask a word when that tile fits (no shift to place the bit), else two a word
    static std::atomic<int> optin{0};
    int m = optin.load(std::memory_order_relaxed);
    if (!m) {
        int dev = 0;
        cudaGetDevice(&dev);
        if (cudaDeviceGetAttribute(&m, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) m = 48 * 1024;
        optin.store(m, std::memory_order_relaxed);
    }
    const size_t wide = scatter_smem_bytes(ax, t, true);
    if (wide + 1024 <= (size_t)m)
        return launch_scatter_tpb<1>(p, t.threads, wide, grid, stream);
    const size_t smem = scatter_smem_bytes(ax, t, false);
    return launch_scatter_tpb<0>(p, t.threads, smem, grid, stream);
}

cudaError_t launch_vote(const Axes &ax, const Workspace &w, const Tiling &t, float refine_eps,
                        cudaStream_t stream)
{
    if (t.vote_mode == HOUGH_VOTE_SCATTER) return launch_scatter(ax, w, t, refine_eps, false, stream);
    // gather every table layer (fused with the peak search under HOUGH_VOTE_FUSED), then let the
    // scatter kernel add the layers whose radii differ
    cudaError_t err = launch_gather(ax, w, t, stream);
    if (err) return err;
    return launch_scatter(ax, w, t, refine_eps, true, stream);
}


cudaError_t launch_band_peaks(const Axes &ax, const Workspace &w, const Tiling &t, cudaStream_t stream)
{
    const int nb = n_bands(ax, w.band_rows);
    const size_t smem = ax.counts ? band_smem_bytes(ax, w.band_rows) : peak_smem_bytes(w.band_rows, ax.n_phi);
    auto kernel = ax.n_d0 ? (ax.counts ? peaks3_count_kernel : peaks_mask_kernel<true>)
                          : (ax.counts ? peaks_count_kernel : peaks_mask_kernel<false>);
    cudaError_t err;
    if ((err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem))) return err;
    if ((err = launch_chained(kernel, dim3(w.n_events * nb), dim3(kPeakThreads), smem, stream, ax, w))) return err;
    return cudaGetLastError();
}

cudaError_t launch_compact(const Axes &ax, const Workspace &w, cudaStream_t stream, bool records)
{
    cudaError_t err = launch_chained(band_scan_kernel, dim3(w.n_events), dim3(kCompactThreads), 0, stream, ax, w);
    if (err) return err;
    const int64_t bands = (int64_t)w.n_events * n_bands(ax, w.band_rows);
    const int blocks = (int)std::min<int64_t>((bands + 7) / 8, 1216);
    return launch_chained(band_copy_kernel, dim3(blocks), dim3(256), 0, stream, ax, w, records ? 1 : 0);
}

cudaError_t launch_copy_candidates(const Workspace &w, hough_candidate *out, cudaStream_t stream, long long limit)
{
    return launch_chained(copy_candidates_kernel, dim3(1216), dim3(256), 0, stream, w, out, limit);
}

}  // namespace hough
