// Confirmation of the candidates (Sec. 4: candidates found as local maxima are confirmed by "more
// expensive computations"): for each candidate, the hits whose stage-1 vote fell in its cell
// (membership) and their vote in a (cot theta, z0) grid of layer masks (stage 2).
//
// One kernel, confirm_kernel.  A warp takes a group of C consecutive candidates of the flattened
// list (three for detectors of at most 10 layers, two for more; fewer when there are not enough
// candidates to fill the GPU's warps) and goes through
//
//   1. Ranges.  Only layers present in a candidate's mask can hold members (with the count
//      accumulator every layer is scanned).  For a layer whose hits share one radius the vote
//      inverts exactly -- a hit of bucket J votes into column j on row i when
//      J = j + I_i + (f < g_i) -- so two neighbouring buckets of the (layer, azimuth bucket)-sorted
//      hits hold all of that layer's members: bucket j + I_i with f >= g_i and the one after it
//      with f < g_i.  A lane per (candidate, layer) forms that one range, its split point and the
//      jump at the split where the second bucket wraps around phi.  Other layers give the buckets
//      their radius range allows, whose hits redo the vote (FP32 with FP64 refinement, as in the
//      vote kernel).
//   2. Membership.  The warp tests the flattened union of all C candidates' ranges, a lane per hit.
//      A lane's range is found without a search: the ranges starting inside the window of 32 hits
//      are OR-reduced into one bit mask (a redux), and a population count below the lane gives its
//      range.  Members are listed by ballot in the fixed order (candidate, layer, position).
//   3. Coefficients, a lane per listed member, 32 members a round whatever candidates they belong
//      to: the z0 coordinate of its vote on cot row m,
//      w(m) = n_z0 (z - s t_m - z0_min) / (z0_max - z0_min) = a - (m - m_ref) b, evaluated in FP32
//      around the row m_ref where it crosses z0_min, from coefficients formed in two-float
//      arithmetic (to within 2e-5 bin of its exact value), and the run of rows whose vote falls
//      inside the z0 range (w is monotone in m, so they form one run).
//   4. Stage-2 vote, candidate by candidate.  The (member, row) pairs of a candidate's runs are
//      spread over the lanes -- a pair's member found by a population count of a bit array that
//      marks each run's first pair -- and voted with a shared atomicOr into the warp's
//      n_cot x n_z0 grid (16-bit masks, or for detectors of at most 10 layers 10-bit masks three
//      to a word, 5.3 KB for 64 x 64).  The word the atomic returns judges the cell: the last OR
//      into a cell sees its final mask and every earlier one a subset, so the largest popcount
//      seen is the grid's maximum and the lowest cell seen with it the row-major-first arg-max.
//      Each lane keeps the best as one 32-bit key (popcount, then the complement of the cell
//      index), and a redux finds the warp's.
//   5. The cell's final mask is read back, the grid cleared, the record written.
//
// Why groups of candidates: a candidate of a batch scans about 30 hits of 9 layers, has 15 members
// and casts 140 stage-2 votes, so with one candidate a warp the lanes of steps 1-3 were half idle
// and their fixed cost (prefix sums, compactions, broadcasts) was paid per candidate.  Only the
// vote needs a grid of its own, and it alone is done a candidate at a time, so a group costs no
// more shared memory than a candidate did.
//
// When the list is full its members go through steps 3 and 4 before further hits are tested, a
// candidate's grid, best key and counts being carried on.  The member lists are kept for contexts (hough_get_members
// reads them), in the event's member pool, where a slot is reserved once a candidate's members are
// counted; a batch keeps none.  The event's member and stage-2 vote counters are summed per warp
// and added once per event a warp visits.
#include <algorithm>
#include <atomic>
#include <climits>

#include "hough_internal.cuh"

namespace hough {

namespace {

constexpr int kWarps = 4;             // warps per CTA at most (fewer when their grids do not fit)
constexpr int kListCap = 96;          // members a warp lists at a time
constexpr int kMaxBandsRead = 8192;   // bands of a single event whose lists the confirmation reads itself
constexpr int kTeamRounds = 2;        // one event with at most so many candidates per CTA: its warps share each candidate
constexpr int kBandChunks = 64;       // coarse band offsets a CTA holds to do so

// Per-warp scratch; the start bits of the runs and the grid follow it.
struct __align__(16) Scratch {
    int4 par[32];           // a round's members with a run of cot rows: a, b, (first row - first pair - m_ref) (float bits);
                            // (first row - first pair) * n_z0 * 32 + layer
    float4 zco[32];         // stage-2 terms {S hi, S lo, B hi, B lo} by lane (candidate, layer)
    int4 seg[32];           // the non-empty ranges: staged position less flattened index, flattened index of the
                            // split, g (float bits), jump of the staged position at the split
    int list_p[kListCap];   // the chunk's members: staged position
    unsigned char list_slot[kListCap];   // and slot
    unsigned char seg_slot[32];          // lane (candidate, layer) of a range, bit 5: a layer of several radii
};

// What the warps of a team exchange.
struct Team {
    unsigned best[kWarps];
    int members[kWarps];
    int pool_base, pool_n;
};

__device__ __forceinline__ unsigned lanes_below() { return (1u << (threadIdx.x & 31)) - 1u; }

__device__ __forceinline__ TabEntry load_tab(const TabEntry *p)
{
    const int2 v = __ldg(reinterpret_cast<const int2 *>(p));
    return TabEntry{v.x, __int_as_float(v.y)};
}

__device__ __forceinline__ int warp_incl_scan(int v)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int t = __shfl_up_sync(0xFFFFFFFFu, v, d);
        if (lane >= d) v += t;
    }
    return v;
}

// The (up to two) ranges of staged hits of a layer whose hits lie at several radii that can hold
// members of candidate (i, j): the buckets its radius range allows on row i.  Returns the count.
__device__ int general_ranges(const Axes &ax, const Workspace &w, const int32_t *offs, int l, int i, int j, float s32,
                              int st[2], int en[2])
{
    const int nphi = ax.n_phi;
    const int lstart = offs[l * nphi], lend = offs[(l + 1) * nphi];
    if (ax.n_d0) {   // a grid with a d0 axis: every hit of the layer
        st[0] = lstart;
        en[0] = lend;
        return 1;
    }
    const float k = w.kq32[i];
    const float c_lo = 0.15f * (float)ax.b / 100.f * __uint_as_float(w.radii->rmin[l]) * 0.999f;
    const float c_hi = 0.15f * (float)ax.b / 100.f * __uint_as_float(w.radii->rmax[l]) * 1.001f;
    const float a1 = asinf(fminf(fmaxf(c_lo * k, -1.f), 1.f));
    const float a2 = asinf(fminf(fmaxf(c_hi * k, -1.f), 1.f));
    const int ja = (int)floorf(j + s32 * fminf(a1, a2)) - 2;
    const int jb = (int)floorf(j + 1 + s32 * fmaxf(a1, a2)) + 2;
    if (jb - ja + 1 >= nphi) {
        st[0] = lstart;
        en[0] = lend;
        return 1;
    }
    const int a = wrap_col(ja, nphi), b = wrap_col(jb, nphi);   // within nphi / 4 + 3 of [0, nphi)
    if (a <= b) {
        st[0] = offs[l * nphi + a];
        en[0] = offs[l * nphi + b + 1];
        return 1;
    }
    st[0] = offs[l * nphi + a];
    en[0] = lend;
    st[1] = lstart;
    en[1] = offs[l * nphi + b + 1];
    return 2;
}

// Whether the staged hit at position p of a layer whose hits lie at several radii votes into cell
// (i, j): the vote redone per hit, as the vote kernel casts it.
__device__ __forceinline__ bool general_member(const Axes &ax, const Workspace &w, const HotHit *hot,
                                               const ColdHit *cold, int p, int i, int j, float s32, float refine_eps)
{
    const HotHit hh = hot[p];
    int jj = 0;
    if (ax.n_d0) {   // every vote in FP64 on a grid with a d0 axis
        const ColdHit ch = cold[p];
        return exact_vote(ax, (double)ch.r, (double)ch.phi, i, &jj) && jj == j;
    }
    const int rlo = (int)(hh.rows & 0xFFFFu), rhi = (int)(hh.rows >> 16);
    if (i < rlo || i > rhi) return false;
    const float x = fminf(fmaxf(hh.c * w.kq32[i], -1.f), 1.f);
    const float vq = fmaf(-asinf(x), s32, hh.f);
    const float fl = floorf(vq);
    const float d = vq - fl;
    jj = (int)(hh.jl & 0xFFFFu) + (int)fl;
    if (d < refine_eps || d > 1.f - refine_eps || fabsf(x) > kRefineXLim) {
        const ColdHit ch = cold[p];
        jj = exact_bin(ax, (double)ch.phi, __dmul_rn(sagitta_coef(ax, (double)ch.r), qpt_centre(ax, i)));
    }
    return wrap_col(jj, ax.n_phi) == j;
}

// Stage-2 coefficients of a member of a layer of one radius at row i: z0 coordinate
// w(m) = a - (m - m_ref) b in FP32.  The per-row terms S = zscale s t_0 and B = zscale s dt come
// from the table and w(m_ref) = zscale (z - z0_min) - S - m_ref B is formed in two-float
// arithmetic (about 2^-44 relative before the final rounding), which keeps a within a few 1e-6
// bins of the exact value.
__device__ __forceinline__ void table_coefficients(const Axes &ax, const float4 zc, float rb, float z, float *a_out,
                                                   float *b_out, float *mref_out)
{
    // d = z - z0_min and Z = zscale d as two-float values
    float2 d = two_sum(z, -ax.zmin_hi);
    d.y = __fsub_rn(d.y, ax.zmin_lo);
    const float2 zp = two_prod(d.x, ax.zs_hi);
    const float zlo = zp.y + d.x * ax.zs_lo + d.y * ax.zs_hi;
    // A = Z - S
    float2 A = two_sum(zp.x, -zc.x);
    A.y = A.y + (zlo - zc.y);
    // any nearby row will do
    const float fm = zc.z > 0.f ? fminf(fmaxf(rintf(A.x * rb), 0.f), (float)(ax.n_cot - 1)) : 0.f;
    // a = A - m_ref B; m_ref B.hi is exact as a two-float product
    const float2 q = two_prod(fm, zc.z);
    *a_out = __fsub_rn(A.x, q.x) + (A.y - q.y - fm * zc.w);
    *b_out = zc.z;
    *mref_out = fm;
}

// The same for a member of a layer whose hits lie at several radii: the arc length from the
// closest approach in FP64 (r asin(|x|) / |x| for prompt tracks).
__device__ __forceinline__ void exact_coefficients(const Axes &ax, int i, const ColdHit &ch, float *a_out,
                                                   float *b_out, float *mref_out)
{
    const double rd = (double)ch.r;
    const double x = __dmul_rn(sagitta_coef(ax, rd), qpt_centre(ax, i));
    const double d0 = d0_centre(ax, i);
    double y = x;
    track_sin(rd, x, d0, &y);   // a member's track passes its radius: its vote was cast
    const double s = track_arc(rd, x, d0, y);
    const double t0 = __dadd_rn(ax.cot_min, __dmul_rn(0.5, ax.dt));
    const double A = __dmul_rn(ax.zscale, __dsub_rn(__dsub_rn((double)ch.z, ax.z0_min), __dmul_rn(s, t0)));
    const double B = __dmul_rn(ax.zscale, __dmul_rn(s, ax.dt));
    float mref = 0.f;
    if (B > 0.0) mref = fminf(fmaxf(rintf((float)A / (float)B), 0.f), (float)(ax.n_cot - 1));
    *a_out = (float)(A - (double)mref * B);
    *b_out = (float)B;
    *mref_out = mref;
}

// The run of cot rows whose vote of the member can fall inside the z0 range.  w(m) is the rounding
// of a quantity strictly decreasing in m (b > 0), so it is non-increasing and the rows with
// 0 <= w(m) < n_z0 form one run.  Approximate quotients bound the run from outside by about a row
// on each side; one step at each end then drops a bound whose own vote falls outside, which
// leaves the exact run in all but rare cases (a row of an outer bound still outside: every pair
// is tested again when it votes).  Rows are whole numbers held as floats (at most 256, exact).
// *len receives the length (0: no row).
__device__ __forceinline__ void member_run(float n_cot, float n_z0, float a, float b, float rb, float mref, float *lo_out,
                                           int *len_out)
{
    const float top = n_cot - 1.f;
    const float alo = a - n_z0;
    float lo = fminf(fmaxf(floorf(fmaf(alo, rb, mref)), 0.f), n_cot);   // rb: about 1 / b
    float hi = fminf(fmaxf(floorf(fmaf(a, rb, mref)) + 1.f, -1.f), top);
    const float wlo = fmaf(-(lo - mref), b, a), whi = fmaf(-(hi - mref), b, a);
    if (!(wlo >= 0.f && wlo < n_z0)) lo += 1.f;   // (of an empty run too: it stays empty)
    if (!(whi >= 0.f && whi < n_z0)) hi -= 1.f;
    if (!(b > 0.f)) {   // w constant in m: every row or none
        lo = 0.f;
        hi = a >= 0.f && a < n_z0 ? top : -1.f;
    }
    *lo_out = lo;
    *len_out = (int)fmaxf(hi - lo + 1.f, 0.f);
}

template <bool P10>
__device__ __forceinline__ uint32_t grid_mask(const uint32_t *grid, unsigned cell)
{
    const unsigned word = P10 ? cell / 3u : cell >> 1;
    const unsigned shift = P10 ? (cell - word * 3u) * 10u : (cell & 1u) << 4;
    return (grid[word] >> shift) & (P10 ? 0x3FFu : 0xFFFFu);
}

// A candidate record as two 16-byte vectors (the arrays are 16-byte aligned, 32 bytes an entry).
__device__ __forceinline__ void store_candidate(hough_candidate *p, const hough_candidate &c)
{
    reinterpret_cast<uint4 *>(p)[0] = make_uint4(c.iq, c.jphi, c.mask, c.n_members);
    reinterpret_cast<uint4 *>(p)[1] = make_uint4(c.icot, c.jz0, c.mask2, c.flags);
}


// A candidate as the confirmation takes it: (row << 16 | column), mask, event, the event's first hit.
struct ListEntry {
    unsigned ij, mask;
    int e, hstart;
};

// One event whose list was not compacted: the CTA scans the band counts, keeping the offset of the
// first band of each of kBandChunks chunks of `chunk` bands in `coarse` (coarse[kBandChunks]: the
// total).  A candidate's band is then found by a search over the coarse offsets and a walk over the
// counts of one chunk.
__device__ int scan_bands(const int32_t *counts, int nb, int chunk, int *coarse)
{
    __shared__ int s_w[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int carry = 0;
    for (int c0 = 0; c0 < kBandChunks; c0 += blockDim.x) {
        const int c = c0 + threadIdx.x;
        const int k0 = min(nb, c * chunk), k1 = min(nb, k0 + chunk);
        int sum = 0;
        for (int k = k0; k < k1; ++k) sum += counts[k];
        const int incl = warp_incl_scan(sum);
        __syncthreads();
        if (lane == 31) s_w[warp] = incl;
        __syncthreads();
        int before = carry, all = 0;
        for (int k = 0; k < nw; ++k) {
            before += k < warp ? s_w[k] : 0;
            all += s_w[k];
        }
        if (c < kBandChunks) coarse[c] = before + incl - sum;
        carry += all;
    }
    if (threadIdx.x == 0) coarse[kBandChunks] = carry;
    __syncthreads();
    return carry;
}

// Membership and stage 2 of every group of C candidates the warp takes.  NL: layers a candidate has
// lanes for.  GEN: some layer's hits lie at several radii (their votes are redone per hit, partly in
// FP64); without it that code is left out, which spares the common path its registers.
// G64: the stage-2 grid is 64 x 64 (its sizes are then constants of the code).
// TEAM: the CTA's kWarps warps share one candidate at a time (C is 1): each takes every kWarps-th
// window of its hits through steps 2-4 with a list of its own, voting into one grid, and they meet
// to combine their keys.  KEEP: the member lists are kept.
template <int NL, bool P10, bool G64, bool GEN, bool KEEP, bool TEAM>
__device__ __forceinline__ void confirm_groups(const Axes &ax, const Workspace &w, float s32, float refine_eps,
                                               Scratch &S, Team *team, unsigned *starts, uint32_t *grid, const int grid_vecs,
                                               unsigned layers_present, unsigned layers_general, int C, int first, int step,
                                               int total, const int *coarse, int chunk)
{
    const int lane = threadIdx.x & 31;
    constexpr int TW = TEAM ? kWarps : 1;
    const int wpos = TEAM ? (int)(threadIdx.x >> 5) : 0;
    const unsigned upto = (2u << lane) - 1u;
    const int nphi = ax.n_phi, nkeys = ax.n_layers * nphi;
    const int kc = lane / NL, l = lane - kc * NL;   // the lane's candidate of the group and layer
    const bool lane_on = kc < C && l < ax.n_layers;
    const int n_z0 = G64 ? 64 : ax.n_z0;
    const float n_z0f = (float)n_z0, n_cotf = G64 ? 64.f : (float)ax.n_cot;
    const unsigned grid_s = smem_u32(grid);
    // the event's counters, summed over the candidates of one event and added when it changes (a
    // lane's own votes are added up over the warp only then)
    int acc_e = 0;
    unsigned acc_members = 0u, acc_votes = 0u;
    auto flush = [&](int e) {
        const unsigned long long v = (unsigned long long)__reduce_add_sync(0xFFFFFFFFu, acc_votes & 0xFFFFu) +
                                     ((unsigned long long)__reduce_add_sync(0xFFFFFFFFu, acc_votes >> 16) << 16);
        if (lane == 0) {
            if (acc_members) atomicAdd(&w.stats[acc_e].n_members, acc_members);
            if (v) atomicAdd(&w.stats[acc_e].stage2_votes, v);
        }
        acc_e = e;
        acc_members = acc_votes = 0u;
    };

    auto fetch = [&](int f0) {
        ListEntry r{0u, 0u, 0, 0};
        const int f = f0 + kc;
        if (kc >= C || f >= total) return r;
        if (!coarse) {
            const uint4 v = __ldg(reinterpret_cast<const uint4 *>(w.cand_list) + f);
            r.ij = v.x;
            r.mask = v.y;
            r.e = (int)v.z;
            r.hstart = (int)v.w;
            return r;
        }
        int b = 0;   // the last chunk of bands starting at or before f
#pragma unroll
        for (int d = kBandChunks / 2; d > 0; d >>= 1)
            if (coarse[b + d] <= f) b += d;
        int rem = f - coarse[b];
        for (b *= chunk;; b += 4) {   // four counts at a time; the walk ends inside the chunk
            int c[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) c[q] = b + q < w.n_band_lists ? __ldg(&w.band_counts[b + q]) : INT_MAX;
            if (rem < c[0]) break;
            rem -= c[0];
            if (rem < c[1]) { b += 1; break; }
            rem -= c[1];
            if (rem < c[2]) { b += 2; break; }
            rem -= c[2];
            if (rem < c[3]) { b += 3; break; }
            rem -= c[3];
        }
        const uint2 v = __ldg(&w.band_cands[(int64_t)b * w.band_cap + rem]);
        r.ij = v.x;
        r.mask = v.y;
        return r;
    };

    ListEntry next = fetch(first * C);
    for (int gq = first; gq * C < total; gq += step) {
        const int f0 = gq * C;
        const ListEntry rec = next;
        if ((gq + step) * C < total) next = fetch((gq + step) * C);
        // step 1: the range of the lane's (candidate, layer)
        const int i = (int)(rec.ij >> 16), j = (int)(rec.ij & 0xFFFFu);
        int st = 0, n0 = 0, len = 0, jump = 0;
        unsigned slot = (unsigned)lane;
        float g = 0.f;
        float4 zc = make_float4(0.f, 0.f, 0.f, 0.f);
        // (a count names no layers)
        if (lane_on && (((ax.counts && f0 + kc < total ? 0xFFFFu : rec.mask) & layers_present) >> l & 1u)) {
            const int32_t *offs = w.offs + (int64_t)rec.e * (nkeys + 1) + l * nphi;
            if (!GEN || !((layers_general >> l) & 1u)) {
                const TabEntry te = load_tab(&w.tab[l * ax.n_qpt + i]);
                zc = __ldg(&w.zco[l * ax.n_qpt + i]);
                if (te.I != kNoVote) {
                    const int J = wrap_col(j + te.I, nphi);   // |I| <= nphi / 4 + 1
                    const bool last = J + 1 == nphi;          // the second bucket is the layer's first
                    const int o0 = __ldg(&offs[J]), o1 = __ldg(&offs[J + 1]);
                    const int p0 = last ? __ldg(&offs[0]) : o1, p1 = __ldg(&offs[last ? 1 : J + 2]);
                    st = rec.hstart + o0;
                    n0 = o1 - o0;
                    len = n0 + (p1 - p0);
                    jump = p0 - o1;
                    g = te.g;
                }
            } else {
                int sts[2] = {0, 0}, ens[2] = {0, 0};
                const int nr = general_ranges(ax, w, w.offs + (int64_t)rec.e * (nkeys + 1), l, i, j, s32, sts, ens);
                st = rec.hstart + sts[0];
                n0 = ens[0] - sts[0];
                len = n0;
                if (nr > 1) {
                    jump = sts[1] - ens[0];
                    len += ens[1] - sts[1];
                }
                slot |= 32u;
            }
        }
        const int incl = warp_incl_scan(len);
        const int excl = incl - len;
        const int T = __shfl_sync(0xFFFFFFFFu, incl, 31);
        const unsigned ne = __ballot_sync(0xFFFFFFFFu, len > 0);
        __syncwarp();   // the last group's readers are done
        S.zco[lane] = zc;
        if (len > 0) {
            const int q = __popc(ne & lanes_below());
            S.seg[q] = make_int4(st - excl, excl + n0, __float_as_int(g), jump);
            S.seg_slot[q] = (unsigned char)slot;
        }
        const int my_start = len > 0 ? excl : INT_MAX;
        __syncwarp();

        // the hit at flattened index base + lane: its staged position, slot, g, f and whether that has
        // to lie below g
        auto locate = [&](int base, int &p, unsigned &sl, float &f, float &gq, bool &after) {
            const int qb = __popc(__ballot_sync(0xFFFFFFFFu, my_start <= base)) - 1;   // the range owning base
            const int d = my_start - base;
            const unsigned bits = __reduce_or_sync(0xFFFFFFFFu, (d > 0 && d < 32) ? 1u << d : 0u);
            const int q = qb + __popc(bits & upto);
            const int4 sg = S.seg[q];
            sl = S.seg_slot[q];
            const int idx = base + lane;
            after = idx >= sg.y;
            gq = __int_as_float(sg.z);
            p = sg.x + idx + (after ? sg.w : 0);
            f = idx < T ? __ldg(&w.fsort[p]) : 0.f;
        };
        auto is_member = [&](int base, int p, unsigned sl, float f, float gq, bool after) {
            bool mem = (f < gq) == after;
            if (GEN) {
                const unsigned ij = __shfl_sync(0xFFFFFFFFu, rec.ij, (int)(sl & 31u));
                if (base + lane < T && (sl & 32u))
                    mem = general_member(ax, w, w.hot, w.cold, p, (int)(ij >> 16), (int)(ij & 0xFFFFu), s32, refine_eps);
            }
            return mem && base + lane < T;
        };

        // member lists of a context: a pool slot per candidate, reserved once its members are counted
        // (lane k holds candidate k's count, base and entries written; in a team, lane 0 the warp's
        // own part of them)
        int cnt = 0, pool_base = 0, pool_n = 0;
        auto count_window = [&](bool mem, unsigned sl) {
            const int kq = (int)(sl & 31u) / NL;
            for (int k = 0; k < C; ++k) {
                const int c = __popc(__ballot_sync(0xFFFFFFFFu, mem && kq == k));
                if (lane == k) cnt += c;
            }
        };
        auto reserve = [&]() {
            if (TEAM) {
                if (lane == 0) team->members[wpos] = cnt;
                __syncthreads();
                int before = 0, all = 0;
#pragma unroll
                for (int k = 0; k < kWarps; ++k) {
                    before += k < wpos ? team->members[k] : 0;
                    all += team->members[k];
                }
                if (threadIdx.x == 0) {
                    const unsigned reserved = all ? atomicAdd(&w.stats[0].pool_used, (unsigned)all) : 0u;
                    const long long room = (long long)w.max_members - (long long)reserved;
                    team->pool_base = (int)min((long long)reserved, (long long)w.max_members);
                    team->pool_n = all ? (int)max(0LL, min((long long)all, room)) : 0;
                    w.mem_start[f0] = team->pool_base;
                    w.mem_count[f0] = team->pool_n;
                }
                __syncthreads();
                pool_base = team->pool_base + before;
                pool_n = max(0, team->pool_n - before);
            } else if (lane < C && f0 + lane < total) {
                const unsigned reserved = cnt ? atomicAdd(&w.stats[0].pool_used, (unsigned)cnt) : 0u;
                const long long room = (long long)w.max_members - (long long)reserved;
                pool_base = (int)min((long long)reserved, (long long)w.max_members);
                pool_n = cnt ? (int)max(0LL, min((long long)cnt, room)) : 0;
                w.mem_start[f0 + lane] = pool_base;
                w.mem_count[f0 + lane] = pool_n;
            }
        };
        // the candidate being voted: its best key and members so far
        int cur = 0;
        unsigned best = 0u;
        int n_members = 0;
        // the record of the lane's candidate, kept by the lanes of its first layer
        unsigned r_best = 0u, r_mask2 = 0u;
        int r_members = 0;
        const bool one_event = __all_sync(0xFFFFFFFFu, rec.e == acc_e || rec.mask == 0u);
        // step 5
        auto finish = [&]() {
            best = __reduce_max_sync(0xFFFFFFFFu, best);
            acc_members += (unsigned)n_members;
            if (TEAM) {
                if (lane == 0) {
                    team->best[wpos] = best;
                    team->members[wpos] = n_members;
                }
                __syncthreads();   // every vote has landed
                n_members = 0;
#pragma unroll
                for (int k = 0; k < kWarps; ++k) {
                    best = max(best, team->best[k]);
                    n_members += team->members[k];
                }
            } else {
                __syncwarp();   // every vote has landed
            }
            uint32_t mask2 = 0u;
            if (best) {
                mask2 = grid_mask<P10>(grid, 0xFFFFu - (best & 0xFFFFu));
                if (TEAM) __syncthreads(); else __syncwarp();   // read before the clear
                uint4 *g4 = reinterpret_cast<uint4 *>(grid) + lane;
                if (TEAM) {
                    for (int q = threadIdx.x; q < grid_vecs; q += 32 * kWarps)
                        reinterpret_cast<uint4 *>(grid)[q] = make_uint4(0u, 0u, 0u, 0u);
                } else if (G64) {
                    constexpr int kVecs = ((P10 ? (64 * 64 + 2) / 3 : 64 * 64 / 2) + 3) / 4;
#pragma unroll
                    for (int q = 0; q < kVecs; q += 32)
                        if (q + 32 <= kVecs || lane < kVecs - q) g4[q] = make_uint4(0u, 0u, 0u, 0u);
                } else {
#pragma unroll 1
                    for (int q = lane; q < grid_vecs; q += 32, g4 += 32) *g4 = make_uint4(0u, 0u, 0u, 0u);
                }
            }
            if (lane == cur * NL) {
                r_best = best;
                r_mask2 = mask2;
                r_members = n_members;
            }
            ++cur;
            best = 0u;
            n_members = 0;
            if (TEAM) __syncthreads(); else __syncwarp();   // the grid is clear
        };

        // step 2: the members among the hits at base + lane, listed behind the nm there are; a lane's
        // place in the list is given by ballots
        int nm = 0;
        auto append = [&](bool mem, int p, unsigned sl) {
            const unsigned b = __ballot_sync(0xFFFFFFFFu, mem);
            if (mem) {
                const int r = nm + __popc(b & lanes_below());
                S.list_p[r] = p;
                S.list_slot[r] = (unsigned char)sl;
            }
            nm += __popc(b);
        };
        // the first windows' loads are all in flight before the first test
        int h = 32 * wpos;   // the next window's first hit
        {
            int p[kListCap / 32];
            unsigned sl[kListCap / 32];
            float f[kListCap / 32], gq[kListCap / 32];
            bool after[kListCap / 32];
#pragma unroll
            for (int u = 0; u < kListCap / 32; ++u)
                if (h + 32 * TW * u < T) locate(h + 32 * TW * u, p[u], sl[u], f[u], gq[u], after[u]);
#pragma unroll
            for (int u = 0; u < kListCap / 32; ++u) {
                if (h + 32 * TW * u < T) {
                    const bool mem = is_member(h + 32 * TW * u, p[u], sl[u], f[u], gq[u], after[u]);
                    append(mem, p[u], sl[u]);
                    if (KEEP) count_window(mem, sl[u]);
                }
            }
            h += 32 * TW * (kListCap / 32);
        }
        bool counting = KEEP;   // windows from here on are counted as they are first tested
        for (;;) {
            // more windows while the list has room for one
            while (h < T && nm <= kListCap - 32) {
                int p;
                unsigned sl;
                float f, gq;
                bool after;
                locate(h, p, sl, f, gq, after);
                const bool mem = is_member(h, p, sl, f, gq, after);
                append(mem, p, sl);
                if (KEEP && counting) count_window(mem, sl);
                h += 32 * TW;
            }
            if (KEEP && counting) {
                // the members of the windows that wait for the list, then the candidates' pool slots
                for (int base = h; base < T; base += 32 * TW) {
                    int p;
                    unsigned sl;
                    float f, gq;
                    bool after;
                    locate(base, p, sl, f, gq, after);
                    count_window(is_member(base, p, sl, f, gq, after), sl);
                }
                reserve();
                counting = false;
            }
            __syncwarp();   // the list is complete
            for (int r0 = 0; r0 < nm; r0 += 32) {
                // step 3: coefficients and run of each of the round's members (a lane past the list
                // repeats an entry and is dropped)
                const int nr = min(32, nm - r0);
                const bool valid = lane < nr;
                const int at = r0 + min(lane, nr - 1);
                const int p = S.list_p[at];
                const unsigned sl = S.list_slot[at];
                const float z = __ldg(&w.zsort[p]);
                const int slot_r = (int)(sl & 31u);
                const int k_r = slot_r / NL, l_r = slot_r - k_r * NL;
                const float4 zcr = S.zco[slot_r];
                float rb = zcr.z > 0.f ? __fdividef(1.f, zcr.z) : 0.f;   // approximate suffices
                float a, b, mref, lo;
                int len_r;
                table_coefficients(ax, zcr, rb, z, &a, &b, &mref);
                if (GEN) {
                    const int i_r = (int)(__shfl_sync(0xFFFFFFFFu, rec.ij, slot_r) >> 16);
                    if (sl & 32u) {
                        exact_coefficients(ax, i_r, w.cold[p], &a, &b, &mref);
                        rb = b > 0.f ? __frcp_rn(b) : 0.f;
                    }
                }
                member_run(n_cotf, n_z0f, a, b, rb, mref, &lo, &len_r);
                if (!valid) len_r = 0;
                const int incl_r = warp_incl_scan(len_r);
                const int st_r = incl_r - len_r;
                const unsigned bkeep = __ballot_sync(0xFFFFFFFFu, len_r > 0);
                const int last_word = (__shfl_sync(0xFFFFFFFFu, incl_r, 31) >> 5) + 1;
                if (lane <= last_word) starts[lane] = 0u;
#pragma unroll 1
                for (int q = lane + 32; q <= last_word; q += 32) starts[q] = 0u;
                __syncwarp();
                if (len_r > 0) {
                    const float c0 = lo - (float)st_r;
                    S.par[__popc(bkeep & lanes_below())] = make_int4(
                        __float_as_int(a), __float_as_int(b), __float_as_int(c0 - mref), (((int)c0 * n_z0) << 5) | l_r);
                    atomicOr(&starts[st_r >> 5], 1u << (st_r & 31));
                }
                __syncwarp();
                // step 4, a candidate's members at a time
                for (int s0 = 0; s0 < nr;) {
                    const int k = __shfl_sync(0xFFFFFFFFu, k_r, s0);
                    const int s1 = s0 + __popc(__ballot_sync(0xFFFFFFFFu, valid && k_r == k));
                    while (cur < k) finish();
                    if (!one_event) {
                        const int e = __shfl_sync(0xFFFFFFFFu, rec.e, k * NL);
                        if (e != acc_e) flush(e);
                    }
                    if (KEEP) {
                        const int base = __shfl_sync(0xFFFFFFFFu, pool_base, k), n = __shfl_sync(0xFFFFFFFFu, pool_n, k);
                        const int r = n_members + lane - s0;   // the member's rank among its candidate's
                        if (lane >= s0 && lane < s1 && r < n) w.mem_pool[base + r] = p;
                    }
                    n_members += s1 - s0;
                    const int v0 = __shfl_sync(0xFFFFFFFFu, st_r, s0), v1 = __shfl_sync(0xFFFFFFFFu, incl_r, s1 - 1);
                    // owner of a pair: the kept members before the candidate's, plus the runs starting at
                    // or before the pair, less one
                    const int4 *owner0 = S.par + (__popc(bkeep & ((1u << s0) - 1u)) - 1);
                    const unsigned *sw = starts + (v0 >> 5);
                    float row = (float)(v0 + lane);
                    unsigned cv = (unsigned)((v0 + lane) * n_z0);
                    unsigned word0 = *sw;
#pragma unroll 1
                    for (int left = v1 - v0 - lane; left > -lane; left -= 32) {   // (left + lane: the pairs to go)
                        const unsigned word1 = *++sw;
                        const unsigned bits = __funnelshift_r(word0, word1, v0);
                        word0 = word1;
                        const int4 pr = owner0[__popc(bits & upto)];
                        owner0 += __popc(bits);
                        // w(m) at the pair's row; its floor from the sum with 2^23 rounded down: below 0 that
                        // falls under the bits of 2^23, above n_z0 it stays above n_z0
                        const float wv = fmaf(-(row + __int_as_float(pr.z)), __int_as_float(pr.y), __int_as_float(pr.x));
                        const unsigned n = (unsigned)__float_as_int(__fadd_rd(wv, 8388608.f)) - 0x4B000000u;
                        const unsigned cell = cv + (unsigned)(pr.w >> 5) + n;
                        const unsigned word = P10 ? __umulhi(cell, 0x55555556u) : cell >> 1;   // cell < 2^15: cell / 3
                        const unsigned shift = P10 ? cell * 10u - word * 30u : (cell & 1u) << 4;
                        const unsigned bit = __funnelshift_l(0u, 1u, pr.w);   // 1 << (pr.w & 31)
                        // the vote and its judgement, predicated on the pair being in range
                        asm volatile(
                            "{\n\t.reg .pred p;\n\t.reg .b32 o, k;\n\t"
                            "setp.lt.u32 p, %2, %3;\n\t"
                            "setp.gt.and.s32 p, %4, 0, p;\n\t"
                            "@p atom.shared.or.b32 o, [%5], %6;\n\t"
                            "shr.u32 o, o, %7;\n\t"
                            "lop3.b32 o, o, %8, %9, 0xEA;\n\t"   // (o & field) | bit
                            "popc.b32 k, o;\n\t"
                            "mad.lo.u32 k, k, 65536, %10;\n\t"
                            "@p max.u32 %0, %0, k;\n\t"
                            "@p add.u32 %1, %1, 1;\n\t}"
                            : "+r"(best), "+r"(acc_votes)
                            : "r"(n), "r"(n_z0), "r"(left), "r"(grid_s + word * 4u), "r"(bit << shift), "r"(shift),
                              "r"(P10 ? 0x3FFu : 0xFFFFu), "r"(bit), "r"(0xFFFFu - cell)
                            : "memory");
                        row += 32.f;
                        cv += 32u * (unsigned)n_z0;
                    }
                    s0 = s1;
                }
                __syncwarp();   // the round's entries are read before the next one's are written
            }
            if (h >= T) break;
            nm = 0;
        }
        const int nc = min(C, total - f0);
        while (cur < nc) finish();
        const int written = !KEEP ? r_members : TEAM ? team->pool_n : __shfl_sync(0xFFFFFFFFu, pool_n, kc);
        if (l == 0 && kc < nc && wpos == 0) {
            const unsigned cell = r_best ? 0xFFFFu - (r_best & 0xFFFFu) : 0u;
            // cell / n_z0: cell < 2^14 and n_z0 <= 256, so the quotient of the half-shifted cell stays
            // far enough from a whole number for its roundings
            const unsigned icot = G64 ? cell >> 6 : (unsigned)(((float)cell + 0.5f) * __frcp_rn(n_z0f));
            hough_candidate out;
            out.iq = (unsigned)i;
            out.jphi = (unsigned)j;
            out.mask = rec.mask;
            out.n_members = (uint32_t)r_members;
            out.icot = icot;
            out.jz0 = cell - icot * (unsigned)n_z0;
            out.mask2 = r_mask2;
            out.flags = ((int)(r_best >> 16) >= min(ax.threshold, ax.n_layers) ? 1u : 0u) | (written < r_members ? 2u : 0u);
            store_candidate(w.cands + f0 + kc, out);
            if (KEEP && f0 + kc < w.out_limit) store_candidate(w.out_cands + f0 + kc, out);
        }
    }
    flush(0);
}

// Membership and stage 2 of every candidate of every event.  EVENT: one event of a context, whose few
// candidates are each shared by a CTA's warps.
template <int NL, bool P10, bool G64, bool EVENT>
__global__ void __launch_bounds__(32 * kWarps, P10 && !EVENT ? 7 : 5)
    confirm_kernel(Axes ax, Workspace w, float s32, float refine_eps, int grid_words, int start_words, int group_warps,
                   int chunk)
{
    pdl_enter();
    extern __shared__ __align__(16) unsigned char smem_c[];
    __shared__ int s_coarse[kBandChunks + 1];
    __shared__ Team s_team;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // the layer records, one a lane
    LayerInfo li{};
    if (lane < ax.n_layers) li = w.info[lane];
    const unsigned present = __ballot_sync(0xFFFFFFFFu, lane < ax.n_layers && li.present);
    const unsigned general = __ballot_sync(0xFFFFFFFFu, lane < ax.n_layers && li.present && !li.uniform);
    // one event of a context whose candidate list was not compacted: every CTA scans the band counts
    // and reads its candidates from the band lists; the first CTA records the totals the compaction
    // would have
    int total;
    const int *coarse = nullptr;
    if (EVENT && w.cands_from_bands) {
        const int found = scan_bands(w.band_counts, w.n_band_lists, chunk, s_coarse);
        total = min(found, w.max_cand);
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            w.stats[0].n_candidates = (unsigned)found;
            if (found > w.max_cand) atomicOr(&w.stats[0].device_error, HOUGH_DEVERR_CAND);
            w.cand_base[0] = 0;
            w.cand_base[1] = total;
            w.counters->total_cands = (unsigned)total;
        }
        coarse = s_coarse;
    } else {
        total = (int)w.counters->total_cands;
    }
    const size_t scratch = sizeof(Scratch) + (size_t)start_words * 4;
    int workers = 1;   // CTAs with candidates
    if (EVENT && total <= kTeamRounds * (int)gridDim.x) {
        workers = max(1, min((int)gridDim.x, total));
        if ((int)blockIdx.x < total) {
            Scratch &S = *reinterpret_cast<Scratch *>(smem_c + warp * scratch);
            unsigned *starts = reinterpret_cast<unsigned *>(&S + 1);
            uint32_t *grid = reinterpret_cast<uint32_t *>(smem_c + kWarps * scratch);
            for (int q = threadIdx.x; q < grid_words >> 2; q += 32 * kWarps)
                reinterpret_cast<uint4 *>(grid)[q] = make_uint4(0u, 0u, 0u, 0u);
            __syncthreads();
            if (general)
                confirm_groups<NL, P10, G64, true, true, true>(ax, w, s32, refine_eps, S, &s_team, starts, grid, grid_words >> 2,
                                                               present, general, 1, blockIdx.x, gridDim.x, total, coarse, chunk);
            else
                confirm_groups<NL, P10, G64, false, true, true>(ax, w, s32, refine_eps, S, &s_team, starts, grid,
                                                                grid_words >> 2, present, 0u, 1, blockIdx.x, gridDim.x, total,
                                                                coarse, chunk);
        }
    } else {
        // candidates per warp: as many as its lanes hold, fewer when that would leave warps without any;
        // group q goes to CTA q mod gridDim, so that a few candidates spread over all SMs
        const int nwarps = group_warps * gridDim.x;
        const int C = max(1, min(32 / NL, total / nwarps));
        const int first = warp * gridDim.x + blockIdx.x;
        workers = max(1, min((int)gridDim.x, (total + C - 1) / C));
        if (warp < group_warps && (int64_t)first * C < total) {
            Scratch &S = *reinterpret_cast<Scratch *>(smem_c + warp * (scratch + (size_t)grid_words * 4));
            unsigned *starts = reinterpret_cast<unsigned *>(&S + 1);
            uint32_t *grid = starts + start_words;
            for (int q = lane; q < grid_words >> 2; q += 32) reinterpret_cast<uint4 *>(grid)[q] = make_uint4(0u, 0u, 0u, 0u);
            __syncwarp();
            if (general)
                confirm_groups<NL, P10, G64, true, EVENT, false>(ax, w, s32, refine_eps, S, nullptr, starts, grid,
                                                                 grid_words >> 2, present, general, C, first, nwarps, total,
                                                                 coarse, chunk);
            else
                confirm_groups<NL, P10, G64, false, EVENT, false>(ax, w, s32, refine_eps, S, nullptr, starts, grid,
                                                                  grid_words >> 2, present, 0u, C, first, nwarps, total, coarse,
                                                                  chunk);
        }
    }
    if (!EVENT || !w.out_stats || (int)blockIdx.x >= workers) return;
    // the CTA that finishes last of those with candidates (the first, if there are none) reports the
    // event's counters, complete by then
    __shared__ int s_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(&w.counters->confirms_done, 1u) == (unsigned)workers - 1u;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    static_assert(sizeof(DevStats) % 4 == 0, "the counters are copied as 32-bit words");
    for (int q = threadIdx.x; q < (int)(sizeof(DevStats) / 4); q += blockDim.x)
        reinterpret_cast<uint32_t *>(w.out_stats)[q] = __ldcg(reinterpret_cast<const uint32_t *>(w.stats) + q);
    if (threadIdx.x == 0) w.counters->confirms_done = 0u;   // ready for the next event
}

__global__ void member_index_kernel(Workspace w, int32_t *idx_out, int64_t total)
{
    pdl_enter();
    const int32_t *isort = w.isort + w.hit_start[0];
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < total; q += (int64_t)gridDim.x * blockDim.x)
        idx_out[q] = isort[w.mem_pool[q]];
}

// Words of a grid of 16-bit masks, two to a word, or of 10-bit masks, three to a word, rounded up
// to whole 16-byte vectors.
int grid_words_for(const Axes &ax, bool p10)
{
    const int cells = ax.n_cot * ax.n_z0;
    return ((p10 ? (cells + 2) / 3 : (cells + 1) / 2) + 3) & ~3;
}

// Resident CTAs per SM of a kernel at a block size and dynamic shared-memory size, asked once per
// pair (the answer depends on the kernel and the device only; the library drives one device model).
template <typename K>
int resident_ctas(K kernel, int threads, size_t smem, std::atomic<unsigned long long> &memo)
{
    const unsigned long long key = (unsigned long long)smem | ((unsigned long long)threads << 20);
    const unsigned long long m = memo.load(std::memory_order_relaxed);
    if (m && (m >> 32) == key) return (int)(m & 0xFFFFFFFFull);
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, threads, smem) != cudaSuccess || n < 1) n = 1;
    memo.store((key << 32) | (unsigned)n, std::memory_order_relaxed);
    return n;
}

std::atomic<unsigned long long> g_ctas[8];
std::atomic<int> g_smem_optin{-1};

int smem_optin()
{
    int m = g_smem_optin.load(std::memory_order_relaxed);
    if (m < 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        if (cudaDeviceGetAttribute(&m, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) m = 48 * 1024;
        g_smem_optin.store(m, std::memory_order_relaxed);
    }
    return m;
}

template <int NL, bool P10, bool G64, bool EVENT>
cudaError_t launch_confirm(const Axes &ax, const Workspace &w, int sms, float s32, float refine_eps,
                           cudaStream_t stream, std::atomic<unsigned long long> &memo)
{
    auto kernel = confirm_kernel<NL, P10, G64, EVENT>;
    const int words = grid_words_for(ax, P10);
    const int start_words = (ax.n_cot + 2 + 3) & ~3;   // 32 members' runs of at most n_cot rows
    const size_t scratch = sizeof(Scratch) + (size_t)start_words * 4, grid = (size_t)words * 4;
    // as many warps with a grid of their own per CTA (up to kWarps) as shared memory holds
    const int room = smem_optin() - 2048;
    const int warps = std::max(1, std::min(kWarps, room / (int)(scratch + grid)));
    const size_t smem = std::max((size_t)warps * (scratch + grid), EVENT ? kWarps * scratch + grid : (size_t)0);
    cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (!err) err = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                         cudaSharedmemCarveoutMaxShared);
    if (err) return err;
    const int threads = 32 * (EVENT ? kWarps : warps);
    const int ctas = resident_ctas(kernel, threads, smem, memo);
    const int chunk = (n_bands(ax, w.band_rows) + kBandChunks - 1) / kBandChunks;
    // the number of candidates is known on the device only: a persistent grid of exactly the
    // resident CTAs, each warp striding over the flattened list
    return launch_chained(kernel, dim3(ctas * sms), dim3(threads), smem, stream, ax, w, s32, refine_eps, words,
                          start_words, warps, chunk);
}

template <bool EVENT>
cudaError_t launch_confirm_for(const Axes &ax, const Workspace &w, int sms, float refine_eps, cudaStream_t stream)
{
    const float s32 = (float)(ax.n_phi * kInvTwoPi);
    std::atomic<unsigned long long> *memo = g_ctas + (EVENT ? 4 : 0);
    // at most 10 layers: 10 lanes a candidate, the grid's masks packed three to a word
    const bool g64 = ax.n_cot == 64 && ax.n_z0 == 64;
    if (ax.n_layers <= 10)
        return g64 ? launch_confirm<10, true, true, EVENT>(ax, w, sms, s32, refine_eps, stream, memo[0])
                   : launch_confirm<10, true, false, EVENT>(ax, w, sms, s32, refine_eps, stream, memo[1]);
    return g64 ? launch_confirm<16, false, true, EVENT>(ax, w, sms, s32, refine_eps, stream, memo[2])
               : launch_confirm<16, false, false, EVENT>(ax, w, sms, s32, refine_eps, stream, memo[3]);
}

}  // namespace

size_t stage2_smem_bytes(const Axes &ax) { return (size_t)grid_words_for(ax, false) * 4; }

bool stage2_reads_bands(const Axes &ax, int band_rows) { return n_bands(ax, band_rows) <= kMaxBandsRead; }

cudaError_t launch_stage2(const Axes &ax, const Workspace &w, int sms, float refine_eps, cudaStream_t stream,
                          cudaEvent_t between)
{
    if (w.keep_members && w.n_events != 1) return cudaErrorInvalidValue;   // only single events keep member lists
    cudaError_t err = w.keep_members ? launch_confirm_for<true>(ax, w, sms, refine_eps, stream)
                                     : launch_confirm_for<false>(ax, w, sms, refine_eps, stream);
    if (err) return err;
    if (between && (err = cudaEventRecord(between, stream))) return err;
    return cudaSuccess;
}

cudaError_t launch_member_index(const Workspace &w, int32_t *idx_out, int64_t total, cudaStream_t stream)
{
    if (total <= 0) return cudaSuccess;
    const int g = (int)min((total + 255) / 256, (int64_t)4096);
    cudaError_t err = launch_chained(member_index_kernel, dim3(g), dim3(256), 0, stream, w, idx_out, total);
    if (err) return err;
    return cudaGetLastError();
}

}  // namespace hough
