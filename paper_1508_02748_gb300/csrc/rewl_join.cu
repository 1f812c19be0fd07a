// Final merge, join and normalisation of librewl, all in FP64 on the device
// (arXiv:1508.02748, Sec. 2, Eqs. 3-4):
//   1. each window's walkers are merged: every walker is shifted by the mean,
//      over the bins all walkers of the window visited, of its difference to
//      walker 0; each bin is the mean over the walkers that visited it;
//   2. within each row of windows (same M range), pieces are joined along E:
//      g(E) = sum_M g(E,M) (Eq. 3) of each piece, beta(E) = d ln g / dE as the
//      forward difference over one bin (dE = 4), E_mat = the overlap bin with
//      minimal |beta_i - beta_j| (lowest on ties, never below the previous
//      matching point), piece j rescaled to agree with piece i at E_mat, and
//      piece i used for E < E_mat, piece j for E >= E_mat (Eq. 4);
//   3. the rows are joined along M by the same rule on g(M) = sum_E g(E,M)
//      (dM = 2), "one at a time" as Sec. 2 prescribes for both axes split;
//   4. the joined table is shifted so that sum g = 2^N.
// The sums run in a fixed order (lanes, then warps, then blocks), so a join of
// the same tables gives the same bits; results differ from a serial evaluation
// by the rounding of exp/log and of the sums.
#include <math.h>

#include <algorithm>

#include <math_constants.h>

#include "rewl_tab.cuh"

namespace rewl {

namespace {

// One walker's table entries by format.  ln g = base + max(H, 0) ln f in the
// exact formats (a caller's plain table is read with ln f = 0); REWL_F32 holds
// ln g itself, and its H only says which bins were visited.
template <int PREC>
__device__ __forceinline__ const typename tab::Tab<PREC>::Elem *table_of(const Params &p)
{
    using Elem = typename tab::Tab<PREC>::Elem;
    if constexpr (PREC == REWL_FP64) return reinterpret_cast<const Elem *>(p.lng);
    else if constexpr (PREC == REWL_F32X2) return reinterpret_cast<const Elem *>(p.lng2);
    else return reinterpret_cast<const Elem *>(p.lng1);
}

// Two adjacent entries from an even one on can be read at once (a caller's
// unpadded tables may start anywhere).
template <int PREC>
__device__ __forceinline__ bool pairs_aligned(const Params &p)
{
    return (p.tstride & 1) == 0 && ((uintptr_t)table_of<PREC>(p) & 15) == 0 && ((uintptr_t)p.H & 7) == 0;
}

// Terms of a sum of exp(v - max) this far below the largest (e^-60 < 1e-26)
// are left out: all (N+1)^2 of them together stay below 2e-19 of the sum, a
// thousandth of its rounding.  Most bins of a window are that far down.
constexpr double LSE_FAR = 60.0;

__device__ __forceinline__ double warp_sum(double v)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}

// Sums of exp(v - top) find the top, the largest value, by integers (an FP64
// comparison occupies its pipe like an addition does): the bits of a double,
// the negative ones' flipped but for the sign, order like the value, and a
// value's rank is how far it lies below +infinity in that order.  All 64 bits
// count: a top that misses the largest value by a part in 2^20 lets exp overflow
// from ln g = 2^30 on, and cuts all terms off below -2^26.  What is not a number
// ranks behind -infinity, so that it is never the top.
typedef unsigned long long Rank;
constexpr Rank RANK_NONE = 0xFFE0000000000001ull;              // of -infinity

__device__ __forceinline__ int order_of(double v)              // of the upper word alone
{
    const int h = __double2hiint(v);
    return h ^ ((h >> 31) & 0x7FFFFFFF);
}

__device__ __forceinline__ Rank rank_of(double v)
{
    const unsigned lo = (unsigned)__double2loint(v) ^ (unsigned)(__double2hiint(v) >> 31);
    return 0x7FF0000000000000ull - ((Rank)(unsigned)order_of(v) << 32 | lo);
}

__device__ __forceinline__ double value_of(Rank r)
{
    const Rank k = 0x7FF0000000000000ull - r;
    const int h = (int)(k >> 32);
    return __hiloint2double(h ^ ((h >> 31) & 0x7FFFFFFF), (int)((unsigned)k ^ (unsigned)(h >> 31)));
}

__device__ __forceinline__ Rank warp_first(Rank r)
{
    const unsigned h = (unsigned)(r >> 32), m = __reduce_min_sync(0xFFFFFFFFu, h);
    return (Rank)m << 32 | __reduce_min_sync(0xFFFFFFFFu, h == m ? (unsigned)r : 0xFFFFFFFFu);
}

// The upper words tell which terms are certainly LSE_FAR below the top, `far`
// the order of top - LSE_FAR; what is not a number counts as a term.
__device__ __forceinline__ bool counts(double v, int far)
{
    constexpr unsigned none = 0xFFF00000u ^ 0x7FFFFFFFu;       // of -infinity
    return (unsigned)order_of(v) - none >= (unsigned)far - none;
}

// ln sum_i exp(v[i]) over the finite v[0..n) by one warp: the top, then the
// sum in a fixed order (lane by lane, then the lanes).
__device__ __forceinline__ double lse_warp(const double *v, int n)
{
    const int lane = threadIdx.x & 31;
    Rank first = RANK_NONE;
    for (int i = lane; i < n; i += 32) first = min(first, rank_of(v[i]));
    first = warp_first(first);
    if (first == RANK_NONE) return -INFINITY;
    const double top = value_of(first);
    const int far = order_of(top - LSE_FAR);
    double acc = 0.0;
    for (int i = lane; i < n; i += 32) {
        const double x = v[i];
        if (counts(x, far)) acc += exp(x - top);
    }
    return top + log(warp_sum(acc));
}

// Matching point (Eq. 4) between marginals Ga, Gb over [lo, hi], q >= floor:
// the overlap bin q minimising |beta_a(q) - beta_b(q)|, beta the forward
// difference over one bin divided by the bin step (a power of two, so its
// reciprocal divides exactly), taken only where both marginals are finite at q
// and q + 1; the lowest such q on ties.  Without any, the lowest q where both
// are finite; -1 if none.
// It is computed by a whole block (every thread calls it and gets the
// result): each thread scans a stride of q keeping its first minimum, and
// the (difference, q) pairs are reduced lexicographically, so the lowest q
// wins ties.
constexpr int MATCH_THREADS = 128;

// Lexicographic minimum of (d, q) over the block, d >= 0 by its bits (which
// order like the values), so that no comparison needs the FP64 pipe.
__device__ void block_min_pair(long long &d, int &q, long long *s_d, int *s_q)
{
    for (int o = 16; o > 0; o >>= 1) {
        const long long od = __shfl_xor_sync(0xFFFFFFFFu, d, o);
        const int oq = __shfl_xor_sync(0xFFFFFFFFu, q, o);
        if (od < d || (od == d && oq < q)) { d = od; q = oq; }
    }
    __syncthreads();
    if ((threadIdx.x & 31) == 0) { s_d[threadIdx.x >> 5] = d; s_q[threadIdx.x >> 5] = q; }
    __syncthreads();
    d = s_d[0];
    q = s_q[0];
    for (int k = 1; k < MATCH_THREADS / 32; ++k)
        if (s_d[k] < d || (s_d[k] == d && s_q[k] < q)) { d = s_d[k]; q = s_q[k]; }
}

// v is not -infinity (by its words: a 64-bit comparison of the bits becomes an
// FP64 one)
__device__ __forceinline__ bool some(double v)
{
    return __double2hiint(v) != (int)0xFFF00000 || __double2loint(v) != 0;
}

__device__ int match_point_block(const double *Ga, const double *Gb, int lo, int hi, int floor_p, double inv_step)
{
    __shared__ long long s_d[MATCH_THREADS / 32];
    __shared__ int s_q[MATCH_THREADS / 32];
    const long long none = 0x7FF0000000000000ll;        // +infinity
    const int start = lo > floor_p ? lo : floor_p;
    long long bestd = none;
    int best = 0x7FFFFFFF;
    for (int q = start + (int)threadIdx.x; q + 1 <= hi; q += MATCH_THREADS) {
        const double a0 = Ga[q], a1 = Ga[q + 1], b0 = Gb[q], b1 = Gb[q + 1];
        if (!some(a0) || !some(a1) || !some(b0) || !some(b1)) continue;
        const double ba = (a1 - a0) * inv_step;
        const double bb = (b1 - b0) * inv_step;
        // (the sign by an integer operation: fabs may make the bits of what is not
        // a number negative, and so the smallest)
        const double x = ba - bb;
        const long long d = (long long)(__double2hiint(x) & 0x7FFFFFFF) << 32 | (unsigned)__double2loint(x);
        if (d < bestd) { bestd = d; best = q; }
    }
    block_min_pair(bestd, best, s_d, s_q);
    if (best != 0x7FFFFFFF) return best;
    bestd = 0;
    best = 0x7FFFFFFF;
    for (int q = start + (int)threadIdx.x; q <= hi; q += MATCH_THREADS)
        if (some(Ga[q]) && some(Gb[q])) { best = q; break; }
    block_min_pair(bestd, best, s_d, s_q);
    return best == 0x7FFFFFFF ? -1 : best;
}

}  // namespace

// 1a. Offsets of each window's walkers relative to the first one taking part
// (walker join_exclude, if >= 0, is left out: the jackknife replicates): the
// mean of ln g_k - ln g_ref over the bins that all of them visited.
//
// Bounded by the FP64 pipe (two lanes an SM and cycle) and by HBM: the tables
// are read once and the visits twice (the second time from L2).  A block takes
// a chunk of a window's bins for all its walkers: which bins all walkers
// visited is found once per window (it was found again for each walker, W^2
// reads of H), then each warp takes walkers in turn and adds up base_k -
// base_ref, two FP64 operations a bin; the visits are added up as integers.
// Chunk sums are folded in chunk order.  L = 32, 2048 walkers (3.1 GB): 12.4
// -> 1.2 ms; L = 16, 256 walkers 0.85 -> 0.05 ms.
constexpr int OFF_THREADS = 256, OFF_BINS = 2048;

// Bins a chunk: all of a small window (its block then finishes the offsets),
// else as many as leave some six blocks for each SM, and at least 4 W (the
// chunk sums of a window take the place of at most its bins' entries).
int off_chunk(const Params &p)
{
    int chunk = OFF_BINS;
    if (p.T <= OFF_BINS) return chunk;
    while (chunk > 512 && (long long)(p.T / chunk) * p.nwin < 152 * 6) chunk /= 2;
    while (chunk < 4 * p.W) chunk *= 2;
    return chunk;
}

// Offset of walker k from its sum over the common bins, and the window's
// typical visit count of a bin (in efrom until 2b writes it), which 1b takes
// out of the walkers' visits to keep its sums small.
__device__ __forceinline__ double offset_of(const Params &p, int k, int ref, double sum, double common)
{
    if (k == ref || k == p.join_exclude) return 0.0;
    if (common == 0.0) { atomicExch(&p.st->join_error, 1); return 0.0; }
    return sum / common;
}

__device__ __forceinline__ int typical_visits(const Params &p, double common, double ref_visits)
{
    return common > 0.0 && p.precision != REWL_F32 ? (int)(ref_visits / common) : 0;
}

template <int PREC>
__global__ void __launch_bounds__(OFF_THREADS) k_off_part(Params p, JoinScratch j, int chunk, int nchunks)
{
    after_previous();
    using TB = tab::Tab<PREC>;
    using Elem = typename TB::Elem;
    const int win = blockIdx.y, c = blockIdx.x, W = p.W;
    if (!p.active[win]) return;
    const int ref = p.join_exclude == 0 ? 1 : 0;   // the first walker taking part
    __shared__ double s_ref[OFF_BINS];
    __shared__ int s_h[OFF_BINS];                  // the reference's visits
    __shared__ unsigned s_all[OFF_BINS / 32];      // bit: all walkers visited the bin
    __shared__ long long s_hits[OFF_THREADS / 32], s_href[OFF_THREADS / 32];
    __shared__ double s_common, s_visits, s_acc[OFF_THREADS / 32];
    const int share = W <= 2 ? 8 : W <= 4 ? 2 : 1;
    // per chunk W sums, then the number of common bins and the reference's
    // visits of them; several chunks leave them where 1b writes the piece (at
    // most half of its entries), a single one finishes the offsets itself
    const bool single = nchunks == 1;
    double *part = single ? j.off + (size_t)win * W : j.piece + (size_t)win * p.tstride + (size_t)c * (W + 2);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const Elem *B0 = table_of<PREC>(p) + (size_t)(win * W) * p.tstride;
    const int32_t *H0 = p.H + (size_t)(win * W) * p.tstride;
    long long hits = 0, href = 0;
    for (int at = c * chunk; at < min(p.T, (c + 1) * chunk); at += OFF_BINS) {
        const int n = min(OFF_BINS, min(p.T, (c + 1) * chunk) - at);
        __syncthreads();
        for (int b0 = 0; b0 < n; b0 += OFF_THREADS) {
            const int b = b0 + (int)threadIdx.x;
            int any = b < n ? 0 : -1;              // sign: some walker has not been there
            if (b < n) {
                #pragma unroll 8
                for (int k = 0; k < W; ++k)
                    if (k != p.join_exclude) any |= H0[(size_t)k * p.tstride + at + b];
                s_ref[b] = TB::exact(B0[(size_t)ref * p.tstride + at + b]);
                s_h[b] = H0[(size_t)ref * p.tstride + at + b];
            }
            const unsigned m = __ballot_sync(0xFFFFFFFFu, any >= 0);
            if (lane == 0) s_all[(b0 >> 5) + wid] = m;
            if (any >= 0) {
                ++hits;
                href += s_h[b];
            }
        }
        __syncthreads();
        // few walkers: `share` warps to each, every share-th 32 bins a warp
        const int turns = OFF_THREADS / 32 / share, mine = wid % share;
        for (int k0 = 0; k0 < W; k0 += turns) {
            const int k = k0 + wid / share;
            const bool on = k < W && k != ref && k != p.join_exclude;
            double acc = 0.0;
            if (on) {
                const Elem *B = B0 + (size_t)k * p.tstride + at;
                const int32_t *H = H0 + (size_t)k * p.tstride + at;
                long long hk = 0;
                #pragma unroll 4
                for (int b = lane + 32 * mine; b < n; b += 32 * share)
                    if ((s_all[b >> 5] >> lane) & 1u) {
                        acc += TB::exact(B[b]) - s_ref[b];
                        hk += H[b] - s_h[b];
                    }
                acc = warp_sum(acc);
                for (int o = 16; o > 0; o >>= 1) hk += __shfl_xor_sync(0xFFFFFFFFu, hk, o);
                if (PREC != REWL_F32) acc = fma((double)hk, p.st->lnf, acc);
            }
            if (share > 1) {
                if (lane == 0) s_acc[wid] = acc;
                __syncthreads();
                for (int q = 1; q < share; ++q) acc += s_acc[(wid / share) * share + q];
                __syncthreads();
            }
            if (on && lane == 0 && mine == 0) part[k] = at == c * chunk ? acc : part[k] + acc;
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        hits += __shfl_xor_sync(0xFFFFFFFFu, hits, o);
        href += __shfl_xor_sync(0xFFFFFFFFu, href, o);
    }
    if (lane == 0) { s_hits[wid] = hits; s_href[wid] = href; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < OFF_THREADS / 32; ++k) { hits += s_hits[k]; href += s_href[k]; }
        s_common = (double)hits;
        s_visits = (double)href;
        if (!single) { part[W] = s_common; part[W + 1] = s_visits; }
    }
    if (!single) return;
    __syncthreads();
    const double common = s_common, visits = s_visits;
    for (int k = threadIdx.x; k < W; k += OFF_THREADS)
        part[k] = offset_of(p, k, ref, part[k], common);
    if (threadIdx.x == 0) j.efrom[win] = typical_visits(p, common, visits);
}

// One block per window, one warp per walker in turn: the chunks' sums in a
// fixed order (lane by lane, then the lanes).
__global__ void __launch_bounds__(256) k_off_fold(Params p, JoinScratch j, int nchunks)
{
    after_previous();
    const int win = blockIdx.x, W = p.W, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (!p.active[win]) return;
    const int ref = p.join_exclude == 0 ? 1 : 0;
    const double *part = j.piece + (size_t)win * p.tstride;
    auto total = [&](int k) -> double {
        double v = 0.0;
        for (int c = lane; c < nchunks; c += 32) v += part[(size_t)c * (W + 2) + k];
        return warp_sum(v);
    };
    const double common = total(W);
    for (int k = wid; k < W; k += 8) {
        const double sum = k != ref && k != p.join_exclude ? total(k) : 0.0;
        if (lane == 0) j.off[(size_t)win * W + k] = offset_of(p, k, ref, sum, common);
    }
    if (wid == 0) {
        const double visits = total(W + 1);
        if (lane == 0) j.efrom[win] = typical_visits(p, common, visits);
    }
}

// 1b. Merged piece: the mean of ln g_k - off_k over the walkers that visited
// the bin, walkers in order; one thread per two bins of a window.
//
// Bounded by the FP64 pipe and HBM: base_k - off_k and its sum are two FP64
// operations an entry, the visits are summed as integers (less the window's
// typical count, whose ln g goes into the offset, so that neither sum grows
// beyond the spread of the values).  L = 32, 2048 walkers (3.1 GB): 1.41 -> 1.1
// ms (four FP64 operations an entry and one bin a thread before).
template <int PREC>
__global__ void __launch_bounds__(256) k_merge(Params p, JoinScratch j)
{
    after_previous();
    using TB = tab::Tab<PREC>;
    using Elem = typename TB::Elem;
    extern __shared__ double s_off[];
    const int win = blockIdx.y, W = p.W;
    const int b = 2 * (int)(blockIdx.x * blockDim.x + threadIdx.x);
    const bool act = p.active[win] != 0;
    double *out = j.piece + (size_t)win * p.tstride;
    const double lnf = PREC == REWL_F32 ? 0.0 : p.st->lnf;
    const int h0 = act && PREC != REWL_F32 ? j.efrom[win] : 0;
    if (act)
        for (int k = threadIdx.x; k < W; k += blockDim.x) s_off[k] = fma(-(double)h0, lnf, j.off[win * W + k]);
    __syncthreads();
    if (b >= p.T) return;
    const bool two = b + 1 < p.T;
    double a0 = 0.0, a1 = 0.0;
    int n0 = 0, n1 = 0;
    long long v0 = 0, v1 = 0;
    if (act) {
        const Elem *B = table_of<PREC>(p) + (size_t)(win * W) * p.tstride + b;
        const int32_t *H = p.H + (size_t)(win * W) * p.tstride + b;
        struct __align__(2 * sizeof(Elem)) Pair { Elem x, y; };
        const bool wide = pairs_aligned<PREC>(p);
        #pragma unroll 4
        for (int k = 0; k < W; ++k) {
            if (k == p.join_exclude) continue;
            const size_t q = (size_t)k * p.tstride;
            int hx, hy = -1;
            Elem x, y = Elem();
            if (wide && two) {
                const int2 h = *reinterpret_cast<const int2 *>(H + q);
                const Pair e = *reinterpret_cast<const Pair *>(B + q);
                hx = h.x; hy = h.y; x = e.x; y = e.y;
            } else {
                hx = H[q]; x = B[q];
                if (two) { hy = H[q + 1]; y = B[q + 1]; }
            }
            if (hx >= 0) { a0 += TB::exact(x) - s_off[k]; v0 += hx - h0; ++n0; }
            if (hy >= 0) { a1 += TB::exact(y) - s_off[k]; v1 += hy - h0; ++n1; }
        }
    }
    auto mean = [&](double a, long long v, int n) -> double {
        if (n == 0) return -INFINITY;
        if (PREC != REWL_F32) a = fma((double)v, lnf, a);
        if ((n & (n - 1)) == 0) return a * __hiloint2double((1023 - (31 - __clz(n))) << 20, 0);   // / 2^i
        return a / (double)n;
    };
    out[b] = mean(a0, v0, n0);
    if (two) out[b + 1] = mean(a1, v1, n1);
}

// 2a. E marginal of each piece over its M range (Eq. 3): one warp per
// (window, e).  (One thread each before: 514 -> 240 us at L = 32.)
__global__ void __launch_bounds__(256) k_marg_piece(Params p, JoinScratch j)
{
    after_previous();
    const int idx = (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5));
    if (idx >= p.nwin * p.wE) return;
    const int win = idx / p.wE, el = idx % p.wE;
    const double g = p.active[win] ? lse_warp(j.piece + (size_t)win * p.tstride + (size_t)el * p.wM, p.wM) : -INFINITY;
    if ((threadIdx.x & 31) == 0) j.GE[idx] = g;
}

// 2b. One block per row b: chain of E matching points along the row (the
// chain is sequential; each matching point and slice rule is block-parallel).
__global__ void __launch_bounds__(MATCH_THREADS) k_match_e(Params p, JoinScratch j)
{
    after_previous();
    const int b = blockIdx.x;
    if (b >= p.nM) return;
    const int nE = p.nE, t0 = threadIdx.x == 0;
    __shared__ int s_first, s_last, s_bad;
    if (t0) {
        for (int a = 0; a < nE; ++a) {
            j.efrom[b * nE + a] = 0; j.eto[b * nE + a] = 0; j.eshift[b * nE + a] = 0.0;
            if (a < nE - 1) j.ematch[b * (nE - 1) + a] = -1;
        }
        if (nE == 1) j.ematch[b] = -1;
        int first = -1, last = -1, bad = 0;
        for (int a = 0; a < nE; ++a)
            if (p.active[b * nE + a]) { if (first < 0) first = a; last = a; }
        j.rowok[b] = first >= 0;
        for (int a = first; first >= 0 && a <= last; ++a)
            if (!p.active[b * nE + a]) bad = 1;
        if (bad) atomicExch(&p.st->join_error, 2);
        s_first = first; s_last = last; s_bad = bad;
    }
    __syncthreads();
    const int first = s_first, last = s_last;
    if (first < 0 || s_bad) return;
    double shift = 0.0;
    if (p.join_rule == 1)
        for (int ml = threadIdx.x; ml < p.wM; ml += blockDim.x) j.eslice[(size_t)(b * nE + first) * p.wM + ml] = 0.0;
    int from = p.rect[b * nE + first].x;
    for (int a = first; a <= last; ++a) {
        const int A = b * nE + a;
        const int4 RA = p.rect[A];
        int to;
        double next_shift = 0.0;
        __syncthreads();                      // the last piece's buffers and slices are complete
        if (a < last) {
            const int4 RB = p.rect[A + 1];
            // the two marginals by absolute bin, read in the overlap [RB.x, RA.y] alone
            const double *Ga = j.GE + (ptrdiff_t)A * p.wE - RA.x, *Gb = j.GE + (ptrdiff_t)(A + 1) * p.wE - RB.x;
            const int q = match_point_block(Ga, Gb, RB.x, RA.y, from, 0.25);
            if (q < 0) { if (t0) atomicExch(&p.st->join_error, 3); return; }
            if (t0) j.ematch[b * (nE - 1) + a] = q;
            next_shift = shift + (Ga[q] - Gb[q]);
            if (p.join_rule == 1) {
                // the next piece's M slices: each matched at (E_mat, M) where
                // both pieces have the bin, else by the marginals
                const double *pa = j.piece + (size_t)A * p.tstride + (size_t)(q - RA.x) * p.wM;
                const double *pb = j.piece + (size_t)(A + 1) * p.tstride + (size_t)(q - RB.x) * p.wM;
                const double *sa = j.eslice + (size_t)A * p.wM;
                double *sb = j.eslice + (size_t)(A + 1) * p.wM;
                for (int ml = threadIdx.x; ml < p.wM; ml += blockDim.x) {
                    const double va = pa[ml], vb = pb[ml];
                    sb[ml] = sa[ml] + (some(va) && some(vb) ? va - vb : Ga[q] - Gb[q]);
                }
            }
            to = q;
        } else {
            to = RA.y + 1;
        }
        if (t0) { j.efrom[A] = from; j.eto[A] = to; j.eshift[A] = shift; }
        shift = next_shift;
        from = to;
    }
}

// Value of row b at (e, m): the piece covering e in that row, shifted.
__device__ __forceinline__ double row_value(const Params &p, const JoinScratch &j, int b, int e, int m)
{
    for (int a = 0; a < p.nE; ++a) {
        const int A = b * p.nE + a;
        if (e >= j.efrom[A] && e < j.eto[A]) {
            const int4 R = p.rect[A];
            if (m < R.z || m > R.w) return -INFINITY;
            const double v = j.piece[(size_t)A * p.tstride + (size_t)(e - R.x) * p.wM + (m - R.z)];
            const double c = p.join_rule == 1 ? j.eslice[(size_t)A * p.wM + (m - R.z)] : j.eshift[A];
            return some(v) ? v + c : v;
        }
    }
    return -INFINITY;
}

// 3a. M marginal of each row: F_b(m) = ln sum_E g_b(E, m).  A block takes
// ROW_COLS adjacent m of a row, its threads every ROW_ES-th e, piece by piece
// (the pieces tile the row, so no entry has to look for its piece); the threads'
// parts meet in shared memory.  Few columns a block: exp is FP64 work, which an
// SM does at two lanes a cycle, so it has to be spread over the SMs.  (One
// thread per m, all e twice, looking for each entry's piece before: 2.84 ->
// 0.12 ms at L = 32, 0.40 -> 0.02 ms at L = 16.)
constexpr int ROW_COLS = 8, ROW_ES = 32;

__global__ void __launch_bounds__(ROW_COLS * ROW_ES) k_marg_row(Params p, JoinScratch j)
{
    after_previous();
    const int B = p.N + 1, b = blockIdx.y, cx = threadIdx.x % ROW_COLS, ex = threadIdx.x / ROW_COLS;
    const int m = (int)blockIdx.x * ROW_COLS + cx;
    __shared__ double s_part[ROW_ES][ROW_COLS];
    const int4 R0 = p.rect[b * p.nE];              // the row's m range is its pieces'
    const bool in = j.rowok[b] && m >= R0.z && m <= R0.w;
    auto each = [&](auto f) {
        if (!in) return;
        for (int a = 0; a < p.nE; ++a) {
            const int A = b * p.nE + a, from = j.efrom[A], to = j.eto[A];
            const double *col = j.piece + (size_t)A * p.tstride + (m - R0.z);
            const int e0 = p.rect[A].x;
            const double c = p.join_rule == 1 && to > from ? j.eslice[(size_t)A * p.wM + (m - R0.z)] : j.eshift[A];
            if (isfinite(c)) {
                #pragma unroll 4
                for (int e = from + ex; e < to; e += ROW_ES) f(col[(size_t)(e - e0) * p.wM] + c);
            } else {                               // a bin without a visit stays one
                for (int e = from + ex; e < to; e += ROW_ES) {
                    const double v = col[(size_t)(e - e0) * p.wM];
                    f(some(v) ? v + c : v);
                }
            }
        }
    };
    __shared__ Rank s_top[ROW_ES][ROW_COLS];
    Rank first = RANK_NONE;
    each([&](double v) { first = min(first, rank_of(v)); });
    s_top[ex][cx] = first;
    __syncthreads();
    for (int k = 0; k < ROW_ES; ++k) first = min(first, s_top[k][cx]);
    const double top = value_of(first);
    double acc = 0.0;
    if (first != RANK_NONE) {
        const int far = order_of(top - LSE_FAR);
        each([&](double v) { if (counts(v, far)) acc += exp(v - top); });
    }
    s_part[ex][cx] = acc;
    __syncthreads();
    if (ex == 0 && m < B) {
        for (int k = 1; k < ROW_ES; ++k) acc += s_part[k][cx];
        j.F[(size_t)b * B + m] = first == RANK_NONE ? -INFINITY : top + log(acc);
    }
}

// 3b. One block: chain of M matching points over the rows (sequential
// chain, block-parallel matching point and slice rule).
__global__ void __launch_bounds__(MATCH_THREADS) k_match_m(Params p, JoinScratch j)
{
    after_previous();
    const int nM = p.nM, nE = p.nE, B = p.N + 1, t0 = threadIdx.x == 0;
    __shared__ int s_first, s_last, s_bad;
    if (t0) {
        for (int b = 0; b < nM; ++b) { j.mfrom[b] = 0; j.mto[b] = 0; j.mshift[b] = 0.0; }
        for (int b = 0; b < (nM > 1 ? nM - 1 : 1); ++b) j.mmatch[b] = -1;
        int first = -1, last = -1, bad = 0;
        for (int b = 0; b < nM; ++b) if (j.rowok[b]) { if (first < 0) first = b; last = b; }
        if (first < 0) { bad = 1; atomicExch(&p.st->join_error, 4); }
        for (int b = first; first >= 0 && b <= last; ++b) if (!j.rowok[b]) bad = 1;
        if (bad && first >= 0) atomicExch(&p.st->join_error, 5);
        s_first = first; s_last = last; s_bad = bad;
    }
    __syncthreads();
    const int first = s_first, last = s_last;
    if (s_bad) return;
    double shift = 0.0;
    if (p.join_rule == 1)
        for (int e = threadIdx.x; e < B; e += blockDim.x) j.mslice[(size_t)first * B + e] = 0.0;
    int from = p.rect[first * nE].z;
    for (int b = first; b <= last; ++b) {
        int to;
        double next_shift = 0.0;
        __syncthreads();                      // the last row's slices are complete
        if (b < last) {
            const double *Ga = j.F + (size_t)b * B, *Gb = j.F + (size_t)(b + 1) * B;
            const int lo = p.rect[(b + 1) * nE].z, hi = p.rect[b * nE].w;
            const int q = match_point_block(Ga, Gb, lo, hi, from, 0.5);
            if (q < 0) { if (t0) atomicExch(&p.st->join_error, 6); return; }
            if (t0) j.mmatch[b] = q;
            next_shift = shift + (Ga[q] - Gb[q]);
            if (p.join_rule == 1)
                for (int e = threadIdx.x; e < B; e += blockDim.x) {
                    const double va = row_value(p, j, b, e, q), vb = row_value(p, j, b + 1, e, q);
                    j.mslice[(size_t)(b + 1) * B + e] = j.mslice[(size_t)b * B + e]
                        + (some(va) && some(vb) ? va - vb : Ga[q] - Gb[q]);
                }
            to = q;
        } else {
            to = p.rect[b * nE].w + 1;
        }
        if (t0) { j.mfrom[b] = from; j.mto[b] = to; j.mshift[b] = shift; }
        shift = next_shift;
        from = to;
    }
}

// 3c. Assemble the joined table; each block leaves the rank of the largest value
// of its part in red[].
constexpr int RED_BLOCKS = 512;     // red[]: 512 maxima (their ranks), then from entry 512 on the sums

__global__ void __launch_bounds__(256) k_assemble(Params p, JoinScratch j)
{
    after_previous();
    const int B = p.N + 1;
    Rank first = RANK_NONE;
    for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < (size_t)B * B; idx += (size_t)gridDim.x * blockDim.x) {
        const int e = (int)(idx / B), m = (int)(idx % B);
        double v = -INFINITY;
        for (int b = 0; b < p.nM; ++b) {
            if (m >= j.mfrom[b] && m < j.mto[b]) {
                const double r = row_value(p, j, b, e, m);
                const double c = p.join_rule == 1 ? j.mslice[(size_t)b * B + e] : j.mshift[b];
                v = some(r) ? r + c : r;
                break;
            }
        }
        j.J[idx] = v;
        first = min(first, rank_of(v));
    }
    first = warp_first(first);
    __shared__ Rank s[8];
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = first;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < 8; ++k) first = min(first, s[k]);
        reinterpret_cast<Rank *>(j.red)[blockIdx.x] = first;
    }
}

// 4. Normalisation: sums of exp(v - max) by blocks, then the shift that makes
// sum g = 2^N.  Each block folds the blocks' maxima (sums) itself, all in the
// same order, instead of waiting for a kernel that does.
__device__ __forceinline__ Rank fold_max(const double *red, int n)
{
    __shared__ Rank s_m[8];
    Rank first = RANK_NONE;
    for (int k = threadIdx.x; k < n; k += 256) first = min(first, reinterpret_cast<const Rank *>(red)[k]);
    first = warp_first(first);
    if ((threadIdx.x & 31) == 0) s_m[threadIdx.x >> 5] = first;
    __syncthreads();
    for (int k = 0; k < 8; ++k) first = min(first, s_m[k]);
    return first;
}

__global__ void __launch_bounds__(256) k_red_sumexp(const double *v, size_t n, double *red, int nblk)
{
    after_previous();
    const Rank first = fold_max(red, nblk);
    const double top = value_of(first);
    double acc = 0.0;
    if (first != RANK_NONE) {
        const int far = order_of(top - LSE_FAR);
        for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
            const double x = v[i];
            if (counts(x, far)) acc += exp(x - top);
        }
    }
    acc = warp_sum(acc);
    __shared__ double s[8];
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < 8; ++k) acc += s[k];
        red[RED_BLOCKS + blockIdx.x] = acc;
    }
}

__global__ void __launch_bounds__(256) k_normalise(double *v, size_t n, const double *red, int nblk, int N)
{
    after_previous();
    const double top = value_of(fold_max(red, nblk));
    double acc = 0.0;
    for (int k = threadIdx.x; k < nblk; k += 256) acc += red[RED_BLOCKS + k];
    acc = warp_sum(acc);
    __shared__ double s[8], s_c;
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < 8; ++k) acc += s[k];
        s_c = (double)N * log(2.0) - (top + log(acc));
    }
    __syncthreads();
    const double c = s_c;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const double x = v[i];
        if (some(x)) v[i] = x + c;
    }
}

namespace {

// Warps a block of the kernels that take a row a warp: one while there is an SM
// for each row (their FP64 work is an SM's bottleneck), eight when there are many.
int row_warps(int rows) { return rows >= 152 * 8 ? 8 : rows >= 152 * 2 ? 2 : 1; }

// The windows lie along the grid's y, which ends at 65,535; there may be (N+1)^2
// of them, and those past a launch's are the first ones of the next.  (Windows
// along x or z cost the kernels a division or a product a block: L = 32's join
// 2.67 -> 2.69 ms.)
template <int PREC>
cudaError_t launch_merge(Params p, JoinScratch j, cudaStream_t s)
{
    const int chunk = off_chunk(p), nchunks = (p.T + chunk - 1) / chunk;
    for (int left = p.nwin; left > 0;) {
        const int n = std::min(left, 65535);
        cudaError_t e = launch_next(k_off_part<PREC>, dim3(nchunks, n), dim3(OFF_THREADS), 0, s, p, j, chunk, nchunks);
        if (e == cudaSuccess && nchunks > 1) e = launch_next(k_off_fold, dim3(n), dim3(256), 0, s, p, j, nchunks);
        if (e == cudaSuccess) e = launch_next(k_merge<PREC>, dim3((p.T + 511) / 512, n), dim3(256), sizeof(double) * p.W, s, p, j);
        if (e != cudaSuccess) return e;
        const size_t walkers = (size_t)n * p.W, entries = walkers * p.tstride;
        if (PREC == REWL_FP64) p.lng += entries;
        else if (PREC == REWL_F32X2) p.lng2 += entries;
        else p.lng1 += entries;
        p.H += entries;
        p.active += n;
        j.off += walkers;
        j.piece += (size_t)n * p.tstride;
        j.efrom += n;
        left -= n;
    }
    return cudaSuccess;
}

}  // namespace

// The first launch that fails ends the chain.
cudaError_t launch_join(const Params &p, const JoinScratch &j, cudaStream_t s)
{
    const int B = p.N + 1;
    cudaError_t e = p.precision == REWL_FP64 ? launch_merge<REWL_FP64>(p, j, s)
                  : p.precision == REWL_F32X2 ? launch_merge<REWL_F32X2>(p, j, s) : launch_merge<REWL_F32>(p, j, s);
    auto next = [&](auto kernel, dim3 grid, int threads, auto... args) {
        if (e == cudaSuccess) e = launch_next(kernel, grid, dim3(threads), 0, s, args...);
    };
    const int rows = p.nwin * p.wE, warps = row_warps(rows);
    next(k_marg_piece, dim3((rows + warps - 1) / warps), 32 * warps, p, j);
    next(k_match_e, dim3(p.nM), MATCH_THREADS, p, j);
    next(k_marg_row, dim3((B + ROW_COLS - 1) / ROW_COLS, p.nM), ROW_COLS * ROW_ES, p, j);
    next(k_match_m, dim3(1), MATCH_THREADS, p, j);
    const size_t nJ = (size_t)B * B;
    const int nblk = (int)std::min<size_t>(RED_BLOCKS, (nJ + 255) / 256);
    next(k_assemble, dim3(nblk), 256, p, j);
    next(k_red_sumexp, dim3(nblk), 256, j.J, nJ, j.red, nblk);
    next(k_normalise, dim3(nblk), 256, j.J, nJ, j.red, nblk, p.N);
    return e;
}

// Eq. 3 on the joined table: ln sum_m g(e, m), one warp per e.
__global__ void __launch_bounds__(256) k_marg_out(Params p, JoinScratch j)
{
    after_previous();
    const int B = p.N + 1;
    const int e = (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5));
    if (e >= B) return;
    const double g = lse_warp(j.J + (size_t)e * B, B);
    if ((threadIdx.x & 31) == 0) j.marg[e] = g;
}

cudaError_t launch_marginal_e(const Params &p, const JoinScratch &j, cudaStream_t s)
{
    const int rows = p.N + 1, warps = row_warps(rows);
    launch_next(k_marg_out, dim3((rows + warps - 1) / warps), dim3(32 * warps), 0, s, p, j);
    return cudaGetLastError();
}

// Jackknife accumulation over replicates k = 0..W-1 (walker k left out of
// every window's merge): differences to replicate 0 are summed; an entry that
// is missing (-inf) in any replicate is marked NaN in jk_ref.
__global__ void k_jk_accum(Params p, JoinScratch j, const double *x, size_t n, int k, int32_t *fail)
{
    after_previous();
    if (blockIdx.x == 0 && threadIdx.x == 0 && p.st->join_error && *fail == 0) *fail = k << 8 | p.st->join_error;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const double v = x[i];
        if (k == 0) {
            j.jk_ref[i] = isfinite(v) ? v : NAN;
            j.jk_sum[i] = 0.0;
            j.jk_sq[i] = 0.0;
        } else if (!isfinite(v)) {
            j.jk_ref[i] = NAN;
        } else {
            const double d = v - j.jk_ref[i];
            j.jk_sum[i] += d;
            j.jk_sq[i] += d * d;
        }
    }
}

__global__ void k_jk_final(JoinScratch j, double *mean, double *err, size_t n, int W)
{
    after_previous();
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const double r = j.jk_ref[i];
        if (isnan(r)) {
            mean[i] = -INFINITY;
            err[i] = NAN;
            continue;
        }
        const double s1 = j.jk_sum[i], s2 = j.jk_sq[i];
        mean[i] = r + s1 / W;
        const double var = (double)(W - 1) / W * (s2 - s1 * s1 / W);
        err[i] = sqrt(var > 0.0 ? var : 0.0);
    }
}

cudaError_t launch_jk_accum(const Params &p, const JoinScratch &j, const double *x, size_t n, int k, int32_t *fail,
                            cudaStream_t s)
{
    launch_next(k_jk_accum, dim3(256), dim3(256), 0, s, p, j, x, n, k, fail);
    return cudaGetLastError();
}

cudaError_t launch_jk_final(const JoinScratch &j, double *mean, double *err, size_t n, int W, cudaStream_t s)
{
    launch_next(k_jk_final, dim3(256), dim3(256), 0, s, j, mean, err, n, W);
    return cudaGetLastError();
}

// Eq. 5 per bin: |g_a - g_b| / ((g_a + g_b) / 2) = 2 tanh(x / 2), x = |ln g_a -
// ln g_b|; 2 where one table is empty, NaN where both are.
//
// Bounded by the FP64 pipe (two lanes an SM and cycle), on which tanh is some
// thirty operations.  Tables of one system differ little, and below x = 1/8 the
// odd series of tanh does with eight: 2 tanh(x/2) = x + x u q(u), u = x^2, with
// the Taylor coefficients of tanh over powers of 4; the first term left out is
// 0.1 ulp at x = 1/8.  tanh stays out of line, so that warps without a
// difference above 1/8 issue none of it.  4097 x 4097 bins: 369 -> 142 us.
__device__ __noinline__ double rel_diff_large(double x) { return 2.0 * tanh(0.5 * x); }

__device__ __forceinline__ double rel_diff(double a, double b)
{
    const bool ea = !some(a), eb = !some(b);
    if (ea || eb) return ea && eb ? CUDART_NAN : 2.0;
    const double s = a - b, x = __hiloint2double(__double2hiint(s) & 0x7FFFFFFF, __double2loint(s));
    // x < 1/8 by its bits; infinities and NaN are not
    if ((unsigned)__double2hiint(x) >= 0x3FC00000u) return rel_diff_large(x);
    const double u = x * x;
    double q = -1382.0 / 155925.0 / 1024.0;
    q = fma(q, u, 62.0 / 2835.0 / 256.0);
    q = fma(q, u, -17.0 / 315.0 / 64.0);
    q = fma(q, u, 2.0 / 15.0 / 16.0);
    q = fma(q, u, -1.0 / 3.0 / 4.0);
    return fma(x * u, q, x);
}

// Two bins a thread at a time where the three tables allow 16-byte accesses
// (the last bin of an odd count alone) and there are enough for all SMs' threads;
// below that a thread's two tanh in a row are the call's time (4097 bins that
// differ by more than 1/8: 12.4 us a call with one bin a thread, 15.2 with two;
// 132,000: 21.2 and 20.5).
constexpr size_t PAIRS_FROM = 152 * 512;

template <bool PAIRS>
__global__ void __launch_bounds__(256) k_rel_diff(const double *a, const double *b, double *out, size_t n)
{
    const size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x, step = (size_t)gridDim.x * blockDim.x;
    if constexpr (PAIRS) {
        for (size_t i = t; i < n / 2; i += step) {
            const double2 x = reinterpret_cast<const double2 *>(a)[i], y = reinterpret_cast<const double2 *>(b)[i];
            reinterpret_cast<double2 *>(out)[i] = make_double2(rel_diff(x.x, y.x), rel_diff(x.y, y.y));
        }
        if (t == 0 && (n & 1)) out[n - 1] = rel_diff(a[n - 1], b[n - 1]);
    } else {
        for (size_t i = t; i < n; i += step) out[i] = rel_diff(a[i], b[i]);
    }
}

cudaError_t launch_rel_diff(const double *a, const double *b, double *out, size_t n, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    const bool pairs = n >= PAIRS_FROM && (((uintptr_t)a | (uintptr_t)b | (uintptr_t)out) & 15) == 0;
    const size_t want = ((pairs ? (n + 1) / 2 : n) + 255) / 256;
    const int blocks = (int)std::min<size_t>(want, 152 * 16);
    if (pairs) k_rel_diff<true><<<blocks, 256, 0, s>>>(a, b, out, n);
    else k_rel_diff<false><<<blocks, 256, 0, s>>>(a, b, out, n);
    return cudaGetLastError();
}

}  // namespace rewl
