// Group-per-walker Wang-Landau sampling with tree speculation (sm_103a).
//
// The trials of one walker form a sequential Markov chain (Eq. 1 and the
// update rule of Sec. 2 of arXiv:1508.02748): each trial depends on the
// accept/reject outcome of the one before.  A group of G lanes (G = 8, 16 or
// 32; 32/G walkers per warp) runs one walker and resolves DEPTH+1 trials per
// step (DEPTH = log2(G) - 1): lanes 0..G-2 form a binary tree; lane l sits at
// depth d = floor(log2(l+1)) and evaluates trial t+d under the history
// h = l + 1 - 2^d (bit k of h = outcome assumed for trial t+k).
//
// Per step every lane
//   1. takes its trial from the ring and the five spins around its site from
//      the committed lattice, corrected for the sites its history flips, and
//      so has its trial's move;
//   2. takes the moves of the accepted trials of its history by shuffle, the
//      latest first, and adds them up: the position before and after its own
//      trial.  A bin the path was in 2 accepted trials ago is the current one
//      again iff the two moves cancel, so three sums say which bins were met
//      before, and how often is a constant of the lane's history;
//   3. reads the proposed bin's screen and visits and decides its own trial
//      (Eq. 1) from the values the sequential chain sees there, ln g(b) =
//      base(b) + (H(b) + visits earlier in the step) ln f.  The current bin
//      needs no read: it is the bin the last accepted trial of the history
//      proposed (a shuffle), or the step's first bin, which the lane without a
//      node (G-1) reads.
// One ballot gives the true path from the root: a lane is on it iff the
// ballot bits of its ancestors are the outcomes its history assumes.  The
// path's last lane hands the new position and the path's outcomes round by
// shuffle.  Each on-path lane that accepts writes the visits of the bin it
// enters: the count it read, the path's earlier visits of that bin, and the
// trials until the path leaves it, all known to it; a bin entered twice is
// written in path order (few ordered stores).
//
// Nothing in a step branches by lane, and all groups of a warp step together:
// collectives over part of a warp, and lanes that branch, run the groups of a
// warp one after the other.
//
// Tables (exact formats only; REWL_F32 runs on the thread sampler): ln g(b)
// = base(b) + max(H(b), 0) ln f, the base fixed during an iteration, so a
// visit changes H alone and no floating-point table update runs here.  The
// decision is screened in float from a 32-bit screen per bin, S(b) =
// base(b) - c_w rounded to nearest (c_w one constant per walker, which
// cancels in the difference and keeps the screened magnitudes small), and
// re-taken exactly in double on near-ties of the true path.  Tables live in
// global memory (L1-cached) or, when small, are staged in shared memory for
// the launch (S and H; the bases are read only by the exact re-decision).
//
// The outcome is the sequential chain itself, trial for trial:
//   - random numbers are drawn per trial index from the TRIAL stream of
//     Philox4x32-10, independent of the state (a ring per walker,
//     refilled from the even trial at or below the launch's first trial);
//   - base(b) + n ln f is evaluated exactly in double (fma; the compensated
//     pair converts exactly) and equals the sequential additions whenever
//     ln f = 2^-k and the values stay within 53 (pair: 48) bits;
//   - the float screen is decided only outside a margin that bounds its
//     error.  With x = S + H ln f of a bin in float, t = (ln u + v ln f) - (x_c
//     - x_n), v the difference of the step's visits, errs by at most
//       2^-24 |S| + 2^-24 (|x| + |S|) + 2^-24 |x| per bin (the screen, the
//         count converted to float, the fma),
//       2^-24 (|x_c| + |x_n|) (their difference),
//       2^-24 (|t| + |x_c| + |x_n|) + 2^-24 |t| (ln u + v ln f, which is t and
//         the difference together, and the last subtraction), and
//       0.51 2^-20 (|ln u| + 1) (u rounds with relative error below 2^-23;
//         __logf errs by at most 2^-21.41 in [1/2, 1] and 3 ulp below),
//     below 0.51 M + 2^-22 |t| with M = 2^-20 (|S_c| + |x_c| + |S_n| + |x_n| +
//     |ln u|) + 2^-20, so the sign of t is the decision whenever |t| > M.
//     Otherwise the decision is re-taken from the exact difference: against
//     the float ln u where the two are farther apart than 2^-20 (|ln u| + 1),
//     else against ln u in double.
//
// What bounds it: the instructions of a step (about 150 a warp at G = 32, the
// ring's refill included) and, with few walkers, the step's dependent chain
// (lattice -> move -> shuffles -> bin -> read -> decision -> ballots ->
// shuffle).  Reading one bin a lane instead of two, the visit counts by three
// comparisons, the leaf by shuffle instead of a mailbox, the trial read a step
// ahead and near-ties looked at on the path alone took 266-302 instructions a
// step to 149-157.  Sampling launches of 10^4 trials per walker, GB300, 2070
// MHz, before -> after: L = 8 (36 walkers, 32 lanes, staged) 0.72 -> 0.34 ms; L
// = 16 (256 walkers, 32 lanes) 0.95 -> 0.63 ms; L = 32 (2048 walkers, 32 lanes)
// 1.64 -> 1.03 ms; L = 64 (3904 walkers, 16 lanes) 2.71 -> 1.56 ms.
// Tried and slower: the visits of recent bins in a shared-memory cache (L1
// loses the space), prefetching the neighbourhood's lines (its instructions
// cost what it saves), the path's end by a warp reduction, flips or stores
// under a branch.
#include <algorithm>
#include <type_traits>

#include "rewl_tab.cuh"

namespace rewl {

using namespace tab;

namespace {

// Trials drawn per refill of a walker's ring, which holds two refills.  With a
// whole warp for a walker whose tables are staged (few walkers) a refill's
// latency counts, and two Philox calls a lane at once take hardly longer than
// one (L = 8, 36 walkers: 0.370 -> 0.357 ms); else its shared memory does.
__host__ __device__ constexpr int chunk_of(bool staged, int G) { return staged && G == 32 ? 128 : 64; }
constexpr unsigned FULL = 0xFFFFFFFFu;

// The lattice in shared memory: each row is cut into nblk blocks of at most
// 30 columns, one 32-bit word each, with the column left of the block in bit
// 0, the block's columns from bit 1 and the column right of it after them, so
// that a site's left neighbour, itself and its right neighbour are three
// adjacent bits of one word whatever L is.  L = 32 needs no such copies: its
// row is one word and the three bits are adjacent after a rotation.
struct Blocks {
    int n, width;   // blocks per row, columns per block (the last one may have fewer, never one)
};

__host__ __device__ __forceinline__ Blocks blocks_of(int L)
{
    Blocks b;
    b.n = L <= 30 || L == 32 ? 1 : L <= 60 ? 2 : 3;
    b.width = (L + b.n - 1) / b.n;
    return b;
}

// Entries per row of a staged window (moves within a step change m by at most
// 5, so rows of 16 or more keep the positions of a step apart).
__host__ __device__ __forceinline__ int staged_ld(int wM) { return wM < 15 ? 16 : wM + 1; }

// One buffered trial (16 bytes, one shared-memory vector load).  Everything
// about a trial that does not depend on the walker's state is computed when
// the ring is refilled.  The first RING_TAIL entries are kept twice, the second
// time behind the last one, so that a step's trials are adjacent.
constexpr int RING_TAIL = 8;
struct RingEntry {
    uint32_t a;    // shared lattice: rotation that brings left, site, right to bits 0-2 | the lattice words
                   //   of the site's row << 8, of the row above << 16 and of the row below << 24
                   // register lattice: mask of the four neighbours, bits 0-31
    uint32_t b;    // shared lattice: for lag 1..4 (5 bits each), which of (left, site, right, up, down) is the
                   //   site of trial t - lag (one-hot, or 0); the site i*L+j << 20
                   // register lattice: mask of the four neighbours, bits 32-63
    uint32_t f;    // shared lattice, one block a row: mask of the site's bit(s) in its word
                   // shared lattice, several blocks: the site's copy in another block: 1 | its bit << 1 |
                   //   its word minus the site's, plus 2, << 6 (0: none)
    float lnu;     // ln u in float
};
static_assert(sizeof(RingEntry) == 16, "one vector load per trial");
__host__ __device__ constexpr size_t ring_bytes(bool staged, int G)
{
    return (2 * chunk_of(staged, G) + RING_TAIL) * sizeof(RingEntry);
}

// Register lattice: each trial's site as a 64-bit mask, beside the ring.
__host__ __device__ constexpr size_t bits_bytes(bool staged, int G) { return ring_bytes(staged, G) / 2; }
static_assert(2 * sizeof(uint2) == sizeof(RingEntry), "half a ring entry");

// Eq. 1 decided from the exact values (near-ties of the float screen on the
// true path only).
// ccnt and ncnt are the visit counts the chain has at that point; the
// difference is exact in double.  q: the trial's index (its acceptance word
// is drawn again where ln u is needed in double).
template <class TB>
__device__ __forceinline__ int exact_accept(const typename TB::Elem *gb, unsigned ci, int ccnt, unsigned ni, int ncnt,
                                         double lnf, float lnu32, unsigned long long q, uint32_t w, uint32_t key0,
                                         uint32_t key1)
{
    const double delta = fma((double)ccnt, lnf, TB::exact(gb[ci])) - fma((double)ncnt, lnf, TB::exact(gb[ni]));
    if (delta >= 0.0) return 1;
    const double lu = (double)lnu32;
    const double band = (fabs(lu) + 1.0) * 0x1p-20;
    if (lu < delta - band) return 1;
    if (lu > delta + band) return 0;
    const u32x4 x = philox10((uint32_t)(q >> 1), (uint32_t)(q >> 33), w, TAG_TRIAL, key0, key1);
    return log(unit_open_d((q & 1ull) ? x.w : x.y)) < delta ? 1 : 0;
}

// Four bytes into shared memory; no register waits for them, so that one warp
// has a whole window under way.
__device__ __forceinline__ void async4(void *to, const void *from)
{
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(to);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(a), "l"(from) : "memory");
}

__device__ __forceinline__ void async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

template <int G>
struct TreeShape {
    static constexpr int DEPTH = G == 32 ? 4 : G == 16 ? 3 : 2;
};

}  // namespace

// LAT: the lattice (N <= 32 or N <= 64 sites, bit i*L + j) is held in one or two
// registers by every lane (LAT = 1, 2); otherwise it lives in shared memory
// (Blocks), its rows one block each (0) or several (3).  SMT: S and H staged in
// shared memory for the launch.
template <bool SMT, int G, int PREC, int LAT>
__global__ void __launch_bounds__(256) k_sweep_tree(Params p, unsigned ntrials, int smem_per_walker)
{
    after_previous();
    using TB = Tab<PREC>;
    using Elem = typename TB::Elem;
    constexpr int DEPTH = TreeShape<G>::DEPTH;
    constexpr int GPW = 32 / G;   // walkers per warp
    constexpr unsigned GBITS = G == 32 ? 0xFFFFFFFFu : ((1u << G) - 1u);
    constexpr bool REG = LAT == 1 || LAT == 2, HI = LAT == 2, WIDE = LAT == 3;
    constexpr int CHUNK = chunk_of(SMT, G), RING = 2 * CHUNK;
    constexpr size_t RING_BYTES = ring_bytes(SMT, G), BITS_BYTES = bits_bytes(SMT, G);
    constexpr unsigned RMASK = RING - 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int gl = lane & (G - 1), grp = lane / G;
    const int slot = wid * GPW + grp;   // walker slot within the block
    if (ntrials == 0 || p.st->done) return;
    // The groups of a warp run in lockstep (every collective takes the whole
    // warp), so a group without a walker to sample (past the last walker, or
    // of an empty window) goes along idle: it reads a walker's data, never has
    // a lane on the true path and writes nothing.
    const int wany = blockIdx.x * ((blockDim.x >> 5) * GPW) + slot;
    const int w = min(wany, p.nwalk - 1);
    const bool idle = wany >= p.nwalk || !p.active[w / p.W];
    if (__all_sync(FULL, idle)) return;

    unsigned char *base = smem_raw + (size_t)slot * smem_per_walker;
    RingEntry *ring = reinterpret_cast<RingEntry *>(base);
    uint2 *bits = reinterpret_cast<uint2 *>(base + RING_BYTES);        // REG
    uint32_t *lat = reinterpret_cast<uint32_t *>(base + RING_BYTES);   // nlat words and G that take the idle lanes' flips
    const int L = p.L;
    const Blocks bk = blocks_of(L);
    const int nlat = REG ? 0 : L * bk.n;
    const Elem *g_base = reinterpret_cast<const Elem *>(PREC == REWL_FP64 ? (const void *)p.lng : (const void *)p.lng2)
                       + (size_t)w * p.tstride;
    int32_t *gH = p.H + (size_t)w * p.tstride;
    const float *gS = p.scr + (size_t)w * p.tstride;
    // staged: (screen, visits >= 0) of each bin, rows of ld entries, with two
    // rows before and after the window's and at least one entry after each row
    // that are marked outside (visits -1), so a proposed bin's entry says itself
    // whether it is in the window; a bin without a visit goes back unwritten
    const int wM = p.wM;
    const int ld = staged_ld(wM);
    const int nstaged = (p.wE + 4) * ld;
    int2 *tab = reinterpret_cast<int2 *>(base + RING_BYTES + (REG ? BITS_BYTES : ((nlat + G) * 4 + 15) & ~15));
    // Staging in and out of a window by one warp: the entries come by copies
    // that no register waits for, their addresses by a walk through the rows
    // (loads, stores and a division an entry before: 3.4 ns a bin in and out, 1.4
    // so; L = 8, 36 walkers, 64 cycles 23.2 -> 22.4 ms).  Windows of at most 26 x
    // 26 bins (N <= 32) keep the short form: they have little to stage, and the
    // step compiled with the walk took 2% longer there.
    constexpr bool WALK = SMT && LAT != 1;
    auto each_bin = [&](auto f) {                   // f(bin, its entry), every G-th one
        const int by = G / wM;                      // rows that G bins are on
        int m = gl % wM, k = (gl / wM + 2) * ld + m;
        #pragma unroll 4
        for (int b = gl; b < p.T; b += G) {
            f(b, k);
            m += G - by * wM;
            k += G + by * (ld - wM);
            if (m >= wM) {
                m -= wM;
                k += ld - wM;
            }
        }
    };
    if constexpr (WALK) {
        each_bin([&](int b, int k) {
            async4(&tab[k].x, gS + b);
            async4(&tab[k].y, gH + b);
        });
        for (int k = gl; k < 2 * ld; k += G) tab[k] = tab[nstaged - 1 - k] = make_int2(0, -1);
        for (int e = 2 + gl; e < p.wE + 2; e += G)
            for (int m = wM; m < ld; ++m) tab[e * ld + m] = make_int2(0, -1);
        async_wait();
        each_bin([&](int, int k) { atomicMax(&tab[k].y, 0); });
    } else if constexpr (SMT) {
        #pragma unroll 4
        for (int k = gl; k < nstaged; k += G) {
            const int e = k / ld - 2, m = k - (e + 2) * ld;
            const bool in = e >= 0 && e < p.wE && m < wM;
            tab[k] = in ? make_int2(__float_as_int(gS[e * wM + m]), max(gH[e * wM + m], 0))
                        : make_int2(0, -1);
        }
    }
    // row r of the stored lattice as 64 bits
    auto stored_row = [&](int r) -> unsigned long long {
        unsigned long long v = p.spins[(size_t)(r * p.wpr) * p.nwalk + w];
        if (p.wpr == 2) v |= (unsigned long long)p.spins[(size_t)(r * 2 + 1) * p.nwalk + w] << 32;
        return v;
    };
    uint32_t lo = 0, hi = 0;            // REG: the committed lattice
    if (REG) {
        unsigned long long v = 0;
        for (int r = 0; r < L; ++r) v |= stored_row(r) << (r * L);
        lo = (uint32_t)v;
        hi = (uint32_t)(v >> 32);
    } else {
        for (int k = gl; k < nlat; k += G) {
            const int r = k / bk.n, q = k - r * bk.n, c0 = q * bk.width;
            const unsigned long long v = stored_row(r);
            if (L == 32) {
                lat[k] = (uint32_t)v;
            } else {
                unsigned long long x = c0 ? v >> (c0 - 1) : (v << 1) | ((v >> (L - 1)) & 1ull);
                if (L - c0 <= bk.width) x |= (v & 1ull) << (L - c0 + 1);
                lat[k] = (uint32_t)x;
            }
        }
    }
    __syncwarp();

    // positions: staged, the bin's entry; else (e - e0) << 16 | (m - m0).  A
    // move changes e by de and m by dm, the position by de * erow + dm.
    const int4 R = p.rect[w / p.W];
    const int erow = SMT ? ld : 65536;
    const int estep = wM - 65536;       // global tables: index = position + e * estep
    const unsigned Tm1 = (unsigned)(p.T - 1);
    const double lnf = p.st->lnf;
    const float lnf32 = __double2float_rn(lnf);
    const uint32_t N = (uint32_t)p.N;
    const uint32_t divL = p.divL;

    // This lane's node of the tree.  Lane G-1 holds none: it never accepts and
    // its move is 0; it goes along with the root's trial, which the ring always
    // holds (the entry after the step's last trial may not be filled yet, and
    // says which lattice words to read).
    const bool node = gl < G - 1;
    const int dl = node ? 31 - __clz(gl + 1) : 0;
    const int hist = node ? gl + 1 - (1 << dl) : 0;
    const int spanp = node ? ((R.y - R.x) << 16) | (R.w - R.z) : (int)0xC0000000;
    // Lanes of the accepted trials of the history, the latest first (lane G-1
    // where there are fewer), and how many of the step's trials end in the
    // bins the history passes: n0 in the current one since the last accepted
    // trial, n1, n2, n3 in the ones before it.
    int src[DEPTH], seg[DEPTH + 1];
    #pragma unroll
    for (int j = 0; j < DEPTH; ++j) src[j] = grp * G + G - 1;
    #pragma unroll
    for (int j = 0; j <= DEPTH; ++j) seg[j] = 0;
    {
        int j = 0, last = dl;            // last: the trial after the segment's end
        for (int k = DEPTH - 1; k >= 0; --k)
            if (node && k < dl && ((hist >> k) & 1)) {
                #pragma unroll
                for (int q = 0; q < DEPTH; ++q)
                    if (q == j) { src[q] = grp * G + (1 << k) - 1 + (hist & ((1 << k) - 1)); seg[q] = last - k; }
                last = k;
                ++j;
            }
        #pragma unroll
        for (int q = 0; q <= DEPTH; ++q)
            if (node && q == j) seg[q] = last;
    }
    const int n0 = seg[0], n1 = seg[1], n2 = DEPTH >= 3 ? seg[2] : 0, n3 = DEPTH >= 4 ? seg[DEPTH >= 4 ? 3 : 0] : 0;
    // On the true path iff the ballot bits of the ancestors (lane 2^k - 1 +
    // (h mod 2^k) at depth k < d) are the outcomes the history assumes: anc
    // marks the ancestors, want holds those outcomes.  Lane G-1 of the group
    // never accepts: asking for its acceptance takes a lane off every path.
    const unsigned never = 1u << (grp * G + G - 1);
    unsigned anc = 0, want = 0;
    #pragma unroll
    for (int k = 0; k <= DEPTH; ++k)
        if (k < dl) {
            const int a = grp * G + (1 << k) - 1 + (hist & ((1 << k) - 1));
            anc |= 1u << a;
            want |= (unsigned)((hist >> k) & 1) << a;
        }
    if (idle || !node) { anc |= never; want |= never; }
    // A lane that accepts on the path writes the visits of the bin it enters,
    // lane G-1 those of the step's first bin.  later: the trials after the
    // lane's; rank: order among the bins of the path that could be the same one
    // (those an even number of accepted trials apart, and visited in the step).
    const bool first = !node && !idle;
    const int later = node ? dl + 1 : 0;
    const int rank = node ? (__popc(hist) + 1 - (dl == 0 ? 1 : hist & 1)) >> 1 : 0;
    const int hacc = node ? hist | (1 << dl) : 0;
    // relation fields of the lags whose trials the history accepts: trial t+k
    // (k < d) is lag d - k of this lane's trial; REG: the accepted trials
    uint32_t sel = 0, flip[DEPTH];
    #pragma unroll
    for (int k = 0; k < DEPTH; ++k) {
        const bool on = node && k < dl && ((hist >> k) & 1);
        if (on) sel |= 0x1Fu << (5 * (dl - k - 1));
        flip[k] = on ? FULL : 0u;
    }
    // move (position difference) of a trial whose five spins (left, site,
    // right, up, down) are the lane's number: looked up by shuffle
    const int nup_l = __popc(lane & 0x1D);
    const int lut = (lane & 2) ? (nup_l - 2) * erow - 1 : (2 - nup_l) * erow + 1;
    const int mvA = node ? erow : 0, mvB = node ? 2 * erow + 1 : 0;   // REG: the move is +-(nup mvA - mvB)

    // committed position (uniform over the group)
    int P0 = (p.we[w] - R.x + (SMT ? 2 : 0)) * erow + (p.wm[w] - R.z);
    const unsigned long long t0 = p.wt[w];
    const unsigned r0 = (unsigned)t0 & RMASK;
    const unsigned long long c0 = t0 >> 1;   // first Philox call
    unsigned u = 0;                 // trials done in this launch
    unsigned cfill = 0;             // calls done: the ring holds trials t0 - (t0 & 1) + [0, 2 cfill)
    unsigned end = 1u << (DEPTH + 1);
    int err = 0;                    // sign: a count passed INT_MAX

    while (u < ntrials) {
        // ---- refill the ring (the test leaves the parity of t0 out, so the
        // warp's groups refill together)
        if (2 * cfill < u + CHUNK / 2 + 1) {
            #pragma unroll (CHUNK == 128 ? 2 : 1)
            for (int r = 0; r < CHUNK / 2 / G; ++r) {
                const unsigned long long c = c0 + cfill + (unsigned)(gl + r * G);
                const u32x4 x = philox10((uint32_t)c, (uint32_t)(c >> 32), (uint32_t)w, TAG_TRIAL, p.key0, p.key1);
                uint32_t si[2], sj[2];
                #pragma unroll
                for (int hh = 0; hh < 2; ++hh) {
                    const uint32_t xs = hh ? x.z : x.x, xu = hh ? x.w : x.y;
                    const uint32_t site = __umulhi(xs, N);
                    const uint32_t i = __umulhi(site, divL);
                    const uint32_t j = site - i * (uint32_t)L;
                    si[hh] = i;
                    sj[hh] = j;
                    const uint32_t iu = i == 0 ? L - 1 : i - 1, id = i == (uint32_t)L - 1 ? 0 : i + 1;
                    RingEntry en;
                    uint2 own = make_uint2(0u, 0u);
                    if (REG) {
                        const uint32_t jl = j == 0 ? L - 1 : j - 1, jr = j == (uint32_t)L - 1 ? 0 : j + 1;
                        const unsigned long long nb = (1ull << (iu * L + j)) | (1ull << (id * L + j))
                                                    | (1ull << (i * L + jl)) | (1ull << (i * L + jr));
                        en.a = (uint32_t)nb;
                        en.b = (uint32_t)(nb >> 32);
                        en.f = 0;
                        const unsigned long long o = 1ull << site;
                        own = make_uint2((uint32_t)o, (uint32_t)(o >> 32));
                    } else {
                        en.b = site << 20;
                        if (WIDE) {
                            // the first column of a block is also the bit after the previous block's last
                            // column, the last one also bit 0 of the next block
                            const uint32_t q = (uint32_t)((int)j >= bk.width) + (uint32_t)((int)j >= 2 * bk.width);
                            const uint32_t amt = j - q * bk.width, qn = (uint32_t)bk.n - 1u;
                            en.a = amt | ((i * bk.n + q) << 8) | ((iu * bk.n + q) << 16) | ((id * bk.n + q) << 24);
                            const bool fc = amt == 0, lc = (int)amt == bk.width - 1 || (int)j == L - 1;
                            const uint32_t qo = fc ? (q == 0 ? qn : q - 1) : (q == qn ? 0u : q + 1);
                            const uint32_t bit = fc ? (q == 0 ? (uint32_t)L - qn * bk.width : (uint32_t)bk.width) + 1u : 0u;
                            en.f = fc || lc ? 1u | (bit << 1) | ((qo + 2u - q) << 6) : 0u;
                        } else {
                            const uint32_t amt = L == 32 ? (j + 31u) & 31u : j;
                            en.a = amt | (i << 8) | (iu << 16) | (id << 24);
                            en.f = __funnelshift_l(2u, 2u, amt);
                            if (L != 32) en.f |= (j == 0 ? 2u << L : 0u) | (uint32_t)(j == (uint32_t)L - 1);
                        }
                    }
                    en.lnu = __logf(__fmaf_rn(__uint2float_rn(xu), 0x1p-32f, 0x1p-33f));
                    const unsigned at = (unsigned)(2 * c + hh) & RMASK;
                    ring[at] = en;
                    if (REG) bits[at] = own;
                    if (at < RING_TAIL) {
                        ring[at + RING] = en;
                        if (REG) bits[at + RING] = own;
                    }
                }
                if (!REG) {
                    // relation codes of the two trials to the DEPTH trials before each
                    __syncwarp();
                    uint32_t f[DEPTH + 1];          // sites of the trials before the second one, the nearest first
                    f[0] = si[0] * (uint32_t)L + sj[0];
                    #pragma unroll
                    for (int lag = 1; lag <= DEPTH; ++lag) f[lag] = ring[((unsigned)(2 * c) - lag) & RMASK].b >> 20;
                    #pragma unroll
                    for (int hh = 0; hh < 2; ++hh) {
                        const uint32_t i = si[hh], j = sj[hh], site = i * (uint32_t)L + j;
                        const uint32_t pos[5] = {j == 0 ? site + L - 1 : site - 1, site, j == (uint32_t)L - 1 ? site + 1 - L : site + 1,
                                                 i == 0 ? site + N - L : site - L, i == (uint32_t)L - 1 ? site + L - N : site + L};
                        uint32_t rel = site << 20;
                        #pragma unroll
                        for (int lag = 1; lag <= DEPTH; ++lag) {
                            #pragma unroll
                            for (int k = 0; k < 5; ++k)
                                if (f[lag - hh] == pos[k]) rel |= 1u << (5 * (lag - 1) + k);
                        }
                        const unsigned at = (unsigned)(2 * c + hh) & RMASK;
                        ring[at].b = rel;
                        if (at < RING_TAIL) ring[at + RING].b = rel;
                    }
                }
            }
            cfill += CHUNK / 2;
            __syncwarp();
        }
        // steps until the ring runs low or the launch ends; its last step may
        // be a short one, whose lanes past the last trial leave the path
        unsigned nsteps = (2 * cfill - 1 - u) / (DEPTH + 1);
        if (ntrials - u <= (unsigned)DEPTH) {
            nsteps = 1;
            end = 1u << (ntrials - u);
            if (dl >= (int)(ntrials - u)) { anc |= never; want |= never; }
        } else {
            nsteps = min(nsteps, (ntrials - u) / (DEPTH + 1));
        }
        // what the step's trials need that does not depend on the state is read
        // a step ahead: the lane's trial and, REG, the sites its history flips
        RingEntry nxt;
        uint32_t nlo = 0, nhi = 0;
        uint2 nbit = make_uint2(0u, 0u);
        auto ahead = [&](unsigned at) {
            const unsigned now = at & RMASK;
            nxt = ring[now + dl];
            if (REG) {
                nlo = nhi = 0;
                #pragma unroll
                for (int k = 0; k < DEPTH; ++k) {
                    const uint2 b = bits[now + k];
                    nlo ^= b.x & flip[k];
                    if (HI) nhi ^= b.y & flip[k];
                }
                nbit = bits[now + dl];
            }
        };
        ahead(r0 + u);
        #pragma unroll 2
        for (unsigned it = 0; it < nsteps; ++it) {
        // ---- 1. own trial under own history: its move, as a position difference
        const RingEntry me = nxt;
        uint32_t hlo = 0, hhi = 0, olo = 0, ohi = 0;   // REG: the lattice under the history; the site's bit
        int pk;
        if (REG) {
            hlo = lo ^ nlo;
            olo = nbit.x;
            bool sup = (hlo & olo) != 0u;
            int nup = __popc(hlo & me.a);
            if (HI) {
                hhi = hi ^ nhi;
                ohi = nbit.y;
                sup = ((hlo & olo) | (hhi & ohi)) != 0u;
                nup += __popc(hhi & me.b);
            }
            pk = nup * (sup ? mvA : -mvA) + (sup ? -mvB : mvB);
        } else {
            const uint32_t wc = lat[(me.a >> 8) & 0xFFu], wu = lat[(me.a >> 16) & 0xFFu], wd = lat[me.a >> 24];
            uint32_t v5 = (__funnelshift_r(wc, wc, me.a) & 7u) | (__funnelshift_r(wu, wu, me.a - 2u) & 8u)
                        | (__funnelshift_r(wd, wd, me.a - 3u) & 16u);
            uint32_t corr = me.b & sel;
            if (DEPTH > 2) corr ^= corr >> 10;
            corr ^= corr >> 5;
            v5 ^= corr;
            pk = __shfl_sync(FULL, lut, v5);        // (the low five bits select)
            if (!node) pk = 0;
        }

        // ---- 2. position under the history (Pc) and after the own move (Pn),
        // and by how much the step's earlier trials visited the current bin more
        // often than the proposed one (the bin before the last 2 accepted trials
        // is the current one again iff their moves cancel, and so on)
        int y[DEPTH];
        #pragma unroll
        for (int j = 0; j < DEPTH; ++j) y[j] = __shfl_sync(FULL, pk, src[j]);
        const int z2 = y[0] + y[1];
        const int zl = DEPTH >= 4 ? y[DEPTH >= 3 ? 2 : 0] + y[DEPTH >= 4 ? 3 : 0] : DEPTH >= 3 ? y[DEPTH >= 3 ? 2 : 0] : 0;
        const int Pc = P0 + z2 + zl, Pn = (P0 + pk) + z2 + zl;
        int vnew = pk + y[0] == 0 ? n1 : 0;
        if (DEPTH >= 4) vnew += pk + z2 + y[DEPTH >= 3 ? 2 : 0] == 0 ? n3 : 0;
        int vcur = n0;
        if (DEPTH >= 3) vcur += z2 == 0 ? n2 : 0;

        // ---- 3. decision of the own trial (Eq. 1).  Off-path lanes may hold
        // positions outside the window: clamped reads.  With global tables a lane
        // reads the proposed bin alone: the current one is the bin the history's
        // last accepted trial proposed, or the step's first bin, which lane G-1
        // reads; with staged ones a second read is cheaper than that shuffle.
        unsigned nu;
        bool live = node;                 // the proposed bin is in the window
        float xn, mn, xc, mc;
        int hn;
        if constexpr (SMT) {
            nu = min((unsigned)Pn, (unsigned)nstaged - 1u);
            const int2 n = tab[nu], c = tab[min((unsigned)Pc, (unsigned)nstaged - 1u)];
            hn = n.y;
            live = node && n.y >= 0;
            xn = __fmaf_rn(__int2float_rn(n.y), lnf32, __int_as_float(n.x));
            xc = __fmaf_rn(__int2float_rn(c.y), lnf32, __int_as_float(c.x));
            mn = fabsf(__int_as_float(n.x)) + fabsf(xn);
            mc = fabsf(__int_as_float(c.x)) + fabsf(xc);
        } else {
            nu = min((unsigned)(Pn + (Pn >> 16) * estep), Tm1);
            const float sn = gS[nu];
            hn = max(gH[nu], 0);
            live = ((Pn | (spanp - Pn)) & 0x80008000) == 0;
            xn = __fmaf_rn(__int2float_rn(hn), lnf32, sn);
            mn = fabsf(sn) + fabsf(xn);
            xc = __shfl_sync(FULL, xn, src[0]);
            mc = __shfl_sync(FULL, mn, src[0]);
        }
        ahead(r0 + u + DEPTH + 1);
        const float t32 = __fsub_rn(__fmaf_rn(__int2float_rn(vnew - vcur), lnf32, me.lnu), __fsub_rn(xc, xn));
        const float M = __fmaf_rn(mc + mn + fabsf(me.lnu), 0x1p-20f, 0x1p-20f);
        bool acc = live && t32 < 0.0f;
        bool near = live && !(fabsf(t32) > M);      // (not a number counts as near)

        // ---- the true path: the lanes whose ancestors decided as their
        // histories assume, and the state after its last trial
        unsigned bal, nearb, pm, path;
        bool onp;
        int Pa;
        uint32_t lo2 = 0, hi2 = 0;
        auto follow = [&]() {
            bal = __ballot_sync(FULL, acc);
            nearb = __ballot_sync(FULL, near);
            onp = ((bal ^ want) & anc) == 0u;
            pm = __ballot_sync(FULL, onp);
            const int leaf = 31 - __clz(pm & (GBITS << (grp * G)));
            Pa = __shfl_sync(FULL, acc ? Pn : Pc, leaf);
            if (REG) {
                lo2 = __shfl_sync(FULL, acc ? hlo ^ olo : hlo, leaf);
                if (HI) hi2 = __shfl_sync(FULL, acc ? hhi ^ ohi : hhi, leaf);
            }
            path = __shfl_sync(FULL, acc ? hacc : hist, leaf);   // bit k: trial k accepted
        };
        follow();
        while (pm & nearb) {
              // near-ties on the path are decided exactly
            if (onp && near) {
                unsigned ib, jb;          // the bins' entries in the window's table
                int hc;
                if constexpr (SMT) {
                    ib = (unsigned)(Pc - (Pc / ld) * (ld - wM) - 2 * wM);
                    jb = (unsigned)(Pn - (Pn / ld) * (ld - wM) - 2 * wM);
                    hc = tab[Pc].y;
                } else {
                    ib = (unsigned)(Pc + (Pc >> 16) * estep);
                    jb = nu;
                    hc = max(gH[ib], 0);
                }
                acc = exact_accept<TB>(g_base, ib, hc + vcur, jb, hn + vnew, lnf, me.lnu, t0 + u + dl, (uint32_t)w, p.key0,
                                       p.key1);
                near = false;
            }
            __syncwarp();
            follow();
        }

        // ---- commit: the visits of the path's bins are written: the count a bin
        // had, plus its earlier visits in the step, plus those until the path
        // leaves it.  A bin the path comes back to is written again with the
        // larger count; global stores of such bins are ordered by rank.
        P0 = Pa;
        if (REG) {
            lo = lo2;
            hi = hi2;
        } else {
            // lanes without a flip go to a word of their own (a branch would
            // cost the warp more than the added traffic)
            const bool flip = onp && acc;
            uint32_t *const own = lat + nlat + gl, *const word = lat + ((me.a >> 8) & 0xFFu);
            atomicXor(flip ? word : own, WIDE ? 2u << (me.a & 31u) : me.f);
            if (WIDE) atomicXor(flip && (me.f & 1u) ? word + (int)(me.f >> 6) - 2 : own, 1u << ((me.f >> 1) & 31u));
        }
        const unsigned ahead_of = (path | end) >> later;
        const int stay = __popc(ahead_of ^ (ahead_of - 1u)) - (node ? 0 : 1);   // trials up to its lowest bit
        const bool st = node ? onp && acc : first && stay > 0;
        const int val = hn + vnew + stay;
        if (st) err |= val;
        if constexpr (SMT) {
            // (visits only grow: the larger count stays, in whatever order; lanes
            // without a bin to write go to an entry outside the window)
            atomicMax(&tab[st ? nu : (unsigned)gl].y, st ? val : -1);
        } else {
            #pragma unroll
            for (int k = 0; k < (DEPTH >= 4 ? 3 : 2); ++k) {
                if (k) __syncwarp();
                if (st && rank == k) gH[nu] = val;
            }
        }
        __syncwarp();
        u += (unsigned)(DEPTH + 1);
        }
    }

    // ---- the state
    if (__any_sync(FULL, err < 0) && lane == 0) atomicOr(&p.st->error, ERR_OVERFLOW);
    __syncwarp();
    if (idle) return;
    if constexpr (WALK) {
        each_bin([&](int b, int k) {
            const int h = tab[k].y;
            if (h > 0) gH[b] = h;
        });
    } else if constexpr (SMT) {
        for (int k = gl + 2 * ld; k < nstaged - 2 * ld; k += G) {
            const int e = k / ld - 2, m = k - (e + 2) * ld, h = tab[k].y;
            if (m < wM && h > 0) gH[e * wM + m] = h;
        }
    }
    for (int r = gl; r < L; r += G) {
        unsigned long long v;
        if (REG) {
            v = ((((unsigned long long)hi << 32) | lo) >> (r * L)) & ((1ull << L) - 1);
        } else if (L == 32) {
            v = lat[r];
        } else {
            v = 0;
            for (int q = 0; q < bk.n; ++q)
                v |= (unsigned long long)((lat[r * bk.n + q] >> 1) & ((1u << bk.width) - 1u)) << (q * bk.width);
            if (L < 64) v &= (1ull << L) - 1;
        }
        p.spins[(size_t)(r * p.wpr) * p.nwalk + w] = (uint32_t)v;
        if (p.wpr == 2) p.spins[(size_t)(r * 2 + 1) * p.nwalk + w] = (uint32_t)(v >> 32);
    }
    if (gl == 0) {
        const int e = P0 / erow;
        p.we[w] = e - (SMT ? 2 : 0) + R.x;
        p.wm[w] = P0 - e * erow + R.z;
        p.wt[w] = t0 + ntrials;
    }
}

// Shared memory per walker: ring, lattice (16-byte padded) and, when staged,
// S and H (8 bytes per entry).
size_t tree_smem_per_warp(const Params &p, bool smt, int group)
{
    const size_t nlat = (size_t)p.L * blocks_of(p.L).n + group;
    size_t b = ring_bytes(smt, group) + (p.lattice_reg ? bits_bytes(smt, group) : (nlat * 4 + 15) & ~(size_t)15);
    if (smt) b += (size_t)(p.wE + 4) * staged_ld(p.wM) * 8;
    return (b + 15) & ~(size_t)15;
}

// group: lanes per walker (8, 16 or 32); warps: warps per block.  One
// launch runs fewer than 2^31 trials per walker (launch_sweep splits).
// Exact table formats only.
cudaError_t launch_sweep_tree(const Params &p, uint64_t ntrials, int group, int warps, bool smt, cudaStream_t s)
{
    if (p.precision != REWL_FP64 && p.precision != REWL_F32X2) return cudaErrorInvalidValue;
    if (group != 8 && group != 16 && group != 32) group = 32;
    const int gpw = 32 / group;
    const size_t max_smem = 227 * 1024;
    // a window whose bins fit in a block's shared memory, but not with the
    // entries around them, is sampled from global memory
    if (smt && tree_smem_per_warp(p, true, group) * gpw > max_smem
        && (128 * sizeof(RingEntry) + 48 + (((size_t)p.nwords * 4 + 15) & ~(size_t)15) + 8 * (size_t)p.T) * gpw <= max_smem)
        smt = false;
    const size_t per = tree_smem_per_warp(p, smt, group);
    // one warp a block: blocks of several warps leave when their last walker
    // does (16 lanes, L = 16: 0.90 ms at 1 warp, 1.00 at 4; 32 lanes: the same);
    // with four 8-lane groups a warp two (L = 32, shared memory set aside as
    // below: 9600 walkers 2.61 ms at 1 warp, 2.50 at 2 and 4; 10,752: 2.97, 2.72,
    // 2.74; 11,520: 4.23, 3.03, 2.81)
    if (warps <= 0) warps = group == 8 ? 2 : 1;
    // no more warps per block than the shared memory of one block holds
    while (warps > 1 && per * (size_t)gpw * warps > max_smem) --warps;
    if (per * (size_t)gpw * warps > max_smem) return cudaErrorInvalidValue;
    const size_t smem = per * (size_t)gpw * warps;
    const int walkers_per_block = gpw * warps;
    const int blocks = (p.nwalk + walkers_per_block - 1) / walkers_per_block;
    const int threads = 32 * warps;
    // Shared memory for the blocks an SM gets and little more: the rest is L1,
    // which the tables live in.  The driver's choice goes by the blocks that could be
    // resident, and may leave 28 KB of L1 (10,752 walkers at L = 32, 8 lanes: 4.3
    // ms; 2.8 with 60 KB or more).  Past some 11,000 walkers their blocks take
    // turns, and only those that an SM holds at once count (12,288 walkers 5.6 ->
    // 3.7 ms, 16,384 7.4 -> 4.9, 24,576 9.9 -> 6.4).  Other runs' blocks find a
    // place beside a small run's only within its carve-out: 64 KB are 14 of their
    // 32-lane warps (8 runs of 128 walkers at L = 16, each on its own stream: 2.11
    // ms a cycle without, 0.79 so, one alone 0.61), and staged walkers, which need
    // no L1, leave them all of it (32 runs of 36 at L = 8: 2.53 and 0.59).
    const long long share = (p.sharing + 152ll * walkers_per_block - 1) / (152ll * walkers_per_block);
    auto go = [&](auto kern) -> cudaError_t {
        cudaError_t e = cudaSuccess;
        if (smem > 48 * 1024) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        long long held = share;
        if (e == cudaSuccess && share * warps > 16) {
            int fit = 0;
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, kern, threads, smem);
            held = std::min<long long>(share, std::max(fit, 1));
        }
        if (e != cudaSuccess) return e;
        const long long all = 228 * 1024;
        const long long room = smt ? all : std::max<long long>((long long)(smem + 1024) * held, 64 * 1024);
        return launch_next_with((int)std::min<long long>(100, (room * 100 + all - 1) / all), kern, dim3(blocks), dim3(threads), smem, s, p,
                                (unsigned)ntrials, (int)per);
    };
    const int lat = p.lattice_reg ? (p.N <= 32 ? 1 : 2) : blocks_of(p.L).n > 1 ? 3 : 0;
    auto with = [&](auto staged, auto g, auto prec) -> cudaError_t {
        constexpr bool S = decltype(staged)::value;
        constexpr int G = decltype(g)::value, P = decltype(prec)::value;
        if (lat == 1) return go(k_sweep_tree<S, G, P, 1>);
        if (lat == 2) return go(k_sweep_tree<S, G, P, 2>);
        if (lat == 3) return go(k_sweep_tree<S, G, P, 3>);
        return go(k_sweep_tree<S, G, P, 0>);
    };
    auto lanes = [&](auto staged, auto prec) -> cudaError_t {
        if (group == 32) return with(staged, std::integral_constant<int, 32>(), prec);
        if (group == 16) return with(staged, std::integral_constant<int, 16>(), prec);
        return with(staged, std::integral_constant<int, 8>(), prec);
    };
    auto tables = [&](auto prec) -> cudaError_t {
        return smt ? lanes(std::true_type(), prec) : lanes(std::false_type(), prec);
    };
    return p.precision == REWL_FP64 ? tables(std::integral_constant<int, REWL_FP64>())
                                    : tables(std::integral_constant<int, REWL_F32X2>());
}

}  // namespace rewl
