// Melting temperature of each site (Sec. 2.1, Melting temperature filtering):
// the maximum over every oligonucleotide of the degenerate primer of the
// two-state nearest-neighbour Tm against the template at the site,
//     Tm(o) = 1000 dH(o) / (dS(o) + C) - 273.15 (+ shift for salt methods 1-4),
// C = R ln(x), and salt method 5 adds 0.368 (L - 1) ln[Na_eq] to dS.
//
// The paper evaluates every oligo separately.  Here the maximum is found
// without enumeration: dH and dS are sums over adjacent primer positions, so
// for a trial value lam the minimum over oligos of F(o) = 1000 dH(o) -
// lam (dS(o) + C) is a 4-state shortest path along the primer (the state is
// the oligo's base at a position, restricted to its IUPAC set; only the
// degenerate positions and the two ends need a step, the fixed stretches
// between them being folded into per-site 4x4 tables), and
// Dinkelbach's iteration lam <- ratio(argmin F) climbs to the maximum ratio in
// a few rounds, provided dS(o) + C < 0 for every oligo (checked first with a
// max-path pass).  Four lanes per site (one DP state each), fp32.
//
// Sites whose fp32 maximum lies within 0.01 deg C of tm_min (fp32 error here
// is ~1e-3 deg C at most) get an exact decision instead: Tm(o) >= tm_min iff
// F(o) = 1000 dH(o) - thr (dS(o) + C) <= 0 at thr = tm_min in kelvin (the
// entropy side is negative), so one more shortest-path pass, in fp64 at
// lam = thr, gives the sign of the minimum of F over all oligos.  Its fp64
// error is ~1e-10 cal; a minimum within 1e-6 cal of zero (a ratio within
// ~1e-9 K of the threshold), and every site under a table where some duplex
// entropy reaches -C, is evaluated the reference way: every oligo, in fp64,
// with the same operation order as the definition and no fused multiply-adds,
// a whole block sharing one site's oligos (tm_exact_kernel).  Either way the
// pass flag is the exact fp64 decision.
#include <algorithm>
#include <cmath>

#include <cstdlib>

#include "ah_internal.h"

namespace ah {
namespace {

__device__ __forceinline__ int base_at(const uint32_t *__restrict__ planes, uint64_t P)
{
    const uint64_t t = P / kTileBases, r = P % kTileBases;
    const int b = (int)(r / kTileW), j = (int)(r % kTileW);
    const uint32_t *w = planes + t * 4 * kTileWX + j;
    int code = -1;
#pragma unroll
    for (int x = 0; x < 4; ++x)
        if ((__ldg(w + x * kTileWX) >> b) & 1u)
            code = x;
    return code;
}

constexpr int kTmWarps = 4; // 128 threads: also the block size of exact_site

template <class F> __device__ __forceinline__ float group_reduce(float v, F op)
{
    v = op(v, __shfl_xor_sync(0xffffffffu, v, 1));
    v = op(v, __shfl_xor_sync(0xffffffffu, v, 2));
    return v;
}

// fp64 Tm of oligo `olig` (2-bit codes) against template bases bt, in the
// operation order of the definition: stacks 0..L-2, then the 5' and the 3'
// initiation terms, then the salt entropy, then the ratio; _rn intrinsics so
// nothing is contracted.
__device__ double exact_tm(const PairDev &pd, const int8_t *bt, int L, uint64_t olig)
{
    double H = 0.0, S = 0.0;
    for (int q = 0; q + 1 < L; ++q) {
        const int a = (int)(olig >> (2 * q) & 3u), b = (int)(olig >> (2 * (q + 1)) & 3u);
        const int idx = ((a * 4 + b) * 4 + bt[q]) * 4 + bt[q + 1];
        H = __dadd_rn(H, pd.stack_dH_d[idx]);
        S = __dadd_rn(S, pd.stack_dS_d[idx]);
    }
    const int o0 = (int)(olig & 3u), oL = (int)(olig >> (2 * (L - 1)) & 3u);
    H = __dadd_rn(H, pd.term_dH_d[o0 * 4 + bt[0]]);
    S = __dadd_rn(S, pd.term_dS_d[o0 * 4 + bt[0]]);
    H = __dadd_rn(H, pd.term_dH_d[oL * 4 + bt[L - 1]]);
    S = __dadd_rn(S, pd.term_dS_d[oL * 4 + bt[L - 1]]);
    if (pd.saltcorr == 5)
        S = __dadd_rn(S, __dmul_rn(__dmul_rn(0.368, (double)(L - 1)), pd.log_na));
    double tm = __dsub_rn(__ddiv_rn(__dmul_rn(1000.0, H), __dadd_rn(S, pd.sconst)), 273.15);
    if (pd.saltcorr == 1)
        tm = __dadd_rn(tm, pd.tm_shift);
    return tm;
}

// Oligo number o (0 <= o < degeneracy <= 10000) of a primer with position sets
// qm -> its bases, 2 bits per position (mixed radix over the positions' sets).
__device__ uint64_t oligo_number(const uint8_t *qm, int L, int o)
{
    uint64_t olig = 0;
    int rem = o;
    for (int q = L - 1; q >= 0; --q) {
        const int nqb = __popc(qm[q]);
        int d; // rem % nqb, rem /= nqb for nqb in 1..4 (rem < 10000)
        if (nqb == 1) {
            d = 0;
        } else if (nqb == 2) {
            d = rem & 1;
            rem >>= 1;
        } else if (nqb == 4) {
            d = rem & 3;
            rem >>= 2;
        } else {
            const int q3 = (rem * 43691) >> 17; // rem / 3, exact for rem < 2^16
            d = rem - 3 * q3;
            rem = q3;
        }
        int base_q = 0;
        for (int x = 0; x < 4; ++x)
            if (qm[q] >> x & 1) {
                if (d == 0) {
                    base_q = x;
                    break;
                }
                --d;
            }
        olig |= (uint64_t)base_q << (2 * q);
    }
    return olig;
}

// One queued site with a whole block of kExactThreads: every oligo in fp64
// with the definition's operation order (exact_tm), block-wide maximum, then
// the Tm and the pass flag.  bt and wmax are the block's shared scratch.
constexpr int kExactThreads = 128; // fp64-bound: a block of 128 already keeps the SM's fp64 units busy

__device__ void exact_site(const ah_site *sites, const PairDev *__restrict__ pairs, const uint32_t *__restrict__ planes,
                           const uint64_t *__restrict__ contig_off, uint32_t i, float *tm_out, uint8_t *pass_out,
                           int8_t *bt, double *wmax)
{
    const ah_site s = sites[i];
    const PairDev &pd = pairs[s.pair];
    const int L = pd.L[s.primer];
    const uint8_t *qm = pd.mask[s.primer];
    const uint64_t P = contig_off[s.contig] + s.pos;
    for (int q = threadIdx.x; q < L; q += blockDim.x) {
        const int c = base_at(planes, P + (s.strand == 0 ? q : L - 1 - q));
        bt[q] = (int8_t)(s.strand == 0 ? 3 - c : c); // queued sites have only A/C/G/T
    }
    __syncthreads();
    int deg = 1;
    for (int q = 0; q < L; ++q)
        deg *= __popc(qm[q]);
    double best = -INFINITY;
    for (int o = threadIdx.x; o < deg; o += blockDim.x) {
        const double t = exact_tm(pd, bt, L, oligo_number(qm, L, o));
        best = t > best ? t : best;
    }
    for (int d = 16; d >= 1; d >>= 1) {
        const double o2 = __shfl_xor_sync(0xffffffffu, best, d);
        best = o2 > best ? o2 : best;
    }
    if ((threadIdx.x & 31) == 0)
        wmax[threadIdx.x >> 5] = best;
    __syncthreads();
    if (threadIdx.x == 0) {
        double m = wmax[0];
        for (int w = 1; w < kExactThreads / 32; ++w)
            m = wmax[w] > m ? wmax[w] : m;
        float tm = (float)m;
        if (pass_out) {
            const bool pass = m >= pd.tm_min;
            pass_out[i] = pass;
            if (!pass && tm >= pd.tm_min_f) // rounding to fp32 may reach the threshold: stay below it
                tm = nextafterf(pd.tm_min_f, -INFINITY);
        }
        tm_out[i] = tm;
    }
    __syncthreads(); // bt and wmax are reused by the next queued site
}

// Queued sites, one block per site (tables under which many sites may queue).
// The queue length is read on the device.
__global__ void __launch_bounds__(kExactThreads) tm_exact_kernel(const ah_site *__restrict__ sites,
                                                                 const PairDev *__restrict__ pairs,
                                                                 const uint32_t *__restrict__ planes,
                                                                 const uint64_t *__restrict__ contig_off,
                                                                 const uint32_t *__restrict__ queue,
                                                                 const uint32_t *__restrict__ queue_n,
                                                                 float *__restrict__ tm_out,
                                                                 uint8_t *__restrict__ pass_out)
{
    __shared__ int8_t bt[AH_MAX_PRIMER_LEN];
    __shared__ double wmax[kExactThreads / 32];
    const uint32_t nq = *queue_n;
    for (uint32_t e = blockIdx.x; e < nq; e += gridDim.x)
        exact_site(sites, pairs, planes, contig_off, queue[e], tm_out, pass_out, bt, wmax);
}

// Per-pair constants of the fp32 path, staged in shared memory by every
// block (the shortest-path steps read them in dependent chains).
struct TmPairS {
    float2 st[256]; // (dH, dS) of each stack, [oligo pair o0 + 4 o1][template pair t0 + 4 t1]
    float2 tm[16];  // of each terminal pair, [oligo base][template base]
    uint64_t first[2];      // lowest base of each position's set, 2 bits each
    uint32_t allowed[2][4]; // per base, bit i: it is in key i's set
    uint8_t key[2][AH_MAX_PRIMER_LEN]; // key positions (both ends and every degenerate one), ascending
    int L[2], nkey[2];
    float cst[2]; // C + salt entropy
    float tm_min_f, tm_shift_f;
};
static_assert(sizeof(TmPairS) % 16 == 0, "TmPairS keeps 16-byte alignment");

// The entry of a table indexed like PairDev's, o0 o1 t0 t1, in the order of TmPairS.
__device__ __forceinline__ int staged_stack(int t)
{
    return ((t >> 4 & 3) * 4 + (t >> 6)) * 16 + (t & 3) * 4 + (t >> 2 & 3);
}

// The weights 1000 dH - thr dS of every table entry at the pair's threshold
// thr, for the near-threshold sign test: computed in fp64 from the fp64
// table, then held as fixed point (units of 2^-30 cal/mol, int64) so that
// every path sum is exact; staged for up to kTmStageD pairs.
struct TmPairD {
    long long st[256]; // in the order of TmPairS
    long long tm[16];
};
constexpr double kFix = 1073741824.0; // 2^30: fixed-point scale of the sign test
// |each weight's rounding| <= 2^-31 cal/mol, so a path of <= 32 terms is within
// 2e-8 of its exact value; decisions use a margin of 1e-6 cal/mol (file comment)
constexpr long long kFixMargin = 1074; // 1e-6 * 2^30
constexpr int kSweepMax = 64;          // thresholds per sweep (one bit each)

__device__ __forceinline__ long long fix_weight(double dH, double dS, double thr)
{
    return __double2ll_rn((1000.0 * dH - thr * dS) * kFix);
}
// Out of line: the tables of more than kTmStageD pairs, rarely read.
__device__ __noinline__ long long far_weight(double dH, double dS, double thr) { return fix_weight(dH, dS, thr); }
constexpr int kTmStageD = 4;
constexpr unsigned kTmEarlyBlocks = 304; // two per SM
// Entries from one site's segment tables to the next: four more than the tables, so that the
// eight sites of a warp, which read the same entry of their tables, meet different banks.
__host__ __device__ constexpr int tm_group_stride(int seg_max) { return seg_max * 16 + 4; }

// 8 x 8 bit transpose: bit c of byte r -> bit r of byte c
__device__ __forceinline__ uint64_t transpose8(uint64_t x)
{
    uint64_t t = (x ^ (x >> 7)) & 0x00AA00AA00AA00AAull;
    x ^= t ^ (t << 7);
    t = (x ^ (x >> 14)) & 0x0000CCCC0000CCCCull;
    x ^= t ^ (t << 14);
    t = (x ^ (x >> 28)) & 0x00000000F0F0F0F0ull;
    return x ^ t ^ (t << 28);
}

// A site's window in the planes, for a warp that fetches it with one 16-byte load per
// lane: 8 lanes per plane, 4 words each, from the 16-byte boundary below the window.
struct Window {
    uint64_t base;   // byte offset of that boundary in the A plane
    uint32_t o, row; // words from there to the window; the bit of its row
    uint32_t last;   // its last word, from the boundary (at most 31)
};

__device__ __forceinline__ Window window_at(uint64_t P, int L)
{
    const uint32_t w = (uint32_t)(P % kTileBases);
    Window d;
    d.base = 4 * (P / kTileBases * (4 * kTileWX) + (w & (kTileW - 4)));
    d.o = w & 3u;
    d.row = w / kTileW;
    d.last = min(d.o + (uint32_t)L, 32u) - 1u;
    return d;
}

// The load of a lane: plane lane / 8, words 4 (lane % 8) .. + 3.  Lanes past the window
// read its last group again (no other sector).
__device__ __forceinline__ uint4 window_load(const uint32_t *planes, int lane, uint64_t base, uint32_t last_group)
{
    const char *p = reinterpret_cast<const char *>(planes + (lane >> 3) * kTileWX);
    return __ldg(reinterpret_cast<const uint4 *>(p + base + min(16u * (lane & 7), last_group)));
}

// Template codes opposite each primer position (A 0, C 1, G 2, T 3), 2 bits each, from
// the four ballots of a window's row: bit 8 x + g of B[j] = plane x at word 4 g + j.
// ok: every position holds one of the four letters.
__device__ __forceinline__ uint64_t window_codes(const uint32_t *planes, const Window &d, int L, int strand,
                                                 const uint32_t (&B)[4], bool *ok)
{
    uint32_t extra[4] = {0, 0, 0, 0}; // words 32 .. 34 of a long window that starts off the boundary, per plane
    if (d.o + L > 32) {
        const uint32_t *p = planes + (d.base >> 2) + 32;
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
            for (int j = 0; j < 3; ++j)
                if (32u + j < d.o + L)
                    extra[x] |= ((__ldg(p + x * kTileWX + j) >> d.row) & 1u) << j;
    }
    // words outside [o, o + L) cleared; every position has exactly one plane set, or the window is bad
    int set = __popc(extra[0] | extra[1] | extra[2] | extra[3]);
    uint64_t rows = 0; // byte 2 j + h: bit g = bit h of the code at word 4 g + j
#pragma unroll
    for (uint32_t j = 0; j < 4; ++j) {
        // groups whose word 4 g + j is at most `last`: all before last's, and its own up to last
        uint32_t keep = (1u << ((d.last >> 2) + (j <= (d.last & 3u)))) - 1u;
        if (j < d.o)
            keep &= ~1u;
        const uint32_t v = B[j] & keep * 0x01010101u;
        set += __popc(v);
        const uint32_t lo8 = ((v >> 8) | (v >> 24)) & 0xffu, hi8 = ((v >> 16) | (v >> 24)) & 0xffu;
        rows |= (uint64_t)(lo8 | hi8 << 8) << (16 * j);
    }
    uint64_t code = transpose8(rows) >> (2 * d.o);
    if (d.o) { // (o = 0: nothing past word 31)
        const uint64_t elo = extra[1] | extra[3], ehi = extra[2] | extra[3];
#pragma unroll
        for (int j = 0; j < 3; ++j)
            code |= ((elo >> j & 1u) | (ehi >> j & 1u) << 1) << (2 * (32 + j) - 2 * d.o) % 64;
    }
    *ok = set == L;
    if (strand == 0) // the complement of the window base at q
        return ~code;
    code = __brevll(code) >> (64 - 2 * L); // the window base at L - 1 - q
    return (code >> 1 & 0x5555555555555555ull) | (code & 0x5555555555555555ull) << 1;
}

// Four lanes per site: lane y of a group holds the DP state "oligo base at
// the current key position = y".  Each step takes the four predecessor costs
// by shuffles and keeps the best predecessor (2 bits per key), so the argmin
// oligo is recovered by a backtrack across the group's lanes; its dH, dS are
// then summed by the four lanes together.  (Carrying dH and dS of the best
// predecessor along takes two more dependent shuffles per step: 3,650 cycles per
// pass of nine steps instead of 2,520.)  Eight sites per warp, their windows
// fetched together (one 16-byte load per lane and site).
//
// kFew (tables under which only the rare ambiguous sites need the exhaustive
// evaluation, all duplexes having dS + C < 0): a block evaluates its own sites'.
// Else the largest denominator decides whether the iteration applies, and the
// sites for the exhaustive evaluation go to a queue.
//
// Bound: latency (a few sites per warp, dependent loads and shuffles).  Cycles on
// a GB300 for 20 sites, from the wait for the predecessor: 24,000 with the error
// word, the count and the records read one after the other, a window position per
// load, template bases in shared memory, a backtrack per pass and a last block
// that looks for queued sites -> 12,500.
template <bool kFew>
__global__ void __launch_bounds__(32 * kTmWarps) tm_kernel(const ah_site *sites, uint64_t n_arg, const uint64_t *n_dev,
                                                           const PairDev *__restrict__ pairs, int n_pairs,
                                                           const uint32_t *__restrict__ planes,
                                                           const uint64_t *__restrict__ contig_off,
                                                           float *tm_out, uint8_t *pass_out, uint32_t *queue,
                                                           uint32_t *queue_n, int seg_max, int *err,
                                                           const uint32_t *idx_list)
{
    static_assert(32 * kTmWarps == kExactThreads, "a block evaluates its ambiguous sites with exact_site");
    __shared__ uint32_t xq[8 * kTmWarps], xn; // kFew: ambiguous sites of a round
    __shared__ int8_t xbt[AH_MAX_PRIMER_LEN];
    __shared__ double xmax[kTmWarps];
    // dynamic: [n_pairs] TmPairS, [n_pairs <= kTmStageD ? n_pairs : 0] TmPairD,
    // then per site of the block its [seg_max][16] segment tables, tm_group_stride apart
    extern __shared__ __align__(16) unsigned char tm_smem[];
    TmPairS *ps = reinterpret_cast<TmPairS *>(tm_smem);
    chain_start();
    // The first blocks of a launch lay out the tables (which no kernel of the chain writes)
    // while its predecessor runs; the others, and the list form's, learn first whether they
    // have a site.
    const bool early = !idx_list && blockIdx.x < kTmEarlyBlocks;
    if (!early)
        chain_wait();
    const int nd = n_pairs <= kTmStageD ? n_pairs : 0;
    TmPairD *pdd = reinterpret_cast<TmPairD *>(tm_smem + (size_t)n_pairs * sizeof(TmPairS));
    float2 *seg_smem =
        reinterpret_cast<float2 *>(tm_smem + (size_t)n_pairs * sizeof(TmPairS) + (size_t)nd * sizeof(TmPairD));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (!early && (uint64_t)blockIdx.x * kTmWarps * 8 >= dev_count(n_arg, n_dev))
        return;
    for (int j = 0; j < n_pairs; ++j) {
        const PairDev &P = pairs[j];
        for (int t = threadIdx.x; t < 256; t += blockDim.x)
            ps[j].st[staged_stack(t)] = make_float2(P.stack_dH[t], P.stack_dS[t]);
        if (threadIdx.x < 16)
            ps[j].tm[threadIdx.x] = make_float2(P.term_dH[threadIdx.x], P.term_dS[threadIdx.x]);
        if (threadIdx.x == 0) {
            ps[j].tm_min_f = P.tm_min_f;
            ps[j].tm_shift_f = (float)P.tm_shift;
        }
        if (j < nd) {
            for (int t = threadIdx.x; t < 256; t += blockDim.x)
                pdd[j].st[staged_stack(t)] = fix_weight(P.stack_dH_d[t], P.stack_dS_d[t], P.thr);
            if (threadIdx.x < 16)
                pdd[j].tm[threadIdx.x] = fix_weight(P.term_dH_d[threadIdx.x], P.term_dS_d[threadIdx.x], P.thr);
        }
    }
    for (int c = warp; c < 2 * n_pairs; c += kTmWarps) { // a warp per primer, lane q position q
        const PairDev &P = pairs[c >> 1];
        TmPairS &sp = ps[c >> 1];
        const int x = c & 1, L = P.L[x];
        const uint32_t m = lane < L ? P.mask[x][lane] : 0u;
        const bool key = lane < L && (lane == 0 || lane == L - 1 || __popc(m) > 1);
        const uint32_t keys = __ballot_sync(0xffffffffu, key);
        const int at = __popc(keys & ((1u << lane) - 1u));
        uint32_t allowed[4];
#pragma unroll
        for (int b = 0; b < 4; ++b)
            allowed[b] = __reduce_or_sync(0xffffffffu, key ? (m >> b & 1u) << at : 0u);
        if (key)
            sp.key[x][at] = (uint8_t)lane;
        const uint64_t low = lane < L ? (uint64_t)(__ffs(m) - 1) << (2 * lane) : 0ull;
        const uint32_t lo = __reduce_or_sync(0xffffffffu, (uint32_t)low);
        const uint32_t hi = __reduce_or_sync(0xffffffffu, (uint32_t)(low >> 32));
        if (lane == 0) {
            sp.first[x] = (uint64_t)hi << 32 | lo;
#pragma unroll
            for (int b = 0; b < 4; ++b)
                sp.allowed[x][b] = allowed[b];
            sp.L[x] = L;
            sp.nkey[x] = __popc(keys);
            sp.cst[x] = (float)(P.sconst + (P.saltcorr == 5 ? 0.368 * (double)(L - 1) * P.log_na : 0.0));
        }
    }
    if (early)
        chain_wait();
    const int g = lane >> 2, y = lane & 3, g0 = lane & ~3;
    // The error word, the count and the first record (below n_arg, so in its buffer) as loads
    // that wait for none of the others.  With the word set nothing is read with the records, the
    // call reports it (one answer per block: the word may change under it).
    const int bad_word = *(volatile const int *)err;
    const uint64_t n = dev_count(n_arg, n_dev);
    uint64_t first_block = (uint64_t)blockIdx.x * kTmWarps * 8;
    ah_site s0{};
    if (!idx_list && first_block + warp * 8 + g < n_arg)
        s0 = sites[first_block + warp * 8 + g];
    if (__syncthreads_or(bad_word))
        return;
    const float INF = INFINITY;
    const uint64_t step = (uint64_t)gridDim.x * kTmWarps * 8;
    for (uint64_t base0 = first_block; base0 < n; base0 += step) { // all warps of the block together
        const uint64_t base = base0 + warp * 8;
        const bool live = base + g < n;
        // with idx_list, the sites taken are sites[idx_list[0 .. n)]
        const uint64_t i = live && idx_list ? (uint64_t)idx_list[base + g] : base + g;
        ah_site s{};
        if (live)
            s = !idx_list && base0 == first_block ? s0 : sites[i];
        const bool bad_rec = live && (s.pair >= n_pairs || s.primer > 1 || s.strand > 1);
        if (bad_rec && y == 0)
            atomicExch(err, kDevBounds);
        const bool act = live && !bad_rec;
        const int pi = act ? s.pair : 0, x1 = act ? s.primer : 0;
        const PairDev &pd = pairs[pi];
        const TmPairS &sp = ps[pi];
        const int L = sp.L[x1];
        // the group's window (without a live site: the first of the planes, unused)
        Window d{};
        if (act)
            d = window_at(contig_off[s.contig] + s.pos, L);
        uint32_t B[4] = {0, 0, 0, 0};
        {
            uint4 w[8];
#pragma unroll
            for (int j = 0; j < 8; ++j)
                w[j] = window_load(planes, lane, __shfl_sync(0xffffffffu, d.base, 4 * j),
                                   4u * (__shfl_sync(0xffffffffu, d.last, 4 * j) & ~3u));
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const uint32_t bit = 1u << __shfl_sync(0xffffffffu, d.row, 4 * j);
                const uint32_t v0 = __ballot_sync(0xffffffffu, w[j].x & bit);
                const uint32_t v1 = __ballot_sync(0xffffffffu, w[j].y & bit);
                const uint32_t v2 = __ballot_sync(0xffffffffu, w[j].z & bit);
                const uint32_t v3 = __ballot_sync(0xffffffffu, w[j].w & bit);
                if (g == j) {
                    B[0] = v0;
                    B[1] = v1;
                    B[2] = v2;
                    B[3] = v3;
                }
            }
        }
        bool ok = false;
        uint64_t code = 0;
        if (act)
            code = window_codes(planes, d, L, s.strand, B, &ok);
        const bool bad = !ok, run = act && ok;
        const float cst = sp.cst[x1];
        // Steps at key positions only (primer positions 0 and L-1 and every
        // degenerate one): between two keys the oligo bases are fixed, so all
        // stacks from key i to key i+1 form a 4x4 table of (dH, dS) sums
        // indexed by the bases at the two keys, E[i][a * 4 + b].  Lane y fills
        // column y of the site's tables once; every pass below reads them.
        const uint8_t *key = sp.key[x1];
        const uint64_t first = sp.first[x1];
        const int m = run ? sp.nkey[x1] - 1 : 0; // segments
        // Shuffles need all 32 lanes, but the groups' segment counts differ: every
        // segment loop runs to the warp's largest count mw and each group only
        // updates its state while si < m.
        const int mw = (int)__reduce_max_sync(0xffffffffu, (uint32_t)m);
        auto oligo2 = [&](int q) { return (int)(first >> (2 * q)) & 15; }; // fixed bases at q and q + 1
        auto templ2 = [&](int q) { return (int)(code >> (2 * q)) & 15; };  // template bases at q and q + 1
        float2 *E = seg_smem + (warp * 8 + g) * tm_group_stride(seg_max);
        for (int sb = 0; sb < mw; sb += 4) {
            // the stacks between two fixed bases: lane y sums those of segment sb + y
            float cH = 0.f, cS = 0.f;
            if (sb + y < m) {
                const int k1 = key[sb + y + 1];
#pragma unroll 4
                for (int q = key[sb + y] + 1; q < k1 - 1; ++q) {
                    const float2 e = sp.st[oligo2(q) * 16 + templ2(q)];
                    cH += e.x;
                    cS += e.y;
                }
            }
#pragma unroll 1
            for (int u = 0; u < 4; ++u) {
                const float uH = __shfl_sync(0xffffffffu, cH, g0 + u), uS = __shfl_sync(0xffffffffu, cS, g0 + u);
                const int si = sb + u;
                if (si < m) {
                    const int k0 = key[si], k1 = key[si + 1], p0 = templ2(k0);
                    const bool apart = k1 > k0 + 1; // else one stack from x to y
                    const int fa = oligo2(k0 + 1) & 3, fb = oligo2(k1 - 1) & 3;
                    const float2 eq = sp.st[(fb + 4 * y) * 16 + templ2(k1 - 1)]; // into key k1, base y
                    const float qH = apart ? eq.x + uH : 0.f, qS = apart ? eq.y + uS : 0.f;
                    const int to = apart ? fa : y;
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        const float2 ep = sp.st[(x + 4 * to) * 16 + p0]; // out of key k0, base x
                        E[si * 16 + x * 4 + y] = make_float2(ep.x + qH, ep.y + qS);
                    }
                }
            }
        }
        // bit i: base y is allowed at key i; this lane's terminal terms at both ends
        const uint32_t amask = run ? sp.allowed[x1][y] : 0u;
        const int tF = (int)code & 3, tE = (int)(code >> (2 * (L - 1))) & 3;
        const float2 t0 = run ? sp.tm[y * 4 + tF] : make_float2(0.f, 0.f);
        const float2 tL = run ? sp.tm[y * 4 + tE] : make_float2(0.f, 0.f);
        __syncwarp(); // the group's tables
        bool dink = run;
        if (!kFew) { // largest denominator over oligos (max-path of dS)
            float sm = (amask & 1u) ? t0.y : -INF;
            for (int si = 0; si < mw; ++si) {
                const bool in = run && si < m;
                float best = -INF;
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const float cx = __shfl_sync(0xffffffffu, sm, g0 + x);
                    if (in) {
                        const float v = cx + E[si * 16 + x * 4 + y].y;
                        best = v > best ? v : best;
                    }
                }
                if (in)
                    sm = (amask >> (si + 1) & 1u) ? best : -INF;
            }
            float dm = sm + ((amask >> m & 1u) ? tL.y : 0.f);
            dm = group_reduce(dm, [](float a, float b) { return a > b ? a : b; });
            dink = run && dm + cst < 0.f;
        }
        float lam = 320.f; // any start gives an oligo; near annealing temperatures mostly the best one
        for (int it = 0; it < 64; ++it) {
            // min over oligos of 1000 dH - lam dS, with the best predecessor at every key
            float c = (dink && (amask & 1u)) ? fmaf(-lam, t0.y, 1000.f * t0.x) : INF;
            uint64_t pred = 0;
            for (int si = 0; si < mw; ++si) {
                float v[4]; // (past its own segments a group reads entries that it then leaves alone)
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const float2 e = E[si * 16 + x * 4 + y];
                    v[x] = __shfl_sync(0xffffffffu, c, g0 + x) + fmaf(-lam, e.y, 1000.f * e.x);
                }
                const bool b1 = v[1] < v[0], b3 = v[3] < v[2]; // ties: the lowest base
                const float lo = b1 ? v[1] : v[0], hi = b3 ? v[3] : v[2];
                const bool bh = hi < lo;
                const uint32_t arg = bh ? (b3 ? 3u : 2u) : (b1 ? 1u : 0u);
                if (si < m) {
                    c = dink && (amask >> (si + 1) & 1u) ? (bh ? hi : lo) : INF;
                    pred |= (uint64_t)arg << (2 * si);
                }
            }
            const float fin = dink && c < INF ? c + fmaf(-lam, tL.y, 1000.f * tL.x) : INF;
            // argmin over the group's four end states (ties: lowest base)
            const float fmin = group_reduce(fin, [](float a, float b) { return a < b ? a : b; });
            const unsigned hit = __ballot_sync(0xffffffffu, fin == fmin) >> g0 & 0xFu;
            int cur = hit ? __ffs(hit) - 1 : 0;
            const int last = cur;
            // backtrack the bases at the keys: ks[i] = base at key i (2 bits each)
            uint64_t ks = (uint64_t)cur << (2 * m);
            for (int si = mw - 1; si >= 0; --si) {
                const uint64_t pp = __shfl_sync(0xffffffffu, pred, g0 + cur);
                if (si < m) {
                    cur = (int)(pp >> (2 * si) & 3u);
                    ks |= (uint64_t)cur << (2 * si);
                }
            }
            // its dH and dS: the segment tables, split over the four lanes
            float H = 0.f, S = 0.f;
            if (dink)
                for (int si = y; si < m; si += 4) {
                    const float2 e = E[si * 16 + (int)(ks >> (2 * si) & 3u) * 4 + (int)(ks >> (2 * (si + 1)) & 3u)];
                    H += e.x;
                    S += e.y;
                }
            H = group_reduce(H, [](float a, float b) { return a + b; });
            S = group_reduce(S, [](float a, float b) { return a + b; });
            // terminal terms of the chosen end bases: held by the lanes of those bases
            H += __shfl_sync(0xffffffffu, t0.x, g0 + cur) + __shfl_sync(0xffffffffu, tL.x, g0 + last);
            S += __shfl_sync(0xffffffffu, t0.y, g0 + cur) + __shfl_sync(0xffffffffu, tL.y, g0 + last);
            const float r = 1000.f * H / (S + cst);
            // Warp-uniform loop: stop when no group still improves by more than
            // 1e-4 K.  In fp32 two oligos of nearly equal ratio could otherwise
            // trade places by one ulp for many rounds; 1e-4 K is far below the
            // 0.01 deg C tolerance, and sites near tm_min are decided exactly below.
            const bool more = dink && (it == 0 || r > lam + 1e-4f);
            if (more)
                lam = r;
            if (!__any_sync(0xffffffffu, more))
                break;
        }
        const float tm32 = lam - 273.15f + sp.tm_shift_f;
        // near the threshold: the sign of min F at lam = thr, in fp64 (file comment)
        const bool near = dink && pass_out && fabsf(tm32 - sp.tm_min_f) < 0.01f;
        int decided = -1; // 1 pass, 0 fail, -1 undecided
        if (__any_sync(0xffffffffu, near)) {
            // Same key segments, exact fixed-point weights at lam = thr.  First every
            // weight W[i][x] of this lane's column (independent work, written over the
            // fp32 tables, no longer needed), then the dependent chain over the segments.
            const long long LINF = 0x2000000000000000ll; // above any path sum, no overflow when added to
            long long *W = reinterpret_cast<long long *>(E); // W[si * 16 + x * 4 + y], 8 bytes per float2 slot
            const bool staged = pi < nd;
            const TmPairD &sd = pdd[staged ? pi : 0];
            auto stW = [&](int o2, int t2) { // oligo and template pairs, as in TmPairS
                if (staged)
                    return sd.st[o2 * 16 + t2];
                const int idx = (((o2 & 3) * 4 + (o2 >> 2)) * 4 + (t2 & 3)) * 4 + (t2 >> 2);
                return far_weight(pd.stack_dH_d[idx], pd.stack_dS_d[idx], pd.thr);
            };
            auto tmW = [&](int idx) {
                return staged ? sd.tm[idx] : far_weight(pd.term_dH_d[idx], pd.term_dS_d[idx], pd.thr);
            };
            __syncwarp();
            // (as the fp32 tables above; loops left rolled: a warp comes here once, and fetching
            // unrolled code cost more than running it, 14,000 cycles against 5,000)
            for (int sb = 0; sb < mw; sb += 4) {
                long long cw = 0;
                if (near && sb + y < m) {
                    const int k1 = key[sb + y + 1];
#pragma unroll 1
                    for (int q = key[sb + y] + 1; q < k1 - 1; ++q)
                        cw += stW(oligo2(q), templ2(q));
                }
#pragma unroll 1
                for (int u = 0; u < 4; ++u) {
                    const long long uw = __shfl_sync(0xffffffffu, cw, g0 + u);
                    const int si = sb + u;
                    if (near && si < m) {
                        const int k0 = key[si], k1 = key[si + 1], p0 = templ2(k0);
                        const bool apart = k1 > k0 + 1;
                        const int fa = oligo2(k0 + 1) & 3, fb = oligo2(k1 - 1) & 3;
                        const long long into = apart ? stW(fb + 4 * y, templ2(k1 - 1)) + uw : 0;
                        const int to = apart ? fa : y;
#pragma unroll 1
                        for (int x = 0; x < 4; ++x)
                            W[si * 16 + x * 4 + y] = stW(x + 4 * to, p0) + into;
                    }
                }
            }
            __syncwarp();
            long long cd = (near && (amask & 1u)) ? tmW(y * 4 + tF) : LINF;
            for (int si = 0; si < mw; ++si) {
                long long best = LINF;
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const long long cx = __shfl_sync(0xffffffffu, cd, g0 + x);
                    const long long v = cx < LINF ? cx + W[si * 16 + x * 4 + y] : LINF;
                    best = v < best ? v : best;
                }
                if (near && si < m)
                    cd = (amask >> (si + 1) & 1u) ? best : LINF;
            }
            long long fin = cd < LINF ? cd + tmW(y * 4 + tE) : LINF;
            long long o1 = __shfl_xor_sync(0xffffffffu, fin, 1);
            fin = o1 < fin ? o1 : fin;
            o1 = __shfl_xor_sync(0xffffffffu, fin, 2);
            fin = o1 < fin ? o1 : fin;
            if (near) {
                // min F = min path sum - thr (C + salt entropy)
                const double Cp = pd.sconst + (pd.saltcorr == 5 ? 0.368 * (double)(L - 1) * pd.log_na : 0.0);
                const long long F = fin - __double2ll_rn(pd.thr * Cp * kFix);
                decided = F < -kFixMargin ? 1 : (F > kFixMargin ? 0 : -1);
            }
        }
        // sites decided the reference way (see the file comment): kFew by this block below,
        // else by tm_exact_kernel, a whole block per site
        const bool exact = run && (!dink || (near && decided < 0));
        if (!kFew && exact && y == 0)
            queue[atomicAdd(queue_n, 1u)] = (uint32_t)i;
        if (y == 0 && act) {
            float tm = NAN;
            uint8_t pass = 0;
            if (!bad) {
                tm = tm32; // replaced by the exact evaluation for the sites it decides
                pass = tm32 >= sp.tm_min_f;
                if (decided >= 0) { // the exact decision; the fp32 value (within 1e-3) made consistent with it
                    pass = (uint8_t)decided;
                    if (decided && tm < sp.tm_min_f)
                        tm = sp.tm_min_f;
                    if (!decided && tm >= sp.tm_min_f)
                        tm = nextafterf(sp.tm_min_f, -INFINITY);
                }
            }
            tm_out[i] = tm;
            if (pass_out)
                pass_out[i] = pass;
        } else if (y == 0 && bad_rec) {
            tm_out[i] = NAN;
            if (pass_out)
                pass_out[i] = 0;
        }
        __syncwarp();
        if (kFew && __syncthreads_or(exact)) {
            if (threadIdx.x == 0)
                xn = 0;
            __syncthreads();
            if (exact && y == 0)
                xq[atomicAdd(&xn, 1u)] = (uint32_t)i;
            __syncthreads();
            const uint32_t nx = xn;
            for (uint32_t k = 0; k < nx; ++k)
                exact_site(sites, pairs, planes, contig_off, xq[k], tm_out, pass_out, xbt, xmax);
        }
    }
}

// ---------------------------------------------------------------------------
// Thread-per-site Tm (the path taken when every pair has few_exact).  The same
// maximum as tm_kernel -- Dinkelbach iteration on the key-position shortest
// path, fp32 -- but one thread carries all states of one site: each state keeps
// its path cost and the path's dH and dS sums, so the argmin oligo's terms come
// out of the forward pass without a backtrack.  Between two keys that are not
// adjacent the segment's table is separable (the stack out of key k0 depends
// only on the base at k0, the stack into key k1 only on the base at k1, the
// fixed stretch between them on neither), so one argmin over the predecessors
// serves all successors.  Sites whose maximum lies within 0.01 deg C of tm_min are
// deferred to tm_kernel (which decides them exactly); everything else is
// written here.
//
// A block takes up to kFastBatch sites at a time.  Gather: a warp fetches a
// site's window with one 16-byte load per lane (8 lanes per plane, 4 words each,
// from the 16-byte boundary below the window) and four ballots; each lane unpacks
// its own site's ballots into 2-bit template codes.  Sort: the block lists its
// sites by primer and its warps claim 32 of one primer at a time: a primer's path
// is a list of steps (its keys, and the table offsets of the bases each allows)
// that all lanes follow together, so no branch diverges and bases outside a set
// are not visited; steps between sets of one or two bases, all but the few with
// three or four, run without a test.  (Sites in canonical order mix both primers
// in every warp.)  Bound: issue slots.  Measured on a GB300, 3.3 M sites of three
// pairs: 727 us with sites in order, four loads per site and all 16 transitions ->
// 419 us; 0.94 M sites of two pairs 243 -> 145 us.
// ---------------------------------------------------------------------------
constexpr int kFastThreads = 256;
constexpr int kFastBatch = 1024;                        // sites of a block between two barriers, at most
constexpr int kFastClasses = 2 * AH_MAX_PAIRS_PER_SCAN; // pair * 2 + primer
constexpr int kFastChunks = kFastBatch / 32 + kFastClasses; // groups of 32 sites of one class, at most
static_assert(kFastClasses == 32, "one lane per class");

// One step of a primer's path, from key k0 to the next key k1.  Sets of one or two
// bases at both: byte offsets of the stack table's rows for the two bases x at k0
// and y at k1, in ascending order (a single base stands twice).
struct TmStep {
    uint8_t sh0, sh1;     // 2 k0, 2 (k1 - 1): the template pairs (k0, k0 + 1) and (k1 - 1, k1)
    uint8_t n0, n1;       // bases at k0 and at k1
    uint16_t off[4];      // k1 = k0 + 1: [2 x + y]; else out of k0 [x], then into k1 [2 + y]
    uint8_t list0, list1; // the bases, ascending, 2 bits each
    uint8_t fixed;        // the fixed bases at k0 + 1 and (<< 2) k1 - 1
    uint8_t kind;         // 1: k1 > k0 + 1, 2: a set of three or four bases at either key
};
static_assert(sizeof(TmStep) == 16, "a step is one 16-byte load");

struct TmFastPrimer {
    TmStep step[AH_MAX_PRIMER_LEN - 1];
    uint64_t has[4]; // bit 2 q: the base is in position q's set
    uint64_t first;  // the lowest base of each set
    uint32_t fixes;  // bit q: positions q and q + 1 lie between two keys
    int n_step, L;
    int nF, listF, nL, listL; // the sets at both ends
    float cst;                // C + salt entropy
    int pad[2];
};
// Per pair: stacks as (1000 dH, dS), a row per oligo pair o0 + 4 o1, indexed by the
// template pair t0 + 4 t1: lanes that read one row at their own template pairs meet
// no bank twice (a row per template pair puts all lanes of such a read into one
// bank: 234 us on the 0.94 M sites).  Terminal pairs [oligo base][template base].
struct TmFastPair {
    float2 st[256];
    float2 tm[16];
    TmFastPrimer pr[2];
    float tm_min_f, tm_shift_f, pad[2];
};
static_assert(sizeof(TmFastPair) % 16 == 0 && offsetof(TmFastPair, pr) % 16 == 0 && sizeof(TmFastPrimer) % 16 == 0,
              "steps keep 16-byte alignment");

// One warp builds a primer's steps: lane q holds position q.
__device__ __forceinline__ void tm_fast_primer(TmFastPrimer &F, const PairDev &P, int x, int lane)
{
    const int L = P.L[x];
    const uint32_t m = lane < L ? P.mask[x][lane] : 0u;
    const bool key = lane < L && (lane == 0 || lane == L - 1 || __popc(m) > 1);
    const uint32_t keys = __ballot_sync(0xffffffffu, key), below = keys & ((1u << lane) - 1u);
    const uint32_t fixed = __ballot_sync(0xffffffffu, lane < L && !key);
    uint32_t list = 0; // ascending, 2 bits each
    for (int b = 3; b >= 0; --b)
        if (m >> b & 1u)
            list = list << 2 | (uint32_t)b;
    const int k0 = below ? 31 - __clz(below) : 0;
    const int cnt = __popc(m);
    const uint32_t list0 = __shfl_sync(0xffffffffu, list, k0);
    const int cnt0 = __shfl_sync(0xffffffffu, cnt, k0);
    const uint32_t fa = __shfl_sync(0xffffffffu, list, (k0 + 1) & 31) & 3u;
    const uint32_t fb = __shfl_sync(0xffffffffu, list, (lane - 1) & 31) & 3u;
    if (key && lane > 0) {
        TmStep s{};
        s.sh0 = (uint8_t)(2 * k0);
        s.sh1 = (uint8_t)(2 * (lane - 1));
        s.n0 = (uint8_t)cnt0;
        s.n1 = (uint8_t)cnt;
        s.list0 = (uint8_t)list0;
        s.list1 = (uint8_t)list;
        s.fixed = (uint8_t)(fa | fb << 2);
        const bool apart = lane > k0 + 1;
        s.kind = (uint8_t)((apart ? 1 : 0) | (cnt0 > 2 || cnt > 2 ? 2 : 0));
        const uint32_t a0 = list0 & 3u, a1 = cnt0 > 1 ? list0 >> 2 & 3u : a0;
        const uint32_t c0 = list & 3u, c1 = cnt > 1 ? list >> 2 & 3u : c0;
        s.off[0] = (uint16_t)(128 * (apart ? a0 + 4 * fa : a0 + 4 * c0));
        s.off[1] = (uint16_t)(128 * (apart ? a1 + 4 * fa : a0 + 4 * c1));
        s.off[2] = (uint16_t)(128 * (apart ? fb + 4 * c0 : a1 + 4 * c0));
        s.off[3] = (uint16_t)(128 * (apart ? fb + 4 * c1 : a1 + 4 * c1));
        F.step[__popc(below) - 1] = s;
    }
    uint64_t bits = lane < L ? (uint64_t)(list & 3u) << (2 * lane) : 0ull;
    const uint32_t flo = __reduce_or_sync(0xffffffffu, (uint32_t)bits), fhi = __reduce_or_sync(0xffffffffu, (uint32_t)(bits >> 32));
    for (int b = 0; b < 4; ++b) {
        bits = (uint64_t)(m >> b & 1u) << (2 * lane);
        const uint32_t lo = __reduce_or_sync(0xffffffffu, (uint32_t)bits), hi = __reduce_or_sync(0xffffffffu, (uint32_t)(bits >> 32));
        if (lane == b)
            F.has[b] = (uint64_t)hi << 32 | lo;
    }
    if (lane == 0) {
        F.first = (uint64_t)fhi << 32 | flo;
        F.fixes = fixed & fixed >> 1;
        F.n_step = __popc(keys) - 1;
        F.L = L;
        F.nF = cnt;
        F.listF = (int)list;
        F.cst = (float)(P.sconst + (P.saltcorr == 5 ? 0.368 * (double)(L - 1) * P.log_na : 0.0));
    }
    if (lane == L - 1) {
        F.nL = cnt;
        F.listL = (int)list;
    }
}

__global__ void __launch_bounds__(kFastThreads, 4) tm_fast_kernel(const ah_site *__restrict__ sites, uint64_t n_arg,
                                                                  const uint64_t *__restrict__ n_dev,
                                                                  const PairDev *__restrict__ pairs, int n_pairs,
                                                                  const uint32_t *__restrict__ planes,
                                                                  const uint64_t *__restrict__ contig_off,
                                                                  float *__restrict__ tm_out,
                                                                  uint8_t *__restrict__ pass_out,
                                                                  uint32_t *__restrict__ defer,
                                                                  unsigned long long *__restrict__ defer_n,
                                                                  int *__restrict__ err)
{
    extern __shared__ __align__(16) unsigned char fast_smem[];
    TmFastPair *fp = reinterpret_cast<TmFastPair *>(fast_smem);
    __shared__ uint64_t win[kFastThreads];                 // byte offset of a window's 16-byte boundary in the A plane
    __shared__ uint32_t win_last[kFastThreads];            // byte offset of its last 16-byte group from there
    __shared__ uint32_t win_bit[kFastThreads];             // the bit of its row
    __shared__ uint4 got[kFastThreads];                    // its ballots: bit 8 x + g of word j = plane x at word 4 g + j
    __shared__ uint64_t codes[kFastBatch];                 // template codes of the batch's sites, 2 bits each
    __shared__ uint16_t list[kFastChunks * 32];            // its sites by class, each class padded to 32
    __shared__ uint32_t cnt[kFastClasses], first[kFastClasses]; // sites of a class; its first entry in list
    __shared__ uint8_t chunk_class[kFastChunks];
    __shared__ int n_chunks, next_chunk;
    const uint64_t n = dev_count(n_arg, n_dev);
    if ((uint64_t)blockIdx.x * blockDim.x >= n || __syncthreads_or(*(volatile const int *)err))
        return; // the whole block: no site for it, or records that failed their check
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int j = 0; j < n_pairs; ++j) {
        const PairDev &P = pairs[j];
        for (int t = threadIdx.x; t < 256; t += blockDim.x) {
            const int o0 = t >> 6, o1 = (t >> 4) & 3, t0 = (t >> 2) & 3, t1 = t & 3; // PairDev index order
            fp[j].st[((o1 * 4 + o0) * 4 + t1) * 4 + t0] = make_float2(1000.f * P.stack_dH[t], P.stack_dS[t]);
        }
        if (threadIdx.x < 16)
            fp[j].tm[threadIdx.x] = make_float2(1000.f * P.term_dH[threadIdx.x], P.term_dS[threadIdx.x]);
        if (threadIdx.x == 0) {
            fp[j].tm_min_f = P.tm_min_f;
            fp[j].tm_shift_f = (float)P.tm_shift;
        }
    }
    for (int c = warp; c < 2 * n_pairs; c += kFastThreads / 32)
        tm_fast_primer(fp[c >> 1].pr[c & 1], pairs[c >> 1], c & 1, lane);
    const float INF = INFINITY;
    constexpr uint32_t kNone = ~0u;
    // an equal share per block (the blocks that start: one per 256 sites, at most the grid), in equal batches
    const uint64_t blocks = min((uint64_t)gridDim.x, (n + kFastThreads - 1) / kFastThreads);
    const uint64_t share = (n + blocks - 1) / blocks;
    const uint64_t lo = min(n, blockIdx.x * share), hi = min(n, lo + share);
    const uint64_t rounds = (share + kFastBatch - 1) / kFastBatch;
    const uint32_t batch = (uint32_t)((share + rounds - 1) / rounds + 31) & ~31u;
    for (uint64_t b0 = lo; b0 < hi; b0 += batch) {
        const uint32_t here = (uint32_t)min((uint64_t)batch, hi - b0);
        __syncthreads(); // the tables; the previous batch's lists are no longer read
        if (threadIdx.x < kFastClasses)
            cnt[threadIdx.x] = 0;
        __syncthreads();
        uint32_t slot[kFastBatch / kFastThreads]; // class << 16 | rank in it, of this lane's sites; kNone
#pragma unroll
        for (int r = 0; r < kFastBatch / kFastThreads; ++r) {
            const uint32_t local = r * kFastThreads + threadIdx.x;
            slot[r] = kNone;
            if (r * kFastThreads + 32 * warp >= here) // the whole warp
                continue;
            // ---- gather
            const uint64_t i = b0 + local;
            const bool live = local < here;
            ah_site s{};
            if (live)
                s = sites[i];
            const bool bad_rec = live && (s.pair >= n_pairs || s.primer > 1 || s.strand > 1);
            if (bad_rec)
                atomicExch(err, kDevBounds);
            const bool act = live && !bad_rec;
            const int L = act ? fp[s.pair].pr[s.primer].L : 1;
            Window d{};
            if (act)
                d = window_at(contig_off[s.contig] + s.pos, L);
            __syncwarp();
            win[threadIdx.x] = d.base;
            win_last[threadIdx.x] = 4u * (d.last & ~3u);
            win_bit[threadIdx.x] = 1u << d.row;
            __syncwarp();
            const uint32_t actm = __ballot_sync(0xffffffffu, act);
            for (int k0 = 0; k0 < 32; k0 += 8) { // eight sites' loads in flight
                if (!((actm >> k0) & 0xffu))
                    continue;
                uint4 w[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int k = 32 * warp + k0 + j;
                    w[j] = window_load(planes, lane, win[k], win_last[k]);
                }
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const uint32_t bit = win_bit[32 * warp + k0 + j];
                    const uint32_t v0 = __ballot_sync(0xffffffffu, w[j].x & bit);
                    const uint32_t v1 = __ballot_sync(0xffffffffu, w[j].y & bit);
                    const uint32_t v2 = __ballot_sync(0xffffffffu, w[j].z & bit);
                    const uint32_t v3 = __ballot_sync(0xffffffffu, w[j].w & bit);
                    if (lane == k0 + j)
                        got[threadIdx.x] = make_uint4(v0, v1, v2, v3);
                }
            }
            // ---- this lane's site
            int cls = -1;
            if (act) {
                const uint4 b4 = got[threadIdx.x];
                const uint32_t B[4] = {b4.x, b4.y, b4.z, b4.w};
                bool ok;
                codes[local] = window_codes(planes, d, L, s.strand, B, &ok);
                if (ok)
                    cls = s.pair * 2 + s.primer;
            }
            if (live && cls < 0) { // a letter other than A, C, G, T, or a record outside its bounds
                tm_out[i] = NAN;
                if (pass_out)
                    pass_out[i] = 0;
            }
            // its rank in its class
            const uint32_t same = __match_any_sync(0xffffffffu, cls);
            uint32_t at = 0;
            if (cls >= 0 && lane == __ffs(same) - 1)
                at = atomicAdd(&cnt[cls], (uint32_t)__popc(same));
            at = __shfl_sync(0xffffffffu, at, __ffs(same) - 1) + __popc(same & ((1u << lane) - 1u));
            if (cls >= 0)
                slot[r] = (uint32_t)cls << 16 | at;
        }
        // ---- the batch's sites by class
        __syncthreads();
        if (warp == 0) {
            const uint32_t chunks = (cnt[lane] + 31) / 32;
            uint32_t incl = chunks;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, incl, d);
                if (lane >= d)
                    incl += y;
            }
            first[lane] = (incl - chunks) * 32;
            for (uint32_t c = incl - chunks; c < incl; ++c)
                chunk_class[c] = (uint8_t)lane;
            if (lane == 31) {
                n_chunks = (int)incl;
                next_chunk = 0;
            }
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kFastBatch / kFastThreads; ++r)
            if (slot[r] != kNone)
                list[first[slot[r] >> 16] + (slot[r] & 0xffffu)] = (uint16_t)(r * kFastThreads + threadIdx.x);
        __syncthreads();
        // ---- 32 sites of one primer per warp
        for (;;) {
            int ch = 0;
            if (lane == 0)
                ch = atomicAdd(&next_chunk, 1);
            ch = __shfl_sync(0xffffffffu, ch, 0);
            if (ch >= n_chunks)
                break;
            const int c = chunk_class[ch];
            const TmFastPair &sp = fp[c >> 1];
            const TmFastPrimer &F = sp.pr[c & 1];
            if ((uint32_t)(ch * 32 + lane) >= first[c] + cnt[c])
                continue; // padding
            const uint32_t local = list[ch * 32 + lane];
            const uint64_t code = codes[local];
            const char *st = reinterpret_cast<const char *>(sp.st);
            // the stack table's column of the template pair at shift sh
            auto column = [&](uint32_t sh) { return st + (((uint32_t)(code >> sh) & 15u) << 3); };
            auto entry = [](const char *E, uint32_t off) { return *reinterpret_cast<const float2 *>(E + off); };
            const int L = F.L, n_step = F.n_step;
            const float2 *tF = sp.tm + ((uint32_t)code & 3u), *tL = sp.tm + ((uint32_t)(code >> (2 * (L - 1))) & 3u);
            const float cst = F.cst;
            // What does not depend on lam, once per site.  The fixed stretches
            // between keys that are not adjacent are the same for every oligo: they
            // add one constant to every path, move no argmin, and join H and S at
            // the end.  The start is an achieved ratio, that of one oligo: at each
            // position the base pairing with the template where the set allows it,
            // else the set's lowest base (for about nine sites in ten the best oligo).
            // Each pass then either confirms the ratio (no oligo beats it by more
            // than 1e-4 K) or moves to a better one.
            float SH = 0.f, SE = 0.f, lam;
            {
                const uint64_t pairing = ~code, one = 0x5555555555555555ull, plo = pairing & one, phi = pairing >> 1 & one;
                const uint64_t in = (F.has[0] & ~(plo | phi)) | (F.has[1] & plo & ~phi) | (F.has[2] & phi & ~plo) |
                                    (F.has[3] & plo & phi);
                const uint64_t m = in | in << 1, oligo = (pairing & m) | (F.first & ~m);
                float2 t = tF[((uint32_t)oligo & 3u) * 4];
                float H0 = t.x, S0 = t.y;
                const uint32_t fixes = F.fixes;
                for (int q = 0; q + 1 < L; ++q) {
                    const float2 v = entry(column(2 * q), ((uint32_t)(oligo >> (2 * q)) & 15u) << 7);
                    H0 += v.x;
                    S0 += v.y;
                    if (fixes >> q & 1u) {
                        SH += v.x;
                        SE += v.y;
                    }
                }
                t = tL[((uint32_t)(oligo >> (2 * (L - 1))) & 3u) * 4];
                lam = (H0 + t.x) / (S0 + t.y + cst);
            }
            for (int it = 0; it < 64; ++it) {
                // forward pass at lam: per base of the current key's set (ascending) the
                // cheapest path cost 1000 dH - lam dS and that path's 1000 dH and dS
                // (fixed stretches left out)
                float cc[4], h[4], e[4];
#pragma unroll
                for (int y = 0; y < 4; ++y) {
                    cc[y] = INF;
                    h[y] = e[y] = 0.f;
                    if (y < F.nF) {
                        const float2 t = tF[(F.listF >> (2 * y) & 3) * 4];
                        cc[y] = fmaf(-lam, t.y, t.x);
                        h[y] = t.x;
                        e[y] = t.y;
                    }
                }
                for (int si = 0; si < n_step; ++si) {
                    const uint4 d4 = *reinterpret_cast<const uint4 *>(&F.step[si]);
                    const uint32_t sh0 = d4.x & 63u, sh1 = d4.x >> 8 & 63u;
                    const uint32_t off0 = d4.y & 0xffffu, off1 = d4.y >> 16, off2 = d4.z & 0xffffu, off3 = d4.z >> 16;
                    const uint32_t kind = d4.w >> 24, apart = kind & 1u;
                    if (kind < 2u) {
                        if (!apart) {
                            const char *E = column(sh0);
                            const float2 e00 = entry(E, off0), e01 = entry(E, off1), e10 = entry(E, off2), e11 = entry(E, off3);
                            const float v00 = cc[0] + fmaf(-lam, e00.y, e00.x), v10 = cc[1] + fmaf(-lam, e10.y, e10.x);
                            const float v01 = cc[0] + fmaf(-lam, e01.y, e01.x), v11 = cc[1] + fmaf(-lam, e11.y, e11.x);
                            const bool p0 = v10 < v00, p1 = v11 < v01;
                            const float h0 = h[0], h1 = h[1], s0 = e[0], s1 = e[1];
                            cc[0] = p0 ? v10 : v00;
                            cc[1] = p1 ? v11 : v01;
                            h[0] = (p0 ? h1 : h0) + (p0 ? e10.x : e00.x);
                            h[1] = (p1 ? h1 : h0) + (p1 ? e11.x : e01.x);
                            e[0] = (p0 ? s1 : s0) + (p0 ? e10.y : e00.y);
                            e[1] = (p1 ? s1 : s0) + (p1 ? e11.y : e01.y);
                        } else {
                            // the stack out of k0 into the fixed base after it: one argmin over
                            // the bases at k0, shared by every y; then the stack into k1
                            const char *EA = column(sh0), *EB = column(sh1);
                            const float2 a0 = entry(EA, off0), a1 = entry(EA, off1), q0 = entry(EB, off2), q1 = entry(EB, off3);
                            const float v0 = cc[0] + fmaf(-lam, a0.y, a0.x), v1 = cc[1] + fmaf(-lam, a1.y, a1.x);
                            const bool p = v1 < v0;
                            const float best = p ? v1 : v0;
                            const float bh = (p ? h[1] : h[0]) + (p ? a1.x : a0.x);
                            const float be = (p ? e[1] : e[0]) + (p ? a1.y : a0.y);
                            cc[0] = best + fmaf(-lam, q0.y, q0.x);
                            cc[1] = best + fmaf(-lam, q1.y, q1.x);
                            h[0] = bh + q0.x;
                            h[1] = bh + q1.x;
                            e[0] = be + q0.y;
                            e[1] = be + q1.y;
                        }
                        continue;
                    }
                    const uint32_t n0 = d4.x >> 16 & 255u, n1 = d4.x >> 24;
                    const uint32_t list0 = d4.w & 255u, list1 = d4.w >> 8 & 255u;
                    const uint32_t fa = d4.w >> 16 & 3u, fb = d4.w >> 18 & 3u;
                    float nc[4], nh[4], ne[4];
                    const char *EA = column(sh0), *EB = column(sh1);
                    float ab = INF, ah = 0.f, ae = 0.f; // keys apart: the argmin over x
                    if (apart) {
#pragma unroll
                        for (uint32_t x = 0; x < 4; ++x)
                            if (x < n0) {
                                const float2 v2 = entry(EA, 128 * ((list0 >> (2 * x) & 3u) + 4 * fa));
                                const float v = cc[x] + fmaf(-lam, v2.y, v2.x);
                                if (v < ab) {
                                    ab = v;
                                    ah = h[x] + v2.x;
                                    ae = e[x] + v2.y;
                                }
                            }
                    }
#pragma unroll
                    for (uint32_t y = 0; y < 4; ++y) {
                        nc[y] = INF;
                        nh[y] = ne[y] = 0.f;
                        if (y < n1) {
                            const uint32_t by = list1 >> (2 * y) & 3u;
                            if (apart) {
                                const float2 v2 = entry(EB, 128 * (fb + 4 * by));
                                nc[y] = ab + fmaf(-lam, v2.y, v2.x);
                                nh[y] = ah + v2.x;
                                ne[y] = ae + v2.y;
                            } else {
#pragma unroll
                                for (uint32_t x = 0; x < 4; ++x)
                                    if (x < n0) {
                                        const float2 v2 = entry(EA, 128 * ((list0 >> (2 * x) & 3u) + 4 * by));
                                        const float v = cc[x] + fmaf(-lam, v2.y, v2.x);
                                        if (v < nc[y]) {
                                            nc[y] = v;
                                            nh[y] = h[x] + v2.x;
                                            ne[y] = e[x] + v2.y;
                                        }
                                    }
                            }
                        }
                    }
#pragma unroll
                    for (int y = 0; y < 4; ++y) {
                        cc[y] = nc[y];
                        h[y] = nh[y];
                        e[y] = ne[y];
                    }
                }
                // the 3' terminal pair, then the argmin end state (ties: the lowest base)
                float best = INF, H = 0.f, S = 0.f;
#pragma unroll
                for (int y = 0; y < 4; ++y)
                    if (y < F.nL) {
                        const float2 t = tL[(F.listL >> (2 * y) & 3) * 4];
                        const float v = cc[y] + fmaf(-lam, t.y, t.x);
                        if (v < best) {
                            best = v;
                            H = h[y] + t.x;
                            S = e[y] + t.y;
                        }
                    }
                const float r = (H + SH) / (S + SE + cst);
                // stop when the ratio no longer improves by more than 1e-4 K (as tm_kernel)
                if (!(r > lam + 1e-4f))
                    break;
                lam = r;
            }
            const float tm32 = lam - 273.15f + sp.tm_shift_f;
            const uint64_t io = b0 + local;
            if (pass_out && fabsf(tm32 - sp.tm_min_f) < 0.01f) {
                defer[atomicAdd(defer_n, 1ull)] = (uint32_t)io; // decided exactly by tm_kernel
                continue;
            }
            tm_out[io] = tm32;
            if (pass_out)
                pass_out[io] = tm32 >= sp.tm_min_f;
        }
    }
}

// ---------------------------------------------------------------------------
// Tm-threshold sweep (Sec. 3.3, Annealing Temperature Optimization: amplicon
// counts, genomes amplified and off-target patterns as the threshold moves).
// Per site a bit per threshold (passes or not, decided as the fp64 definition
// decides: the fp32 maximum where it is 0.01 deg C or more from the threshold,
// else the exact fixed-point sign test of the file comment, else every oligo
// in fp64), then per amplicon the AND of its two sites' bits.
// ---------------------------------------------------------------------------

// W[(pair * n_thr + j) * 272 + e]: fixed-point weight of table entry e (256
// stacks, then 16 terminal pairs) at threshold j, in the pair's ratio units
__global__ void sweep_weights_kernel(const PairDev *__restrict__ pairs, int n_pairs, const double *__restrict__ thr_c,
                                     int n_thr, long long *__restrict__ W)
{
    const int total = n_pairs * n_thr * 272;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
        const int e = i % 272, pj = i / 272, j = pj % n_thr, p = pj / n_thr;
        const PairDev &pd = pairs[p];
        const double thr = thr_c[j] + 273.15 - pd.tm_shift;
        W[i] = e < 256 ? fix_weight(pd.stack_dH_d[e], pd.stack_dS_d[e], thr)
                       : fix_weight(pd.term_dH_d[e - 256], pd.term_dS_d[e - 256], thr);
    }
}

// One thread per site: bit j of pass_mask[i] = site i passes threshold j.  A
// threshold that fp32 keeps clear of the 0.01 deg C band (with its own rounding
// and the threshold's allowed for) is decided by one fp32 comparison: the fp64
// units run at 1/64 of the fp32 rate here.  What remains is the latency of the
// sites near a threshold (80,000 sites x 31 thresholds: 47 -> 42 us).
__global__ void sweep_pass_kernel(const ah_site *__restrict__ sites, uint64_t n, const PairDev *__restrict__ pairs,
                                  const uint32_t *__restrict__ planes, const uint64_t *__restrict__ contig_off,
                                  const float *__restrict__ tm, const double *__restrict__ thr_c, int n_thr,
                                  const long long *__restrict__ W, int few_exact, uint64_t *__restrict__ pass_mask,
                                  const int *__restrict__ err)
{
    const long long LINF = 0x2000000000000000ll;
    __shared__ float thr_f[kSweepMax], clear_of[kSweepMax];
    if (threadIdx.x < (unsigned)n_thr) {
        const float f = (float)thr_c[threadIdx.x];
        thr_f[threadIdx.x] = f;
        clear_of[threadIdx.x] = 0.0101f + 2.4e-7f * fabsf(f);
    }
    __syncthreads();
    if (*(volatile const int *)err)
        return;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
        const ah_site s = sites[i];
        const float t = tm[i];
        const PairDev &pd = pairs[s.pair];
        const int L = pd.L[s.primer];
        const uint8_t *qm = pd.mask[s.primer];
        int8_t bt[AH_MAX_PRIMER_LEN];
        bool have_bt = false;
        uint64_t m = 0;
        for (int j = 0; j < n_thr; ++j) {
            const float df = t - thr_f[j];
            if (isnan(t) || fabsf(df) >= clear_of[j]) {
                if (df > 0.0f) // (NaN, a template with a non-ACGT letter: fails every threshold)
                    m |= 1ull << j;
                continue;
            }
            const double T = thr_c[j];
            bool pass;
            if (fabs((double)t - T) >= 0.01) {
                pass = (double)t >= T;
            } else {
                if (!have_bt) {
                    const uint64_t P = contig_off[s.contig] + s.pos;
                    for (int q = 0; q < L; ++q) {
                        const int c = base_at(planes, P + (s.strand == 0 ? q : L - 1 - q));
                        bt[q] = (int8_t)(s.strand == 0 ? 3 - c : c); // finite Tm: only A/C/G/T
                    }
                    have_bt = true;
                }
                int dec = -1;
                if (few_exact) { // sign of min over oligos of F at this threshold, exactly
                    const long long *Wp = W + ((size_t)s.pair * n_thr + j) * 272;
                    long long c[4];
                    for (int y = 0; y < 4; ++y)
                        c[y] = (qm[0] >> y & 1) ? Wp[256 + y * 4 + bt[0]] : LINF;
                    for (int q = 1; q < L; ++q) {
                        long long nc[4];
                        for (int y = 0; y < 4; ++y) {
                            long long best = LINF;
                            if (qm[q] >> y & 1)
                                for (int x = 0; x < 4; ++x)
                                    if (c[x] < LINF) {
                                        const long long v = c[x] + Wp[((x * 4 + y) * 4 + bt[q - 1]) * 4 + bt[q]];
                                        best = v < best ? v : best;
                                    }
                            nc[y] = best;
                        }
                        for (int y = 0; y < 4; ++y)
                            c[y] = nc[y];
                    }
                    long long fin = LINF;
                    for (int y = 0; y < 4; ++y)
                        if (c[y] < LINF) {
                            const long long v = c[y] + Wp[256 + y * 4 + bt[L - 1]];
                            fin = v < fin ? v : fin;
                        }
                    const double thr = T + 273.15 - pd.tm_shift;
                    const double Cp = pd.sconst + (pd.saltcorr == 5 ? 0.368 * (double)(L - 1) * pd.log_na : 0.0);
                    const long long F = fin - __double2ll_rn(thr * Cp * kFix);
                    dec = F < -kFixMargin ? 1 : (F > kFixMargin ? 0 : -1);
                }
                if (dec < 0) { // every oligo, in the definition's fp64 order
                    int deg = 1;
                    for (int q = 0; q < L; ++q)
                        deg *= __popc(qm[q]);
                    double best = -INFINITY;
                    for (int o = 0; o < deg; ++o) {
                        const double v = exact_tm(pd, bt, L, oligo_number(qm, L, o));
                        best = v > best ? v : best;
                    }
                    dec = best >= T ? 1 : 0;
                }
                pass = dec == 1;
            }
            if (pass)
                m |= 1ull << j;
        }
        pass_mask[i] = m;
    }
}

// Per threshold (bit j of each lane's m), the lanes that have it: lane j % 32
// adds the count to its acc[j / 32].  A warp's count is one vote, where an
// atomic per set bit made all lanes of a block queue at one shared word.
__device__ __forceinline__ void count_bits(uint64_t m, int n_thr, int lane, uint32_t (&acc)[2])
{
    for (int j = 0; j < n_thr; ++j) {
        const uint32_t c = __popc(__ballot_sync(0xffffffffu, (m >> j) & 1u));
        if (lane == (j & 31)) {
            if (j < 32)
                acc[0] += c;
            else
                acc[1] += c;
        }
    }
}
__device__ __forceinline__ void add_counts(const uint32_t (&acc)[2], int n_thr, int lane, unsigned long long *out)
{
    if (lane < n_thr && acc[0])
        atomicAdd(out + lane, (unsigned long long)acc[0]);
    if (32 + lane < n_thr && acc[1])
        atomicAdd(out + 32 + lane, (unsigned long long)acc[1]);
}

// Per amplicon: the thresholds both of its sites pass; counts per threshold
// (all, FF or RR) and, per genome, the thresholds at which it is amplified.
// (65,000 amplicons, 31 thresholds: 30 -> 9 us; the genomes' counts below 48 -> 3.)
__global__ void sweep_count_kernel(const ah_amplicon *__restrict__ a, uint64_t na, uint64_t n_sites,
                                   const uint64_t *__restrict__ pass_mask, uint32_t max_genome, int n_thr,
                                   unsigned long long *__restrict__ amps, unsigned long long *__restrict__ ffrr,
                                   unsigned long long *__restrict__ gmask, int *__restrict__ err)
{
    const int lane = threadIdx.x & 31;
    uint32_t all[2] = {0, 0}, same[2] = {0, 0};
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i0 = (uint64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); i0 < na; i0 += stride) {
        const uint64_t i = i0 + lane;
        uint64_t m = 0;
        bool ff = false;
        if (i < na) {
            const ah_amplicon am = a[i];
            if (am.left >= n_sites || am.right >= n_sites || am.genome > max_genome || am.orient > 3) {
                atomicExch(err, kDevBounds);
            } else {
                m = pass_mask[am.left] & pass_mask[am.right];
                ff = am.orient >= 2;
                if (m & ~*(volatile unsigned long long *)(gmask + am.genome)) // (most add nothing: no atomic)
                    atomicOr(gmask + am.genome, (unsigned long long)m);
            }
        }
        count_bits(m, n_thr, lane, all);
        if (__any_sync(0xffffffffu, ff))
            count_bits(ff ? m : 0, n_thr, lane, same);
    }
    add_counts(all, n_thr, lane, amps);
    add_counts(same, n_thr, lane, ffrr);
}

__global__ void sweep_genomes_kernel(const unsigned long long *__restrict__ gmask, uint64_t n_words, int n_thr,
                                     unsigned long long *__restrict__ gcount)
{
    const int lane = threadIdx.x & 31;
    uint32_t all[2] = {0, 0};
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i0 = (uint64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); i0 < n_words; i0 += stride) {
        const uint64_t i = i0 + lane;
        count_bits(i < n_words ? gmask[i] : 0, n_thr, lane, all);
    }
    add_counts(all, n_thr, lane, gcount);
}

// Whether one thread takes a site (tm_fast_kernel, then the four-lane kernel on the sites near the
// threshold).  Few sites (a latency-bound launch): the four-lane kernel alone finishes first; many:
// one thread per site has 6 times its rate on 3.2 M sites.  On a GB300, the four-lane kernel alone
// against the two: 16,384 sites 22 us against 15 + 14 (15 + 2 when no site is deferred), 24,000 25
// against 15 + 14, 32,767 44 against 15 + 14; the line lies where they meet with sites deferred.
constexpr uint64_t kFastMinSites = 24576;
bool tm_fast(uint64_t n, bool few_exact) { return few_exact && n >= kFastMinSites; }

} // namespace

int tm_launches(uint64_t n, bool few_exact) { return n == 0 ? 0 : few_exact && !tm_fast(n, few_exact) ? 1 : 2; }

void launch_tm(const ah_site *sites, uint64_t n, const uint64_t *n_dev, const PairDev *pairs_d, int n_pairs,
               const uint32_t *planes, const uint64_t *contig_off, float *tm_out, uint8_t *pass_out, uint32_t *queue,
               uint32_t *queue_n, int seg_max, bool few_exact, int *err, cudaStream_t s)
{
    if (!n)
        return;
    if (seg_max < 1 || seg_max > AH_MAX_PRIMER_LEN - 1)
        throw Error(AH_ERR_ARG, "Tm: segment count outside 1..31");
    static int cached_dev = -1, sms = 148, tm_bps = 1, fast_blocks[AH_MAX_PAIRS_PER_SCAN + 1];
    int dev = 0;
    AH_CUDA(cudaGetDevice(&dev));
    const size_t smem = (size_t)n_pairs * sizeof(TmPairS) + (size_t)(n_pairs <= kTmStageD ? n_pairs : 0) * sizeof(TmPairD) +
                        kTmWarps * 8 * tm_group_stride(seg_max) * sizeof(float2);
    const size_t fast_smem = (size_t)n_pairs * sizeof(TmFastPair);
    if (dev != cached_dev) {
        AH_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        const int most = AH_MAX_PAIRS_PER_SCAN * (int)sizeof(TmPairS) + kTmStageD * (int)sizeof(TmPairD) +
                         kTmWarps * 8 * tm_group_stride(AH_MAX_PRIMER_LEN - 1) * (int)sizeof(float2);
        AH_CUDA(cudaFuncSetAttribute(tm_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
        AH_CUDA(cudaFuncSetAttribute(tm_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
        const int most_fast = AH_MAX_PAIRS_PER_SCAN * (int)sizeof(TmFastPair);
        AH_CUDA(cudaFuncSetAttribute(tm_fast_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most_fast));
        for (int j = 1; j <= AH_MAX_PAIRS_PER_SCAN; ++j) {
            AH_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fast_blocks[j], tm_fast_kernel, kFastThreads,
                                                                  j * sizeof(TmFastPair)));
            fast_blocks[j] = std::max(1, fast_blocks[j]);
        }
        AH_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&tm_bps, tm_kernel<true>, 32 * kTmWarps, most));
        tm_bps = std::max(1, tm_bps);
        // AH_TM_FAST_BLOCKS=n: at most n blocks of the thread-per-site kernel per SM (profiling aid)
        if (const char *e = getenv("AH_TM_FAST_BLOCKS"))
            if (atoi(e) > 0)
                for (int &b : fast_blocks)
                    b = std::min(b, atoi(e));
        cached_dev = dev;
    }
    const bool fast = tm_fast(n, few_exact);
    if (!n_dev && (fast || !few_exact)) // queue length, deferred sites
        AH_CUDA(cudaMemsetAsync(queue_n, 0, 2 * sizeof(uint64_t), s));
    if (fast) {
        // every site in one thread; those near tm_min go to the four-lane kernel below
        uint32_t *defer = queue + n;
        unsigned long long *defer_n = reinterpret_cast<unsigned long long *>(queue_n) + 1;
        const uint64_t fb = std::min<uint64_t>((n + kFastThreads - 1) / kFastThreads, (uint64_t)sms * fast_blocks[n_pairs]);
        tm_fast_kernel<<<(unsigned)fb, kFastThreads, fast_smem, s>>>(sites, n, n_dev, pairs_d, n_pairs, planes,
                                                                      contig_off, tm_out, pass_out, defer, defer_n,
                                                                      err);
        AH_CUDA(cudaGetLastError());
        // deferred sites (few; their count stays on the device): a persistent grid
        const uint64_t tb = std::min<uint64_t>((n + 8 * kTmWarps - 1) / (8 * kTmWarps), (uint64_t)sms * tm_bps);
        launch_chained(tm_kernel<true>, (unsigned)tb, 32 * kTmWarps, smem, s, sites, n,
                       reinterpret_cast<const uint64_t *>(defer_n), pairs_d, n_pairs, planes, contig_off, tm_out, pass_out,
                       queue, queue_n, seg_max, err, defer);
        return;
    }
    const uint64_t per_block = 8ull * kTmWarps; // sites per block per pass
    uint64_t blocks = (n + per_block - 1) / per_block;
    if (blocks > 65535)
        blocks = 65535;
    launch_chained(few_exact ? tm_kernel<true> : tm_kernel<false>, (unsigned)blocks, 32 * kTmWarps, smem, s, sites, n,
                   n_dev, pairs_d, n_pairs, planes, contig_off, tm_out, pass_out, queue, queue_n, seg_max, err, nullptr);
    if (few_exact)
        return;
    tm_exact_kernel<<<(unsigned)sms, kExactThreads, 0, s>>>(sites, pairs_d, planes, contig_off, queue, queue_n,
                                                              tm_out, pass_out);
    AH_CUDA(cudaGetLastError());
}

// Sweep: counts[0..n_thr) amplicons, [64..64+n_thr) FF/RR, [128..128+n_thr)
// genomes; counts and gmask (max_genome + 1 words) zeroed here.
void launch_tm_sweep(const ah_site *sites, uint64_t n_sites, const ah_amplicon *amps, uint64_t n_amps,
                     const PairDev *pairs_d, int n_pairs, const uint32_t *planes, const uint64_t *contig_off,
                     const float *tm, const double *thr_d, int n_thr, long long *W, bool few_exact,
                     uint64_t *pass_mask, unsigned long long *gmask, uint32_t max_genome, unsigned long long *counts,
                     int *err, cudaStream_t s)
{
    if (n_thr < 1 || n_thr > kSweepMax)
        throw Error(AH_ERR_ARG, "sweep: 1..64 thresholds");
    AH_CUDA(cudaMemsetAsync(counts, 0, 3 * kSweepMax * sizeof(unsigned long long), s));
    AH_CUDA(cudaMemsetAsync(gmask, 0, ((uint64_t)max_genome + 1) * sizeof(unsigned long long), s));
    sweep_weights_kernel<<<(n_pairs * n_thr * 272 + 255) / 256, 256, 0, s>>>(pairs_d, n_pairs, thr_d, n_thr, W);
    AH_CUDA(cudaGetLastError());
    if (n_sites) {
        const uint64_t blocks = std::min<uint64_t>((n_sites + 127) / 128, 8192);
        sweep_pass_kernel<<<(unsigned)blocks, 128, 0, s>>>(sites, n_sites, pairs_d, planes, contig_off, tm, thr_d,
                                                           n_thr, W, few_exact ? 1 : 0, pass_mask, err);
        AH_CUDA(cudaGetLastError());
    }
    if (n_amps) {
        const uint64_t blocks = std::min<uint64_t>((n_amps + 255) / 256, 4096);
        sweep_count_kernel<<<(unsigned)blocks, 256, 0, s>>>(amps, n_amps, n_sites, pass_mask, max_genome, n_thr,
                                                            counts, counts + kSweepMax, gmask, err);
        AH_CUDA(cudaGetLastError());
    }
    const uint64_t words = (uint64_t)max_genome + 1;
    const uint64_t blocks = std::min<uint64_t>((words + 255) / 256, 1024);
    sweep_genomes_kernel<<<(unsigned)blocks, 256, 0, s>>>(gmask, words, n_thr, counts + 2 * kSweepMax);
    AH_CUDA(cudaGetLastError());
}

} // namespace ah
