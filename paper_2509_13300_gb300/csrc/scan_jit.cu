// Scan kernel generator (primer matching, Sec. 2.1) and its run-time compiler.
//
// Why generate: the mismatch count of a window against a degenerate primer is
// a sum of L one-bit terms, and on this GPU its cost is set by integer issue
// slots.  With the primer's IUPAC codes known when the kernel is compiled,
// the match word of a single-base position is a plane word itself (0 ops), a
// two- or three-base position is a sum of disjoint plane words (integer adds,
// which do not use the logic pipe), and the count runs through a carry-save
// network whose shape depends on L and k.  So each set of patterns gets its
// own straight-line kernel, built here as CUDA source and compiled with NVRTC
// for sm_103a; compiled kernels are cached per process.
//
// Bit-sliced counting.  A thread owns R consecutive words of a tile; word j
// holds starts p = b * W + j for b = 0..31 (tile-strided layout), so the
// window base at offset i of all 32 starts is word j + i.  For each pattern
// and word the kernel forms match words M_i (bit b = 1 when the base at
// p_b + i is in the pattern's set) and reduces them column by column with
// full adders.  It works in the "match" domain: a full adder on match words
// yields the complements of the sum and carry of the mismatch bits, so no
// inversion is ever needed, and padding uses all-ones words (a match).  With
// K2 the smallest power of two above k, columns of weight < K2 are reduced
// to one bit each; a mismatch count >= K2 shows as a zero bit in any carry
// word of weight K2, so those are AND-ed; the low bits are compared with k by
// one or two LOP3s.  Full adders are either two LOP3s (xor3, majority) or one
// majority LOP3 plus integer adds for the sum (s = a + b + c - 2 maj), a mix
// chosen by the tuner to balance the logic and integer pipes.
//
// The network is a filter: it counts only the positions that pay for
// themselves (choose_positions), because every hit start is re-counted
// exactly anyway.  A position costs ~1.75 LOP3s per word and pattern; leaving
// it out lets more false starts through, each of which costs a visit.  N
// positions filter nothing and are always left out.  Complements are free
// (a full adder's table takes inverted inputs), so R, M, W and the three-base
// codes are the complements of Y, K, S and single planes; such a term also
// lets a non-base through, which the exact count rejects.
//
// Hits.  The network's hit words of the four patterns of one primer pair are
// OR-ed into one word per pair and thread word.  A warp with any hit publishes
// its hit words to shared memory and visits the hit starts together: the warp
// gathers the 32 window bases as four ballots of the plane bits (bit i = base
// at window position i) and four lanes keep them, one per pattern; eight
// starts fill the warp, and one evaluation counts all 32 (start, pattern)
// combinations exactly (AND/OR/popc against the pattern's position masks),
// tests the 3' clamp and the contig end.  Windows never cross a contig end: a
// start within the first contig of its tile takes that contig's end from a
// per-tile table loaded while the network runs; any other searches the tile's
// contigs.  Surviving keys collect in a per-warp stash in shared memory and
// are appended 32 at a time with one atomic (the rest when the warp ends).
// Key = ((pair << pbits | flat position) << 10) | primer << 9 | strand << 8
// | mm, so sorting keys gives the canonical site order.
//
// Bound: the logic pipe (LOP3s at 64 lanes/clk/SM); ncu on 0.6 Gbp, three pairs
// at k = 4: ALU pipe 83 % active, of which the network is nearly all, issue
// 0.58, DRAM 20 %.  At k <= 1 the reads of the planes (0.516 B/base) come near:
// 2 Gbp at k = 1 in 243 us = 4.2 TB/s.  Measured, 4 Gbp and three pairs at k = 4
// (960, 64 and 256 oligos): 4,286 us with every position counted, a visit per
// start and pattern list and a slice pipeline per warp; 3,694 us with the
// chosen positions; 2,997 us with the tile ring and batched evaluation; 2,850 us
// in one launch.  1.5 Gbp, four pairs of k = 2, 3, 4, 2: 1,687 -> 943 us;
// 0.41 Gbp, one 960-oligo pair at k = 3: 125 -> 88 us.
#include <nvrtc.h>

#include <algorithm>
#include <cstdio>
#include <cstring>
#include <deque>
#include <mutex>
#include <sstream>

#include "ah_internal.h"

namespace ah {
namespace {

const char *kPrelude = R"CUDA(
typedef unsigned int u32;
typedef unsigned long long u64;
typedef unsigned char u8;
template <int IMM> __device__ __forceinline__ u32 lop3(u32 a, u32 b, u32 c)
{
    u32 d;
    asm("lop3.b32 %0, %1, %2, %3, %4;" : "=r"(d) : "r"(a), "r"(b), "r"(c), "n"(IMM));
    return d;
}
__device__ __forceinline__ u32 smem_addr(const void *p) { return (u32)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(u64 *bar, u32 count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
// one thread: start a bulk copy (TMA) whose bytes complete on `bar`; the
// generic-proxy reads of the buffer are ordered before the async write
__device__ __forceinline__ void tma_copy(void *dst, const void *src, u32 bytes, u64 *bar)
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_addr(dst)), "l"(src), "r"(bytes), "r"(smem_addr(bar))
                 : "memory");
}
__device__ __forceinline__ bool mbar_try(u64 *bar, u32 parity)
{
    u32 ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
                 : "=r"(ok) : "r"(smem_addr(bar)), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ u64 global_ns()
{
    u64 t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ bool mbar_test(u64 *bar, u32 parity)
{
    u32 ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
                 : "=r"(ok) : "r"(smem_addr(bar)), "r"(parity) : "memory");
    return ok != 0;
}
// bounded wait for a barrier phase: gives up after limit_ns instead of hanging.
// Limits of a millisecond and more poll with try_wait (the thread may be
// suspended between tests); shorter ones poll with the non-blocking test, so
// that the limit itself decides.
__device__ __forceinline__ bool mbar_wait(u64 *bar, u32 parity, u64 limit_ns)
{
    if (mbar_test(bar, parity))
        return true;
    const u64 t0 = global_ns();
    if (limit_ns >= 1000000ull) {
        while (!mbar_try(bar, parity))
            if (global_ns() - t0 > limit_ns)
                return false;
    } else {
        while (!mbar_test(bar, parity))
            if (global_ns() - t0 > limit_ns)
                return false;
    }
    return true;
}
)CUDA";

// Body of the kernel after the generated hit words.  Uses: hg[NHG] (hit words
// per pattern group and thread word), any, lane, sm (the warp's words of the
// tile's planes, stride WX), tile, wbase, room, and the warp's state: hit-word
// buffer hs, visited starts vs (nb of them) and key stash ws (nv keys) in
// shared memory.
const char *kEmit = R"CUDA(
    if (__any_sync(0xffffffffu, any != 0u)) {
        u32 lanes = __ballot_sync(0xffffffffu, any != 0u);
        u32 nz = 0u; // bit i: hg[i] != 0
        if (any != 0u) {
#pragma unroll
            for (int i = 0; i < NHG; i += 4)
                *reinterpret_cast<uint4 *>(hs + lane * NHG + i) = make_uint4(hg[i], hg[i + 1], hg[i + 2], hg[i + 3]);
#pragma unroll
            for (int i = 0; i < NHG; ++i) nz |= hg[i] != 0u ? 1u << i : 0u;
        }
        __syncwarp();
#pragma unroll 1
        while (lanes) {
            const int src = __ffs(lanes) - 1;
            lanes &= lanes - 1;
            u32 words = __shfl_sync(0xffffffffu, nz, src);
#pragma unroll 1
            while (words) {
                const int i = __ffs(words) - 1;
                words &= words - 1;
                u32 m = hs[src * NHG + i];
                const int jr = src * R + i % R; // the starts' word, from the warp's first
                const u32 *wp = sm + jr + lane;
#pragma unroll 1
                while (m) {
                    const int b = __ffs(m) - 1;
                    const u32 bit = m & (0u - m);
                    m &= m - 1;
                    // window bases, bit i = base at position i of the window
                    const u32 cA = __ballot_sync(0xffffffffu, (wp[0] & bit) != 0u);
                    const u32 cC = __ballot_sync(0xffffffffu, (wp[WX] & bit) != 0u);
                    const u32 cG = __ballot_sync(0xffffffffu, (wp[2 * WX] & bit) != 0u);
                    const u32 cT = __ballot_sync(0xffffffffu, (wp[3 * WX] & bit) != 0u);
                    if (lane == 0) {
                        vs[2 * nb] = make_uint4(cA, cC, cG, cT);
                        vs[2 * nb + 1] = make_uint4((u32)(b * W + wbase + jr), (u32)(i / R), (u32)tile, room);
                    }
                    if (++nb == 8) evaluate();
                }
            }
        }
        __syncwarp();
    }
)CUDA";

// One input of the network: a word variable, taken inverted or not.
struct Term {
    std::string v;
    bool inv = false;
};

// LOP3 immediate of f over (a, b, c): bit index (a << 2) | (b << 1) | c; the
// inputs are inverted where ia, ib, ic say so.
template <class F> int lut3(F f, bool ia = false, bool ib = false, bool ic = false)
{
    int imm = 0;
    for (int a = 0; a < 2; ++a)
        for (int b = 0; b < 2; ++b)
            for (int c = 0; c < 2; ++c)
                if (f(a ^ (int)ia, b ^ (int)ib, c ^ (int)ic))
                    imm |= 1 << ((a << 2) | (b << 1) | c);
    return imm;
}

struct Gen {
    std::ostringstream os;
    int n = 0;
    int fa_total = 0, fa_arith = 0;
    int arith_pct = 0;

    std::string tmp() { return "v" + std::to_string(n++); }
    std::string lop(const std::string &a, const std::string &b, const std::string &c, int imm)
    {
        std::string v = tmp();
        os << "    const u32 " << v << " = lop3<0x" << std::hex << imm << std::dec << ">(" << a << ", " << b << ", "
           << c << ");\n";
        return v;
    }
    // full adder on match-domain words -> (sum, carry)
    void fa(const Term &a, const Term &b, const Term &c, std::string &s, std::string &cy)
    {
        ++fa_total;
        cy = lop(a.v, b.v, c.v, lut3([](int x, int y, int z) { return x + y + z >= 2; }, a.inv, b.inv, c.inv));
        // Bresenham-style spread of the arithmetic full adders
        bool arith = (fa_arith * 100 < arith_pct * fa_total);
        if (arith) {
            ++fa_arith;
            s = tmp();
            os << "    const u32 " << s << " = " << (a.inv ? "~" : "") << a.v << " + " << (b.inv ? "~" : "") << b.v
               << " + " << (c.inv ? "~" : "") << c.v << " - " << cy << " - " << cy << ";\n";
        } else {
            s = lop(a.v, b.v, c.v, lut3([](int x, int y, int z) { return (x + y + z) & 1; }, a.inv, b.inv, c.inv));
        }
    }
};

int popc4(int m) { return (m & 1) + ((m >> 1) & 1) + ((m >> 2) & 1) + ((m >> 3) & 1); }

using WordCache = std::map<std::pair<int, int>, std::string>;

// Sum of the planes of `mask` at window word w: the match word of that set
// (disjoint planes: add = or; adds keep the logic pipe free).
std::string plane_sum(Gen &g, int mask, int w, WordCache &cache)
{
    static const char *P[4] = {"pA", "pC", "pG", "pT"};
    if (popc4(mask) == 1)
        return std::string(P[__builtin_ctz(mask)]) + "[" + std::to_string(w) + "]";
    auto key = std::make_pair(mask, w);
    auto it = cache.find(key);
    if (it != cache.end())
        return it->second;
    const std::string r = g.tmp();
    g.os << "    const u32 " << r << " = ";
    bool first = true;
    for (int x = 0; x < 4; ++x)
        if (mask & (1 << x)) {
            g.os << (first ? "" : " + ") << P[x] << "[" << w << "]";
            first = false;
        }
    g.os << ";\n";
    cache[key] = r;
    return r;
}

// Match word of an IUPAC mask at window word w.  With complements allowed,
// a three-base set is the complement of its missing plane, and of the six
// two-base sets only C|T, G|T and C|G are formed (the others are their
// complements), so fewer distinct words are summed and kept.
Term match_word(Gen &g, int mask, int w, bool complements, WordCache &cache)
{
    constexpr int kC = 2, kG = 4, kT = 8;
    const int n = popc4(mask);
    if (complements && (n == 3 || (n == 2 && mask != (kC | kT) && mask != (kG | kT) && mask != (kC | kG))))
        return {plane_sum(g, 15 & ~mask, w, cache), true};
    return {plane_sum(g, mask, w, cache), false};
}

std::string and_reduce(Gen &g, std::deque<Term> v)
{
    if (v.empty())
        return "0xffffffffu";
    while (v.size() > 1) {
        Term a = v.front();
        v.pop_front();
        Term b = v.front();
        v.pop_front();
        Term c{"0xffffffffu"};
        if (!v.empty()) {
            c = v.front();
            v.pop_front();
        }
        v.push_back({g.lop(a.v, b.v, c.v, lut3([](int x, int y, int z) { return x & y & z; }, a.inv, b.inv, c.inv))});
    }
    return (v.front().inv ? "~" : "") + v.front().v;
}

int low_columns(int k) // columns of weight below K2 = 2^klog, the smallest power of two above k
{
    int klog = 0;
    while ((1 << klog) <= k)
        ++klog;
    return klog;
}

// LOP3s of the network over n positions at threshold k (as gen_hit emits them).
int network_lops(int n, int k)
{
    if (k >= n)
        return 0;
    const int klog = low_columns(k);
    int col[6] = {n, 0, 0, 0, 0, 0}, ops = 0;
    for (int w = 0; w < klog; ++w)
        while (col[w] > 1) {
            col[w] -= std::min(3, col[w]) - 1;
            ++col[w + 1];
            ops += 2;
        }
    for (int m = col[klog]; m > 1; ++ops)
        m -= std::min(3, m) - 1;
    return ops + (k == (1 << klog) - 1 ? 0 : klog == 2 ? 1 : 2);
}

// Share of random starts with at most k mismatches at positions of the given
// sets, averaged over genomes of three GC contents.
double pass_rate(const std::vector<int> &masks, int k)
{
    double total = 0;
    for (double gc : {0.35, 0.5, 0.65}) {
        std::vector<double> d(masks.size() + 1, 0.0);
        d[0] = 1.0;
        for (int m : masks) {
            const double hit = ((m & 1) + (m >> 3 & 1)) * (1 - gc) / 2 + ((m >> 1 & 1) + (m >> 2 & 1)) * gc / 2;
            for (size_t j = d.size() - 1; j > 0; --j)
                d[j] = d[j] * hit + d[j - 1] * (1 - hit);
            d[0] *= hit;
        }
        for (int j = 0; j <= k && j < (int)d.size(); ++j)
            total += d[j] / 3;
    }
    return total;
}

// Cycles a scheduler spends on one visited start and on one LOP3 (half rate).
// Visits measured by sweeping the figure (three pairs at k = 4, 4 Gbp): 25 3,549 us,
// 40 3,043, 60 2,996, 90 2,997, 130 2,986; four pairs of k = 2..4, 1.5 Gbp: 40 1,089 us,
// 60 1,035, 90 972, 130 974.
constexpr double kVisitCycles = 100, kLopCycles = 2;

// The window positions the network of a pattern counts, ascending.  Positions
// are taken by information (fewest bases first, then leftmost: a short window
// needs fewer words in registers); their number minimises LOP3 cycles plus
// visits per warp and word (1,024 starts).  At least k + 1 positions, so that
// a run of non-bases never passes.
std::vector<int> choose_positions(const ScanPattern &p)
{
    std::vector<int> order, all;
    for (int n = 1; n <= 3; ++n)
        for (int i = 0; i < p.L; ++i)
            if (popc4(p.mask[i]) == n)
                order.push_back(i);
    for (int i = 0; i < p.L; ++i)
        all.push_back(i);
    if ((int)order.size() <= p.k)
        return all;
    std::vector<int> masks;
    size_t best = 0;
    double best_cost = 0;
    for (size_t n = 1; n <= order.size(); ++n) {
        masks.push_back(p.mask[order[n - 1]]);
        if ((int)n <= p.k)
            continue;
        const double cost = kLopCycles * network_lops((int)n, p.k) + 1024 * kVisitCycles * pass_rate(masks, p.k);
        if (!best || cost < best_cost) {
            best = n;
            best_cost = cost;
        }
    }
    std::vector<int> out(order.begin(), order.begin() + best);
    std::sort(out.begin(), out.end());
    return out;
}

// Hit word of pattern p for the thread's word r: bit b set where the window at
// start p_b has <= k mismatches among the positions `pos`.
std::string gen_hit(Gen &g, const ScanPattern &p, const std::vector<int> &pos, int r, WordCache &cache)
{
    if (p.k >= p.L)
        return "0xffffffffu";
    const int klog = low_columns(p.k);
    // complements let non-bases through: only beside more than k single-base positions
    int singles = 0;
    for (int i : pos)
        singles += popc4(p.mask[i]) == 1;
    std::deque<Term> col[6];
    for (int i : pos)
        col[0].push_back(match_word(g, p.mask[i], r + i, singles > p.k, cache));
    for (int w = 0; w < klog; ++w) {
        while (col[w].size() > 1) {
            Term a = col[w].front();
            col[w].pop_front();
            Term b = col[w].front();
            col[w].pop_front();
            Term c{"0xffffffffu"};
            if (!col[w].empty()) {
                c = col[w].front();
                col[w].pop_front();
            }
            std::string s, cy;
            g.fa(a, b, c, s, cy);
            col[w].push_back({s});
            col[w + 1].push_back({cy});
        }
    }
    const std::string hi = and_reduce(g, col[klog]); // (at k = 0 the match words themselves)
    if (p.k == (1 << klog) - 1)
        return hi;
    // low part: match-domain bits s_w (mismatch bit = ~s_w), value v = sum 2^w (1 - s_w) <= k
    Term s[4];
    for (int w = 0; w < klog; ++w)
        s[w] = col[w].empty() ? Term{"0xffffffffu"} : col[w].front();
    const int k = p.k;
    if (klog == 2) { // k == 2 (k == 3 handled above)
        int imm = lut3([&](int a, int b, int c) { return a && ((1 - b) + 2 * (1 - c) <= k); }, false, s[0].inv, s[1].inv);
        return g.lop(hi, s[0].v, s[1].v, imm);
    }
    if (klog == 3) { // k in 4..6
        int imm = lut3([&](int a, int b, int c) { return ((1 - a) + 2 * (1 - b) + 4 * (1 - c)) <= k; }, s[0].inv,
                       s[1].inv, s[2].inv);
        std::string lo = g.lop(s[0].v, s[1].v, s[2].v, imm);
        return "(" + hi + " & " + lo + ")"; // joins the OR over the pair's patterns
    }
    // klog == 4, k in 8..10: v = low3 + 8 (1 - s3); low3 <= 7 <= k, so v <= k iff s3 or low3 <= k - 8
    int imm = lut3([&](int a, int b, int c) { return ((1 - a) + 2 * (1 - b) + 4 * (1 - c)) <= k - 8; }, s[0].inv,
                   s[1].inv, s[2].inv);
    std::string lo = g.lop(s[0].v, s[1].v, s[2].v, imm);
    int imm2 = lut3([](int a, int b, int c) { return a && (b || c); }, false, s[3].inv, false);
    return g.lop(hi, s[3].v, lo, imm2);
}

} // namespace

std::string scan_source(const std::vector<ScanPattern> &pats, const ScanTuning &t)
{
    const int npat = (int)pats.size();
    std::vector<std::vector<int>> pos(npat);
    int span = 1; // window words the networks read
    for (int q = 0; q < npat; ++q) {
        pos[q] = choose_positions(pats[q]);
        span = std::max(span, pos[q].back() + 1);
    }
    const int R = t.R;
    if (R != 4 && R != 8) // the loader reads 16-byte vectors at a warp's word lane * R
        throw Error(AH_ERR_ARG, "scan kernel: R must be 4 or 8");
    const int nwin = 4 * ((R + span - 1 + 3) / 4);
    Gen g;
    g.arith_pct = t.arith_pct;
    std::ostringstream &os = g.os;
    os << kPrelude;
    os << "#define W " << kTileW << "\n#define WX " << kTileWX << "\n#define TB " << kTileBases << "ull\n";
    os << "#define R " << R << "\n#define NWIN " << nwin << "\n";
    // pattern groups: the four patterns of each primer pair
    if (npat % 4 != 0)
        throw Error(AH_ERR_ARG, "scan kernel: four patterns per primer pair");
    const int ngrp = npat / 4;
    os << "#define NGRP " << ngrp << "\n#define NHG (NGRP * R)\n";
    // per pattern: position masks of A, C, G, T; then length mask, clamp mask, k << 8 | length,
    // pair << 2 | primer << 1 | strand
    os << "__constant__ u32 PT[" << npat * 8 << "] = {";
    for (const ScanPattern &p : pats) {
        uint32_t m[4] = {0, 0, 0, 0}, lm = 0, cm = 0;
        for (int i = 0; i < p.L; ++i) {
            for (int x = 0; x < 4; ++x)
                if (p.mask[i] & (1 << x))
                    m[x] |= 1u << i;
            lm |= 1u << i;
            if (p.strand == 0 ? (i >= p.L - p.clamp) : (i < p.clamp)) // the c 3'-most positions
                cm |= 1u << i;
        }
        os << m[0] << "u, " << m[1] << "u, " << m[2] << "u, " << m[3] << "u, " << lm << "u, " << cm << "u, "
           << (p.k << 8 | p.L) << "u, " << (p.pair << 2 | p.primer << 1 | p.strand) << "u,\n    ";
    }
    os << "};\n";
    os << "#define S " << t.stages << "\n#define WPC (W / (32 * R))\n";
    os << "extern \"C\" __global__ void __launch_bounds__(32 * WPC, " << t.min_blocks << ")\n"
       << "ah_scan_kernel(const u32 *__restrict__ planes, u64 n_tiles, const u64 *__restrict__ contig_off,\n"
       << "               u32 n_contigs, u64 *__restrict__ keys, u64 cap, u64 *__restrict__ counter, int pbits,\n"
       << "               int *__restrict__ err, u64 *__restrict__ work, const u64 *__restrict__ tile_list,\n"
       << "               const u32 *__restrict__ tile_contig, const u32 *__restrict__ tile_room, u64 wait_ns,\n"
       << "               int stall_first, u32 per_claim)\n{\n"
       << "  // A CTA runs a ring of S tiles in shared memory, one mbarrier and one bulk async\n"
       << "  // copy (TMA) per tile; its WPC warps each take 32 * R words of a tile and drift up\n"
       << "  // to S tiles apart (no CTA-wide barrier after the start).  The warp that finishes a\n"
       << "  // tile last refills its stage.  The first S tiles of a CTA are fixed; later ones are\n"
       << "  // claimed, `per_claim` at a time, from the shared counter `work` (zeroed before the\n"
       << "  // launch), so SMs that run faster take more.  Tiles of a CTA only grow, so after the\n"
       << "  // first stage that holds none (kNone, its barrier completed without a copy) none\n"
       << "  // follows.  With tile_list, the tiles scanned are tile_list[0 .. n_tiles).\n"
       << "  extern __shared__ __align__(128) u32 smbuf[];\n"
       << "  __shared__ __align__(8) u64 bars[S];\n"
       << "  __shared__ u64 tiles[S], next_item, last_item; // per stage: its tile; items claimed, not yet taken\n"
       << "  __shared__ u32 done[S]; // warps that finished the stage's tile\n"
       << "  __shared__ __align__(16) uint4 ptab[NGRP * 8]; // the patterns' masks (PT)\n"
       << "  const u64 kNone = ~0ull;\n"
       << "  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;\n"
       << "  // per warp: published hit words, visited starts (8), key stash (up to 31 + 32 keys)\n"
       << "  u32 *hs = smbuf + S * (4 * WX) + warp * (32 * NHG + 64 + 128);\n"
       << "  uint4 *vs = reinterpret_cast<uint4 *>(hs + 32 * NHG);\n"
       << "  u64 *ws = reinterpret_cast<u64 *>(hs + 32 * NHG + 64);\n"
       << "  u32 nv = 0u;  // keys in the stash\n"
       << "  int nb = 0;   // starts visited and not yet evaluated\n"
       << "  const u64 n_fixed = (u64)gridDim.x * S; // items taken without a claim\n"
       << "  // one thread: the tile of item w (kNone past the end) into stage stg.  stall_first (a\n"
       << "  // test of the timeout path): a CTA's first tile is armed without a copy, so its wait\n"
       << "  // can only run out\n"
       << "  auto fill = [&](u64 w, int stg, bool copy) {\n"
       << "    if (w >= n_tiles) {\n"
       << "      tiles[stg] = kNone;\n"
       << "      asm volatile(\"mbarrier.arrive.shared::cta.b64 _, [%0];\" ::\"r\"(smem_addr(&bars[stg])) : \"memory\");\n"
       << "      return;\n"
       << "    }\n"
       << "    const u64 tl = tile_list ? tile_list[w] : w;\n"
       << "    tiles[stg] = tl;\n"
       << "    asm volatile(\"mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\" ::\"r\"(smem_addr(&bars[stg])),\n"
       << "                 \"r\"((u32)(16 * WX)) : \"memory\");\n"
       << "    if (copy) tma_copy(smbuf + stg * (4 * WX), planes + tl * (4 * WX), 16 * WX, &bars[stg]);\n"
       << "  };\n"
       << "  // append the n keys ws[0 .. n) with one atomic\n"
       << "  auto flush = [&](u32 n) {\n"
       << "    u64 base = 0;\n"
       << "    if (lane == 0) base = atomicAdd(counter, (u64)n);\n"
       << "    base = __shfl_sync(0xffffffffu, base, 0);\n"
       << "    if ((u32)lane < n && base + lane < cap) keys[base + lane] = ws[lane];\n"
       << "  };\n"
       << "  // the exact count of the visited starts against the four patterns of their pair: lanes\n"
       << "  // 4 n .. 4 n + 3 take start n\n"
       << "  auto evaluate = [&]() {\n"
       << "    __syncwarp();\n"
       << "    const uint4 c = vs[2 * (lane >> 2)], o = vs[2 * (lane >> 2) + 1]; // columns; start, group, tile, room\n"
       << "    bool ok = (lane >> 2) < nb;\n"
       << "    const u32 pat = ok ? o.y * 4u + (u32)(lane & 3) : 0u;\n"
       << "    const uint4 pm = ptab[pat * 2u];\n"
       << "    const uint4 pi = ptab[pat * 2u + 1u]; // length mask, clamp mask, k << 8 | length, key bits\n"
       << "    const u32 mis = ~((c.x & pm.x) | (c.y & pm.y) | (c.z & pm.z) | (c.w & pm.w)) & pi.x;\n"
       << "    const u32 mm = __popc(mis), len = pi.z & 255u;\n"
       << "    ok = ok && mm <= (pi.z >> 8) && (mis & pi.y) == 0u;\n"
       << "    const u64 P = (u64)o.z * TB + o.x;\n"
       << "    if (ok) {\n"
       << "      if (o.x < o.w) {\n"
       << "        ok = o.x + len <= o.w;\n"
       << "      } else { // the first contig end above P among the tile's contigs\n"
       << "        u32 lo = tile_contig[o.z] + 1u;\n"
       << "        const u32 last = min(n_contigs, tile_contig[o.z + 1u] + 1u);\n"
       << "        u32 hi = last + 1u;\n"
       << "        while (lo < hi) {\n"
       << "          const u32 mid = (lo + hi) >> 1;\n"
       << "          if (contig_off[mid] > P) hi = mid;\n"
       << "          else lo = mid + 1u;\n"
       << "        }\n"
       << "        ok = lo <= last && P + len <= contig_off[lo];\n"
       << "      }\n"
       << "    }\n"
       << "    const u32 okm = __ballot_sync(0xffffffffu, ok);\n"
       << "    if (ok)\n"
       << "      ws[nv + __popc(okm & ((1u << lane) - 1u))] =\n"
       << "          (((((u64)(pi.w >> 2)) << pbits) | P) << 10) | (u64)(((pi.w & 3u) << 8) | mm);\n"
       << "    nv += __popc(okm);\n"
       << "    __syncwarp();\n"
       << "    if (nv >= 32u) {\n"
       << "      flush(32u);\n"
       << "      nv -= 32u;\n"
       << "      const u64 rest = ws[32 + lane];\n"
       << "      __syncwarp();\n"
       << "      if ((u32)lane < nv) ws[lane] = rest;\n"
       << "      __syncwarp();\n"
       << "    }\n"
       << "    nb = 0;\n"
       << "  };\n"
       << "  if (threadIdx.x == 0) {\n"
       << "    for (int q = 0; q < S; ++q) {\n"
       << "      mbar_init(&bars[q], 1);\n"
       << "      done[q] = 0u;\n"
       << "    }\n"
       << "    asm volatile(\"fence.mbarrier_init.release.cluster;\" ::: \"memory\");\n"
       << "    next_item = last_item = 0ull;\n"
       << "    for (int q = 0; q < S; ++q)\n"
       << "      fill((u64)q * gridDim.x + blockIdx.x, q, !(stall_first && q == 0));\n"
       << "  }\n"
       << "  for (int i = threadIdx.x; i < NGRP * 32; i += 32 * WPC)\n"
       << "    reinterpret_cast<u32 *>(ptab)[i] = PT[i];\n"
       << "  __syncthreads();\n"
       << "  for (u32 k = 0;; ++k) {\n"
       << "    const u32 stg = k % S;\n"
       << "    const bool landed = mbar_wait(&bars[stg], (k / S) & 1u, wait_ns);\n"
       << "    if (!__all_sync(0xffffffffu, landed)) {\n"
       << "      // a copy did not land in time: report, wait (bounded, ~2 s) for every copy\n"
       << "      // still in flight, this stage's included, then leave\n"
       << "      if (lane == 0) {\n"
       << "        atomicExch(err, 1);\n"
       << "        for (u32 d = 0; d < S; ++d)\n"
       << "          if (tiles[(k + d) % S] != kNone && !(stall_first && k + d == 0)) // no copy was issued there\n"
       << "            mbar_wait(&bars[(k + d) % S], ((k + d) / S) & 1u, 2000000000ull);\n"
       << "      }\n"
       << "      break;\n"
       << "    }\n"
       << "    const u64 tile = tiles[stg];\n"
       << "    if (tile == kNone) break;\n"
       << "    const int wbase = warp * (32 * R);\n"
       << "    const u32 room = tile_room[tile]; // used only on hits; the load overlaps the network\n"
       << "    const u32 *sm = smbuf + stg * (4 * WX) + wbase;\n"
       << "    const int j0 = lane * R;\n"
       << "    u32 pA[NWIN], pC[NWIN], pG[NWIN], pT[NWIN];\n"
       << "#pragma unroll\n"
       << "    for (int c = 0; c < NWIN / 4; ++c) {\n"
       << "      uint4 a = reinterpret_cast<const uint4 *>(sm + 0 * WX + j0)[c];\n"
       << "      uint4 cc = reinterpret_cast<const uint4 *>(sm + 1 * WX + j0)[c];\n"
       << "      uint4 gg = reinterpret_cast<const uint4 *>(sm + 2 * WX + j0)[c];\n"
       << "      uint4 tt = reinterpret_cast<const uint4 *>(sm + 3 * WX + j0)[c];\n"
       << "      pA[4*c] = a.x; pA[4*c+1] = a.y; pA[4*c+2] = a.z; pA[4*c+3] = a.w;\n"
       << "      pC[4*c] = cc.x; pC[4*c+1] = cc.y; pC[4*c+2] = cc.z; pC[4*c+3] = cc.w;\n"
       << "      pG[4*c] = gg.x; pG[4*c+1] = gg.y; pG[4*c+2] = gg.z; pG[4*c+3] = gg.w;\n"
       << "      pT[4*c] = tt.x; pT[4*c+1] = tt.y; pT[4*c+2] = tt.z; pT[4*c+3] = tt.w;\n"
       << "    }\n"
       << "    u32 hg[NGRP * R];\n";
    WordCache cache;
    std::vector<bool> assigned(ngrp * R, false);
    auto one = [&](int q, int r) {
        os << "    // pattern " << q << ", word " << r << "\n";
        std::string hw = gen_hit(g, pats[q], pos[q], r, cache);
        const int i = q / 4 * R + r;
        os << "    hg[" << i << "] " << (assigned[i] ? "|=" : "=") << " " << hw << ";\n";
        assigned[i] = true;
    };
    if (t.order == 0) {
        for (int r = 0; r < R; ++r)
            for (int q = 0; q < npat; ++q)
                one(q, r);
    } else {
        for (int q = 0; q < npat; ++q)
            for (int r = 0; r < R; ++r)
                one(q, r);
    }
    os << "    u32 any = 0u;\n";
    for (int i = 0; i < ngrp * R; ++i)
        os << "    any |= hg[" << i << "];\n";
    os << kEmit;
    os << "    __syncwarp(); // every lane has read what it needs of the tile\n"
       << "    if (lane == 0) {\n"
       << "      u32 before;\n"
       << "      asm volatile(\"atom.acq_rel.cta.shared::cta.add.u32 %0, [%1], 1;\" : \"=r\"(before) : \"r\"(smem_addr(&done[stg])) : \"memory\");\n"
       << "      // the last warp of the tile refills its stage (it does so before it takes part in the\n"
       << "      // next stage's count, so refills run one after another, in stage order)\n"
       << "      if (before == WPC - 1) {\n"
       << "        done[stg] = 0u;\n"
       << "        u64 w = n_tiles;\n"
       << "        if (n_tiles > n_fixed) {\n"
       << "          if (next_item == last_item) {\n"
       << "            next_item = n_fixed + atomicAdd(work, 1ull) * per_claim;\n"
       << "            last_item = next_item + per_claim;\n"
       << "          }\n"
       << "          w = next_item++;\n"
       << "        }\n"
       << "        fill(w, (int)stg, true);\n"
       << "      }\n"
       << "    }\n"
       << "    __syncwarp();\n"
       << "  }\n"
       << "  if (nb) evaluate();\n"
       << "  __syncwarp();\n"
       << "  if (nv) flush(nv); // keys still in the stash (at most 31)\n"
       << "}\n";
    return os.str();
}

// Logic and integer operations of one pattern's network per thread word (the
// generator's own statement count).
static int pattern_ops(const ScanPattern &p)
{
    Gen g;
    WordCache cache;
    gen_hit(g, p, choose_positions(p), 0, cache);
    const std::string src = g.os.str();
    return (int)std::count(src.begin(), src.end(), ';');
}

// Pairs one launch scans at most: their hit words take 512 bytes of shared
// memory per pair and warp.
constexpr int kMaxPairsPerLaunch = 4;

std::vector<std::pair<int, int>> scan_launch_groups(const std::vector<ScanPattern> &pats)
{
    // Pairs that share a launch share the loads of the planes and the tile ring; too long a
    // network spills and misses in the instruction cache.  Measured: three pairs at k = 4 (~320
    // operations per word) in three launches 3,180 us, in two 2,997, in one 2,850; four pairs
    // of k = 2, 3, 4, 2 (~350) in two launches 994 us, in one 943.
    int budget = 480;
    if (const char *e = getenv("AH_SCAN_GROUP_OPS"))
        budget = std::max(1, atoi(e));
    static std::mutex mu;
    static std::map<std::string, std::vector<std::pair<int, int>>> cache;
    std::string key = std::to_string(budget) + "|";
    for (const auto &p : pats) {
        key += std::to_string(p.L) + "," + std::to_string(p.k) + "," + std::to_string(p.pair) + ":";
        for (int i = 0; i < p.L; ++i)
            key += (char)('a' + p.mask[i]);
        key += ";";
    }
    std::lock_guard<std::mutex> lock(mu);
    auto it = cache.find(key);
    if (it != cache.end())
        return it->second;
    std::vector<std::pair<int, int>> out;
    int q = 0, start = 0, ops = 0;
    const int n = (int)pats.size();
    while (q < n) {
        int e = q, pops = 0; // the pair starting at q: [q, e)
        while (e < n && pats[e].pair == pats[q].pair)
            pops += pattern_ops(pats[e++]);
        if (q > start && (ops + pops > budget || e - start > 4 * kMaxPairsPerLaunch)) {
            out.push_back({start, q});
            start = q;
            ops = 0;
        }
        ops += pops;
        q = e;
    }
    if (n > start)
        out.push_back({start, n});
    cache[key] = out;
    return out;
}

namespace {
std::mutex g_mu;
std::map<std::string, std::unique_ptr<ScanKernel>> g_cache; // key: device + source

std::string nvrtc_err(nvrtcResult r) { return nvrtcGetErrorString(r); }
} // namespace

namespace {
std::string compile_cubin(const std::string &src, std::vector<char> *cubin, bool *ok)
{
    nvrtcProgram prog;
    nvrtcResult r = nvrtcCreateProgram(&prog, src.c_str(), "ah_scan_generated.cu", 0, nullptr, nullptr);
    if (r != NVRTC_SUCCESS)
        throw Error(AH_ERR_JIT, "nvrtcCreateProgram: " + nvrtc_err(r));
    const char *opts[] = {"-arch=sm_103a", "-std=c++17", "-lineinfo", "--ptxas-options=-v", "-DNDEBUG"};
    r = nvrtcCompileProgram(prog, 5, opts);
    size_t log_size = 0;
    nvrtcGetProgramLogSize(prog, &log_size);
    std::string log(log_size, '\0');
    if (log_size)
        nvrtcGetProgramLog(prog, &log[0]);
    *ok = (r == NVRTC_SUCCESS);
    if (*ok && cubin) {
        size_t cubin_size = 0;
        nvrtcGetCUBINSize(prog, &cubin_size);
        cubin->resize(cubin_size);
        nvrtcGetCUBIN(prog, cubin->data());
    }
    nvrtcDestroyProgram(&prog);
    return log;
}
} // namespace

std::string scan_compile_only(const std::vector<ScanPattern> &pats, const ScanTuning &t, bool *ok)
{
    return compile_cubin(scan_source(pats, t), nullptr, ok);
}

ScanKernel *scan_kernel(const std::vector<ScanPattern> &pats, const ScanTuning &t, int device)
{
    // cache key: device, tuning and the patterns (cheap; the source is only generated on a miss)
    std::string key = std::to_string(device) + "|" + std::to_string(t.R) + "," + std::to_string(t.arith_pct) + "," +
                      std::to_string(t.min_blocks) + "," + std::to_string(t.order) + "," + std::to_string(t.stages) +
                      "," + std::to_string(t.resident) + "|";
    for (auto &p : pats) {
        key += std::to_string(p.L) + "," + std::to_string(p.k) + "," + std::to_string(p.clamp) + "," +
               std::to_string(p.pair) + "," + std::to_string(p.primer) + "," + std::to_string(p.strand) + ":";
        for (int i = 0; i < p.L; ++i)
            key += (char)('a' + p.mask[i]);
        key += ";";
    }
    std::lock_guard<std::mutex> lock(g_mu);
    auto it = g_cache.find(key);
    if (it != g_cache.end())
        return it->second.get();
    const std::string src = scan_source(pats, t);
    bool ok = false;
    std::vector<char> cubin;
    std::string log = compile_cubin(src, &cubin, &ok);
    if (!ok)
        throw Error(AH_ERR_JIT, "scan kernel compilation failed: " + log.substr(0, 2000));

    auto k = std::make_unique<ScanKernel>();
    k->log = log;
    AH_CUDA(cudaLibraryLoadData(&k->lib, cubin.data(), nullptr, nullptr, 0, nullptr, nullptr, 0));
    AH_CUDA(cudaLibraryGetKernel(&k->fn, k->lib, "ah_scan_kernel"));
    const int warps = kTileW / (32 * t.R);
    k->threads = 32 * warps;
    // the ring of tiles; per warp the published hit words, the visited starts and the key stash
    k->smem = t.stages * kTileBytes + (size_t)warps * (32 * (pats.size() / 4) * t.R + 64 + 128) * sizeof(uint32_t);
    if (k->smem > 48 * 1024)
        AH_CUDA(cudaKernelSetAttributeForDevice(k->fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)k->smem,
                                                device));
    auto pos = log.find("Used ");
    if (pos != std::string::npos)
        k->regs = atoi(log.c_str() + pos + 5);
    int bps = 0;
    AH_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, (const void *)k->fn, k->threads, k->smem));
    k->blocks_per_sm = std::max(1, bps);
    if (t.resident > 0)
        k->blocks_per_sm = std::min(k->blocks_per_sm, t.resident);
    ScanKernel *raw = k.get();
    g_cache[key] = std::move(k);
    return raw;
}

} // namespace ah

// Generate and compile (no GPU needed) the scan kernel of one primer pair;
// writes the NVRTC/ptxas log (register use) into log[0..log_cap).  Returns 0
// on success.  A development aid; not part of the public header.
static int debug_scan(const char *fwd, const char *rev, int k, int R, int arith_pct, int order, char *log,
                      size_t log_cap, bool compile)
{
    try {
        std::vector<ah::ScanPattern> pats;
        const char *pr[2] = {fwd, rev};
        for (int primer = 0; primer < 2; ++primer)
            for (int strand = 0; strand < 2; ++strand) {
                ah::ScanPattern p;
                p.L = (int)strlen(pr[primer]);
                if (p.L < 1 || p.L > AH_MAX_PRIMER_LEN)
                    return 2;
                p.k = k;
                p.primer = primer;
                p.strand = strand;
                for (int i = 0; i < p.L; ++i) {
                    int m = strand == 0 ? ah::iupac_mask(pr[primer][i]) : ah::comp_mask(ah::iupac_mask(pr[primer][p.L - 1 - i]));
                    if (!m)
                        return 2;
                    p.mask[i] = (uint8_t)m;
                }
                pats.push_back(p);
            }
        ah::ScanTuning t; // no register cap: the log reports the generator's own register use
        t.R = R;
        t.arith_pct = arith_pct;
        t.order = order;
        t.min_blocks = 1;
        bool ok = false;
        std::string l = compile ? ah::scan_compile_only(pats, t, &ok) : ah::scan_source(pats, t);
        if (!compile)
            ok = true;
        if (log && log_cap) {
            size_t n = std::min(log_cap - 1, l.size());
            memcpy(log, l.data(), n);
            log[n] = 0;
        }
        return ok ? 0 : 1;
    } catch (const std::exception &e) {
        if (log && log_cap)
            snprintf(log, log_cap, "%s", e.what());
        return 3;
    }
}

extern "C" int ah_debug_compile_scan(const char *fwd, const char *rev, int k, int R, int arith_pct, int order,
                                     char *log, size_t log_cap)
{
    return debug_scan(fwd, rev, k, R, arith_pct, order, log, log_cap, true);
}

// The generated source of one pair's scan kernel (development aid).
extern "C" int ah_debug_scan_source(const char *fwd, const char *rev, int k, int R, int arith_pct, int order,
                                    char *out, size_t cap)
{
    return debug_scan(fwd, rev, k, R, arith_pct, order, out, cap, false);
}
