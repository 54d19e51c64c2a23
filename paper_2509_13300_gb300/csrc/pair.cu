// Amplicon calling (Sec. 2.1): pair '+' sites with '-' sites of the same pair
// and contig inside the length window, labelled FR/RF/FF/RR (Sec. 2.1,
// Amplicon analysis, item 1).
//
// Sites arrive in canonical order, so all sites at one (pair, contig, pos)
// are adjacent (at most F+, F-, R+, R-).  One thread owns each "start group"
// -- the '+' sites at one position (F+ and/or R+) -- and walks the sorted
// sites after it whose position can close an amplicon: right sites t with
// t >= s and t + L_Y - s in [min_len, max_len].  A count pass, an exclusive
// scan and a write pass place every group's amplicons at fixed offsets; the
// write pass merges the up-to-four (left primer, right primer) streams of its
// group by (end, orient), each of which is already sorted by end, so the
// output comes out in canonical order with no global sort.  Bound: the latency of
// a thread's dependent loads (own site, neighbours, candidates).  A site that is
// not '+' is left after its own record, the neighbours beyond the next are read
// only at a shared position, and the write pass starts from the counts, as most
// sites lead no amplicon.  Measured on a GB300: 0.94 M sites, count 20 -> 13 us,
// write 28 -> 13; 3.3 M sites, write 68 -> 20.
#include <cooperative_groups.h>
#include <cub/device/device_scan.cuh>

#include "ah_internal.h"

namespace ah {
namespace {

__device__ __forceinline__ bool same_group(const ah_site &a, const ah_site &b)
{
    return a.pair == b.pair && a.contig == b.contig && a.pos == b.pos;
}

__device__ __forceinline__ bool site_less(const ah_site &m, uint32_t pair, uint32_t contig, uint64_t t)
{
    return (m.pair < pair) || (m.pair == pair && (m.contig < contig || (m.contig == contig && m.pos < t)));
}

// First index in [lo, n) whose (pair, contig, pos) >= (pair, contig, t), by
// galloping from lo: probes lo, lo+1, lo+3, lo+7, ... then a binary search in
// the last gap.  Candidates usually sit right after the group, so this takes
// one or two dependent loads where a plain binary search over all sites takes
// log2(n).
__device__ uint64_t lower_bound_pos(const ah_site *s, uint64_t lo, uint64_t n, uint32_t pair,
                                    uint32_t contig, uint64_t t)
{
    uint64_t step = 1, hi = lo;
    while (hi < n && site_less(s[hi], pair, contig, t)) {
        lo = hi + 1;
        hi = lo + step - 1;
        step <<= 1;
    }
    if (hi > n)
        hi = n;
    while (lo < hi) { // s[lo-1] is less (or lo is the start), s[hi] is not (or hi == n)
        const uint64_t mid = (lo + hi) >> 1;
        if (site_less(s[mid], pair, contig, t))
            lo = mid + 1;
        else
            hi = mid;
    }
    return lo;
}

struct Group {
    int nl;          // number of passing left sites (0..2)
    uint64_t li[2];  // their indices
    int lx[2];       // their primers
    uint64_t first;  // first candidate index
    uint64_t tmax;   // last candidate position
    bool valid;
};

__device__ Group make_group(const ah_site *s, uint64_t n, const uint8_t *pass,
                            const PairDev *__restrict__ pairs, uint64_t a)
{
    Group g;
    g.valid = false;
    g.nl = 0;
    const ah_site sa = s[a];
    if (sa.strand != 0)
        return g;
    ah_site p = sa, q = sa; // the neighbours, loaded together; most sites are alone at their position
    if (a > 0)
        p = s[a - 1];
    if (a + 1 < n)
        q = s[a + 1];
    uint64_t g0 = a; // first site of this (pair, contig, pos) group
    for (uint64_t d = 1; d <= 3 && d <= a; ++d) {
        if (d > 1)
            p = s[a - d];
        if (!same_group(p, sa))
            break;
        if (p.strand == 0)
            return g; // an earlier '+' site leads this group
        g0 = a - d;
    }
    if (!pass || pass[a]) {
        g.li[0] = a;
        g.lx[0] = sa.primer;
        g.nl = 1;
    }
    for (uint64_t d = 1; d <= 3 && a + d < n; ++d) {
        if (d > 1)
            q = s[a + d];
        if (!same_group(q, sa))
            break;
        if (q.strand == 0 && (!pass || pass[a + d])) {
            (g.nl ? g.li[1] : g.li[0]) = a + d;
            (g.nl ? g.lx[1] : g.lx[0]) = q.primer;
            ++g.nl;
        }
    }
    if (g.nl == 0)
        return g;
    const PairDev &pd = pairs[sa.pair];
    const int Lmin = min(pd.L[0], pd.L[1]), Lmax = max(pd.L[0], pd.L[1]);
    const int64_t lo = max((int64_t)0, (int64_t)pd.min_len - Lmax);
    const int64_t hi = (int64_t)pd.max_len - Lmin;
    if (hi < lo)
        return g;
    g.first = lower_bound_pos(s, g0, n, sa.pair, sa.contig, (uint64_t)sa.pos + (uint64_t)lo);
    g.tmax = (uint64_t)sa.pos + (uint64_t)hi;
    g.valid = true;
    return g;
}

__device__ __forceinline__ bool in_window(const PairDev &pd, uint32_t s_pos, const ah_site &r, uint32_t *end)
{
    const int64_t e = (int64_t)r.pos + pd.L[r.primer];
    const int64_t len = e - (int64_t)s_pos;
    *end = (uint32_t)e;
    return r.pos >= s_pos && len >= pd.min_len && len <= pd.max_len;
}

__device__ __forceinline__ int orient_of(int x, int y) { return (x == 0 && y == 1) ? 0 : (x == 1 && y == 0) ? 1 : (x == 0 ? 2 : 3); }

// Amplicons of the group that site a leads, and the sum of their lengths.
__device__ __forceinline__ uint64_t count_group(const ah_site *s, uint64_t n, const uint8_t *pass,
                                                const PairDev *__restrict__ pairs, uint64_t a, uint64_t *bases)
{
    uint64_t cnt = 0;
    *bases = 0;
    const Group g = make_group(s, n, pass, pairs, a);
    if (!g.valid)
        return 0;
    const ah_site sa = s[a];
    const PairDev &pd = pairs[sa.pair];
    for (uint64_t b = g.first; b < n; ++b) {
        const ah_site r = s[b];
        if (r.pair != sa.pair || r.contig != sa.contig || r.pos > g.tmax)
            break;
        if (r.strand != 1 || (pass && !pass[b]))
            continue;
        uint32_t end;
        if (in_window(pd, sa.pos, r, &end)) {
            cnt += g.nl;
            *bases += (uint64_t)g.nl * (end - sa.pos);
        }
    }
    return cnt;
}

// Write them from out[o] on, those below cap; with qoff, also the sequence offset of each, the
// first at base.
__device__ __forceinline__ void write_group(const ah_site *s, uint64_t n, const uint8_t *pass,
                                            const PairDev *__restrict__ pairs, uint64_t a, uint64_t o, uint64_t base,
                                            ah_amplicon *out, uint64_t *qoff, uint64_t cap)
{
    const Group g = make_group(s, n, pass, pairs, a);
    if (!g.valid)
        return;
    const ah_site sa = s[a];
    const PairDev &pd = pairs[sa.pair];
    // streams: (left index li, right primer y); cursor = next candidate index
    uint64_t cur[4];
    const int ns = g.nl * 2;
    auto advance = [&](int st, uint64_t from) -> uint64_t {
        const int y = st & 1;
        for (uint64_t b = from; b < n; ++b) {
            const ah_site r = s[b];
            if (r.pair != sa.pair || r.contig != sa.contig || r.pos > g.tmax)
                return n;
            if (r.strand != 1 || r.primer != y || (pass && !pass[b]))
                continue;
            uint32_t end;
            if (in_window(pd, sa.pos, r, &end))
                return b;
        }
        return n;
    };
    for (int st = 0; st < ns; ++st)
        cur[st] = advance(st, g.first);
    for (;;) {
        int best = -1;
        uint32_t bend = 0;
        int bor = 0;
        for (int st = 0; st < ns; ++st) {
            if (cur[st] >= n)
                continue;
            const ah_site r = s[cur[st]];
            const uint32_t end = r.pos + pd.L[r.primer];
            const int orr = orient_of(g.lx[st >> 1], r.primer);
            if (best < 0 || end < bend || (end == bend && orr < bor)) {
                best = st;
                bend = end;
                bor = orr;
            }
        }
        if (best < 0)
            break;
        if (o < cap) {
            ah_amplicon am;
            am.genome = sa.genome;
            am.contig = sa.contig;
            am.start = sa.pos;
            am.end = bend;
            am.left = (uint32_t)g.li[best >> 1];
            am.right = (uint32_t)cur[best];
            am.orient = (uint8_t)bor;
            am.pair = sa.pair;
            am.pad0 = am.pad1 = 0;
            out[o] = am;
            if (qoff) {
                qoff[o] = base;
                base += bend - sa.pos;
            }
        }
        ++o;
        cur[best] = advance(best, cur[best] + 1);
    }
}

__global__ void pair_count_kernel(const ah_site *s, uint64_t n, const uint8_t *pass, const PairDev *__restrict__ pairs,
                                  uint64_t *counts, const int *err)
{
    chain_start();
    chain_wait();
    if (err && *(volatile const int *)err) // the records' check failed: nothing is indexed with them
        return;
    for (uint64_t a = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; a < n; a += (uint64_t)gridDim.x * blockDim.x) {
        uint64_t bases;
        counts[a] = count_group(s, n, pass, pairs, a, &bases);
    }
}

__global__ void pair_write_kernel(const ah_site *s, uint64_t n, const uint8_t *pass, const PairDev *__restrict__ pairs,
                                  const uint64_t *counts, const uint64_t *offsets, ah_amplicon *out, uint64_t cap)
{
    chain_start();
    chain_wait();
    for (uint64_t a = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; a < n; a += (uint64_t)gridDim.x * blockDim.x)
        if (counts[a]) // most sites lead no amplicon
            write_group(s, n, pass, pairs, a, offsets[a], 0, out, nullptr, cap);
}

// Both passes and the scan between them in one launch, for at most kSmallSort sites whose count
// is on the device: a cluster of kPairCtas CTAs, a thread per site.  Counts and lengths stay in
// registers; they are scanned within the warp, and every CTA scans the totals of all the cluster's
// warps, read through distributed shared memory.  The sequence offsets follow from the same scan.
// Groups of 32 sites go to the CTAs in turn: few sites, or the neighbouring sites of a hot spot
// that lead many amplicons each, keep all 16 SMs at work (5,000 sites of 62,500 amplicons: 103
// us with 1,024 neighbours per CTA, five SMs at work, 62 so; 6,000 sites 2 us less).  Sixteen
// CTAs are beyond the cluster size that every device has room for (eight): where
// pair_run_available finds none, runs go step by step, with the kernels above.
// Bound: latency, and the host's launches around it.  Measured on a GB300 from the end of the
// Tm kernel to the sequence decode: four launches (count, scan, write, scan of the lengths)
// 9.3 us for 14 sites, 15 for 6,000 -> 8 to 9 and 10; the run of a small resident set, which waits
// for the host's launches too, 93 -> 88.  A cluster of eight with two sites per thread took
// 18 us for 10,000 sites against 15.  Beside another stream's packing, whose blocks it waits for
// (16 SMs of one GPC must have room at once), 28 us against 13 alone for 10,000 sites; the
// launches it replaces took 39 and 26 there.
constexpr int kPairCtas = 16, kPairThreads = 1024, kPairWarps = kPairThreads / 32;
constexpr int kPairSets = kPairCtas * kPairWarps; // groups of 32 sites
static_assert(kPairSets * 32 == kSmallSort && kPairSets <= kPairThreads && kPairCtas == 16, "a thread per site, and per set");

__global__ void __cluster_dims__(kPairCtas, 1, 1) __launch_bounds__(kPairThreads)
    pair_run_kernel(const ah_site *s, uint64_t n_arg, const uint64_t *n_dev, const uint8_t *pass,
                    const PairDev *__restrict__ pairs, ah_amplicon *out, uint64_t *qoff, uint64_t amps_max,
                    uint64_t seq_max, uint64_t *n_amps, uint64_t *n_seq, uint64_t *redo)
{
    namespace cg = cooperative_groups;
    __shared__ ulonglong2 warp_sum[kPairWarps];               // amplicons and bases of this CTA's warps
    __shared__ ulonglong2 before_warp[kPairWarps];            // ... of all sites before them
    __shared__ ulonglong2 set_sum[kPairSets / 32];            // ... of 32 sets
    const cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank(), tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // inclusive over the lanes
    auto scan2 = [&](uint64_t &c, uint64_t &l) {
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint64_t x = __shfl_up_sync(0xffffffffu, c, d), y = __shfl_up_sync(0xffffffffu, l, d);
            if (lane >= d) {
                c += x;
                l += y;
            }
        }
    };
    chain_start();
    chain_wait();
    const uint64_t n = dev_count(n_arg, n_dev);
    const uint64_t a = (uint64_t)(warp * kPairCtas + rank) * 32 + lane; // set (warp, rank) of the sites
    uint64_t cnt = 0, len = 0;
    if (a < n)
        cnt = count_group(s, n, pass, pairs, a, &len);
    uint64_t icnt = cnt, ilen = len; // inclusive in the warp
    scan2(icnt, ilen);
    if (lane == 31)
        warp_sum[warp] = make_ulonglong2(icnt, ilen);
    cluster.sync(); // every warp's totals
    uint64_t c = 0, l = 0;
    ulonglong2 own = make_ulonglong2(0, 0); // of set tid, in the sites' order
    if (tid < kPairSets) {
        own = *cluster.map_shared_rank(&warp_sum[tid / kPairCtas], tid % kPairCtas);
        c = own.x;
        l = own.y;
        scan2(c, l);
        if (lane == 31)
            set_sum[warp] = make_ulonglong2(c, l);
    }
    __syncthreads();
    uint64_t total = 0, bases = 0; // of all sites
#pragma unroll
    for (int w = 0; w < kPairSets / 32; ++w) {
        if (w == warp) {
            c += total;
            l += bases;
        }
        total += set_sum[w].x;
        bases += set_sum[w].y;
    }
    if (tid < kPairSets && tid % kPairCtas == rank)
        before_warp[tid / kPairCtas] = make_ulonglong2(c - own.x, l - own.y);
    cluster.sync(); // before_warp; and no block leaves while its totals are read
    const bool fits = total <= amps_max;
    if (rank == 0 && tid == 0) {
        *n_amps = fits ? total : 0;
        const bool seq_fits = !fits || bases <= seq_max;
        *n_seq = fits && seq_fits ? bases : 0;
        qoff[fits ? total : 0] = fits ? bases : 0;
        if (!fits || !seq_fits)
            atomicOr((unsigned long long *)redo, (unsigned long long)(!fits ? kRedoAmps : kRedoSeq));
    }
    if (fits && cnt)
        write_group(s, n, pass, pairs, a, before_warp[warp].x + icnt - cnt, before_warp[warp].y + ilen - len, out, qoff,
                    amps_max);
}

__global__ void total_kernel(const uint64_t *offs, const uint64_t *counts, uint64_t n, uint64_t *out)
{
    chain_start();
    chain_wait();
    *out = n ? offs[n - 1] + counts[n - 1] : 0;
}

// One-block exclusive scan of n u64 values, 4096 at a time: coalesced loads (four per thread in
// flight) staged through shared memory, each thread scans four consecutive values, warp shuffles
// and one shared pass scan the 1024 thread sums, and the results leave through shared memory as
// coalesced stores.
__global__ void __launch_bounds__(1024) scan_small_kernel(const uint64_t *in, uint64_t *out, uint32_t n)
{
    chain_start();
    chain_wait();
    __shared__ uint64_t buf[4096];
    __shared__ uint64_t wsum[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint64_t carry = 0;
    for (uint32_t base = 0; base < n; base += 4096) {
        uint64_t v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const uint32_t i = base + tid + 1024u * u;
            v[u] = i < n ? in[i] : 0;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            buf[tid + 1024 * u] = v[u];
        __syncthreads();
        const uint64_t x0 = buf[4 * tid], x1 = buf[4 * tid + 1], x2 = buf[4 * tid + 2], x3 = buf[4 * tid + 3];
        const uint64_t sum = x0 + x1 + x2 + x3;
        uint64_t incl = sum;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint64_t y = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d)
                incl += y;
        }
        if (lane == 31)
            wsum[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            uint64_t w = wsum[lane];
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint64_t y = __shfl_up_sync(0xffffffffu, w, d);
                if (lane >= d)
                    w += y;
            }
            wsum[lane] = w;
        }
        __syncthreads();
        const uint64_t ex = carry + (warp ? wsum[warp - 1] : 0) + incl - sum;
        buf[4 * tid] = ex;
        buf[4 * tid + 1] = ex + x0;
        buf[4 * tid + 2] = ex + x0 + x1;
        buf[4 * tid + 3] = ex + x0 + x1 + x2;
        carry += wsum[31];
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const uint32_t i = base + tid + 1024u * u;
            if (i < n)
                out[i] = buf[tid + 1024 * u];
        }
        __syncthreads(); // buf and wsum are rewritten by the next chunk
    }
}

unsigned grid_for(uint64_t n, int threads)
{
    uint64_t b = (n + threads - 1) / threads;
    if (b > 16384)
        b = 16384;
    if (b == 0)
        b = 1;
    return (unsigned)b;
}

} // namespace

void launch_pair_count(const ah_site *sites, uint64_t n, const uint8_t *pass, const PairDev *pairs_d, uint64_t *counts,
                       const int *err, cudaStream_t s)
{
    if (!n)
        return;
    launch_chained(pair_count_kernel, grid_for(n, 128), 128, 0, s, sites, n, pass, pairs_d, counts, err);
}

bool pair_run_available()
{
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = kPairCtas;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(kPairCtas);
    cfg.blockDim = dim3(kPairThreads);
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    int clusters = 0;
    const bool ok =
        cudaFuncSetAttribute(pair_run_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&clusters, pair_run_kernel, &cfg) == cudaSuccess && clusters > 0;
    if (!ok)
        cudaGetLastError(); // (not an error: the step-by-step form needs no cluster)
    return ok;
}

void launch_pair_run(const ah_site *sites, uint64_t n, const uint64_t *n_dev, const uint8_t *pass,
                     const PairDev *pairs_d, ah_amplicon *out, uint64_t *seq_offsets, uint64_t amps_max,
                     uint64_t seq_max, uint64_t *n_amps, uint64_t *n_seq, uint64_t *redo, cudaStream_t s)
{
    if (n == 0 || n > kSmallSort)
        throw Error(AH_ERR_ARG, "pairing with a device count: size outside 1..16384");
    launch_chained(pair_run_kernel, kPairCtas, kPairThreads, 0, s, sites, n, n_dev, pass, pairs_d, out, seq_offsets,
                   amps_max, seq_max, n_amps, n_seq, redo);
}

void launch_total(const uint64_t *offs, const uint64_t *counts, uint64_t n, uint64_t *out, cudaStream_t s)
{
    launch_chained(total_kernel, 1, 1, 0, s, offs, counts, n, out);
}

size_t scan_u64_temp_bytes(uint64_t n)
{
    size_t bytes = 0;
    AH_CUDA(cub::DeviceScan::ExclusiveSum(nullptr, bytes, (const uint64_t *)nullptr, (uint64_t *)nullptr, (int64_t)n));
    return bytes;
}

void exclusive_scan_u64(void *temp, size_t temp_bytes, const uint64_t *in, uint64_t *out, uint64_t n, cudaStream_t s)
{
    if (n == 0)
        return;
    if (n <= kOneBlockScan) {
        launch_chained(scan_small_kernel, 1, 1024, 0, s, in, out, (uint32_t)n);
        return;
    }
    AH_CUDA(cub::DeviceScan::ExclusiveSum(temp, temp_bytes, in, out, (int64_t)n, s));
}

int scan_u64_launches(uint64_t n) { return n == 0 ? 0 : n <= kOneBlockScan ? 1 : 2; }

void launch_pair_write(const ah_site *sites, uint64_t n, const uint8_t *pass, const PairDev *pairs_d,
                       const uint64_t *counts, const uint64_t *offsets, ah_amplicon *out, uint64_t cap, cudaStream_t s)
{
    if (!n)
        return;
    launch_chained(pair_write_kernel, grid_for(n, 128), 128, 0, s, sites, n, pass, pairs_d, counts, offsets, out, cap);
}

} // namespace ah
