// Amplicon sequence variants and amplitypes (Sec. 3.3, Amplicon Pattern
// Visualization: an amplitype is a genome's combination of amplicon sequence
// variants and their copy numbers; genomes sharing one are grouped).
//
// Variants: each amplicon's sequence (as ah_fetch returns it: RF reverse-
// complemented, N for any non-ACGT letter) is hashed straight from the packed
// planes with two polynomial hashes modulo the Mersenne prime 2^61 - 1 (the second
// with the length's low three bits beside it); amplicons with equal pairs are one
// variant.  Variants, and then
// amplitypes, are numbered by first occurrence: every element enters a hash
// table in device memory (open addressing) that keeps the smallest index seen
// per key, so the elements that are their key's smallest are the first
// occurrences, and their ranks in input order are the ids.  Which slot a key
// lands in depends on the order of arrival, the ids do not.  Amplitype of a
// genome: the multiset of (variant, copies), hashed as a sum of mixed 64-bit
// words per (variant, copies) pair (two independent sums, order-free), the
// copies counted in a second table keyed by (genome, variant).
//
// Bound: launches, memory latency and, in the hashing, issue slots (ncu: issue 0.68,
// ALU pipe 65 %, of the 16 bytes of planes per letter five in six from L1, 264 MB from
// L2, 76 from DRAM; a sixth fewer instructions per letter changed nothing).
// Measured on a GB300, 65,000 amplicons of ~1,500 letters: hashing 399 us (a lane per
// 1/32 of an amplicon, letter by letter) -> 122; the rest of a call 3 x 16 radix-sort
// passes and ~60 small launches, 0.7 ms -> 15 launches, 0.13 ms.  (Fewer blocks for the
// kernels that enter a table, so that common keys are entered before most elements
// look: 39 -> 58 us, not kept.)
#include <algorithm>

#include "ah_internal.h"

namespace ah {
namespace {

constexpr uint64_t kM61 = (1ull << 61) - 1;
constexpr uint64_t kB1 = 0x1d2e3f4a5b6c7d8ull % kM61; // hash bases (any values in [2, 2^61 - 2])
constexpr uint64_t kB2 = 0x0f1e2d3c4b5a697ull % kM61;
constexpr unsigned long long kEmpty = ~0ull;

__host__ __device__ constexpr uint64_t mod61(uint64_t x)
{
    x = (x & kM61) + (x >> 61);
    return x >= kM61 ? x - kM61 : x;
}

// a * b mod 2^61 - 1 for a, b < 2^61: the 122-bit product folded at bit 61
__device__ __forceinline__ uint64_t mulmod61(uint64_t a, uint64_t b)
{
    const uint64_t lo = a * b, hi = __umul64hi(a, b);
    return mod61((lo & kM61) + (lo >> 61) + (hi << 3));
}

// base^(31 - lane) for the 32 lanes and, last, base^32 (built at compile time)
constexpr uint64_t mul61(uint64_t a, uint64_t b)
{
    const unsigned __int128 p = (unsigned __int128)a * b;
    return mod61((uint64_t)(p & kM61) + (uint64_t)(p >> 61));
}
struct Powers {
    uint64_t v[33];
};
constexpr Powers powers(uint64_t base)
{
    Powers p{};
    p.v[31] = 1;
    for (int i = 30; i >= 0; --i)
        p.v[i] = mul61(p.v[i + 1], base);
    p.v[32] = mul61(p.v[0], base);
    return p;
}
__constant__ Powers kPow1 = powers(kB1);
__constant__ Powers kPow2 = powers(kB2);

// 64-bit finaliser of the SplitMix generator (Steele, Lea and Flood, 2014)
__device__ __forceinline__ uint64_t mix64(uint64_t x)
{
    x ^= x >> 30;
    x *= 0xbf58476d1ce4e5b9ull;
    x ^= x >> 27;
    x *= 0x94d049bb133111ebull;
    x ^= x >> 31;
    return x;
}

// Sum of the lanes' values modulo 2^61 - 1 (each below 2^61), in every lane.
__device__ __forceinline__ uint64_t sum61(uint64_t v)
{
#pragma unroll
    for (int d = 1; d <= 4; d <<= 1) // eight values stay below 2^64
        v += __shfl_xor_sync(0xffffffffu, v, d);
    v = mod61(v);
    v += __shfl_xor_sync(0xffffffffu, v, 8);
    v += __shfl_xor_sync(0xffffffffu, v, 16);
    return mod61(v);
}

// The slot of key (a, b) in an open-addressing table; claims a free one.  Keys
// of a slot never change once set, and every element of a key meets the slots
// in the same order, so equal keys always end at the same slot.  With one
// word per key pass k2 = nullptr.
__device__ uint64_t table_slot(unsigned long long *k1, unsigned long long *k2, uint64_t size, uint64_t a, uint64_t b)
{
    uint64_t i = __umul64hi(mix64(a ^ (b * 0x9e3779b97f4a7c15ull)), size);
    for (;;) {
        unsigned long long x = *(volatile unsigned long long *)(k1 + i);
        if (x == kEmpty)
            x = atomicCAS(k1 + i, kEmpty, (unsigned long long)a);
        if (x == kEmpty || x == a) {
            if (!k2)
                return i;
            unsigned long long y = *(volatile unsigned long long *)(k2 + i);
            if (y == kEmpty)
                y = atomicCAS(k2 + i, kEmpty, (unsigned long long)b);
            if (y == kEmpty || y == b)
                return i;
        }
        i = i + 1 == size ? 0 : i + 1;
    }
}

__device__ __forceinline__ void note_first(unsigned int *first, uint64_t slot, uint32_t i)
{
    if (*(volatile unsigned int *)(first + slot) > i) // (most are not smaller: no atomic)
        atomicMin(first + slot, i);
}

constexpr int kDigitLetters = 20;

// Lane `lane`'s digit of the group of 32 * kDigitLetters letters at `first` (the
// flat position of the group's letter 0), of which `left` are in the amplicon:
// the letters lane, lane + 32, ..., three bits each (a base: 4 + its code with
// A 0, C 1, G 2, T 3; else 0).  RC: the letters run backwards and are
// complemented (code 3 - code: the planes in reverse order).  Positions are
// counted from the start of the group's tile (RC: of the tile before it), so
// they fit in 32 bits and reach one tile further at most.
template <bool RC>
__device__ __forceinline__ uint64_t group_digit(const uint32_t *__restrict__ planes, uint64_t first, uint32_t left, int lane)
{
    const uint32_t *tile = planes + (int64_t)(first / kTileBases - (RC ? 1 : 0)) * (4 * kTileWX);
    const uint32_t rel0 = (uint32_t)(first % kTileBases) + (RC ? (uint32_t)kTileBases - lane : (uint32_t)lane);
    uint64_t d = 0;
    for (uint32_t c0 = 0; c0 < kDigitLetters && 32 * c0 < left; c0 += 4) { // four letters' loads in flight
        uint32_t w[4][4], b[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t q = 32 * (c0 + j), rel = RC ? rel0 - q : rel0 + q;
            b[j] = (rel / kTileW) & 31u;
            const uint32_t *wp = tile + (rel / (uint32_t)kTileBases * (4 * kTileWX) + rel % kTileW);
            const bool in = q + lane < left;
#pragma unroll
            for (int x = 0; x < 4; ++x)
                w[j][x] = in ? __ldg(wp + (RC ? 3 - x : x) * kTileWX) : 0u;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t lo = w[j][1] | w[j][3], hi = w[j][2] | w[j][3], any = lo | w[j][2] | w[j][0];
            d = d << 3 | (((any >> b[j]) & 1u) << 2 | ((hi >> b[j]) & 1u) << 1 | ((lo >> b[j]) & 1u));
        }
    }
    return d;
}

// One warp per amplicon: the record's check and its two hashes.  A group of 640
// letters is 32 digits of 60 bits, one per lane (four coalesced loads per 32
// letters: consecutive positions lie in consecutive words), each times its
// power of the base; hash = the groups in order (zeros beyond the end), then
// the length.  (Neither word is ever the empty key: the low 61 bits are below 2^61 - 1.)
// A bad record sets *err.  65,000 amplicons of ~1,500 letters: 121 us.
__global__ void amp_hash_kernel(const ah_amplicon *__restrict__ a, uint64_t n, const uint32_t *__restrict__ planes,
                                const uint64_t *__restrict__ contig_off, const uint32_t *__restrict__ contig_genome,
                                uint32_t n_contigs, uint64_t *__restrict__ hash1, uint64_t *__restrict__ hash2,
                                int *__restrict__ err)
{
    constexpr uint32_t kGroup = 32 * kDigitLetters;
    const int lane = threadIdx.x & 31;
    const uint64_t pow1 = kPow1.v[lane], pow2 = kPow2.v[lane];
    const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x / 32);
    for (uint64_t i = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32; i < n; i += warps) {
        const ah_amplicon am = a[i];
        bool ok = am.contig < n_contigs && am.start <= am.end && am.orient <= 3;
        if (ok)
            ok = (uint64_t)am.end <= contig_off[am.contig + 1] - contig_off[am.contig] &&
                 am.genome == contig_genome[am.contig];
        if (!ok) {
            if (lane == 0) {
                atomicExch(err, kDevBounds);
                hash1[i] = hash2[i] = 0;
            }
            continue;
        }
        const uint32_t len = am.end - am.start;
        const uint64_t base = contig_off[am.contig] + am.start;
        uint64_t h1 = 0, h2 = 0;
        for (uint64_t g = 0; g < len; g += kGroup) {
            const uint32_t left = (uint32_t)min((uint64_t)kGroup, len - g);
            const uint64_t d = am.orient == 1 ? group_digit<true>(planes, base + len - 1 - g, left, lane)
                                              : group_digit<false>(planes, base + g, left, lane);
            h1 = mod61(mulmod61(h1, kPow1.v[32]) + sum61(mulmod61(d, pow1)));
            h2 = mod61(mulmod61(h2, kPow2.v[32]) + sum61(mulmod61(d, pow2)));
        }
        if (lane == 0) {
            hash1[i] = mod61(mulmod61(h1, kB1) + len);
            hash2[i] = mod61(mulmod61(h2, kB2) + len) | (uint64_t)len << 61; // its low three bits beside the hash
        }
    }
}

// Every amplicon's slot in the variant table.  Equal keys of a warp enter the
// table once, by their first lane (the smallest index): a common variant's slot
// is one address for the whole GPU.
__global__ void variant_slots_kernel(uint64_t n, const uint64_t *__restrict__ hash1, const uint64_t *__restrict__ hash2,
                                     AmpliTables t, uint32_t *__restrict__ slot)
{
    const int lane = threadIdx.x & 31;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i0 = (uint64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); i0 < n; i0 += stride) {
        const uint64_t i = i0 + lane;
        const bool in = i < n;
        const uint64_t a = in ? hash1[i] : kEmpty, b = in ? hash2[i] : kEmpty;
        const uint32_t same = __match_any_sync(0xffffffffu, a) & __match_any_sync(0xffffffffu, b);
        const int lead = __ffs(same) - 1;
        uint32_t s = 0;
        if (in && lane == lead) {
            s = (uint32_t)table_slot(t.k1, t.k2, t.size, a, b);
            note_first(t.first, s, (uint32_t)i);
        }
        s = __shfl_sync(0xffffffffu, s, lead);
        if (in)
            slot[i] = s;
    }
}

// flag[i] = element i is its key's first occurrence; 0 for i in [n, cap)
__global__ void first_flags_kernel(const unsigned int *__restrict__ first, const uint32_t *__restrict__ slot,
                                   const uint64_t *__restrict__ n_dev, uint64_t cap, uint64_t *__restrict__ flag)
{
    const uint64_t n = dev_count(cap, n_dev);
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < cap; i += (uint64_t)gridDim.x * blockDim.x)
        flag[i] = i < n && first[slot[i]] == (uint32_t)i ? 1 : 0;
}

// variant ids, and the copies of every (genome, variant) in the second table
__global__ void variants_kernel(const ah_amplicon *__restrict__ a, uint64_t n, AmpliTables t,
                                const uint32_t *__restrict__ slot, const uint64_t *__restrict__ flag,
                                const uint64_t *__restrict__ rank, uint32_t *__restrict__ variant,
                                uint64_t *__restrict__ n_variants, const int *__restrict__ err)
{
    if (__syncthreads_or(*(volatile const int *)err)) // (the records are not to be trusted; the call reports it)
        return;
    const int lane = threadIdx.x & 31;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i0 = (uint64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); i0 < n; i0 += stride) {
        const uint64_t i = i0 + lane;
        const bool in = i < n;
        uint64_t key = kEmpty;
        if (in) {
            const uint32_t v = (uint32_t)rank[t.first[slot[i]]];
            variant[i] = v;
            key = (uint64_t)a[i].genome << 32 | v;
            if (i == n - 1)
                *n_variants = rank[i] + flag[i];
        }
        const uint32_t same = __match_any_sync(0xffffffffu, key); // (amplicons of a genome are neighbours)
        if (in && lane == __ffs(same) - 1)
            atomicAdd(t.pair_n + table_slot(t.pair_key, nullptr, t.size, key, 0), (unsigned int)__popc(same));
    }
}

// per (genome, variant) with its copies: the genome's sums
__global__ void genome_sums_kernel(AmpliTables t, unsigned long long *__restrict__ g1, unsigned long long *__restrict__ g2,
                                   unsigned int *__restrict__ gamp, unsigned int *__restrict__ gvar)
{
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < t.size; i += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t key = t.pair_key[i];
        if (key == kEmpty)
            continue;
        const uint32_t g = (uint32_t)(key >> 32), copies = t.pair_n[i];
        const uint64_t v = key & 0xffffffffull;
        atomicAdd(g1 + g, (unsigned long long)mix64((v << 32 | copies) * 2 + 1));
        atomicAdd(g2 + g, (unsigned long long)mix64((v << 32 | copies) ^ 0x9e3779b97f4a7c15ull));
        atomicAdd(gamp + g, copies);
        atomicAdd(gvar + g, 1u);
    }
}

__global__ void genome_flags_kernel(const unsigned int *__restrict__ gamp, uint64_t n, uint64_t *__restrict__ has)
{
    for (uint64_t g = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; g < n; g += (uint64_t)gridDim.x * blockDim.x)
        has[g] = gamp[g] ? 1 : 0;
}

// genomes with amplicons (ascending id) as rows, and each row's slot in the amplitype table
__global__ void genome_rows_kernel(const uint64_t *__restrict__ has, const uint64_t *__restrict__ pos, uint64_t n,
                                   const unsigned long long *__restrict__ g1, const unsigned long long *__restrict__ g2,
                                   AmpliTables t, uint32_t *__restrict__ gid, uint32_t *__restrict__ slot,
                                   uint64_t *__restrict__ n_rows)
{
    for (uint64_t g = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; g < n; g += (uint64_t)gridDim.x * blockDim.x) {
        if (has[g]) {
            const uint64_t r = pos[g];
            gid[r] = (uint32_t)g;
            // (without its top bit a sum is never the empty key)
            const uint64_t s = table_slot(t.k1, t.k2, t.size, g1[g] & ~(1ull << 63), g2[g] & ~(1ull << 63));
            note_first(t.first, s, (uint32_t)r);
            slot[r] = (uint32_t)s;
        }
        if (g == n - 1)
            *n_rows = pos[g] + has[g];
    }
}

__global__ void rows_kernel(const uint32_t *__restrict__ gid, const uint32_t *__restrict__ slot, AmpliTables t,
                            const uint64_t *__restrict__ n_rows, uint64_t cap, const uint64_t *__restrict__ flag,
                            const uint64_t *__restrict__ rank, const unsigned int *__restrict__ gamp,
                            const unsigned int *__restrict__ gvar, ah_genome_amplitype *__restrict__ rows,
                            uint64_t *__restrict__ n_types)
{
    const uint64_t n = dev_count(cap, n_rows);
    if (n == 0 && blockIdx.x == 0 && threadIdx.x == 0)
        *n_types = 0;
    for (uint64_t r = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t g = gid[r];
        rows[r] = {g, (uint32_t)rank[t.first[slot[r]]], gamp[g], gvar[g]};
        if (r == n - 1)
            *n_types = rank[r] + flag[r];
    }
}

unsigned grid(uint64_t n, int threads = 256)
{
    const uint64_t b = (n + threads - 1) / threads;
    return (unsigned)std::max<uint64_t>(1, std::min<uint64_t>(b, 8192));
}

} // namespace

// Slots for n keys: at most two in three are taken.
// Slots are numbered in 32 bits; there is always one for every key (n < 2^32).
uint64_t amplitype_slots(uint64_t n) { return std::min<uint64_t>(n + n / 2 + 64, 0xffffffffull); }

void launch_amplitypes(const ah_amplicon *a, uint64_t n, const uint32_t *planes, const uint64_t *contig_off,
                       const uint32_t *contig_genome, uint32_t n_contigs, uint64_t n_ids, const AmpliScratch &S,
                       uint64_t *counts, int *err, cudaStream_t s)
{
    if (!n)
        return;
    // the tables' keys and first occurrences empty; counts and sums zero
    AH_CUDA(cudaMemsetAsync(S.ones, 0xff, S.ones_bytes, s));
    AH_CUDA(cudaMemsetAsync(S.zeros, 0, S.zeros_bytes, s));
    amp_hash_kernel<<<grid(n * 32), 256, 0, s>>>(a, n, planes, contig_off, contig_genome, n_contigs, S.flag, S.rank, err);
    AH_CUDA(cudaGetLastError());
    variant_slots_kernel<<<grid(n), 256, 0, s>>>(n, S.flag, S.rank, S.t, S.slot); // (the hashes' arrays are free after it)
    AH_CUDA(cudaGetLastError());
    first_flags_kernel<<<grid(n), 256, 0, s>>>(S.t.first, S.slot, nullptr, n, S.flag);
    AH_CUDA(cudaGetLastError());
    exclusive_scan_u64(S.scan_temp, S.scan_bytes, S.flag, S.rank, n, s);
    variants_kernel<<<grid(n), 256, 0, s>>>(a, n, S.t, S.slot, S.flag, S.rank, S.variant, counts + 0, err);
    AH_CUDA(cudaGetLastError());
    genome_sums_kernel<<<grid(S.t.size), 256, 0, s>>>(S.t, S.g1, S.g2, S.gamp, S.gvar);
    AH_CUDA(cudaGetLastError());
    genome_flags_kernel<<<grid(n_ids), 256, 0, s>>>(S.gamp, n_ids, S.has);
    AH_CUDA(cudaGetLastError());
    exclusive_scan_u64(S.scan_temp, S.scan_bytes, S.has, S.pos, n_ids, s);
    // the first table again, for the genomes' sums (at most min(n, n_ids) rows)
    const uint64_t most = std::min(n, n_ids);
    AH_CUDA(cudaMemsetAsync(S.ones, 0xff, S.ones_bytes, s));
    genome_rows_kernel<<<grid(n_ids), 256, 0, s>>>(S.has, S.pos, n_ids, S.g1, S.g2, S.t, S.gid, S.slot, counts + 1);
    AH_CUDA(cudaGetLastError());
    first_flags_kernel<<<grid(most), 256, 0, s>>>(S.t.first, S.slot, counts + 1, most, S.flag);
    AH_CUDA(cudaGetLastError());
    exclusive_scan_u64(S.scan_temp, S.scan_bytes, S.flag, S.rank, most, s);
    rows_kernel<<<grid(most), 256, 0, s>>>(S.gid, S.slot, S.t, counts + 1, most, S.flag, S.rank, S.gamp, S.gvar, S.rows,
                                           counts + 2);
    AH_CUDA(cudaGetLastError());
}

int amplitype_launches(uint64_t n, uint64_t n_ids)
{
    return 9 + scan_u64_launches(n) + scan_u64_launches(n_ids) + scan_u64_launches(std::min(n, n_ids));
}

} // namespace ah
