// Site keys -> canonical order -> site records.
//
// The scan appends 64-bit keys in whatever order warps finish; a radix sort
// over the key bits that carry (pair, flat position, primer, strand) gives
// the canonical order (pair, contig, pos, primer, strand), since contigs are
// laid out in load order.  The decode kernel then finds each key's contig by
// binary search over the contig offsets.
#include <cub/device/device_radix_sort.cuh>

#include "ah_internal.h"

namespace ah {
namespace {

__global__ void decode_keys_kernel(const uint64_t *__restrict__ keys, uint64_t n, int pbits,
                                   const uint64_t *__restrict__ contig_off, uint32_t n_contigs,
                                   const uint32_t *__restrict__ contig_genome, ah_site *__restrict__ out)
{
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t key = keys[i];
        const uint64_t pp = key >> 10;
        const uint64_t P = pp & ((1ull << pbits) - 1);
        const uint32_t pair = (uint32_t)(pp >> pbits);
        uint32_t lo = 0, hi = n_contigs;
        while (hi - lo > 1) {
            uint32_t mid = (lo + hi) >> 1;
            if (contig_off[mid] <= P)
                lo = mid;
            else
                hi = mid;
        }
        ah_site s;
        s.genome = contig_genome[lo];
        s.contig = lo;
        s.pos = (uint32_t)(P - contig_off[lo]);
        s.primer = (uint8_t)((key >> 9) & 1);
        s.strand = (uint8_t)((key >> 8) & 1);
        s.mm = (uint8_t)(key & 0xff);
        s.pair = (uint8_t)pair;
        out[i] = s;
    }
}

__global__ void validate_sites_kernel(const ah_site *__restrict__ sites, uint64_t n, const PairDev *__restrict__ pairs,
                                      int n_pairs, const uint64_t *__restrict__ contig_off, uint32_t n_contigs,
                                      int *__restrict__ err)
{
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
        const ah_site s = sites[i];
        bool ok = s.pair < n_pairs && s.primer <= 1 && s.strand <= 1 && s.contig < n_contigs;
        if (ok) {
            const uint64_t len = contig_off[s.contig + 1] - contig_off[s.contig];
            ok = (uint64_t)s.pos + (uint64_t)pairs[s.pair].L[s.primer] <= len;
        }
        if (!ok)
            atomicExch(err, kDevBounds);
    }
}

} // namespace

void launch_validate_sites(const ah_site *sites, uint64_t n, const PairDev *pairs_d, int n_pairs,
                           const uint64_t *contig_off, uint32_t n_contigs, int *err, cudaStream_t s)
{
    if (!n)
        return;
    uint64_t blocks = (n + 255) / 256;
    if (blocks > 8192)
        blocks = 8192;
    validate_sites_kernel<<<(unsigned)blocks, 256, 0, s>>>(sites, n, pairs_d, n_pairs, contig_off, n_contigs, err);
    AH_CUDA(cudaGetLastError());
}

size_t sort_keys_temp_bytes(uint64_t n, int end_bit)
{
    size_t bytes = 0;
    AH_CUDA(cub::DeviceRadixSort::SortKeys(nullptr, bytes, (const uint64_t *)nullptr, (uint64_t *)nullptr,
                                           (int64_t)n, 8, end_bit));
    return bytes;
}

void sort_keys(void *temp, size_t temp_bytes, const uint64_t *in, uint64_t *out, uint64_t n, int begin_bit,
               int end_bit, cudaStream_t s)
{
    AH_CUDA(cub::DeviceRadixSort::SortKeys(temp, temp_bytes, in, out, (int64_t)n, begin_bit, end_bit, s));
}

void launch_decode_keys(const uint64_t *keys, uint64_t n, int pbits, const uint64_t *contig_off, uint32_t n_contigs,
                        const uint32_t *contig_genome, ah_site *out, cudaStream_t s)
{
    if (!n)
        return;
    uint64_t blocks = (n + 255) / 256;
    if (blocks > 8192)
        blocks = 8192;
    decode_keys_kernel<<<(unsigned)blocks, 256, 0, s>>>(keys, n, pbits, contig_off, n_contigs, contig_genome, out);
    AH_CUDA(cudaGetLastError());
}

} // namespace ah

// ---------------------------------------------------------------------------
// Small-count path: rank sort.  Site keys are distinct in their bits
// [8, end_bit) -- (pair, flat position, primer, strand) names one site -- so
// a key's place in canonical order is the number of keys below it.  Every block
// sorts all keys into kRankBuckets ranges of equal width in shared memory (count,
// scan, scatter; up to 1,024 keys stay one range; a range that holds too many is divided
// into equal parts first), then ranks its own share of them, a warp per key against the
// keys of its range or part, decodes them and writes each record at its rank: no block
// waits for another, one launch.
// Bound: latency (the count and the scatter are one shared-memory atomic per key
// and thread).  Measured on a GB300, against the former n^2 compares of all keys
// over the GPU: 6,000 sites 14 -> 7 us; 10,000 sites of 33 sort bits 25 -> 12; 14 sites 3.2 -> 3.4;
// 16,000 sites within 0.4 Mbp of a 400 Mbp set, all in one range, 44 -> 18 (undivided 71).
// ---------------------------------------------------------------------------
namespace ah {
namespace {

constexpr int kRankThreads = 512;
constexpr int kRankKeys = 16;    // keys of a thread held in registers; more are read twice
constexpr int kRankBuckets = 1024;
// A range of more keys is divided again (2,000 keys in one range: 10.0 us undivided, 11.6
// divided; 6,000: 19 and 12); at most seven of the 16,384 keys' ranges are.
constexpr uint32_t kRankCrowd = 2048;
static_assert(kSmallSort / (kRankCrowd + 1) < 8, "a divided range has at least 128 parts");
constexpr uint32_t kRankStageContigs = 4096; // contig offset tables up to this size are staged in shared memory

// Shared memory: the keys by range, then the contig offsets when stage_contigs.
__global__ void __launch_bounds__(kRankThreads, 2)
    rank_sort_decode_kernel(const uint64_t *keys, uint64_t n_arg, const uint64_t *n_dev, int shift, int pbits,
                            const uint64_t *__restrict__ contig_off, uint32_t n_contigs, bool stage_contigs,
                            const uint32_t *__restrict__ contig_genome, ah_site *out, uint64_t *n_out, uint64_t *redo)
{
    extern __shared__ __align__(16) uint64_t rank_smem[];
    __shared__ uint32_t end[kRankBuckets]; // keys of a range; then where it ends in cand
    __shared__ uint32_t wsum[kRankThreads / 32];
    // divided ranges: their numbers (kNone: not divided), the keys of their parts, then where these end in cand
    constexpr uint32_t kNone = 0xffu;
    __shared__ uint8_t number[kRankBuckets];
    __shared__ uint32_t part_end[kRankBuckets];
    __shared__ uint32_t n_divided, part0[8]; // part0: a divided range's start in cand, less that of its parts
    __shared__ uint64_t query[kRankThreads];
    __shared__ uint32_t rank[kRankThreads];
    uint64_t *cand = rank_smem, *coff = rank_smem + n_arg;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    chain_start();
    if (stage_contigs) // (no kernel of the chain writes them)
        for (uint32_t i = tid; i <= n_contigs; i += kRankThreads)
            coff[i] = __ldg(contig_off + i);
    for (int i = tid; i < kRankBuckets; i += kRankThreads)
        end[i] = 0;
    chain_wait();
    const uint64_t n64 = n_dev ? *(const volatile uint64_t *)n_dev : n_arg;
    if (n64 > n_arg) { // device count above the launch's size: the host redoes this step
        if (blockIdx.x == 0 && tid == 0) {
            *n_out = 0;
            atomicOr((unsigned long long *)redo, (unsigned long long)kRedoSites);
        }
        return;
    }
    const uint32_t n = (uint32_t)n64;
    if (n_out && blockIdx.x == 0 && tid == 0)
        *n_out = n;
    const uint32_t share = (n + gridDim.x - 1) / gridDim.x, q0 = blockIdx.x * share;
    if (q0 >= n)
        return;
    const uint32_t q1 = min(n, q0 + share);
    if ((uint32_t)tid < q1 - q0) // the block's first queries
        query[tid] = keys[q0 + tid];
    const bool flat = n <= kRankBuckets; // few keys: one range
    bool crowded = false;                // some range is divided
    int part_bits = 0, part_shift = 0;   // parts of a divided range: 2^part_bits
    auto part_of = [&](uint64_t key, uint32_t num) {
        return num << part_bits | ((uint32_t)(key >> part_shift) & ((1u << part_bits) - 1u));
    };
    if (flat) {
        for (uint32_t i = tid; i < n; i += kRankThreads)
            cand[i] = keys[i];
    } else {
        // count
        uint64_t k[kRankKeys];
#pragma unroll
        for (int u = 0; u < kRankKeys; ++u) {
            const uint32_t i = tid + u * kRankThreads;
            k[u] = i < n ? keys[i] : 0;
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < kRankKeys; ++u)
            if (tid + u * kRankThreads < n)
                atomicAdd(&end[k[u] >> shift], 1u);
        for (uint32_t i = tid + kRankKeys * kRankThreads; i < n; i += kRankThreads)
            atomicAdd(&end[keys[i] >> shift], 1u);
        __syncthreads();
        // exclusive scan: each thread its kRankBuckets / kRankThreads = 2 ranges
        static_assert(kRankBuckets == 2 * kRankThreads, "two ranges per thread");
        const uint32_t c0 = end[2 * tid], c1 = end[2 * tid + 1];
        auto before_pair = [&](uint32_t sum) { // the threads' sums before this one's; whether a range is crowded
            uint32_t incl = sum;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, incl, d);
                if (lane >= d)
                    incl += y;
            }
            if (lane == 31)
                wsum[warp] = incl;
            crowded = __syncthreads_or(max(c0, c1) > kRankCrowd);
            uint32_t before = incl - sum;
            for (int w = 0; w < warp; ++w)
                before += wsum[w];
            return before;
        };
        const uint32_t before = before_pair(c0 + c1);
        end[2 * tid] = before;
        end[2 * tid + 1] = before + c0;
        if (!crowded) {
            __syncthreads();
            // scatter: `end` moves from a range's start to its end
#pragma unroll
            for (int u = 0; u < kRankKeys; ++u)
                if (tid + u * kRankThreads < n)
                    cand[atomicAdd(&end[k[u] >> shift], 1u)] = k[u];
            for (uint32_t i = tid + kRankKeys * kRankThreads; i < n; i += kRankThreads) {
                const uint64_t key = keys[i];
                cand[atomicAdd(&end[key >> shift], 1u)] = key;
            }
        } else {
            // The crowded ranges share kRankBuckets parts.  (They hold more than 2^11 keys, which
            // differ above bit 8, so a range spans more than 2^19 and a part is wider than a key.)
            if (tid == 0)
                n_divided = 0;
            part_end[2 * tid] = part_end[2 * tid + 1] = 0;
            __syncthreads();
            auto divide = [&](uint32_t r, uint32_t start, uint32_t c) {
                uint32_t num = kNone;
                if (c > kRankCrowd) {
                    num = atomicAdd(&n_divided, 1u);
                    part0[num] = start;
                    end[r] = start + c; // (its keys go by parts)
                }
                number[r] = (uint8_t)num;
            };
            divide(2 * tid, before, c0);
            divide(2 * tid + 1, before + c0, c1);
            __syncthreads();
            part_bits = 10 - (32 - __clz(n_divided - 1)); // (one range: __clz(0) = 32)
            part_shift = shift - part_bits;
            auto count_part = [&](uint64_t key) {
                const uint32_t num = number[key >> shift];
                if (num != kNone)
                    atomicAdd(&part_end[part_of(key, num)], 1u);
            };
#pragma unroll
            for (int u = 0; u < kRankKeys; ++u)
                if (tid + u * kRankThreads < n)
                    count_part(k[u]);
            for (uint32_t i = tid + kRankKeys * kRankThreads; i < n; i += kRankThreads)
                count_part(keys[i]);
            __syncthreads();
            const uint32_t p0 = part_end[2 * tid], p1 = part_end[2 * tid + 1], at = before_pair(p0 + p1);
            const uint32_t num = (2u * tid) >> part_bits; // (of both: a divided range has an even number of parts)
            if ((2u * tid) == num << part_bits && num < n_divided)
                part0[num] -= at;
            __syncthreads();
            if (num < n_divided) {
                part_end[2 * tid] = part0[num] + at;
                part_end[2 * tid + 1] = part0[num] + at + p0;
            }
            __syncthreads();
            auto place = [&](uint64_t key) {
                const uint32_t r = (uint32_t)(key >> shift), num = number[r];
                cand[atomicAdd(num == kNone ? &end[r] : &part_end[part_of(key, num)], 1u)] = key;
            };
#pragma unroll
            for (int u = 0; u < kRankKeys; ++u)
                if (tid + u * kRankThreads < n)
                    place(k[u]);
            for (uint32_t i = tid + kRankKeys * kRankThreads; i < n; i += kRankThreads)
                place(keys[i]);
        }
    }
    __syncthreads();
    // the block's keys, kRankThreads at a time
    for (uint32_t qb = q0; qb < q1; qb += kRankThreads) {
        const uint32_t m = min(q1 - qb, (uint32_t)kRankThreads);
        if (qb > q0) { // (the first ones are there)
            __syncthreads();
            if ((uint32_t)tid < m)
                query[tid] = keys[qb + tid];
            __syncthreads();
        }
        for (uint32_t j = warp; j < m; j += kRankThreads / 32) {
            const uint64_t key = query[j];
            const uint32_t b = (uint32_t)(key >> shift);
            uint32_t first = flat || !b ? 0u : end[b - 1], last = flat ? n : end[b];
            if (crowded && number[b] != kNone) {
                const uint32_t q = part_of(key, number[b]);
                if (q & ((1u << part_bits) - 1u))
                    first = part_end[q - 1];
                last = part_end[q];
            }
            uint32_t below = 0;
            for (uint32_t i = first + lane; i < last; i += 32)
                below += cand[i] < key ? 1u : 0u;
            below = __reduce_add_sync(0xffffffffu, below);
            if (lane == 0)
                rank[j] = first + below;
        }
        __syncthreads();
        if ((uint32_t)tid < m) {
            const uint64_t key = query[tid], pp = key >> 10;
            const uint64_t P = pp & ((1ull << pbits) - 1);
            const uint64_t *co = stage_contigs ? coff : contig_off;
            uint32_t lo = 0, hi = n_contigs;
            while (hi - lo > 1) {
                const uint32_t mid = (lo + hi) >> 1;
                if (co[mid] <= P)
                    lo = mid;
                else
                    hi = mid;
            }
            ah_site s;
            s.genome = __ldg(contig_genome + lo);
            s.contig = lo;
            s.pos = (uint32_t)(P - co[lo]);
            s.primer = (uint8_t)((key >> 9) & 1);
            s.strand = (uint8_t)((key >> 8) & 1);
            s.mm = (uint8_t)(key & 0xff);
            s.pair = (uint8_t)(pp >> pbits);
            out[rank[tid]] = s;
        }
    }
}

} // namespace

void launch_rank_sort_decode(const uint64_t *keys, uint64_t n, const uint64_t *n_dev, int end_bit, int pbits,
                             const uint64_t *contig_off, uint32_t n_contigs, const uint32_t *contig_genome,
                             ah_site *out, uint64_t *n_out, uint64_t *redo, cudaStream_t s)
{
    if (n == 0 || n > kSmallSort)
        throw Error(AH_ERR_ARG, "rank sort: count outside 1..16384");
    const bool stage = n_contigs + 1 <= kRankStageContigs;
    const size_t smem = (n + (stage ? n_contigs + 1 : 0)) * sizeof(uint64_t);
    static int attr_dev = -1, sms = 148; // opt in to the largest size once per device
    int dev = 0;
    AH_CUDA(cudaGetDevice(&dev));
    if (dev != attr_dev) {
        AH_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        AH_CUDA(cudaFuncSetAttribute(rank_sort_decode_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)((kSmallSort + kRankStageContigs) * sizeof(uint64_t))));
        attr_dev = dev;
    }
    // a block per SM, but at least a key per warp
    const unsigned blocks = (unsigned)std::min<uint64_t>((uint64_t)sms, (n + kRankThreads / 32 - 1) / (kRankThreads / 32));
    const int shift = end_bit > 10 + 8 ? end_bit - 10 : 8; // kRankBuckets ranges of the bits below end_bit
    launch_chained(rank_sort_decode_kernel, blocks, kRankThreads, smem, s, keys, n, n_dev, shift, pbits, contig_off,
                   n_contigs, stage, contig_genome, out, n_out, redo);
}

} // namespace ah
