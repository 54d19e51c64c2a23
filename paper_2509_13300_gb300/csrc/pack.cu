// Packer: ASCII genome -> tile-strided one-hot bitplanes (layout in ah_internal.h).
//
// One CTA packs one tile at a time.  The tile's 32 KB of ASCII are 32 rows of
// kTileW bytes (row b = flat positions t*kTileBases + b*kTileW + [0, kTileW)),
// plus the next tile's first 32 bytes ("row 32") for the extension words; bulk
// async copies (TMA) bring them into shared memory, two tiles staged per CTA
// so the next copy overlaps the current packing.  Word j of plane x takes bit
// b from row b, column j, so thread i builds the four words of columns
// 4i .. 4i+3 alone, with no cross-lane traffic.  Per block of 4 rows it reads
// 4 row words (4 columns each) and transposes the 4x4 bytes with PRMT, giving
// one register per column (4 rows), and then:
//   - a letter's base is read from bits 1 and 2 of its byte (A 00, C 01,
//     T 10, G 11).  Bit 2 is copied up to bit 5, and one multiply by a
//     constant whose partial products never share a bit (so no carries)
//     moves bit 1 of the 4 bytes to bits 0..3 and bit 5 to bits 4..7 of the
//     product's high word; PRMT drops that byte into the column's even- or
//     odd-block word, and two masks per plane turn these into the column's
//     32-bit bit-1 and bit-2 words;
//   - a byte is a base only if it is exactly A/C/G/T in either case.  The
//     fast test: the byte must equal, up to case, the letter its low nibble
//     names (1 A, 3 C, 4 T, 7 G; an 8-entry PRMT table).  The low nibbles of
//     two rows interleave into a selector whose byte order is that of the
//     transpose's first stage, so one PRMT and one XOR per 4 bytes give 0 or
//     0x20 for every base byte; the thread ORs them over its 128 bytes.  Only
//     when some byte fails does the thread run the exact per-byte test for its
//     columns (a per-byte zero test and a gather by multiply).
// Plane words then follow from (h, l, valid) with one LOP3 each.  The work is
// split between the logic and the multiply pipes (shifts by constants are
// multiplies by run-time powers of two) so that the kernel is bound by HBM:
// 1 byte read and 0.516 bytes written per base.
//
// Input at any address, and contigs packed reversed (decoy sets): the tile's
// bytes are copied from the 16-byte boundary below their first, so the staged
// tile is shifted by 0..15 bytes (the same for every tile), and a row word is two
// staged words and a funnel shift; a reversed tile that lies in one contig is
// the contig's mirrored stretch staged as it is, read backwards with the bytes
// of each word reversed.  Tiles with a contig end inside (reversed) or at the
// end of the input are gathered word by word.  Measured on a GB300: a reversed set
// of 0.1 Gbp 233 us for a reversal pass and 41 for the packing -> 52 us; 4.6 Mbp at
// an odd address 11.5 -> 8 us (byte loads before).
#include <algorithm>
#include <cstdlib>

#include "ah_internal.h"

namespace ah {
namespace {

constexpr int kRowWords = kTileW / 4; // u32 words per ASCII row in shared memory
constexpr int kPackThreads = kTileW / 4;
constexpr int kRows = 33;                    // 32 rows + the next tile's head
constexpr int kBufWords = kRows * kRowWords; // one staged tile

// PRMT table: byte n is the (upper-case) letter whose low nibble is n, 0xFF
// where no letter has that nibble
constexpr uint32_t kLetterLo = 0x43FF41FFu, kLetterHi = 0x47FFFF54u;
// bit 8k+1 -> bit 32+k and bit 8k+5 -> bit 36+k of the 64-bit product: byte k
// moves by 31 - 7k; every partial product lands on its own bit
constexpr uint32_t kGatherLH = (1u << 31) | (1u << 24) | (1u << 17) | (1u << 10);

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void tma_load(void *dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_addr(dst)),
                 "l"(src), "r"(bytes), "r"(smem_addr(bar))
                 : "memory");
}

__device__ __forceinline__ bool mbar_try(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
                 : "=r"(ok)
                 : "r"(smem_addr(bar)), "r"(parity)
                 : "memory");
    return ok != 0;
}

__device__ __forceinline__ uint64_t global_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// bounded wait: false after ~2 s instead of hanging
__device__ bool mbar_wait(uint64_t *bar, uint32_t parity)
{
    if (mbar_try(bar, parity))
        return true;
    const uint64_t t0 = global_ns();
    while (!mbar_try(bar, parity))
        if (global_ns() - t0 > 2000000000ull)
            return false;
    return true;
}

// Exact validity of 4 bytes (one column, 4 rows): bit k set iff byte k is
// exactly one of A C G T in either case.
__device__ __forceinline__ uint32_t valid4(uint32_t raw, uint32_t sixteen, uint32_t top4)
{
    const uint32_t n = raw & 0x0F0F0F0Fu;
    const uint32_t x = n + __umulhi(n, top4);                       // nibbles n0 n1 | n2 n3 (n | n >> 4)
    const uint32_t sel = __byte_perm(x, 0, 0x4420);                 // 4 selector nibbles
    const uint32_t expect = __byte_perm(kLetterLo, kLetterHi, sel); // letter the nibble names
    const uint32_t z = (raw & 0xDFDFDFDFu) ^ expect;                // upper-cased letter vs expected
    const uint32_t s = (z & 0x7F7F7F7Fu) + 0x7F7F7F7Fu;             // byte MSB: low 7 bits non-zero
    const uint32_t valid = ~(s | z) & 0x80808080u;                  // byte MSB: z byte == 0
    return __umulhi(valid * 0x00204081u, sixteen);                  // byte k MSB -> bit k
}

// Classify 4 bytes (one column, 4 rows) and add their bits at the nibble
// given by pw (a run-time power of two) of the column's L (bit 1 of the
// letter), H (bit 2) and V (exactly one of A C G T, either case) words.
__device__ __forceinline__ void classify4(uint32_t raw, uint32_t pw, uint32_t sixteen, uint32_t top4, uint32_t &L,
                                          uint32_t &H, uint32_t &V)
{
    const uint32_t l4 = __umulhi((raw & 0x02020202u) * 0x08102040u, sixteen); // byte k bit 1 -> bit k
    const uint32_t h4 = __umulhi((raw & 0x04040404u) * 0x04081020u, sixteen); // byte k bit 2 -> bit k
    L = l4 * pw + L; // the nibbles are disjoint: add = or
    H = h4 * pw + H;
    V = valid4(raw, sixteen, top4) * pw + V;
}

// 4x4 byte transpose of rows r .. r+3 (row(q) = this thread's word of row q,
// 4 columns): col[k] = byte k of each row; t[] = the first stage, (a0 b0 a1
// b1), (a2 b2 a3 b3), (c0 d0 c1 d1), (c2 d2 c3 d3).
template <class Row>
__device__ __forceinline__ void load_block(const Row &rowf, int r, uint32_t (&row)[4], uint32_t (&t)[4],
                                           uint32_t (&col)[4])
{
#pragma unroll
    for (int q = 0; q < 4; ++q)
        row[q] = rowf(r + q);
    t[0] = __byte_perm(row[0], row[1], 0x5140);
    t[1] = __byte_perm(row[0], row[1], 0x7362);
    t[2] = __byte_perm(row[2], row[3], 0x5140);
    t[3] = __byte_perm(row[2], row[3], 0x7362);
    col[0] = __byte_perm(t[0], t[2], 0x5410);
    col[1] = __byte_perm(t[0], t[2], 0x7632);
    col[2] = __byte_perm(t[1], t[3], 0x5410);
    col[3] = __byte_perm(t[1], t[3], 0x7632);
}

// Build plane words for columns 4*ci .. 4*ci+3 from rows 0 .. 31 of the
// staged tile and store them as words 4*ci .. 4*ci+3 of the tile's planes.
// Threads of columns below kTileExt also store the extension words W + 4*ci
// .. W + 4*ci + 3: bit b of extension word W + j is the base at row b + 1,
// column j, i.e. the column's own word shifted right by one with bit 31 from
// row 32 (the next tile's first row, staged with the tile).
template <class Row>
__device__ __forceinline__ void pack_columns(const Row &rowf, int ci, uint32_t *__restrict__ dst, uint32_t one)
{
    const int j0 = 4 * ci;
    const uint32_t eight = one << 3, sixteen = one << 4, top4 = one << 28;
    // per column: byte m of ev / od = bits 1 (low nibble) and 2 (high nibble)
    // of rows 8m .. 8m+3 / 8m+4 .. 8m+7
    uint32_t ev[4] = {0, 0, 0, 0}, od[4] = {0, 0, 0, 0};
    uint32_t bad = 0; // OR of (byte ^ letter its nibble names): only 0x20 bits if all are bases
#pragma unroll
    for (int rb = 0; rb < 8; ++rb) {
        uint32_t row[4], t[4], col[4];
        load_block(rowf, 4 * rb, row, t, col);
        const uint32_t s01 = (row[0] & 0x0F0F0F0Fu) | ((row[1] * sixteen) & 0xF0F0F0F0u);
        const uint32_t s23 = (row[2] & 0x0F0F0F0Fu) | ((row[3] * sixteen) & 0xF0F0F0F0u);
        bad |= (t[0] ^ __byte_perm(kLetterLo, kLetterHi, s01)) | (t[1] ^ __byte_perm(kLetterLo, kLetterHi, s01 >> 16));
        bad |= (t[2] ^ __byte_perm(kLetterLo, kLetterHi, s23)) | (t[3] ^ __byte_perm(kLetterLo, kLetterHi, s23 >> 16));
        // byte 0 of the gathered word goes to byte rb / 2
        const uint32_t put = rb / 2 == 0 ? 0x3214u : rb / 2 == 1 ? 0x3240u : rb / 2 == 2 ? 0x3410u : 0x4210u;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t w = (col[k] & 0x02020202u) | ((col[k] * eight) & 0x20202020u);
            const uint32_t g = __umulhi(w, kGatherLH); // bits 0..3: bit 1 of rows 4rb.., bits 4..7: bit 2
            if (rb & 1)
                od[k] = __byte_perm(od[k], g, put);
            else
                ev[k] = __byte_perm(ev[k], g, put);
        }
    }
    uint32_t V[4] = {~0u, ~0u, ~0u, ~0u};
    if (bad & 0xDFDFDFDFu) { // some byte is not a base: exact per-byte test for these columns
#pragma unroll
        for (int k = 0; k < 4; ++k)
            V[k] = 0;
#pragma unroll
        for (int rb = 0; rb < 8; ++rb) {
            uint32_t row[4], t[4], col[4];
            load_block(rowf, 4 * rb, row, t, col);
            const uint32_t pw = one << (4 * rb);
#pragma unroll
            for (int k = 0; k < 4; ++k)
                V[k] = valid4(col[k], sixteen, top4) * pw + V[k];
        }
    }
    uint4 pa, pc, pg, pt;
    uint32_t *A = &pa.x, *C = &pc.x, *G = &pg.x, *T = &pt.x;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint32_t L = (ev[k] & 0x0F0F0F0Fu) | ((od[k] * sixteen) & 0xF0F0F0F0u);
        const uint32_t H = (__umulhi(ev[k], top4) & 0x0F0F0F0Fu) | (od[k] & 0xF0F0F0F0u);
        A[k] = V[k] & ~H & ~L;
        C[k] = V[k] & ~H & L;
        T[k] = V[k] & H & ~L;
        G[k] = V[k] & H & L;
    }
    *reinterpret_cast<uint4 *>(dst + 0 * kTileWX + j0) = pa;
    *reinterpret_cast<uint4 *>(dst + 1 * kTileWX + j0) = pc;
    *reinterpret_cast<uint4 *>(dst + 2 * kTileWX + j0) = pg;
    *reinterpret_cast<uint4 *>(dst + 3 * kTileWX + j0) = pt;
    if (j0 < kTileExt) {
        // row 32 of these four columns: bit k of hl / hh / hv = byte k's letter bits and validity
        uint32_t hl = 0, hh = 0, hv = 0;
        classify4(rowf(32), one, one << 4, one << 28, hl, hh, hv);
        const uint32_t ha = hv & ~hh & ~hl, hc = hv & ~hh & hl, ht = hv & hh & ~hl, hg = hv & hh & hl;
        uint4 ea, ec, eg, et;
        uint32_t *EA = &ea.x, *EC = &ec.x, *EG = &eg.x, *ET = &et.x;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            EA[k] = (A[k] >> 1) | ((ha >> k & 1u) << 31);
            EC[k] = (C[k] >> 1) | ((hc >> k & 1u) << 31);
            EG[k] = (G[k] >> 1) | ((hg >> k & 1u) << 31);
            ET[k] = (T[k] >> 1) | ((ht >> k & 1u) << 31);
        }
        *reinterpret_cast<uint4 *>(dst + 0 * kTileWX + kTileW + j0) = ea;
        *reinterpret_cast<uint4 *>(dst + 1 * kTileWX + kTileW + j0) = ec;
        *reinterpret_cast<uint4 *>(dst + 2 * kTileWX + kTileW + j0) = eg;
        *reinterpret_cast<uint4 *>(dst + 3 * kTileWX + kTileW + j0) = et;
    }
}

// Four bytes from any address, as aligned words.
__device__ __forceinline__ uint32_t load4(const uint8_t *a)
{
    const uintptr_t u = reinterpret_cast<uintptr_t>(a);
    const uint32_t *w = reinterpret_cast<const uint32_t *>(u & ~(uintptr_t)3);
    const uint32_t sh = (uint32_t)(u & 3u) * 8u;
    const uint32_t lo = __ldg(w), hi = sh ? __ldg(w + 1) : 0u;
    return __funnelshift_r(lo, hi, sh);
}

// What the input is to the packer: at a 16-byte boundary, at any address, or a
// set whose contigs are packed reversed (at any address; position P of contig
// [o, e) takes byte o + e - 1 - P).
enum PackInput { kAligned, kShifted, kReversed };

// A reversed tile of few contigs' parts, c_end the last of them, into the staging
// buffer: part by part, so that a thread's loads do not wait for the search of each
// word's contig, then the words that hold an end, byte by byte; zero past the end.
// Measured on a GB300, mirrored 100 Mbp of 409 contigs (361 of 3,052 tiles hold an end): 58 us
// with the search in every word -> 52.  (One contig 43, 1,500 contigs 61, 4,000 82; not
// mirrored 39.  Loading a tile's contig once instead of twice, or six blocks per SM instead
// of five, changed nothing.)
constexpr uint32_t kFewParts = 16;

__device__ __forceinline__ void gather_parts(const uint8_t *__restrict__ seq, uint64_t lim, uint64_t p0,
                                             const uint64_t *__restrict__ contig_off, uint32_t c0, uint32_t c_end,
                                             uint32_t *rows)
{
    constexpr uint32_t kNeed = (uint32_t)kTileBases + 32, kWords = kNeed / 4;
    const uint32_t end = lim <= p0 ? 0u : lim - p0 < kNeed ? (uint32_t)(lim - p0) : kNeed; // positions that exist
    auto rel = [&](uint64_t p) { return p <= p0 ? 0u : p - p0 < end ? (uint32_t)(p - p0) : end; };
    for (uint32_t c = c0; c <= c_end; ++c) {
        const uint64_t b = contig_off[c], e = contig_off[c + 1];
        const uint32_t w1 = rel(e) / 4;
        const uint8_t *src = seq + (b + e - 4 - p0); // word w: the four bytes at src - 4 w
#pragma unroll 8
        for (uint32_t w = (rel(b) + 3) / 4 + threadIdx.x; w < w1; w += kPackThreads)
            rows[kWords - 1 - w] = load4(src - 4 * (uint64_t)w);
        // the word that the part starts in (parts that end in it too write the same)
        if (threadIdx.x == c - c0 && (rel(b) & 3u)) {
            const uint32_t w = rel(b) / 4;
            uint32_t v = 0, cc = c0;
            for (uint32_t q = 4 * w; q < 4 * w + 4 && q < end; ++q) {
                while (contig_off[cc + 1] <= p0 + q)
                    ++cc;
                v |= (uint32_t)seq[contig_off[cc] + contig_off[cc + 1] - 1 - (p0 + q)] << (8 * (q & 3u));
            }
            rows[kWords - 1 - w] = __byte_perm(v, 0, 0x0123);
        }
    }
    if (threadIdx.x == 0 && (end & 3u)) { // the word with the end of all
        const uint32_t w = end / 4;
        uint32_t v = 0, cc = c0;
        for (uint32_t q = 4 * w; q < end; ++q) {
            while (contig_off[cc + 1] <= p0 + q)
                ++cc;
            v |= (uint32_t)seq[contig_off[cc] + contig_off[cc + 1] - 1 - (p0 + q)] << (8 * (q & 3u));
        }
        rows[kWords - 1 - w] = __byte_perm(v, 0, 0x0123);
    }
    for (uint32_t w = (end + 3) / 4 + threadIdx.x; w < kWords; w += kPackThreads)
        rows[kWords - 1 - w] = 0;
}

// A tile at the end of the input, or (reversed) with many contigs' ends, into the
// staging buffer: word by word, byte by byte where a word holds such an end;
// zero past the end.
template <int In>
__device__ __forceinline__ void gather_tile(const uint8_t *__restrict__ seq, uint64_t seq_base, uint64_t lim, uint64_t p0,
                                         const uint64_t *__restrict__ contig_off, uint32_t c, uint32_t *rows)
{
    constexpr uint32_t kWords = ((uint32_t)kTileBases + 32) / 4;
    for (uint32_t w = threadIdx.x; w < kWords; w += blockDim.x) {
        const uint64_t pos = p0 + 4ull * w;
        uint32_t v = 0;
        if (In == kReversed) {
            if (pos < lim) {
                while (contig_off[c + 1] <= pos)
                    ++c;
                if (pos + 4 <= contig_off[c + 1]) {
                    v = __byte_perm(load4(seq + (contig_off[c] + contig_off[c + 1] - 4 - pos)), 0, 0x0123);
                } else {
                    uint32_t cc = c;
                    for (int q = 0; q < 4 && pos + q < lim; ++q) {
                        while (contig_off[cc + 1] <= pos + q)
                            ++cc;
                        v |= (uint32_t)seq[contig_off[cc] + contig_off[cc + 1] - 1 - (pos + q)] << (8 * q);
                    }
                }
            }
            rows[kWords - 1 - w] = __byte_perm(v, 0, 0x0123); // where a mirrored tile has it
        } else {
            if (pos >= seq_base && pos + 4 <= lim) {
                v = load4(seq + (pos - seq_base));
            } else {
                for (int q = 0; q < 4; ++q)
                    if (pos + q >= seq_base && pos + q < lim)
                        v |= (uint32_t)seq[pos + q - seq_base] << (8 * q);
            }
            rows[w] = v;
        }
    }
}

// (five blocks per SM for shifted input: the second word and the shift do not fit in 40 registers)
template <int In>
__global__ void __launch_bounds__(kPackThreads, In == kAligned ? 6 : 5) pack_kernel(const uint8_t *__restrict__ seq, uint64_t seq_base,
                                                            uint64_t seq_len, uint64_t n_bases,
                                                            uint32_t *__restrict__ planes, uint64_t t0, uint64_t t1,
                                                            const uint64_t *__restrict__ contig_off,
                                                            const uint32_t *__restrict__ tile_contig, uint32_t one,
                                                            int *__restrict__ err)
{
    extern __shared__ __align__(128) uint32_t smem[]; // two staged tiles
    __shared__ __align__(8) uint64_t bar[2];
    constexpr uint32_t kNeed = (uint32_t)kTileBases + 32; // the tile and the next one's head
    const uint64_t lim = n_bases < seq_base + seq_len ? n_bases : seq_base + seq_len;
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&bar[0])) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&bar[1])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    // a tile goes through TMA when all of its bytes (and the next tile's head) are present
    // (reversed: and in one contig)
    auto full = [&](uint64_t t) {
        const uint64_t p0 = t * kTileBases;
        if (In == kReversed)
            return p0 + kNeed <= contig_off[tile_contig[t] + 1];
        return p0 >= seq_base && p0 + kNeed <= lim;
    };
    // the first source byte of a full tile
    auto source = [&](uint64_t t) {
        const uint64_t p0 = t * kTileBases;
        if (In == kReversed) {
            const uint32_t c = tile_contig[t];
            return seq + (contig_off[c] + contig_off[c + 1] - (p0 + kNeed));
        }
        return seq + (p0 - seq_base);
    };
    auto issue = [&](uint64_t t, int sb) {
        uint32_t *rows = smem + sb * kBufWords;
        const uint8_t *src = source(t);
        const uint32_t shift = In == kAligned ? 0u : (uint32_t)(reinterpret_cast<uintptr_t>(src) & 15u);
        const uint32_t bytes = (kNeed + shift + 15u) & ~15u; // (both ends stay in their 16-byte granules)
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(&bar[sb])), "r"(bytes)
                     : "memory");
        tma_load(rows, src - shift, bytes, &bar[sb]);
    };
    uint32_t phase0 = 0, phase1 = 0;
    const uint64_t first = t0 + blockIdx.x;
    if (threadIdx.x == 0 && first < t1 && full(first))
        issue(first, 0);
    int it = 0;
    for (uint64_t t = first; t < t1; t += gridDim.x, ++it) {
        const int sb = it & 1;
        uint32_t *rows = smem + sb * kBufWords;
        const uint64_t next = t + gridDim.x;
        // the other buffer was released by the barrier that ended the previous tile
        if (threadIdx.x == 0 && next < t1 && full(next))
            issue(next, sb ^ 1);
        const uint64_t p0 = t * kTileBases;
        uint32_t shift = 0; // of the staged tile, in bytes
        if (full(t)) {
            if (In != kAligned)
                shift = (uint32_t)(reinterpret_cast<uintptr_t>(source(t)) & 15u);
            const bool ok = mbar_wait(&bar[sb], sb ? phase1 : phase0);
            if (sb)
                phase1 ^= 1;
            else
                phase0 ^= 1;
            if (!__syncthreads_and(ok)) {
                if (threadIdx.x == 0) {
                    atomicExch(err, kDevTimeout);
                    if (next < t1 && full(next)) // bounded wait for the copy still in flight
                        mbar_wait(&bar[sb ^ 1], sb ? phase0 : phase1);
                }
                return;
            }
        } else {
            uint32_t c = 0, c_end = ~0u; // reversed: the first contig of the tile, the last that starts in it or its extension
            if (In == kReversed) {
                c = tile_contig[t];
                const uint64_t stop = p0 + kNeed < lim ? p0 + kNeed : lim;
                for (c_end = c; c_end - c <= kFewParts && contig_off[c_end + 1] < stop;)
                    ++c_end;
            }
            if (In == kReversed && c_end - c <= kFewParts)
                gather_parts(seq, lim, p0, contig_off, c, c_end, rows);
            else
                gather_tile<In>(seq, seq_base, lim, p0, contig_off, c, rows);
            __syncthreads();
        }
        const int ci = threadIdx.x;
        const uint32_t *staged = rows + shift / 4;
        const uint32_t sh = (shift & 3u) * 8u;
        if constexpr (In == kAligned)
            pack_columns([&](int r) { return rows[r * kRowWords + ci]; }, ci, planes + t * 4 * kTileWX, one);
        else
            pack_columns([&](int r) {
                const uint32_t *w = In == kReversed ? staged + (kNeed / 4 - 1 - r * kRowWords - ci)
                                                    : staged + (r * kRowWords + ci);
                const uint32_t v = __funnelshift_r(w[0], w[1], sh);
                return In == kReversed ? __byte_perm(v, 0, 0x0123) : v;
            }, ci, planes + t * 4 * kTileWX, one);
        __syncthreads(); // this buffer is refilled two tiles from now
    }
}

// ---------------------------------------------------------------------------
// Packer from 2-bit base codes (the load form whose host input is a quarter
// of ASCII's size): base p is bits 2 (p % 4) .. 2 (p % 4) + 1 of byte p / 4,
// A 0, C 1, G 2, T 3; positions listed in `gaps` (sorted, disjoint (start,
// length) pairs) and positions at or past n_bases are no base (all four
// planes 0).  One block per tile: the tile's 8 KB of codes and the next
// tile's first 8 bytes (the extension row) are loaded into shared memory with
// coalesced 16-byte loads; thread ci builds the plane words of columns
// 4 ci .. 4 ci + 3, for which row b holds exactly byte ci of the row: a 32 x 8
// bit matrix, transposed in registers by three rounds of masked exchanges.  The
// no-base runs of a tile (tile_gap, built at load by a merge walk) become masks
// per column: the rows of column j that a run [a, b) covers are consecutive.
// Bound: HBM (0.25 B read + 0.516 B written per base), then the latency of one
// tile (its loads, a barrier, the matrix).  Measured, 1.5 Gbp with 0.1 % of no-base
// bases on a GB300: 416 us with persistent blocks, a serial search of the tile's
// runs and a bitmap read back row by row -> 205 us (5.6 TB/s).  (Packing pieces of a
// host set while later pieces cross the link gains nothing: the copies stand
// still for as long as the packing runs.)
// ---------------------------------------------------------------------------
constexpr int kCodeRowBytes = kTileW / 4;                  // 256 bytes of codes per row
constexpr int kCodeWords = (32 * kCodeRowBytes + 16) / 4;  // the tile + the extension row (16 bytes read)
constexpr int kFewGaps = 16;                               // runs of a tile turned into masks by every thread

// The rows b of column j (bit b) whose position b * kTileW + j lies in [a, e).
__device__ __forceinline__ uint32_t rows_of(uint32_t a, uint32_t e, uint32_t j)
{
    const uint32_t r0 = a > j ? (a - j + kTileW - 1) / kTileW : 0u; // first row at or above a
    const uint32_t r1 = e > j ? (e - j + kTileW - 1) / kTileW : 0u; // first row at or above e
    const uint32_t lo = r0 >= 32 ? 0xffffffffu : (1u << r0) - 1u, hi = r1 >= 32 ? 0xffffffffu : (1u << r1) - 1u;
    return hi & ~lo;
}

__global__ void __launch_bounds__(kPackThreads, 8) pack2_kernel(const uint8_t *__restrict__ codes, uint64_t base0,
                                                                uint64_t n_avail, uint64_t n_bases,
                                                                const ulonglong2 *__restrict__ gaps,
                                                                const uint2 *__restrict__ tile_gap,
                                                                uint32_t *__restrict__ planes, uint64_t t0)
{
    __shared__ __align__(16) uint32_t cw[kCodeWords];
    __shared__ uint2 run[kFewGaps + 1];             // the tile's runs, relative to its start
    __shared__ __align__(16) uint32_t none[kTileW]; // many runs: per column, the rows that are no base
    __shared__ uint32_t none_head;                  // ... and of the extension row's 32 positions
    const int ci = threadIdx.x;
    const uint64_t avail_end = base0 + n_avail < n_bases ? base0 + n_avail : n_bases; // bases present here
    const uint64_t t = t0 + blockIdx.x;
    const uint64_t p0 = t * kTileBases;
    constexpr uint32_t kEnd = (uint32_t)kTileBases + 32; // the tile and its extension row
    const uint2 tg = __ldg(tile_gap + t);                // its runs: gaps[tg.x .. tg.y)
    // codes: bytes (p0 - base0) / 4 .. + 8208 of `codes`; zero past the available bytes
    const uint64_t cb0 = (p0 - base0) / 4;
    const uint64_t bytes_avail = (avail_end > p0 ? (avail_end - p0 + 3) / 4 : 0);
    if (bytes_avail >= (uint64_t)kCodeWords * 4) {
        const uint4 *src = reinterpret_cast<const uint4 *>(codes + cb0);
        for (int w = ci; w < kCodeWords / 4; w += kPackThreads)
            reinterpret_cast<uint4 *>(cw)[w] = __ldg(src + w);
    } else {
        for (int w = ci; w < kCodeWords; w += kPackThreads) {
            uint32_t v = 0;
            for (int q = 0; q < 4; ++q)
                if ((uint64_t)(4 * w + q) < bytes_avail)
                    v |= (uint32_t)codes[cb0 + 4 * w + q] << (8 * q);
            cw[w] = v;
        }
    }
    const uint32_t listed = tg.y - tg.x;
    const bool few = listed <= kFewGaps;
    const bool cut = avail_end < p0 + kEnd; // everything at or past avail_end is no base
    auto clipped = [&](uint32_t g) {        // run g of the tile, relative to p0
        const ulonglong2 x = __ldg(gaps + tg.x + g);
        auto rel = [&](uint64_t p) { return p <= p0 ? 0u : p - p0 < kEnd ? (uint32_t)(p - p0) : kEnd; };
        return make_uint2(rel(x.x), rel(x.x + x.y));
    };
    if (few) {
        if ((uint32_t)ci < listed)
            run[ci] = clipped(ci);
        if (cut && ci == 0)
            run[listed] = make_uint2((uint32_t)(avail_end > p0 ? avail_end - p0 : 0ull), kEnd);
    } else { // mark every position of every run, a run per warp
        for (int w = ci; w < kTileW; w += kPackThreads)
            none[w] = 0u;
        if (ci == 0)
            none_head = 0u;
        __syncthreads();
        for (uint32_t g = ci / 32; g < listed + (cut ? 1u : 0u); g += kPackThreads / 32) {
            const uint2 r = g < listed ? clipped(g) : make_uint2((uint32_t)(avail_end > p0 ? avail_end - p0 : 0ull), kEnd);
            for (uint32_t x = r.x + ci % 32; x < r.y; x += 32)
                if (x < kTileBases)
                    atomicOr(&none[x % kTileW], 1u << (x / kTileW));
                else
                    atomicOr(&none_head, 1u << (x - kTileBases));
        }
    }
    __syncthreads();
    const int j0 = 4 * ci;
    const uint8_t *cbytes = reinterpret_cast<const uint8_t *>(cw);
    // x[r], byte q = the codes of row r + 8 q (4 columns, 2 bits each) ...
    uint32_t x[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        const uint32_t b0 = cbytes[r * kCodeRowBytes + ci], b1 = cbytes[(r + 8) * kCodeRowBytes + ci],
                       b2 = cbytes[(r + 16) * kCodeRowBytes + ci], b3 = cbytes[(r + 24) * kCodeRowBytes + ci];
        x[r] = __byte_perm(__byte_perm(b0, b1, 0x0040), __byte_perm(b2, b3, 0x0040), 0x5410);
    }
    // ... transposed as an 8 x 8 bit matrix in every byte: x[k], bit 8 q + r = bit k of that row's codes
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const int sft = 1 << i;
        const uint32_t m = i == 0 ? 0x55555555u : i == 1 ? 0x33333333u : 0x0f0f0f0fu;
#pragma unroll
        for (int r = 0; r < 8; ++r)
            if (!(r & sft)) {
                const uint32_t u = x[r], v = x[r | sft];
                x[r] = (u & m) | ((v << sft) & ~m);
                x[r | sft] = ((u >> sft) & m) | (v & ~m);
            }
    }
    // the rows that are no base, per column (bit k of head: position k of this thread's part of the extension row)
    uint32_t bad[4] = {0, 0, 0, 0}, head = 0;
    if (few) {
        for (uint32_t g = 0; g < listed + (cut ? 1u : 0u); ++g) {
            const uint2 r = run[g];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                bad[k] |= rows_of(r.x, r.y, j0 + k);
                const uint32_t h = (uint32_t)kTileBases + j0 + k;
                head |= (h >= r.x && h < r.y ? 1u : 0u) << k;
            }
        }
    } else {
        const uint4 v = *reinterpret_cast<const uint4 *>(none + j0);
        bad[0] = v.x;
        bad[1] = v.y;
        bad[2] = v.z;
        bad[3] = v.w;
        head = j0 < kTileExt ? none_head >> j0 : 0u;
    }
    uint32_t *dst = planes + t * 4 * kTileWX;
    const uint32_t hb = j0 < kTileExt ? (uint32_t)cbytes[32 * kCodeRowBytes + ci] : 0u;
#pragma unroll
    for (int pl = 0; pl < 4; ++pl) { // A 00, C 01, G 10, T 11
        uint4 w;
        uint32_t *W = &w.x;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            W[k] = ~bad[k] & (pl & 1 ? x[2 * k] : ~x[2 * k]) & (pl & 2 ? x[2 * k + 1] : ~x[2 * k + 1]);
        *reinterpret_cast<uint4 *>(dst + pl * kTileWX + j0) = w;
        if (j0 < kTileExt) { // extension words: row b + 1 of the same column, bit 31 from the next tile's head
            uint4 ew;
            uint32_t *EW = &ew.x;
#pragma unroll
            for (int k = 0; k < 4; ++k)
                EW[k] = (W[k] >> 1) | ((((hb >> (2 * k)) & 3u) == (uint32_t)pl && !(head >> k & 1u) ? 1u : 0u) << 31);
            *reinterpret_cast<uint4 *>(dst + pl * kTileWX + kTileW + j0) = ew;
        }
    }
}

// Decode the planes back to one byte per position (0 = no base, 1..4 = A C G T,
// 5 = more than one plane set, which the packer never produces).  Test aid.
__global__ void unpack_kernel(const uint32_t *__restrict__ planes, uint8_t *__restrict__ codes, uint64_t n_bases)
{
    for (uint64_t p = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n_bases;
         p += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t t = p / kTileBases, r = p % kTileBases;
        const int b = (int)(r / kTileW), j = (int)(r % kTileW);
        const uint32_t *base = planes + t * 4 * kTileWX + j;
        int n = 0, code = 0;
        for (int x = 0; x < 4; ++x)
            if ((base[x * kTileWX] >> b) & 1u) {
                ++n;
                code = x + 1;
            }
        codes[p] = (uint8_t)(n > 1 ? 5 : code);
    }
}

} // namespace


namespace {
__global__ void copy_words_kernel(const uint32_t *__restrict__ src, uint32_t *__restrict__ dst, uint64_t n)
{
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x)
        dst[i] = src[i];
}
} // namespace

void launch_pack2(const uint8_t *codes, uint64_t base0, uint64_t n_avail, uint64_t n_bases, const uint64_t *gaps,
                  const uint2 *tile_gap, uint32_t *planes, uint64_t t0, uint64_t t1, cudaStream_t s)
{
    if (t1 <= t0)
        return;
    if (reinterpret_cast<uintptr_t>(codes) % 16 != 0 || base0 % kTileBases != 0)
        throw Error(AH_ERR_ARG, "2-bit codes must start 16-byte aligned at a tile boundary");
    // one block per tile (blocks end as tiles are done, as in launch_pack)
    pack2_kernel<<<(unsigned)(t1 - t0), kPackThreads, 0, s>>>(codes, base0, n_avail, n_bases,
                                                              reinterpret_cast<const ulonglong2 *>(gaps), tile_gap,
                                                              planes, t0);
    AH_CUDA(cudaGetLastError());
}

void launch_copy_words(const uint32_t *src, uint32_t *dst, uint64_t n_words, cudaStream_t s)
{
    if (!n_words)
        return;
    const uint64_t blocks = std::min<uint64_t>((n_words + 255) / 256, 1024);
    copy_words_kernel<<<(unsigned)blocks, 256, 0, s>>>(src, dst, n_words);
    AH_CUDA(cudaGetLastError());
}

namespace {
template <int In>
void launch_pack_as(const uint8_t *seq, uint64_t seq_base, uint64_t seq_len, uint64_t n_bases, uint32_t *planes,
                    uint64_t t0, uint64_t t1, const uint64_t *contig_off, const uint32_t *tile_contig, int *err,
                    cudaStream_t s)
{
    static_assert(kTileW % 128 == 0 && kTileExt == 32, "pack layout");
    static_assert(kBufWords * 4 >= kTileBases + 32 + 32, "a staged tile with its shift");
    const size_t smem = 2ull * kBufWords * sizeof(uint32_t); // two staged tiles (67.6 KB)
    // grid size and the shared-memory opt-in, once per device
    static int cached_dev = -1, sms = 148, per_sm = 1;
    int dev = 0;
    AH_CUDA(cudaGetDevice(&dev));
    if (dev != cached_dev) {
        AH_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        AH_CUDA(cudaFuncSetAttribute(pack_kernel<In>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        AH_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, pack_kernel<In>, kPackThreads, smem));
        // one block per tile: blocks end as tiles are done, so kernels that run
        // beside the packing (a run's later stages) get SMs as they free up;
        // AH_PACK_BLOCKS=n keeps n persistent blocks per SM instead (profiling aid)
        const char *e = getenv("AH_PACK_BLOCKS");
        per_sm = (e && atoi(e) > 0) ? std::max(1, std::min(per_sm, atoi(e))) : (1 << 20);
        cached_dev = dev;
    }
    uint64_t blocks = (uint64_t)sms * (uint64_t)(per_sm > 0 ? per_sm : 1);
    // AH_PACK_TILES=n: n tiles per block (the second staged while the first is packed)
    static int tiles_per_block = -1;
    if (tiles_per_block < 0) {
        const char *e = getenv("AH_PACK_TILES");
        tiles_per_block = (e && atoi(e) > 0) ? atoi(e) : 1;
    }
    blocks = std::min<uint64_t>(blocks, (t1 - t0 + tiles_per_block - 1) / tiles_per_block);
    // A block that packs one tile reserves the one staging buffer it uses: six
    // blocks per SM (measured on the large workload: the packing alone at 0.97
    // of the copy peak against 0.84 with two buffers reserved, and a pass 2.4 %
    // shorter; the collection step unchanged).  AH_PACK_SMEM_KB sets the
    // reservation (profiling aid; at least one buffer).
    size_t smem_launch = blocks >= t1 - t0 ? smem / 2 : smem;
    if (const char *e = getenv("AH_PACK_SMEM_KB"))
        smem_launch = std::min(smem, std::max(blocks >= t1 - t0 ? smem / 2 : smem, (size_t)atoi(e) * 1024));
    pack_kernel<In><<<(unsigned)blocks, kPackThreads, smem_launch, s>>>(seq, seq_base, seq_len, n_bases, planes, t0,
                                                                        t1, contig_off, tile_contig, 1u, err);
    AH_CUDA(cudaGetLastError());
}
} // namespace

void launch_pack(const uint8_t *seq, uint64_t seq_base, uint64_t seq_len, uint64_t n_bases, uint32_t *planes,
                 uint64_t t0, uint64_t t1, int *err, cudaStream_t s)
{
    if (t1 <= t0)
        return;
    // (tiles start 32 KB apart, so all of an input's tiles are shifted alike)
    if ((reinterpret_cast<uintptr_t>(seq) - seq_base) % 16 == 0)
        launch_pack_as<kAligned>(seq, seq_base, seq_len, n_bases, planes, t0, t1, nullptr, nullptr, err, s);
    else
        launch_pack_as<kShifted>(seq, seq_base, seq_len, n_bases, planes, t0, t1, nullptr, nullptr, err, s);
}

void launch_pack_reversed(const uint8_t *seq, uint64_t n_bases, uint32_t *planes, uint64_t n_tiles,
                          const uint64_t *contig_off, const uint32_t *tile_contig, int *err, cudaStream_t s)
{
    if (n_tiles)
        launch_pack_as<kReversed>(seq, 0, n_bases, n_bases, planes, 0, n_tiles, contig_off, tile_contig, err, s);
}

void launch_unpack_check(const uint32_t *planes, uint64_t n_tiles, uint8_t *codes, uint64_t n_bases, cudaStream_t s)
{
    (void)n_tiles;
    if (n_bases == 0)
        return;
    uint64_t blocks = (n_bases + 255) / 256;
    if (blocks > 4096)
        blocks = 4096;
    unpack_kernel<<<(unsigned)blocks, 256, 0, s>>>(planes, codes, n_bases);
    AH_CUDA(cudaGetLastError());
}

} // namespace ah
