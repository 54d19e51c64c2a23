// Profile-HMM homology scores of amplicons (Sec. 2.1, Amplicon analysis,
// item 2: a profile HMM trained on amplicons whose primers match exactly
// scores every predicted amplicon).
//
// Profile (built on the host, build_profile): the most frequent training
// sequence is the reference (first occurrence on ties); every training
// sequence is aligned to it globally with unit costs (equal A/C/G/T letters
// cost 0, any other pair 1, a gap 1), the traceback preferring a diagonal
// step, then a step that consumes a letter of the sequence (an insertion
// after the current column), then a step that consumes a column (a
// deletion); the state path of each alignment (B = M_0, M_j, I_j, D_j, E)
// gives transition counts from every state to the next column's M (E after
// column m), to I_j and to the next column's D, and letter counts for each
// match column; probabilities are counts + 1 normalised over the allowed
// moves (and over A/C/G/T); insert states emit the background.  Scores are
// bits against the uniform background: log2(p / (1/4)) for match emissions
// (0 for an unknown letter), 0 for insert emissions, log2 p for moves.
//
// Scores: the glocal Viterbi log-odds score of each amplicon's sequence (as
// ah_fetch returns it) against the profile, fp32, or the glocal Forward score:
// the same recurrence with the maximum of the predecessors replaced by
// log2(2^a + 2^b) (the log-sum semiring).  Two kernels compute the recurrence.
//
// hmm_wave_kernel (the default; hmm_use_wave): a warp runs one stripe of 32 * K columns of one
// amplicon; lane l owns K consecutive columns with their nine move scores in
// registers and, at step s, computes row i = s - l (an anti-diagonal
// wavefront): M and I of its columns from its own previous row, the delete
// chain along its K columns.  The left neighbour's last column arrives by one
// shuffle per state (its row i from the previous step; its row i - 1 is kept
// from the step before); lane 0 takes it from the previous stripe, through a
// buffer in global memory that is read 32 rows at a time, two blocks ahead.  The
// stripes of a block's amplicons are one sequence of tasks dealt to its four
// warps in turn, each stripe about 100 rows behind the one before it, so one
// amplicon already fills four warps and a call's last amplicons leave no warp
// idle for a whole amplicon.  Forward scores are computed as odds (sums and
// products, no logarithms: the log-sum took an exp2 and a log2 per term, and
// its roundings of scores of ~1,000 bits were the larger error) with a common
// exponent per lane, brought up to date every fourth row and wherever what comes
// in from the left outweighs the lane by far.
// Bound: issue slots, with latency next (three warps per scheduler by registers):
// 143 instructions per step of 256 cells for Viterbi, 157 for Forward, issue 0.68
// and 0.66.  K = 8 needs half the steps of K = 4 per profile; packed two-wide
// fp32 instructions were measured no faster (they take two dispatch cycles, and
// the packing moves come on top).  Measured on a GB300: Viterbi, 4,000 amplicons x
// 1,461 columns 22.8 -> 6.3 ms (1.36 T cells/s); Forward, 5,000 x 460 11.3 -> 1.0 ms
// (1.05 T cells/s); one amplicon of 1,461 letters 1,577 -> 500 us (Viterbi).
//
// hmm_score_kernel (Viterbi scores of amplicons much shorter than the profile,
// both scores where a memory budget has no room for the wavefront's buffers, and
// AH_HMM_KERNEL=rows): a block scores a group of amplicons of
// similar length in lockstep, rows = sequence letters: each thread owns K
// consecutive profile columns with their 13 scores in registers; M and I of a
// row depend only on the previous row (the left neighbour's values come by
// shuffle, or through shared memory across warps); the delete chain
// D_j = max(E_j, D_{j-1} + t_DD) is a block-wide scan in the (max, +)
// semiring over (t_DD, E_j) pairs (for the Forward score, in (log-sum, +)).
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <type_traits>

#include "ah_internal.h"
#include "hmm.h"

namespace ah {
namespace {

int letter_code(char c)
{
    switch (c) {
    case 'A': case 'a': return 0;
    case 'C': case 'c': return 1;
    case 'G': case 'g': return 2;
    case 'T': case 't': return 3;
    default: return 4;
    }
}

enum { kM = 0, kI = 1, kD = 2 };

} // namespace

static HmmProfile::Odds odds_form(const HmmProfile &p);

void build_profile(const char *seqs, const uint64_t *off, uint64_t n, HmmProfile &p)
{
    // the reference: most frequent sequence, first occurrence on ties (by hashing)
    std::map<std::string, std::pair<uint64_t, uint64_t>> freq; // sequence -> (count, first index)
    for (uint64_t q = 0; q < n; ++q) {
        std::string s(seqs + off[q], seqs + off[q + 1]);
        auto it = freq.find(s);
        if (it == freq.end())
            freq.emplace(std::move(s), std::make_pair(1ull, q));
        else
            ++it->second.first;
    }
    uint64_t best_q = 0, best_n = 0;
    for (const auto &kv : freq)
        if (kv.second.first > best_n || (kv.second.first == best_n && kv.second.second < best_q)) {
            best_n = kv.second.first;
            best_q = kv.second.second;
        }
    const char *R = seqs + off[best_q];
    const int64_t m = (int64_t)(off[best_q + 1] - off[best_q]);
    p.m = (int)m;
    p.reference = best_q;
    std::vector<double> ct((size_t)(m + 1) * 9, 0.0), ce((size_t)(m + 1) * 4, 0.0);
    std::vector<int> rc(m);
    for (int64_t j = 0; j < m; ++j)
        rc[j] = letter_code(R[j]);
    std::vector<uint32_t> dist; // (len + 1) x (m + 1) alignment costs
    std::vector<uint8_t> moves;
    for (uint64_t q = 0; q < n; ++q) {
        const char *S = seqs + off[q];
        const int64_t ls = (int64_t)(off[q + 1] - off[q]);
        const int64_t W = m + 1;
        dist.assign((size_t)(ls + 1) * W, 0);
        for (int64_t j = 0; j <= m; ++j)
            dist[j] = (uint32_t)j;
        for (int64_t i = 1; i <= ls; ++i) {
            const int si = letter_code(S[i - 1]);
            uint32_t *row = &dist[i * W];
            const uint32_t *up = &dist[(i - 1) * W];
            row[0] = (uint32_t)i;
            for (int64_t j = 1; j <= m; ++j) {
                const uint32_t sub = up[j - 1] + ((si < 4 && si == rc[j - 1]) ? 0u : 1u);
                row[j] = std::min(sub, std::min(up[j], row[j - 1]) + 1u);
            }
        }
        moves.clear();
        int64_t i = ls, j = m;
        while (i > 0 || j > 0) {
            const uint32_t here = dist[i * W + j];
            if (i > 0 && j > 0) {
                const int si = letter_code(S[i - 1]);
                const uint32_t sub = dist[(i - 1) * W + j - 1] + ((si < 4 && si == rc[j - 1]) ? 0u : 1u);
                if (here == sub) {
                    moves.push_back(kM);
                    --i;
                    --j;
                    continue;
                }
            }
            if (i > 0 && here == dist[(i - 1) * W + j] + 1u) {
                moves.push_back(kI);
                --i;
            } else {
                moves.push_back(kD);
                --j;
            }
        }
        int from = kM; // B = M_0
        int64_t col = 0, pos = 0;
        for (auto it = moves.rbegin(); it != moves.rend(); ++it) {
            const int to = *it;
            ct[(size_t)col * 9 + from * 3 + to] += 1.0;
            if (to == kM) {
                ++col;
                const int l = letter_code(S[pos]);
                if (l < 4)
                    ce[(size_t)col * 4 + l] += 1.0;
                ++pos;
            } else if (to == kI) {
                ++pos;
            } else {
                ++col;
            }
            from = to;
        }
        ct[(size_t)col * 9 + from * 3 + kM] += 1.0; // to E
    }
    p.t.assign((size_t)(m + 1) * 9, -INFINITY);
    p.e.assign((size_t)(m + 1) * 4, 0.0f);
    for (int64_t j = 0; j <= m; ++j) {
        for (int x = 0; x < 3; ++x) {
            if (j == 0 && x == kD)
                continue; // D_0 does not exist
            const bool has_d = j < m;
            double tot = 0.0;
            for (int y = 0; y < 3; ++y)
                if (y != kD || has_d)
                    tot += ct[(size_t)j * 9 + x * 3 + y] + 1.0;
            for (int y = 0; y < 3; ++y)
                if (y != kD || has_d)
                    p.t[(size_t)j * 9 + x * 3 + y] = (float)std::log2((ct[(size_t)j * 9 + x * 3 + y] + 1.0) / tot);
        }
        if (j > 0) {
            const double tot = ce[j * 4] + ce[j * 4 + 1] + ce[j * 4 + 2] + ce[j * 4 + 3] + 4.0;
            for (int l = 0; l < 4; ++l)
                p.e[(size_t)j * 4 + l] = (float)std::log2((ce[(size_t)j * 4 + l] + 1.0) / tot * 4.0);
        }
    }
    p.odds = odds_form(p);
}

namespace {

constexpr int kHmmThreads = 512;
constexpr float kNeg = -INFINITY;

// The semiring's "sum" of two log2 scores: Viterbi takes the larger, Forward
// log2(2^a + 2^b) (exp2f and the __log2f intrinsic of CUDA's math library).
struct MaxSum {
    __device__ static __forceinline__ float add(float a, float b) { return fmaxf(a, b); }
};
struct LogSum {
    __device__ static __forceinline__ float add(float a, float b)
    {
        const float hi = fmaxf(a, b), lo = fminf(a, b);
        if (lo == kNeg) // also both -inf
            return hi;
        return hi + __log2f(1.0f + exp2f(lo - hi)); // 1 + 2^d in [1, 2]: absolute error ~2^-22
    }
};

// Letter codes of amplicon `am` (as fetched: RF reverse-complemented) into seq.
__device__ void decode_letters(const ah_amplicon &am, const uint32_t *__restrict__ planes,
                               const uint64_t *__restrict__ contig_off, uint8_t *seq, int len)
{
    const uint64_t base = contig_off[am.contig] + am.start;
    const bool rc = am.orient == 1;
    for (int q = threadIdx.x; q < len; q += blockDim.x) {
        const uint64_t P = base + (rc ? (uint64_t)(len - 1 - q) : (uint64_t)q);
        const uint64_t t = P / kTileBases, r = P % kTileBases;
        const int b = (int)(r / kTileW), j = (int)(r % kTileW);
        const uint32_t *w = planes + t * 4 * kTileWX + j;
        int code = 4;
#pragma unroll
        for (int x = 0; x < 4; ++x)
            if ((__ldg(w + x * kTileWX) >> b) & 1u)
                code = x;
        if (code < 4 && rc)
            code = 3 - code;
        seq[q] = (uint8_t)code;
    }
}

// A amplicons per block, in lockstep over rows (the host groups amplicons of
// similar length): the barriers of a row serve A rows of work.  The delete
// chain's (max, +) pairs share their t_DD part across the A amplicons.
template <class Op, int K, int A, int NT>
__global__ void __launch_bounds__(NT) hmm_score_kernel(const ah_amplicon *__restrict__ amps,
                                                                  const uint32_t *__restrict__ order, uint64_t n_amps,
                                                                  const uint32_t *__restrict__ planes,
                                                                  const uint64_t *__restrict__ contig_off,
                                                                  uint32_t n_contigs, const float *__restrict__ t,
                                                                  const float *__restrict__ e, int m, int max_len,
                                                                  float *__restrict__ score_out, int *__restrict__ err)
{
    extern __shared__ uint8_t seq[];                    // A x max_len letter codes
    __shared__ float edge_prev[A][3][NT / 32]; // M, I, D of each warp's last column, previous row
    __shared__ float edge_cur[A][2][NT / 32];  // M, I of each warp's last column, current row
    __shared__ float wtot_a[NT / 32], wtot_b[A][NT / 32];
    __shared__ float wpre_a[NT / 32], wpre_b[A][NT / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int c0 = threadIdx.x * K;
    // this thread's columns: scores of the moves into M_j (from j-1), into D_j
    // (from j-1) and into I_j (from j), and M_j's emissions
    float toM[K][3], toD[K][3], toI[K][3], em[K][4];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int j = c0 + k;
#pragma unroll
        for (int x = 0; x < 3; ++x) {
            toM[k][x] = (j >= 1 && j <= m) ? t[(j - 1) * 9 + x * 3 + 0] : kNeg;
            toD[k][x] = (j >= 1 && j <= m) ? t[(j - 1) * 9 + x * 3 + 2] : kNeg;
            toI[k][x] = (j <= m) ? t[j * 9 + x * 3 + 1] : kNeg;
        }
#pragma unroll
        for (int l = 0; l < 4; ++l)
            em[k][l] = (j >= 1 && j <= m) ? e[j * 4 + l] : 0.0f;
    }
    // the delete chain's t_DD prefix of this thread's columns (the same for every amplicon)
    float tdd_sum = 0.0f;
#pragma unroll
    for (int k = 0; k < K; ++k)
        tdd_sum += toD[k][kD];
    const uint64_t n_groups = (n_amps + A - 1) / A;
    for (uint64_t gi = blockIdx.x; gi < n_groups; gi += gridDim.x) {
        int len[A];
        uint32_t idx[A];
        int rows = 0;
        __syncthreads(); // the previous group's letters are no longer read
#pragma unroll
        for (int s = 0; s < A; ++s) {
            const uint64_t q = gi * A + s;
            len[s] = -1; // -1: no amplicon in this slot
            idx[s] = 0;
            if (q < n_amps) {
                idx[s] = order[q];
                const ah_amplicon am = amps[idx[s]];
                bool ok = am.contig < n_contigs && am.start <= am.end;
                if (ok)
                    ok = (uint64_t)am.end <= contig_off[am.contig + 1] - contig_off[am.contig] &&
                         am.end - am.start <= (uint32_t)max_len;
                if (ok) {
                    len[s] = (int)(am.end - am.start);
                    decode_letters(am, planes, contig_off, seq + s * max_len, len[s]);
                    rows = max(rows, len[s]);
                } else if (threadIdx.x == 0) { // checked on the host; reported, not read
                    atomicExch(err, kDevBounds);
                    score_out[idx[s]] = kNeg;
                }
            }
        }
        float pM[A][K], pI[A][K], pD[A][K];
#pragma unroll
        for (int s = 0; s < A; ++s)
#pragma unroll
            for (int k = 0; k < K; ++k) {
                pM[s][k] = (c0 + k == 0) ? 0.0f : kNeg;
                pI[s][k] = kNeg;
                pD[s][k] = kNeg;
            }
        // the delete chains of a row from its M and I values
        auto delete_chain = [&](const float (&cM)[A][K], const float (&cI)[A][K], float (&cD)[A][K]) {
            float lM[A], lI[A];
#pragma unroll
            for (int s = 0; s < A; ++s) {
                lM[s] = __shfl_up_sync(0xffffffffu, cM[s][K - 1], 1);
                lI[s] = __shfl_up_sync(0xffffffffu, cI[s][K - 1], 1);
                if (lane == 31) {
                    edge_cur[s][0][warp] = cM[s][K - 1];
                    edge_cur[s][1][warp] = cI[s][K - 1];
                }
            }
            __syncthreads();
            if (lane == 0)
#pragma unroll
                for (int s = 0; s < A; ++s) {
                    lM[s] = warp > 0 ? edge_cur[s][0][warp - 1] : kNeg;
                    lI[s] = warp > 0 ? edge_cur[s][1][warp - 1] : kNeg;
                }
            // per column: D_j = max(b_j, D_{j-1} + a_j); thread aggregate (a, b[s])
            float eb[A][K], agg_b[A];
#pragma unroll
            for (int s = 0; s < A; ++s) {
                float acc = kNeg;
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    const float pm = k ? cM[s][k - 1] : lM[s], pi = k ? cI[s][k - 1] : lI[s];
                    eb[s][k] = Op::add(pm + toD[k][kM], pi + toD[k][kI]);
                    acc = Op::add(eb[s][k], acc + toD[k][kD]);
                }
                agg_b[s] = acc;
            }
            // inclusive warp scan: (a1, b1) then (a2, b2) = (a1 + a2, max(b2, b1 + a2))
            float inc_a = tdd_sum, inc_b[A];
#pragma unroll
            for (int s = 0; s < A; ++s)
                inc_b[s] = agg_b[s];
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const float oa = __shfl_up_sync(0xffffffffu, inc_a, d);
#pragma unroll
                for (int s = 0; s < A; ++s) {
                    const float ob = __shfl_up_sync(0xffffffffu, inc_b[s], d);
                    if (lane >= d)
                        inc_b[s] = Op::add(inc_b[s], ob + inc_a);
                }
                if (lane >= d)
                    inc_a = oa + inc_a;
            }
            if (lane == 31) {
                wtot_a[warp] = inc_a;
#pragma unroll
                for (int s = 0; s < A; ++s)
                    wtot_b[s][warp] = inc_b[s];
            }
            __syncthreads();
            if (warp == 0) {
                float wa = lane < nwarps ? wtot_a[lane] : 0.0f, wb[A];
#pragma unroll
                for (int s = 0; s < A; ++s)
                    wb[s] = lane < nwarps ? wtot_b[s][lane] : kNeg;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const float oa = __shfl_up_sync(0xffffffffu, wa, d);
#pragma unroll
                    for (int s = 0; s < A; ++s) {
                        const float ob = __shfl_up_sync(0xffffffffu, wb[s], d);
                        if (lane >= d)
                            wb[s] = Op::add(wb[s], ob + wa);
                    }
                    if (lane >= d)
                        wa = oa + wa;
                }
                // exclusive prefix of the warps
                const float xa = __shfl_up_sync(0xffffffffu, wa, 1);
                if (lane < nwarps)
                    wpre_a[lane] = lane ? xa : 0.0f;
#pragma unroll
                for (int s = 0; s < A; ++s) {
                    const float xb = __shfl_up_sync(0xffffffffu, wb[s], 1);
                    if (lane < nwarps)
                        wpre_b[s][lane] = lane ? xb : kNeg;
                }
            }
            __syncthreads();
            // this thread's exclusive prefix = (warps before) then (lanes before)
            const float xa = __shfl_up_sync(0xffffffffu, inc_a, 1);
#pragma unroll
            for (int s = 0; s < A; ++s) {
                float xb = __shfl_up_sync(0xffffffffu, inc_b[s], 1);
                if (lane == 0)
                    xb = kNeg;
                const float lane_a = lane ? xa : 0.0f;
                float d = Op::add(xb, wpre_b[s][warp] + lane_a); // D at column c0 - 1
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    d = Op::add(eb[s][k], d + toD[k][kD]);
                    cD[s][k] = d;
                }
            }
        };
        auto finish = [&](int i) { // amplicons whose last row is i: the holder of column m scores them
#pragma unroll
            for (int s = 0; s < A; ++s)
                if (len[s] == i)
#pragma unroll
                    for (int k = 0; k < K; ++k)
                        if (c0 + k == m)
                            score_out[idx[s]] =
                                Op::add(Op::add(pM[s][k] + t[m * 9 + kM * 3], pI[s][k] + t[m * 9 + kI * 3]),
                                      pD[s][k] + t[m * 9 + kD * 3]);
        };
        __syncthreads(); // the letters are decoded
        delete_chain(pM, pI, pD);
        finish(0);
        for (int i = 1; i <= rows; ++i) {
            float lM[A], lI[A], lD[A];
#pragma unroll
            for (int s = 0; s < A; ++s) {
                lM[s] = __shfl_up_sync(0xffffffffu, pM[s][K - 1], 1);
                lI[s] = __shfl_up_sync(0xffffffffu, pI[s][K - 1], 1);
                lD[s] = __shfl_up_sync(0xffffffffu, pD[s][K - 1], 1);
                if (lane == 31) {
                    edge_prev[s][0][warp] = pM[s][K - 1];
                    edge_prev[s][1][warp] = pI[s][K - 1];
                    edge_prev[s][2][warp] = pD[s][K - 1];
                }
            }
            __syncthreads();
            if (lane == 0)
#pragma unroll
                for (int s = 0; s < A; ++s) {
                    lM[s] = warp > 0 ? edge_prev[s][0][warp - 1] : kNeg;
                    lI[s] = warp > 0 ? edge_prev[s][1][warp - 1] : kNeg;
                    lD[s] = warp > 0 ? edge_prev[s][2][warp - 1] : kNeg;
                }
            float cM[A][K], cI[A][K], cD[A][K];
#pragma unroll
            for (int s = 0; s < A; ++s) {
                const int x = i <= len[s] ? seq[s * max_len + i - 1] : 4;
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    const float qm = k ? pM[s][k - 1] : lM[s], qi = k ? pI[s][k - 1] : lI[s],
                                qd = k ? pD[s][k - 1] : lD[s];
                    // (a select, not an indexed load: the emission scores stay in registers)
                    const float ex = x == 0 ? em[k][0] : x == 1 ? em[k][1] : x == 2 ? em[k][2] : x == 3 ? em[k][3] : 0.0f;
                    cM[s][k] = ex + Op::add(Op::add(qm + toM[k][kM], qi + toM[k][kI]), qd + toM[k][kD]);
                    cI[s][k] = Op::add(Op::add(pM[s][k] + toI[k][kM], pI[s][k] + toI[k][kI]), pD[s][k] + toI[k][kD]);
                }
            }
            delete_chain(cM, cI, cD);
#pragma unroll
            for (int s = 0; s < A; ++s)
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    pM[s][k] = cM[s][k];
                    pI[s][k] = cI[s][k];
                    pD[s][k] = cD[s][k];
                }
            finish(i);
        }
    }
}

// NT: the most threads a block may have (the register budget per thread follows from it)
template <class Op, int K, int A, int NT>
bool launch_k(const ah_amplicon *amps, const uint32_t *order, uint64_t n, const uint32_t *planes,
              const uint64_t *contig_off, uint32_t n_contigs, const float *t, const float *e, int m, int max_len,
              float *out, int *err, int sms, cudaStream_t s)
{
    const int threads = 32 * (((m + 1) + 32 * K - 1) / (32 * K));
    if (threads > NT)
        return false; // the profile needs more columns than this variant holds
    const size_t smem = (size_t)A * (size_t)max_len;
    AH_CUDA(cudaFuncSetAttribute(hmm_score_kernel<Op, K, A, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)std::max<size_t>(smem, 1)));
    int per_sm = 1;
    AH_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, hmm_score_kernel<Op, K, A, NT>, threads, smem));
    const uint64_t groups = (n + A - 1) / A;
    const uint64_t blocks = std::min<uint64_t>(groups, (uint64_t)sms * (uint64_t)std::max(1, per_sm));
    hmm_score_kernel<Op, K, A, NT><<<(unsigned)blocks, threads, smem, s>>>(amps, order, n, planes, contig_off,
                                                                          n_contigs, t, e, m, max_len, out, err);
    AH_CUDA(cudaGetLastError());
    return true;
}

// ---------------------------------------------------------------------------
// The warp wavefront (see the head of this file).
// ---------------------------------------------------------------------------
constexpr int kWaveWarps = 4;       // warps per block: a pipeline over stripes
constexpr int kWaveRing = 64 + 8;   // float4s per warp: 64 boundary rows, and one lane's columns at the end
constexpr int kSeqPad = 64;         // letters of padding on either side of a warp's sequence in shared memory
constexpr uint64_t kWaveScratchMax = 256ull << 20;
constexpr uint64_t kWaveWaitNs = 2000000000ull; // bound of a wait on another warp's progress

// The wavefront's two semirings.  Viterbi: scores in bits, (max, +).  Forward:
// odds (2^score) with an exponent per lane, (+, x).  ext(a, t): a path
// extended by a move; acc(s, a, t): the sum of s and a extended by t; acc3: the
// sum of three extended paths.
struct WaveMax {
    static constexpr bool kScaled = false, kWatch = false;
    static constexpr int kTop = 0;
    static constexpr float kZero = -INFINITY, kOne = 0.0f;
    __device__ static __forceinline__ float ext(float a, float t) { return a + t; }
    __device__ static __forceinline__ float acc(float s, float a, float t) { return fmaxf(s, a + t); }
    __device__ static __forceinline__ float acc3(float a, float ta, float b, float tb, float c, float tc)
    {
        return fmaxf(fmaxf(a + ta, b + tb), c + tc); // one three-input maximum
    }
};
template <bool Watch> struct WaveSum {
    static constexpr bool kScaled = true, kWatch = Watch;
    static constexpr int kTop = Watch ? 80 : 0;
    static constexpr float kZero = 0.0f, kOne = 1.0f;
    __device__ static __forceinline__ float ext(float a, float t) { return a * t; }
    __device__ static __forceinline__ float acc(float s, float a, float t) { return fmaf(a, t, s); }
    __device__ static __forceinline__ float acc3(float a, float ta, float b, float tb, float c, float tc)
    {
        return fmaf(c, tc, fmaf(b, tb, a * ta)); // (the last term may be the one that arrives late)
    }
};

// Exponents of the scaled odds: a value is mantissa * 2^E with one E per lane.
// Every four rows a lane's largest mantissa is brought to 2^kTop, and the factor
// 2^(left lane's exponent - this one's) for what comes in from the left is renewed.
// Let a move into a deletion cost at most a bits, one into an insertion b, from a
// deletion to the next d, from an insertion to itself i, any move c.
//   fall: the smallest cell that counts is the deletion state of a lane's last column,
//     through which a row's mass must go where no letters are left for it.  It is at
//     least its lane's largest cell less a + 6 d; that one falls by b + 3 i at most in
//     the rows between two settlings (by insertions, if nothing better) and lies at most a
//     below what came in.  The other states of that column count down to c + 24 bits less.
//     kTop - (c + 2 a + 6 d + b + 3 i) >= -125 keeps all of it among the floats.
//   rise: a lane holds at least what deletions bring to it within a row.  A path that
//     reaches it within the next four rows crosses the same columns with at most four
//     matches, so it is at most a + 8 d bits above that: the columns of the matches and
//     those after them.  Four letters give 4^4, and at most 2^13.2 cells add up.
//     kTop + 22.2 + a + 8 d <= 127 keeps every mantissa finite.
//   far: by the same counts the left lane's exponent lies at most 15.2 + 2 a + 10 d above
//     this lane's (a row and a lane further), or a + 8 d + b + 3 i where a stripe's boundary
//     rows share that of three rows ago; up to 127 the factor is a float.
// Where all three hold (calm: kTop = 0), a look at what comes in is needed only while mass
// reaches the lanes for the first time, the first 32 steps of a stripe.  Else (watched) each
// step looks: a lane that is outweighed by more than 2^kRise, or whose left neighbour's
// exponent lies kHot above its own, takes the level of what comes in, so four rows end below
// 2^(kTop + kRise + 13), and kTop = 80 leaves fall 205 bits.  Beyond that the scores go by
// logarithms (hmm_score_kernel).  With every move down to 2^-c, calm holds up to c = 9.3
// (600 training sequences that each delete and insert everywhere), watched to 15.7; the 2,416
// of an operon family, which seldom delete, are calm.  On a GB300, calm against watched: 5,000
// amplicons x 460 columns 1,101 us and 1,270, 5,023 x 639 on that family's profile 2.02 ms and
// 3.05.  (With kTop = 30 and the left lane's exponent taken over where it lay 80 above,
// profiles lost mass or overflowed from c = 8 on.)
constexpr int kRise = 24, kHot = 100;
constexpr double kFallRoom = 125.0, kRiseRoom = 104.8, kFarRoom = 127.0; // at kTop = 0
constexpr int kNoMass = -(1 << 20); // exponent of a lane that holds only zeros
template <int Top> __device__ __forceinline__ int level_of(float x) { return (int)(__float_as_uint(x) >> 23) - 127 - Top; }
__device__ __forceinline__ float power_of_two(int e) // 2^e for e <= 127; 0 below the normal range
{
    return e < -126 ? 0.0f : __uint_as_float((uint32_t)(e + 127) << 23);
}

// Letter codes of amplicon `am` into seq[0 .. len), the warp's lanes in turn, and
// "unknown" on either side.
__device__ void decode_letters_warp(const ah_amplicon &am, const uint32_t *__restrict__ planes,
                                    const uint64_t *__restrict__ contig_off, uint8_t *seq, int len, int lane)
{
    const uint64_t base = contig_off[am.contig] + am.start;
    const bool rc = am.orient == 1;
    for (int q = lane - kSeqPad; q < len + kSeqPad; q += 32) {
        int code = 4;
        if (q >= 0 && q < len) {
            const uint64_t P = base + (rc ? (uint64_t)(len - 1 - q) : (uint64_t)q);
            const uint64_t tt = P / kTileBases, r = P % kTileBases;
            const int b = (int)(r / kTileW), j = (int)(r % kTileW);
            const uint32_t *w = planes + tt * 4 * kTileWX + j;
#pragma unroll
            for (int x = 0; x < 4; ++x)
                if ((__ldg(w + x * kTileWX) >> b) & 1u)
                    code = x;
            if (code < 4 && rc)
                code = 3 - code;
        }
        seq[q] = (uint8_t)code;
    }
}

// Waits (bounded) until *p >= need: another warp of the block has got that far.
__device__ __forceinline__ bool wait_for(volatile uint64_t *p, uint64_t need)
{
    if (*p >= need)
        return true;
    uint64_t t0, t1;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    while (*p < need) {
        __nanosleep(100);
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t1));
        if (t1 - t0 > kWaveWaitNs)
            return false;
    }
    return true;
}

// A block scores the amplicons order[blockIdx.x + i * gridDim.x].  Their stripes
// form one sequence of tasks (task = i * n_stripes + stripe), and warp w takes
// the tasks with task % kWaveWarps == w, so the stripes of an amplicon run
// behind one another and no warp waits for a whole amplicon.  A task hands its
// last column on through one of its warp's two buffers in bnd_all (max_len + 1
// float4s each: M, I, D and their exponent, per row): rows[w] = (task + 1) << 20
// | rows written, and used[w] = task + 1 once the next warp has read all of a
// task's rows (a buffer is reused two tasks later).
// t, e: the profile's moves and emissions in the semiring's values (bits, or
// odds).  Shared memory: the emissions of every column for letter codes 0..4;
// per warp the boundary ring, the last row's states and the letters.
template <class Op, int K>
__global__ void __launch_bounds__(32 * kWaveWarps, K <= 4 ? 4 : 3) hmm_wave_kernel(
    const ah_amplicon *__restrict__ amps, const uint32_t *__restrict__ order, uint64_t n_amps,
    const uint32_t *__restrict__ planes, const uint64_t *__restrict__ contig_off, uint32_t n_contigs,
    const float *__restrict__ t, const float *__restrict__ e, int m, int max_len, float4 *bnd_all,
    float *__restrict__ score_out, int *__restrict__ err)
{
    constexpr int span = 32 * K;
    constexpr int kVec = K / 4; // float4s of a lane's emissions
    static_assert(K % 4 == 0, "emissions are read as float4s");
    extern __shared__ __align__(16) float4 wave_smem[];
    __shared__ volatile uint64_t rows[kWaveWarps], used[kWaveWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n_stripes = (m + span) / span;
    const int letter_stride = n_stripes * kVec * 32; // float4s
    float4 *emi = wave_smem;                         // [letter][stripe][vector][lane]
    float4 *ring = wave_smem + 5 * letter_stride + warp * kWaveRing;
    float4 *at_end = ring + 64; // the states of the lane of column m at the last row
    const int seq_stride = ((max_len + 15) & ~15) + 2 * kSeqPad;
    uint8_t *seq = reinterpret_cast<uint8_t *>(wave_smem + 5 * letter_stride + kWaveWarps * kWaveRing) + warp * seq_stride + kSeqPad;
    for (int i = threadIdx.x; i < 5 * letter_stride; i += blockDim.x) {
        const int l = i % 32, c = (i / 32) % kVec, sl = i / (32 * kVec); // sl: letter * n_stripes + stripe
        const int letter = sl / n_stripes, j0 = (sl % n_stripes) * span + l * K + 4 * c;
        auto at = [&](int j) { return letter < 4 && j >= 1 && j <= m ? e[j * 4 + letter] : Op::kOne; };
        emi[i] = make_float4(at(j0), at(j0 + 1), at(j0 + 2), at(j0 + 3));
    }
    if (threadIdx.x < kWaveWarps)
        rows[threadIdx.x] = used[threadIdx.x] = 0;
    __syncthreads();
    const int before = (warp + kWaveWarps - 1) % kWaveWarps; // the warp of the previous stripe
    const uint64_t buffer = (uint64_t)(max_len + 1);
    auto buffer_of = [&](int w, uint64_t task) {
        return bnd_all + (((uint64_t)blockIdx.x * kWaveWarps + w) * 2 + (task / kWaveWarps & 1)) * buffer;
    };
    const uint64_t n_mine = (n_amps - blockIdx.x + gridDim.x - 1) / gridDim.x; // (gridDim.x <= n_amps)
    const uint64_t n_tasks = n_mine * n_stripes;
    bool failed = false; // a wait ran out: reported, and nothing more is waited for
    uint64_t have = ~0ull; // the amplicon whose letters are in seq
    int len = 0;
    uint32_t idx = 0;
    bool ok = false;
    for (uint64_t task = warp; task < n_tasks; task += kWaveWarps) {
        const uint64_t mine = task / n_stripes;
        const int s = (int)(task % n_stripes);
        const bool last_stripe = s + 1 == n_stripes;
        if (mine != have) {
            have = mine;
            idx = order[blockIdx.x + mine * gridDim.x];
            const ah_amplicon am = amps[idx];
            ok = am.contig < n_contigs && am.start <= am.end;
            if (ok)
                ok = (uint64_t)am.end <= contig_off[am.contig + 1] - contig_off[am.contig] &&
                     am.end - am.start <= (uint32_t)max_len;
            len = ok ? (int)(am.end - am.start) : 0;
            __syncwarp(); // the previous amplicon's letters are no longer read
            if (ok)
                decode_letters_warp(am, planes, contig_off, seq, len, lane);
            __syncwarp();
        }
        if (!ok) { // checked on the host; reported, not read
            if (lane == 0) {
                if (s == 0) {
                    atomicExch(err, kDevBounds);
                    score_out[idx] = kNeg;
                } else {
                    used[before] = task;
                }
            }
            continue;
        }
        float4 *out_rows = buffer_of(warp, task);
        const float4 *in_rows = buffer_of(before, task - 1); // (s > 0)
        // The task that used this buffer before, eight back, has been read.  (Where that was a last
        // stripe, which hands nothing on, the user before it is sixteen back: its reader, the
        // next warp, has read task - 12 since, for which task - 4 waited here: neither of these
        // is a last stripe unless this one is too, as then the stripes divide four.)
        if (!last_stripe && task >= 2 * kWaveWarps && (task - 2 * kWaveWarps) % n_stripes + 1 != n_stripes && !failed &&
            !wait_for(&used[warp], task - 2 * kWaveWarps + 1))
            failed = true;
        const int c0 = s * span + lane * K;
        // the moves into M_j and D_j (from j - 1) and into I_j (from j), by state left
        float toM[K][3], toI[K][3], toD[K][3];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int j = c0 + k;
#pragma unroll
            for (int x = 0; x < 3; ++x) {
                toM[k][x] = (j >= 1 && j <= m) ? t[(j - 1) * 9 + x * 3 + kM] : Op::kZero;
                toD[k][x] = (j >= 1 && j <= m) ? t[(j - 1) * 9 + x * 3 + kD] : Op::kZero;
                toI[k][x] = (j <= m) ? t[j * 9 + x * 3 + kI] : Op::kZero;
            }
        }
        // this lane's columns at its previous row, and column c0 - 1 there
        float pM[K], pI[K], pD[K];
#pragma unroll
        for (int k = 0; k < K; ++k)
            pM[k] = pI[k] = pD[k] = Op::kZero;
        float lM = Op::kZero, lI = Op::kZero, lD = Op::kZero;
        int E = kNoMass;
        if (Op::kScaled && c0 == 0) // row 0 begins there
            E = -Op::kTop;
        const int lane_m = (m - s * span) / K; // (last stripe) the lane of column m
        const int steps = len + 1 + (last_stripe ? lane_m : 31);
        // rows r0 + lane of the previous stripe's boundary, once they are written; each four rows
        // (one group of steps of lane 0) at one exponent
        auto boundary = [&](int r0) {
            const int r = r0 + lane;
            if (r0 <= len && !failed) {
                if (!wait_for(&rows[before], task << 20 | (uint64_t)min(r0 + 32, len + 1)))
                    failed = true;
                __threadfence_block();
            }
            failed = __any_sync(0xffffffffu, failed);
            float4 v = r <= len && !failed ? in_rows[r]
                                           : make_float4(Op::kZero, Op::kZero, Op::kZero, __int_as_float(kNoMass));
            if constexpr (Op::kScaled) {
                const int x = __float_as_int(v.w);
                int top = max(x, __shfl_xor_sync(0xffffffffu, x, 1));
                top = max(top, __shfl_xor_sync(0xffffffffu, top, 2));
                const float f = power_of_two(x - top);
                v = make_float4(v.x * f, v.y * f, v.z * f, __int_as_float(top));
            }
            if (r0 <= len && r0 + 32 > len) { // that was the last of them
                __syncwarp();
                if (lane == 0) {
                    __threadfence_block();
                    used[before] = task;
                }
            }
            return v;
        };
        // rows 0..31 in the ring, the next 32 in registers
        float4 ahead;
        if (s > 0) {
            __syncwarp();
            ring[lane] = boundary(0);
            ahead = boundary(32);
            __syncwarp();
        }
        const float4 *emi_s = emi + s * kVec * 32 + lane;
        // emissions of the current row's letter, and the next row's letter (rows below 1 and
        // above len: unknown)
        float4 em[kVec];
#pragma unroll
        for (int c = 0; c < kVec; ++c)
            em[c] = emi_s[4 * letter_stride + c * 32];
        int x_next = seq[-lane];
        // 2^(left lane's exponent - this lane's); with a look at what comes in, infinite where that is
        // no number to go by (nothing ever comes into columns above m)
        float from_left = 1.0f;
        auto link = [&](int left_e, auto look) {
            const int d = left_e - E;
            if (decltype(look)::value && d > kHot)
                from_left = c0 <= m ? INFINITY : 0.0f;
            else
                from_left = power_of_two(min(d, 127));
        };
        if constexpr (Op::kScaled) {
            const int rE = __shfl_up_sync(0xffffffffu, E, 1);
            link(lane > 0 ? rE : s > 0 ? __float_as_int(ring[0].w) : kNoMass, std::true_type());
        }
        auto scale_own = [&](float f) {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                pM[k] *= f;
                pI[k] *= f;
                pD[k] *= f;
            }
            lM *= f;
            lI *= f;
            lD *= f;
        };
        // One step.  kFirst: among the first 32, which bring mass to each lane for the first time;
        // they look at what comes in.  (Rows below 0: every state is zero, and so is what the
        // recurrence makes of them; rows above len: unused.)
        auto step = [&](int st, auto first) {
            constexpr bool kFirst = decltype(first)::value, kLook = Op::kScaled && (kFirst || Op::kWatch);
            // column c0 - 1 at this row: the left lane's latest row, or the previous stripe's boundary
            float rM, rI, rD;
            auto come = [&] {
                rM = __shfl_up_sync(0xffffffffu, pM[K - 1], 1);
                rI = __shfl_up_sync(0xffffffffu, pI[K - 1], 1);
                rD = __shfl_up_sync(0xffffffffu, pD[K - 1], 1);
                int rE = kNoMass;
                if (lane == 0) {
                    rM = rI = rD = Op::kZero;
                    if (s > 0) {
                        const float4 v = ring[st & 63];
                        rM = v.x;
                        rI = v.y;
                        rD = v.z;
                        rE = __float_as_int(v.w);
                    }
                }
                return rE; // lane 0's
            };
            come();
            // the next row's emissions and the letter after it, for the next step
            float4 em_next[kVec];
#pragma unroll
            for (int c = 0; c < kVec; ++c)
                em_next[c] = emi_s[x_next * letter_stride + c * 32];
            x_next = seq[st + 1 - lane];
            if constexpr (Op::kScaled) {
                rM *= from_left;
                rI *= from_left;
                rD *= from_left;
            }
            if constexpr (kLook) {
                // (an infinite factor leaves nothing that compares as less)
                const bool over = !(fmaxf(fmaxf(rM, rI), rD) <= power_of_two(Op::kTop + kRise));
                if (__any_sync(0xffffffffu, over)) {
                    const int e0 = come(), e1 = __shfl_up_sync(0xffffffffu, E, 1), rE = lane == 0 ? e0 : e1;
                    const float x = fmaxf(fmaxf(rM, rI), rD);
                    const int level = rE + level_of<Op::kTop>(x);
                    if (over && level > E && x > 0.0f) { // it outweighs the lane: the lane takes its level
                        scale_own(power_of_two(E - level));
                        E = level;
                    }
                    const int d = max(-252, min(rE - E, 254));
                    const float f1 = power_of_two(d / 2), f2 = power_of_two(d - d / 2);
                    rM = rM * f1 * f2;
                    rI = rI * f1 * f2;
                    rD = rD * f1 * f2;
                    const int e2 = __shfl_up_sync(0xffffffffu, E, 1);
                    link(lane == 0 ? e0 : e2, std::true_type());
                }
            }
            float cM[K], cI[K];
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const float4 v = em[k / 4];
                const float ex = k % 4 == 0 ? v.x : k % 4 == 1 ? v.y : k % 4 == 2 ? v.z : v.w;
                cM[k] = Op::ext(Op::acc3(k ? pM[k - 1] : lM, toM[k][kM], k ? pI[k - 1] : lI, toM[k][kI],
                                         k ? pD[k - 1] : lD, toM[k][kD]),
                                ex);
                cI[k] = Op::acc3(pM[k], toI[k][kM], pI[k], toI[k][kI], pD[k], toI[k][kD]);
            }
            if constexpr (kFirst)
                if (st == 0 && s == 0 && lane == 0) // B = M_0 at row 0
                    cM[0] = Op::kScaled ? power_of_two(Op::kTop) : Op::kOne;
            // the delete chain along the row
#pragma unroll
            for (int k = 0; k < K; ++k)
                pD[k] = Op::acc3(k ? cM[k - 1] : rM, toD[k][kM], k ? cI[k - 1] : rI, toD[k][kI], k ? pD[k - 1] : rD,
                                 toD[k][kD]);
#pragma unroll
            for (int k = 0; k < K; ++k) {
                pM[k] = cM[k];
                pI[k] = cI[k];
            }
            lM = rM;
            lI = rI;
            lD = rD;
#pragma unroll
            for (int c = 0; c < kVec; ++c)
                em[c] = em_next[c];
            if (!last_stripe) {
                if (lane == 31 && st >= 31 && st - 31 <= len)
                    out_rows[st - 31] = make_float4(pM[K - 1], pI[K - 1], pD[K - 1], __int_as_float(E));
            } else if (st + 1 == steps && lane == lane_m) { // row len: kept for the end state
#pragma unroll
                for (int k = 0; k < K; ++k)
                    at_end[k] = make_float4(pM[k], pI[k], pD[k], __int_as_float(E));
            }
        };
        // after every fourth step (its last: st); look: those that follow look at what comes in
        auto settle = [&](int st, auto look) {
            if ((st & 31) == 31) {
                if (!last_stripe && lane == 31) { // rows .. st - 31 are written
                    __threadfence_block();
                    rows[warp] = (task + 1) << 20 | (uint64_t)min(st - 30, len + 1);
                }
                if (s > 0) { // rows st + 1 .. st + 32 into the ring; the block after them
                    ring[(st + 1 + lane) & 63] = ahead;
                    ahead = boundary(st + 33);
                    __syncwarp();
                }
            }
            if constexpr (Op::kScaled) { // the lane's largest mantissa back to 2^kTop
                float big[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    big[0] = fmaxf(big[0], pM[k]);
                    big[1] = fmaxf(big[1], pI[k]);
                    big[2] = fmaxf(big[2], pD[k]);
                }
                const float b = fmaxf(fmaxf(big[0], big[1]), big[2]);
                const int up = b > 0.0f ? max(level_of<Op::kTop>(b), -126) : 0;
                scale_own(power_of_two(-up));
                E += up;
                // what comes in during the next four steps
                int rE = __shfl_up_sync(0xffffffffu, E, 1);
                if (lane == 0)
                    rE = s > 0 ? __float_as_int(ring[(st + 1) & 63].w) : kNoMass;
                link(rE, look);
            }
        };
        int st = 0;
        const std::bool_constant<Op::kWatch> watch;
#pragma unroll 1
        for (; st < 32 && st < steps; ++st) {
            step(st, std::true_type());
            if (st == 31)
                settle(st, watch);
            else if ((st & 3) == 3)
                settle(st, std::true_type());
        }
#pragma unroll 1
        for (; st < steps; st += 4) { // (up to three steps more than needed)
            step(st, std::false_type());
            step(st + 1, std::false_type());
            step(st + 2, std::false_type());
            step(st + 3, std::false_type());
            settle(st + 3, watch);
        }
        if (!last_stripe) {
            if (lane == 31) { // every row is written
                __threadfence_block();
                rows[warp] = (task + 1) << 20 | (uint64_t)(len + 1);
            }
        } else {
            __syncwarp();
            if (lane == 0) {
                const float4 v = at_end[(m - s * span) % K];
                const float endM = t[m * 9 + kM * 3], endI = t[m * 9 + kI * 3], endD = t[m * 9 + kD * 3];
                float sum = Op::acc(Op::acc(Op::ext(v.x, endM), v.y, endI), v.z, endD);
                if constexpr (Op::kScaled) {
                    int x = 0;
                    const float f = frexpf(sum, &x);
                    sum = sum > 0.0f ? (float)((double)log2f(f) + (double)(x + __float_as_int(v.w))) : kNeg;
                }
                score_out[idx] = sum;
            }
        }
        __syncwarp();
    }
    if (__any_sync(0xffffffffu, failed) && lane == 0)
        atomicExch(err, kDevTimeout);
}

// columns per lane: 4 holds up to 128 columns in one stripe; above that 8 halves the steps
bool wave_narrow(int m) { return m + 1 <= 128; }
int wave_stripes(int m) { return wave_narrow(m) ? 1 : (m + 256) / 256; }
constexpr int kWaveBlocksPerSm = 4; // most blocks per SM (the register budgets of the kernels)

template <class Op, int K>
void launch_wave(const ah_amplicon *amps, const uint32_t *order, uint64_t n, const uint32_t *planes,
                 const uint64_t *contig_off, uint32_t n_contigs, const float *t, const float *e, int m, int max_len,
                 float4 *bnd, uint64_t blocks, float *out, int *err, int sms, cudaStream_t s)
{
    const size_t smem = (size_t)5 * wave_stripes(m) * 32 * K * sizeof(float) +
                        (size_t)kWaveWarps * kWaveRing * sizeof(float4) +
                        (size_t)kWaveWarps * (size_t)(((max_len + 15) & ~15) + 2 * kSeqPad);
    AH_CUDA(cudaFuncSetAttribute(hmm_wave_kernel<Op, K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int per_sm = 1;
    AH_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, hmm_wave_kernel<Op, K>, 32 * kWaveWarps, smem));
    blocks = std::min<uint64_t>(blocks, (uint64_t)sms * (uint64_t)std::max(1, per_sm));
    hmm_wave_kernel<Op, K><<<(unsigned)blocks, 32 * kWaveWarps, smem, s>>>(amps, order, n, planes, contig_off,
                                                                           n_contigs, t, e, m, max_len, bnd, out, err);
    AH_CUDA(cudaGetLastError());
}

} // namespace

// The form of the odds that a profile's moves leave room for (see kTop).
static HmmProfile::Odds odds_form(const HmmProfile &p)
{
    double a = 0, b = 0, c = 0, d = 0, i = 0;
    for (int j = 0; j <= p.m; ++j)
        for (int x = 0; x < 3; ++x) {
            const float *t = &p.t[(size_t)j * 9 + x * 3];
            for (int y = 0; y < 3; ++y) {
                if (!std::isfinite(t[y])) // no such move
                    continue;
                double &most = y == kD ? a : y == kI ? b : c;
                most = std::max(most, -(double)t[y]);
                if (x == y && x != kM)
                    (x == kD ? d : i) = std::max(x == kD ? d : i, -(double)t[y]);
            }
        }
    c = std::max(c, std::max(a, b));
    const double fall = c + 2 * a + 6 * d + b + 3 * i, rise = a + 8 * d;
    const double far = std::max(15.2 + 2 * a + 10 * d, a + 8 * d + b + 3 * i);
    if (fall <= kFallRoom && rise <= kRiseRoom && far <= kFarRoom)
        return HmmProfile::kCalm;
    return fall <= kFallRoom + WaveSum<true>::kTop ? HmmProfile::kWatched : HmmProfile::kLogs;
}

// One block per amplicon up to a full GPU; a profile of one stripe runs an amplicon per warp.
uint64_t hmm_wave_blocks(uint64_t n, int m, int max_len, int sms)
{
    uint64_t b = std::min<uint64_t>(wave_stripes(m) == 1 ? (n + kWaveWarps - 1) / kWaveWarps : n,
                                    (uint64_t)sms * kWaveBlocksPerSm);
    const uint64_t per_block = hmm_scratch_bytes(1, m, max_len);
    if (per_block)
        b = std::min<uint64_t>(b, std::max<uint64_t>((uint64_t)sms, kWaveScratchMax / per_block));
    return std::max<uint64_t>(b, 1);
}

size_t hmm_scratch_bytes(uint64_t blocks, int m, int max_len)
{
    return wave_stripes(m) == 1 ? 0 : blocks * kWaveWarps * 2ull * (uint64_t)(max_len + 1) * sizeof(float4);
}

// Viterbi scores of amplicons much shorter than the profile go to the kernel that walks rows: a
// stripe of the wavefront takes 31 steps to fill and the stripes follow one another, while that
// kernel has all columns at work from the first row.  The line, in letters of the mean amplicon
// (of the longest where the call does not fill the GPU and its longest amplicon decides), is where
// the two met on a GB300 or a little above; wavefront against rows, us: one amplicon,
// 1,461 columns 20 letters 67, 34; 60 letters 102, 76; 150 letters 116, 188; 3,070 columns 100
// letters 214, 127; 300 letters 262, 345; 5,000 amplicons, 3,070 columns 20 letters 1,214, 807;
// 60 letters 1,954, 2,305.  (Forward scores stay with the wavefront: on odds they are more exact.)
bool hmm_use_wave(const HmmProfile &p, bool forward, uint64_t n, uint64_t letters, int max_len)
{
    if (forward && p.odds == HmmProfile::kLogs)
        return false;
    if (const char *kern = getenv("AH_HMM_KERNEL"))
        if (!strcmp(kern, "rows") || !strcmp(kern, "wave"))
            return kern[0] == 'w';
    if (forward || n == 0)
        return true;
    constexpr uint64_t kFull = 608; // amplicons that fill the GPU: four blocks for each of 152 SMs
    const uint64_t line = 20 * (uint64_t)wave_stripes(p.m) - 12;
    return n <= kFull ? (uint64_t)max_len > line : letters > n * std::min<uint64_t>(line, 75);
}

void launch_hmm_wave(const ah_amplicon *amps, const uint32_t *order, uint64_t n, const uint32_t *planes,
                     const uint64_t *contig_off, uint32_t n_contigs, const HmmProfile &p, int max_len, bool forward,
                     void *bnd, uint64_t blocks, float *score_out, int *err, int sms, cudaStream_t s)
{
    if (n == 0)
        return;
    if (p.m + 1 > kHmmMaxColumns)
        throw Error(AH_ERR_ARG, "ah_hmm_score: profile longer than " + std::to_string(kHmmMaxColumns) + " columns");
    blocks = std::min<uint64_t>(blocks, n);
    auto go = [&](auto *launch) {
        launch(amps, order, n, planes, contig_off, n_contigs, forward ? p.d_t_odds : p.d_t,
               forward ? p.d_e_odds : p.d_e, p.m, max_len, (float4 *)bnd, blocks, score_out, err, sms, s);
    };
    if (forward && p.odds == HmmProfile::kCalm)
        wave_narrow(p.m) ? go(launch_wave<WaveSum<false>, 4>) : go(launch_wave<WaveSum<false>, 8>);
    else if (forward)
        wave_narrow(p.m) ? go(launch_wave<WaveSum<true>, 4>) : go(launch_wave<WaveSum<true>, 8>);
    else
        wave_narrow(p.m) ? go(launch_wave<WaveMax, 4>) : go(launch_wave<WaveMax, 8>);
}

void launch_hmm_score(const ah_amplicon *amps, const uint32_t *order, uint64_t n, const uint32_t *planes,
                      const uint64_t *contig_off, uint32_t n_contigs, const float *t, const float *e, int m,
                      int max_len, bool forward, float *score_out, int *err, int sms, cudaStream_t s)
{
    if (n == 0)
        return;
    const int cols = m + 1;
    // AH_HMM_VARIANT="K,A" picks columns per thread and amplicons per block (profiling aid)
    int vk = 0, va = 0;
    if (const char *v = getenv("AH_HMM_VARIANT"))
        if (sscanf(v, "%d,%d", &vk, &va) != 2)
            vk = va = 0;
#define AH_HMM_TRY_OP(OP_, K_, A_, NT_)                                                                          \
    if ((vk == 0 || (vk == K_ && va == A_)) &&                                                                   \
        launch_k<OP_, K_, A_, NT_>(amps, order, n, planes, contig_off, n_contigs, t, e, m, max_len, score_out, err, \
                                   sms, s))                                                                      \
        return;
    if (forward) { // the default variants only
        vk = va = 0;
        AH_HMM_TRY_OP(LogSum, 4, 2, 512)
        AH_HMM_TRY_OP(LogSum, 6, 1, 512)
        throw Error(AH_ERR_ARG, "ah_hmm_forward: profile longer than " + std::to_string(kHmmMaxColumns) + " columns");
    }
#define AH_HMM_TRY(K_, A_, NT_) AH_HMM_TRY_OP(MaxSum, K_, A_, NT_)
    if (vk) { // the named variant (when it covers the profile)
        AH_HMM_TRY(2, 2, 512)
        AH_HMM_TRY(4, 1, 512)
        AH_HMM_TRY(4, 2, 512)
        AH_HMM_TRY(4, 4, 256)
        AH_HMM_TRY(8, 2, 256)
        AH_HMM_TRY(8, 1, 256)
        vk = va = 0;
    }
    // 4 columns x 2 amplicons (on 639 columns 398 GCUPS; 2 x 2 272; 4 x 1 315; 8 x 1 234,
    // register-capped); longer profiles take 6 columns x 1 amplicon
    AH_HMM_TRY(4, 2, 512)
    AH_HMM_TRY(6, 1, 512)
#undef AH_HMM_TRY
#undef AH_HMM_TRY_OP
    throw Error(AH_ERR_ARG, "ah_hmm_score: profile longer than " + std::to_string(kHmmMaxColumns) + " columns");
}

} // namespace ah

// The profile of a training set without a context or a GPU (development aid:
// lets the host-side builder be compared with an independent implementation on
// machines without a GPU).  Returns 0 and writes m and the reference index;
// when t and e are not NULL they receive (m + 1) * 9 and (m + 1) * 4 scores.
// Returns 1 for no training sequence, 2 when t or e is given and m exceeds
// m_cap.
extern "C" int ah_debug_hmm_profile(const char *seqs, const uint64_t *offsets, uint64_t n, uint64_t m_cap,
                                    uint64_t *m_out, uint64_t *reference_out, float *t, float *e)
{
    if (n == 0 || !offsets || !m_out || !reference_out)
        return 1;
    ah::HmmProfile p;
    ah::build_profile(seqs, offsets, n, p);
    *m_out = (uint64_t)p.m;
    *reference_out = p.reference;
    if (t || e) {
        if ((uint64_t)p.m > m_cap)
            return 2;
        if (t)
            memcpy(t, p.t.data(), p.t.size() * sizeof(float));
        if (e)
            memcpy(e, p.e.data(), p.e.size() * sizeof(float));
    }
    return 0;
}
