// Profile-HMM scoring by the warp wavefront (hmm.cu): the launch, its device
// scratch and the choice between it and the block-per-group kernel that
// launch_hmm_score (ah_internal.h) starts.
#pragma once

#include "ah_internal.h"

namespace ah {

// Whether the wavefront scores a call of n amplicons (their letters in all, the longest) against a
// profile; AH_HMM_KERNEL=rows or wave decides instead (a profiling aid) where both can.
bool hmm_use_wave(const HmmProfile &p, bool forward, uint64_t n, uint64_t letters, int max_len);

// Blocks the wavefront takes for n amplicons of at most max_len letters, and the
// device scratch of `blocks` of them in bytes: two stripe-boundary buffers of
// max_len + 1 float4s per warp (none for a profile of one stripe; at most
// 256 MB beyond one block per SM).
uint64_t hmm_wave_blocks(uint64_t n, int m, int max_len, int sms);
size_t hmm_scratch_bytes(uint64_t blocks, int m, int max_len);

// The scores of n amplicons, as launch_hmm_score computes them, by the warp
// wavefront in at most `blocks` blocks (any number from 1); bnd holds
// hmm_scratch_bytes(blocks, m, max_len) bytes.
void launch_hmm_wave(const ah_amplicon *amps, const uint32_t *order, uint64_t n, const uint32_t *planes,
                     const uint64_t *contig_off, uint32_t n_contigs, const HmmProfile &p, int max_len, bool forward,
                     void *bnd, uint64_t blocks, float *score_out, int *err, int sms, cudaStream_t s);

} // namespace ah
