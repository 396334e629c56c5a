// accept_launch.h -- host side of the two-launch LM head (calls that one_launch() in
// verify_accept.cu does not take): lm_head_pairs.cu and accept_rows.cu.
#pragma once
#include "accept_common.cuh"

namespace spade {
namespace accept {

// Vocabulary slices (CTAs) of the pair kernel on a device of `sms` SMs.
int pair_slices(int V, int sms);

// Statistics of every row and the logits of the rows of sampled sequences, on
// pairs of SMs.  c.NC is pair_slices(...).
spade_status launch_lm_head_pairs(const Call &c, const void *hidden, const void *w_lm, int H, cudaStream_t stream);

// The rows phase as a launch of its own, after launch_lm_head_pairs.
spade_status launch_accept_rows(const Call &c, int sms, cudaStream_t stream);

}  // namespace accept
}  // namespace spade
