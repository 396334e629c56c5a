// accept_rows.cu -- second launch of the two-launch LM head: merge of the slice
// statistics, accept tests alpha(x) = min(1, p(x)/q(x)), KV commit and the draw
// of the correction / bonus token (Sec. III-C, Algorithm 1) from the logits
// that lm_head_pairs.cu stored.  Bound by latency: each sampled sequence reads
// one logits row and one q row (1.2 MB at 152064 entries), spread over a group of
// CTAs.  The launch is cooperative, as the CTAs of a group meet at barriers, and
// programmatic: its CTAs start while the last ones of the statistics finish.
#include "accept_launch.h"

namespace spade {
namespace accept {

__global__ void __launch_bounds__(kThreads, 1) accept_rows_kernel(const __grid_constant__ Call c) {
  extern __shared__ __align__(128) uint8_t smem_rows[];
  __shared__ SeqTable seqs;
  griddep_wait();
  griddep_launch_dependents();
  fill_table(c, seqs, threadIdx.x / 32, kWarps, threadIdx.x % 32, false);  // (reported by the first launch)
  block_sync();
  if (threadIdx.x < 32) fill_lists(c, seqs, blockIdx.x, gridDim.x, threadIdx.x);
  block_sync();
  rows_phase(c, *reinterpret_cast<RowsSmem *>(smem_rows), seqs, RowTables{}, blockIdx.x, gridDim.x);
}

spade_status launch_accept_rows(const Call &c, int sms, cudaStream_t stream) {
  static OncePerDevice once;
  const cudaError_t es = set_max_smem(once, static_cast<int>(kRowsBytesDouble), accept_rows_kernel);
  if (es != cudaSuccess) return cuda_fail(es, "cudaFuncSetAttribute(accept_rows)");
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(sms < kMaxNC ? sms : kMaxNC);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kRowsBytesDouble;  // two buffers for the draw's pieces
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeCooperative;
  attr[1].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, accept_rows_kernel, c);
  if (e != cudaSuccess) return cuda_fail(e, "accept_rows launch");
  return SPADE_OK;
}

}  // namespace accept
}  // namespace spade
