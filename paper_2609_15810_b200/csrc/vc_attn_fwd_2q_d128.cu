#include "vc_attn_fwd_2q.cuh"

namespace vc {

cudaError_t launch_2q_d128(const Problem& pr, const QuantLayout& ql, const WorkLayout& wl, const uint8_t* quant, void* o,
                          uint8_t* work, cudaStream_t s) {
  return run_2q<128>(pr, ql, wl, quant, o, work, s);
}

}  // namespace vc
