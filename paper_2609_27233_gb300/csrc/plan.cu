// The span metadata kernel of prompt compaction, and of rollbacks whose map is a
// kernel of its own.
#include "plan_block.cuh"

namespace umim {
namespace {

__global__ void __launch_bounds__(kPlanThreads) span_plan_kernel(PlanArgs a, PlanArrays arr) {
  griddep_wait();
  const PlanSeq q = plan_sequence(a, arr, nullptr);
  if (q.last) plan_totals(a, arr);
}

}  // namespace

cudaError_t launch_span_plan(const PlanArgs &args, const PlanArrays &arr, cudaStream_t stream) {
  return launch_pdl(span_plan_kernel, dim3(args.B), dim3(kPlanThreads), 0, stream, args, arr);
}

}  // namespace umim
