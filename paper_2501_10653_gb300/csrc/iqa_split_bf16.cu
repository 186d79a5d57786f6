// iqa_split_bf16.cu -- batch sums of split tiles for __nv_bfloat16 pixel storage.
#include "iqa_split.cuh"

namespace iqa {

cudaError_t launch_split_sums_bf16(const SplitArgs &p, int vec, int maps, cudaStream_t st)
{
    return launch_split_sums_t<__nv_bfloat16>(p, vec, maps, st);
}

}  // namespace iqa

IQA_VIOLATION_READER(iqa_read_violations_split_bf16)
