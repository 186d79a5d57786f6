// iqa_split_f16.cu -- batch sums of split tiles for __half pixel storage.
#include "iqa_split.cuh"

namespace iqa {

cudaError_t launch_split_sums_f16(const SplitArgs &p, int vec, int maps, cudaStream_t st)
{
    return launch_split_sums_t<__half>(p, vec, maps, st);
}

}  // namespace iqa

IQA_VIOLATION_READER(iqa_read_violations_split_f16)
