// iqa_split_f32.cu -- batch sums of split tiles for float pixel storage.
#include "iqa_split.cuh"

namespace iqa {

cudaError_t launch_split_sums_f32(const SplitArgs &p, int vec, int maps, cudaStream_t st)
{
    return launch_split_sums_t<float>(p, vec, maps, st);
}

}  // namespace iqa

IQA_VIOLATION_READER(iqa_read_violations_split_f32)
