// k_stream_f32.cu -- the f32 instances of the streaming detection pass
// (k_stream_impl.cuh); one translation unit per dtype so they compile in
// parallel.
#include "k_stream_impl.cuh"

namespace gp {

cudaError_t launch_stream_f32(const DetectArgs* args, const DetectArgs* batch, int nframes, bool fast,
                             const CUtensorMap* maps, cudaStream_t st)
{
    return launch_stream_dtype<true>(args, batch, nframes, fast, maps, st);
}

}  // namespace gp
