// Forward render kernels with float leaf storage (fp32 arithmetic).
#include "pot_render.cuh"

namespace pot {
cudaError_t launch_render_f32(const RenderParams &p, int K, bool cams, bool count, cudaStream_t s)
{
    return launch_render_t<float>(p, K, cams, count, s);
}
}  // namespace pot
