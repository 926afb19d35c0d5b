// The x passes of any_x.cuh on complex64 vectors (a file of its own: it compiles beside the others).
#include "any_x.cuh"

namespace vie {
template vie_status launch_x_any<float2>(bool, const PassPtrs<float2>&, int, int, int, int, int, const float2*, int,
                                      cudaStream_t, int, bool*);
}  // namespace vie
