// Pass B of any_b.cuh on complex64 vectors (a file of its own: it compiles beside the others).
#include "any_b.cuh"

namespace vie {
template vie_status launch_b_any<float2>(const PassPtrs<float2>&, int, const PassBGeom&, int, const float2*, double,
                                      const float2*, cudaStream_t, bool*);
}  // namespace vie
