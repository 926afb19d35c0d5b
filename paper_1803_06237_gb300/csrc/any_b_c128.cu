// Pass B of any_b.cuh on complex128 vectors (a file of its own: it compiles beside the others).
#include "any_b.cuh"

namespace vie {
template vie_status launch_b_any<double2>(const PassPtrs<double2>&, int, const PassBGeom&, int, const double2*, double,
                                      const double2*, cudaStream_t, bool*);
}  // namespace vie
