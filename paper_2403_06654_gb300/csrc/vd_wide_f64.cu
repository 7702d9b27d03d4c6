// The passes of vd_wide.cuh in double (a unit of its own: it compiles beside the other type's).
#include "vd_wide.cuh"

namespace vd {
template void wide_axis<double>(const AxisProg&, int, const GridDesc&, const void*, int, int, cudaStream_t);
template void wide_xpass<double>(const XProg&, const GridDesc&, const void*, int, int, cudaStream_t);
}  // namespace vd
