// complex64 plane kernel
#include "plane_launch.cuh"
template void plane_launch<float2>(aim_ctx*, int, int, int, const int*, float2*, int, size_t);
template void plane_rhs<float2>(aim_ctx*, int, const SlabList&, float2*);
template bool plane_holds<float2>(const aim_ctx*);
template float2* plane_tables<float2>(aim_ctx*, int, const float2*);
