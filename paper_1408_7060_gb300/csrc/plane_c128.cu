// complex128 plane kernel
#include "plane_launch.cuh"
template void plane_launch<double2>(aim_ctx*, int, int, int, const int*, double2*, int, size_t);
template void plane_rhs<double2>(aim_ctx*, int, const SlabList&, double2*);
template bool plane_holds<double2>(const aim_ctx*);
template double2* plane_tables<double2>(aim_ctx*, int, const double2*);
