// FP64 instantiation of the strip spreading kernel (see strips.cuh).
#include "strips.cuh"
namespace fres {
template <>
void launch_spread_strips<double>(const NodeRec<double>* sorted, long long n, int cap, bool merge, double2* grid,
                              int nf1, int nf2, const KernelShape& ks, cudaStream_t st) {
    launch_strips_impl<double>(sorted, n, cap, merge, grid, nf1, nf2, ks, st);
}
}  // namespace fres
