// lb_k3_d3q19.cu -- compiled tiles of the step in moment form for D3Q19.
// Each entry: storage / arithmetic type, tile bx x by, TMA ring depth, CTAs
// per SM; and the brick cross-sections whose contexts can end a
// run: all that are compiled, so that no batch, autotuner or requested brick takes a
// context's runs away.
#include "lb_k3_launch.cuh"

namespace lbgb {

extern const K3Variant k3_variants_d3q19[] = {
    K3Impl<D3Q19, float, float, 32, 16, 3, 1>::variant(LB_D3Q19, LB_F32),
    K3Impl<D3Q19, float, float, 32, 4, 2, 2>::variant(LB_D3Q19, LB_F32),  // small domains
    K3Impl<D3Q19, double, double, 32, 8, 2, 1>::variant(LB_D3Q19, LB_F64),
    K3Impl<D3Q19, __half, float, 32, 16, 3, 1>::variant(LB_D3Q19, LB_F16S),
    K3Impl<D3Q19, __nv_bfloat16, float, 32, 16, 3, 1>::variant(LB_D3Q19, LB_BF16S),
};
extern const int k3_n_variants_d3q19 = sizeof(k3_variants_d3q19) / sizeof(k3_variants_d3q19[0]);

extern const LeaveVariant leave_variants_d3q19[] = {
    LeaveImpl<D3Q19, float, float, 64, 8, 3>::variant(LB_D3Q19, LB_F32),
    LeaveImpl<D3Q19, float, float, 32, 16, 3>::variant(LB_D3Q19, LB_F32),
    LeaveImpl<D3Q19, float, float, 32, 8, 2>::variant(LB_D3Q19, LB_F32),
    LeaveImpl<D3Q19, float, float, 64, 7, 3>::variant(LB_D3Q19, LB_F32),
    LeaveImpl<D3Q19, float, float, 64, 6, 3>::variant(LB_D3Q19, LB_F32),
    LeaveImpl<D3Q19, float, float, 32, 14, 3>::variant(LB_D3Q19, LB_F32),
    LeaveImpl<D3Q19, double, double, 32, 8, 2>::variant(LB_D3Q19, LB_F64),
};
extern const int leave_n_variants_d3q19 = sizeof(leave_variants_d3q19) / sizeof(leave_variants_d3q19[0]);

}  // namespace lbgb
