// lb_k3_d3q27.cu -- compiled tiles of the step in moment form for D3Q27.
// Each entry: storage / arithmetic type, tile bx x by, TMA ring depth, CTAs
// per SM; and the brick cross-sections whose contexts can end a
// run: all that are compiled, so that no batch, autotuner or requested brick takes a
// context's runs away.
#include "lb_k3_launch.cuh"

namespace lbgb {

extern const K3Variant k3_variants_d3q27[] = {
    K3Impl<D3Q27, float, float, 32, 12, 3, 1>::variant(LB_D3Q27, LB_F32),
    K3Impl<D3Q27, double, double, 32, 6, 2, 1>::variant(LB_D3Q27, LB_F64),
    K3Impl<D3Q27, __half, float, 32, 12, 3, 1>::variant(LB_D3Q27, LB_F16S),
    K3Impl<D3Q27, __nv_bfloat16, float, 32, 12, 3, 1>::variant(LB_D3Q27, LB_BF16S),
};
extern const int k3_n_variants_d3q27 = sizeof(k3_variants_d3q27) / sizeof(k3_variants_d3q27[0]);

extern const LeaveVariant leave_variants_d3q27[] = {
    LeaveImpl<D3Q27, float, float, 32, 14, 2>::variant(LB_D3Q27, LB_F32),
    LeaveImpl<D3Q27, float, float, 32, 12, 2>::variant(LB_D3Q27, LB_F32),
    LeaveImpl<D3Q27, float, float, 32, 10, 2>::variant(LB_D3Q27, LB_F32),
    LeaveImpl<D3Q27, float, float, 32, 8, 2>::variant(LB_D3Q27, LB_F32),
    LeaveImpl<D3Q27, float, float, 64, 6, 2>::variant(LB_D3Q27, LB_F32),
    LeaveImpl<D3Q27, double, double, 32, 4, 2>::variant(LB_D3Q27, LB_F64),
};
extern const int leave_n_variants_d3q27 = sizeof(leave_variants_d3q27) / sizeof(leave_variants_d3q27[0]);

}  // namespace lbgb
