// The step of an RK stage, shared by the kernels that update cells.
#pragma once

#include "launch.h"

namespace wz {

__device__ __forceinline__ double bits_to_double(unsigned long long b) {
    return __longlong_as_double((long long)b);
}

// CFL step of the current RK3 step from the LF speeds of U^n (slot 0), in the operation
// order of the oracle: 1D cfl dx / a_x (Sec. 4.3); 2D cfl dtx dty / (dtx + dty) with
// dtx = dx / a_x, dty = dy / a_y (Sec. 4.4); advection cfl dx / |a|.
__device__ __forceinline__ double step_dt(const UpdateArgs& a, int system) {
    double dt = a.dt_fixed;
    if (!(dt > 0.0)) {
        if (system == 0) {
            dt = __ddiv_rn(__dmul_rn(a.cfl, a.dx), fabs(a.adv_speed));
        } else {
            const double ax = bits_to_double(a.ctrl->alpha[0][0]);
            if (system == 1) {
                dt = __ddiv_rn(__dmul_rn(a.cfl, a.dx), ax);
            } else {
                const double ay = bits_to_double(a.ctrl->alpha[0][1]);
                const double tx = __ddiv_rn(a.dx, ax), ty = __ddiv_rn(a.dy, ay);
                dt = __ddiv_rn(__dmul_rn(__dmul_rn(a.cfl, tx), ty), __dadd_rn(tx, ty));
            }
        }
    }
    if (a.t_remaining > 0.0 && dt > a.t_remaining) dt = a.t_remaining;
    return dt;
}

}  // namespace wz
