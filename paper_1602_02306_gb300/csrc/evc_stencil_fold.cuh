// evc_stencil_fold.cuh -- the FP64 arithmetic of a stencil point.
//
// The FP64 passes are bound by the FP64 units (0.5 TFMA/s in all): every operation
// counts.  With the scale of the operand's column, the pass's scale k1 and the
// stencil's coefficients folded into per-column constants,
//   insc (k1 (c1 S1 + c2 S2) + (k1 cd + k0 + V_p - sigma) x)
//     = A1 S1 + A2 S2 + (B + insc V_p) x
// costs 5 additions, one product and one fused multiply-add for the 7-point
// stencil (6 and one more with V, 13-point) where the FP32 form, whose roundings
// are kept, spends 11.  40^3, 64 columns, 17 passes: 1.76 -> 1.2 ms per step.
#pragma once

#include "evc_internal.cuh"

namespace evc {
namespace {

template <int LPP>
struct Fold64 {
    struct alignas(16) Two { double v[2]; };
    Two a1[LPP], a2[LPP], b[LPP];

    __device__ void set(int l, int w, const StencilPass& p, const StencilOp& op, double insc, double sigma)
    {
        a1[l].v[w] = insc * p.k1 * op.c1;
        a2[l].v[w] = insc * p.k1 * op.c2;
        b[l].v[w] = insc * (p.k1 * op.cd + p.k0 - sigma);
    }
    template <int R, bool VS>
    __device__ __forceinline__ double apply(int l, int w, double s1, double s2, double x, double insc,
                                            double vp) const
    {
        const double coef = VS ? fma(insc, vp, b[l].v[w]) : b[l].v[w];
        double r = fma(a1[l].v[w], s1, coef * x);
        if (R == 2) r = fma(a2[l].v[w], s2, r);
        return r;
    }
};

}  // namespace
}  // namespace evc
