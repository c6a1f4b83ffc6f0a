// Host arithmetic of the coefficient table: neighbour coefficients of one position of an
// axis (Eq. pml-1d-s).
//
// A last bit here is a difference of up to 5e-9 in the solution of a complex64 solve, so
// the products' rounding is fixed by the source: this file is compiled with
// -ffp-contract=off and says itself which of them go into a multiply-add (std::fma rounds
// once on every machine).  Left to gcc they depend on what the compiler inlines around
// them on aarch64, and there are none on plain x86-64.  Which product goes in unrounded
// is as gcc 13 had it on aarch64, in the table and in the plan's bound, so that solutions
// keep their bits.  (1 / s is libgcc's complex division, one library call.)
#include <cmath>

#include "mxp_internal.h"

namespace mxp {

using cd = std::complex<double>;

// a b with one multiply-add per component.  Unrounded goes in: re_ii: the product of the
// imaginary parts, else of the real parts; im_ir: Im a Re b, else Re a Im b.
static cd cmul_fma(cd a, cd b, bool re_ii, bool im_ir)
{
    const double ar = a.real(), ai = a.imag(), br = b.real(), bi = b.imag();
    return cd(re_ii ? std::fma(-ai, bi, ar * br) : std::fma(ar, br, -(ai * bi)),
              im_ir ? std::fma(ai, br, ar * bi) : std::fma(ar, bi, ai * br));
}

// 1 / s at coordinate x
static cd inv_stretch(const PmlAxis &ax, double x)
{
    if (ax.npml == 0) return 1.0;
    const double L = (double)ax.n_interior * ax.h, delta = ax.npml * ax.h;
    double dist = 0.0;
    if (x < 0.0) dist = -x;
    if (x > L) dist = x - L;
    const double r = dist / delta;
    return 1.0 / cd(1.0, ax.c_pml / (delta * ax.omega) * r * r);
}

void pml_neighbours(const PmlAxis &ax, int64_t i, bool bound, cd *wp, cd *wm)
{
    const double h = ax.h, ih2 = 1.0 / (h * h);
    const double x = ((double)i - ax.npml + 0.5) * h;
    const cd a = inv_stretch(ax, x);
    *wp = cmul_fma(a, inv_stretch(ax, x + 0.5 * h), !bound, false) * ih2;
    *wm = cmul_fma(a, inv_stretch(ax, x - 0.5 * h), false, bound) * ih2;
}

}  // namespace mxp
