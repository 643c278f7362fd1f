// vof_curvature_pair.cuh -- the PLIC offsets of two neighbours of an interface
// cell at once, for the one-thread-per-cell kernels of the curvature step and of
// its adjoint.
#pragma once
#include "plic_pair.cuh"
#include "vof_curvature.cuh"

namespace plic {

// Offsets d0(V0, n) of two neighbours of a cell (both with the centre normal
// of `pl`): for the optimised SZ solution, CellPlic<M_SZ_OPT>::offset on the
// paired FP32 instructions (two neighbours per instruction; the case-(1) cube
// root of the paired path); other methods solve one after the other.  These
// solves are most of an interface cell's instructions, and the kernels are
// issue bound: with the arcsine, the sine and a Newton step on Eq. 10 the batch of
// 64 fields (2.59 M cells) took 252 us, with a root of one polynomial and one step 207 us
// (and 189 -> 191 with that step carried to the accuracy of the former, CentreRoot).
template <int METHOD>
__device__ __forceinline__ p2::f2 offset_two(const CellPlic<METHOD>& pl, p2::f2 V0) {
    return make_float2(pl.offset(V0.x), pl.offset(V0.y));
}
template <>
__device__ __forceinline__ p2::f2 offset_two<M_SZ_OPT>(const CellPlic<M_SZ_OPT>& P, p2::f2 V0) {
    using namespace p2;
    typedef CentreRoot R;
    const f2 V = make_float2(fminf(V0.x, 1.0f - V0.x), fminf(V0.y, 1.0f - V0.y));
    // the root of cases (3)/(4), as CentreRoot::eval
    const b2 three = lt(V, mk(P.V3));
    const f2 k = sel(three, mk(-P.m3), mk(P.k4)), c = sel(three, mk(P.c3), mk(P.c4));
    const f2 X = fma(k, V, c);
    f2 z = mul(mul(X, X), sel(three, mk(P.i3), mk(P.i4)));
    z = make_float2(fminf(z.x, R::zmax), fminf(z.y, R::zmax));
    f2 p = fma(mk(R::c4), z, mk(R::c3));
    p = fma(p, z, mk(R::c2));
    p = fma(p, z, mk(R::c1));
    p = fma(p, z, mk(R::c0));
    const f2 w = mul(X, p), h = mul(mul(p, p), z);
    const f2 f = fma(w, h, fma(k, V, sub(c, w)));
    f2 s = fma(f, rcp(fma(mk(-3.0f), h, mk(1.0f))), add(w, sel(three, mk(P.b3), mk(0.0f))));
    // cases (2), (1), (5)
    s = sel(lt(V, mk(P.V2)), sub(mk(P.h2), sqrtp(fmax0(fma(mk(P.k2a), V, mk(-P.k2b))))), s);
    s = sel(lt(V, mk(P.V1)), fma(mk(-P.cb1), cbrt_(V), mk(0.5f)), s);
    s = sel(le(mk(P.V5), V), mul(mk(P.m3), sub(mk(0.5f), V)), s);
    s = mul(mk(P.L), s);
    return make_float2(copysignf(s.x, V0.x - 0.5f), copysignf(s.y, V0.y - 0.5f));
}

}  // namespace plic
