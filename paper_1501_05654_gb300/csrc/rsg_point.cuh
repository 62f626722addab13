// Per-point pieces shared by the one-thread-per-value stencil kernels: row
// lookup, projector terms, and the FP64 epilogue.
#pragma once

#include "rsg_internal.h"
#include "rsg_vec.cuh"

namespace rsg {

__device__ __forceinline__ Row load_row(const Row *rows, int y, int z, int ny, int nz) {
    if (y < 0 || y >= ny || z < 0 || z >= nz) return Row{0, 1, 0, 0};
    return rows[(int64_t)z * ny + y];
}

// Projector entries of one point: their range, and the atom of the first
// (read ahead of use: pointer, atom, coefficients is a chain of three loads).
struct NlPoint {
    int e0, e1, at;
};
// acc += sum over the point's entries of p_ai D_ai, entries in list order.
template <typename R>
__device__ __forceinline__ void add_projectors(const ApplyArgs<R> &a, const NlPoint &n, int v,
                                               typename VT<R>::T &acc) {
    using T = typename VT<R>::T;
    for (int e = n.e0; e < n.e1; e++) {
        const int at = e == n.e0 ? n.at : a.e_atom[e];
        const R *pv = a.e_p + (int64_t)e * a.npmax;
        const T *Da = (const T *)a.D + (int64_t)at * a.npmax * a.SV + v;
        for (int i = 0; i < a.npmax; i++) VT<R>::fma(acc, pv[i], Da[(int64_t)i * a.SV]);
    }
}
template <typename R>
__device__ __forceinline__ NlPoint load_projectors(const ApplyArgs<R> &a, int64_t idx) {
    NlPoint n{0, 0, 0};
    if (a.nl_ptr != nullptr) {
        n.e0 = a.nl_ptr[idx];
        n.e1 = a.nl_ptr[idx + 1];
        if (n.e0 < n.e1) n.at = a.e_atom[n.e0];
    }
    return n;
}

// FP64 epilogue: the general one costs 20 FP64 instructions
// a value, which the FP64 pipe (two a clock per SM) pays next to the 50 of
// the stencil.  The host's flags (ApplyArgs::ef) name the terms that are
// absent or whose scale is purely real or imaginary, and those cost nothing.
__device__ __forceinline__ void finish_fp64(const ApplyArgs<double> &a, int64_t idx, int x, int y, int z, int v,
                                            const double2 &c, double2 acc, double d, const double2 &b,
                                            const NlPoint &nl) {
    const int SV = a.SV, ef = a.ef;
    if (a.twocol)
        d += a.cf[v][0] + a.cf[v][1] * (double)x + a.cf[v][2] * (double)y + a.cf[v][3] * (double)z;
    else if (ef & EF_FIELD)
        d += a.f0 + a.fx * (double)x + a.fy * (double)y + a.fz * (double)z;
    else if (ef & EF_SHIFT)
        d += a.f0;
    acc.x = fma(d, c.x, acc.x);
    acc.y = fma(d, c.y, acc.y);
    add_projectors<double>(a, nl, v, acc);
    const int64_t o = idx * SV + v;
    const double ar = a.twocol ? a.ca[v][0] : a.ar, ai = a.twocol ? a.ca[v][1] : a.ai;
    double2 y0 = b;   // base scale 1, or no base (b = 0)
    if (a.base != nullptr && !(ef & EF_BASE1))
        y0 = ef & EF_BASER ? make_double2(a.br * b.x, a.br * b.y) : VT<double>::cmul(a.br, a.bi, b);
    if (ef & EF_IMAG) {
        y0.x = fma(-ai, acc.y, y0.x);
        y0.y = fma(ai, acc.x, y0.y);
    } else if (ef & EF_REAL) {
        y0.x = fma(ar, acc.x, y0.x);
        y0.y = fma(ar, acc.y, y0.y);
    } else {
        VT<double>::cfma(y0, ar, ai, acc);
    }
    ((double2 *)a.out)[o] = y0;
    if (a.acc != nullptr) {
        double2 s = a.acc_base != nullptr ? ((const double2 *)a.acc_base)[o] : ((double2 *)a.acc)[o];
        if (ef & EF_GAMR) {
            s.x = fma(a.gr, y0.x, s.x);
            s.y = fma(a.gr, y0.y, s.y);
        } else {
            VT<double>::cfma(s, a.gr, a.gi, y0);
        }
        ((double2 *)a.acc)[o] = s;
    }
}

}  // namespace rsg
