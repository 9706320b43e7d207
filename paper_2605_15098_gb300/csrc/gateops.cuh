// One gate on one amplitude or amplitude pair: the arithmetic shared by the
// per-gate kernels (pergate.cu) and the resident kernel (small.cu), so that
// both give the same bits.  Included inside namespace sv.
#pragma once

#include "common.h"

namespace sv {
namespace {

template <typename R>
struct Coef {
    R re[4], im[4];
};

enum Op { OP_U = 0, OP_H = 1, OP_X = 2, OP_PHASE = 3, OP_NEG = 4, OP_SWAP = 5 };

template <typename R>
__device__ __forceinline__ R scale_h(R x, const Coef<R> &c) {
    if constexpr (sizeof(R) == 4)
        return fmaf(x, c.re[0], x * c.im[0]);
    else
        return x * c.re[0];
}

// (a, b) <- U (a, b) for one amplitude pair, by kind.
template <typename R, int OP>
__device__ __forceinline__ void pair_update(R &ar, R &ai, R &br, R &bi, const Coef<R> &c) {
    if (OP == OP_U) {
        R xr = c.re[0] * ar - c.im[0] * ai + c.re[1] * br - c.im[1] * bi;
        R xi = c.re[0] * ai + c.im[0] * ar + c.re[1] * bi + c.im[1] * br;
        R yr = c.re[2] * ar - c.im[2] * ai + c.re[3] * br - c.im[3] * bi;
        R yi = c.re[2] * ai + c.im[2] * ar + c.re[3] * bi + c.im[3] * br;
        ar = xr; ai = xi; br = yr; bi = yi;
    } else if (OP == OP_H) {
        // complex64: 1/sqrt(2) = s_hi + s_lo (two floats) so that the product
        // is rounded once, without the bias of a rounded constant
        R xr = ar + br, xi = ai + bi, yr = ar - br, yi = ai - bi;
        ar = scale_h(xr, c); ai = scale_h(xi, c); br = scale_h(yr, c); bi = scale_h(yi, c);
    } else if (OP == OP_X || OP == OP_SWAP) {
        R tr = ar, ti = ai;
        ar = br; ai = bi; br = tr; bi = ti;
    }
}

template <typename R, int OP>
__device__ __forceinline__ void single_update(R &ar, R &ai, const Coef<R> &c) {
    if (OP == OP_PHASE) {
        R xr = ar * c.re[0] - ai * c.im[0];
        R xi = ar * c.im[0] + ai * c.re[0];
        ar = xr; ai = xi;
    } else if (OP == OP_NEG) {
        ar = -ar; ai = -ai;
    }
}

template <typename R>
Coef<R> to_coef(const Mat2 &m) {
    Coef<R> c;
    for (int e = 0; e < 4; e++) {
        c.re[e] = (R)m.re[e];
        c.im[e] = (R)m.im[e];
    }
    return c;
}

// Operation and coefficients of a gate of the paper's set.
inline int gate_op(const sv_gate &g, sv_dtype dt, Mat2 *m) {
    int op = -1;
    switch (g.kind) {
        case SV_X: op = OP_X; break;
        case SV_H: op = OP_H; break;
        case SV_U3: case SV_U: case SV_CU: op = OP_U; break;
        case SV_CZ: op = OP_NEG; break;
        case SV_P: case SV_CP: case SV_PK: case SV_CPK: op = OP_PHASE; break;
        case SV_SWAP: op = OP_SWAP; break;
        default: return -1;
    }
    *m = Mat2{};
    if (op != OP_SWAP && op != OP_NEG) *m = gate_matrix(g);
    if (op == OP_H) {
        const double r = 0.70710678118654752440084436210485;
        m->re[0] = r;
        m->im[0] = dt == SV_C64 ? r - (double)(float)r : 0.0;  // low part for complex64
    }
    if (op == OP_PHASE) {  // coefficient on |1>
        m->re[0] = m->re[3];
        m->im[0] = m->im[3];
    }
    return op;
}

}  // namespace
}  // namespace sv
