// Full-state integration in absolute coordinates, T = float (plain FP32 tracer) or
// double (FP64 tracer and its adjoint): the field at a point and one Sharma RKN or classic
// RK4 step of dr/dt = v, dv/dt = eta grad eta (Sec. 2.2, Eq. 1).  Shared by the forward
// and the adjoint, which recomputes the forward's steps with it (to rounding: what is fused is the
// compiler's choice in each kernel).
#pragma once

#include "bos_comp.cuh"
#include "bos_device.cuh"

namespace bos {

template <class T>
struct FullField;

// ---- the field in float64
//
// GB300 runs float64 at a 64th of the float32 rate: its pipe bounds these tracers (82 % busy,
// issue 8 %), so what counts is the number of float64 operations.  A point inside the cell of
// the ray's previous one takes 15 for its fractions (a saturating conversion and integer
// clamps; a division by h and float64 clamps took 48) and 28 for the cell's trilinear
// polynomial (56 as lerps of the corners); forming the polynomial (48) is shared by the six or
// so points of a cell.  Registers are free beside that: a few warps keep the pipe busy.

// A cell's trilinear polynomial in its fractions (x, y, z):
// c[0] + x c[1] + y (c[2] + x c[3]) + z (c[4] + x c[5] + y (c[6] + x c[7])).
struct DCell {
    int i[3];       // base node; -1: no cell yet
    D4 c[8];
};

__device__ __forceinline__ D4 dsub4(D4 a, D4 b) { return D4{a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w}; }
__device__ __forceinline__ D4 dfma4(double t, D4 a, D4 b) {
    return D4{fma(t, a.x, b.x), fma(t, a.y, b.y), fma(t, a.z, b.z), fma(t, a.w, b.w)};
}

// Base node i (clamped to the grid) and fraction f of a point along each axis.
__device__ __forceinline__ void split_point(const GridDev& g, const double x[3], int i[3], double f[3]) {
    for (int a = 0; a < 3; ++a) {
        const double u = fma(x[a] - g.origin[a], g.inv_h[a], -0.5);
        i[a] = min(max(__double2int_rd(u), 0), g.n[a] - 2);
        f[a] = u - (double)i[a];
    }
}

// Fractions of x; moves m to the cell of x where it is another one.
__device__ __forceinline__ void dcell_point(const GridDev& g, const double x[3], DCell& m, double f[3]) {
    int i[3];
    split_point(g, x, i, f);
    if (i[0] == m.i[0] && i[1] == m.i[1] && i[2] == m.i[2]) return;
    for (int a = 0; a < 3; ++a) m.i[a] = i[a];
    uint32_t o = bounded(brick_offset(i[0], i[1], i[2]) + 91u, g.store_elems, g.err);
    o = o ? o - 91u : 0u;
    const D4* s = static_cast<const D4*>(g.store);
    const D4 c0 = load_d4(s, o), c2 = load_d4(s, o + 9), c4 = load_d4(s, o + 81), c6 = load_d4(s, o + 90);
    const D4 d0 = dsub4(load_d4(s, o + 1), c0), d2 = dsub4(load_d4(s, o + 10), c2), d4 = dsub4(load_d4(s, o + 82), c4),
             d6 = dsub4(load_d4(s, o + 91), c6);
    m.c[0] = c0;
    m.c[1] = d0;
    m.c[2] = dsub4(c2, c0);
    m.c[3] = dsub4(d2, d0);
    m.c[4] = dsub4(c4, c0);
    m.c[5] = dsub4(d4, d0);
    m.c[6] = dsub4(dsub4(c6, c4), m.c[2]);
    m.c[7] = dsub4(dsub4(d6, d4), m.c[3]);
}

__device__ __forceinline__ D4 dcell_value(const DCell& m, const double f[3]) {
    const D4 e0 = dfma4(f[0], m.c[1], m.c[0]), e1 = dfma4(f[0], m.c[3], m.c[2]);
    const D4 e2 = dfma4(f[0], m.c[5], m.c[4]), e3 = dfma4(f[0], m.c[7], m.c[6]);
    return dfma4(f[2], dfma4(f[1], e3, e2), dfma4(f[1], e1, e0));
}

template <>
struct FullField<double> {
    GridDev g;
    mutable DCell m = {{-1, -1, -1}, {}};
    __device__ __forceinline__ D4 at(const double x[3]) const {
        double f[3];
        dcell_point(g, x, m, f);
        return dcell_value(m, f);
    }
    __device__ __forceinline__ void rhs(const double x[3], double D[3]) const {
        const D4 v = at(x);
        const double eta = 1.0 + v.x;
        D[0] = eta * v.y;
        D[1] = eta * v.z;
        D[2] = eta * v.w;
    }
    __device__ __forceinline__ double eta(const double x[3]) const { return 1.0 + at(x).x; }
};

template <>
struct FullField<float> {
    GridDev g;
    __device__ __forceinline__ float4 at(const float x[3]) const {
        int i[3];
        float f[3];
        for (int a = 0; a < 3; ++a) {
            float u = (x[a] - (float)g.origin[a]) * g.inv_hf[a] - 0.5f;
            split_coord(u, g.n[a], i[a], f[a]);
        }
        uint32_t o = bounded(brick_offset(i[0], i[1], i[2]) + 90u, g.store_elems, g.err);
        o = o ? o - 90u : 0u;
        return trilinear(static_cast<const F4P*>(g.store), o, f[0], f[1], f[2]);
    }
    __device__ __forceinline__ void rhs(const float x[3], float D[3]) const { rhs_of(at(x), D); }
    __device__ __forceinline__ float eta(const float x[3]) const { return 1.0f + at(x).x; }
};

// A float64 division takes about nine operations of its pipe, the product one.
__device__ __forceinline__ float sixth(float x) { return x / 6.0f; }
__device__ __forceinline__ double sixth(double x) { return x * (1.0 / 6.0); }

template <class T, int INTEG>
__device__ __forceinline__ void full_step(const FullField<T>& F, T r[3], T v[3], T dt) {
    if (INTEG == 0) {
        T A[3], B[3], C[3], p[3], D[3];
        F.rhs(r, D);
        for (int a = 0; a < 3; ++a) A[a] = dt * D[a];
        for (int a = 0; a < 3; ++a) p[a] = r[a] + (dt * T(0.5)) * v[a] + (dt * T(0.125)) * A[a];
        F.rhs(p, D);
        for (int a = 0; a < 3; ++a) B[a] = dt * D[a];
        for (int a = 0; a < 3; ++a) p[a] = r[a] + dt * v[a] + (dt * T(0.5)) * B[a];
        F.rhs(p, D);
        for (int a = 0; a < 3; ++a) C[a] = dt * D[a];
        for (int a = 0; a < 3; ++a) {
            r[a] = r[a] + dt * (v[a] + sixth(A[a] + T(2) * B[a]));
            v[a] = v[a] + sixth(A[a] + T(4) * B[a] + C[a]);
        }
    } else {
        T k1v[3], k2v[3], k3v[3], k4v[3], k2r[3], k3r[3], k4r[3], p[3];
        F.rhs(r, k1v);
        for (int a = 0; a < 3; ++a) {
            k2r[a] = v[a] + (dt * T(0.5)) * k1v[a];
            p[a] = r[a] + (dt * T(0.5)) * v[a];
        }
        F.rhs(p, k2v);
        for (int a = 0; a < 3; ++a) {
            k3r[a] = v[a] + (dt * T(0.5)) * k2v[a];
            p[a] = r[a] + (dt * T(0.5)) * k2r[a];
        }
        F.rhs(p, k3v);
        for (int a = 0; a < 3; ++a) {
            k4r[a] = v[a] + dt * k3v[a];
            p[a] = r[a] + dt * k3r[a];
        }
        F.rhs(p, k4v);
        for (int a = 0; a < 3; ++a) {
            r[a] = r[a] + dt / T(6) * (v[a] + T(2) * k2r[a] + T(2) * k3r[a] + k4r[a]);
            v[a] = v[a] + dt / T(6) * (k1v[a] + T(2) * k2v[a] + T(2) * k3v[a] + k4v[a]);
        }
    }
}

}  // namespace bos
