// Marching a ray through the brick store cell by cell (compensated tracers).
//
// A ray's stage points (the start, middle and end of every step) sit on its fixed-point
// straight line plus a small deviation.  Consecutive points are a quarter of a cell apart or
// less, so a ray stays in a cell for several of them.  The marcher keeps, per ray:
//   - the cell's trilinear polynomial in registers (8 coefficients of (deta, grad eta),
//     formed once per cell from its 4 paired records), so a point inside the cell costs 14
//     packed FMAs and no load;
//   - its line split into float32 parts relative to that cell, so a point's fraction is three
//     operations per axis and needs no integer arithmetic or conversions.
// What bounds it: instruction issue (63 % of the slots; float32 FMA instructions, most of them
// packed, fill 39 % of their pipe's, L1 is at 20 %) with 16 warps per SM.  A point inside its cell takes ~35 instructions where gathering each stage through the 64-bit
// line position, the brick address and seven packed lerps took ~90; the rest is cell changes
// (~80 each, and rays of a warp that cross an x or z face one after the other each pay theirs).
// Flow render of 128x128x96 cells, 1024^2 x 4 rays: 13.71 ms stage by stage, 10.45 ms so; of
// 256x256x192 cells at 256^2 rays: 745 us, 450 us.  At 96 registers (20 warps per SM) 10.74 ms
// and 580 us, at 168 (12 warps) 12.5 ms and 712 us.  Its displacements are nearer the float64
// result (4.0e-8 rms of the largest against 9.2e-8) since the acceleration's scale is rounded
// once per ray.
#pragma once

#include "bos_comp.cuh"

namespace bos {

__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 neg2(f32x2 a) { return a ^ 0x8000000080000000ull; }
__device__ __forceinline__ f32x2 splat2(float a) { return pack2(a, a); }
__device__ __forceinline__ float lo2(f32x2 v) {
    float a, b;
    unpack2(v, a, b);
    return a;
}
__device__ __forceinline__ float hi2(f32x2 v) {
    float a, b;
    unpack2(v, a, b);
    return b;
}

// A 3-vector as x and the packed pair (y, z): a record's second pair is (g_y, g_z), so field
// gradients need no shuffling.
struct P3 {
    float x;
    f32x2 yz;
};
__device__ __forceinline__ P3 p3(float x, float y, float z) { return P3{x, pack2(y, z)}; }
__device__ __forceinline__ P3 add3(P3 a, P3 b) { return P3{__fadd_rn(a.x, b.x), add2(a.yz, b.yz)}; }
__device__ __forceinline__ P3 sub3(P3 a, P3 b) { return P3{__fsub_rn(a.x, b.x), sub2(a.yz, b.yz)}; }
__device__ __forceinline__ P3 fma3(float s, P3 a, P3 b) { return P3{fmaf(s, a.x, b.x), fma2(splat2(s), a.yz, b.yz)}; }
__device__ __forceinline__ P3 mul3(float s, P3 a) { return P3{__fmul_rn(s, a.x), mul2(splat2(s), a.yz)}; }
__device__ __forceinline__ float dot3(P3 a, P3 b) {
    const f32x2 p = mul2(a.yz, b.yz);
    return fmaf(a.x, b.x, __fadd_rn(lo2(p), hi2(p)));
}
// The largest one; NaN where any is (fmaxf drops a NaN).
__device__ __forceinline__ float max_nan(float a, float b) {
    float r;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float max_nan(float a, float b, float c) {
    float r;
    asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ float maxabs3(P3 a) { return max_nan(fabsf(a.x), fabsf(lo2(a.yz)), fabsf(hi2(a.yz))); }

// s += x with Kahan compensation c, x already reduced by c (y = x - c).
__device__ __forceinline__ void kahan3(P3& s, P3& c, P3 y) {
    const P3 t = add3(s, y);
    c = sub3(sub3(t, s), y);
    s = t;
}

// The trilinear polynomial of a cell in its fractions (x, y, z), per channel pair:
// c[0] + x c[1] + y (c[2] + x c[3]) + z (c[4] + x c[5] + y (c[6] + x c[7])).
struct CellPoly {
    Cell2 c[8];
};

__device__ __forceinline__ Cell2 csub(Cell2 a, Cell2 b) { return Cell2{sub2(a.lo, b.lo), sub2(a.hi, b.hi)}; }
__device__ __forceinline__ Cell2 cfma(f32x2 t, Cell2 a, Cell2 b) { return Cell2{fma2(t, a.lo, b.lo), fma2(t, a.hi, b.hi)}; }

template <class E>
__device__ __forceinline__ void load_poly(const E* s, uint32_t o, CellPoly& p) {
    Cell2 v1, d1, v2, d2, v3, d3;
    load_rec(s, o, p.c[0], p.c[1]);
    load_rec(s, o + 9, v1, d1);
    load_rec(s, o + 81, v2, d2);
    load_rec(s, o + 90, v3, d3);
    p.c[2] = csub(v1, p.c[0]);
    p.c[3] = csub(d1, p.c[1]);
    p.c[4] = csub(v2, p.c[0]);
    p.c[5] = csub(d2, p.c[1]);
    p.c[6] = csub(csub(v3, v2), p.c[2]);
    p.c[7] = csub(csub(d3, d2), p.c[3]);
}

__device__ __forceinline__ Cell2 poly_value(const CellPoly& p, f32x2 x, f32x2 y, f32x2 z) {
    const Cell2 e0 = cfma(x, p.c[1], p.c[0]), e1 = cfma(x, p.c[3], p.c[2]);
    const Cell2 e2 = cfma(x, p.c[5], p.c[4]), e3 = cfma(x, p.c[7], p.c[6]);
    return cfma(z, cfma(y, e3, e2), cfma(y, e1, e0));
}

// A ray's straight line u(h) = u0 + h du at half step h (in cells), split so that float32
// evaluates it anywhere to the resolution of a fraction: u(h) - cell = fma(h, dh, base) +
// corr, base = (u0 rounded to 2^-9) - cell exact, one rounding in the fma, and
// corr = (the rest of u0) + h (du - dh) kept from the half step where the cell was entered (it
// drifts by at most 2^-25 of a cell before the ray leaves the cell).
struct MarchLine {
    P3 dh, dlo;       // half step in cells: float32 and the rest
    P3 ulo;           // rest of u0
    P3 ih;            // 1 / h
};

struct MarchCell {
    P3 base, corr;
    P3 ci;            // base corner of the cell, each + kCellBias (so that its bits hold the integer)
    uint32_t brick;   // store element of the cell's brick
    CellPoly p;
};

// Cell indices live in the mantissas of floats (2^23 + i): clamping, moving and reading them
// takes float32 operations only, where F2I, I2F and FRND have a quarter of the rate or less and
// several times the latency.
constexpr float kCellBias = 8388608.0f;
constexpr float kFloorBias = 12582912.0f;   // 1.5 2^23: adding it rounding down leaves the floor

constexpr int kLineSteps = 1 << 20;   // steps after which the line is set up anew (h stays exact in float32)

// A value formed from float64 operations before a loop, opaque to the compiler: it otherwise
// repeats the operations inside the loop (next to a use, or in the cell change) to save a
// register, and the float64 pipe takes 64 cycles per warp instruction.
__device__ __forceinline__ float kept(float v) {
    asm volatile("" : "+f"(v));
    return v;
}

// The line u0 + h du (grid units, du per half step), and a cell that no point lies in yet.
__device__ __forceinline__ void march_line(const float inv_h[3], const double u0[3], const double du[3], MarchLine& L,
                                           MarchCell& m) {
    float dh[3], dlo[3], ulo[3], base[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        dh[a] = (float)du[a];
        dlo[a] = (float)(du[a] - (double)dh[a]);
        // u0 to a multiple of 2^-9: 3 2^42 puts that bit last in a double
        const double r = (u0[a] + 13194139533312.0) - 13194139533312.0;
        base[a] = (float)r;
        ulo[a] = (float)(u0[a] - r);
        dh[a] = kept(dh[a]), dlo[a] = kept(dlo[a]), ulo[a] = kept(ulo[a]), base[a] = kept(base[a]);
    }
    L.dh = p3(dh[0], dh[1], dh[2]);
    L.dlo = p3(dlo[0], dlo[1], dlo[2]);
    L.ulo = p3(ulo[0], ulo[1], ulo[2]);
    L.ih = p3(inv_h[0], inv_h[1], inv_h[2]);
    m.base = p3(base[0], base[1], base[2]);
    m.corr = L.ulo;
    m.ci = P3{kCellBias, splat2(kCellBias)};
}

// march_line leaves the ray in cell (0, 0, 0), whose polynomial is not loaded yet: the next point
// is found by march_point<true>, or, where that would be a second copy of it, after this: the
// indices go to -2^14 on every axis, outside any grid (at most 8192 cells), so that march_point
// sees a change of cell and of brick (the base stays exact, and the estimate of the new cell is
// off by one only within 2^-9 of a face, where both cells' polynomials agree to that).
__device__ __forceinline__ void march_leave(MarchCell& m) {
    const P3 away = {16384.0f, splat2(16384.0f)};
    m.ci = sub3(m.ci, away);
    m.base = add3(m.base, away);
}

// LINE: the point on the line itself (q is not looked at).
template <bool LINE>
__device__ __forceinline__ P3 march_frac(const MarchLine& L, const MarchCell& m, f32x2 h, P3 q) {
    const P3 u = P3{fmaf(lo2(h), L.dh.x, m.base.x), fma2(h, L.dh.yz, m.base.yz)};
    if constexpr (LINE) return add3(u, m.corr);
    return add3(u, P3{fmaf(q.x, L.ih.x, m.corr.x), fma2(q.yz, L.ih.yz, m.corr.yz)});
}

struct Frac3 {
    float x, y, z;
};

// Fractions of the point of half step h (both halves) with deviation q (metres).  Where they
// fall outside the cell the ray is moved to the cell of the point (clamped to the grid: the
// edge cells extrapolate) and that cell's polynomial is loaded.  FIRST: no cell is loaded yet.
// Returns true where the cell changed.
template <bool FIRST, bool LINE = false, class E>
__device__ __forceinline__ bool march_point(const CompField<E>& F, const MarchLine& L, MarchCell& m, f32x2 h, P3 q,
                                            Frac3& f) {
    P3 u = march_frac<LINE>(L, m, h, q);
    f = Frac3{u.x, lo2(u.yz), hi2(u.yz)};
    // 0 <= f < 1 exactly when the bit pattern is below that of 1.0f
    const uint32_t top = max(__float_as_uint(f.x), max(__float_as_uint(f.y), __float_as_uint(f.z)));
    if (!FIRST && top < 0x3f800000u) return false;
    const float cf[3] = {f.x, f.y, f.z}, old[3] = {m.ci.x, lo2(m.ci.yz), hi2(m.ci.yz)};
    float ci[3], back[3];
    uint32_t c[3], moved = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float fl = __fsub_rn(__fadd_rd(cf[a], kFloorBias), kFloorBias);
        ci[a] = fminf(fmaxf(__fadd_rn(old[a], fl), kCellBias), kCellBias + (float)(F.n[a] - 2));
        back[a] = __fsub_rn(old[a], ci[a]);
        c[a] = __float_as_uint(ci[a]);
        moved |= c[a] ^ __float_as_uint(old[a]);
    }
    if (!FIRST && moved == 0u) return false;
    m.ci = p3(ci[0], ci[1], ci[2]);
    m.base = add3(m.base, p3(back[0], back[1], back[2]));
    m.corr = P3{fmaf(lo2(h), L.dlo.x, L.ulo.x), fma2(h, L.dlo.yz, L.ulo.yz)};
    u = march_frac<LINE>(L, m, h, q);
    f = Frac3{u.x, lo2(u.yz), hi2(u.yz)};
    if (FIRST || (moved >> 3) != 0u)
        m.brick = morton3((c[0] & 0x7fffffu) >> 3, (c[1] & 0x7fffffu) >> 3, (c[2] & 0x7fffffu) >> 3) *
                  (uint32_t)kBrickCells;
    uint32_t o = m.brick + ((c[2] & 7u) * kBrickSide + (c[1] & 7u)) * kBrickSide + (c[0] & 7u);
#if BOS_CHECKED
    o = bounded(o + 90u, F.nelem, F.err);
    o = o ? o - 90u : 0u;
#endif
    load_poly(F.store, o, m.p);
    return true;
}

// (deta, grad eta) at a point.
template <bool FIRST = false, bool LINE = false, class E>
__device__ __forceinline__ Cell2 march_value(const CompField<E>& F, const MarchLine& L, MarchCell& m, f32x2 h, P3 q) {
    Frac3 f;
    march_point<FIRST, LINE>(F, L, m, h, q, f);
    return poly_value(m.p, splat2(f.x), splat2(f.y), splat2(f.z));
}

// s eta grad eta there (s = dt^2 / 6: the acceleration scaled to metres per step).
__device__ __forceinline__ P3 march_accel(Cell2 v, float s) {
    const float se = fmaf(s, lo2(v.lo), s);
    return P3{__fmul_rn(se, hi2(v.lo)), mul2(splat2(se), v.hi)};
}

// Two stage points closer than this fraction of a cell are one point to the resolution that a
// float32 fraction in [0, 1) has: rounding alone moves a fraction by up to 2^-24.
constexpr float kSamePoint = 5.9604645e-8f;   // 2^-24 cells

// Bound of the same difference for reversing a ray without its stage terms (see
// bos_adjoint.cu): it enters the gradient relative to one, so four times the resolution.
constexpr float kSameReverse = 2.3841858e-7f;   // 2^-22 cells

__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

}  // namespace bos
