// Forward kernels of the BOS library for sm_103a:
//   build_store   -- step a1: T -> (eta - 1, grad eta) bricks                 (Sec. 2.1)
//   render        -- steps a2-a5: rays, Sharma RKN tracing, wall, radiance    (Eq. 1, Eq. 2)
//   ray_steps     -- the integer step count of every ray (step a2)
//   export_nodes  -- read the store back through the brick addressing
//   loss_l2       -- L_BOS and its seed dL/dI                                 (Sec. 2.4)
#include "bos_comp.cuh"
#include "bos_device.cuh"
#include "bos_full.cuh"
#include "bos_internal.h"
#include "bos_march.cuh"

namespace bos {

// ===================================================================== a1: field store

__device__ __forceinline__ double deta_at(const GridDev& g, const float* T, int i, int j, int k) {
    double t = (double)__ldg(T + ((size_t)k * g.n[1] + j) * g.n[0] + i);
    return ddiv(g.K, t);
}

// One block per brick: deta = K / T is computed once for every cell of the brick's 9^3
// records plus a one-cell halo (11^3 values in shared memory), then each record takes
// its central or one-sided differences from there.  Bricks cover base cells 0..n-2;
// coordinates beyond the grid are clamped (those records are never read).
constexpr int kHalo = kBrickSide + 2;   // 11

// Store element of each record type: float32 and bfloat16 records are stored as x pairs
// (F4P, B4P), float64 records as they are.
template <class R>
struct StoreElem {
    using type = R;
};
template <>
struct StoreElem<float4> {
    using type = F4P;
};
template <>
struct StoreElem<uint2> {
    using type = B4P;
};

__device__ __forceinline__ void write_elem(F4P* dst, const float4* rec, int l, bool next) {
    const float4 a = rec[l], b = next ? rec[l + 1] : a;
    F4P p;
    p.v = a;
    p.d = make_float4(b.x - a.x, b.y - a.y, b.z - a.z, b.w - a.w);   // float32 subtractions
    *dst = p;
}
__device__ __forceinline__ void write_elem(B4P* dst, const uint2* rec, int l, bool next) {
    B4P p;
    p.a = rec[l];
    p.b = next ? rec[l + 1] : make_uint2(0u, 0u);
    *dst = p;
}

// The float64 store, evaluated in float64.
__global__ void __launch_bounds__(256) build_store_kernel(GridDev g, const float* __restrict__ T, D4* __restrict__ store) {
    __shared__ double de[kHalo * kHalo * kHalo];
    const int b = blockIdx.x;
    const int bx = b % g.nb[0], by = (b / g.nb[0]) % g.nb[1], bz = b / (g.nb[0] * g.nb[1]);
    const int ox = bx * kBrick - 1, oy = by * kBrick - 1, oz = bz * kBrick - 1;
    for (int t = threadIdx.x; t < kHalo * kHalo * kHalo; t += blockDim.x) {
        const int hx = t % kHalo, hy = (t / kHalo) % kHalo, hz = t / (kHalo * kHalo);
        const int i = min(max(ox + hx, 0), g.n[0] - 1), j = min(max(oy + hy, 0), g.n[1] - 1),
                  k = min(max(oz + hz, 0), g.n[2] - 1);
        de[t] = deta_at(g, T, i, j, k);
    }
    __syncthreads();
    const size_t slot = morton3((uint32_t)bx, (uint32_t)by, (uint32_t)bz);
    for (int local = threadIdx.x; local < kBrickCells; local += blockDim.x) {
        const int lx = local % kBrickSide, ly = (local / kBrickSide) % kBrickSide, lz = local / (kBrickSide * kBrickSide);
        const int c[3] = {min(bx * kBrick + lx, g.n[0] - 1), min(by * kBrick + ly, g.n[1] - 1),
                          min(bz * kBrick + lz, g.n[2] - 1)};
        // halo index of a (clamped) grid cell
        auto at = [&](int i, int j, int k) { return de[((k - oz) * kHalo + (j - oy)) * kHalo + (i - ox)]; };
        double gr[3];
        for (int a = 0; a < 3; ++a) {
            int lo[3] = {c[0], c[1], c[2]}, hi[3] = {c[0], c[1], c[2]};
            double den = dmul(2.0, g.h[a]);
            lo[a] = c[a] - 1;
            hi[a] = c[a] + 1;
            if (lo[a] < 0) {
                lo[a] = c[a];
                den = g.h[a];
            }
            if (hi[a] > g.n[a] - 1) {
                hi[a] = c[a];
                den = g.h[a];
            }
            gr[a] = ddiv(dsub(at(hi[0], hi[1], hi[2]), at(lo[0], lo[1], lo[2])), den);
        }
        double2* dst = reinterpret_cast<double2*>(store + slot * kBrickCells + local);
        dst[0] = make_double2(at(c[0], c[1], c[2]), gr[0]);
        dst[1] = make_double2(gr[1], gr[2]);
    }
}

// ---- float32 and bfloat16 records without the float64 pipe
//
// A record's values are float64 results rounded once to float32 or bfloat16: RN(K / T) and
// RN(RN(K / T_hi - K / T_lo) / den).  GB300 runs float64 at a 64th of the float32 rate, and
// build_store_kernel's seven divisions per cell kept that pipe busy for 1.66 ms on 256x256x192
// cells.  Here the same values are formed from unevaluated sums of float32: K / T in three
// terms (long division, each remainder exact by an fma; Dekker 1971), differences by two-sums
// (Knuth), the product with 1 / den in two terms.  The result's float32 rounding f and what
// is left, rho, are kept with a bound E of everything the float64 evaluation or the sums round
// off; |rho| + E < ulp(f) / 2 proves that the float64 evaluation rounds to f too.  Otherwise
// (one value in ~10^4 of a field with structure; smoother ones more often) the value is
// evaluated in float64 as above.  The node values are the same bits.
// What bounds it: issue (~150 instructions per record) and the store's 32 bytes per element;
// 256x256x192 cells: 1.66 ms before, 324 us now (64^3: 44 us, 11.5 us; bfloat16 192x192x144: 706 us,
// 138 us), against 0.12 ms to write 717 MB.

struct Split3 {          // K, or K / T
    float a, b, c;
};
struct BuildConst {
    Split3 K;
    float rh[3][2], rl[3][2];   // 1 / (2 h) and 1 / h per axis in two terms
    float rm[3][2];             // upper bounds of both, times 2^-51
};

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float t = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
}

// K / T to 2^-66 relative; NaN in the second term where a remainder could leave float32's range.
__device__ __forceinline__ Split3 divide3(const Split3& K, float T) {
    const float y = __frcp_rn(T);
    Split3 q;
    q.a = __fdiv_rn(K.a, T);
    float r = fmaf(-q.a, T, K.a), e;             // exact for a correctly rounded quotient
    two_sum(r, K.b, r, e);
    q.b = __fmul_rn(r, y);
    r = __fadd_rn(fmaf(-q.b, T, r), __fadd_rn(e, K.c));
    q.c = __fmul_rn(r, y);
    const float m = fabsf(q.a);
    if (!(fabsf(T) > 1.0e-15f && fabsf(T) < 1.0e15f && m > 1.0e-12f && m < 1.0e12f))
        q.b = __int_as_float(0x7fc00000);
    return q;
}

// f = RN(p + e), |e| << |p|; true where a value within E of p + e rounds to f as well.
__device__ __forceinline__ bool rounds_to(float p, float e, float E, float& f) {
    f = __fadd_rn(p, e);
    const float rho = __fsub_rn(e, __fsub_rn(f, p));
    const uint32_t b = __float_as_uint(f);
    // half an ulp; a power of two has half of that below it, and tiny results are left out
    const float half = __uint_as_float((b & 0x7f800000u) - (24u << 23));
    return (b & 0x7fffffu) != 0u && (b & 0x7f800000u) > (64u << 23) && fabsf(rho) + E < half;
}
__device__ __forceinline__ bool rounds_to(float p, float e, float E, uint16_t& h) {
    float f;
    if (!rounds_to(p, e, E, f)) return false;
    h = __bfloat16_as_ushort(__float2bfloat16_rn(f));
    return (__float_as_uint(f) & 0xffffu) != 0x8000u;   // halfway: the rest decides
}

__device__ __forceinline__ void round_exact(double v, float& f) { f = __double2float_rn(v); }
__device__ __forceinline__ void round_exact(double v, uint16_t& h) { h = __bfloat16_as_ushort(__double2bfloat16(v)); }

__device__ __forceinline__ float4 make_record(const float v[4]) { return make_float4(v[0], v[1], v[2], v[3]); }
__device__ __forceinline__ uint2 make_record(const uint16_t v[4]) {
    return make_uint2((uint32_t)v[0] | ((uint32_t)v[1] << 16), (uint32_t)v[2] | ((uint32_t)v[3] << 16));
}

// One block per brick, as build_store_kernel; V = float or uint16_t (bfloat16 bits).
template <class R, class V>
__global__ void __launch_bounds__(256) build_split_kernel(GridDev g, BuildConst bc, const float* __restrict__ T,
                                                          typename StoreElem<R>::type* __restrict__ store) {
    constexpr int kCells = kHalo * kHalo * kHalo;
    __shared__ float qa[kCells], qb[kCells], qc[kCells];
    __shared__ __align__(32) R rec[kBrickCells];
    const uint32_t b = blockIdx.x, nbx = (uint32_t)g.nb[0], nby = (uint32_t)g.nb[1];
    const int bx = (int)(b % nbx), by = (int)((b / nbx) % nby), bz = (int)(b / (nbx * nby));
    const int ox = bx * kBrick - 1, oy = by * kBrick - 1, oz = bz * kBrick - 1;
    for (int t = threadIdx.x; t < kCells; t += 256) {
        const int hx = t % kHalo, hy = (t / kHalo) % kHalo, hz = t / (kHalo * kHalo);
        const int i = min(max(ox + hx, 0), g.n[0] - 1), j = min(max(oy + hy, 0), g.n[1] - 1),
                  k = min(max(oz + hz, 0), g.n[2] - 1);
        const Split3 q = divide3(bc.K, __ldg(T + ((size_t)k * g.n[1] + j) * g.n[0] + i));
        qa[t] = q.a, qb[t] = q.b, qc[t] = q.c;
    }
    __syncthreads();
    for (int local = threadIdx.x; local < kBrickCells; local += 256) {
        const int lx = local % kBrickSide, ly = (local / kBrickSide) % kBrickSide, lz = local / (kBrickSide * kBrickSide);
        const int c[3] = {min(bx * kBrick + lx, g.n[0] - 1), min(by * kBrick + ly, g.n[1] - 1),
                          min(bz * kBrick + lz, g.n[2] - 1)};
        const int at = ((c[2] - oz) * kHalo + (c[1] - oy)) * kHalo + (c[0] - ox);
        const int step[3] = {1, kHalo, kHalo * kHalo};
        const float de = qa[at];
        V v[4];
        bool sure[4];
        sure[0] = rounds_to(de, __fadd_rn(qb[at], qc[at]), fabsf(de) * 1.4210855e-14f, v[0]);   // 2^-46
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int lo = c[a] > 0 ? at - step[a] : at, hi = c[a] < g.n[a] - 1 ? at + step[a] : at;
            // (selected, not indexed: a per-lane index into the parameters takes the constant-load
            // unit a cycle per thread, which bounded this kernel at 734 us)
            const bool one = c[a] == 0 || c[a] == g.n[a] - 1;   // one-sided
            const float rh = one ? bc.rh[a][1] : bc.rh[a][0], rl = one ? bc.rl[a][1] : bc.rl[a][0],
                        rm = one ? bc.rm[a][1] : bc.rm[a][0];
            const float s0 = __fsub_rn(qa[hi], qa[lo]);        // exact for values within a factor of two
            float s1, e1, p, e;
            two_sum(qb[hi], -qb[lo], s1, e1);
            e1 = __fadd_rn(e1, __fsub_rn(qc[hi], qc[lo]));
            two_sum(s0, s1, p, e);
            e = __fadd_rn(e, e1);
            two_sum(p, e, p, e);                               // difference = p + e
            const float w = __fmul_rn(p, rh);
            const float we = fmaf(p, rl, fmaf(e, rh, fmaf(p, rh, -w)));
            const float big = fmaxf(fabsf(qa[hi]), fabsf(qa[lo]));
            const bool near = big <= 2.0f * fminf(fabsf(qa[hi]), fabsf(qa[lo])) && __fmul_rn(qa[hi], qa[lo]) > 0.0f;
            sure[1 + a] = near && rounds_to(w, we, fmaf(fabsf(w), 5.6843419e-14f, big * rm), v[1 + a]);   // 2^-44
            if (p == 0.0f && e == 0.0f && near) {              // equal temperatures
                v[1 + a] = V(0);
                sure[1 + a] = true;
            }
        }
        if (!(sure[0] && sure[1] && sure[2] && sure[3])) {
            if (!sure[0]) round_exact(deta_at(g, T, c[0], c[1], c[2]), v[0]);
            for (int a = 0; a < 3; ++a) {
                if (sure[1 + a]) continue;
                int lo[3] = {c[0], c[1], c[2]}, hi[3] = {c[0], c[1], c[2]};
                lo[a] = max(c[a] - 1, 0);
                hi[a] = min(c[a] + 1, g.n[a] - 1);
                const double den = hi[a] - lo[a] == 2 ? dmul(2.0, g.h[a]) : g.h[a];
                round_exact(ddiv(dsub(deta_at(g, T, hi[0], hi[1], hi[2]), deta_at(g, T, lo[0], lo[1], lo[2])), den),
                            v[1 + a]);
            }
        }
        rec[local] = make_record(v);
    }
    __syncthreads();
    const uint32_t slot = morton3((uint32_t)bx, (uint32_t)by, (uint32_t)bz);
    for (int local = threadIdx.x; local < kBrickCells; local += 256)
        write_elem(store + (size_t)slot * kBrickCells + local, rec, local, local % kBrickSide < kBrickSide - 1);
}

// ===================================================================== a2-a5: render

struct Sums {
    double I, du, dv, hu, hv;
};

// A ray's float64 set-up values wait in shared memory while it is traced.  Kept in registers
// they cost 12, and the assembler then repeats conversions of them to float32 inside the loop
// to save others: three per step, which held the float64 pipe at 47 % of a render.
constexpr int kRenderThreads = 128;
template <int SLOT>
__device__ __forceinline__ volatile double* ray_park() {
    __shared__ double buf[6 * kRenderThreads];
    return buf + threadIdx.x;
}
__device__ __forceinline__ void park_ray(volatile double* p, const Ray& R) {
    for (int a = 0; a < 3; ++a) p[a * kRenderThreads] = R.d[a];
    p[3 * kRenderThreads] = R.tw;
    p[4 * kRenderThreads] = R.t_in;
    p[5 * kRenderThreads] = R.ell;
}
__device__ __forceinline__ void unpark_ray(volatile double* p, Ray& R) {
    for (int a = 0; a < 3; ++a) R.d[a] = p[a * kRenderThreads];
    R.tw = p[3 * kRenderThreads];
    R.t_in = p[4 * kRenderThreads];
    R.ell = p[5 * kRenderThreads];
}

// Steps of one ray through the cell marcher (QUASI: quasi-linear, else Sharma's), in the scaled
// variables V = dt dv and a = (dt^2 / 6) D (metres per step), so that
//   p2 = S(n+1/2) + dr + V/2 + 3a/4,   p3 = S(n+1) + dr + V + 3b
//   dr += V + a + 2b,                  V += a + 4b + c
// with a, b, c taken at dr, p2 and p3, and every constant exact in float32.  The next step's
// first point and p3 differ by a - b, second order in the step: where that is below the resolution of a float32
// fraction (kSamePoint cells; the usual case, ~1e-9 cells on a half-cell step), the two are
// one point and a' = c, which leaves two field evaluations per step; where it is not (a
// coarse step through a steep field), that lane evaluates a' at its own point.  The path
// excess sum |dS + inc| - |dS| is d.(sum of inc) + sum (|inc|^2 - (d.inc)^2) / (2L + d.inc):
// the first term is the end deviation, so only the small second one is summed.
// Quasi-linear tracing (Sec. 2.2) takes the same weights at the start, middle and end of each
// step on the straight line: the end sample is the next step's start sample.  (Only where nothing
// is kept for an adjoint, see line_run.)
template <class E, bool QUASI>
__device__ __forceinline__ void march_run(const SceneDev& S, const CompField<E>& F, const double rs[3], const Ray& R,
                                          volatile double* park, float dr_end[3], float dv_end[3], float& excess_end,
                                          float& eta_out) {
    MarchLine L;
    MarchCell m;
    const double sl = R.ell / (double)R.N;
    double u0[3], du[3];
    for (int a = 0; a < 3; ++a) {
        u0[a] = (rs[a] + R.t_in * R.d[a] - S.g.origin[a]) * S.g.inv_h[a] - 0.5;
        du[a] = (0.5 * sl) * R.d[a] * S.g.inv_h[a];
    }
    march_line(F.inv_h, u0, du, L, m);
    const P3 d = p3(kept((float)R.d[0]), kept((float)R.d[1]), kept((float)R.d[2]));
    const float near = kSamePoint / fmaxf(F.inv_h[0], fmaxf(F.inv_h[1], F.inv_h[2]));
    const float len2 = kept((float)(2.0 * sl));
    P3 dr = {0.0f, 0ull}, cr = dr, V = dr, cv = dr;
    float excess = 0.0f;
    f32x2 h = 0ull;   // half step, in both halves
    const Cell2 v0 = march_value<true>(F, L, m, h, dr);
    const double eta_in = 1.0 + (double)lo2(v0.lo);
    eta_out = __fadd_rn(1.0f, lo2(v0.lo));
    // dt = (ell / N) / eta_in; dt^2 / 6 scales every acceleration of the ray, so it is rounded
    // once, from float64 (one Newton step on the float32 reciprocal)
    const double ie0 = (double)(1.0f / (float)eta_in), dt = sl * (ie0 * (2.0 - eta_in * ie0));
    const float s = kept((float)(dt * dt * (1.0 / 6.0))), idt = kept(1.0f / (float)dt);
    P3 a = march_accel(v0, s);
    int n = 0;
    while (n < R.N) {
        if (lo2(h) >= 2.0f * kLineSteps) {
            Ray Q;
            unpark_ray(park, Q);
            for (int q = 0; q < 3; ++q) {
                du[q] = (0.5 * (Q.ell / (double)R.N)) * Q.d[q] * S.g.inv_h[q];
                u0[q] = (rs[q] + Q.t_in * Q.d[q] - S.g.origin[q]) * S.g.inv_h[q] - 0.5 + 2.0 * n * du[q];
            }
            march_line(F.inv_h, u0, du, L, m);   // the cell is found again: back to cell 0 first
            h = 0ull;
            Frac3 f;
            march_point<true>(F, L, m, h, dr, f);
        }
        const int n1 = min(R.N, n + kLineSteps);
        for (; n < n1; ++n) {
            h = add2(h, splat2(1.0f));
            if constexpr (QUASI) {
                const P3 b = march_accel(march_value<false, true>(F, L, m, h, dr), s);
                h = add2(h, splat2(1.0f));
                const P3 c = march_accel(march_value<false, true>(F, L, m, h, dr), s);
                const P3 t = fma3(2.0f, b, a);
                const P3 y = add3(t, sub3(V, cr));
                kahan3(dr, cr, y);
                kahan3(V, cv, sub3(add3(fma3(2.0f, b, t), c), cv));
                const float di = dot3(d, y);
                excess = fmaf(fmaf(-di, di, dot3(y, y)), rcp_approx(__fadd_rn(len2, di)), excess);
                a = c;
                continue;
            }
            const P3 b = march_accel(march_value(F, L, m, h, fma3(0.75f, a, fma3(0.5f, V, dr))), s);
            h = add2(h, splat2(1.0f));
            P3 p = fma3(3.0f, b, add3(dr, V));
            const P3 t = fma3(2.0f, b, a);
            const P3 y = add3(t, sub3(V, cr));
            const bool same = maxabs3(sub3(a, b)) <= near;
            kahan3(dr, cr, y);
            P3 c;
#pragma unroll 1
            for (int pass = 0;; ++pass) {
                a = march_accel(march_value(F, L, m, h, p), s);
                if (pass == 0) c = a;
                if (same || pass == 1 || n + 1 == R.N) break;
                p = dr;
            }
            kahan3(V, cv, sub3(add3(fma3(2.0f, b, t), c), cv));
            const float di = dot3(d, y);
            excess = fmaf(fmaf(-di, di, dot3(y, y)), rcp_approx(__fadd_rn(len2, di)), excess);
        }
    }
    const P3 e = sub3(dr, cr), w = mul3(idt, sub3(V, cv));
    dr_end[0] = e.x, dr_end[1] = lo2(e.yz), dr_end[2] = hi2(e.yz);
    dv_end[0] = w.x, dv_end[1] = lo2(w.yz), dv_end[2] = hi2(w.yz);
    excess_end = excess + dot3(d, e);
}

// Sharma steps of one ray with checkpoints, stage by stage on the 32.32 fixed-point line: the
// arithmetic whose result seeds a gradient.  (Where adjoint_kernel recomputes a segment it takes
// comp_step, which agrees with this to rounding.)  Every operation is explicitly rounded (left to the assembler, a product and a sum are fused or not depending
// on the register budget), in packed pairs where three components do the same.  The next
// step's first stage needs only the new position, not C, so it is evaluated beside this
// step's third stage.
//
// The ray keeps its last cell's four paired records and that cell's indices: a point whose line
// position is in the same cell and whose fractions are in [0, 1) takes the records as they
// are, without an address.
//
// What bounds it: instruction issue (57 % of the slots, FMA instructions 33 % of their pipe's) at 16
// warps per SM.  256x256x192 cells, 2048^2 rays with checkpoints: 28.7 ms with an address per point
// and scalar updates, 22.5 ms so (27.1 ms with the address kept and explicit rounding only, 25.6
// without the address, 23.9 with the equal-fractions test, 21.9 with the ray parked, 22.5 with the
// bound on A - C); before that bound 96 registers and 20 warps 24.1 ms, 168 and 12 23.3 ms.  Same
// bits.  With the refracted connection 168 registers are
// best (1.79 ms; 128: 2.08; 96: 2.85; before: 2.11, 128x128x96 cells at 512^2).
struct StageCell {
    int c[3];
    BrickCache bc;
    Cell2 v[4], d[4];      // pairs at o, o + 9, o + 81, o + 90: records and x differences
};

// Fraction of a line position's low words.
__device__ __forceinline__ P3 line_frac(const long long U[3]) {
    auto fr = [](long long u) { return __fsub_rn(__uint_as_float(((uint32_t)u >> 9) | 0x3f800000u), 1.0f); };   // see comp_cell
    return p3(fr(U[0]), fr(U[1]), fr(U[2]));
}

// D = (1 + deta) grad eta at line position U (fractions fr) plus deviation q (LINE: on the line
// itself; q and ih are not looked at).
template <bool LINE = false, class E>
__device__ __forceinline__ P3 stage_rhs(const CompField<E>& F, const long long U[3], P3 fr, P3 ih, P3 q, StageCell& m) {
    P3 u = fr;
    if constexpr (!LINE) u = P3{fmaf(q.x, ih.x, fr.x), fma2(q.yz, ih.yz, fr.yz)};
    float f[3] = {u.x, lo2(u.yz), hi2(u.yz)};
    const int c0 = (int)(U[0] >> 32), c1 = (int)(U[1] >> 32), c2 = (int)(U[2] >> 32);
    const uint32_t top = max(__float_as_uint(f[0]), max(__float_as_uint(f[1]), __float_as_uint(f[2])));
    if (top >= 0x3f800000u || ((c0 ^ m.c[0]) | (c1 ^ m.c[1]) | (c2 ^ m.c[2])) != 0) {
        int ci[3] = {c0, c1, c2};
#pragma unroll
        for (int a = 0; a < 3; ++a) {   // comp_cell's clamping (a no-op inside the grid)
            const float fl = floorf(f[a]);
            const int I = ci[a] + (int)fl;
            ci[a] = min(max(I, 0), F.n[a] - 2);
            f[a] = __fadd_rn(__fsub_rn(f[a], fl), (float)(I - ci[a]));
        }
        if (((ci[0] ^ m.c[0]) | (ci[1] ^ m.c[1]) | (ci[2] ^ m.c[2])) != 0) {
            m.c[0] = ci[0], m.c[1] = ci[1], m.c[2] = ci[2];
            const uint32_t o = comp_offset(F, m.bc, ci);
            load_rec(F.store, o, m.v[0], m.d[0]);
            load_rec(F.store, o + 9, m.v[1], m.d[1]);
            load_rec(F.store, o + 81, m.v[2], m.d[2]);
            load_rec(F.store, o + 90, m.v[3], m.d[3]);
        }
    }
    const f32x2 t0 = splat2(f[0]), t1 = splat2(f[1]), t2 = splat2(f[2]);
    Cell2 a[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) a[i] = Cell2{fma2(t0, m.d[i].lo, m.v[i].lo), fma2(t0, m.d[i].hi, m.v[i].hi)};
    const Cell2 r = lerpc(lerpc(a[0], a[1], t1), lerpc(a[2], a[3], t1), t2);
    const float eta = __fadd_rn(1.0f, lo2(r.lo));
    return P3{__fmul_rn(eta, hi2(r.lo)), mul2(splat2(eta), r.hi)};
}

template <class E>
__device__ __forceinline__ void stage_run(const CompField<E>& F, const Ray& R, const CompConst& k, const CkptDev& ck,
                                          float4* state, long long ray, CompState& st, float* apart_cells) {
    const P3 ih = p3(F.inv_h[0], F.inv_h[1], F.inv_h[2]);
    const P3 d = p3(kept(k.dhat[0]), kept(k.dhat[1]), kept(k.dhat[2]));
    const float dt = kept(k.dt), len2 = kept(2.0f * k.step_len);
    const float h1 = __fmul_rn(0.5f, dt), e1 = __fmul_rn(0.125f, dt);
    long long U[3], dU[3];
    for (int a = 0; a < 3; ++a) {
        U[a] = st.U[a];
        dU[a] = k.dU[a];
        asm volatile("" : "+l"(U[a]), "+l"(dU[a]));   // see kept()
    }
    StageCell m;
    m.c[0] = m.c[1] = m.c[2] = -2;   // no cell
    m.bc = {0xffffffffu, 0u};
    P3 dr = {0.0f, 0ull}, cr = dr, dv = dr, cv = dr;
    float excess = 0.0f, apart = 0.0f, change = 0.0f;   // largest |A - B| and |A - C| of the steps
    P3 A = mul3(dt, stage_rhs(F, U, line_frac(U), ih, dr, m));
    const int K = ck.every;
    int left = K;                        // steps before the next checkpoint
    for (int n = 0; n < R.N; ++n) {
        if (state != nullptr && left == 0) {
            left = K;
            const size_t c = bounded((size_t)(n / K), (size_t)ck.max_ckpt, ck.err);
            state[(c * 3 + 0) * ck.nrays + ray] = make_float4(dr.x, lo2(dr.yz), hi2(dr.yz), cr.x);
            state[(c * 3 + 1) * ck.nrays + ray] = make_float4(dv.x, lo2(dv.yz), hi2(dv.yz), lo2(cr.yz));
            state[(c * 3 + 2) * ck.nrays + ray] = make_float4(cv.x, lo2(cv.yz), hi2(cv.yz), hi2(cr.yz));
        }
        --left;
        long long U2[3];
        for (int a = 0; a < 3; ++a) {
            U2[a] = U[a] + (dU[a] >> 1);
            U[a] += dU[a];
        }
        const P3 B = mul3(dt, stage_rhs(F, U2, line_frac(U2), ih, fma3(e1, A, fma3(h1, dv, dr)), m));
        apart = max_nan(apart, maxabs3(sub3(A, B)));
        const P3 q = fma3(h1, B, fma3(dt, dv, dr));
        const P3 X = fma3(1.0f / 6.0f, fma3(2.0f, B, A), dv);
        const P3 inc = mul3(dt, X);
        const P3 y = P3{fmaf(dt, X.x, -cr.x), fma2(splat2(dt), X.yz, neg2(cr.yz))};
        const P3 fr = line_frac(U);
        const P3 D = stage_rhs(F, U, fr, ih, q, m), C = mul3(dt, D);
        change = max_nan(change, maxabs3(sub3(A, C)));
        kahan3(dr, cr, y);
        // the third stage's point and the new position differ by second order in the step: where
        // their fractions round to the same bits, so does D there
        P3 A1 = {0.0f, 0ull};
        const P3 u1 = P3{fmaf(q.x, ih.x, fr.x), fma2(q.yz, ih.yz, fr.yz)};
        const P3 u2 = P3{fmaf(dr.x, ih.x, fr.x), fma2(dr.yz, ih.yz, fr.yz)};
        if (u1.yz == u2.yz && __float_as_uint(u1.x) == __float_as_uint(u2.x)) A1 = C;
        else if (n + 1 < R.N) A1 = mul3(dt, stage_rhs(F, U, fr, ih, dr, m));
        const P3 s = fma3(dt, D, fma3(4.0f, B, A));
        kahan3(dv, cv, P3{fmaf(s.x, 1.0f / 6.0f, -cv.x), fma2(s.yz, splat2(1.0f / 6.0f), neg2(cv.yz))});
        A = A1;
        // |dS + inc| - |dS|, dS = L d:  d.inc (summed as the end deviation) plus the rest
        const float di = dot3(d, inc);
        excess = fmaf(fmaf(-di, di, dot3(inc, inc)), rcp_approx(__fadd_rn(len2, di)), excess);
    }
    st.dr[0] = dr.x, st.dr[1] = lo2(dr.yz), st.dr[2] = hi2(dr.yz);
    st.cr[0] = cr.x, st.cr[1] = lo2(cr.yz), st.cr[2] = hi2(cr.yz);
    st.dv[0] = dv.x, st.dv[1] = lo2(dv.yz), st.dv[2] = hi2(dv.yz);
    st.cv[0] = cv.x, st.cv[1] = lo2(cv.yz), st.cv[2] = hi2(cv.yz);
    st.excess = __fadd_rn(excess, dot3(d, sub3(dr, cr)));
    if (state != nullptr) {
        // the first checkpoint is the entry state, which is zero: its slot holds the end state
        state[0 * ck.nrays + ray] = make_float4(st.dr[0], st.dr[1], st.dr[2], st.cr[0]);
        state[1 * ck.nrays + ray] = make_float4(st.dv[0], st.dv[1], st.dv[2], st.cr[1]);
        state[2 * ck.nrays + ray] = make_float4(st.cv[0], st.cv[1], st.cv[2], st.cr[2]);
        // steps that the adjoint can reverse without their stage terms (see bos_adjoint.cu): the
        // third stage's point is the new position, dt |A - B| / 6, and the second stage's point may
        // take C for A, dt |A - C| / 24, both within kSameReverse cells (not so: NaN, too).  The one
        // does not bound the other: a layer may lie between a step's middle and its end.
        const float ihm = fmaxf(F.inv_h[0], fmaxf(F.inv_h[1], F.inv_h[2]));
        *apart_cells = max_nan(apart, 0.25f * change) * dt * (ihm * (1.0f / 6.0f));
    }
}

// Quasi-linear steps of one ray whose end state is kept: Sharma's weights, the field at the start,
// middle and end of every step on the line; the end sample is the next step's start sample.
// Stage by stage on the fixed-point line like stage_run, and explicitly rounded for the same
// reason: the luminance is read at a float32 texel coordinate, so an end state an ulp away moves
// the pixels beside one of its steps by 1e-5 of the image, and a residual of one per cent, which
// seeds the gradient, by a few per mille.  What bounds it: instruction issue (60 % of the slots, FMA
// 36 %, L1 24 %) at 16 warps per SM.  Render and adjoint of 256x256x192 cells at 1024 x 768 rays: 14.2 ms with an address and four gathers per pair of steps, 13.3 ms so (12.8 ms marched;
// 168 registers 13.7 ms, 96 13.3 ms).
template <class E>
__device__ __forceinline__ void line_run(const CompField<E>& F, const Ray& R, const CompConst& k, CompState& st) {
    const P3 d = p3(kept(k.dhat[0]), kept(k.dhat[1]), kept(k.dhat[2]));
    const float dt = kept(k.dt), len2 = kept(2.0f * k.step_len);
    long long U[3], dU[3];
    for (int a = 0; a < 3; ++a) {
        U[a] = st.U[a];
        dU[a] = k.dU[a];
        asm volatile("" : "+l"(U[a]), "+l"(dU[a]));   // see kept()
    }
    StageCell m;
    m.c[0] = m.c[1] = m.c[2] = -2;   // no cell
    m.bc = {0xffffffffu, 0u};
    const P3 none = {0.0f, 0ull};
    P3 dr = none, cr = none, dv = none, cv = none;
    float excess = 0.0f;
    P3 A = mul3(dt, stage_rhs<true>(F, U, line_frac(U), none, none, m));
    for (int n = 0; n < R.N; ++n) {
        long long U2[3];
        for (int a = 0; a < 3; ++a) {
            U2[a] = U[a] + (dU[a] >> 1);
            U[a] += dU[a];
        }
        const P3 B = mul3(dt, stage_rhs<true>(F, U2, line_frac(U2), none, none, m));
        const P3 C = mul3(dt, stage_rhs<true>(F, U, line_frac(U), none, none, m));
        const P3 inc = mul3(dt, fma3(1.0f / 6.0f, fma3(2.0f, B, A), dv));
        const P3 s = add3(fma3(4.0f, B, A), C);
        kahan3(dr, cr, sub3(inc, cr));
        kahan3(dv, cv, P3{fmaf(s.x, 1.0f / 6.0f, -cv.x), fma2(s.yz, splat2(1.0f / 6.0f), neg2(cv.yz))});
        A = C;
        const float di = dot3(d, inc);   // as in stage_run
        excess = fmaf(fmaf(-di, di, dot3(inc, inc)), rcp_approx(__fadd_rn(len2, di)), excess);
    }
    st.dr[0] = dr.x, st.dr[1] = lo2(dr.yz), st.dr[2] = hi2(dr.yz);
    st.cr[0] = cr.x, st.cr[1] = lo2(cr.yz), st.cr[2] = hi2(cr.yz);
    st.dv[0] = dv.x, st.dv[1] = lo2(dv.yz), st.dv[2] = hi2(dv.yz);
    st.cv[0] = cv.x, st.cv[1] = lo2(cv.yz), st.cv[2] = hi2(cv.yz);
    st.excess = __fadd_rn(excess, dot3(d, sub3(dr, cr)));
}

// Integrate one ray of the comp path (N > 0) from the pinhole rs stage by stage; Sharma's tracer
// stores its checkpoints every K steps in `state` (slot `ray`) where that is set (renders of the
// classical integrator keep none).  Leaves the end state in st.
template <class E, int INTEG>
__device__ __forceinline__ void comp_run(const SceneDev& S, const CompField<E>& F, const double rs[3], const Ray& R,
                                         const CkptDev& ck, float4* state, long long ray, CompState& st,
                                         double& eta_in, float* apart_cells) {
    CompConst k;
    double rin[3];
    comp_setup(S, F, rs, R, st, k, eta_in, rin);
    if constexpr (INTEG == 0) {
        stage_run(F, R, k, ck, state, ray, st, apart_cells);
    } else if constexpr (INTEG == 2) {
        line_run(F, R, k, st);
    } else {
        BrickCache bc = {0xffffffffu, 0u};
        for (int n = 0; n < R.N; ++n) comp_step<E, INTEG>(F, st, k, bc);
    }
}

__device__ __forceinline__ void comp_end(const CompState& st, float dr[3], float dv[3]) {
    for (int a = 0; a < 3; ++a) {
        dr[a] = st.dr[a] - st.cr[a];
        dv[a] = st.dv[a] - st.cv[a];
    }
}

// End deviation, path excess and entry index of a ray: Sharma and the quasi-linear tracer march
// from cell to cell where nothing is kept for an adjoint; everything else goes stage by stage.
template <class E, int INTEG, bool SAVE>
__device__ __forceinline__ void trace_end(const SceneDev& S, const CompField<E>& F, const double rs[3], Ray& R,
                                          volatile double* park,
                                          const CkptDev& ck, float4* state, long long ray, float dr[3], float dv[3],
                                          float& excess, float& eta, float* apart) {
    if constexpr (INTEG != 1) park_ray(park, R);   // (classical steps have registers to spare)
    if constexpr (INTEG != 1 && !SAVE) {
        march_run<E, INTEG == 2>(S, F, rs, R, park, dr, dv, excess, eta);
    } else {
        CompState st;
        double eta_in;
        comp_run<E, INTEG>(S, F, rs, R, ck, state, ray, st, eta_in, apart);
        eta = (float)eta_in;
        comp_end(st, dr, dv);
        excess = st.excess;
        if (INTEG == 2 && state != nullptr) {   // the end state, from which the adjoint reverses the ray
            state[0 * ck.nrays + ray] = make_float4(dr[0], dr[1], dr[2], excess);
            state[1 * ck.nrays + ray] = make_float4(dv[0], dv[1], dv[2], 0.0f);
        }
    }
    if constexpr (INTEG != 1) unpark_ray(park, R);
}

// Trace one camera ray of the comp path (checkpoints every K steps when ck.state is set).
// With CONN (light mode 2) the luminance is read at the refracted projector connection of
// the wall point x_w = x_ref + dx: M rounds of a <- a + (x_w - y(a)) from a = x_w, y(a) the
// wall hit of the projector ray aimed at a (traced like a camera ray), so that
// a = x_ref + e with e <- dx - (y(a) - (P + t_w d_p)) - ((P + t_w d_p) - a).
template <class E, int INTEG, bool CONN, bool SAVE>
__device__ RayResult trace_comp(const SceneDev& S, const CompField<E>& F, Ray R, const CkptDev& ck,
                                long long ray, bool want_hit, unsigned long long& steps) {
    WallRel h;
    float path = 0.0f, apart = 0.0f;   // path excess; largest stage distance of a step (cells)
    if (R.N > 0) {
        float dr[3], dv[3], excess;
        float eta_in;
        trace_end<E, INTEG, SAVE>(S, F, S.cam.pos, R, ray_park<0>(), ck, ck.state, ray, dr, dv, excess, eta_in, &apart);
        path = excess;
        steps += (unsigned long long)R.N;
        h = comp_wall(S, R, eta_in, dr, dv, excess);
    } else {   // straight camera ray (only with CONN: the projector rays may still bend)
        h.dx[0] = h.dx[1] = h.dx[2] = 0.0f;
        h.cosw = (float)(R.d[0] * S.w.normal[0] + R.d[1] * S.w.normal[1] + R.d[2] * S.w.normal[2]);
        h.len = (float)R.tw;
        h.valid = h.cosw > 0.0f;
    }
    float e[3] = {h.dx[0], h.dx[1], h.dx[2]};
    if constexpr (CONN) {
        if (h.valid) {
            double xref[3];
            for (int a = 0; a < 3; ++a) xref[a] = S.cam.pos[a] + R.tw * R.d[a];
            const double* P = S.L.proj.pos;
            if constexpr (INTEG != 1) park_ray(ray_park<0>(), R);
            for (int m = 0; m < S.L.connect_iters; ++m) {
                Ray Rp = projector_setup(S, xref, e);
                float yrel[3] = {0.0f, 0.0f, 0.0f};
                if (Rp.wall && Rp.N > 0) {
                    float eta_p;
                    float pr[3], pv[3], pexcess, papart = 0.0f;
                    trace_end<E, INTEG, SAVE>(S, F, P, Rp, ray_park<1>(), ck, m == 0 ? ck.pstate : nullptr, ray, pr, pv, pexcess,
                                                    eta_p, &papart);
                    apart = max_nan(apart, papart);
                    steps += (unsigned long long)Rp.N;
                    const WallRel hp = comp_wall(S, Rp, eta_p, pr, pv, 0.0f);
                    if (hp.valid)
                        for (int a = 0; a < 3; ++a) yrel[a] = hp.dx[a];
                }
                if constexpr (INTEG != 1) {
                    unpark_ray(ray_park<0>(), R);
                    for (int a = 0; a < 3; ++a) xref[a] = S.cam.pos[a] + R.tw * R.d[a];
                }
                for (int a = 0; a < 3; ++a) {
                    const double eps = (xref[a] + (double)e[a]) - (P[a] + Rp.tw * Rp.d[a]);
                    e[a] = (h.dx[a] - yrel[a]) + (float)eps;
                }
            }
        }
        if constexpr (INTEG != 1)
            if (h.valid) unpark_ray(ray_park<0>(), R);
        if (ck.conn != nullptr) {   // (a zero cosine factor marks a ray that misses the wall)
            ck.conn[2 * ray] = make_float4(h.dx[0], h.dx[1], h.dx[2], h.valid ? h.cosw / h.len : 0.0f);
            ck.conn[2 * ray + 1] = make_float4(h.dx[0] - e[0], h.dx[1] - e[1], h.dx[2] - e[2], 0.0f);
        }
    }
    // the path record's last bit: whether the adjoint needs the ray's stage terms kept
    if (ck.state != nullptr)
        ck.excess[ray] = __uint_as_float((__float_as_uint(path) & ~1u) | (apart <= kSameReverse ? 0u : 1u));
    return comp_finish(S, R, h, e, want_hit);
}

// Plain FP32 / FP64 tracer.  For the float64 adjoint (T = double, Sharma RKN) the state
// (r, v) is kept every K steps as six doubles, plane q of checkpoint c at
// ((c * 6 + q) * nrays + ray) of ck.state, and the path length of the traced steps per ray
// in ck.excess (as a double).
template <class T, int INTEG>
__device__ RayResult trace_full(const SceneDev& S, const FullField<T>& F, const Ray& R, const CkptDev& ck,
                                long long ray) {
    T r[3], v[3];
    double rin[3];
    double* const save = (sizeof(T) == 8 && INTEG == 0) ? reinterpret_cast<double*>(ck.state) : nullptr;
    for (int a = 0; a < 3; ++a) {
        rin[a] = S.cam.pos[a] + R.t_in * R.d[a];
        r[a] = (T)rin[a];
    }
    T eta_in = F.eta(r);
    for (int a = 0; a < 3; ++a) v[a] = eta_in * (T)R.d[a];
    T dt = (T)R.ell / ((T)R.N * eta_in);
    T lensum = 0;
    const T rl[3] = {r[0], r[1], r[2]}, v0[3] = {v[0], v[1], v[2]};
    for (int n = 0; n < R.N; ++n) {
        if (save != nullptr && n % ck.every == 0) {
            const size_t c = bounded((size_t)(n / ck.every), (size_t)ck.max_ckpt, ck.err);
            for (int q = 0; q < 3; ++q) {
                save[(c * 6 + q) * ck.nrays + ray] = (double)r[q];
                save[(c * 6 + 3 + q) * ck.nrays + ray] = (double)v[q];
            }
        }
        T r0[3] = {r[0], r[1], r[2]};
        if constexpr (INTEG == 2) {
            // quasi-linear: the field on the straight line at the start, middle and end of the step
            T A[3], B[3], C[3], p[3], D[3];
            for (int a = 0; a < 3; ++a) p[a] = rl[a] + ((T)n * dt) * v0[a];
            F.rhs(p, D);
            for (int a = 0; a < 3; ++a) A[a] = dt * D[a];
            for (int a = 0; a < 3; ++a) p[a] = rl[a] + (((T)n + T(0.5)) * dt) * v0[a];
            F.rhs(p, D);
            for (int a = 0; a < 3; ++a) B[a] = dt * D[a];
            for (int a = 0; a < 3; ++a) p[a] = rl[a] + (((T)n + T(1)) * dt) * v0[a];
            F.rhs(p, D);
            for (int a = 0; a < 3; ++a) C[a] = dt * D[a];
            for (int a = 0; a < 3; ++a) {
                r[a] = r[a] + dt * (v[a] + sixth(A[a] + T(2) * B[a]));
                v[a] = v[a] + sixth(A[a] + T(4) * B[a] + C[a]);
            }
        } else {
            full_step<T, INTEG>(F, r, v, dt);
        }
        T d0 = r[0] - r0[0], d1 = r[1] - r0[1], d2 = r[2] - r0[2];
        lensum += sqrt(d0 * d0 + d1 * d1 + d2 * d2);
    }
    if (save != nullptr) reinterpret_cast<double*>(ck.excess)[ray] = (double)lensum;
    double rN[3] = {(double)r[0], (double)r[1], (double)r[2]};
    double vN[3] = {(double)v[0], (double)v[1], (double)v[2]};
    return wall_epilogue(S, S.cam.pos, R, rN, vN, R.t_in + (double)lensum);
}

template <int MODE>   // 0 straight, 1 comp fp32, 2 comp bf16, 3 full fp32, 4 full fp64
struct Tracer;

template <int MODE, int INTEG, bool CONN, bool SAVE>
__device__ __forceinline__ RayResult trace_ray(const SceneDev& S, const Ray& R, const CkptDev& ck, long long ray,
                                               bool want_hit, unsigned long long& steps) {
    if constexpr (MODE == 0) {
        return straight_epilogue(S, R, want_hit);
    } else if constexpr (MODE == 1) {
        const CompField<F4P> F = comp_field<F4P>(S.g);
        return trace_comp<F4P, INTEG, CONN, SAVE>(S, F, R, ck, ray, want_hit, steps);
    } else if constexpr (MODE == 2) {
        const CompField<B4P> F = comp_field<B4P>(S.g);
        return trace_comp<B4P, INTEG, CONN, SAVE>(S, F, R, ck, ray, want_hit, steps);
    } else if constexpr (MODE == 3) {
        FullField<float> F = {S.g};
        steps += (unsigned long long)R.N;
        return trace_full<float, INTEG>(S, F, R, ck, ray);
    } else {
        FullField<double> F = {S.g};
        steps += (unsigned long long)R.N;
        return trace_full<double, INTEG>(S, F, R, ck, ray);
    }
}

// Resident 128-thread blocks per SM that each tracer's register budget is cut for.
#ifndef BOS_FWD_MIN_BLOCKS
#define BOS_FWD_MIN_BLOCKS 6
#endif
#ifndef BOS_FWD_MARCH_MIN_BLOCKS
#define BOS_FWD_MARCH_MIN_BLOCKS 4        // Sharma through the cell marcher (32 polynomial values per ray)
#endif
#ifndef BOS_FWD_STAGE_MIN_BLOCKS
#define BOS_FWD_STAGE_MIN_BLOCKS 4        // Sharma with checkpoints (32 values of the last cell per ray)
#endif
#ifndef BOS_FWD_STAGE_CONN_MIN_BLOCKS
#define BOS_FWD_STAGE_CONN_MIN_BLOCKS 3   // the same with the refracted connection
#endif
#ifndef BOS_FWD_QUASI_MIN_BLOCKS
#define BOS_FWD_QUASI_MIN_BLOCKS 4        // quasi-linear tracing through the cell marcher
#endif
#ifndef BOS_FWD_LINE_MIN_BLOCKS
#define BOS_FWD_LINE_MIN_BLOCKS 4         // quasi-linear tracing whose end state is kept
#endif
#ifndef BOS_FWD_RK4_MIN_BLOCKS
#define BOS_FWD_RK4_MIN_BLOCKS 5          // classical steps on the paired stores (96x96x72 cells, 512^2: 6: 1190 us, 5: 995, 4: 1047)
#endif
#ifndef BOS_FWD_FP64_MIN_BLOCKS
#define BOS_FWD_FP64_MIN_BLOCKS 3         // float64: its pipe is full with a few warps, the cell's polynomial is 64 registers
#endif
constexpr int render_min_blocks(int mode, int integ, bool conn, bool save) {
    return mode == 4 ? BOS_FWD_FP64_MIN_BLOCKS
           : integ == 2 ? (save ? BOS_FWD_LINE_MIN_BLOCKS : BOS_FWD_QUASI_MIN_BLOCKS)
           : mode != 1 && mode != 2 ? BOS_FWD_MIN_BLOCKS
           : integ == 1 ? BOS_FWD_RK4_MIN_BLOCKS
           : save ? (conn ? BOS_FWD_STAGE_CONN_MIN_BLOCKS : BOS_FWD_STAGE_MIN_BLOCKS) : BOS_FWD_MARCH_MIN_BLOCKS;
}
// One warp tile of a render: the rays of its (up to) 32 lanes, averaged per pixel, written
// to the outputs; adds the traced ray-steps to my_steps.
template <int MODE, int INTEG, bool CONN, bool SAVE>
__device__ __forceinline__ void render_tile(const SceneDev& S, const RenderOut& out, const WorkDev& wk,
                                            const CkptDev& ck, const TileShape& ts, int t, int lane,
                                            unsigned long long& my_steps) {
    const int spp = S.cam.spp;
    const int sl = lane % ts.G;
    const TilePix tp = tile_pixel(S, ts, t, lane);
    if (tp.bad) flag_error(wk.err, DEV_BAD_PIXEL);
    const int px = tp.px, py = tp.py;
    const bool valid = tp.valid;
    Sums acc = {0, 0, 0, 0, 0};
    if (valid) {
        for (int q = 0; q < ts.samples_per_lane; ++q) {
            const int s = ts.samples_per_lane == 1 ? sl : q;
            const long long ray = ((long long)t * 32 + lane) * ts.samples_per_lane + q;   // checkpoint slot
            Ray R = ray_setup<MODE != 0>(S, px, py, s);
            if (!R.wall || R.N < 0) {
                if ((MODE == 1 || MODE == 2) && ck.state != nullptr) ck.excess[ray] = 0.0f;
                if (R.wall) flag_error(wk.err, DEV_STEP_BUDGET);
                continue;
            }
            RayResult r;
            if (MODE == 0 || (R.N == 0 && !CONN)) {
                r = straight_epilogue(S, R, out.hit != nullptr);
                if (MODE != 0 && R.N == 0 && ck.state != nullptr) {
                    if (MODE == 4) reinterpret_cast<double*>(ck.excess)[ray] = 0.0;
                    else ck.excess[ray] = 0.0f;
                }
            } else {
                r = trace_ray<MODE, INTEG, CONN, SAVE>(S, R, ck, ray, out.hit != nullptr, my_steps);
            }
            acc.I += r.I;
            acc.du += r.disp[0];
            acc.dv += r.disp[1];
            acc.hu += r.hit[0];
            acc.hv += r.hit[1];
        }
    }
    for (int m = 1; m < ts.G; m <<= 1) {
        acc.I += __shfl_xor_sync(0xffffffffu, acc.I, m);
        acc.du += __shfl_xor_sync(0xffffffffu, acc.du, m);
        acc.dv += __shfl_xor_sync(0xffffffffu, acc.dv, m);
        acc.hu += __shfl_xor_sync(0xffffffffu, acc.hu, m);
        acc.hv += __shfl_xor_sync(0xffffffffu, acc.hv, m);
    }
    if (valid && sl == 0) {
        const size_t p = (size_t)tp.out;
        const double inv = 1.0 / spp;
        out.I[p] = (float)(acc.I * inv);
        if (out.disp) {
            out.disp[2 * p] = (float)(acc.du * inv);
            out.disp[2 * p + 1] = (float)(acc.dv * inv);
        }
        if (out.hit) {
            out.hit[2 * p] = acc.hu * inv;
            out.hit[2 * p + 1] = acc.hv * inv;
        }
    }
}

__device__ __forceinline__ void add_steps(unsigned long long* steps, unsigned long long my_steps, int lane) {
    for (int m = 16; m >= 1; m >>= 1) my_steps += __shfl_xor_sync(0xffffffffu, my_steps, m);
    if (lane == 0 && my_steps) atomicAdd(steps, my_steps);
}

// FEW: the form for launches with few warp tiles (a pixel minibatch), without a register
// cap: the GPU is not full either way, and each ray finishes sooner without spills.
// SAVE (Sharma on the paired stores): with checkpoints; the other tracers look at ck.state.
template <int MODE, int INTEG, bool CONN, bool FEW = false, bool SAVE = true>
__global__ void __launch_bounds__(128, FEW ? 1 : render_min_blocks(MODE, INTEG, CONN, SAVE))
    render_kernel(SceneDev S, RenderOut out, WorkDev wk, CkptDev ck) {
    const TileShape ts = tile_shape(S.cam.width, S.cam.height, S.cam.spp);
    const int ntiles = tile_count(S, ts);
    const int lane = threadIdx.x & 31;
    unsigned long long my_steps = 0;
    for (;;) {
        int t = 0;
        if (lane == 0) t = atomicAdd(wk.tile_counter, 1);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= ntiles) break;
        render_tile<MODE, INTEG, CONN, SAVE>(S, out, wk, ck, ts, t, lane, my_steps);
    }
    add_steps(wk.steps, my_steps, lane);
}

// Batched render: one launch covers warp tiles of several requests' renders (the request
// server's continuous batching).  Work item g belongs to job j with jobs[j].first <= g <
// jobs[j + 1].first and is that job's tile jobs[j].tile0 + (g - jobs[j].first).  Warps
// pull items in order, so the jobs' tiles are interleaved as they are listed.
template <int MODE, int INTEG>
__global__ void __launch_bounds__(128, render_min_blocks(MODE, INTEG, false, false))
    render_batch_kernel(const BatchJob* __restrict__ jobs, int njobs, int total, int* counter) {
    const int lane = threadIdx.x & 31;
    for (;;) {
        int g = 0;
        if (lane == 0) g = atomicAdd(counter, 1);
        g = __shfl_sync(0xffffffffu, g, 0);
        if (g >= total) break;
        const int j = batch_job_of(jobs, njobs, g);
        const BatchJob& J = jobs[j];
        const TileShape ts = tile_shape(J.S.cam.width, J.S.cam.height, J.S.cam.spp);
        unsigned long long my_steps = 0;
        const int t = J.tile0 + (g - J.first);
        if (J.ck.state == nullptr)
            render_tile<MODE, INTEG, false, false>(J.S, J.out, J.wk, J.ck, ts, t, lane, my_steps);
        else
            render_tile<MODE, INTEG, false, true>(J.S, J.out, J.wk, J.ck, ts, t, lane, my_steps);
        add_steps(J.wk.steps, my_steps, lane);
    }
}

// ===================================================================== small kernels

__global__ void ray_steps_kernel(SceneDev S, int32_t* __restrict__ nsteps) {
    const long long nrays = (long long)S.cam.width * S.cam.height * S.cam.spp;
    for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < nrays;
         r += (long long)gridDim.x * blockDim.x) {
        long long pix = r / S.cam.spp;
        int s = (int)(r % S.cam.spp);
        Ray R = ray_setup(S, (int)(pix % S.cam.width), (int)(pix / S.cam.width), s);
        nsteps[r] = R.wall ? R.N : 0;
    }
}

__device__ __forceinline__ float4 node_record(const F4P& p) { return p.v; }
__device__ __forceinline__ uint2 node_record(const B4P& p) { return p.a; }
__device__ __forceinline__ D4 node_record(const D4& p) { return p; }

template <class R>
__global__ void export_nodes_kernel(GridDev g, R* __restrict__ out) {
    using E = typename StoreElem<R>::type;
    const long long n = (long long)g.n[0] * g.n[1] * g.n[2];
    const E* st = static_cast<const E*>(g.store);
    for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x) {
        int i = (int)(c % g.n[0]), j = (int)((c / g.n[0]) % g.n[1]), k = (int)(c / ((long long)g.n[0] * g.n[1]));
        // read node (i, j, k) as a corner of the cell whose base is clamped to n-2
        int bi = min(i, g.n[0] - 2), bj = min(j, g.n[1] - 2), bk = min(k, g.n[2] - 2);
        uint32_t o = brick_offset(bi, bj, bk) + (uint32_t)((k - bk) * 81 + (j - bj) * 9 + (i - bi));
        out[c] = node_record(st[o]);
    }
}

__global__ void loss_l2_kernel(const float* __restrict__ I, const float* __restrict__ target, long long n,
                               double* loss, float* __restrict__ dLdI) {
    double acc = 0.0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const double r = (double)target[i] - (double)I[i];     // exact for two floats
        acc += r * r;
        if (dLdI) dLdI[i] = -2.0f * (target[i] - I[i]);
    }
    for (int m = 16; m >= 1; m >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, m);
    __shared__ double part[32];
    int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) part[w] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += part[i];
        atomicAdd(loss, s);
    }
}

// ===================================================================== measurement probe

// Streams `n4` float4 of an L2-resident buffer `repeats` times (grid-stride, L1 bypassed)
// and folds them into a register; measures the L2 read bandwidth.
__global__ void probe_read_kernel(const float4* __restrict__ buf, long long n4, int repeats, float* sink) {
    float acc = 0.0f;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (int r = 0; r < repeats; ++r)
        for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += stride) {
            float4 v = __ldcg(buf + i);
            acc += (v.x + v.y) + (v.z + v.w);
        }
    if (acc == 1234.5678f) sink[0] = acc;
}

cudaError_t launch_probe_read(const void* buf, long long bytes, int repeats, float* sink, int num_sms,
                              cudaStream_t st) {
    probe_read_kernel<<<num_sms * 8, 256, 0, st>>>((const float4*)buf, bytes / 16, repeats, sink);
    return cudaGetLastError();
}

// ===================================================================== launchers

cudaError_t launch_build_store(const GridDev& g, const float* T, void* store, cudaStream_t st) {
    const unsigned blocks = (unsigned)g.nb[0] * g.nb[1] * g.nb[2];
    if (g.prec == 0) {
        build_store_kernel<<<blocks, 256, 0, st>>>(g, T, (D4*)store);
        return cudaGetLastError();
    }
    BuildConst bc;
    bc.K.a = (float)g.K;
    bc.K.b = (float)(g.K - (double)bc.K.a);
    bc.K.c = (float)((g.K - (double)bc.K.a) - (double)bc.K.b);
    for (int a = 0; a < 3; ++a)
        for (int one = 0; one < 2; ++one) {
            const double r = 1.0 / (one ? g.h[a] : 2.0 * g.h[a]);
            bc.rh[a][one] = (float)r;
            bc.rl[a][one] = (float)(r - (double)bc.rh[a][one]);
            bc.rm[a][one] = (float)(r * 4.4408920985006262e-16 * 1.001);   // 2^-51
        }
    if (g.prec == 3) build_split_kernel<uint2, uint16_t><<<blocks, 256, 0, st>>>(g, bc, T, (B4P*)store);
    else build_split_kernel<float4, float><<<blocks, 256, 0, st>>>(g, bc, T, (F4P*)store);
    return cudaGetLastError();
}

template <int MODE, int INTEG, bool CONN, bool FEW = false, bool SAVE = true>
static cudaError_t launch_render_c(const SceneDev& S, const RenderOut& o, const WorkDev& w, const CkptDev& ck,
                                   int num_sms, cudaStream_t st) {
    int threads = kRenderThreads, per_sm = 0;
    if (MODE == 4) threads = fp64_threads(tile_count(S, tile_shape(S.cam.width, S.cam.height, S.cam.spp)), num_sms, threads);
    cudaError_t e = occupancy_prefer_l1(render_kernel<MODE, INTEG, CONN, FEW, SAVE>, threads, 0, per_sm);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    render_kernel<MODE, INTEG, CONN, FEW, SAVE><<<num_sms * per_sm, threads, 0, st>>>(S, o, w, ck);
    return cudaGetLastError();
}

// The refracted projector connection (light mode 2) has its own instantiation for the
// compensated tracers; the straight reference render and the plain tracers do not use it.
template <int MODE, int INTEG>
static cudaError_t launch_render_t(const SceneDev& S, const RenderOut& o, const WorkDev& w, const CkptDev& ck,
                                   int num_sms, cudaStream_t st) {
    if constexpr (MODE == 1 || MODE == 2) {
        const bool few = tile_count(S, tile_shape(S.cam.width, S.cam.height, S.cam.spp)) <= num_sms * kFewTiles;
        // renders that keep nothing march from cell to cell; where the image seeds a gradient it
        // keeps the stage-by-stage arithmetic on the fixed-point line
        if constexpr (INTEG != 1) {
            if (ck.state == nullptr)
                return S.L.mode == 2 ? launch_render_c<MODE, INTEG, true, false, false>(S, o, w, ck, num_sms, st)
                       : few ? launch_render_c<MODE, INTEG, false, true, false>(S, o, w, ck, num_sms, st)
                             : launch_render_c<MODE, INTEG, false, false, false>(S, o, w, ck, num_sms, st);
        }
        if constexpr (INTEG != 2) {   // (no adjoint of the refracted connection for quasi-linear rays)
            if (S.L.mode == 2) return launch_render_c<MODE, INTEG, true>(S, o, w, ck, num_sms, st);
        }
        // a few tiles (up to 8 warps per SM): the uncapped form
        if constexpr (INTEG != 1) {
            if (few) return launch_render_c<MODE, INTEG, false, true>(S, o, w, ck, num_sms, st);
        }
    }
    return launch_render_c<MODE, INTEG, false>(S, o, w, ck, num_sms, st);
}

cudaError_t launch_render(int mode, const SceneDev& S, const RenderOut& o, const WorkDev& w, const CkptDev& ck,
                          int num_sms, cudaStream_t st) {
    const int integ = S.it.integrator;
#define BOS_CASE(M)                                                                        \
    case M:                                                                                \
        return integ == 1   ? launch_render_t<M, 1>(S, o, w, ck, num_sms, st)              \
               : integ == 2 ? launch_render_t<M, 2>(S, o, w, ck, num_sms, st)              \
                            : launch_render_t<M, 0>(S, o, w, ck, num_sms, st);
    switch (mode) {
        BOS_CASE(0)
        BOS_CASE(1)
        BOS_CASE(2)
        BOS_CASE(3)
        BOS_CASE(4)
        default: return cudaErrorInvalidValue;
    }
#undef BOS_CASE
}

template <int MODE, int INTEG>
static cudaError_t launch_render_batch_c(const BatchJob* jobs, int njobs, int total, int* counter, int num_sms,
                                         cudaStream_t st) {
    int per_sm = 0;
    cudaError_t e = occupancy_prefer_l1(render_batch_kernel<MODE, INTEG>, 128, 0, per_sm);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    render_batch_kernel<MODE, INTEG><<<num_sms * per_sm, 128, 0, st>>>(jobs, njobs, total, counter);
    return cudaGetLastError();
}

cudaError_t launch_render_batch(int mode, int integ, const BatchJob* jobs, int njobs, int total, int* counter,
                                int num_sms, cudaStream_t st) {
    if (mode == 1) return integ == 2 ? launch_render_batch_c<1, 2>(jobs, njobs, total, counter, num_sms, st)
                                     : launch_render_batch_c<1, 0>(jobs, njobs, total, counter, num_sms, st);
    if (mode == 2) return integ == 2 ? launch_render_batch_c<2, 2>(jobs, njobs, total, counter, num_sms, st)
                                     : launch_render_batch_c<2, 0>(jobs, njobs, total, counter, num_sms, st);
    return cudaErrorNotSupported;
}

cudaError_t launch_ray_steps(const SceneDev& S, int32_t* nsteps, int num_sms, cudaStream_t st) {
    ray_steps_kernel<<<num_sms * 8, 256, 0, st>>>(S, nsteps);
    return cudaGetLastError();
}

cudaError_t launch_export_nodes(const GridDev& g, void* out, int num_sms, cudaStream_t st) {
    switch (g.prec) {
        case 0: export_nodes_kernel<D4><<<num_sms * 8, 256, 0, st>>>(g, (D4*)out); break;
        case 3: export_nodes_kernel<uint2><<<num_sms * 8, 256, 0, st>>>(g, (uint2*)out); break;
        default: export_nodes_kernel<float4><<<num_sms * 8, 256, 0, st>>>(g, (float4*)out); break;
    }
    return cudaGetLastError();
}

cudaError_t launch_loss_l2(const float* I, const float* target, long long n, double* loss, float* dLdI, int num_sms,
                           cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(loss, 0, sizeof(double), st);
    if (e != cudaSuccess) return e;
    loss_l2_kernel<<<num_sms * 4, 256, 0, st>>>(I, target, n, loss, dLdI);
    return cudaGetLastError();
}

}  // namespace bos
