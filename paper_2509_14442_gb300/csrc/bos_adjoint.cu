// Adjoint of the BOS forward model (step a6, Sec. 2.4): dL/dT for a given dL/dI.
//
//   reverse_kernel  -- per ray, reverse Sharma's steps from the end state the forward kept,
//                      starting from the adjoint of the wall epilogue (luminance, cosine,
//                      path length of Eq. 2), one field point (value and gradient) and one
//                      scatter per half step.
//   adjoint_kernel  -- the tiles with rays whose steps cannot be reversed that way: each
//                      segment of K steps is recomputed forward from its checkpoint, keeping
//                      the steps' states and stage terms, then reversed stage by stage.
//                      In both, the sensitivities of the 8 trilinear corners are summed per
//                      lane while the ray stays in a cell, and flushed into per-node
//                      accumulators (d L/d deta, d L/d grad eta) with warp-aggregated atomics.
//   gradient_kernel -- per node: the transpose of the central-difference stencil applied
//                      to the grad-eta sensitivities, plus the deta sensitivity, times
//                      d deta/dT = -rho0 G T0 / T^2.  A gather, so it is deterministic.
#include "bos_comp.cuh"
#include "bos_device.cuh"
#include "bos_full.cuh"
#include "bos_internal.h"
#include "bos_march.cuh"

namespace bos {

constexpr int kAdjWarps = kAdjWarpsPerBlock;   // warps per block
#ifndef BOS_ADJ_MIN_BLOCKS
#define BOS_ADJ_MIN_BLOCKS 5              // resident blocks per SM the register budget is cut for
#endif
constexpr int kRow = 36;              // floats per lane row of the cell accumulators (16-byte aligned rows)
constexpr int kConnDoubles = 20;      // per-lane shared doubles of the refracted connection's adjoint
constexpr uint32_t kNoKey = 0xffffffffu;

struct InterpGrad {
    float4 v, d0, d1, d2;   // value and derivatives with respect to the three fractions
};

__device__ __forceinline__ float4 to4(Cell2 c) {
    float4 v;
    unpack2(c.lo, v.x, v.y);
    unpack2(c.hi, v.z, v.w);
    return v;
}

// Value (same operations as `trilinear2`, so bit-identical) and its derivatives with respect
// to the three fractions, in packed f32x2 arithmetic.
template <class E>
__device__ __forceinline__ InterpGrad trilinear_grad2(const E* s, uint32_t o, float f0, float f1, float f2) {
    const f32x2 t0 = pack2(f0, f0), t1 = pack2(f1, f1), t2 = pack2(f2, f2);
    Cell2 a0, a1, a2, a3, e0, e1, e2, e3;   // x-interpolated corner pairs and their x differences
    xlerp(s, o, t0, a0, e0);
    xlerp(s, o + 9, t0, a1, e1);
    xlerp(s, o + 81, t0, a2, e2);
    xlerp(s, o + 90, t0, a3, e3);
    const Cell2 b0 = lerpc(a0, a1, t1), b1 = lerpc(a2, a3, t1);
    InterpGrad r;
    r.v = to4(lerpc(b0, b1, t2));
    r.d2 = to4(csub(b1, b0));
    r.d1 = to4(lerpc(csub(a1, a0), csub(a3, a2), t2));
    r.d0 = to4(lerpc(lerpc(e0, e1, t1), lerpc(e2, e3, t1), t2));
    return r;
}

struct Stage {
    uint32_t key;   // node index of the cell's base corner
    float cf[3];
    InterpGrad ig;
};

template <class E>
__device__ __forceinline__ uint32_t cell_key_of(const CompField<E>& F, const int ci[3]) {
    return (uint32_t)ci[0] + (uint32_t)ci[1] * (uint32_t)F.n[0] + (uint32_t)ci[2] * ((uint32_t)F.n[0] * (uint32_t)F.n[1]);
}

__device__ __forceinline__ void rhs_from(const InterpGrad& ig, float D[3]) {
    float eta = 1.0f + ig.v.x;
    D[0] = eta * ig.v.y;
    D[1] = eta * ig.v.z;
    D[2] = eta * ig.v.w;
}

template <class E>
__device__ __forceinline__ void stage_eval(const CompField<E>& F, const long long U[3], const float q[3], BrickCache& bc,
                                           Stage& s) {
    int ci[3];
    comp_cell(F, U, q, ci, s.cf);
    s.key = cell_key_of(F, ci);
    const uint32_t o = comp_offset(F, bc, ci);
    s.ig = trilinear_grad2(F.store, o, s.cf[0], s.cf[1], s.cf[2]);
}

// Adjoint of D = (1 + deta) grad at a stage point: given Db, the position adjoint (metres)
// and the per-corner record Q (corner c receives w_c Q).
template <class E>
__device__ __forceinline__ void rhs_adjoint(const CompField<E>& F, const InterpGrad& ig, const float Db[3], float pb[3],
                                            float4& Q) {
    const float eta = 1.0f + ig.v.x;
    const float Dg = Db[0] * ig.v.y + Db[1] * ig.v.z + Db[2] * ig.v.w;
    const float4 dv[3] = {ig.d0, ig.d1, ig.d2};
#pragma unroll
    for (int a = 0; a < 3; ++a)
        pb[a] = F.inv_h[a] * (dv[a].x * Dg + eta * (Db[0] * dv[a].y + Db[1] * dv[a].z + Db[2] * dv[a].w));
    Q = make_float4(Dg, eta * Db[0], eta * Db[1], eta * Db[2]);
}

// Per-lane accumulation of corner sensitivities for the lane's current cell; the row
// (8 corners x 4 channels) lives in shared memory.  When a lane's stage point leaves the
// cell, the warp flushes: lanes whose rows belong to the same cell are summed column by
// column (lane l owns corner l/4, channel l%4) and each sum is one atomic.
struct CellAcc {
    uint32_t key;      // node index of the accumulated cell's base corner, kNoKey if empty
    uint32_t ncells;   // nodes of the accumulators (the checked build's bound)
    int* err;
};

__device__ __forceinline__ void flush_rows(float* rows, bool flag, CellAcc& ca, float* acc, int nx, int nxy) {
    unsigned pend = __ballot_sync(0xffffffffu, flag);
    if (!pend) return;
    const int lane = threadIdx.x & 31;
    __syncwarp();
    const int corner = lane >> 2;
    const uint32_t off = (uint32_t)(corner & 1) + (uint32_t)((corner >> 1) & 1) * (uint32_t)nx +
                         (uint32_t)(corner >> 2) * (uint32_t)nxy;
    const uint32_t mykey = flag ? ca.key : kNoKey;
    while (pend) {
        const int leader = __ffs(pend) - 1;
        const uint32_t lk = __shfl_sync(0xffffffffu, mykey, leader);
        const unsigned grp = __ballot_sync(0xffffffffu, mykey == lk);
        pend &= ~grp;
        // column sum over the group's rows, sixteen rows at a time with independent loads
        // and a pairwise tree (warp tiles are coherent, so a group is often the whole warp)
        float sum = 0.0f;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const unsigned part = (grp >> (16 * q)) & 0xffffu;
            if (part) {
                float v[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) v[i] = (part >> i) & 1u ? rows[(16 * q + i) * kRow + lane] : 0.0f;
#pragma unroll
                for (int w = 8; w >= 1; w >>= 1)
#pragma unroll
                    for (int i = 0; i < w; ++i) v[i] += v[i + w];
                sum += v[0];
            }
        }
        if (sum != 0.0f) atomicAdd(acc + ((size_t)bounded(lk + off, ca.ncells, ca.err) << 2) + (lane & 3), sum);
    }
    __syncwarp();
    if (flag) {
        float4* row = reinterpret_cast<float4*>(rows + lane * kRow);
#pragma unroll
        for (int c = 0; c < 8; ++c) row[c] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        ca.key = kNoKey;
    }
    __syncwarp();
}

// Warp-collective: add w_c(cf) Q to the lane's cell row (flushing first where the cell changes).
__device__ __forceinline__ void accumulate(float* rows, bool act, uint32_t cell, const float cf[3], float4 Q,
                                           CellAcc& ca, float* acc, int nx, int nxy) {
    const int lane = threadIdx.x & 31;
    const uint32_t key = act ? cell : kNoKey;
    flush_rows(rows, act && ca.key != kNoKey && ca.key != key, ca, acc, nx, nxy);
    if (act) {
        ca.key = key;
        float4* row = reinterpret_cast<float4*>(rows + lane * kRow);
        const float g0 = 1.0f - cf[0], g1 = 1.0f - cf[1], g2 = 1.0f - cf[2];
        const f32x2 qlo = pack2(Q.x, Q.y), qhi = pack2(Q.z, Q.w);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const float w = ((c & 1) ? cf[0] : g0) * ((c & 2) ? cf[1] : g1) * ((c & 4) ? cf[2] : g2);
            const f32x2 ww = pack2(w, w);
            float4 r = row[c];
            f32x2 lo = fma2(ww, qlo, pack2(r.x, r.y)), hi = fma2(ww, qhi, pack2(r.z, r.w));
            unpack2(lo, r.x, r.y);
            unpack2(hi, r.z, r.w);
            row[c] = r;
        }
    }
}

// Warp-collective: add w_c(cf) Q and, where with2 / with1, w_c(cf2) Q2 and w_c(cf1) Q1 (other
// samples in the same cell) to the lane's cell row, in one read and one write of the row.
__device__ __forceinline__ void accumulate3(float* rows, bool act, uint32_t cell, const float cf[3], float4 Q,
                                            bool with2, const float cf2[3], float4 Q2, bool with1, const float cf1[3],
                                            float4 Q1, CellAcc& ca, float* acc, int nx, int nxy) {
    const int lane = threadIdx.x & 31;
    const uint32_t key = act ? cell : kNoKey;
    flush_rows(rows, act && ca.key != kNoKey && ca.key != key, ca, acc, nx, nxy);
    if (act) {
        ca.key = key;
        float4* row = reinterpret_cast<float4*>(rows + lane * kRow);
        const f32x2 qlo = pack2(Q.x, Q.y), qhi = pack2(Q.z, Q.w);
        const f32x2 q2lo = pack2(Q2.x, Q2.y), q2hi = pack2(Q2.z, Q2.w);
        const f32x2 q1lo = pack2(Q1.x, Q1.y), q1hi = pack2(Q1.z, Q1.w);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const float w = ((c & 1) ? cf[0] : 1.0f - cf[0]) * ((c & 2) ? cf[1] : 1.0f - cf[1]) *
                            ((c & 4) ? cf[2] : 1.0f - cf[2]);
            const float w2 = with2 ? ((c & 1) ? cf2[0] : 1.0f - cf2[0]) * ((c & 2) ? cf2[1] : 1.0f - cf2[1]) *
                                         ((c & 4) ? cf2[2] : 1.0f - cf2[2])
                                   : 0.0f;
            const float w1 = with1 ? ((c & 1) ? cf1[0] : 1.0f - cf1[0]) * ((c & 2) ? cf1[1] : 1.0f - cf1[1]) *
                                         ((c & 4) ? cf1[2] : 1.0f - cf1[2])
                                   : 0.0f;
            float4 r = row[c];
            f32x2 lo = fma2(pack2(w, w), qlo, pack2(r.x, r.y)), hi = fma2(pack2(w, w), qhi, pack2(r.z, r.w));
            lo = fma2(pack2(w2, w2), q2lo, lo);
            hi = fma2(pack2(w2, w2), q2hi, hi);
            lo = fma2(pack2(w1, w1), q1lo, lo);
            hi = fma2(pack2(w1, w1), q1hi, hi);
            unpack2(lo, r.x, r.y);
            unpack2(hi, r.z, r.w);
            row[c] = r;
        }
    }
}

// Adjoint of the wall epilogue for seed Ib = dL/dI of this ray: returns the adjoints of
// (r_N, v_N) and of the path length (which the per-step lengths feed).
// With the refracted projector connection the luminance is read at xl (not at x_w) and
// its sensitivity to x_w arrives as xlb; otherwise xl = xlb = nullptr.
__device__ __forceinline__ void wall_adjoint(const SceneDev& S, const double rN[3], const double vN[3],
                                             double len_before, double Ib, double rb[3], double vb[3],
                                             double& lenb, const double* xl = nullptr, const double* xlb = nullptr) {
    const WallDev& w = S.w;
    rb[0] = rb[1] = rb[2] = vb[0] = vb[1] = vb[2] = 0.0;
    lenb = 0.0;
    double vn = vN[0] * w.normal[0] + vN[1] * w.normal[1] + vN[2] * w.normal[2];
    if (!(vn > 0.0)) return;
    double q[3] = {w.origin[0] - rN[0], w.origin[1] - rN[1], w.origin[2] - rN[2]};
    double ts = (q[0] * w.normal[0] + q[1] * w.normal[1] + q[2] * w.normal[2]) / vn;
    double xw[3];
    for (int a = 0; a < 3; ++a) xw[a] = rN[a] + ts * vN[a];
    double vl = sqrt(vN[0] * vN[0] + vN[1] * vN[1] + vN[2] * vN[2]);
    double len = len_before + ts * vl;              // signed continuation x_w - r_N = t* v
    double cw = vn / vl;
    double gL[3];
    double Lw = xl ? wall_luminance(S.L, w, xl) : wall_luminance(S.L, w, xw, gL);
    double Lb = Ib * cw / len, cb = Ib * Lw / len;
    lenb = -Ib * Lw * cw / (len * len);
    double xwb[3];
    for (int a = 0; a < 3; ++a) {
        double u = vN[a] / vl;                      // d(t* |v|) through x_w = r_N + t* v
        xwb[a] = (xl ? xlb[a] : Lb * gL[a]) + lenb * u;
        rb[a] = -lenb * u;
        vb[a] = cb * (w.normal[a] / vl - vn * vN[a] / (vl * vl * vl));
    }
    double tb = xwb[0] * vN[0] + xwb[1] * vN[1] + xwb[2] * vN[2];
    for (int a = 0; a < 3; ++a) {
        rb[a] += xwb[a] - tb * w.normal[a] / vn;
        vb[a] += ts * xwb[a] - tb * ts * w.normal[a] / vn;
    }
}

// Adjoint of a projector ray's wall hit y = r_N + t* v_N, t* = ((o - r_N) . n) / (v_N . n),
// for the seed yb.
__device__ __forceinline__ void hit_adjoint(const SceneDev& S, const double rN[3], const double vN[3],
                                            const double yb[3], double rb[3], double vb[3]) {
    const WallDev& w = S.w;
    rb[0] = rb[1] = rb[2] = vb[0] = vb[1] = vb[2] = 0.0;
    double vn = vN[0] * w.normal[0] + vN[1] * w.normal[1] + vN[2] * w.normal[2];
    if (!(vn > 0.0)) return;
    double q[3] = {w.origin[0] - rN[0], w.origin[1] - rN[1], w.origin[2] - rN[2]};
    double ts = (q[0] * w.normal[0] + q[1] * w.normal[1] + q[2] * w.normal[2]) / vn;
    double tb = yb[0] * vN[0] + yb[1] * vN[1] + yb[2] * vN[2];
    for (int a = 0; a < 3; ++a) {
        rb[a] = yb[a] - tb * w.normal[a] / vn;
        vb[a] = ts * rb[a];
    }
}

// d/d aim of the straight projector ray's wall hit y = P + t_w d (d = q / |q|,
// t_w = ((o - P) . n) / (d . n)), for the seed yb.
__device__ __forceinline__ void straight_aim_adjoint(const SceneDev& S, const Ray& Rp, double nq, const double yb[3],
                                                     double ab[3]) {
    const WallDev& w = S.w;
    double den = Rp.d[0] * w.normal[0] + Rp.d[1] * w.normal[1] + Rp.d[2] * w.normal[2];
    double twb = yb[0] * Rp.d[0] + yb[1] * Rp.d[1] + yb[2] * Rp.d[2];
    double db[3];
    for (int a = 0; a < 3; ++a) db[a] = Rp.tw * yb[a] - twb * Rp.tw * w.normal[a] / den;
    double dd = db[0] * Rp.d[0] + db[1] * Rp.d[1] + db[2] * Rp.d[2];
    for (int a = 0; a < 3; ++a) ab[a] = (db[a] - dd * Rp.d[a]) / nq;
}

// Refracted projector connection (light mode 2, one aiming round): the luminance is read at
// a_1 = 2 x_w - y(x_w), y the wall hit of the projector ray aimed at x_w.  Sets that ray up,
// its seed ybar = -dL/da_1, |q| of its aim and dL/dx_w's straight part; true where the
// projector ray is traced and has to be reversed.
__device__ __forceinline__ bool connection_seed(const SceneDev& S, const CkptDev& ck, long long slot, const Ray& R,
                                                double Ib, bool act0, Ray& Rp, double* xlum, double* xlb, double* ybar,
                                                double* nqp) {
    for (int a = 0; a < 3; ++a) xlum[a] = xlb[a] = ybar[a] = 0.0;
    nqp[0] = 1.0;
    if (!act0) return false;
    const float4 c0 = ck.conn[2 * slot], c1 = ck.conn[2 * slot + 1];
    const float dxf[3] = {c0.x, c0.y, c0.z};
    double xref[3], gL[3], q[3];
    for (int a = 0; a < 3; ++a) {
        xref[a] = S.cam.pos[a] + R.tw * R.d[a];
        xlum[a] = xref[a] + ((double)dxf[a] - (double)(&c1.x)[a]);
    }
    const double Lb = Ib * (double)c0.w;
    wall_luminance(S.L, S.w, xlum, gL);
    for (int a = 0; a < 3; ++a) {
        ybar[a] = -Lb * gL[a];
        xlb[a] = 2.0 * Lb * gL[a];
        q[a] = (xref[a] - S.L.proj.pos[a]) + (double)dxf[a];
    }
    nqp[0] = sqrt(q[0] * q[0] + q[1] * q[1] + q[2] * q[2]);
    Rp = projector_setup(S, xref, dxf);
    if (!Rp.wall) {                 // y = aim
        for (int a = 0; a < 3; ++a) xlb[a] += ybar[a];
    } else if (Rp.N <= 0) {         // straight projector ray
        double ab[3];
        straight_aim_adjoint(S, Rp, nqp[0], ybar, ab);
        for (int a = 0; a < 3; ++a) xlb[a] += ab[a];
    } else {
        return ybar[0] != 0.0 || ybar[1] != 0.0 || ybar[2] != 0.0;
    }
    return false;
}

// A reversed projector ray's entry state as a function of its aim: r_in = P + t_in d,
// v0 = eta_in d (base of v_N), straight step (ell/N) d, dt = ell / (N eta_in),
// eta_in = 1 + deta(r_in), d = q / |q|, t_in and t_end on slab faces or the wall.  rb, etab,
// dtb: adjoints of r_in, eta_in and dt; ge = grad eta(r_in); drbw, dvbw: of the end state; tpb:
// of the straight step.  Adds dL/d aim to xlb.
__device__ __forceinline__ void aim_adjoint(const SceneDev& S, const Ray& RR, double eta_in, double etab, double dtb,
                                            const double ge[3], const float rb[3], const double* drbw,
                                            const double* dvbw, const double* tpb, double nq, double* xlb) {
    const double Nd = (double)RR.N, ds = RR.ell / Nd;
    double dSb[3], rbi[3], db[3];
    for (int a = 0; a < 3; ++a) {
        dSb[a] = tpb[a] + Nd * drbw[a];
        rbi[a] = (double)rb[a] + etab * ge[a];
        db[a] = eta_in * dvbw[a] + ds * dSb[a] + RR.t_in * rbi[a];
    }
    const double ellb = dtb / (Nd * eta_in) + (RR.d[0] * dSb[0] + RR.d[1] * dSb[1] + RR.d[2] * dSb[2]) / Nd;
    const double tinb = RR.d[0] * rbi[0] + RR.d[1] * rbi[1] + RR.d[2] * rbi[2] - ellb;
    if (RR.in_axis >= 0) db[RR.in_axis] += tinb * (-RR.t_in / RR.d[RR.in_axis]);
    if (RR.out_axis == 3) {
        const double den = RR.d[0] * S.w.normal[0] + RR.d[1] * S.w.normal[1] + RR.d[2] * S.w.normal[2];
        for (int a = 0; a < 3; ++a) db[a] += ellb * (-RR.tw * S.w.normal[a] / den);
    } else {
        const int oa = RR.out_axis;
        db[oa] += ellb * (-(RR.t_in + RR.ell) / RR.d[oa]);
    }
    const double dd = db[0] * RR.d[0] + db[1] * RR.d[1] + db[2] * RR.d[2];
    for (int a = 0; a < 3; ++a) xlb[a] += (db[a] - dd * RR.d[a]) / nq;
}

constexpr size_t kWarpRows = (size_t)32 * kRow;   // shared floats of a warp's lane rows

// Floats per lane and step of the recomputed segment: (dr, dv, A, B) of Sharma's step.
constexpr int kSegFloats = 12;

// ---- reversal without stage terms -----------------------------------------------------------
//
// In the scaled variables V = dt dv, a = (dt^2 / 6) D (see march_run) a Sharma step is
//   r' = r + V + a + 2b,  V' = V + a + 4b + c,  p2 = r + V/2 + 3a/4,  p3 = r + V + 3b
// and solving it backwards gives, exactly,
//   p2 = r' - V'/2 + a/4 + c/2,  r = r' - V' + 2b + c,  V = V' - a - 4b - c.
// p3 and r' differ by b - a, second order in the step.  Where the forward found |b - a| and
// |a - c| / 4 below kSameReverse of a cell for all steps of a ray, c is the acceleration at r' and
// c may stand for a in p2, so the step is reversed from (r', V') alone: no segment
// recompute, no kept stage terms, and the third stage of a step and the first stage of the
// next one are one field point with one evaluation and one scatter.  Per step that is two value
// and gradient evaluations and two scatters, where recomputing the segment and reversing the
// three stages took three evaluations, three more with gradients and three scatters.
// Tiles with a ray for which it does not hold are left to adjoint_kernel.
//
// With r_, V_ the adjoints of (r', V') and the path length's share added to r_ (u = unit step
// direction): a_ = r_ + V_, b_ = 2 r_ + 4 V_, c_ = V_, and with P(w) = (dt^2/6) (dD/dx)^T w
//   q3 = P3(c_), b_ += 3 q3;  q2 = P2(b_), a_ += 3/4 q2;  q1 = P1(a_)
//   V_ += r_ + q3 + q2/2,  r_ += q3 + q2 + q1.
// At the point between two steps both c_ of the earlier and a_ of the later step are known, so
// their sum is scattered once.  All adjoints of a ray are held times s = dt^2/6, so that Q
// needs no scaling and the point adjoints take s from the factor 1/h.

// Corner sensitivities of a lane's current cell, in registers: corner c (x + 2y + 4z).
struct CellRows {
    Cell2 c[8];
};

__device__ __forceinline__ void rows_clear(CellRows& r) {
#pragma unroll
    for (int i = 0; i < 8; ++i) r.c[i] = Cell2{0ull, 0ull};
}

// r += w_c(f) Q
__device__ __forceinline__ void rows_add(CellRows& r, const Frac3& f, Cell2 Q) {
    const f32x2 x = splat2(f.x), y = splat2(f.y), z = splat2(f.z), z1 = splat2(1.0f - f.z);
    Cell2 q[4];
    q[1] = Cell2{mul2(x, Q.lo), mul2(x, Q.hi)};
    q[0] = csub(Q, q[1]);
    q[2] = Cell2{mul2(y, q[0].lo), mul2(y, q[0].hi)};
    q[3] = Cell2{mul2(y, q[1].lo), mul2(y, q[1].hi)};
    q[0] = csub(q[0], q[2]);
    q[1] = csub(q[1], q[3]);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        r.c[i] = cfma(z1, q[i], r.c[i]);
        r.c[4 + i] = cfma(z, q[i], r.c[4 + i]);
    }
}

// 16 bytes of shared memory where `on`, else zero: a predicated load, where a conditional one
// compiles to a branch.
__device__ __forceinline__ Cell2 load_if(uint32_t shared_addr, bool on) {
    Cell2 v;
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\tmov.b64 %0, 0;\n\tmov.b64 %1, 0;\n\t"
        "@p ld.shared.v2.u64 {%0, %1}, [%2];\n\t}"
        : "=l"(v.lo), "=l"(v.hi)
        : "r"(shared_addr), "r"((unsigned)on)
        : "memory");
    return v;
}

// Warp-collective: add the rows of the flagged lanes to the node accumulators, lanes of the
// same cell summed first, and clear them.  The rows go through shared memory; each quarter of
// the warp (8 lanes: one pixel row of the tile) sums the rows of its own lanes, one cell per
// pass, lane l taking corner l % 8 (8 lanes read one row: no bank conflict), and issues one
// 16-byte atomic per corner.
__device__ __forceinline__ void rows_flush(float* rows, bool flag, uint32_t key, CellRows& r, float* acc, int nx, int nxy,
                                           uint32_t ncells, int* err) {
    unsigned pend = __ballot_sync(0xffffffffu, flag);
    if (!pend) return;
    const int lane = threadIdx.x & 31, corner = lane & 7, first = lane & 24;
    const uint32_t off = (uint32_t)(corner & 1) + (uint32_t)((corner >> 1) & 1) * (uint32_t)nx +
                         (uint32_t)(corner >> 2) * (uint32_t)nxy;
    const uint32_t mykey = flag ? key : kNoKey;
    if (flag) {
        ulonglong2* row = reinterpret_cast<ulonglong2*>(rows + lane * kRow);
#pragma unroll
        for (int i = 0; i < 8; ++i) row[i] = make_ulonglong2(r.c[i].lo, r.c[i].hi);
        rows_clear(r);
    }
    __syncwarp();
    const uint32_t src = (uint32_t)__cvta_generic_to_shared(rows + first * kRow + corner * 4);
    do {
        const unsigned mine = (pend >> first) & 0xffu;
        const uint32_t lk = __shfl_sync(0xffffffffu, mykey, mine ? first + __ffs(mine) - 1 : lane);
        const unsigned eq = __ballot_sync(0xffffffffu, mykey == lk) & pend;
        pend &= ~eq;
        const unsigned part = (eq >> first) & mine;
        Cell2 v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = load_if(src + i * (kRow * 4), (part >> i) & 1u);
#pragma unroll
        for (int w = 4; w >= 1; w >>= 1)
#pragma unroll
            for (int i = 0; i < w; ++i) v[i] = Cell2{add2(v[i].lo, v[i + w].lo), add2(v[i].hi, v[i + w].hi)};
        if (part) atomicAdd(reinterpret_cast<float4*>(acc) + bounded(lk + off, ncells, err), to4(v[0]));
    } while (pend);
    __syncwarp();
}

// The same where neighbouring rays share few cells: every flagged lane adds its own rows, eight
// 16-byte atomics that nothing waits for.  Then a quarter's lanes are in several cells, and
// rows_flush takes a pass of dependent shared loads and sums for each.
__device__ __forceinline__ void rows_scatter(bool flag, uint32_t key, CellRows& r, float* acc, int nx, int nxy,
                                             uint32_t ncells, int* err) {
    if (!flag) return;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const uint32_t off = (uint32_t)(c & 1) + (uint32_t)((c >> 1) & 1) * (uint32_t)nx + (uint32_t)(c >> 2) * (uint32_t)nxy;
        atomicAdd(reinterpret_cast<float4*>(acc) + bounded(key + off, ncells, err), to4(r.c[c]));
    }
    rows_clear(r);
}

template <bool SCATTER>
__device__ __forceinline__ void rows_out(float* rows, bool flag, uint32_t key, CellRows& r, float* acc, int nx, int nxy,
                                         uint32_t ncells, int* err) {
    if constexpr (SCATTER) rows_scatter(flag, key, r, acc, nx, nxy, ncells, err);
    else rows_flush(rows, flag, key, r, acc, nx, nxy, ncells, err);
}

// Whether a launch's lanes are sparse enough for that: per cell of the grid's smallest cross
// section at most 12, with the refracted connection (whose two rays visit other cells) at most
// 24.  Whole steps at n lanes per cell, rows_flush -> rows_scatter: 200x200x150 cells, n = 0.7: 1306 ->
// 1075 us; 64x64x48 cells, n = 7: 357 -> 335; a 64^3 minibatch, n = 2.4: 437 -> 390; even at n = 12;
// 200x200x150 cells, n = 19: 9.6 -> 10.0 ms, 40: 19.0 -> 20.7 ms; 24x24x18 cells, n = 83: 204 -> 260 us.
// With the connection the line lies where the first grid turns: 32x32x24 cells, n = 20: 446 -> 432 us,
// 24: 444 -> 439, 28: 444 -> 445, 36: 443 -> 453, 120: 960 -> 1026.  24x24x18 turns at 34 (24: 384 -> 375 us; 80: 380
// -> 428); finer grids would gain beyond it, 64x64x48 at n = 28: 1478 -> 1368 us, 80: 3448 -> 3350,
// 128x128x96 at 22: 6.48 -> 5.81 ms, 45: 12.4 -> 11.4 ms.
__host__ __device__ __forceinline__ bool sparse_lanes(const SceneDev& S, const TileShape& ts, bool conn) {
    const long long nx = S.g.n[0], ny = S.g.n[1], nz = S.g.n[2];
    const long long longest = nx > ny ? (nx > nz ? nx : nz) : (ny > nz ? ny : nz);
    return (long long)tile_count(S, ts) * 32 <= (conn ? 24 : 12) * (nx * ny * nz / longest);
}

// Value and fraction derivatives of the cell polynomial.
struct PolyGrad {
    Cell2 v, x, y, z;
};
__device__ __forceinline__ PolyGrad poly_grad(const CellPoly& p, const Frac3& f) {
    const f32x2 x = splat2(f.x), y = splat2(f.y), z = splat2(f.z);
    const Cell2 e0 = cfma(x, p.c[1], p.c[0]), e1 = cfma(x, p.c[3], p.c[2]);
    const Cell2 e2 = cfma(x, p.c[5], p.c[4]), e3 = cfma(x, p.c[7], p.c[6]);
    PolyGrad g;
    g.z = cfma(y, e3, e2);
    g.v = cfma(z, g.z, cfma(y, e1, e0));
    g.y = cfma(z, e3, e1);
    g.x = cfma(z, cfma(y, p.c[7], p.c[5]), cfma(y, p.c[3], p.c[1]));
    return g;
}

template <bool VALUE_ONLY>
__device__ __forceinline__ PolyGrad poly_point(const CellPoly& p, const Frac3& f) {
    if constexpr (!VALUE_ONLY) return poly_grad(p, f);
    PolyGrad g = {};
    g.v = poly_value(p, splat2(f.x), splat2(f.y), splat2(f.z));
    return g;
}

// The marcher's line of a ray with step 0 at its step `origin`.
template <class E>
__device__ __forceinline__ void set_line(const SceneDev& S, const CompField<E>& F, const double rs[3], const Ray& R,
                                         int origin, MarchLine& L, MarchCell& m) {
    const double half = 0.5 * (R.ell / (double)R.N);
    double u0[3], du[3];
    for (int a = 0; a < 3; ++a) {
        du[a] = half * R.d[a] * S.g.inv_h[a];
        u0[a] = (rs[a] + R.t_in * R.d[a] - S.g.origin[a]) * S.g.inv_h[a] - 0.5 + 2.0 * (double)origin * du[a];
    }
    march_line(F.inv_h, u0, du, L, m);
}

// (dD/d record)^T w: the record adjoint Q that the corners share.
__device__ __forceinline__ Cell2 record_adjoint(const PolyGrad& g, float eta, P3 w) {
    const f32x2 t = mul2(w.yz, g.v.hi);
    return Cell2{pack2(fmaf(w.x, hi2(g.v.lo), __fadd_rn(lo2(t), hi2(t))), eta * w.x), mul2(splat2(eta), w.yz)};
}

// s (d record / dx)^T Q, ih = s / h
__device__ __forceinline__ P3 point_adjoint(const PolyGrad& g, Cell2 Q, P3 ih) {
    const f32x2 a = fma2(g.x.hi, Q.hi, mul2(g.x.lo, Q.lo)), b = fma2(g.y.hi, Q.hi, mul2(g.y.lo, Q.lo)),
                c = fma2(g.z.hi, Q.hi, mul2(g.z.lo, Q.lo));
    return P3{ih.x * (lo2(a) + hi2(a)), mul2(ih.yz, pack2(lo2(b) + hi2(b), lo2(c) + hi2(c)))};
}

// Node index of a cell's base corner from its biased float indices.
__device__ __forceinline__ uint32_t march_key(const MarchCell& m, uint32_t nx, uint32_t nxy) {
    return (__float_as_uint(m.ci.x) & 0x7fffffu) + (__float_as_uint(lo2(m.ci.yz)) & 0x7fffffu) * nx +
           (__float_as_uint(hi2(m.ci.yz)) & 0x7fffffu) * nxy;
}

// A ray of the tile has steps that cannot be reversed without their stage terms (the last bit
// of its path record; every ray of the image has one).
__device__ __forceinline__ bool tile_needs_stages(const CkptDev& ck, const TileShape& ts, int t, int lane, bool valid) {
    bool strong = false;
    for (int q = 0; q < ts.samples_per_lane; ++q)
        if (valid) strong |= (__float_as_uint(ck.excess[((long long)t * 32 + lane) * ts.samples_per_lane + q]) & 1u) != 0u;
    return __any_sync(0xffffffffu, strong);
}

// One warp tile of the adjoint by reversal.  Rows are empty on entry and on return.  QUASI: the
// quasi-linear tracer, whose points lie on the straight line: the same recurrences for V and
// the adjoints without the point adjoints (its outputs are linear in the sampled values), for
// every ray.
template <class E, bool CONN, bool QUASI, bool SCATTER>
__device__ __forceinline__ void reverse_tile(const SceneDev& S, const CkptDev& ck, const AdjDev& adj,
                                             const CompField<E>& F, const TileShape& ts, int t, int lane, float* rows,
                                             float* acc, uint32_t ncells, int* err, int* deferred, double* xlum) {
    const int nx = S.g.n[0], nxy = S.g.n[0] * S.g.n[1];
    const int spp = S.cam.spp;
    double* const xlb = xlum + 3;
    double* const ybar = xlum + 6;
    double* const drbw = xlum + 9;
    double* const dvbw = xlum + 12;
    double* const tpb = xlum + 15;
    double* const nqp = xlum + 18;
    const TilePix tp = tile_pixel(S, ts, t, lane);
    if (!QUASI && tile_needs_stages(ck, ts, t, lane, tp.valid)) {
        if (lane == 0) atomicAdd(deferred, 1);
        return;
    }
    for (int qs = 0; qs < ts.samples_per_lane; ++qs) {
        const int s = ts.samples_per_lane == 1 ? lane % ts.G : qs;
        const long long slot = ((long long)t * 32 + lane) * ts.samples_per_lane + qs;
        Ray R;
        R.N = 0;
        R.wall = false;
        double Ib = 0.0;
        if (tp.valid) {
            R = ray_setup(S, tp.px, tp.py, s);
            Ib = (double)adj.dLdI[(size_t)tp.out] / spp;
        }
        const bool act0 = tp.valid && R.wall && R.N >= 0 && Ib != 0.0;
        Ray Rp;
        Rp.N = 0;
        Rp.wall = false;
        bool pact = false;
        if constexpr (CONN) pact = connection_seed(S, ck, slot, R, Ib, act0, Rp, xlum, xlb, ybar, nqp);
        for (int pass = CONN ? 0 : 1; pass < 2; ++pass) {
            const bool proj = CONN && pass == 0;
            const Ray& RR = proj ? Rp : R;
            const double* rs = proj ? S.L.proj.pos : S.cam.pos;
            const float4* cstate = proj ? ck.pstate : ck.state;
            const bool act = proj ? pact : (act0 && R.N > 0);
            const int N = act ? RR.N : -1;
            const int n_max = (int)__reduce_max_sync(0xffffffffu, (unsigned)(N + 1)) - 1;
            if (n_max < 0) continue;
            MarchLine L;
            MarchCell m;
            P3 dr = {0.0f, 0ull}, V = dr, rb = dr, Vb = dr, dS = dr, sih = dr;
            float sc = 0.0f, lenb = 0.0f, dt = 0.0f;
            double eta_in = 1.0, etab = 0.0;
            uint32_t key = 0u;                // node of the cell's base corner
            bool far_off = false;
            if (act) {
                const double sl = RR.ell / (double)RR.N;
                double rin[3];
                for (int a = 0; a < 3; ++a) rin[a] = rs[a] + RR.t_in * RR.d[a];
                set_line(S, F, rs, RR, 0, L, m);
                Frac3 f;
                march_point<true>(F, L, m, 0ull, dr, f);
                key = march_key(m, (uint32_t)nx, (uint32_t)nxy);
                eta_in = 1.0 + (double)lo2(poly_value(m.p, splat2(f.x), splat2(f.y), splat2(f.z)).lo);
                const double ie0 = (double)(1.0f / (float)eta_in), dtd = sl * (ie0 * (2.0 - eta_in * ie0));
                dt = kept((float)dtd);
                sc = kept((float)(dtd * dtd * (1.0 / 6.0)));
                dS = p3(kept((float)(sl * RR.d[0])), kept((float)(sl * RR.d[1])), kept((float)(sl * RR.d[2])));
                const float4 s0 = cstate[slot], s1 = cstate[ck.nrays + slot];
                float4 s2 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if (!QUASI) s2 = cstate[2 * ck.nrays + slot];
                // (quasi-linear tracing keeps its end state uncompensated, with the path excess)
                const float er[3] = {s0.x - (QUASI ? 0.0f : s0.w), s0.y - (QUASI ? 0.0f : s1.w),
                                     s0.z - s2.w};
                const float ev[3] = {s1.x - s2.x, s1.y - s2.y, s1.z - s2.z};
                double rN[3], vN[3], drb[3], dvb[3], lb = 0.0;
                for (int a = 0; a < 3; ++a) {
                    rN[a] = rin[a] + RR.ell * RR.d[a] + (double)er[a];
                    vN[a] = eta_in * RR.d[a] + (double)ev[a];
                }
                if (proj) {
                    hit_adjoint(S, rN, vN, ybar, drb, dvb);
                    for (int a = 0; a < 3; ++a) {
                        drbw[a] = drb[a];
                        dvbw[a] = dvb[a];
                        tpb[a] = 0.0;
                    }
                } else {
                    const double len_before = R.t_in + R.ell + (double)(QUASI ? s0.w : ck.excess[slot]);
                    wall_adjoint(S, rN, vN, len_before, Ib, drb, dvb, lb, CONN ? xlum : nullptr, CONN ? xlb : nullptr);
                }
                lenb = kept((float)lb) * sc;
                // eta_in's adjoint through v0 and (below) dt = ell / (N eta_in); dv_N = V_N / dt
                etab = dvb[0] * RR.d[0] + dvb[1] * RR.d[1] + dvb[2] * RR.d[2] +
                       (dvb[0] * (double)ev[0] + dvb[1] * (double)ev[1] + dvb[2] * (double)ev[2]) / eta_in;
                const float idt = 1.0f / dt;
                dr = p3(er[0], er[1], er[2]);
                V = mul3(dt, p3(ev[0], ev[1], ev[2]));
                rb = p3(kept(sc * (float)drb[0]), kept(sc * (float)drb[1]), kept(sc * (float)drb[2]));
                const float si = sc * idt;
                Vb = p3(kept((float)dvb[0] * si), kept((float)dvb[1] * si), kept((float)dvb[2] * si));
                sih = mul3(sc, L.ih);
                if (QUASI) dr = P3{0.0f, 0ull};
                far_off = !QUASI && !(maxabs3(P3{dr.x * L.ih.x, mul2(dr.yz, L.ih.yz)}) <= 0.0625f);
            }
            // A ray that ends more than a sixteenth of a cell off its line takes its state from
            // the checkpoints where there is one: its deviation's rounding, 2^-29 of a cell and
            // less otherwise, would build up over the steps.
            const bool resync = __any_sync(0xffffffffu, far_off);
            const int K = ck.every;
            int to_ckpt = n_max % K;          // node n_max - to_ckpt is the next checkpointed one
            CellRows row;
            rows_clear(row);
            P3 ab = {0.0f, 0ull};             // a_ of the later step, waiting for its point
            float work = 0.0f;                // sum of a_.a + b_.b + c_.c
            const P3 VbN = Vb;
            P3 ulen = {0.0f, 0ull};           // quasi-linear: lenb times the unit directions so far
            float tps[3] = {0.0f, 0.0f, 0.0f};
            P3 rseg = rb;
            int seg0 = n_max - to_ckpt;       // first node of the segment (the refracted sums)
            int origin = n_max / kLineSteps * kLineSteps;   // the step that the line is set up from
            if (origin > 0 && act) {
                set_line(S, F, rs, RR, origin, L, m);
                march_leave(m);
            }
            f32x2 h = splat2(2.0f * (float)(n_max - origin));
            bool used = false;                // the rows hold something
            bool later = false;               // a later step of this ray has been reversed
            for (int n = n_max;; --n, --to_ckpt) {
                const bool on = n <= N;
                if (n < origin) {
                    origin -= kLineSteps;
                    if (act) {
                        set_line(S, F, rs, RR, origin, L, m);
                        march_leave(m);
                    }
                    h = splat2(2.0f * (float)(n - origin));
                }
                // ---- the point between steps n - 1 and n
                P3 c = {0.0f, 0ull}, q3 = c;
                Frac3 f;
                bool moved = false;
                bool kept_state = false;
                P3 Vk = c;
                if (on) {
                    if (resync && to_ckpt == 0 && n < N && n > 0) {
                        const size_t cc = bounded((size_t)(n / K), (size_t)ck.max_ckpt, ck.err);
                        const float4 s0 = cstate[(cc * 3 + 0) * ck.nrays + slot];
                        const float4 s1 = cstate[(cc * 3 + 1) * ck.nrays + slot];
                        const float4 s2 = cstate[(cc * 3 + 2) * ck.nrays + slot];
                        dr = p3(s0.x - s0.w, s0.y - s1.w, s0.z - s2.w);
                        Vk = mul3(dt, p3(s1.x - s2.x, s1.y - s2.y, s1.z - s2.z));
                        kept_state = true;
                    }
                    moved = march_point<false, QUASI>(F, L, m, h, dr, f);
                }
                if (__any_sync(0xffffffffu, moved)) {
                    rows_out<SCATTER>(rows, moved && used, key, row, acc, nx, nxy, ncells, err);
                    if (moved) key = march_key(m, (uint32_t)nx, (uint32_t)nxy);
                }
                if (on) {
                    const PolyGrad g = poly_point<QUASI>(m.p, f);
                    const float eta = 1.0f + lo2(g.v.lo);
                    c = march_accel(g.v, sc);
                    if (later) V = kept_state ? Vk : sub3(V, c);
                    P3 w = ab;
                    if (n > 0) {
                        w = add3(w, Vb);
                        if (!QUASI) q3 = point_adjoint(g, record_adjoint(g, eta, Vb), sih);
                    }
                    Cell2 Q = record_adjoint(g, eta, w);
                    work = fmaf(eta, lo2(Q.lo), work);
                    P3 q = {0.0f, 0ull};
                    if (!QUASI) {
                        q = point_adjoint(g, Q, sih);
                        rb = add3(rb, sub3(q, q3));
                    }
                    if constexpr (CONN) {
                        const float tn = (float)(n - seg0);
                        const P3 q1 = sub3(q, q3);
                        tps[0] += tn * q1.x, tps[1] += tn * lo2(q1.yz), tps[2] += tn * hi2(q1.yz);
                    }
                    if (n == 0) {
                        // entry: v0 = eta_in d and dt = ell / (N eta_in), eta_in = 1 + deta(r_in);
                        // a, b and c carry dt^2, so dL/d dt = 2 work / dt (- dv_N . dL/d v_N / dt, above)
                        etab -= 2.0 * (double)work / eta_in;
                        Q.lo = pack2(lo2(Q.lo) + (float)etab, hi2(Q.lo));
                    }
                    rows_add(row, f, Q);
                    used = true;
                }
                if constexpr (CONN) {
                    if (proj && on && to_ckpt == 0) {
                        const P3 e = sub3(rb, rseg);
                        const float ee[3] = {e.x, lo2(e.yz), hi2(e.yz)};
                        for (int a = 0; a < 3; ++a) {
                            tpb[a] += ((double)tps[a] + (double)seg0 * (double)ee[a]) / (double)sc;
                            tps[a] = 0.0f;
                        }
                        rseg = rb;
                    }
                }
                if (to_ckpt == 0) {
                    to_ckpt = K;
                    seg0 -= K;
                }
                if (n == 0) break;
                // ---- the middle of step n - 1
                h = add2(h, splat2(-1.0f));
                moved = false;
                if (on) moved = march_point<false, QUASI>(F, L, m, h, QUASI ? dr : fma3(0.75f, c, fma3(-0.5f, V, dr)), f);
                if (__any_sync(0xffffffffu, moved)) {
                    rows_out<SCATTER>(rows, moved && used, key, row, acc, nx, nxy, ncells, err);
                    if (moved) key = march_key(m, (uint32_t)nx, (uint32_t)nxy);
                }
                if (on) {
                    const PolyGrad g = poly_point<QUASI>(m.p, f);
                    const float eta = 1.0f + lo2(g.v.lo);
                    const P3 b = march_accel(g.v, sc);
                    const P3 inc = sub3(V, fma3(2.0f, b, c));          // r' - r
                    if (!QUASI) dr = sub3(dr, inc);
                    V = sub3(V, fma3(4.0f, b, c));                     // less a, at the next point
                    const P3 step = add3(dS, inc);
                    const float ln = lenb * rsqrtf(dot3(step, step));
                    const P3 sg = fma3(ln, step, rb);                  // r_ with the path length's share
                    P3 bb = mul3(4.0f, Vb), q2 = {0.0f, 0ull};
                    if (!QUASI) bb = fma3(3.0f, q3, bb);
                    bb = fma3(2.0f, sg, bb);
                    const Cell2 Q = record_adjoint(g, eta, bb);
                    work = fmaf(eta, lo2(Q.lo), work);
                    rows_add(row, f, Q);
                    ab = add3(sg, Vb);
                    if (QUASI) {
                        // r_ is constant: V_ from its closed form, whose float32 error does not
                        // build up over the steps (their number from the integers: a float that
                        // counts them stops at 2^24)
                        ulen = fma3(ln, step, ulen);
                        Vb = add3(fma3((float)(N - n + 1), rb, VbN), ulen);
                    } else {
                        Vb = add3(Vb, sg);
                    }
                    if (!QUASI) {
                        q2 = point_adjoint(g, Q, sih);
                        rb = add3(rb, add3(q3, q2));
                        ab = fma3(0.75f, q2, ab);
                        Vb = add3(Vb, fma3(0.5f, q2, q3));
                    }
                    later = true;
                    if constexpr (CONN) {
                        const P3 t = fma3((float)(n - seg0), q3, mul3((float)(n - seg0) - 0.5f, q2));
                        tps[0] += t.x, tps[1] += lo2(t.yz), tps[2] += hi2(t.yz);
                    }
                }
                h = add2(h, splat2(-1.0f));
            }
            rows_out<SCATTER>(rows, used, key, row, acc, nx, nxy, ncells, err);
            if constexpr (CONN) {
                if (proj && act) {
                    Frac3 f;
                    march_point<false>(F, L, m, 0ull, P3{0.0f, 0ull}, f);
                    const PolyGrad g = poly_grad(m.p, f);
                    const double ge[3] = {(double)lo2(g.x.lo) * (double)F.inv_h[0], (double)lo2(g.y.lo) * (double)F.inv_h[1],
                                          (double)lo2(g.z.lo) * (double)F.inv_h[2]};
                    // etab = dvb . d - dtb dt / eta_in
                    const double dtb = (dvbw[0] * RR.d[0] + dvbw[1] * RR.d[1] + dvbw[2] * RR.d[2] - etab) * eta_in /
                                       (double)dt;
                    const float rbf[3] = {rb.x / sc, lo2(rb.yz) / sc, hi2(rb.yz) / sc};
                    aim_adjoint(S, RR, eta_in, etab, dtb, ge, rbf, drbw, dvbw, tpb, nqp[0], xlb);
                }
            }
        }   // passes
    }
}

// One warp tile of the Sharma adjoint: reverse every ray of the tile from its checkpoints
// and scatter its sensitivities into the lane rows (flushed into acc as the cells change).
template <class E, bool CONN>
__device__ __forceinline__ void adjoint_tile(const SceneDev& S, const CkptDev& ck, const AdjDev& adj,
                                             const CompField<E>& F, const TileShape& ts, int t, int lane,
                                             float* rows, float* st_buf, float* acc, CellAcc& ca, double* xlum) {
    const int nx = S.g.n[0], nxy = S.g.n[0] * S.g.n[1];
    const int spp = S.cam.spp;
    const int K = ck.every;
    double* const xlb = xlum + 3;
    double* const ybar = xlum + 6;
    double* const drbw = xlum + 9;
    double* const dvbw = xlum + 12;
    double* const tpb = xlum + 15;
    double* const nqp = xlum + 18;
    const int sl = lane % ts.G;
    const TilePix tp = tile_pixel(S, ts, t, lane);
    const int px = tp.px, py = tp.py;
    const bool valid = tp.valid;
    for (int qs = 0; qs < ts.samples_per_lane; ++qs) {
        const int s = ts.samples_per_lane == 1 ? sl : qs;
        const long long slot = ((long long)t * 32 + lane) * ts.samples_per_lane + qs;
        bool act = valid;
        Ray R;
        R.N = 0;
        R.wall = false;
        double Ib = 0.0;
        if (act) {
            R = ray_setup(S, px, py, s);
            Ib = (double)adj.dLdI[(size_t)tp.out] / spp;
        }
        const bool act0 = act && R.wall && R.N >= 0 && Ib != 0.0;
        // Refracted projector connection (light mode 2, one aiming round): the luminance is
        // read at a_1 = 2 x_w - y(x_w), y the wall hit of the projector ray aimed at x_w.
        // Pass 0 reverses that projector ray for the seed -dL/da_1 and turns its entry state
        // into dL/d aim; pass 1 reverses the camera ray with dL/dx_w = 2 dL/da_1 + dL/d aim.
        Ray Rp;
        Rp.N = 0;
        Rp.wall = false;
        bool pact = false;
        if constexpr (CONN) {
            pact = connection_seed(S, ck, slot, R, Ib, act0, Rp, xlum, xlb, ybar, nqp);
        }
        for (int pass = CONN ? 0 : 1; pass < 2; ++pass) {
        const bool proj = CONN && pass == 0;
        const Ray& RR = proj ? Rp : R;
        const double* rs = proj ? S.L.proj.pos : S.cam.pos;
        const float4* cstate = proj ? ck.pstate : ck.state;
        act = proj ? pact : (act0 && R.N > 0);
        CompState st0;
        CompConst k;
        double eta_in = 1.0, rin[3] = {0, 0, 0};
        if (act) comp_setup(S, F, rs, RR, st0, k, eta_in, rin);
        const int N = act ? RR.N : 0;
        const int nseg = (N + K - 1) / K;
        const int nseg_max = __reduce_max_sync(0xffffffffu, (unsigned)nseg);
        float rb[3] = {0, 0, 0}, vb[3] = {0, 0, 0}, dtb = 0.0f, lenb = 0.0f;
        double etab = 0.0;
        if constexpr (CONN)
            for (int a = 0; a < 3; ++a) tpb[a] = 0.0;
        const float dt = act ? k.dt : 0.0f;
        BrickCache bc = {kNoKey, 0u};
        for (int c = nseg_max - 1; c >= 0; --c) {
            const int n0 = c * K;
            const int n1 = min(n0 + K, N);
            const bool seg = act && n0 < N;
            // ---- recompute the segment from its checkpoint, keeping each step's state
            if (seg) {
                CompState st;
                const size_t cc = bounded((size_t)c, (size_t)ck.max_ckpt, ck.err);
                float4 s0 = make_float4(0.0f, 0.0f, 0.0f, 0.0f), s1 = s0, s2 = s0;   // the entry state
                if (c > 0) {
                    s0 = cstate[(cc * 3 + 0) * ck.nrays + slot];
                    s1 = cstate[(cc * 3 + 1) * ck.nrays + slot];
                    s2 = cstate[(cc * 3 + 2) * ck.nrays + slot];
                }
                st.dr[0] = s0.x; st.dr[1] = s0.y; st.dr[2] = s0.z;
                st.dv[0] = s1.x; st.dv[1] = s1.y; st.dv[2] = s1.z;
                st.cv[0] = s2.x; st.cv[1] = s2.y; st.cv[2] = s2.z;
                st.cr[0] = s0.w; st.cr[1] = s1.w; st.cr[2] = s2.w;
                st.excess = 0.0f;
                for (int a = 0; a < 3; ++a) st.U[a] = st0.U[a] + (long long)n0 * k.dU[a];
                for (int n = n0; n < n1; ++n) {
                    float* p = st_buf + (size_t)(n - n0) * kSegFloats * 32 + lane;
                    p[0] = st.dr[0]; p[32] = st.dr[1]; p[64] = st.dr[2];
                    p[96] = st.dv[0]; p[128] = st.dv[1]; p[160] = st.dv[2];
                    float AB[6];
                    comp_step<E, 0>(F, st, k, bc, AB);
                    for (int q = 0; q < 6; ++q) p[192 + 32 * q] = AB[q];
                }
                if (c == nseg - 1) {
                    // the lane's last segment: start from the adjoint of the wall epilogue
                    double rN[3], vN[3], drb[3], dvb[3], lb = 0.0;
                    for (int a = 0; a < 3; ++a) {
                        rN[a] = rin[a] + RR.ell * RR.d[a] + ((double)st.dr[a] - (double)st.cr[a]);
                        vN[a] = eta_in * RR.d[a] + ((double)st.dv[a] - (double)st.cv[a]);
                    }
                    if (proj) {
                        hit_adjoint(S, rN, vN, ybar, drb, dvb);
                        for (int a = 0; a < 3; ++a) {
                            drbw[a] = drb[a];
                            dvbw[a] = dvb[a];
                        }
                    } else {
                        double len_before = R.t_in + R.ell + (double)ck.excess[slot];
                        wall_adjoint(S, rN, vN, len_before, Ib, drb, dvb, lb, CONN ? xlum : nullptr,
                                     CONN ? xlb : nullptr);
                    }
                    for (int a = 0; a < 3; ++a) {
                        rb[a] = (float)drb[a];
                        vb[a] = (float)dvb[a];
                    }
                    lenb = (float)lb;
                    etab += dvb[0] * RR.d[0] + dvb[1] * RR.d[1] + dvb[2] * RR.d[2];
                }
            }
            __syncwarp();
            const float rseg[3] = {rb[0], rb[1], rb[2]};   // rb before this segment's steps
            // ---- reverse the segment's steps
            const int n_hi = __reduce_max_sync(0xffffffffu, (unsigned)(seg ? n1 : 0));
            float tps[3] = {0.0f, 0.0f, 0.0f};   // sum over the segment's stages of (t / dt_step) pb
            for (int n = n_hi - 1; n >= n0; --n) {
                const bool a_ = seg && n < n1;
                // the step's state and stage terms from the recompute: all three stage
                // points are known, so each stage is evaluated (value and gradient) when
                // its adjoint is formed, in the order 3, 2, 1
                float dr[3] = {0, 0, 0}, dvv[3] = {0, 0, 0}, A[3] = {0, 0, 0}, B[3] = {0, 0, 0};
                if (a_) {
                    const float* p = st_buf + (size_t)(n - n0) * kSegFloats * 32 + lane;
                    dr[0] = p[0]; dr[1] = p[32]; dr[2] = p[64];
                    dvv[0] = p[96]; dvv[1] = p[128]; dvv[2] = p[160];
                    A[0] = p[192]; A[1] = p[224]; A[2] = p[256];
                    B[0] = p[288]; B[1] = p[320]; B[2] = p[352];
                }
                long long U[3];
                for (int a = 0; a < 3; ++a) U[a] = st0.U[a] + (long long)n * k.dU[a];
                float u[3] = {0, 0, 0};
                if (a_) {
                    float inc[3], nn = 0.0f;
                    for (int a = 0; a < 3; ++a) {
                        inc[a] = k.dS[a] + dt * (dvv[a] + (A[a] + 2.0f * B[a]) * (1.0f / 6.0f));
                        nn += inc[a] * inc[a];
                    }
                    const float rn = rsqrtf(nn);
                    for (int a = 0; a < 3; ++a) {
                        u[a] = inc[a] * rn;             // unit step direction: d|r_{n+1} - r_n|
                        rb[a] += lenb * u[a];
                    }
                }
                // r' = r + dt (v + (A + 2B)/6),  v' = v + (A + 4B + C)/6
                float Ab[3], Bb[3], Cb[3], rn_[3], vn_[3];
                for (int a = 0; a < 3; ++a) {
                    Ab[a] = (dt * (1.0f / 6.0f)) * rb[a] + vb[a] * (1.0f / 6.0f);
                    Bb[a] = (dt * (1.0f / 3.0f)) * rb[a] + vb[a] * (4.0f / 6.0f);
                    Cb[a] = vb[a] * (1.0f / 6.0f);
                    rn_[a] = rb[a];
                    vn_[a] = vb[a] + dt * rb[a];
                    dtb += rb[a] * (dvv[a] + (A[a] + 2.0f * B[a]) * (1.0f / 6.0f));
                }
                float Db[3], pb[3] = {0, 0, 0}, D[3] = {0, 0, 0}, q[3];
                long long Us[3];
                Stage s;
                float4 Q3 = make_float4(0, 0, 0, 0), Q2 = Q3, Q1 = Q3;
                uint32_t key3 = kNoKey, key2 = kNoKey, key1 = kNoKey;
                float cf3[3] = {0, 0, 0}, cf2[3] = {0, 0, 0}, cf1[3] = {0, 0, 0};
                // C = dt D(p3),  p3 = S(n+1) + dr + dt dv + dt/2 B
                if (a_) {
                    for (int a = 0; a < 3; ++a) {
                        q[a] = dr[a] + dt * dvv[a] + (0.5f * dt) * B[a];
                        Us[a] = U[a] + k.dU[a];
                    }
                    stage_eval(F, Us, q, bc, s);
                    rhs_from(s.ig, D);
                }
                for (int a = 0; a < 3; ++a) {
                    dtb += Cb[a] * D[a];
                    Db[a] = dt * Cb[a];
                }
                if (a_) {
                    rhs_adjoint(F, s.ig, Db, pb, Q3);
                    key3 = s.key;
                    for (int a = 0; a < 3; ++a) cf3[a] = s.cf[a];
                }
                if constexpr (CONN) {
                    const float tn = (float)(n + 1 - n0);
                    for (int a = 0; a < 3; ++a) tps[a] += tn * pb[a];
                }
                for (int a = 0; a < 3; ++a) {
                    rn_[a] += pb[a];
                    vn_[a] += dt * pb[a];
                    Bb[a] += (0.5f * dt) * pb[a];
                    dtb += pb[a] * (dvv[a] + 0.5f * B[a]);
                }
                // B = dt D(p2),  p2 = S(n+1/2) + dr + dt/2 dv + dt/8 A
                if (a_) {
                    for (int a = 0; a < 3; ++a) {
                        q[a] = dr[a] + (0.5f * dt) * dvv[a] + (0.125f * dt) * A[a];
                        Us[a] = U[a] + k.dUh[a];
                    }
                    stage_eval(F, Us, q, bc, s);
                    rhs_from(s.ig, D);
                }
                for (int a = 0; a < 3; ++a) {
                    dtb += Bb[a] * D[a];
                    Db[a] = dt * Bb[a];
                }
                if (a_) {
                    rhs_adjoint(F, s.ig, Db, pb, Q2);
                    key2 = s.key;
                    for (int a = 0; a < 3; ++a) cf2[a] = s.cf[a];
                }
                if constexpr (CONN) {
                    const float tn = (float)(n - n0) + 0.5f;
                    for (int a = 0; a < 3; ++a) tps[a] += tn * pb[a];
                }
                for (int a = 0; a < 3; ++a) {
                    rn_[a] += pb[a];
                    vn_[a] += (0.5f * dt) * pb[a];
                    Ab[a] += (0.125f * dt) * pb[a];
                    dtb += pb[a] * (0.5f * dvv[a] + 0.125f * A[a]);
                }
                // A = dt D(p1),  p1 = S(n) + dr
                if (a_) {
                    stage_eval(F, U, dr, bc, s);
                    rhs_from(s.ig, D);
                }
                for (int a = 0; a < 3; ++a) {
                    dtb += Ab[a] * D[a];
                    Db[a] = dt * Ab[a];
                }
                if (a_) {
                    rhs_adjoint(F, s.ig, Db, pb, Q1);
                    key1 = s.key;
                    for (int a = 0; a < 3; ++a) cf1[a] = s.cf[a];
                }
                if constexpr (CONN) {
                    const float tn = (float)(n - n0);
                    for (int a = 0; a < 3; ++a) tps[a] += tn * pb[a];
                }
                if (a_) {
                    for (int a = 0; a < 3; ++a) {
                        rb[a] = rn_[a] + pb[a] - lenb * u[a];
                        vb[a] = vn_[a];
                    }
                }
                // scatter the three stages: one pass over the lane's cell row for the
                // stages in stage 3's cell, then the others (a step that crosses a face)
#ifndef BOS_ADJ_ONE_PASS
#define BOS_ADJ_ONE_PASS 1
#endif
                const bool same2 = BOS_ADJ_ONE_PASS && key2 == key3, same1 = BOS_ADJ_ONE_PASS && key1 == key3;
                accumulate3(rows, a_, key3, cf3, Q3, same2, cf2, Q2, same1, cf1, Q1, ca, acc, nx, nxy);
                accumulate(rows, a_ && !same2, key2, cf2, Q2, ca, acc, nx, nxy);
                accumulate(rows, a_ && !same1, key1, cf1, Q1, ca, acc, nx, nxy);
            }
            if constexpr (CONN) {
                if (proj && seg)
                    for (int a = 0; a < 3; ++a) tpb[a] += (double)tps[a] + (double)n0 * (double)(rb[a] - rseg[a]);
            }
            __syncwarp();
        }
        // ---- entry: v0 = eta_in d and dt = ell / (N eta_in), eta_in = 1 + deta(r_in)
        int ci[3] = {0, 0, 0};
        float cf[3] = {0, 0, 0};
        if (act) {
            etab -= (double)dtb * (double)dt / eta_in;
            const float zero[3] = {0, 0, 0};
            comp_cell(F, st0.U, zero, ci, cf);
        }
        accumulate(rows, act, cell_key_of(F, ci), cf, make_float4((float)etab, 0.0f, 0.0f, 0.0f), ca, acc, nx, nxy);
        if constexpr (CONN) {
            if (proj && act) {
                Stage se;
                const float zero[3] = {0, 0, 0};
                stage_eval(F, st0.U, zero, bc, se);
                const double ge[3] = {(double)se.ig.d0.x * (double)F.inv_h[0], (double)se.ig.d1.x * (double)F.inv_h[1],
                                      (double)se.ig.d2.x * (double)F.inv_h[2]};
                aim_adjoint(S, RR, eta_in, etab, (double)dtb, ge, rb, drbw, dvbw, tpb, nqp[0], xlb);
            }
        }
        }   // passes
    }
}

#ifndef BOS_REV_MIN_BLOCKS
#define BOS_REV_MIN_BLOCKS 7              // resident 2-warp blocks per SM the register budget is cut for
#endif
#ifndef BOS_REV_CONN_MIN_BLOCKS
#define BOS_REV_CONN_MIN_BLOCKS 6         // the same with the refracted connection
#endif
// What bounds it: instruction issue and dependent arithmetic (45 to 58 % of the issue slots, FMA
// instructions 28 % of their pipe's, at 12 to 16 warps per SM), ~500 warp instructions per step of a
// tile, a quarter of them in the row flushes; memory is at 44 to 61 % (L1) and 1 to 3 % (DRAM).
// 256x256x192 cells, 2048^2 rays: 48.8 ms, where recomputing the segments took 128.4 ms; 192x192x144 cells in
// bfloat16 at 768^2: 6.0 ms, 18.6 ms; with the refracted connection, 128x128x96 cells at 512^2:
// 4.3 ms, 11.2 ms.  Against the float64 oracle the gradients are 10 to 35 % nearer than with the
// recompute (relative L2 2e-7 .. 7e-7).  128 registers and 16 warps beat 168 and 12 by 2 to 3 %;
// with the connection, whose spills then reach the loop, 168 are 7 % faster.  Summing the rows
// of a whole warp one cell at a time, with branches around the row reads, took 62.7 ms.
// SCATTER: rows_scatter (see sparse_lanes).
template <class E, bool CONN, bool QUASI, bool FEW, bool SCATTER>
__global__ void __launch_bounds__(kAdjWarps * 32, FEW ? 1 : CONN ? BOS_REV_CONN_MIN_BLOCKS : BOS_REV_MIN_BLOCKS)
    reverse_kernel(SceneDev S, CkptDev ck, AdjDev adj, WorkDev wk) {
    extern __shared__ float4 smem4[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __shared__ double conn_sh[CONN ? kAdjWarps * 32 * kConnDoubles : 1];   // as in adjoint_kernel
    double* const xlum = conn_sh + (CONN ? (warp * 32 + lane) * kConnDoubles : 0);
    float* rows = reinterpret_cast<float*>(smem4) + (size_t)warp * kWarpRows;
    const CompField<E> F = comp_field<E>(S.g);
    const TileShape ts = tile_shape(S.cam.width, S.cam.height, S.cam.spp);
    const int ntiles = tile_count(S, ts);
    const uint32_t ncells = (uint32_t)S.g.n[0] * S.g.n[1] * S.g.n[2];
    for (;;) {
        int t = 0;
        if (lane == 0) t = atomicAdd(wk.tile_counter, 1);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= ntiles) break;
        reverse_tile<E, CONN, QUASI, SCATTER>(S, ck, adj, F, ts, t, lane, rows, reinterpret_cast<float*>(adj.acc), ncells, S.g.err,
                              wk.tile_counter + 1, xlum);
    }
}

// The tiles that reverse_kernel left (wk.tile_counter[1] of them; its queue is entry 2).
template <class E, bool CONN_T>
__global__ void __launch_bounds__(kAdjWarps * 32, BOS_ADJ_MIN_BLOCKS) adjoint_kernel(SceneDev S, CkptDev ck, AdjDev adj, WorkDev wk) {
    constexpr bool CONN = CONN_T;
    if (wk.tile_counter[1] == 0) return;
    extern __shared__ float4 smem4[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // Refracted connection: values that live across a whole ray reversal are parked in
    // shared memory (per lane: a_1, dL/dx_w, the projector seed, the projector's wall-seed
    // adjoints, the straight-step adjoint sum and |q|) rather than held in registers
    // through the hot loop.
    __shared__ double conn_sh[CONN ? kAdjWarps * 32 * kConnDoubles : 1];
    double* const xlum = conn_sh + (CONN ? (warp * 32 + lane) * kConnDoubles : 0);
    const int K = ck.every;
    float* rows = reinterpret_cast<float*>(smem4) + (size_t)warp * kWarpRows;      // [32][kRow]
    // [K][12][32] step states and stage terms (dr, dv, A, B) of the segment being reversed
    // (this warp's slice)
    float* st_buf = adj.seg + ((size_t)blockIdx.x * kAdjWarps + warp) * ((size_t)K * kSegFloats * 32);
    const CompField<E> F = comp_field<E>(S.g);
    const TileShape ts = tile_shape(S.cam.width, S.cam.height, S.cam.spp);
    const int ntiles = tile_count(S, ts);
    float* acc = reinterpret_cast<float*>(adj.acc);
    {
        float4* row = reinterpret_cast<float4*>(rows + lane * kRow);
        for (int c = 0; c < 8; ++c) row[c] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }
    __syncwarp();
    CellAcc ca = {kNoKey, (uint32_t)S.g.n[0] * S.g.n[1] * S.g.n[2], S.g.err};
    for (;;) {
        int t = 0;
        if (lane == 0) t = atomicAdd(wk.tile_counter + 2, 1);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= ntiles) break;
        if (!tile_needs_stages(ck, ts, t, lane, tile_pixel(S, ts, t, lane).valid)) continue;
        adjoint_tile<E, CONN>(S, ck, adj, F, ts, t, lane, rows, st_buf, acc, ca, xlum);
    }
    flush_rows(rows, ca.key != kNoKey, ca, acc, S.g.n[0], S.g.n[0] * S.g.n[1]);
}

// ---- float64 adjoint (FP64 store and tracer, Sharma RKN) -------------------------------------
//
// The same discrete adjoint in float64 throughout, for the plain float64 tracer: the state
// is the absolute (r, v), kept every K steps by the forward render (six doubles); each
// segment is recomputed into this warp's slice of global memory and reversed; every stage's
// corner sensitivities go to float64 node accumulators.  GB300 runs float64 at 1/64 of the
// float32 rate, so this path is for accuracy, not speed: it separates the method's own error
// from float32 rounding.

struct D4Grad {
    D4 v, d0, d1, d2;   // value and derivatives with respect to the three fractions
};

// Value (dcell_value's operations, so bit-identical) and fraction derivatives.
__device__ __forceinline__ D4Grad dcell_grad(const DCell& m, const double f[3]) {
    const D4 e0 = dfma4(f[0], m.c[1], m.c[0]), e1 = dfma4(f[0], m.c[3], m.c[2]);
    const D4 e2 = dfma4(f[0], m.c[5], m.c[4]), e3 = dfma4(f[0], m.c[7], m.c[6]);
    D4Grad r;
    r.d2 = dfma4(f[1], e3, e2);
    r.v = dfma4(f[2], r.d2, dfma4(f[1], e1, e0));
    r.d1 = dfma4(f[2], e3, e1);
    r.d0 = dfma4(f[2], dfma4(f[1], m.c[7], m.c[5]), dfma4(f[1], m.c[3], m.c[1]));
    return r;
}

struct DStage {
    int i[3];       // base cell
    double f[3];    // fractions (unclamped at the edge cells)
    D4Grad g;
};

// Field value and gradient at absolute position x.
__device__ __forceinline__ void dstage_eval(const GridDev& g, const double x[3], DCell& m, DStage& s) {
    dcell_point(g, x, m, s.f);
    for (int a = 0; a < 3; ++a) s.i[a] = m.i[a];
    s.g = dcell_grad(m, s.f);
}

__device__ __forceinline__ void drhs(const DStage& s, double D[3]) {
    const double eta = 1.0 + s.g.v.x;
    D[0] = eta * s.g.v.y;
    D[1] = eta * s.g.v.z;
    D[2] = eta * s.g.v.w;
}

// Adjoint of D = (1 + deta) grad at a stage for Db: the position adjoint pb and the record
// adjoint Q that the corners share.
__device__ __forceinline__ void drhs_adjoint(const GridDev& g, const DStage& s, const double Db[3], double pb[3],
                                             double Q[4]) {
    const double eta = 1.0 + s.g.v.x;
    const double Dg = Db[0] * s.g.v.y + Db[1] * s.g.v.z + Db[2] * s.g.v.w;
    const D4 dv[3] = {s.g.d0, s.g.d1, s.g.d2};
    Q[0] = Dg;
    for (int a = 0; a < 3; ++a) Q[1 + a] = eta * Db[a];
    for (int a = 0; a < 3; ++a) pb[a] = g.inv_h[a] * (dv[a].x * Q[0] + dv[a].y * Q[1] + dv[a].z * Q[2] + dv[a].w * Q[3]);
}

// Corner sensitivities of a lane's current cell in float64, a row of shared memory per lane
// (value 4 c + channel; odd row stride: neither a lane's own accesses nor a warp's read of one
// row conflict).  A ray stays in a cell for six to twelve stage points, and neighbouring rays
// share cells: summed per lane and then over the warp's lanes of a cell, a tile sends a few
// hundred node additions where every point sent 32 per lane.
constexpr int kRowD = 33;

__device__ __forceinline__ void flush_rows_d(double* rows, bool flag, uint32_t& key, double* acc, const GridDev& g) {
    unsigned pend = __ballot_sync(0xffffffffu, flag);
    if (!pend) return;
    __syncwarp();
    const int lane = threadIdx.x & 31, corner = lane >> 2;
    const uint32_t nx = (uint32_t)g.n[0], nxy = nx * (uint32_t)g.n[1];
    const uint32_t off = (uint32_t)(corner & 1) + (uint32_t)((corner >> 1) & 1) * nx + (uint32_t)(corner >> 2) * nxy;
    const uint32_t mykey = flag ? key : kNoKey;
    while (pend) {
        const uint32_t lk = __shfl_sync(0xffffffffu, mykey, __ffs(pend) - 1);
        unsigned grp = __ballot_sync(0xffffffffu, mykey == lk);
        pend &= ~grp;
        double sum = 0.0;
        for (; grp; grp &= grp - 1) sum += rows[(__ffs(grp) - 1) * kRowD + lane];
        atomicAdd(acc + (size_t)bounded(lk + off, nxy * (uint32_t)g.n[2], g.err) * 4 + (lane & 3), sum);
    }
    __syncwarp();
    if (flag) {
        for (int c = 0; c < 32; ++c) rows[lane * kRowD + c] = 0.0;
        key = kNoKey;
    }
    __syncwarp();
}

// Warp-collective: add w_c(f) Q to the lane's row (flushed first where the cell changes).
__device__ __forceinline__ void accumulate_d(double* rows, bool act, const int i[3], const double f[3], const double Q[4],
                                             uint32_t& key, double* acc, const GridDev& g) {
    const uint32_t cell =
        act ? (uint32_t)i[0] + (uint32_t)g.n[0] * ((uint32_t)i[1] + (uint32_t)g.n[1] * (uint32_t)i[2]) : kNoKey;
    flush_rows_d(rows, act && key != kNoKey && key != cell, key, acc, g);
    if (!act) return;
    key = cell;
    double* row = rows + (threadIdx.x & 31) * kRowD;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const double w = ((c & 1) ? f[0] : 1.0 - f[0]) * ((c & 2) ? f[1] : 1.0 - f[1]) * ((c & 4) ? f[2] : 1.0 - f[2]);
#pragma unroll
        for (int ch = 0; ch < 4; ++ch) row[4 * c + ch] = fma(w, Q[ch], row[4 * c + ch]);
    }
}

// G = the seed's type: float (bos_backward) or double (bos_backward_f64).
template <class G>
__global__ void __launch_bounds__(kAdjWarps * 32) adjoint_fp64_kernel(SceneDev S, CkptDev ck, AdjDev adj, WorkDev wk) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int K = ck.every;
    // [K][6][32] step states (r, v) of the segment being reversed (this warp's slice)
    double* buf = reinterpret_cast<double*>(adj.seg) + ((size_t)blockIdx.x * kAdjWarps + warp) * ((size_t)K * 6 * 32);
    const double* ckd = reinterpret_cast<const double*>(ck.state);
    double* acc = reinterpret_cast<double*>(adj.acc);
    const GridDev& g = S.g;
    const FullField<double> F = {S.g};
    __shared__ double rows_sh[kAdjWarps * 32 * kRowD];
    double* const rows = rows_sh + (size_t)warp * 32 * kRowD;
    for (int c = 0; c < 32; ++c) rows[lane * kRowD + c] = 0.0;
    uint32_t key = kNoKey;                // cell of the lane's row
    const int W = S.cam.width, H = S.cam.height, spp = S.cam.spp;
    const TileShape ts = tile_shape(W, H, spp);
    const int ntiles = tile_count(S, ts);
    for (;;) {
        int t = 0;
        if (lane == 0) t = atomicAdd(wk.tile_counter, 1);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= ntiles) break;
        const int sl = lane % ts.G;
        const TilePix tp = tile_pixel(S, ts, t, lane);
        for (int qs = 0; qs < ts.samples_per_lane; ++qs) {
            const int s = ts.samples_per_lane == 1 ? sl : qs;
            const long long slot = ((long long)t * 32 + lane) * ts.samples_per_lane + qs;
            Ray R;
            R.N = 0;
            R.wall = false;
            double Ib = 0.0;
            if (tp.valid) {
                R = ray_setup(S, tp.px, tp.py, s);
                Ib = (double)reinterpret_cast<const G*>(adj.dLdI)[(size_t)tp.out] / spp;
            }
            const bool act = tp.valid && R.wall && R.N > 0 && Ib != 0.0;
            // entry state as the forward forms it: r_in, eta_in, v0 = eta_in d, dt = ell / (N eta_in)
            double rin[3] = {0.0, 0.0, 0.0}, eta_in = 1.0, dt = 0.0;
            if (act) {
                for (int a = 0; a < 3; ++a) rin[a] = S.cam.pos[a] + R.t_in * R.d[a];
                eta_in = F.eta(rin);
                dt = R.ell / ((double)R.N * eta_in);
            }
            const int N = act ? R.N : 0;
            const int nseg = (N + K - 1) / K;
            const int nseg_max = __reduce_max_sync(0xffffffffu, (unsigned)nseg);
            double rb[3] = {0, 0, 0}, vb[3] = {0, 0, 0}, dtb = 0.0, lenb = 0.0;
            const double dt6 = sixth(dt);
            for (int c = nseg_max - 1; c >= 0; --c) {
                const int n0 = c * K, n1 = min(n0 + K, N);
                const bool seg = act && n0 < N;
                if (seg) {
                    // ---- recompute the segment from its checkpoint (full_step's operations)
                    double r[3], v[3];
                    const size_t cc = bounded((size_t)c, (size_t)ck.max_ckpt, ck.err);
                    for (int q = 0; q < 3; ++q) {
                        r[q] = ckd[(cc * 6 + q) * ck.nrays + slot];
                        v[q] = ckd[(cc * 6 + 3 + q) * ck.nrays + slot];
                    }
                    for (int n = n0; n < n1; ++n) {
                        double* p = buf + (size_t)(n - n0) * 6 * 32 + lane;
                        for (int q = 0; q < 3; ++q) {
                            p[32 * q] = r[q];
                            p[32 * (3 + q)] = v[q];
                        }
                        full_step<double, 0>(F, r, v, dt);
                    }
                    if (c == nseg - 1) {
                        double lb = 0.0;
                        const double len_before = R.t_in + reinterpret_cast<const double*>(ck.excess)[slot];
                        wall_adjoint(S, r, v, len_before, Ib, rb, vb, lb);
                        lenb = lb;
                    }
                }
                __syncwarp();
                // ---- reverse the segment's steps
                const int n_hi = __reduce_max_sync(0xffffffffu, (unsigned)(seg ? n1 : 0));
                for (int n = n_hi - 1; n >= n0; --n) {
                    const bool a_ = seg && n < n1;
                    DStage s1, s2, s3;
                    double Q1[4], Q2[4], Q3[4];
                    if (a_) {
                        const double* p = buf + (size_t)(n - n0) * 6 * 32 + lane;
                        double r[3], v[3], A[3], B[3], D1[3], D2[3], D3[3], q[3];
                        for (int a = 0; a < 3; ++a) {
                            r[a] = p[32 * a];
                            v[a] = p[32 * (3 + a)];
                        }
                        dstage_eval(g, r, F.m, s1);
                        drhs(s1, D1);
                        for (int a = 0; a < 3; ++a) A[a] = dt * D1[a];
                        for (int a = 0; a < 3; ++a) q[a] = r[a] + (dt * 0.5) * v[a] + (dt * 0.125) * A[a];
                        dstage_eval(g, q, F.m, s2);
                        drhs(s2, D2);
                        for (int a = 0; a < 3; ++a) B[a] = dt * D2[a];
                        for (int a = 0; a < 3; ++a) q[a] = r[a] + dt * v[a] + (dt * 0.5) * B[a];
                        dstage_eval(g, q, F.m, s3);
                        drhs(s3, D3);
                        // r' = r + dt (v + (A + 2B)/6), |r' - r| enters the path length
                        double inc[3], nn = 0.0, u[3];
                        for (int a = 0; a < 3; ++a) {
                            inc[a] = dt * (v[a] + sixth(A[a] + 2.0 * B[a]));
                            nn += inc[a] * inc[a];
                        }
                        const double rn = rsqrt(nn);
                        double rbs[3], Ab[3], Bb[3], Cb[3], rn_[3], vn_[3], Db[3], pb[3];
                        for (int a = 0; a < 3; ++a) {
                            u[a] = inc[a] * rn;
                            rbs[a] = rb[a] + lenb * u[a];
                        }
                        for (int a = 0; a < 3; ++a) {
                            Cb[a] = sixth(vb[a]);
                            Ab[a] = dt6 * rbs[a] + Cb[a];
                            Bb[a] = 2.0 * (dt6 * rbs[a]) + vb[a] * (4.0 / 6.0);
                            rn_[a] = rbs[a];
                            vn_[a] = vb[a] + dt * rbs[a];
                            dtb += rbs[a] * (v[a] + sixth(A[a] + 2.0 * B[a]));
                        }
                        // C = dt D(p3), p3 = r + dt v + dt/2 B
                        for (int a = 0; a < 3; ++a) {
                            dtb += Cb[a] * D3[a];
                            Db[a] = dt * Cb[a];
                        }
                        drhs_adjoint(g, s3, Db, pb, Q3);
                        for (int a = 0; a < 3; ++a) {
                            rn_[a] += pb[a];
                            vn_[a] += dt * pb[a];
                            Bb[a] += (0.5 * dt) * pb[a];
                            dtb += pb[a] * (v[a] + 0.5 * B[a]);
                        }
                        // B = dt D(p2), p2 = r + dt/2 v + dt/8 A
                        for (int a = 0; a < 3; ++a) {
                            dtb += Bb[a] * D2[a];
                            Db[a] = dt * Bb[a];
                        }
                        drhs_adjoint(g, s2, Db, pb, Q2);
                        for (int a = 0; a < 3; ++a) {
                            rn_[a] += pb[a];
                            vn_[a] += (0.5 * dt) * pb[a];
                            Ab[a] += (0.125 * dt) * pb[a];
                            dtb += pb[a] * (0.5 * v[a] + 0.125 * A[a]);
                        }
                        // A = dt D(p1), p1 = r
                        for (int a = 0; a < 3; ++a) {
                            dtb += Ab[a] * D1[a];
                            Db[a] = dt * Ab[a];
                        }
                        drhs_adjoint(g, s1, Db, pb, Q1);
                        for (int a = 0; a < 3; ++a) {
                            rb[a] = rn_[a] + pb[a] - lenb * u[a];
                            vb[a] = vn_[a];
                        }
                    }
                    accumulate_d(rows, a_, s3.i, s3.f, Q3, key, acc, g);
                    accumulate_d(rows, a_, s2.i, s2.f, Q2, key, acc, g);
                    accumulate_d(rows, a_, s1.i, s1.f, Q1, key, acc, g);
                }
                __syncwarp();
            }
            // ---- entry: v0 = eta_in d, dt = ell / (N eta_in), eta_in = 1 + deta(r_in)
            DStage se;
            double Qe[4] = {0.0, 0.0, 0.0, 0.0};
            if (act) {
                Qe[0] = vb[0] * R.d[0] + vb[1] * R.d[1] + vb[2] * R.d[2] - dtb * dt / eta_in;
                split_point(g, rin, se.i, se.f);
            }
            accumulate_d(rows, act, se.i, se.f, Qe, key, acc, g);
            flush_rows_d(rows, key != kNoKey, key, acc, g);
        }
    }
}

// Transpose of the difference stencil of grad eta at node c, plus d L/d deta, in float64.
template <class A>
__device__ __forceinline__ double stencil_fp64(const GridDev& g, const A* __restrict__ acc, uint32_t c) {
    const uint32_t stride[3] = {1u, (uint32_t)g.n[0], (uint32_t)g.n[0] * (uint32_t)g.n[1]};
    const int idx[3] = {(int)(c % stride[1]), (int)(c / stride[1] % (uint32_t)g.n[1]), (int)(c / stride[2])};
    double tot = acc[(size_t)c * 4];
    for (int a = 0; a < 3; ++a) {
        const int i = idx[a], na = g.n[a];
        const double ih = g.inv_h[a], ih2 = 0.5 * g.inv_h[a];
        const A* p = acc + 1 + a;
        if (i - 1 >= 0) tot += p[(size_t)(c - stride[a]) * 4] * (i - 1 == 0 ? ih : ih2);        // node i-1 reads i as hi
        if (i + 1 <= na - 1) tot -= p[(size_t)(c + stride[a]) * 4] * (i + 1 == na - 1 ? ih : ih2);  // node i+1 reads i as lo
        if (i == 0) tot -= p[(size_t)c * 4] * ih;                                               // one-sided at the faces
        if (i == na - 1) tot += p[(size_t)c * 4] * ih;
    }
    return tot;
}

// dL/dT per node: that times d deta/dT = -K / T^2 (float64 accumulators).
template <class O>
__global__ void gradient_fp64_kernel(GridDev g, const double* __restrict__ acc, const float* __restrict__ T,
                                     O* __restrict__ dLdT) {
    const uint32_t n = (uint32_t)g.n[0] * g.n[1] * g.n[2], c = blockIdx.x * 256u + threadIdx.x;
    if (c >= n) return;
    const double Tc = (double)T[c];
    dLdT[c] = (O)(stencil_fp64(g, acc, c) * (-g.K / (Tc * Tc)));
}

// The same for float32 accumulators.  The sum is carried in two float32 terms (products and
// sums with their rounding errors, Knuth's two-sum), which keeps ~2^-46 of its largest term:
// the float64 sum it replaces held the 12.6 M cells of a 256x256x192 grid for 611 us on the
// float64 pipe and in 64-bit index divisions; this takes 121 us, against 45 us to read the
// accumulators and T and write dL/dT (five rows of accumulators pass through L2 per row).  Where a
// product or the sum leaves float32's range the rounding errors are NaN: there the sum is float64's.
struct GradConst {
    float hi[3][2], lo[3][2];   // 1 / (2 h), 1 / h in two terms
    float K;
};

__device__ __forceinline__ void add_term(float& s, float& e, float a, float kh, float kl) {
    const float p = __fmul_rn(a, kh);
    e = __fadd_rn(e, fmaf(a, kl, fmaf(a, kh, -p)));
    const float t = __fadd_rn(s, p), z = __fsub_rn(t, s);
    e = __fadd_rn(e, __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(p, z)));
    s = t;
}

__global__ void __launch_bounds__(256) gradient_kernel(GridDev g, GradConst k, const float4* __restrict__ acc4,
                                                       const float* __restrict__ T, float* __restrict__ dLdT) {
    const uint32_t n = (uint32_t)g.n[0] * g.n[1] * g.n[2], c = blockIdx.x * 256u + threadIdx.x;
    if (c >= n) return;
    const uint32_t nx = (uint32_t)g.n[0], nxy = nx * (uint32_t)g.n[1];
    const uint32_t z = c / nxy, r = c - z * nxy, y = r / nx;
    const uint32_t idx[3] = {r - y * nx, y, z}, stride[3] = {1u, nx, nxy};
    const float* acc = reinterpret_cast<const float*>(acc4) + (size_t)c * 4;
    float s = acc[0], e = 0.0f;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const uint32_t i = idx[a], last = (uint32_t)g.n[a] - 1u;
        const float* p = acc + 1 + a;
        if (i > 0u) {                                    // node i-1 reads i as hi
            const bool one = i == 1u;                    // (selected: see build_split_kernel)
            add_term(s, e, p[-(ptrdiff_t)stride[a] * 4], one ? k.hi[a][1] : k.hi[a][0], one ? k.lo[a][1] : k.lo[a][0]);
        }
        if (i < last) {                                  // node i+1 reads i as lo
            const bool one = i + 1u == last;
            add_term(s, e, -p[(size_t)stride[a] * 4], one ? k.hi[a][1] : k.hi[a][0], one ? k.lo[a][1] : k.lo[a][0]);
        }
        if (i == 0u) add_term(s, e, -p[0], k.hi[a][1], k.lo[a][1]);      // one-sided at the faces
        if (i == last) add_term(s, e, p[0], k.hi[a][1], k.lo[a][1]);
    }
    s = __fadd_rn(s, e);
    if (!(fabsf(s) <= 3.4028235e38f)) s = (float)stencil_fp64(g, reinterpret_cast<const float*>(acc4), c);
    const float Tc = T[c];
    dLdT[c] = s * (-k.K / (Tc * Tc));
}

// Batched adjoints (the request server): one launch covers warp tiles of several jobs,
// indexed as in render_batch_kernel.  counter: queue, tiles left to adjoint_batch_kernel, its
// queue.
template <class E, bool QUASI>
__global__ void __launch_bounds__(kAdjWarps * 32, BOS_REV_MIN_BLOCKS)
    reverse_batch_kernel(const BatchJob* __restrict__ jobs, int njobs, int total, int* counter) {
    extern __shared__ float4 smem4[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float* rows = reinterpret_cast<float*>(smem4) + (size_t)warp * kWarpRows;
    for (;;) {
        int g = 0;
        if (lane == 0) g = atomicAdd(counter, 1);
        g = __shfl_sync(0xffffffffu, g, 0);
        if (g >= total) break;
        const BatchJob& J = jobs[batch_job_of(jobs, njobs, g)];
        const TileShape ts = tile_shape(J.S.cam.width, J.S.cam.height, J.S.cam.spp);
        const uint32_t ncells = (uint32_t)J.S.g.n[0] * J.S.g.n[1] * J.S.g.n[2];
        float* const acc = reinterpret_cast<float*>(J.adj.acc);
        const int t = J.tile0 + (g - J.first);
        // (a choice of rows_scatter per job: 9.5 ms for a mix of six requests instead of 8.55, by spills)
        reverse_tile<E, false, QUASI, false>(J.S, J.ck, J.adj, comp_field<E>(J.S.g), ts, t, lane, rows, acc, ncells,
                                             J.S.g.err, counter + 1, nullptr);
    }
}

// The Sharma tiles that reverse_batch_kernel left.  The lane rows belong to one job's
// accumulators at a time, so they are flushed whenever a warp moves on to another job's tile.
// The segment slices come from seg_base with room for k_max steps.
template <class E>
__global__ void __launch_bounds__(kAdjWarps * 32, BOS_ADJ_MIN_BLOCKS)
    adjoint_batch_kernel(const BatchJob* __restrict__ jobs, int njobs, int total, int* counter, float* seg_base,
                         int k_max) {
    if (counter[1] == 0) return;
    extern __shared__ float4 smem4[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float* rows = reinterpret_cast<float*>(smem4) + (size_t)warp * kWarpRows;
    float* st_buf = seg_base + ((size_t)blockIdx.x * kAdjWarps + warp) * ((size_t)k_max * kSegFloats * 32);
    {
        float4* row = reinterpret_cast<float4*>(rows + lane * kRow);
        for (int c = 0; c < 8; ++c) row[c] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }
    __syncwarp();
    CellAcc ca = {kNoKey, 0u, nullptr};
    int cur = -1;                      // job whose accumulators the rows belong to
    for (;;) {
        int g = 0;
        if (lane == 0) g = atomicAdd(counter + 2, 1);
        g = __shfl_sync(0xffffffffu, g, 0);
        if (g >= total) break;
        const int j = batch_job_of(jobs, njobs, g);
        if (j != cur && cur >= 0) {
            const BatchJob& P = jobs[cur];
            flush_rows(rows, ca.key != kNoKey, ca, reinterpret_cast<float*>(P.adj.acc), P.S.g.n[0],
                       P.S.g.n[0] * P.S.g.n[1]);
        }
        cur = j;
        const BatchJob& J = jobs[j];
        ca.ncells = (uint32_t)J.S.g.n[0] * J.S.g.n[1] * J.S.g.n[2];
        ca.err = J.S.g.err;
        const CompField<E> F = comp_field<E>(J.S.g);
        const TileShape ts = tile_shape(J.S.cam.width, J.S.cam.height, J.S.cam.spp);
        const int t = J.tile0 + (g - J.first);
        if (tile_needs_stages(J.ck, ts, t, lane, tile_pixel(J.S, ts, t, lane).valid))
            adjoint_tile<E, false>(J.S, J.ck, J.adj, F, ts, t, lane, rows, st_buf,
                                   reinterpret_cast<float*>(J.adj.acc), ca, nullptr);
    }
    if (cur >= 0) {
        const BatchJob& P = jobs[cur];
        flush_rows(rows, ca.key != kNoKey, ca, reinterpret_cast<float*>(P.adj.acc), P.S.g.n[0], P.S.g.n[0] * P.S.g.n[1]);
    }
}

template <class E, bool QUASI>
static cudaError_t launch_adjoint_batch_c(const BatchJob* jobs, int njobs, int total, int* counter, float* seg_base,
                                          int k_max, int num_sms, cudaStream_t st) {
    const size_t smem = (size_t)kAdjWarps * kWarpRows * sizeof(float);
    int per_sm = 0;
    cudaError_t e = occupancy_prefer_l1(reverse_batch_kernel<E, QUASI>, kAdjWarps * 32, smem, per_sm);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    reverse_batch_kernel<E, QUASI><<<num_sms * per_sm, kAdjWarps * 32, smem, st>>>(jobs, njobs, total, counter);
    if ((e = cudaGetLastError()) != cudaSuccess || QUASI) return e;
    e = occupancy_prefer_l1(adjoint_batch_kernel<E>, kAdjWarps * 32, smem, per_sm);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    const int blocks = num_sms * per_sm < kAdjMaxBlocks ? num_sms * per_sm : kAdjMaxBlocks;
    adjoint_batch_kernel<E><<<blocks, kAdjWarps * 32, smem, st>>>(jobs, njobs, total, counter, seg_base, k_max);
    return cudaGetLastError();
}

cudaError_t launch_adjoint_batch(int mode, int integ, const BatchJob* jobs, int njobs, int total, int* counter,
                                 float* seg_base, int k_max, int num_sms, cudaStream_t st) {
    if (k_max > 64 || (integ != 0 && integ != 2)) return cudaErrorNotSupported;
    if (mode == 1) return integ == 2 ? launch_adjoint_batch_c<F4P, true>(jobs, njobs, total, counter, seg_base, k_max, num_sms, st)
                                     : launch_adjoint_batch_c<F4P, false>(jobs, njobs, total, counter, seg_base, k_max, num_sms, st);
    if (mode == 2) return integ == 2 ? launch_adjoint_batch_c<B4P, true>(jobs, njobs, total, counter, seg_base, k_max, num_sms, st)
                                     : launch_adjoint_batch_c<B4P, false>(jobs, njobs, total, counter, seg_base, k_max, num_sms, st);
    return cudaErrorNotSupported;
}

static unsigned cell_blocks(const GridDev& g) {
    return (unsigned)(((long long)g.n[0] * g.n[1] * g.n[2] + 255) / 256);
}

cudaError_t launch_gradient(const GridDev& g, const float4* acc, const float* T, float* dLdT, cudaStream_t st) {
    GradConst k;
    k.K = (float)g.K;
    for (int a = 0; a < 3; ++a)
        for (int one = 0; one < 2; ++one) {
            const double v = one ? g.inv_h[a] : 0.5 * g.inv_h[a];
            k.hi[a][one] = (float)v;
            k.lo[a][one] = (float)(v - (double)k.hi[a][one]);
        }
    gradient_kernel<<<cell_blocks(g), 256, 0, st>>>(g, k, acc, T, dLdT);
    return cudaGetLastError();
}

template <class E, bool CONN, bool QUASI, bool FEW, bool SCATTER>
static cudaError_t launch_reverse_f(const SceneDev& S, const CkptDev& ck, const AdjDev& adj, const WorkDev& w,
                                    int num_sms, cudaStream_t st) {
    const size_t smem = SCATTER ? 0 : (size_t)kAdjWarps * kWarpRows * sizeof(float);
    int per_sm = 0;
    cudaError_t e = occupancy_prefer_l1(reverse_kernel<E, CONN, QUASI, FEW, SCATTER>, kAdjWarps * 32, smem, per_sm);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    reverse_kernel<E, CONN, QUASI, FEW, SCATTER><<<num_sms * per_sm, kAdjWarps * 32, smem, st>>>(S, ck, adj, w);
    return cudaGetLastError();
}

// Launches of at most kFewTiles warp tiles per SM take the form without a register cap (~230
// registers, which leaves 8 warps per SM resident): the GPU is not full either way and each
// ray finishes sooner without spills.
template <class E, bool CONN, bool QUASI>
static cudaError_t launch_reverse(const SceneDev& S, const CkptDev& ck, const AdjDev& adj, const WorkDev& w, int num_sms,
                                  cudaStream_t st) {
    const TileShape ts = tile_shape(S.cam.width, S.cam.height, S.cam.spp);
    const bool sparse = sparse_lanes(S, ts, CONN);
    if (tile_count(S, ts) <= num_sms * kFewTiles)
        return sparse ? launch_reverse_f<E, CONN, QUASI, true, true>(S, ck, adj, w, num_sms, st)
                      : launch_reverse_f<E, CONN, QUASI, true, false>(S, ck, adj, w, num_sms, st);
    return sparse ? launch_reverse_f<E, CONN, QUASI, false, true>(S, ck, adj, w, num_sms, st)
                  : launch_reverse_f<E, CONN, QUASI, false, false>(S, ck, adj, w, num_sms, st);
}

template <class E, bool CONN>
static cudaError_t launch_adjoint_c(const SceneDev& S, const CkptDev& ck, const AdjDev& adj, const WorkDev& w,
                                    int num_sms, cudaStream_t st) {
    const size_t smem = (size_t)kAdjWarps * kWarpRows * sizeof(float);
    cudaError_t e =
        cudaFuncSetAttribute(adjoint_kernel<E, CONN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = occupancy_prefer_l1(adjoint_kernel<E, CONN>, kAdjWarps * 32, smem, per_sm);
    if (e != cudaSuccess) return e;
    if (per_sm < 1 || adj.seg == nullptr) return cudaErrorInvalidConfiguration;
    e = launch_reverse<E, CONN, false>(S, ck, adj, w, num_sms, st);
    if (e != cudaSuccess) return e;
    const int blocks = num_sms * per_sm < kAdjMaxBlocks ? num_sms * per_sm : kAdjMaxBlocks;
    adjoint_kernel<E, CONN><<<blocks, kAdjWarps * 32, smem, st>>>(S, ck, adj, w);
    return cudaGetLastError();
}

// The refracted projector connection (light mode 2) reverses each sample's projector ray
// too; it has its own instantiation so that the other modes do not carry it.
template <class E>
static cudaError_t launch_adjoint_t(const SceneDev& S, const CkptDev& ck, const AdjDev& adj, const WorkDev& w,
                                    int num_sms, cudaStream_t st) {
    if (S.L.mode == 2) {
        if (ck.pstate == nullptr || ck.conn == nullptr) return cudaErrorInvalidValue;
        return launch_adjoint_c<E, true>(S, ck, adj, w, num_sms, st);
    }
    return launch_adjoint_c<E, false>(S, ck, adj, w, num_sms, st);
}

// Float64 store and tracer: Sharma RKN, float64 accumulators; seed and dL/dT in float32 or
// (f64) float64.
cudaError_t launch_backward_fp64(const SceneDev& S, const CkptDev& ck, const AdjDev& adj, const WorkDev& w,
                                 const float* T, void* dLdT, bool f64, int num_sms, cudaStream_t st) {
    if (S.it.integrator != 0 || S.L.mode == 2 || adj.seg == nullptr || ck.every > 64) return cudaErrorNotSupported;
    const int blocks = num_sms * 8 < kAdjMaxBlocks ? num_sms * 8 : kAdjMaxBlocks;
    const int threads =
        fp64_threads(tile_count(S, tile_shape(S.cam.width, S.cam.height, S.cam.spp)), num_sms, kAdjWarps * 32);
    if (f64) adjoint_fp64_kernel<double><<<blocks, threads, 0, st>>>(S, ck, adj, w);
    else adjoint_fp64_kernel<float><<<blocks, threads, 0, st>>>(S, ck, adj, w);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const double* acc = reinterpret_cast<const double*>(adj.acc);
    if (f64) gradient_fp64_kernel<<<cell_blocks(S.g), 256, 0, st>>>(S.g, acc, T, static_cast<double*>(dLdT));
    else gradient_fp64_kernel<<<cell_blocks(S.g), 256, 0, st>>>(S.g, acc, T, static_cast<float*>(dLdT));
    return cudaGetLastError();
}

cudaError_t launch_backward(int mode, const SceneDev& S, const CkptDev& ck, const AdjDev& adj, const WorkDev& w,
                            const float* T, float* dLdT, int num_sms, cudaStream_t st) {
    const bool quasi = S.it.integrator == 2;
    if (!quasi && ck.every > 64) return cudaErrorNotSupported;
    cudaError_t e;
    if (mode == 4) return launch_backward_fp64(S, ck, adj, w, T, dLdT, false, num_sms, st);
    if (mode == 1) e = quasi ? launch_reverse<F4P, false, true>(S, ck, adj, w, num_sms, st)
                             : launch_adjoint_t<F4P>(S, ck, adj, w, num_sms, st);
    else if (mode == 2) e = quasi ? launch_reverse<B4P, false, true>(S, ck, adj, w, num_sms, st)
                                  : launch_adjoint_t<B4P>(S, ck, adj, w, num_sms, st);
    else return cudaErrorNotSupported;
    return e == cudaSuccess ? launch_gradient(S.g, adj.acc, T, dLdT, st) : e;
}

}  // namespace bos
