// The reduced dipole pair kernel shared by the field traversal and the
// gradient pass (Sec. 2, reduced Eqs. h_dip and f_dip).
#pragma once

#include "ffk.cuh"

namespace ffk {

__device__ __forceinline__ float dip_rsqrt(float x) { return rsqrtf(x); }
__device__ __forceinline__ double dip_rsqrt(double x) { return rsqrt(x); }

__device__ __forceinline__ float rfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double rfma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float pmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double pmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float padd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double padd(double a, double b) { return __dadd_rn(a, b); }

// r^2 of a pair, each fused operation written out: every walk forms the same bits.
template <typename R>
__device__ __forceinline__ R pair_r2(R rx, R ry, R rz)
{
    return rfma(rz, rz, rfma(rx, rx, pmul(ry, ry)));
}
// a.b, likewise.
template <typename R>
__device__ __forceinline__ R pair_dot(R ax, R ay, R az, R bx, R by, R bz)
{
    return rfma(az, bz, rfma(ax, bx, pmul(ay, by)));
}

// Reduced dipolar field of u_j and force on u_k at separation r = rho_k - rho_j
// (Sec. 2, reduced Eqs. h_dip and f_dip), accumulated:
//   h += [3 r (u_j.r) - u_j r^2] / r^5
//   f += 3 [r (u_j.u_k) + u_k (u_j.r) + u_j (u_k.r)] / r^5 - 15 r (u_k.r)(u_j.r) / r^7
template <typename R>
__device__ __forceinline__ void dipole(R rx, R ry, R rz, R r2, R ukx, R uky, R ukz, R ujx, R ujy,
                                       R ujz, R& hx, R& hy, R& hz, R& fx, R& fy, R& fz)
{
    const R ir = dip_rsqrt(r2);
    const R ir2 = ir * ir;
    const R ir3 = ir2 * ir;
    const R ir5 = ir3 * ir2;
    const R ir7 = ir5 * ir2;
    const R bj = ujx * rx + ujy * ry + ujz * rz;
    const R bk = ukx * rx + uky * ry + ukz * rz;
    const R a = ujx * ukx + ujy * uky + ujz * ukz;
    const R s3 = R(3) * ir5;
    const R cuk = s3 * bj, cuj = s3 * bk;  // cuk = 3 (u_j.r) / r^5 serves h and f
    hx += rx * cuk - ujx * ir3;
    hy += ry * cuk - ujy * ir3;
    hz += rz * cuk - ujz * ir3;
    const R cr = s3 * a - R(15) * bk * bj * ir7;
    fx += rx * cr + ukx * cuk + ujx * cuj;
    fy += ry * cr + uky * cuk + ujy * cuj;
    fz += rz * cr + ukz * cuk + ujz * cuj;
}

// The same with each fused operation written out, for the FP32 walks: every walk
// that adds the same terms in the same order gives the same bits.
template <typename R>
__device__ __forceinline__ void walk_dipole(R rx, R ry, R rz, R r2, R ukx, R uky, R ukz, R ujx, R ujy,
                                       R ujz, R& hx, R& hy, R& hz, R& fx, R& fy, R& fz)
{
    const R ir = dip_rsqrt(r2);
    const R ir2 = pmul(ir, ir);
    const R ir3 = pmul(ir2, ir);
    const R ir5 = pmul(ir3, ir2);
    const R ir7 = pmul(ir5, ir2);
    const R bj = pair_dot(ujx, ujy, ujz, rx, ry, rz);
    const R bk = pair_dot(ukx, uky, ukz, rx, ry, rz);
    const R a = pair_dot(ujx, ujy, ujz, ukx, uky, ukz);
    const R s3 = pmul(R(3), ir5);
    const R cuk = pmul(s3, bj), cuj = pmul(s3, bk);  // cuk = 3 (u_j.r) / r^5 serves h and f
    hx = padd(hx, rfma(rx, cuk, -pmul(ujx, ir3)));
    hy = padd(hy, rfma(ry, cuk, -pmul(ujy, ir3)));
    hz = padd(hz, rfma(rz, cuk, -pmul(ujz, ir3)));
    const R cr = rfma(s3, a, -pmul(pmul(pmul(R(15), bk), bj), ir7));
    fx = padd(fx, rfma(ujx, cuj, rfma(ukx, cuk, pmul(rx, cr))));
    fy = padd(fy, rfma(ujy, cuj, rfma(uky, cuk, pmul(ry, cr))));
    fz = padd(fz, rfma(ujz, cuj, rfma(ukz, cuk, pmul(rz, cr))));
}

// The terms of two sources (components .x and .y) for one target, two FP32
// operations per instruction: walk_dipole()'s operations in its order, so
// each source's terms have the same bits.  v = -u_j: with the moment's sign
// turned, (-3 / r^5)(v.r) is 3 (u_j.r) / r^5 and every product below has
// walk_dipole()'s value without an instruction spent on a sign.  The caller adds the
// terms one source after the other (h += t, f += s).
struct DipoleTerms2 {
    float2 tx, ty, tz, sx, sy, sz;
};
__device__ __forceinline__ float2 dup2(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 pair_r2_2(float2 rx, float2 ry, float2 rz)
{
    return __ffma2_rn(rz, rz, __ffma2_rn(rx, rx, __fmul2_rn(ry, ry)));
}
__device__ __forceinline__ DipoleTerms2 dipole2(float2 rx, float2 ry, float2 rz, float2 ir,
                                                float2 ukx, float2 uky, float2 ukz, float2 vx,
                                                float2 vy, float2 vz)
{
    DipoleTerms2 o;
    const float2 ir2 = __fmul2_rn(ir, ir);
    const float2 ir3 = __fmul2_rn(ir2, ir);
    const float2 ir5 = __fmul2_rn(ir3, ir2);
    const float2 ir7 = __fmul2_rn(ir5, ir2);
    const float2 bj = __ffma2_rn(vz, rz, __ffma2_rn(vx, rx, __fmul2_rn(vy, ry)));    // -u_j.r
    const float2 bk = __ffma2_rn(ukz, rz, __ffma2_rn(ukx, rx, __fmul2_rn(uky, ry)));
    const float2 a = __ffma2_rn(vz, ukz, __ffma2_rn(vx, ukx, __fmul2_rn(vy, uky)));  // -u_j.u_k
    const float2 s3 = __fmul2_rn(dup2(-3.0f), ir5);
    const float2 cuk = __fmul2_rn(s3, bj);
    const float2 cuj = __fmul2_rn(s3, bk);  // -3 (u_k.r) / r^5
    o.tx = __ffma2_rn(rx, cuk, __fmul2_rn(vx, ir3));
    o.ty = __ffma2_rn(ry, cuk, __fmul2_rn(vy, ir3));
    o.tz = __ffma2_rn(rz, cuk, __fmul2_rn(vz, ir3));
    const float2 cr =
        __ffma2_rn(s3, a, __fmul2_rn(__fmul2_rn(__fmul2_rn(dup2(15.0f), bk), bj), ir7));
    o.sx = __ffma2_rn(vx, cuj, __ffma2_rn(ukx, cuk, __fmul2_rn(rx, cr)));
    o.sy = __ffma2_rn(vy, cuj, __ffma2_rn(uky, cuk, __fmul2_rn(ry, cr)));
    o.sz = __ffma2_rn(vz, cuj, __ffma2_rn(ukz, cuk, __fmul2_rn(rz, cr)));
    return o;
}

// The same terms with u_k's part of the force kept as one scalar: adds
//   h += r cuk - u_j / r^3,   f += r cr + u_j cuj,   c += cuk,
// cuk = 3 (u_j.r) / r^5, cuj = 3 (u_k.r) / r^5,
// cr = 3 / r^5 [u_j.u_k - 5 (u_k.r)(u_j.r) / r^2],
// so that the force on u_k is f + u_k c once every source has been added (u_k
// is the same for all of them).  A pair at r2 = 0 adds nothing.  Each operation
// is written out: the counting and the plain walk give the same bits.
template <typename R>
__device__ __forceinline__ void dipole_acc(R rx, R ry, R rz, R r2, R ukx, R uky, R ukz, R ujx,
                                           R ujy, R ujz, R& hx, R& hy, R& hz, R& fx, R& fy,
                                           R& fz, R& c)
{
    const R ir = r2 > R(0) ? dip_rsqrt(r2) : R(0);
    const R ir2 = pmul(ir, ir);
    const R ir3 = pmul(ir2, ir);
    const R s3 = pmul(pmul(R(3), ir2), ir3);
    const R bj = pair_dot(ujx, ujy, ujz, rx, ry, rz);
    const R bk = pair_dot(ukx, uky, ukz, rx, ry, rz);
    const R a = pair_dot(ujx, ujy, ujz, ukx, uky, ukz);
    const R cuk = pmul(s3, bj), cuj = pmul(s3, bk);
    const R cr = pmul(s3, rfma(pmul(R(-5), ir2), pmul(bj, bk), a));
    hx = rfma(-ujx, ir3, rfma(rx, cuk, hx));
    hy = rfma(-ujy, ir3, rfma(ry, cuk, hy));
    hz = rfma(-ujz, ir3, rfma(rz, cuk, hz));
    fx = rfma(ujx, cuj, rfma(rx, cr, fx));
    fy = rfma(ujy, cuj, rfma(ry, cr, fy));
    fz = rfma(ujz, cuj, rfma(rz, cr, fz));
    c = padd(c, cuk);
}

// The traversal's pair terms: FP64 takes the form above with u_k factored out
// (fewer FP64 operations, the scarce ones on this part); FP32 keeps dipole()'s,
// whose extra operations measured no slower than the accumulator they save, and
// in the plain and counting walks with every operation written out (with the
// dipole-position terms around it that order costs 4 %: left to the compiler).
// A pair at r2 = 0 adds nothing in either.
template <bool QUAD>
__device__ __forceinline__ void walk_pair(float rx, float ry, float rz, float r2, float ukx,
                                          float uky, float ukz, float ujx, float ujy, float ujz,
                                          float& hx, float& hy, float& hz, float& fx, float& fy,
                                          float& fz, float&)
{
    if (QUAD) {
        if (r2 > 0.0f)
            dipole<float>(rx, ry, rz, r2, ukx, uky, ukz, ujx, ujy, ujz, hx, hy, hz, fx, fy, fz);
    } else if (r2 > 0.0f) {
        walk_dipole<float>(rx, ry, rz, r2, ukx, uky, ukz, ujx, ujy, ujz, hx, hy, hz, fx, fy, fz);
    }
}

template <bool QUAD>
__device__ __forceinline__ void walk_pair(double rx, double ry, double rz, double r2, double ukx,
                                          double uky, double ukz, double ujx, double ujy,
                                          double ujz, double& hx, double& hy, double& hz,
                                          double& fx, double& fy, double& fz, double& c)
{
    dipole_acc<double>(rx, ry, rz, r2, ukx, uky, ukz, ujx, ujy, ujz, hx, hy, hz, fx, fy, fz, c);
}

// Inverse powers of r shared by the derivative terms below.
template <typename R>
struct PairGeo {
    R rx, ry, rz, ir3, ir5, ir7, ir9;
};

template <typename R>
__device__ __forceinline__ PairGeo<R> pair_geo(R rx, R ry, R rz, R r2)
{
    PairGeo<R> g;
    g.rx = rx;
    g.ry = ry;
    g.rz = rz;
    const R ir = dip_rsqrt(r2);
    const R ir2 = ir * ir;
    g.ir3 = ir2 * ir;
    g.ir5 = g.ir3 * ir2;
    g.ir7 = g.ir5 * ir2;
    g.ir9 = g.ir7 * ir2;
    return g;
}

// grad phi(r; p, q) with phi = p . T(r) q (the printed force with u_k = p,
// u_j = q): 3[p (q.r) + q (p.r) + r (p.q)]/r^5 - 15 r (p.r)(q.r)/r^7, added.
template <typename R>
__device__ __forceinline__ void grad_phi_add(const PairGeo<R>& g, R px, R py, R pz, R qx, R qy,
                                             R qz, R s, R& ox, R& oy, R& oz)
{
    const R pr = px * g.rx + py * g.ry + pz * g.rz;
    const R qr = qx * g.rx + qy * g.ry + qz * g.rz;
    const R pq = px * qx + py * qy + pz * qz;
    const R a = R(3) * g.ir5 * s;
    const R c = (R(3) * pq * g.ir5 - R(15) * pr * qr * g.ir7) * s;
    ox += a * (px * qr + qx * pr) + c * g.rx;
    oy += a * (py * qr + qy * pr) + c * g.ry;
    oz += a * (pz * qr + qz * pr) + c * g.rz;
}

// T(r) p = [3 r (p.r) - p r^2]/r^5, scaled by s and added.
template <typename R>
__device__ __forceinline__ void t_apply_add(const PairGeo<R>& g, R px, R py, R pz, R s, R& ox,
                                            R& oy, R& oz)
{
    const R pr = px * g.rx + py * g.ry + pz * g.rz;
    const R a = R(3) * pr * g.ir5 * s, b = g.ir3 * s;
    ox += a * g.rx - b * px;
    oy += a * g.ry - b * py;
    oz += a * g.rz - b * pz;
}

// H phi(r; p, q) v, the derivative of grad phi(r; p, q) along v:
//   3[(p.v) q + (q.v) p + (p.q) v]/r^5
//   - 15 [r((p.v)(q.r) + (q.v)(p.r) + (r.v)(p.q)) + v (p.r)(q.r) + (r.v)(p (q.r) + q (p.r))]/r^7
//   + 105 r (r.v)(p.r)(q.r)/r^9,   scaled by s and added.
template <typename R>
__device__ __forceinline__ void hess_phi_add(const PairGeo<R>& g, R px, R py, R pz, R qx, R qy,
                                             R qz, R vx, R vy, R vz, R s, R& ox, R& oy, R& oz)
{
    const R pr = px * g.rx + py * g.ry + pz * g.rz;
    const R qr = qx * g.rx + qy * g.ry + qz * g.rz;
    const R rv = g.rx * vx + g.ry * vy + g.rz * vz;
    const R pv = px * vx + py * vy + pz * vz;
    const R qv = qx * vx + qy * vy + qz * vz;
    const R pq = px * qx + py * qy + pz * qz;
    const R a5 = R(3) * g.ir5 * s;
    const R a7 = R(15) * g.ir7 * s;
    const R cr = -a7 * (pv * qr + qv * pr + rv * pq) + R(105) * rv * pr * qr * g.ir9 * s;
    const R cv = a5 * pq - a7 * pr * qr;
    const R cp = a5 * qv - a7 * rv * qr;
    const R cq = a5 * pv - a7 * rv * pr;
    ox += cr * g.rx + cv * vx + cp * px + cq * qx;
    oy += cr * g.ry + cv * vy + cp * py + cq * qy;
    oz += cr * g.rz + cv * vz + cp * pz + cq * qz;
}

}  // namespace ffk
