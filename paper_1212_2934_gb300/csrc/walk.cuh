// Device functions shared by the traversal kernels: the Lennard-Jones pair, the
// opening test, and the shape of a persistent grid.
#pragma once

#include <mutex>

#include "dipole.cuh"
#include "ffk.cuh"

namespace ffk {

namespace {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ float rsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double rsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ float radd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double radd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float rmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double rmul(double a, double b) { return __dmul_rn(a, b); }

// Knuth's TwoSum: s + e == a + b exactly (no fused or reordered operations).
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e)
{
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// sigma^2 - r^2 without the cancellation error of the rounded r^2.  In FP32
// each square is split exactly into its rounded value and the remainder an fma
// recovers, the rounded squares are added with TwoSum so that their rounding
// errors are kept too, and sigma^2 enters as an unevaluated pair (hi, lo): the
// result carries one final rounding relative to the difference itself.  In
// FP64 the plain difference is accurate far beyond the parity bars.
__device__ __forceinline__ float sigma2_minus_r2(const FieldParams<float>& fp, float rx, float ry,
                                                 float rz)
{
    // streamed so that few temporaries are live at once: t gathers every
    // rounding error, a the rounded sum of squares
    float a = __fmul_rn(rx, rx);
    float t = __fmaf_rn(rx, rx, -a);
    float p = __fmul_rn(ry, ry);
    t = __fadd_rn(t, __fmaf_rn(ry, ry, -p));
    float e;
    two_sum(a, p, a, e);
    t = __fadd_rn(t, e);
    p = __fmul_rn(rz, rz);
    t = __fadd_rn(t, __fmaf_rn(rz, rz, -p));
    two_sum(a, p, a, e);
    t = __fadd_rn(t, e);
    two_sum(fp.lj_sigma2, -a, a, e);
    return __fadd_rn(a, __fsub_rn(__fadd_rn(e, fp.lj_sigma2_lo), t));
}

__device__ __forceinline__ double sigma2_minus_r2(const FieldParams<double>& fp, double rx, double ry,
                                                  double rz)
{
    return rsub(fp.lj_sigma2, pair_r2(rx, ry, rz));
}

// Printed LJ force (Sec. 2, Eq. LJ) inside the cut, and half the pair
// energy 2 eps (s/r)^12 - 4 eps (s/r)^6 shifted to zero at the cut.  Whether
// the pair is inside is decided on r^2 = (rx rx + ry ry) + rz rz with every
// operation rounded once (r2 from the field code may carry fused rounding);
// that exact value is formed only near the cut.  Near contact (r ~ sigma) the
// bracket (s/r)^12 - (s/r)^6 is a small difference of two numbers near one, so
// it is formed as s6 (s6 - 1) with s6 - 1 = (s2 - 1)(s2^2 + s2 + 1) and
// s2 - 1 = (sigma^2 - r^2) / r^2, the difference compensated below
// r^2 = 1.5 sigma^2; beyond, sigma^2 - r^2 is at least a third of r^2 and the
// plain difference of the rounded r^2 is accurate to a few ulps.
template <typename R>
__device__ __forceinline__ void lj(const FieldParams<R>& fp, R rx, R ry, R rz, R r2, R& fx, R& fy,
                                   R& fz, R& e)
{
    if (!(r2 < fp.lj_rcut2_hi)) return;
    const R r2e = radd(radd(rmul(rx, rx), rmul(ry, ry)), rmul(rz, rz));
    if (!(r2e < fp.lj_rcut2 && r2e > R(0))) return;
    const R ir2 = R(1) / r2e;
    const R dsr = r2e < R(1.5) * fp.lj_sigma2 ? sigma2_minus_r2(fp, rx, ry, rz)
                                              : rsub(fp.lj_sigma2, r2e);
    const R s2m1 = pmul(dsr, ir2);
    const R s2 = radd(R(1), s2m1);
    const R q = pmul(s2, s2);
    const R s6 = pmul(q, s2);
    const R s6m1 = pmul(s2m1, radd(radd(q, s2), R(1)));
    const R c = pmul(pmul(fp.lj_eps24, pmul(s6, s6m1)), ir2);
    fx = rfma(c, rx, fx);
    fy = rfma(c, ry, fy);
    fz = rfma(c, rz, fz);
    e += R(0.5) * (fp.lj_e2 * s6 * s6 - fp.lj_e4 * s6 - fp.lj_shift);
}

// Opening test in the tree precision, each operation rounded once:
// side^2 < theta^2 ((dx dx + dy dy) + dz dz), and with LJ on, the distance
// from the particle to the cell's cube is at least rcut.  Beyond far2 =
// far2_of(rcut, reach) from the centre (reach: the largest distance from the
// centre to a point of the cube) the exact test cannot fail; the aggregation
// stores far2 with each cell's moment sum.
// (dx, dy, dz) = x - c, each component rounded once.
template <typename R>
__device__ __forceinline__ bool accept(const FieldParams<R>& fp, R dx, R dy, R dz, const vec4<R>& x,
                                       const vec4<R>& c, const vec4<R>* __restrict__ lo_arr, int i,
                                       R far2)
{
    const R d2 = radd(radd(rmul(dx, dx), rmul(dy, dy)), rmul(dz, dz));
    // c.w holds side^2, rounded once
    if (!(c.w < rmul(fp.theta2, d2))) return false;
    if (fp.use_rcut) {
        // the cube is at least d - reach away
        if (d2 >= far2) return true;
        const vec4<R> lo = lo_arr[i];
        const R side = lo.w;
        R t[3];
        const R xs[3] = {x.x, x.y, x.z};
        const R ls[3] = {lo.x, lo.y, lo.z};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const R hi = radd(ls[a], side);
            const R below = rsub(ls[a], xs[a]);
            const R above = rsub(xs[a], hi);
            const R m = below > R(0) ? below : R(0);
            t[a] = above > m ? above : m;
        }
        const R b2 = radd(radd(rmul(t[0], t[0]), rmul(t[1], t[1])), rmul(t[2], t[2]));
        if (b2 < fp.rcut2) return false;
    }
    return true;
}

template <typename R>
__device__ __forceinline__ bool accept(const FieldParams<R>& fp, const vec4<R>& x, const vec4<R>& c,
                                       const vec4<R>* __restrict__ lo_arr, int i, R far2)
{
    return accept<R>(fp, rsub(x.x, c.x), rsub(x.y, c.y), rsub(x.z, c.z), x, c, lo_arr, i, far2);
}

// Shape of a persistent grid on the current device: one work segment per SM
// (at most kWorkSegments) and as many blocks as fit at once.  `occupancy`
// configures the caller's kernel and returns its resident blocks per SM; each
// kernel instance keeps its own per-device cache, guarded by its own mutex.
struct PersistentGrid {
    int blocks = 0;
    int nseg = 0;
};
constexpr int kMaxDevices = 64;

template <typename F>
PersistentGrid persistent_grid(PersistentGrid* cache, std::mutex& mu, F occupancy)
{
    int dev = 0;
    cudaGetDevice(&dev);
    const bool cached = dev >= 0 && dev < kMaxDevices;
    std::lock_guard<std::mutex> lock(mu);
    if (cached && cache[dev].blocks > 0) return cache[dev];
    PersistentGrid g;
    int nsm = 0;
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    int per_sm = occupancy();
    if (per_sm < 1) per_sm = 1;
    if (nsm < 1) nsm = 1;
    if (nsm > kWorkSegments) nsm = kWorkSegments;
    g.nseg = nsm;
    g.blocks = per_sm * nsm;
    if (cached) cache[dev] = g;
    return g;
}

}  // namespace

}  // namespace ffk
