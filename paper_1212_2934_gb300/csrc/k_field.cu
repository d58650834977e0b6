// Dipolar field and force kernels: the Barnes-Hut traversal (Sec. 3.2,
// kernel 5 of the paper's scheme, redesigned) and the all-pairs sum
// (Sec. 3.1, Algorithm 1).
//
// Traversal: a warp serves 32 consecutive particles of the Morton order,
// split into groups of G lanes.  Each lane keeps its own position in the
// depth-first cell list (`nxt`); a group visits cell i = min over its lanes
// of nxt, and only the lanes whose nxt == i act on it.  A lane therefore
// makes exactly the decisions of its own per-particle traversal, in the
// same order (children in octant order), while the cell record is fetched
// once per group (a broadcast load).  Large groups share more loads; small
// groups waste fewer lane slots on cells only some lanes need.  Skip
// pointers replace a stack.  Every lane's nxt strictly increases, so the
// loop ends after at most ncells visits per group.  Small FP32 contexts
// (k_walk.cu) and FP64 ones (k_walk64.cu) have walks of their own, which these
// launchers choose by size, type and options.
#include "walk.cuh"

namespace ffk {

namespace {

// Derivative terms of one LJ pair for a vector-Jacobian product: the pair
// enters L = sum bbar . f through c (bbar_k - bbar_j) . r with c = 24 eps
// (s^12 - s^6) / r^2, whose r-derivative is c db + 2 c'(r^2) (db . r) r,
// c' = 24 eps s^6 (4 - 7 s^6) / r^4 (the same cut and bracket as lj()).
template <typename R>
__device__ __forceinline__ void lj_vjp(const FieldParams<R>& fp, R rx, R ry, R rz, R r2, R dbx,
                                       R dby, R dbz, R& dx, R& dy, R& dz)
{
    if (!(r2 < fp.lj_rcut2_hi)) return;
    const R r2e = radd(radd(rmul(rx, rx), rmul(ry, ry)), rmul(rz, rz));
    if (!(r2e < fp.lj_rcut2 && r2e > R(0))) return;
    const R ir2 = R(1) / r2e;
    const R s2m1 = sigma2_minus_r2(fp, rx, ry, rz) * ir2;
    const R s2 = R(1) + s2m1;
    const R s6 = s2 * s2 * s2;
    const R s6m1 = s2m1 * (s2 * s2 + s2 + R(1));
    const R c = fp.lj_eps24 * (s6 * s6m1) * ir2;
    const R cp = fp.lj_eps24 * s6 * (R(4) - R(7) * s6) * ir2 * ir2;
    const R k = R(2) * cp * (dbx * rx + dby * ry + dbz * rz);
    dx += c * dbx + k * rx;
    dy += c * dby + k * ry;
    dz += c * dbz + k * rz;
}

// Dipole-position (quadrupole) term of an accepted cell (an option beyond the
// paper's pseudo-particles): with S the symmetric part of sum (rho_i - c) (x) u_i
// and m its trace (q1 = (S_xx, S_yy, S_zz, S_xy), q2 = (S_xz, S_yz, m, 0)) and
// Phi(r) = (3 r.S.r - m r^2) / r^5, the field gains -grad Phi and the force
// -H Phi u_k:
//   grad Phi = 6 S r / r^5 + r (3 m / r^5 - 15 q / r^7),           q = r.S.r
//   H Phi u  = 6 S u / r^5 - 30 (r.u) S r / r^7
//            + r (105 q (r.u) / r^9 - 30 (S r.u) / r^7 - 15 m (r.u) / r^7)
//            + u (3 m / r^5 - 15 q / r^7)
template <typename R>
__device__ __forceinline__ void quad_term(R rx, R ry, R rz, R r2, const vec4<R>& q1,
                                          const vec4<R>& q2, R ux, R uy, R uz, R& hx, R& hy,
                                          R& hz, R& fx, R& fy, R& fz)
{
    const PairGeo<R> g = pair_geo<R>(rx, ry, rz, r2);
    const R srx = q1.x * rx + q1.w * ry + q2.x * rz;
    const R sry = q1.w * rx + q1.y * ry + q2.y * rz;
    const R srz = q2.x * rx + q2.y * ry + q1.z * rz;
    const R sux = q1.x * ux + q1.w * uy + q2.x * uz;
    const R suy = q1.w * ux + q1.y * uy + q2.y * uz;
    const R suz = q2.x * ux + q2.y * uy + q1.z * uz;
    const R q = rx * srx + ry * sry + rz * srz;
    const R ru = rx * ux + ry * uy + rz * uz;
    const R sru = srx * ux + sry * uy + srz * uz;
    const R m = q2.z;
    const R c6 = R(6) * g.ir5;
    const R cmq = R(3) * m * g.ir5 - R(15) * q * g.ir7;
    hx -= c6 * srx + cmq * rx;
    hy -= c6 * sry + cmq * ry;
    hz -= c6 * srz + cmq * rz;
    const R cs = R(30) * ru * g.ir7;
    const R cr = R(105) * q * ru * g.ir9 - R(30) * sru * g.ir7 - R(15) * m * ru * g.ir7;
    fx -= c6 * sux - cs * srx + cr * rx + cmq * ux;
    fy -= c6 * suy - cs * sry + cr * ry + cmq * uy;
    fz -= c6 * suz - cs * srz + cr * rz + cmq * uz;
}

// Preferred shared-memory share of the traversal (percent of the maximum):
// 7 % selects 16 KB, room for the per-block reservation of the resident
// blocks; the rest of the unified storage serves as L1 cache.
#ifndef FFK_TRAVERSE_CARVEOUT
#define FFK_TRAVERSE_CARVEOUT 7
#endif
constexpr int kTraverseCarveout = FFK_TRAVERSE_CARVEOUT;

// Traversal block shape: warps work independently (no shared memory, no
// block barrier), so the block size only sets how registers and warps are
// traded.  Registers are allocated per SM sub-partition (16384 each, a warp
// taking 32 x its registers), so 128 x 10 allows 48 registers a thread, room
// for the whole walk without spills.  The plain FP32 walk is lean enough for
// 128 x 12 (40 registers, 48 warps) with a few spilled words, and measures
// slightly faster so; the other walks keep 10 blocks.  The walk with
// dipole-position terms also has a shape with more registers (54 a thread with 8
// blocks asked for, 36 warps an SM): see quad_few_warps().
#ifndef FFK_BH_THREADS
#define FFK_BH_THREADS 128
#endif
#ifndef FFK_BH_MIN_BLOCKS
#define FFK_BH_MIN_BLOCKS 10
#endif
#ifndef FFK_BH_MIN_BLOCKS_LEAN
#define FFK_BH_MIN_BLOCKS_LEAN 12
#endif
constexpr int kBhThreads = FFK_BH_THREADS;
constexpr int kBhMinBlocks = FFK_BH_MIN_BLOCKS;
constexpr int kBhMinBlocksQuadFew = 8;

// FP64 walks hold twice the registers per value.
#ifndef FFK_BH_MIN_BLOCKS_FP64
#define FFK_BH_MIN_BLOCKS_FP64 6
#endif

template <typename R, bool COUNT, bool QUAD>
constexpr int bh_min_blocks()
{
    return sizeof(R) == 8 ? FFK_BH_MIN_BLOCKS_FP64
           : (!COUNT && !QUAD) ? FFK_BH_MIN_BLOCKS_LEAN
                               : FFK_BH_MIN_BLOCKS;
}
static_assert(kBhThreads % 32 == 0, "whole warps");

// The walks that also write the source lists need a few more registers than
// the counting walk: 8 blocks of 128 (64 registers) in FP32.
#ifndef FFK_BH_MIN_BLOCKS_REC
#define FFK_BH_MIN_BLOCKS_REC 8
#endif
template <typename R>
constexpr int bh_rec_min_blocks()
{
    return sizeof(R) == 8 ? FFK_BH_MIN_BLOCKS_FP64 : FFK_BH_MIN_BLOCKS_REC;
}

// Minimum of v over each aligned group of G lanes.
template <int G>
__device__ __forceinline__ unsigned group_min(unsigned v)
{
    if (G == 32) return __reduce_min_sync(kFull, v);
#pragma unroll
    for (int o = 1; o < G; o <<= 1) v = min(v, __shfl_xor_sync(kFull, v, o, G));
    return v;
}

// One task: the 32 consecutive particles task*32 .. task*32+31 of the key order.
template <typename R, bool COUNT, int G>
__device__ __forceinline__ void bh_task(int task, const vec4<R>* __restrict__ pos,
                                        const vec4<R>* __restrict__ u, int n, const Tree<R>& t,
                                        const FieldParams<R>& fp, unsigned ncells,
                                        vec4<R>* __restrict__ h, vec4<R>* __restrict__ f,
                                        R* __restrict__ esr, int4* __restrict__ counts, int* flags,
                                        const uint32_t* __restrict__ off, const Segs& sg)
{
    const int lane = threadIdx.x & 31;
    const int k = task * 32 + lane;
    const bool active = k < n;
    vec4<R> xk, uk;
    if (active) {
        xk = pos[k];
        uk = u[k];
    } else {
        xk.x = xk.y = xk.z = xk.w = R(0);
        uk = xk;
    }
    R hx = 0, hy = 0, hz = 0, fx = 0, fy = 0, fz = 0, sx = 0, sy = 0, sz = 0, es = 0, ck = 0;
    int nacc = 0, npair = 0, nopen = 0;
    // the cells of this particle's system: [first, end)
    unsigned first = 0, end = ncells;
    if (sg.of_pos && active) {
        const int sys = (int)sg.of_pos[k];
        first = off[sg.start[sys]];
        end = off[sg.start[sys + 1]];
    }
    unsigned nxt = active && first < end ? first : 0xffffffffu;
    for (;;) {
        const unsigned i = group_min<G>(nxt);
        if (G == 32) {
            if (i >= ncells) break;
        } else if (!__any_sync(kFull, i < ncells)) {
            break;
        }
        // a finished group keeps looping with i >= ncells while other groups of
        // the warp still work; its lanes must not touch cell i then
        if (nxt == i && i < ncells) {
            const Cell<R> cl = t.cell[i];
            const int4 nd = cl.node;
            const bool inside = nd.x <= k && k < nd.y;
            const bool leaf = (nd.w >> 8) != 0;
            const bool single = (nd.w >> 9) != 0;  // a one-particle leaf
            const vec4<R> c = cl.cen;
            const vec4<R> m = t.mom[i];  // .w: the cell's far2
            const bool acc = !inside && accept<R>(fp, xk, c, t.lo, (int)i, m.w);
            if (acc || (single && !inside)) {
                // the cell's pseudo-particle; for a one-particle leaf it is the
                // particle itself (centre and moment sum of one term are exact)
                const R rx = xk.x - c.x, ry = xk.y - c.y, rz = xk.z - c.z;
                const R r2 = pair_r2(rx, ry, rz);
                walk_pair<false>(rx, ry, rz, r2, uk.x, uk.y, uk.z, m.x, m.y, m.z, hx, hy, hz, fx, fy,
                              fz, ck);
                if (acc) {
                    if (COUNT) ++nacc;
                } else {
                    if (fp.include_sr) lj<R>(fp, rx, ry, rz, r2, sx, sy, sz, es);
                    if (COUNT) ++npair;
                }
                nxt = (unsigned)nd.z;
            } else if (leaf) {
                if (!single) {
                    for (int s = nd.x; s < nd.y; ++s) {
                        if (s == k) continue;
                        const vec4<R> xj = pos[s], uj = u[s];
                        const R rx = xk.x - xj.x, ry = xk.y - xj.y, rz = xk.z - xj.z;
                        const R r2 = pair_r2(rx, ry, rz);
                        if (r2 > R(0)) {
                            walk_pair<false>(rx, ry, rz, r2, uk.x, uk.y, uk.z, uj.x, uj.y, uj.z, hx,
                                          hy, hz, fx, fy, fz, ck);
                            if (fp.include_sr) lj<R>(fp, rx, ry, rz, r2, sx, sy, sz, es);
                        }
                        if (COUNT) ++npair;
                    }
                }
                nxt = (unsigned)nd.z;
            } else {
                if (COUNT) ++nopen;
                nxt = i + 1;
            }
            if (nxt <= i) {  // skip pointers must move forward
                atomicOr(flags, FLAG_TRAVERSE);
                nxt = 0xffffffffu;
            }
            if (nxt >= end) nxt = 0xffffffffu;  // this lane's system is done
        }
    }
    if (!active) return;
    vec4<R> ho, fo;
    ho.x = fp.dip_scale * hx;
    ho.y = fp.dip_scale * hy;
    ho.z = fp.dip_scale * hz;
    ho.w = R(0);
    fo.x = fp.dip_scale * (fx + uk.x * ck) + sx;
    fo.y = fp.dip_scale * (fy + uk.y * ck) + sy;
    fo.z = fp.dip_scale * (fz + uk.z * ck) + sz;
    fo.w = R(0);
    h[k] = ho;
    f[k] = fo;
    if (esr) esr[k] = es;
    if (COUNT) counts[k] = make_int4(nacc, npair, nopen, 0);
}

// A particle's source list in the entry pool: chunk k first, then chunks taken
// from *next.  Sources are kept four at a time and stored as one 16-byte word
// (a chunk holds a multiple of four); the chunk after a full one is taken at
// once.  Nothing is written to chunks at or past cap.
struct ChunkWriter {
    const EntryPool& p;   // the kernel's parameter: read where used, not held
    uint32_t ck, f;       // current chunk, sources so far
    uint32_t s0, s1, s2;  // the current group of four so far

    __device__ __forceinline__ ChunkWriter(const EntryPool& pool, uint32_t own)
        : p(pool), ck(own), f(0), s0(0), s1(0), s2(0)
    {
    }
    __device__ __forceinline__ void put(uint32_t key)
    {
        const uint32_t q = f & 3u;
        if (q == 0u) {
            s0 = key;
        } else if (q == 1u) {
            s1 = key;
        } else if (q == 2u) {
            s2 = key;
        } else {
            const uint32_t o = f & (uint32_t)(kPoolChunk - 1);
            if (ck < p.cap)
                *reinterpret_cast<uint4*>(p.keys + (size_t)ck * kPoolChunk + (o - 3u)) =
                    make_uint4(s0, s1, s2, key);
            if (o == (uint32_t)(kPoolChunk - 1)) {
                const uint32_t nk = p.first + atomicAdd(p.next, 1u);
                if (ck < p.cap) p.link[ck] = nk;
                ck = nk;
            }
        }
        ++f;
    }
    // the last, incomplete group
    __device__ __forceinline__ void flush()
    {
        const uint32_t r = f & 3u;
        if (r == 0u || ck >= p.cap) return;
        uint32_t* q = p.keys + (size_t)ck * kPoolChunk + ((f - r) & (uint32_t)(kPoolChunk - 1));
        q[0] = s0;
        if (r > 1u) q[1] = s1;
        if (r > 2u) q[2] = s2;
    }
};

// pair_r2() with the last operation left for the compiler to fuse (it can only be
// the same one), for the particles of opened leaves: written out there, it cost
// fields with leaves of several particles 1 % (1,048,576 particles, leaf_max 8, theta
// 0.6: 5.69 ms, so 5.65).  In the cell's own r^2 it is the other way round
// (150,000 particles, leaf_max 1, theta 0.4: 1.682 ms written out, 1.695 so).
template <typename R>
__device__ __forceinline__ R lane_r2(R rx, R ry, R rz)
{
    return rfma(rx, rx, ry * ry) + rz * rz;
}

// Independent per-lane walk (group size 1): each lane follows its own path
// through the cell list; no vote or shuffle per visited cell.  With REC (and
// COUNT) each source also goes to the particle's list in the entry pool.
template <typename R, bool COUNT, bool QUAD, bool REC = false>
__device__ __forceinline__ void bh_task1(int task, const vec4<R>* __restrict__ pos,
                                         const vec4<R>* __restrict__ u, int n, const Tree<R>& t,
                                         const FieldParams<R>& fp, unsigned ncells,
                                         vec4<R>* __restrict__ h, vec4<R>* __restrict__ f,
                                         R* __restrict__ esr, int4* __restrict__ counts, int* flags,
                                         const uint32_t* __restrict__ off, const Segs& sg,
                                         const EntryPool& ep = EntryPool())
{
    static_assert(!REC || (COUNT && !QUAD), "sources are recorded by the counting walk");
    const int lane = threadIdx.x & 31;
    const int k = task * 32 + lane;
    if (k >= n) return;
    ChunkWriter cw(ep, (uint32_t)k);
    const vec4<R> xk = pos[k], uk = u[k];
    R hx = 0, hy = 0, hz = 0, fx = 0, fy = 0, fz = 0, sx = 0, sy = 0, sz = 0, es = 0, ck = 0;
    int nacc = 0, npair = 0, nopen = 0;
    // the cells of this particle's system: [i, end)
    unsigned i = 0, end = ncells;
    if (sg.of_pos) {
        const int sys = (int)sg.of_pos[k];
        i = off[sg.start[sys]];
        end = off[sg.start[sys + 1]];
    }
    while (i < end) {
        const Cell<R> cl = t.cell[i];
        // requested with the cell so that one latency covers both loads; .w is
        // the cell's far2 for the opening test
        const vec4<R> m = t.mom[i];
        const int4 nd = cl.node;
        const bool inside = nd.x <= k && k < nd.y;
        const bool leaf = (nd.w >> 8) != 0;
        const bool single = (nd.w >> 9) != 0;  // a one-particle leaf
        const vec4<R> c = cl.cen;
        // the separation serves the opening test (each component rounded once
        // either way) and the pair terms
        const R rx = rsub(xk.x, c.x), ry = rsub(xk.y, c.y), rz = rsub(xk.z, c.z);
        const R r2 = QUAD ? rx * rx + ry * ry + rz * rz : pair_r2(rx, ry, rz);
        const bool out1 = single && !inside;
        // A one-particle leaf adds the same dipole term whether accepted or
        // summed as a pair; the two differ only by the LJ term, which is zero
        // unless r2 < lj_rcut2_hi, and in the counts.  Below lj_rcut2_lo the
        // particle, and so its cube, is within rcut (by a margin far above the
        // rounding of the cube's corners): the opening test fails.  The plain
        // walk therefore decides such a leaf only in between.
        const bool acc =
            (!COUNT && !QUAD && out1)
                ? (fp.include_sr && r2 < fp.lj_rcut2_hi && r2 >= fp.lj_rcut2_lo &&
                   accept<R>(fp, rx, ry, rz, xk, c, t.lo, (int)i, m.w))
                : (!inside && accept<R>(fp, rx, ry, rz, xk, c, t.lo, (int)i, m.w));
        unsigned nxt = i + 1;
        if (acc || out1) {
            // the cell's pseudo-particle; for a one-particle leaf it is the
            // particle itself (centre and moment sum of one term are exact)
            walk_pair<QUAD>(rx, ry, rz, r2, uk.x, uk.y, uk.z, m.x, m.y, m.z, hx, hy, hz, fx, fy, fz,
                          ck);
            if (REC) cw.put(i + (uint32_t)nd.x);
            if (QUAD && acc && r2 > R(0))
                quad_term<R>(rx, ry, rz, r2, t.q1[i], t.q2[i], uk.x, uk.y, uk.z, hx, hy, hz, fx,
                             fy, fz);
            if (acc) {
                if (COUNT) ++nacc;
            } else {
                if (fp.include_sr) lj<R>(fp, rx, ry, rz, r2, sx, sy, sz, es);
                if (COUNT) ++npair;
            }
            nxt = (unsigned)nd.z;
        } else if (leaf) {
            if (!single) {
                for (int s = nd.x; s < nd.y; ++s) {
                    if (s == k) continue;
                    if (REC) cw.put(i + 1u + (uint32_t)s);
                    const vec4<R> xj = pos[s], uj = u[s];
                    const R rx = xk.x - xj.x, ry = xk.y - xj.y, rz = xk.z - xj.z;
                    const R r2 = QUAD ? pair_r2(rx, ry, rz) : lane_r2(rx, ry, rz);
                    if (r2 > R(0)) {
                        walk_pair<QUAD>(rx, ry, rz, r2, uk.x, uk.y, uk.z, uj.x, uj.y, uj.z, hx, hy,
                                      hz, fx, fy, fz, ck);
                        if (fp.include_sr) lj<R>(fp, rx, ry, rz, r2, sx, sy, sz, es);
                    }
                    if (COUNT) ++npair;
                }
            }
            nxt = (unsigned)nd.z;
        } else {
            if (COUNT) ++nopen;
        }
        if (nxt <= i) {  // skip pointers must move forward
            atomicOr(flags, FLAG_TRAVERSE);
            break;
        }
        i = nxt;
    }
    if (REC) cw.flush();
    vec4<R> ho, fo;
    ho.x = fp.dip_scale * hx;
    ho.y = fp.dip_scale * hy;
    ho.z = fp.dip_scale * hz;
    ho.w = R(0);
    fo.x = fp.dip_scale * (fx + uk.x * ck) + sx;
    fo.y = fp.dip_scale * (fy + uk.y * ck) + sy;
    fo.z = fp.dip_scale * (fz + uk.z * ck) + sz;
    fo.w = R(0);
    h[k] = ho;
    f[k] = fo;
    if (esr) esr[k] = es;
    if (COUNT) counts[k] = make_int4(nacc, npair, nopen, 0);
}

// Target-side terms of a vector-Jacobian product of h and f (cotangents abar,
// bbar) for L = sum abar . h + bbar . f, on the walk of bh_task1 (the same
// decisions in the same order):
//   dL/du_k   += ds grad phi(r; bbar_k, w_s)
//   dL/drho_k += ds [grad phi(r; abar_k, w_s) + H phi(r; u_k, w_s) bbar_k] + LJ terms
// written to dxt, dut; the source-side terms come from the source records.
template <typename R>
struct VjpIn {
    const vec4<R>* u;
    const vec4<R>* abar;
    const vec4<R>* bbar;
    vec4<R>* dxt;
    vec4<R>* dut;
};

template <typename R>
__device__ __forceinline__ void vjp_target(const FieldParams<R>& fp, const vec4<R>& xk,
                                           const vec4<R>& uk, const vec4<R>& ak,
                                           const vec4<R>& bk, const vec4<R>& xs,
                                           const vec4<R>& ws, R& dx, R& dy, R& dz, R& ux, R& uy,
                                           R& uz)
{
    const R rx = xk.x - xs.x, ry = xk.y - xs.y, rz = xk.z - xs.z;
    const R r2 = rx * rx + ry * ry + rz * rz;
    if (!(r2 > R(0))) return;
    const PairGeo<R> g = pair_geo<R>(rx, ry, rz, r2);
    const R ds = fp.dip_scale;
    grad_phi_add<R>(g, bk.x, bk.y, bk.z, ws.x, ws.y, ws.z, ds, ux, uy, uz);
    grad_phi_add<R>(g, ak.x, ak.y, ak.z, ws.x, ws.y, ws.z, ds, dx, dy, dz);
    hess_phi_add<R>(g, uk.x, uk.y, uk.z, ws.x, ws.y, ws.z, bk.x, bk.y, bk.z, ds, dx, dy, dz);
}

// With REC the walk also writes each particle's sources to the entry pool and
// their number to counts[k].x (as the counting walk of the gradient pass does).
template <typename R, bool REC = false>
__device__ __forceinline__ void vjp_task(int task, const vec4<R>* __restrict__ pos, int n,
                                         const Tree<R>& t, const FieldParams<R>& fp,
                                         unsigned ncells, int* flags,
                                         const uint32_t* __restrict__ off, const Segs& sg,
                                         const VjpIn<R>& vj, int4* __restrict__ counts = nullptr,
                                         const EntryPool& ep = EntryPool())
{
    const int k = task * 32 + (threadIdx.x & 31);
    if (k >= n) return;
    ChunkWriter cw(ep, (uint32_t)k);
    int nent = 0;
    const vec4<R> xk = pos[k];
    const vec4<R> uk = vj.u[k], ak = vj.abar[k], bk = vj.bbar[k];
    R dx = 0, dy = 0, dz = 0, ux = 0, uy = 0, uz = 0;
    unsigned i = 0, end = ncells;
    if (sg.of_pos) {
        const int sys = (int)sg.of_pos[k];
        i = off[sg.start[sys]];
        end = off[sg.start[sys + 1]];
    }
    while (i < end) {
        const Cell<R> cl = t.cell[i];
        const int4 nd = cl.node;
        const bool inside = nd.x <= k && k < nd.y;
        const bool leaf = (nd.w >> 8) != 0;
        const bool single = (nd.w >> 9) != 0;  // a one-particle leaf
        const vec4<R> ws = t.mom[i];  // moment sum; .w: the cell's far2
        const bool out1 = single && !inside;
        const R rx = rsub(xk.x, cl.cen.x), ry = rsub(xk.y, cl.cen.y), rz = rsub(xk.z, cl.cen.z);
        const R r2 = rx * rx + ry * ry + rz * rz;
        // A one-particle leaf gives the same dipole terms whether accepted or
        // summed as a pair; only the LJ term differs, and it vanishes outside
        // [lj_rcut2_lo, lj_rcut2_hi) (see bh_task1), so it is decided only there.
        const bool acc =
            out1 ? (fp.include_sr && r2 < fp.lj_rcut2_hi && r2 >= fp.lj_rcut2_lo &&
                    accept<R>(fp, rx, ry, rz, xk, cl.cen, t.lo, (int)i, ws.w))
                 : (!inside && accept<R>(fp, rx, ry, rz, xk, cl.cen, t.lo, (int)i, ws.w));
        unsigned nxt = i + 1;
        if (acc || out1) {
            if (REC) {
                cw.put(i + (uint32_t)nd.x);
                ++nent;
            }
            vjp_target<R>(fp, xk, uk, ak, bk, cl.cen, ws, dx, dy, dz, ux, uy, uz);
            if (!acc && fp.include_sr) {
                const vec4<R> bj = vj.bbar[nd.x];
                lj_vjp<R>(fp, rx, ry, rz, r2, bk.x - bj.x, bk.y - bj.y, bk.z - bj.z, dx, dy, dz);
            }
            nxt = (unsigned)nd.z;
        } else if (leaf) {
            if (!single) {
                for (int s = nd.x; s < nd.y; ++s) {
                    if (s == k) continue;
                    if (REC) {
                        cw.put(i + 1u + (uint32_t)s);
                        ++nent;
                    }
                    const vec4<R> xj = pos[s], uj = vj.u[s], bj = vj.bbar[s];
                    vjp_target<R>(fp, xk, uk, ak, bk, xj, uj, dx, dy, dz, ux, uy, uz);
                    if (fp.include_sr) {
                        const R rx = xk.x - xj.x, ry = xk.y - xj.y, rz = xk.z - xj.z;
                        const R r2 = rx * rx + ry * ry + rz * rz;
                        if (r2 > R(0))
                            lj_vjp<R>(fp, rx, ry, rz, r2, bk.x - bj.x, bk.y - bj.y, bk.z - bj.z,
                                      dx, dy, dz);
                    }
                }
            }
            nxt = (unsigned)nd.z;
        }
        if (nxt <= i) {
            atomicOr(flags, FLAG_TRAVERSE);
            break;
        }
        i = nxt;
    }
    vec4<R> o;
    o.x = dx; o.y = dy; o.z = dz; o.w = R(0);
    vj.dxt[k] = o;
    o.x = ux; o.y = uy; o.z = uz;
    vj.dut[k] = o;
    if (REC) {
        cw.flush();
        counts[k] = make_int4(nent, 0, 0, 0);
    }
}

// The target-side walk on the traversal's schedule: warps take 32-particle
// tasks from their SM's Morton segment first (see k_bh).
template <typename R, bool REC>
__global__ void __launch_bounds__(kBhThreads, (REC ? bh_rec_min_blocks<R>() : kBhMinBlocks)) k_bh_vjp(
    const vec4<R>* __restrict__ pos, int n, Tree<R> t, FieldParams<R> fp, int* flags,
    int* __restrict__ work, int nseg, const uint32_t* __restrict__ off, Segs sg, VjpIn<R> vj,
    int4* __restrict__ counts, EntryPool ep)
{
    if (*flags & FLAG_CAPACITY) return;
    const unsigned ncells = (unsigned)*t.ncells;
    const int ntask = (n + 31) / 32;
    unsigned smid;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
    const int home = (int)(smid % (unsigned)nseg);
    const int lane = threadIdx.x & 31;
    for (int probe = 0; probe < nseg; ++probe) {
        const int ws = (home + probe) % nseg;
        const int t0 = (int)((int64_t)ntask * ws / nseg);
        const int t1 = (int)((int64_t)ntask * (ws + 1) / nseg);
        for (;;) {
            int got = 0;
            if (lane == 0) got = atomicAdd(&work[ws], 1);
            got = __shfl_sync(kFull, got, 0);
            const int task = t0 + got;
            if (task >= t1) break;
            vjp_task<R, REC>(task, pos, n, t, fp, ncells, flags, off, sg, vj, counts, ep);
        }
    }
}

// Persistent traversal: the key order is cut into nseg contiguous segments of
// 32-particle tasks; a warp takes tasks from the segment of the SM it runs on
// (so warps sharing an L1 cache walk neighbouring parts of the tree) and then
// from the following segments once its own is used up.  Task counters
// (work[0..nseg)) start at zero; every task is taken exactly once.
template <typename R, bool COUNT, int G, bool QUAD, int THREADS = kBhThreads,
          int MINB = bh_min_blocks<R, COUNT, QUAD>()>
__global__ void __launch_bounds__(THREADS, MINB) k_bh(const vec4<R>* __restrict__ pos,
                                            const vec4<R>* __restrict__ u, int n, Tree<R> t,
                                            FieldParams<R> fp, vec4<R>* __restrict__ h,
                                            vec4<R>* __restrict__ f, R* __restrict__ esr,
                                            int4* __restrict__ counts, int* flags,
                                            int* __restrict__ work, int nseg,
                                            const uint32_t* __restrict__ off, Segs sg)
{
    if (*flags & FLAG_CAPACITY) return;
    const unsigned ncells = (unsigned)*t.ncells;
    const int ntask = (n + 31) / 32;
    unsigned smid;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
    const int home = (int)(smid % (unsigned)nseg);
    const int lane = threadIdx.x & 31;
    for (int probe = 0; probe < nseg; ++probe) {
        const int ws = (home + probe) % nseg;
        const int t0 = (int)((int64_t)ntask * ws / nseg);
        const int t1 = (int)((int64_t)ntask * (ws + 1) / nseg);
        for (;;) {
            int got = 0;
            if (lane == 0) got = atomicAdd(&work[ws], 1);
            got = __shfl_sync(kFull, got, 0);
            const int task = t0 + got;
            if (task >= t1) break;
            if (G == 1)
                bh_task1<R, COUNT, QUAD>(task, pos, u, n, t, fp, ncells, h, f, esr, counts, flags,
                                         off, sg);
            else
                bh_task<R, COUNT, G>(task, pos, u, n, t, fp, ncells, h, f, esr, counts, flags, off,
                                     sg);
        }
    }
}

// The counting walk that also records every particle's sources (energy
// gradient), on the schedule of k_bh.

template <typename R>
__global__ void __launch_bounds__(kBhThreads, (bh_rec_min_blocks<R>())) k_bh_rec(
    const vec4<R>* __restrict__ pos, const vec4<R>* __restrict__ u, int n, Tree<R> t,
    FieldParams<R> fp, vec4<R>* __restrict__ h, vec4<R>* __restrict__ f, R* __restrict__ esr,
    int4* __restrict__ counts, int* flags, int* __restrict__ work, int nseg,
    const uint32_t* __restrict__ off, Segs sg, EntryPool ep)
{
    if (*flags & FLAG_CAPACITY) return;
    const unsigned ncells = (unsigned)*t.ncells;
    const int ntask = (n + 31) / 32;
    unsigned smid;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
    const int home = (int)(smid % (unsigned)nseg);
    const int lane = threadIdx.x & 31;
    for (int probe = 0; probe < nseg; ++probe) {
        const int ws = (home + probe) % nseg;
        const int t0 = (int)((int64_t)ntask * ws / nseg);
        const int t1 = (int)((int64_t)ntask * (ws + 1) / nseg);
        for (;;) {
            int got = 0;
            if (lane == 0) got = atomicAdd(&work[ws], 1);
            got = __shfl_sync(kFull, got, 0);
            const int task = t0 + got;
            if (task >= t1) break;
            bh_task1<R, true, false, true>(task, pos, u, n, t, fp, ncells, h, f, esr, counts,
                                           flags, off, sg, ep);
        }
    }
}

// All pairs in FP64: one thread per target; source records staged through
// shared memory one block-sized tile at a time (Sec. 3.1, Algorithm 1).
constexpr int kApThreads = 256;

template <typename R>
__global__ void __launch_bounds__(kApThreads) k_ap(const vec4<R>* __restrict__ pos,
                                                   const vec4<R>* __restrict__ u, int n,
                                                   FieldParams<R> fp, vec4<R>* __restrict__ h,
                                                   vec4<R>* __restrict__ f, R* __restrict__ esr)
{
    __shared__ vec4<R> sp[kApThreads];
    __shared__ vec4<R> su[kApThreads];
    const int k = blockIdx.x * kApThreads + threadIdx.x;
    const bool active = k < n;
    vec4<R> xk, uk;
    if (active) {
        xk = pos[k];
        uk = u[k];
    } else {
        xk.x = xk.y = xk.z = xk.w = R(0);
        uk = xk;
    }
    // two-level sums: each tile is summed on its own, then added to the total,
    // so rounding grows with sqrt(tile) + sqrt(n / tile) terms instead of sqrt(n)
    R hx = 0, hy = 0, hz = 0, fx = 0, fy = 0, fz = 0, sx = 0, sy = 0, sz = 0, es = 0;
    for (int tile = 0; tile < n; tile += kApThreads) {
        const int j = tile + threadIdx.x;
        if (j < n) {
            sp[threadIdx.x] = pos[j];
            su[threadIdx.x] = u[j];
        }
        __syncthreads();
        const int lim = min(kApThreads, n - tile);
        R thx = 0, thy = 0, thz = 0, tfx = 0, tfy = 0, tfz = 0;
        for (int jj = 0; jj < lim; ++jj) {
            if (tile + jj == k) continue;
            const vec4<R> xj = sp[jj], uj = su[jj];
            const R rx = xk.x - xj.x, ry = xk.y - xj.y, rz = xk.z - xj.z;
            const R r2 = rx * rx + ry * ry + rz * rz;
            if (r2 > R(0)) {
                dipole<R>(rx, ry, rz, r2, uk.x, uk.y, uk.z, uj.x, uj.y, uj.z, thx, thy, thz, tfx,
                          tfy, tfz);
                if (fp.include_sr) lj<R>(fp, rx, ry, rz, r2, sx, sy, sz, es);
            }
        }
        hx += thx;
        hy += thy;
        hz += thz;
        fx += tfx;
        fy += tfy;
        fz += tfz;
        __syncthreads();
    }
    if (!active) return;
    vec4<R> ho, fo;
    ho.x = fp.dip_scale * hx;
    ho.y = fp.dip_scale * hy;
    ho.z = fp.dip_scale * hz;
    ho.w = R(0);
    fo.x = fp.dip_scale * fx + sx;
    fo.y = fp.dip_scale * fy + sy;
    fo.z = fp.dip_scale * fz + sz;
    fo.w = R(0);
    h[k] = ho;
    f[k] = fo;
    if (esr) esr[k] = es;
}

// All pairs in single precision: a block serves T targets (a lane each, 32 / T
// times over) and its warps share out the sources, 32 at a time, each warp (and
// each group of T lanes in it) a batch of its own; the groups' sums are added in
// a fixed order at the end.  One thread per target left the chip idle below
// 150,000 targets (20,011: 79 blocks of 256 on 152 SMs).  Two sources go through
// each FP32 instruction, their sums kept apart, and with the powers of 1/r outside
// the brackets the last operation of each component is one fused multiply-add
// into its sum: 41 instructions for two pairs, 82 cycles of the FP32 pipe, which
// bounds the kernel.  Every 256 sources of a warp the running sums go to the
// totals, so rounding grows with the square root of the two levels, not of n.
// 16 targets a block below kApWide (n = 4,096 still gives 256 blocks); 32 above,
// where staging a source for twice the targets saves 5 %.
constexpr int kAp2Warps = 8;
constexpr int kAp2Pair = 20;           // words per staged pair (14 used)
constexpr int kAp2Stage = 16 * kAp2Pair + 4;
constexpr int64_t kApWide = 65536;

// A target (each value twice) and its sums (two sources at a time, kept apart).
struct Ap2Target {
    float2 x, y, z, ux, uy, uz;
};
struct Ap2Sums {
    float2 hx, hy, hz, fx, fy, fz;
    float sx, sy, sz, es;
};

// This warp's share of the sources on its targets.  A source at r^2 = 0 (the
// target itself, a coincident particle) or at an undefined one (a position that
// is not a number) adds nothing.  1/r = 0 sees to that as long as the rest of
// its terms is finite; EXACT leaves the terms out one by one instead, whatever
// they are, and gives sources past the end an undefined position.
template <int T, bool EXACT>
__device__ __forceinline__ void ap2_sweep(const float4* __restrict__ pos,
                                          const float4* __restrict__ u, int n,
                                          const FieldParams<float>& fp, float* stage,
                                          const Ap2Target& k, Ap2Sums& a)
{
    constexpr int kPairs = 16 / (32 / T);  // staged pairs of each group of T lanes
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, grp = lane / T;
    // (the second group's pairs start 4 words on: other banks)
    float* mine = stage + (lane >> 1) * kAp2Pair + (lane & 1) + ((lane >> 1) >= kPairs ? 4 : 0);
    const float* own = stage + grp * (kPairs * kAp2Pair + 4);
    const float2 zero = dup2(0.0f);
    float2 thx = zero, thy = zero, thz = zero, tfx = zero, tfy = zero, tfz = zero;
    float2 hx = zero, hy = zero, hz = zero, fx = zero, fy = zero, fz = zero;
    float sx = 0.0f, sy = 0.0f, sz = 0.0f, es = 0.0f;
    const float near2 = fp.include_sr ? fp.lj_rcut2_hi : 0.0f;
    // past the end: no moment, far away
    const float far = EXACT ? __int_as_float(0x7fffffff) : 1e18f;
    const float4 none = make_float4(far, far, far, 0.0f);
    int j = w * 32 + lane;
    float4 c = j < n ? pos[j] : none, m = j < n ? u[j] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    for (int base = w * 32, it = 1; base < n; base += 32 * kAp2Warps, ++it) {
        __syncwarp();
        mine[0] = -c.x;
        mine[2] = -c.y;
        mine[4] = -c.z;
        mine[6] = m.x;
        mine[8] = m.y;
        mine[10] = m.z;
        __syncwarp();
        j += 32 * kAp2Warps;  // the next batch, under this one's arithmetic
        c = j < n ? pos[j] : none;
        m = j < n ? u[j] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        uint32_t close = 0u, one = 1u;
        const float4* q = reinterpret_cast<const float4*>(own);
#pragma unroll 2
        for (int p = 0; p < kPairs; ++p, q += kAp2Pair / 4) {
            const float4 q0 = q[0], q1 = q[1], q2 = q[2];
            const float2 rx = __fadd2_rn(k.x, make_float2(q0.x, q0.y));
            const float2 ry = __fadd2_rn(k.y, make_float2(q0.z, q0.w));
            const float2 rz = __fadd2_rn(k.z, make_float2(q1.x, q1.y));
            const float2 vx = make_float2(q1.z, q1.w), vy = make_float2(q2.x, q2.y),
                         vz = make_float2(q2.z, q2.w);
            const float2 r2 = pair_r2_2(rx, ry, rz);
            const bool in0 = r2.x > 0.0f, in1 = r2.y > 0.0f;
            const auto kept = [&](float2 v) {
                return EXACT ? make_float2(in0 ? v.x : 0.0f, in1 ? v.y : 0.0f) : v;
            };
            const float2 ir = make_float2(in0 ? dip_rsqrt(r2.x) : 0.0f, in1 ? dip_rsqrt(r2.y) : 0.0f);
            const float2 ir2 = __fmul2_rn(ir, ir);
            const float2 ir3 = __fmul2_rn(ir2, ir);
            const float2 p3 = __fmul2_rn(dup2(3.0f), ir2);
            const float2 bj = __ffma2_rn(vz, rz, __ffma2_rn(vy, ry, __fmul2_rn(vx, rx)));
            const float2 bk = __ffma2_rn(k.uz, rz, __ffma2_rn(k.uy, ry, __fmul2_rn(k.ux, rx)));
            const float2 ab = __ffma2_rn(vz, k.uz, __ffma2_rn(vy, k.uy, __fmul2_rn(vx, k.ux)));
            // h += [3 r (u_j.r) / r^2 - u_j] / r^3
            const float2 qh = __fmul2_rn(p3, bj);
            const float2 nir3 = make_float2(-ir3.x, -ir3.y);
            const float2 nqh = make_float2(-qh.x, -qh.y);
            thx = __ffma2_rn(nir3, kept(__ffma2_rn(rx, nqh, vx)), thx);
            thy = __ffma2_rn(nir3, kept(__ffma2_rn(ry, nqh, vy)), thy);
            thz = __ffma2_rn(nir3, kept(__ffma2_rn(rz, nqh, vz)), thz);
            // f += 3 / r^5 {r [u_j.u_k - 5 (u_k.r)(u_j.r) / r^2] + u_k (u_j.r) + u_j (u_k.r)}
            const float2 g = __fmul2_rn(p3, ir3);
            const float2 wv = __ffma2_rn(__fmul2_rn(dup2(-5.0f), ir2), __fmul2_rn(bj, bk), ab);
            tfx = __ffma2_rn(g, kept(__ffma2_rn(rx, wv, __ffma2_rn(k.ux, bj, __fmul2_rn(vx, bk)))), tfx);
            tfy = __ffma2_rn(g, kept(__ffma2_rn(ry, wv, __ffma2_rn(k.uy, bj, __fmul2_rn(vy, bk)))), tfy);
            tfz = __ffma2_rn(g, kept(__ffma2_rn(rz, wv, __ffma2_rn(k.uz, bj, __fmul2_rn(vz, bk)))), tfz);
            if (r2.x < near2) close |= one;
            if (r2.y < near2) close |= one << 1;
            one <<= 2;
        }
        // LJ pairs within the cut, each lane its own
        while (close != 0u) {
            const int b = __ffs(close) - 1;
            close &= close - 1u;
            const float* st = own + (b >> 1) * kAp2Pair + (b & 1);
            const float rx = k.x.x + st[0], ry = k.y.x + st[2], rz = k.z.x + st[4];
            lj<float>(fp, rx, ry, rz, pair_r2(rx, ry, rz), sx, sy, sz, es);
        }
        if ((it & 7) == 0) {
            hx = __fadd2_rn(hx, thx); hy = __fadd2_rn(hy, thy); hz = __fadd2_rn(hz, thz);
            fx = __fadd2_rn(fx, tfx); fy = __fadd2_rn(fy, tfy); fz = __fadd2_rn(fz, tfz);
            thx = thy = thz = tfx = tfy = tfz = zero;
        }
    }
    a.hx = __fadd2_rn(hx, thx); a.hy = __fadd2_rn(hy, thy); a.hz = __fadd2_rn(hz, thz);
    a.fx = __fadd2_rn(fx, tfx); a.fy = __fadd2_rn(fy, tfy); a.fz = __fadd2_rn(fz, tfz);
    a.sx = sx; a.sy = sy; a.sz = sz; a.es = es;
}

// A lane's sums to its place among the block's.
__device__ __forceinline__ void ap2_store(const Ap2Sums& a, float* r)
{
    r[0] = a.hx.x + a.hx.y; r[1] = a.hy.x + a.hy.y; r[2] = a.hz.x + a.hz.y;
    r[3] = a.fx.x + a.fx.y; r[4] = a.fy.x + a.fy.y; r[5] = a.fz.x + a.fz.y;
    r[6] = a.sx; r[7] = a.sy; r[8] = a.sz; r[9] = a.es;
}

// A block whose sums hold an undefined value forms them again with EXACT: zero
// times an infinite or undefined term (a moment that is not finite or too large for
// products of two, an undefined position) is undefined and stays so in a sum, so
// nothing is missed, and the test costs other blocks one barrier vote.  (Leaving
// terms out in every pair cost 8 %: n = 65,536 6.78 -> 7.46 ms; in line rather than
// as a call, this code cost 1.5 us of the 74 of a field call at n = 1,000.)
template <int T>
__device__ __noinline__ void ap2_exact(const float4* __restrict__ pos, const float4* __restrict__ u,
                                       int n, const FieldParams<float>& fp, float* stage, float4 xk,
                                       float4 uk, float* r)
{
    const Ap2Target tg = {dup2(xk.x), dup2(xk.y), dup2(xk.z), dup2(uk.x), dup2(uk.y), dup2(uk.z)};
    Ap2Sums a;
    ap2_sweep<T, true>(pos, u, n, fp, stage, tg, a);
    __syncthreads();
    ap2_store(a, r);
}

template <int T>
__global__ void __launch_bounds__(32 * kAp2Warps, 2) k_ap2(const float4* __restrict__ pos,
                                                           const float4* __restrict__ u, int n,
                                                           FieldParams<float> fp,
                                                           float4* __restrict__ h,
                                                           float4* __restrict__ f,
                                                           float* __restrict__ esr)
{
    constexpr int kGroups = 32 / T;         // groups of T lanes in a warp
    constexpr int kSums = 10;
    __shared__ __align__(16) float sm[kAp2Warps * kAp2Stage];
    static_assert(kAp2Warps * kAp2Stage >= kAp2Warps * 32 * kSums, "room for the partial sums");
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int k = blockIdx.x * T + lane % T;
    const float4 xk = pos[min(k, n - 1)], uk = u[min(k, n - 1)];
    const Ap2Target tg = {dup2(xk.x), dup2(xk.y), dup2(xk.z), dup2(uk.x), dup2(uk.y), dup2(uk.z)};
    float* stage = sm + w * kAp2Stage;
    float* r = sm + (w * 32 + lane) * kSums;
    Ap2Sums a;
    ap2_sweep<T, false>(pos, u, n, fp, stage, tg, a);
    const float2 all = __fadd2_rn(__fadd2_rn(__fadd2_rn(a.hx, a.hy), __fadd2_rn(a.hz, a.fx)),
                                  __fadd2_rn(a.fy, a.fz));
    if (__syncthreads_or(isnan(all.x + all.y)))
        ap2_exact<T>(pos, u, n, fp, stage, xk, uk, r);
    else
        ap2_store(a, r);
    __syncthreads();
    // component q of target t: the groups' sums in order
    for (int e = threadIdx.x; e < T * kSums; e += 32 * kAp2Warps) {
        const int t = e / kSums, q = e % kSums;
        float v = 0.0f;
        for (int g = 0; g < kAp2Warps * kGroups; ++g) v += sm[(g * T + t) * kSums + q];
        sm[t * kSums + q] = v;  // (its own slot of group 0, read by no other sum)
    }
    __syncthreads();
    if (threadIdx.x < T && k < n) {
        const float* v = sm + threadIdx.x * kSums;
        h[k] = make_float4(fp.dip_scale * v[0], fp.dip_scale * v[1], fp.dip_scale * v[2], 0.0f);
        f[k] = make_float4(fp.dip_scale * v[3] + v[6], fp.dip_scale * v[4] + v[7],
                           fp.dip_scale * v[5] + v[8], 0.0f);
        if (esr) esr[k] = v[9];
    }
}

}  // namespace

// Whether the walk with dipole-position terms takes the shape with more registers
// and `resident` warps at once (54 registers, 36 warps on each of 152 SMs).  While
// every task has a warp at once, or all but a few that start as the first end (to
// 182,080 particles), fewer warps cost nothing.  Beyond, the 40 warps of the other
// shape hide more of its loads, except at small opening angles with one-particle
// leaves, where a task does more arithmetic a load (but not up to 1.4 waves of
// warps, where what the second wave holds runs alone).  Field calls, ms with 10 / 8
// blocks: 131,071 particles at theta 0.7 0.976 / 0.940; 180,000 at 0.4 3.22 / 3.09;
// 200,000 at 0.5 2.10 / 2.33; 1,048,576 at 0.7 4.36 / 4.65, at 0.5 9.47 / 9.79; at 0.4
// 192,000 3.33 / 3.70, 288,000 5.17 / 4.97, 400,000 6.77 / 6.60, 700,000 11.8 / 11.5
// (leaf_max 2: 300,000 5.16 / 5.27); at 0.3 400,000 15.4 / 14.1.
bool quad_few_warps(int64_t ntask, int64_t resident, double theta2, int leaf_max)
{
    if (25 * ntask <= 26 * resident) return true;
    return theta2 < 0.2 && leaf_max == 1 && 5 * ntask > 7 * resident;
}

// FEW: only where quad_few_warps() (else false, and no launch).
template <typename R, bool COUNT, int G, bool QUAD = false, int THREADS = kBhThreads,
          int MINB = bh_min_blocks<R, COUNT, QUAD>(), bool FEW = false>
bool bh_launch_g(const vec4<R>* pos, const vec4<R>* u, int64_t n, Tree<R> t, FieldParams<R> fp,
                 vec4<R>* h, vec4<R>* f, R* esr, int4* counts, int* flags, int* work,
                 const uint32_t* off, Segs sg, cudaStream_t s)
{
    // persistent grid: as many blocks as fit on the device at once; a small
    // shared-memory carveout (the kernel uses none) leaves the rest to L1
    static std::mutex mu;
    static PersistentGrid cache[kMaxDevices];
    const auto kern = k_bh<R, COUNT, G, QUAD, THREADS, MINB>;
    const PersistentGrid g = persistent_grid(cache, mu, [kern] {
        cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                             kTraverseCarveout);
        int per_sm = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, THREADS, 0);
        return per_sm;
    });
    if (FEW && !quad_few_warps((n + 31) / 32, (int64_t)g.blocks * (THREADS / 32),
                               (double)fp.theta2, t.leaf_max))
        return false;
    cudaMemsetAsync(work, 0, sizeof(int) * g.nseg, s);
    kern<<<g.blocks, THREADS, 0, s>>>(pos, u, (int)n, t, fp, h, f, esr, counts, flags, work,
                                      g.nseg, off, sg);
    return true;
}

template <typename R, bool COUNT>
void bh_launch(const vec4<R>* pos, const vec4<R>* u, int64_t n, Tree<R> t, FieldParams<R> fp,
               vec4<R>* h, vec4<R>* f, R* esr, int4* counts, int* flags, int* work, int group,
               int sched, const uint32_t* off, Segs sg, cudaStream_t s)
{
    if constexpr (sizeof(R) == 4 && !COUNT) {
        // few particles: a warp per task shares its reading of the tree, and no lane
        // group or launch schedule applies
        if (takes_warp_walk(t, n, COUNT)) {
            warp_walk(pos, u, n, t, fp, h, f, esr, flags, work, off, sg, s);
            return;
        }
        // a tuned launch schedule of the plain FP32 walk (see kSchedules)
        if (sched >= 1 && sched <= kNumSchedules && !t.q1) {
#define FFK_SCHED(G, T, B) bh_launch_g<R, false, G, false, T, B>(pos, u, n, t, fp, h, f, esr, counts, flags, work, off, sg, s)
            switch (sched) {
                case 1: FFK_SCHED(1, 128, 12); return;
                case 2: FFK_SCHED(1, 128, 10); return;
                case 3: FFK_SCHED(1, 128, 8); return;
                case 4: FFK_SCHED(1, 256, 6); return;
                case 5: FFK_SCHED(1, 256, 4); return;
                case 6: FFK_SCHED(1, 64, 24); return;
                case 7: FFK_SCHED(1, 64, 16); return;
                case 8: FFK_SCHED(2, 128, 12); return;
                case 9: FFK_SCHED(4, 128, 12); return;
                default: FFK_SCHED(8, 128, 12); return;
            }
#undef FFK_SCHED
        }
    }
    if constexpr (sizeof(R) == 8) {
        // FP64: one walk for every lane group and schedule (trees of more cells than its
        // source words can name, and dipole-position terms, keep the one-lane walk)
        if (t.child && !t.q1 && t.cap <= kWarpWalkCells)
            warp_walk64(pos, u, n, t, fp, h, f, esr, COUNT ? counts : nullptr, flags, work, off, sg, s);
        else if (t.q1)
            bh_launch_g<R, COUNT, 1, true>(pos, u, n, t, fp, h, f, esr, counts, flags, work, off, sg, s);
        else
            bh_launch_g<R, COUNT, 1>(pos, u, n, t, fp, h, f, esr, counts, flags, work, off, sg, s);
        return;
    } else {
    if (sched >= 1 && sched <= kNumSchedules) group = kSchedules[sched - 1].group;
    if (t.q1) {
        // the dipole-position terms are evaluated by the one-lane walk only, in one of
        // two shapes (quad_few_warps)
        if (!bh_launch_g<R, COUNT, 1, true, kBhThreads, kBhMinBlocksQuadFew, true>(
                pos, u, n, t, fp, h, f, esr, counts, flags, work, off, sg, s))
            bh_launch_g<R, COUNT, 1, true>(pos, u, n, t, fp, h, f, esr, counts, flags, work, off,
                                           sg, s);
        return;
    }
#define FFK_BH_CASE(G) bh_launch_g<R, COUNT, G>(pos, u, n, t, fp, h, f, esr, counts, flags, work, off, sg, s)
    switch (group) {
        case 1: FFK_BH_CASE(1); break;
        case 2: FFK_BH_CASE(2); break;
        case 4: FFK_BH_CASE(4); break;
        case 8: FFK_BH_CASE(8); break;
        case 16: FFK_BH_CASE(16); break;
        default: FFK_BH_CASE(32); break;
    }
#undef FFK_BH_CASE
    }
}

template <typename R>
void bh_field(const vec4<R>* pos, const vec4<R>* u, int64_t n, Tree<R> t, FieldParams<R> fp,
              vec4<R>* h, vec4<R>* f, R* esr, int4* counts, int* flags, int* work, int group,
              int sched, const uint32_t* off, Segs sg, cudaStream_t s)
{
    if (counts)
        bh_launch<R, true>(pos, u, n, t, fp, h, f, esr, counts, flags, work, group, sched, off, sg,
                           s);
    else
        bh_launch<R, false>(pos, u, n, t, fp, h, f, esr, counts, flags, work, group, sched, off,
                            sg, s);
    counted();
}

template <typename R>
void bh_field_record(const vec4<R>* pos, const vec4<R>* u, int64_t n, Tree<R> t, FieldParams<R> fp,
                     vec4<R>* h, vec4<R>* f, R* esr, int4* counts, int* flags, int* work,
                     const uint32_t* off, Segs sg, EntryPool pool, cudaStream_t s)
{
    if (n <= 0) return;
    static std::mutex mu;
    static PersistentGrid cache[kMaxDevices];
    const PersistentGrid g = persistent_grid(cache, mu, [] {
        cudaFuncSetAttribute(k_bh_rec<R>, cudaFuncAttributePreferredSharedMemoryCarveout,
                             kTraverseCarveout);
        int per_sm = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_bh_rec<R>, kBhThreads, 0);
        return per_sm;
    });
    cudaMemsetAsync(work, 0, sizeof(int) * g.nseg, s);
    k_bh_rec<R><<<g.blocks, kBhThreads, 0, s>>>(pos, u, (int)n, t, fp, h, f, esr, counts, flags,
                                                work, g.nseg, off, sg, pool);
    counted();
}

template <>
void ap_field<double>(const dvec4* pos, const dvec4* u, int64_t n, FieldParams<double> fp, dvec4* h,
                      dvec4* f, double* esr, cudaStream_t s)
{
    const unsigned g = (unsigned)((n + kApThreads - 1) / kApThreads);
    k_ap<double><<<g, kApThreads, 0, s>>>(pos, u, (int)n, fp, h, f, esr);
    counted();
}

template <>
void ap_field<float>(const float4* pos, const float4* u, int64_t n, FieldParams<float> fp,
                     float4* h, float4* f, float* esr, cudaStream_t s)
{
    if (n < kApWide)
        k_ap2<16><<<(unsigned)((n + 15) / 16), 32 * kAp2Warps, 0, s>>>(pos, u, (int)n, fp, h, f, esr);
    else
        k_ap2<32><<<(unsigned)((n + 31) / 32), 32 * kAp2Warps, 0, s>>>(pos, u, (int)n, fp, h, f, esr);
    counted();
}

template void bh_field<float>(const float4*, const float4*, int64_t, Tree<float>,
                              FieldParams<float>, float4*, float4*, float*, int4*, int*, int*,
                              int, int, const uint32_t*, Segs, cudaStream_t);
template void bh_field<double>(const dvec4*, const dvec4*, int64_t, Tree<double>,
                               FieldParams<double>, dvec4*, dvec4*, double*, int4*, int*, int*,
                               int, int, const uint32_t*, Segs, cudaStream_t);
template void bh_field_record<float>(const float4*, const float4*, int64_t, Tree<float>,
                                     FieldParams<float>, float4*, float4*, float*, int4*, int*,
                                     int*, const uint32_t*, Segs, EntryPool, cudaStream_t);
template void bh_field_record<double>(const dvec4*, const dvec4*, int64_t, Tree<double>,
                                      FieldParams<double>, dvec4*, dvec4*, double*, int4*, int*,
                                      int*, const uint32_t*, Segs, EntryPool, cudaStream_t);

template <typename R, bool REC>
void bh_vjp_launch(const vec4<R>* pos, int64_t n, Tree<R> t, FieldParams<R> fp, int* flags,
                   int* work, const uint32_t* off, Segs sg, VjpIn<R> vj, int4* counts,
                   EntryPool ep, cudaStream_t s)
{
    static std::mutex mu;
    static PersistentGrid cache[kMaxDevices];
    const PersistentGrid g = persistent_grid(cache, mu, [] {
        cudaFuncSetAttribute(k_bh_vjp<R, REC>, cudaFuncAttributePreferredSharedMemoryCarveout,
                             kTraverseCarveout);
        int per_sm = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_bh_vjp<R, REC>, kBhThreads, 0);
        return per_sm;
    });
    cudaMemsetAsync(work, 0, sizeof(int) * g.nseg, s);
    k_bh_vjp<R, REC><<<g.blocks, kBhThreads, 0, s>>>(pos, (int)n, t, fp, flags, work, g.nseg, off,
                                                     sg, vj, counts, ep);
    counted();
}

template <typename R>
void bh_vjp_target(const vec4<R>* pos, const vec4<R>* u, const vec4<R>* abar, const vec4<R>* bbar,
                   int64_t n, Tree<R> t, FieldParams<R> fp, int* flags, int* work,
                   const uint32_t* off, Segs sg, vec4<R>* dxt, vec4<R>* dut, cudaStream_t s,
                   int4* counts, const EntryPool* pool)
{
    if (n <= 0) return;
    VjpIn<R> vj;
    vj.u = u;
    vj.abar = abar;
    vj.bbar = bbar;
    vj.dxt = dxt;
    vj.dut = dut;
    if (pool)
        bh_vjp_launch<R, true>(pos, n, t, fp, flags, work, off, sg, vj, counts, *pool, s);
    else
        bh_vjp_launch<R, false>(pos, n, t, fp, flags, work, off, sg, vj, nullptr, EntryPool(), s);
}

template void bh_vjp_target<float>(const float4*, const float4*, const float4*, const float4*,
                                   int64_t, Tree<float>, FieldParams<float>, int*, int*,
                                   const uint32_t*, Segs, float4*, float4*, cudaStream_t, int4*,
                                   const EntryPool*);
template void bh_vjp_target<double>(const dvec4*, const dvec4*, const dvec4*, const dvec4*,
                                    int64_t, Tree<double>, FieldParams<double>, int*, int*,
                                    const uint32_t*, Segs, dvec4*, dvec4*, cudaStream_t, int4*,
                                    const EntryPool*);

}  // namespace ffk
