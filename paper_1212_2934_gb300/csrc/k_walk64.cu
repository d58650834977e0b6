// The double-precision Barnes-Hut walk (Sec. 3.2, kernel 5 of the paper's scheme,
// redesigned): one warp serves eight consecutive particles of the Morton order.
//
// FP64 arithmetic bounds it: a warp's FP64 instruction holds its quarter of the SM
// for 64 cycles, whatever its lanes do.  The one-lane walk spent such
// instructions on opening tests, on lanes that had taken another branch and on
// the longest walk of 32.  Here the tree is read for the eight particles
// together, a cell per lane (walk_stack.cuh), and decided in single precision
// relative to the first particle, with bounds far above the rounding; only what
// those leave open is decided by the exact test.  Each particle's sources go to a
// list of its own, in depth-first order, and four lanes a particle sum every
// fourth entry: full warps, and four quarters of an SM at work on 32 particles
// where one was.
//
// A particle's sums depend on its own list alone (four partial sums added in a
// fixed order), not on its neighbours in the warp.  Measured on GB300 (volume
// fraction 0.05, theta 0.5), one-lane walk -> this: n = 4,096 1.53 -> 0.39 ms,
// 16,384 1.98 -> 1.14, 50,000 5.57 -> 3.24, 100,000 12.0 -> 6.87, 262,144 29.9 ->
// 19.4; the FP64 units are 86 % busy at n = 100,000.
#include "walk_stack.cuh"

namespace ffk {

namespace {

constexpr int kT = 8;          // particles per warp
constexpr int kSub = 32 / kT;  // lanes per particle
constexpr int kWalk64Threads = 64;
// Sources of a particle summed at a time, and blocks an SM.  The longer the lists,
// the less their lengths differ within a warp; two warps a quarter keep its FP64
// unit busy.  Measured at n = 50,000, ms: 224 / 8 blocks 3.71, 320 / 6 3.41,
// 416 / 5 3.30, 512 / 4 3.26.
constexpr int kCap = 512;
constexpr int kWalk64Blocks = 4;
// uncertainty of a squared distance formed in single precision from coordinates
// relative to the task: below 2e-6 of it plus the task's own extent squared
constexpr float kSlack = 1e-5f;

// Cells decided particle by particle in a round, relative to the task.
struct Mixed64 {
    float4 c[32];     // centre, side^2
    float4 lo[32];    // lower cube corner, the cell (bits)
    float hi[32][3];  // upper cube corner
};

struct Walk64Shared {
    WalkQueue q;
    Mixed64 mixed;
    uint32_t src[kT][kCap];
};

struct Sums64 {
    double hx, hy, hz, fx, fy, fz, ck, sx, sy, sz, es;
    int nacc, npair;
};

// Centre and moment of a source word.
__device__ __forceinline__ void source_of(uint32_t s, const Tree<double>& t,
                                          const dvec4* __restrict__ pos,
                                          const dvec4* __restrict__ u, dvec4& c, dvec4& m)
{
    const uint32_t i = s & kIndex;
    c = (s & kParticle) ? pos[i] : t.cell[i].cen;
    m = (s & kParticle) ? u[i] : t.mom[i];
}

// Sums the particles' lists, the n entries after the particle's first done: lane
// sub of its lanes takes the entries that are sub, sub + 4, ... of all its sources,
// so where the lists are cut, which the longest of the warp's decides, does not
// matter.  LJ pairs (and, counting, the decision of one-particle
// leaves) are left to the end of each 32 entries, so that one lane's pair does
// not hold up the others at every entry.
template <bool COUNT>
__device__ __forceinline__ void sum_lists(const Walk64Shared& w, int n, int& done,
                                          const Tree<double>& t,
                                          const FieldParams<double>& fp,
                                          const dvec4* __restrict__ pos,
                                          const dvec4* __restrict__ u, const dvec4& xk,
                                          const dvec4& uk, Sums64& a)
{
    const int lane = threadIdx.x & 31, g = lane / kSub, sub = lane % kSub;
    const int most = __reduce_max_sync(kFull, n);
    __syncwarp();
    const int first = (sub - done) & (kSub - 1);
    done += n;
    for (int b = first; b - first < most; b += 32 * kSub) {
        uint32_t close = 0u;
        for (int r = 0; r < 32; ++r) {
            const int i = b + r * kSub;
            if (i - first >= most) break;
            if (i < n) {
                const uint32_t s = w.src[g][i];
                dvec4 c, m;
                source_of(s, t, pos, u, c, m);
                const double rx = xk.x - c.x, ry = xk.y - c.y, rz = xk.z - c.z;
                const double r2 = pair_r2(rx, ry, rz);
                dipole_acc<double>(rx, ry, rz, r2, uk.x, uk.y, uk.z, m.x, m.y, m.z, a.hx, a.hy,
                                   a.hz, a.fx, a.fy, a.fz, a.ck);
                if (s & (kLeafCell | kParticle)) {
                    const bool leaf = (s & kLeafCell) != 0u;
                    if ((COUNT && leaf) || (fp.include_sr && r2 < fp.lj_rcut2_hi)) close |= 1u << r;
                    else if (COUNT) ++a.npair;
                } else if (COUNT) {
                    ++a.nacc;
                }
            }
        }
        while (close != 0u) {
            const int r = __ffs(close) - 1;
            close &= close - 1u;
            const uint32_t s = w.src[g][b + r * kSub];
            dvec4 c, m;
            source_of(s, t, pos, u, c, m);
            const double rx = xk.x - c.x, ry = xk.y - c.y, rz = xk.z - c.z;
            const double r2 = pair_r2(rx, ry, rz);
            // a one-particle leaf is accepted or summed as a pair: the two differ by LJ
            if ((s & kLeafCell) && (COUNT || (r2 >= fp.lj_rcut2_lo && r2 < fp.lj_rcut2_hi))) {
                const int i = (int)(s & kIndex);
                if (accept<double>(fp, __dsub_rn(xk.x, c.x), __dsub_rn(xk.y, c.y),
                                   __dsub_rn(xk.z, c.z), xk, t.cell[i].cen, t.lo, i, m.w)) {
                    if (COUNT) ++a.nacc;
                    continue;
                }
            }
            if (COUNT) ++a.npair;
            if (fp.include_sr) lj<double>(fp, rx, ry, rz, r2, a.sx, a.sy, a.sz, a.es);
        }
    }
    __syncwarp();
}

// Hands the first n entries (at most 32) of the list to their particles; mine is
// the length of this lane's particle's list.
__device__ __forceinline__ void hand_out(Walk64Shared& w, int n, int lane, uint32_t lt, int& mine)
{
    __syncwarp();
    uint2 e = make_uint2(0u, 0u);
    if (lane < n) e = w.q.list[lane];
#pragma unroll
    for (int g = 0; g < kT; ++g) {
        const bool has = ((e.y >> g) & 1u) != 0u;
        const uint32_t m = __ballot_sync(kFull, has);
        const int base = __shfl_sync(kFull, mine, g * kSub);
        if (has) w.src[g][base + __popc(m & lt)] = e.x;
        if (lane / kSub == g) mine += __popc(m);
    }
    __syncwarp();
}

__device__ __forceinline__ float warp_min(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(kFull, v, o));
    return v;
}

__device__ __forceinline__ double group_sum(double v)
{
#pragma unroll
    for (int o = 1; o < kSub; o <<= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

template <bool COUNT>
__device__ __forceinline__ void walk64_task(Walk64Shared& w, int task,
                                            const dvec4* __restrict__ pos,
                                            const dvec4* __restrict__ u, int n,
                                            const Tree<double>& t, const FieldParams<double>& fp,
                                            unsigned ncells, dvec4* __restrict__ h,
                                            dvec4* __restrict__ f, double* __restrict__ esr,
                                            int4* __restrict__ counts, int* flags,
                                            const uint32_t* __restrict__ off, const Segs& sg)
{
    const int lane = threadIdx.x & 31, g = lane / kSub, sub = lane % kSub;
    const uint32_t lt = (1u << lane) - 1u;
    const int k0 = task * kT, k = k0 + g;
    const bool active = k < n;
    const dvec4 xk = pos[active ? k : k0], uk = u[active ? k : k0], org = pos[k0];
    const float xf = (float)(xk.x - org.x), yf = (float)(xk.y - org.y), zf = (float)(xk.z - org.z);
    const float lx = warp_min(xf), ly = warp_min(yf), lz = warp_min(zf);
    const float ux = -warp_min(-xf), uy = -warp_min(-yf), uz = -warp_min(-zf);
    const float ext2 = -warp_min(-(xf * xf + yf * yf + zf * zf));
    // quick decisions up to theta = 10, where a cube that may be accepted has its corners
    // within 20 distances of its centre, and so their rounding within the slack; no quick
    // one holds beyond (nor for angles whose square is no normal single-precision number)
    const bool quick = fp.theta2 <= 100.0 && !(fp.theta2 > 0.0 && fp.theta2 < 1e-37);
    const float th2 = quick ? (float)fp.theta2 : __int_as_float(0x7fffffff);
    const float rcut2 = quick && fp.use_rcut ? (float)fp.rcut2 : -3.0e38f;
    Sums64 a = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0, 0};
    int nopen = 0, mine = 0, done = 0, top = 0;
    // the roots of the task's systems, the first on top
    __syncwarp();
    {
        const bool lead0 = active && sub == 0;
        const uint32_t sys = sg.of_pos ? (active ? sg.of_pos[k] : 0xffffffffu)
                                       : (active ? 0u : 0xffffffffu);
        const uint32_t same = __match_any_sync(kFull, sys);
        // a particle's bit from its first lane's
        uint32_t mask = 0u;
#pragma unroll
        for (int q = 0; q < kT; ++q) mask |= ((same >> (q * kSub)) & 1u) << q;
        const bool lead = lead0 && (same & lt) == 0u;
        const uint32_t lm = __ballot_sync(kFull, lead);
        top = __popc(lm);
        if (lead)
            w.q.stack[top - 1 - __popc(lm & lt)] =
                make_uint2(sg.of_pos ? off[sg.start[sys]] : 0u, mask);
    }
    const unsigned max_rounds = 4u * ncells + 64u;
    unsigned rounds = 0;
    while (top > 0) {
        __syncwarp();
        const int seen = min(32, top);
        uint2 e = make_uint2(kDone, 0u);
        if (lane < seen) e = w.q.stack[top - 1 - lane];
        __syncwarp();
        const uint32_t runs = __ballot_sync(kFull, (e.x & kRun) != 0u);
        if (runs & 1u) {
            // an opened leaf of several particles on top: each of them, but to itself
            const uint2 first = make_uint2(__shfl_sync(kFull, e.x, 0), __shfl_sync(kFull, e.y, 0));
            const int4 nd = t.cell[first.x & kIndex].node;
            for (int s0 = nd.x; s0 < nd.y; s0 += 32) {
                const int s = s0 + lane;
                uint32_t mask = s < nd.y ? first.y : 0u;
                if (s >= k0 && s < k0 + kT) mask &= ~(1u << (s - k0));
                w.q.list[lane] = make_uint2((uint32_t)s | kParticle, mask);
                hand_out(w, 32, lane, lt, mine);
                if (__reduce_max_sync(kFull, mine) > kCap - 32) {
                    sum_lists<COUNT>(w, mine, done, t, fp, pos, u, xk, uk, a);
                    mine = 0;
                }
            }
            --top;
            continue;
        }
        const bool fresh = (e.x & kDone) == 0u;
        uint32_t acc = fresh ? 0u : e.y, open = 0u, own = 0u;
        uint32_t src = e.x & ~kDone;
        bool mixed = false;
        int4 nd = make_int4(0, 0, 0, 0);
        float4 c, lo;
        float hx, hy, hz;
        if (fresh) {
            const Cell<double> cl = t.cell[e.x];
            const dvec4 l = t.lo[e.x];
            nd = cl.node;
            const bool meets = nd.x < k0 + kT && nd.y > k0;
            if (meets) {
                const int b = max(nd.x - k0, 0), m = min(nd.y - k0, kT) - b;
                own = ((1u << m) - 1u) << b;
            }
            if ((nd.w >> 9) != 0) {
                acc = e.y & ~own;
                src = e.x | kLeafCell;
            } else {
                asm volatile("prefetch.global.L1 [%0];" ::"l"(t.child + 2 * (int64_t)e.x));
                c = make_float4((float)(cl.cen.x - org.x), (float)(cl.cen.y - org.y),
                                (float)(cl.cen.z - org.z), (float)cl.cen.w);
                lo = make_float4((float)(l.x - org.x), (float)(l.y - org.y), (float)(l.z - org.z),
                                 __uint_as_float(e.x));
                const float side = (float)l.w;
                hx = lo.x + side;
                hy = lo.y + side;
                hz = lo.z + side;
                // bounds over the particles' box: nearest and farthest distance of the
                // centre, and of the cube
                const float ax = lx - c.x, bx = c.x - ux, ay = ly - c.y, by = c.y - uy,
                            az = lz - c.z, bz = c.z - uz;
                const float gx = fmaxf(fmaxf(ax, bx), 0.0f), wx = fminf(ax, bx);
                const float gy = fmaxf(fmaxf(ay, by), 0.0f), wy = fminf(ay, by);
                const float gz = fmaxf(fmaxf(az, bz), 0.0f), wz = fminf(az, bz);
                const float dmin = gx * gx + gy * gy + gz * gz;
                const float dmax = wx * wx + wy * wy + wz * wz;
                const float px = fmaxf(fmaxf(lo.x - ux, lx - hx), 0.0f);
                const float py = fmaxf(fmaxf(lo.y - uy, ly - hy), 0.0f);
                const float pz = fmaxf(fmaxf(lo.z - uz, lz - hz), 0.0f);
                const float qx = fmaxf(fmaxf(lo.x - lx, ux - hx), 0.0f);
                const float qy = fmaxf(fmaxf(lo.y - ly, uy - hy), 0.0f);
                const float qz = fmaxf(fmaxf(lo.z - lz, uz - hz), 0.0f);
                const float bmin = px * px + py * py + pz * pz;
                const float bmax = qx * qx + qy * qy + qz * qz;
                const float slack = kSlack * (dmax + ext2);
                const bool sized = c.w > 1e-30f && dmax < 1e30f;
                const bool all = sized && !meets && c.w * 1.00001f < th2 * (dmin - slack) &&
                                 bmin - slack > rcut2;
                const bool none = sized && (c.w > th2 * 1.00001f * (dmax + slack) ||
                                            bmax + slack < rcut2);
                mixed = !all && !none;
                acc = all ? e.y : 0u;
                open = none ? e.y : 0u;
            }
        }
        const uint32_t mm = __ballot_sync(kFull, mixed);
        if (mm != 0u) {
            const int rank = __popc(mm & lt), nm = __popc(mm);
            uint32_t got = 0u;
            if (mixed) {
                w.mixed.c[rank] = c;
                w.mixed.lo[rank] = lo;
                w.mixed.hi[rank][0] = hx;
                w.mixed.hi[rank][1] = hy;
                w.mixed.hi[rank][2] = hz;
            }
            __syncwarp();
            // four cells at a time, lane sub of each particle's lanes the r0 + sub-th
            for (int r0 = 0; r0 < nm; r0 += kSub) {
                const int r = min(r0 + sub, nm - 1);
                const float4 cj = w.mixed.c[r], lj = w.mixed.lo[r];
                const float dx = xf - cj.x, dy = yf - cj.y, dz = zf - cj.z;
                const float d2 = dx * dx + dy * dy + dz * dz;
                const float bx = fmaxf(fmaxf(lj.x - xf, xf - w.mixed.hi[r][0]), 0.0f);
                const float by = fmaxf(fmaxf(lj.y - yf, yf - w.mixed.hi[r][1]), 0.0f);
                const float bz = fmaxf(fmaxf(lj.z - zf, zf - w.mixed.hi[r][2]), 0.0f);
                const float b2 = bx * bx + by * by + bz * bz;
                const float slack = kSlack * (d2 + ext2);
                const bool sized = cj.w > 1e-30f && d2 < 1e30f;
                bool ok = sized && cj.w * 1.00001f < th2 * (d2 - slack) && b2 - slack > rcut2;
                const bool no = sized && (cj.w > th2 * 1.00001f * (d2 + slack) || b2 + slack < rcut2);
                if (!ok && !no) {  // too near to call: the exact test
                    const int i = (int)__float_as_uint(lj.w);
                    ok = accept<double>(fp, xk, t.cell[i].cen, t.lo, i, t.mom[i].w);
                }
                const uint32_t am = __ballot_sync(kFull, ok);
                if (rank >= r0 && rank < r0 + kSub) {
                    // the bits of the particles' lanes rank - r0, packed
                    uint32_t x = (am >> (rank - r0)) & 0x11111111u;
                    x = (x | x >> 3) & 0x03030303u;
                    x = (x | x >> 6) & 0x000f000fu;
                    got = (x | x >> 12) & 0xffu;
                }
            }
            if (mixed) {
                got &= ~own;
                acc = e.y & got;
                open = e.y & ~got;
            }
        }
        const int emit = settle(w.q, 0, lane, seen, runs, e, src, acc, open, nd.w, t.child, top);
        if (COUNT) {
            const uint32_t inner = (nd.w >> 8) == 0 ? open : 0u;
#pragma unroll
            for (int q = 0; q < kT; ++q) {
                const int m = __popc(__ballot_sync(kFull, ((inner >> q) & 1u) != 0u));
                if (g == q) nopen += m;
            }
        }
        hand_out(w, emit, lane, lt, mine);
        if (__reduce_max_sync(kFull, mine) > kCap - 32) {
            sum_lists<COUNT>(w, mine, done, t, fp, pos, u, xk, uk, a);
            mine = 0;
        }
        if (++rounds > max_rounds) {  // a damaged tree
            if (lane == 0) atomicOr(flags, FLAG_TRAVERSE);
            break;
        }
    }
    sum_lists<COUNT>(w, mine, done, t, fp, pos, u, xk, uk, a);
    a.hx = group_sum(a.hx); a.hy = group_sum(a.hy); a.hz = group_sum(a.hz);
    a.fx = group_sum(a.fx); a.fy = group_sum(a.fy); a.fz = group_sum(a.fz);
    a.sx = group_sum(a.sx); a.sy = group_sum(a.sy); a.sz = group_sum(a.sz);
    a.ck = group_sum(a.ck);
    a.es = group_sum(a.es);
    if (COUNT) {
#pragma unroll
        for (int o = 1; o < kSub; o <<= 1) {
            a.nacc += __shfl_xor_sync(kFull, a.nacc, o);
            a.npair += __shfl_xor_sync(kFull, a.npair, o);
        }
    }
    if (!active || sub != 0) return;
    dvec4 ho, fo;
    ho.x = fp.dip_scale * a.hx;
    ho.y = fp.dip_scale * a.hy;
    ho.z = fp.dip_scale * a.hz;
    ho.w = 0.0;
    fo.x = fp.dip_scale * (a.fx + uk.x * a.ck) + a.sx;
    fo.y = fp.dip_scale * (a.fy + uk.y * a.ck) + a.sy;
    fo.z = fp.dip_scale * (a.fz + uk.z * a.ck) + a.sz;
    fo.w = 0.0;
    h[k] = ho;
    f[k] = fo;
    if (esr) esr[k] = a.es;
    if (COUNT) counts[k] = make_int4(a.nacc, a.npair, nopen, 0);
}

template <bool COUNT>
__global__ void __launch_bounds__(kWalk64Threads, kWalk64Blocks) k_warp_walk64(
    const dvec4* __restrict__ pos, const dvec4* __restrict__ u, int n, Tree<double> t,
    FieldParams<double> fp, dvec4* __restrict__ h, dvec4* __restrict__ f,
    double* __restrict__ esr, int4* __restrict__ counts, int* flags, int* __restrict__ work,
    int nseg, const uint32_t* __restrict__ off, Segs sg)
{
    extern __shared__ __align__(16) unsigned char walk64_smem[];
    Walk64Shared& w = reinterpret_cast<Walk64Shared*>(walk64_smem)[threadIdx.x >> 5];
    // a build that failed leaves no tree to walk (its flag reaches the host)
    if (*flags & (FLAG_CAPACITY | FLAG_SORT | FLAG_AGGREGATE | FLAG_NONFINITE)) return;
    const unsigned ncells = (unsigned)*t.ncells;
    const int ntask = (n + kT - 1) / kT;
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
            walk64_task<COUNT>(w, task, pos, u, n, t, fp, ncells, h, f, esr, counts, flags, off, sg);
        }
    }
}

template <bool COUNT>
void walk64_launch(const dvec4* pos, const dvec4* u, int64_t n, Tree<double> t,
                   FieldParams<double> fp, dvec4* h, dvec4* f, double* esr, int4* counts,
                   int* flags, int* work, const uint32_t* off, Segs sg, cudaStream_t s)
{
    constexpr int smem = (int)sizeof(Walk64Shared) * (kWalk64Threads / 32);
    static std::mutex mu;
    static PersistentGrid cache[kMaxDevices];
    const auto kern = k_warp_walk64<COUNT>;
    const PersistentGrid g = persistent_grid(cache, mu, [kern] {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        int per_sm = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kWalk64Threads, smem);
        return per_sm;
    });
    // no more blocks than tasks: a few tasks then sit on different quarters of the SMs
    const int64_t ntask = (n + kT - 1) / kT, per_block = kWalk64Threads / 32;
    const int64_t want = ((ntask + g.nseg * per_block - 1) / (g.nseg * per_block)) * g.nseg;
    const int blocks = (int)(want < g.blocks ? want : g.blocks);
    cudaMemsetAsync(work, 0, sizeof(int) * g.nseg, s);
    kern<<<blocks, kWalk64Threads, smem, s>>>(pos, u, (int)n, t, fp, h, f, esr, counts, flags,
                                              work, g.nseg, off, sg);
}

}  // namespace

void warp_walk64(const dvec4* pos, const dvec4* u, int64_t n, Tree<double> t,
                 FieldParams<double> fp, dvec4* h, dvec4* f, double* esr, int4* counts, int* flags,
                 int* work, const uint32_t* off, Segs sg, cudaStream_t s)
{
    if (counts)
        walk64_launch<true>(pos, u, n, t, fp, h, f, esr, counts, flags, work, off, sg, s);
    else
        walk64_launch<false>(pos, u, n, t, fp, h, f, esr, counts, flags, work, off, sg, s);
}

}  // namespace ffk
