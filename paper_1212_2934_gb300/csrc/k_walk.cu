// The plain single-precision Barnes-Hut walk of up to kWarpWalkMax particles
// (Sec. 3.2, kernel 5 of the paper's scheme, redesigned): one warp serves T
// consecutive particles of the Morton order and its lanes share the reading of
// the tree.
//
// Below kWarpWalkMax particles the one-lane walk (k_field.cu) does not fill the
// chip and takes the time of one particle's chain of about 900 dependent cell
// loads.  Here the chain is about 80 rounds.  Deciding: a stack of (cell, lanes
// that reach it) in depth-first order; each round takes up to 32 of them, a cell
// per lane, and settles a cell for all of its lanes at once where the
// particles' bounding box allows it (beyond the opening distance of every
// particle, or within it); cells in between are decided particle by particle,
// every lane its own.  An opened cell is replaced by its children, so what
// leaves the top of the stack is each particle's list of sources in depth-first
// order, the order of the one-lane walk.  Summing: sources are staged in shared
// memory two by two and added by every lane that has them, with two FP32
// operations per instruction; the sums themselves are formed one source after
// the other, so fields and forces have the bits of the one-lane walk.
//
// Measured on GB300 (volume fraction 0.05, theta 0.5), one-lane walk -> this:
//   n = 1,000  0.409 -> 0.157 ms     n = 65,536   0.647 -> 0.566 ms
//   n = 16,384 0.525 -> 0.313 ms     n = 100,000  0.741 -> 0.716 ms
// and 4.85 -> 5.45 ms at n = 1,048,576, where the one-lane walk has enough
// warps to hide its loads and this one adds every source of a task in all of
// its lanes (1784 of which a lane uses 813): the summing is bound by the FP32
// pipe (84 % busy), the deciding by the latency of its rounds.
#include "walk_stack.cuh"

namespace ffk {

namespace {

constexpr int kBatch = 64;    // sources summed together once this many are known
constexpr int kPairWords = 20;  // words per staged pair (16 used): fewer bank conflicts
constexpr int kStageWords = 352;  // 16 staged pairs, or a round's mixed cells
constexpr float kNormal = 1.1754944e-38f;  // smallest normal float

// Block shape: 8 blocks of 2 warps an SM leave 128 registers a thread and 112 KB
// of L1.  More warps cost registers and L1 that the walk needs more (65,536
// particles: 0.575 ms, against 0.617 at 20 warps an SM and 0.671 at 28).
constexpr int kWalkThreads = 64;
constexpr int kWalkBlocks = 8;

struct WarpShared {
    WalkQueue q;
    float stage[kStageWords];
};

// Cells decided particle by particle in a round (in the staging space).
struct MixedCell {
    float4 c[32];   // centre, side^2
    float4 lo[32];  // lower cube corner, far2
    float hi[32][3];  // upper cube corner
};
static_assert(sizeof(MixedCell) <= sizeof(float) * kStageWords, "fits the staging space");

struct Target {
    float x, y, z, ux, uy, uz;
};

struct Sums {
    float hx, hy, hz, fx, fy, fz, sx, sy, sz, es;
};

// The records of a task (energy gradient): each source once, with the lanes that
// have it, 64 to a chunk of the pool (the task's own chunk first, then chunks
// handed out by a counter, linked; chunks at or past cap are not written).
constexpr uint32_t kRecChunk = kPoolChunk / 2;

struct RecordWriter {
    uint32_t ck, fill, total;
    int nsrc;  // this lane's sources

    __device__ __forceinline__ void put(const EntryPool& p, bool valid, uint32_t key, uint32_t mask)
    {
        const int lane = threadIdx.x & 31;
        const uint32_t m = __ballot_sync(kFull, valid), c = (uint32_t)__popc(m);
        const uint32_t at = fill + (uint32_t)__popc(m & ((1u << lane) - 1u));
        const bool full = fill + c >= kRecChunk;  // the chunk after a full one is taken at once
        uint32_t nk = 0;
        if (full) {
            if (lane == 0) {
                nk = p.first + atomicAdd(p.next, 1u);
                if (ck < p.cap) p.link[ck] = nk;
            }
            nk = __shfl_sync(kFull, nk, 0);
        }
        const uint32_t to = at < kRecChunk ? ck : nk;
        if (valid && to < p.cap)
            reinterpret_cast<uint2*>(p.keys)[(size_t)to * kRecChunk + at % kRecChunk] =
                make_uint2(key, mask);
        fill += c;
        total += c;
        if (full) {
            ck = nk;
            fill -= kRecChunk;
        }
    }
};

// What one source adds for this lane beyond the dipole terms of an ordinary
// separation (rare): the LJ force of a particle within the cut, where a
// one-particle leaf is first decided between accepting it and summing it as a
// pair, and the dipole terms at a separation below the normal range.
__device__ __forceinline__ void near_source(const FieldParams<float>& fp, const Tree<float>& t,
                                            const Target& k, uint32_t src, float rx, float ry,
                                            float rz, float vx, float vy, float vz, Sums& a)
{
    const float r2 = pair_r2(rx, ry, rz);
    if (r2 > 0.0f && r2 < kNormal)
        walk_dipole<float>(rx, ry, rz, r2, k.ux, k.uy, k.uz, -vx, -vy, -vz, a.hx, a.hy, a.hz,
                           a.fx, a.fy, a.fz);
    if (!fp.include_sr || !(src & (kLeafCell | kParticle))) return;
    if ((src & kLeafCell) && r2 >= fp.lj_rcut2_lo && r2 < fp.lj_rcut2_hi) {
        const int i = (int)(src & kIndex);
        const float4 c = t.cell[i].cen;
        if (accept<float>(fp, rx, ry, rz, make_float4(k.x, k.y, k.z, 0.0f), c, t.lo, i,
                          t.mom[i].w))
            return;
    }
    lj<float>(fp, rx, ry, rz, r2, a.sx, a.sy, a.sz, a.es);
}

// 1/sqrt(x) of a normal x, the bits of rsqrtf() there without its handling of
// subnormal x.
__device__ __forceinline__ float rsqrt_normal(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Adds one source's terms if the lane has it (mask & bit) at a separation in the
// normal range, and marks it in `close` below near2.  Written as predicated
// instructions: as branches the 12 additions of a pair cost more than their own
// issue slots.
__device__ __forceinline__ void add_if(uint32_t mask, uint32_t bit, float r2, float near2,
                                       float tx, float ty, float tz, float sx, float sy, float sz,
                                       Sums& a, uint32_t& close, uint32_t one)
{
    asm("{\n\t"
        ".reg .pred in, p, c;\n\t"
        ".reg .b32 m;\n\t"
        "and.b32 m, %7, %8;\n\t"
        "setp.ne.b32 in, m, 0;\n\t"
        "setp.ge.and.f32 p, %9, %10, in;\n\t"
        "setp.lt.and.f32 c, %9, %11, in;\n\t"
        "@p add.rn.f32 %0, %0, %12;\n\t"
        "@p add.rn.f32 %1, %1, %13;\n\t"
        "@p add.rn.f32 %2, %2, %14;\n\t"
        "@p add.rn.f32 %3, %3, %15;\n\t"
        "@p add.rn.f32 %4, %4, %16;\n\t"
        "@p add.rn.f32 %5, %5, %17;\n\t"
        "@c or.b32 %6, %6, %18;\n\t"
        "}"
        : "+f"(a.hx), "+f"(a.hy), "+f"(a.hz), "+f"(a.fx), "+f"(a.fy), "+f"(a.fz), "+r"(close)
        : "r"(mask), "r"(bit), "f"(r2), "f"(kNormal), "f"(near2), "f"(tx), "f"(ty), "f"(tz),
          "f"(sx), "f"(sy), "f"(sz), "r"(one));
}

// Sums the first cnt sources of the list (REC: and records the cells among them;
// particles are recorded where their leaf is opened).
template <bool REC>
__device__ __forceinline__ void sum_sources(WarpShared& w, int cnt, const Tree<float>& t,
                                            const FieldParams<float>& fp, float near2,
                                            const float4* __restrict__ pos,
                                            const float4* __restrict__ u, const Target& k, Sums& a,
                                            RecordWriter& rw, const EntryPool& ep)
{
    const int lane = threadIdx.x & 31;
    const uint32_t bit = 1u << lane;
    const float2 kx = dup2(k.x), ky = dup2(k.y), kz = dup2(k.z);
    const float2 ukx = dup2(k.ux), uky = dup2(k.uy), ukz = dup2(k.uz);
    for (int b = 0; b < cnt; b += 32) {
        __syncwarp();
        {
            uint2 e = make_uint2(0u, 0u);
            float4 c = make_float4(0.0f, 0.0f, 0.0f, 0.0f), m = c;
            if (b + lane < cnt) {
                e = w.q.list[b + lane];
                const uint32_t i = e.x & kIndex;
                const bool p = (e.x & kParticle) != 0u;
                c = p ? pos[i] : t.cell[i].cen;
                m = p ? u[i] : t.mom[i];
            }
            if (REC) {
                const uint32_t i = e.x & kIndex;
                const bool cell = b + lane < cnt && !(e.x & kParticle);
                // named by its place in the depth-first order of cells and particles
                const uint32_t key = cell ? i + (uint32_t)t.cell[i].node.x : 0u;
                rw.put(ep, cell, key, e.y);
            }
            float* st = w.stage + (lane >> 1) * kPairWords + (lane & 1);
            st[0] = -c.x;
            st[2] = -c.y;
            st[4] = -c.z;
            st[6] = -m.x;
            st[8] = -m.y;
            st[10] = -m.z;
            st[12] = __uint_as_float(e.y);
            st[14] = __uint_as_float(e.x);
        }
        __syncwarp();
        const int pairs = (min(32, cnt - b) + 1) >> 1;
        const float4* q = reinterpret_cast<const float4*>(w.stage);
        // this lane's sources for near_source: pairs' first and second ones
        uint32_t closeA = 0u, closeB = 0u, one = 1u;
#pragma unroll 2
        for (int p = 0; p < pairs; ++p, q += kPairWords / 4) {
            const float4 q0 = q[0], q1 = q[1], q2 = q[2];
            const uint2 mk = *reinterpret_cast<const uint2*>(q + 3);
            const float2 rx = __fadd2_rn(kx, make_float2(q0.x, q0.y));
            const float2 ry = __fadd2_rn(ky, make_float2(q0.z, q0.w));
            const float2 rz = __fadd2_rn(kz, make_float2(q1.x, q1.y));
            const float2 r2 = pair_r2_2(rx, ry, rz);
            if (REC) rw.nsrc += ((mk.x & bit) != 0u ? 1 : 0) + ((mk.y & bit) != 0u ? 1 : 0);
            const float2 ir = make_float2(rsqrt_normal(r2.x), rsqrt_normal(r2.y));
            const DipoleTerms2 d =
                dipole2(rx, ry, rz, ir, ukx, uky, ukz, make_float2(q1.z, q1.w),
                        make_float2(q2.x, q2.y), make_float2(q2.z, q2.w));
            add_if(mk.x, bit, r2.x, near2, d.tx.x, d.ty.x, d.tz.x, d.sx.x, d.sy.x, d.sz.x, a,
                   closeA, one);
            add_if(mk.y, bit, r2.y, near2, d.tx.y, d.ty.y, d.tz.y, d.sx.y, d.sy.y, d.sz.y, a,
                   closeB, one);
            one <<= 1;
        }
        // each lane its own close sources, in order
        while ((closeA | closeB) != 0u) {
            const int p = __ffs(closeA | closeB) - 1;
            const uint32_t pb = 1u << p;
            const float* st = w.stage + p * kPairWords + ((closeA & pb) ? 0 : 1);
            if (closeA & pb) closeA ^= pb;
            else closeB ^= pb;
            near_source(fp, t, k, __float_as_uint(st[14]), __fadd_rn(k.x, st[0]),
                        __fadd_rn(k.y, st[2]), __fadd_rn(k.z, st[4]), st[6], st[8], st[10], a);
        }
    }
    __syncwarp();
}

// Sums the list's full batches of 32 and moves the rest to its front; returns
// how many that is.
template <bool REC>
__device__ __forceinline__ int sum_full(WarpShared& w, int cnt, const Tree<float>& t,
                                        const FieldParams<float>& fp, float near2,
                                        const float4* __restrict__ pos,
                                        const float4* __restrict__ u, const Target& k, Sums& a,
                                        RecordWriter& rw, const EntryPool& ep)
{
    const int lane = threadIdx.x & 31, full = cnt & ~31;
    sum_sources<REC>(w, full, t, fp, near2, pos, u, k, a, rw, ep);
    uint2 e = make_uint2(0u, 0u);
    if (lane < cnt - full) e = w.q.list[full + lane];
    __syncwarp();
    if (lane < cnt - full) w.q.list[lane] = e;
    __syncwarp();
    return cnt - full;
}

__device__ __forceinline__ float warp_min(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(kFull, v, o));
    return v;
}

template <int T, bool REC>
__device__ __forceinline__ void walk_task(WarpShared& w, int task, const float4* __restrict__ pos,
                                          const float4* __restrict__ u, int n,
                                          const Tree<float>& t, const FieldParams<float>& fp,
                                          unsigned ncells, float4* __restrict__ h,
                                          float4* __restrict__ f, float* __restrict__ esr,
                                          int* flags, const uint32_t* __restrict__ off,
                                          const Segs& sg, const EntryPool& ep,
                                          int4* __restrict__ counts, uint32_t* __restrict__ tcount)
{
    const int lane = threadIdx.x & 31;
    const uint32_t lt = (1u << lane) - 1u;
    const int k0 = task * T, k = k0 + lane;
    const bool active = (T == 32 || lane < T) && k < n;
    const float4 xk = pos[active ? k : k0], uk = u[active ? k : k0];
    const Target tg = {xk.x, xk.y, xk.z, uk.x, uk.y, uk.z};
    Sums a = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
    const float lx = warp_min(xk.x), ly = warp_min(xk.y), lz = warp_min(xk.z);
    const float ux = -warp_min(-xk.x), uy = -warp_min(-xk.y), uz = -warp_min(-xk.z);
    // r^2 below which a source goes to near_source
    const float near2 = fp.include_sr ? fmaxf(fp.lj_rcut2_hi, kNormal) : kNormal;
    // the quick tests' bounds; with LJ off no cube is too near (far2 and rcut2 count as 0)
    const float th2lo = fp.theta2 * 0.99999f, th2hi = fp.theta2 * 1.00001f;
    const float rcut2 = fp.use_rcut ? fp.rcut2 : 0.0f;
    const unsigned max_rounds = 4u * ncells + 64u;
    // the roots of the task's systems, the first on top
    int top = 0;
    __syncwarp();
    {
        const uint32_t am = __ballot_sync(kFull, active);
        if (!sg.of_pos) {
            if (lane == 0) w.q.stack[0] = make_uint2(0u, am);
            top = 1;
        } else {
            const uint32_t sys = active ? sg.of_pos[k] : 0xffffffffu;
            const uint32_t mine = __match_any_sync(kFull, sys);
            const bool lead = active && (mine & lt) == 0u;
            const uint32_t lm = __ballot_sync(kFull, lead);
            top = __popc(lm);
            if (lead) w.q.stack[top - 1 - __popc(lm & lt)] = make_uint2(off[sg.start[sys]], mine);
        }
    }
    RecordWriter rw = {(uint32_t)task, 0u, 0u, 0};
    int cnt = 0;
    unsigned rounds = 0;
    while (top > 0) {
        __syncwarp();
        const int seen = min(32, top);
        uint2 e = make_uint2(kDone, 0u);
        if (lane < seen) e = w.q.stack[top - 1 - lane];
        __syncwarp();
        const uint32_t runs = __ballot_sync(kFull, (e.x & kRun) != 0u);
        if (runs & 1u) {
            // an opened leaf of several particles on top: each of them, for its lanes but itself
            const uint2 first = make_uint2(__shfl_sync(kFull, e.x, 0), __shfl_sync(kFull, e.y, 0));
            const int4 nd = t.cell[first.x & kIndex].node;
            for (int s0 = nd.x; s0 < nd.y; s0 += 32) {
                const int s = s0 + lane;
                uint32_t mask = s < nd.y ? first.y : 0u;
                if (s >= k0 && s < k0 + T) mask &= ~(1u << (s - k0));
                const uint32_t keep = __ballot_sync(kFull, mask != 0u);
                if (REC) rw.put(ep, mask != 0u, (first.x & kIndex) + 1u + (uint32_t)s, mask);
                if (mask) w.q.list[cnt + __popc(keep & lt)] = make_uint2((uint32_t)s | kParticle, mask);
                cnt += __popc(keep);
                if (cnt >= kBatch) cnt = sum_full<REC>(w, cnt, t, fp, near2, pos, u, tg, a, rw, ep);
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
        float far2;
        if (fresh) {
            const Cell<float> cl = t.cell[e.x];
            far2 = fp.use_rcut ? t.mom[e.x].w : 0.0f;
            lo = t.lo[e.x];
            nd = cl.node;
            c = cl.cen;
            const bool meets = nd.x < k0 + T && nd.y > k0;
            if (meets) {
                // the lanes whose particles it holds
                const int b = max(nd.x - k0, 0), m = min(nd.y - k0, T) - b;
                own = (m == 32 ? kFull : (1u << m) - 1u) << b;
            }
            if ((nd.w >> 9) != 0) {
                // a one-particle leaf: a source of every lane but its own particle's
                acc = e.y & ~own;
                src = e.x | kLeafCell;
            } else {
                // its children are looked up below if it is opened
                asm volatile("prefetch.global.L1 [%0];" ::"l"(t.child + 2 * (int64_t)e.x));
                const float ax = __fsub_rn(lx, c.x), bx = __fsub_rn(c.x, ux);
                const float ay = __fsub_rn(ly, c.y), by = __fsub_rn(c.y, uy);
                const float az = __fsub_rn(lz, c.z), bz = __fsub_rn(c.z, uz);
                const float gx = fmaxf(fmaxf(ax, bx), 0.0f), wx = fminf(ax, bx);
                const float gy = fmaxf(fmaxf(ay, by), 0.0f), wy = fminf(ay, by);
                const float gz = fmaxf(fmaxf(az, bz), 0.0f), wz = fminf(az, bz);
                // bounds of every lane's rounded d^2, with a margin far above the
                // rounding (a cell too small for the margin to hold is left to the lanes)
                const float dmin = (gx * gx + gy * gy + gz * gz) * 0.99999f;
                const float dmax = (wx * wx + wy * wy + wz * wz) * 1.00001f;
                const bool sized = c.w > 1e-30f;
                const bool all = sized && !meets && c.w < th2lo * dmin && dmin >= far2;
                const bool none = sized && c.w > th2hi * dmax;
                mixed = !all && !none;
                acc = all ? e.y : 0u;
                open = none ? e.y : 0u;
            }
        }
        const uint32_t mm = __ballot_sync(kFull, mixed);
        if (mm != 0u) {
            // handed round through shared memory (the staging space, free here)
            MixedCell* mc = reinterpret_cast<MixedCell*>(w.stage);
            const int rank = __popc(mm & lt), nm = __popc(mm);
            uint32_t got = 0u;
            if (mixed) {
                mc->c[rank] = c;
                mc->lo[rank] = make_float4(lo.x, lo.y, lo.z, far2);
                mc->hi[rank][0] = __fadd_rn(lo.x, lo.w);
                mc->hi[rank][1] = __fadd_rn(lo.y, lo.w);
                mc->hi[rank][2] = __fadd_rn(lo.z, lo.w);
            }
            __syncwarp();
#pragma unroll 2
            for (int r = 0; r < nm; ++r) {
                // accept(), its parts without branches
                const float4 cj = mc->c[r], lj = mc->lo[r];
                const float hx = mc->hi[r][0], hy = mc->hi[r][1], hz = mc->hi[r][2];
                const float dx = __fsub_rn(xk.x, cj.x), dy = __fsub_rn(xk.y, cj.y),
                            dz = __fsub_rn(xk.z, cj.z);
                const float d2 = __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)),
                                           __fmul_rn(dz, dz));
                const float gx = fmaxf(fmaxf(__fsub_rn(lj.x, xk.x), __fsub_rn(xk.x, hx)), 0.0f);
                const float gy = fmaxf(fmaxf(__fsub_rn(lj.y, xk.y), __fsub_rn(xk.y, hy)), 0.0f);
                const float gz = fmaxf(fmaxf(__fsub_rn(lj.z, xk.z), __fsub_rn(xk.z, hz)), 0.0f);
                const float b2 = __fadd_rn(__fadd_rn(__fmul_rn(gx, gx), __fmul_rn(gy, gy)),
                                           __fmul_rn(gz, gz));
                const bool ok = cj.w < __fmul_rn(fp.theta2, d2) && (d2 >= lj.w || !(b2 < rcut2));
                const uint32_t am = __ballot_sync(kFull, ok);
                if (rank == r) got = am;
            }
            if (mixed) {
                got &= ~own;  // its own particles do not accept it
                acc = e.y & got;
                open = e.y & ~got;
            }
        }
        const int emit = settle(w.q, cnt, lane, seen, runs, e, src, acc, open, nd.w, t.child, top);
        cnt += emit;
        if (cnt >= kBatch) {
            __syncwarp();
            cnt = sum_full<REC>(w, cnt, t, fp, near2, pos, u, tg, a, rw, ep);
        }
        // every round opens a cell or clears its part of the stack
        if (++rounds > max_rounds) {  // a damaged tree
            if (lane == 0) atomicOr(flags, FLAG_TRAVERSE);
            break;
        }
    }
    __syncwarp();
    sum_sources<REC>(w, cnt, t, fp, near2, pos, u, tg, a, rw, ep);
    if (REC && lane == 0) tcount[task] = rw.total;
    if (!active) return;
    if (REC) counts[k] = make_int4(rw.nsrc, 0, 0, 0);
    float4 ho, fo;
    ho.x = fp.dip_scale * a.hx;
    ho.y = fp.dip_scale * a.hy;
    ho.z = fp.dip_scale * a.hz;
    ho.w = 0.0f;
    fo.x = fp.dip_scale * a.fx + a.sx;
    fo.y = fp.dip_scale * a.fy + a.sy;
    fo.z = fp.dip_scale * a.fz + a.sz;
    fo.w = 0.0f;
    h[k] = ho;
    f[k] = fo;
    if (esr) esr[k] = a.es;
}

template <int T, bool REC>
__global__ void __launch_bounds__(kWalkThreads, kWalkBlocks) k_warp_walk(
    const float4* __restrict__ pos, const float4* __restrict__ u, int n, Tree<float> t,
    FieldParams<float> fp, float4* __restrict__ h, float4* __restrict__ f,
    float* __restrict__ esr, int* flags, int* __restrict__ work, int nseg,
    const uint32_t* __restrict__ off, Segs sg, EntryPool ep, int4* __restrict__ counts,
    uint32_t* __restrict__ tcount)
{
    extern __shared__ __align__(16) unsigned char walk_smem[];
    WarpShared& w = reinterpret_cast<WarpShared*>(walk_smem)[threadIdx.x >> 5];
    // a build that failed leaves no tree to walk (its flag reaches the host)
    if (*flags & (FLAG_CAPACITY | FLAG_SORT | FLAG_AGGREGATE | FLAG_NONFINITE)) return;
    const unsigned ncells = (unsigned)*t.ncells;
    const int ntask = (n + T - 1) / T;
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
            walk_task<T, REC>(w, task, pos, u, n, t, fp, ncells, h, f, esr, flags, off, sg, ep,
                              counts, tcount);
        }
    }
}

template <int T, bool REC = false>
void warp_walk_launch(const float4* pos, const float4* u, int64_t n, Tree<float> t,
                      FieldParams<float> fp, float4* h, float4* f, float* esr, int* flags,
                      int* work, const uint32_t* off, Segs sg, cudaStream_t s,
                      const EntryPool& ep = EntryPool(), int4* counts = nullptr,
                      uint32_t* tcount = nullptr)
{
    constexpr int smem = (int)sizeof(WarpShared) * (kWalkThreads / 32);
    static std::mutex mu;
    static PersistentGrid cache[kMaxDevices];
    const auto kern = k_warp_walk<T, REC>;
    const PersistentGrid g = persistent_grid(cache, mu, [kern] {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                             100 * ((smem + 1024) * kWalkBlocks) / (228 * 1024) + 1);
        int per_sm = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kWalkThreads, smem);
        return per_sm;
    });
    cudaMemsetAsync(work, 0, sizeof(int) * g.nseg, s);
    kern<<<g.blocks, kWalkThreads, smem, s>>>(pos, u, (int)n, t, fp, h, f, esr, flags, work, g.nseg,
                                              off, sg, ep, counts, tcount);
}

}  // namespace

// Targets per warp: the chip holds 2432 such warps.  Fewer targets a task mean
// more tasks in flight and fewer sources in each (a task of 8 passes 1180 cells
// on average where one of 32 passes 1700), but more work in all.  Measured on
// GB300, gases at volume fraction 0.05, ms per walk with 4 / 8 / 16 / 32 targets:
//   n = 1,000  0.161 / 0.167 / 0.178 / 0.190     n = 16,384  - / 0.337 / 0.316 / 0.334
//   n = 4,000  0.212 / 0.220 / 0.237 / 0.257     n = 32,768  - / 0.511 / 0.453 / 0.412
void warp_walk(const float4* pos, const float4* u, int64_t n, Tree<float> t,
               FieldParams<float> fp, float4* h, float4* f, float* esr, int* flags, int* work,
               const uint32_t* off, Segs sg, cudaStream_t s)
{
    if (n <= 4096)
        warp_walk_launch<4>(pos, u, n, t, fp, h, f, esr, flags, work, off, sg, s);
    else if (n <= 8192)
        warp_walk_launch<8>(pos, u, n, t, fp, h, f, esr, flags, work, off, sg, s);
    else if (n <= 26624)
        warp_walk_launch<16>(pos, u, n, t, fp, h, f, esr, flags, work, off, sg, s);
    else
        warp_walk_launch<32>(pos, u, n, t, fp, h, f, esr, flags, work, off, sg, s);
}

// The walk of the gradient pass, at any n: lists gathered from the one-lane walk
// (its counting instance writing every particle's sources, and a hash table per
// task merging 32 lists) cost 1.1 ms of 5.2 at n = 262,144.  Here a task's sources
// are known once, with the lanes that have them, as the walk goes.
void warp_walk_record(const float4* pos, const float4* u, int64_t n, Tree<float> t,
                      FieldParams<float> fp, float4* h, float4* f, float* esr, int4* counts,
                      uint32_t* tcount, int* flags, int* work, const uint32_t* off, Segs sg,
                      EntryPool pool, cudaStream_t s)
{
    if (n <= 0) return;
    warp_walk_launch<32, true>(pos, u, n, t, fp, h, f, esr, flags, work, off, sg, s, pool, counts,
                               tcount);
    counted();
}

}  // namespace ffk
