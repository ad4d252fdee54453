// ucp_lists.cuh -- the traversal shared by the walks over 32 targets: which boxes
// a chunk's targets accept and which leaves they open (Sec. 3, Eq. 5).
#pragma once

#include "ucp_internal.cuh"

#include <math.h>

namespace ucp {

__device__ __forceinline__ int next_chunk(int* work, int lane)
{
    int c = 0;
    if (lane == 0) c = atomicAdd(work, 1);
    return __shfl_sync(0xffffffffu, c, 0);
}

// The first box of a walk, in lane 0 (-1 elsewhere): the root of the targets' cloud, or
// none once a wait of the build gave up.  The tables are then no tree (children of several
// parents, leaves that end before they begin), and the walks' stacks hold only a tree's.
// gave_up: *a.err, which a kernel reads once at its start.
__device__ __forceinline__ int first_box(const WalkArgs& a, int gave_up, int cloud, int lane)
{
    return lane == 0 && !gave_up ? a.pos_off[a.t.cloud_start ? a.t.cloud_start[cloud] : 0] : -1;
}

// Twigs on the stack: up to kPopWide + 28 while four are popped per step; above
// kPopWide one is popped per step, which adds at most 7 per level below it.
constexpr int kPopWide = 64;
constexpr int kStack = kPopWide + 28 + 7 * (kMaxDepth - 1) + 8;

// x^-1/2 in FP64 by the cubic iteration y + y e (1/2 + 3/8 e), e = 1 - x y^2 (Householder's
// method of order two for the inverse square root), in three FP64 operations: one step of
// it on the special-function unit's value runs on the FP32 and integer units, which the
// FP64 walk leaves idle (an FP64 warp instruction takes its pipe for 16 cycles), with e
// from fused multiply-adds on the two parts of y^2 and of x, and gives 2^-45; that value,
// rounded to 26 bits so that its square is exact, starts the second step, whose factor
// 1/2 + 3/8 e follows from the rounding's remainder (e = 2 rem / y).  Close to
// correctly rounded (at most 1.0 x 2^-53 off, rms as the library's); 8 % of a walk
// against rsqrt() (block of 10 steps at N = 131,072: 86.9 -> 79.5 ms).  Arguments outside [2^-60, 2^100) go to the library.
__device__ __forceinline__ double rsqrt_fp64(double x)
{
    const unsigned int hi = (unsigned int)__double2hiint(x), lo = (unsigned int)__double2loint(x);
    if (hi - 0x3c300000u >= 0x46300000u - 0x3c300000u) return rsqrt(x);
    // x = xf + xl: the leading 24 bits and the other 29 as a float
    const unsigned int fb = __funnelshift_l(lo, hi - 0x38000000u, 3);
    const float xf = __uint_as_float(fb);
    const float xl = (float)(int)(lo & 0x1fffffffu) *
                     __uint_as_float((fb & 0x7f800000u) - (52u << 23));
    const float y = rsqrt_ftz(xf);
    const float p = y * y, pl = fmaf(y, y, -p);
    const float e = fmaf(-xf, pl, fmaf(-xl, p, fmaf(-xf, p, 1.f)));
    const float c = y * e * fmaf(0.375f, e, 0.5f);
    // y + c in units of the last place of a double, then d = its leading 26 bits
    const unsigned int yb = __float_as_uint(y);
    const float unit = __uint_as_float(((52u + 254u) << 23) - (yb & 0x7f800000u));
    const long long y1 = (long long)(((unsigned long long)yb << 29) + 0x3800000000000000ull) +
                         (long long)__float2int_rn(c * unit);
    const long long db = (y1 + (1ll << 26)) & ~((1ll << 27) - 1);
    const int rem = (int)(y1 - db);
    const double d = __longlong_as_double(db);
    // d (1/2 + 3/8 e) = d/2 (1 + 3/4 e)
    const double k = __longlong_as_double(db - (1ll << 52) + (long long)(rem + (rem >> 1)));
    return __fma_rn(k, __fma_rn(-x, __dmul_rn(d, d), 1.0), d);
}

// Eq. 5 for a target and a box's record m in FP64, rounded like the definition
static __device__ __noinline__ bool accepts_fp64(const double* m, const double* x, const double* y,
                                          const double* z)
{
    const double dx = __dsub_rn(*x, m[0]);
    const double dy = __dsub_rn(*y, m[1]);
    const double dz = __dsub_rn(*z, m[2]);
    return m[MR2] < __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

// A target of an FP64 context: its decisions are taken in FP32 on the traversal records and
// again in FP64 within the rounding of d2 - rcrit2.  Per axis R is off by at most 2^-23
// (|x_t| + |R|), so |error| <= 2^-22 sqrt(3) X d + 2^-21 d2 (rcrit2's rounding included),
// X the target's largest coordinate.  With d <= (d2 / u + u) / 2 that lies inside wa d2 + wb;
// u = side / 32 makes the window the same in every unit of length (u was 1: coordinates
// from 4e6 up or 1e-7 down were all decided twice) and keeps it narrow down to the smallest
// boxes.  1e-37 covers what underflows; where FP32's range ends, the window is infinite or
// not a number and FP64 decides.  At N = 20,000 and units of 2^-40, 2^20 and 2^40 a force
// call took 1.68, 1.52 and 1.59 ms, now 1.33 (r^2 past rsqrt_fp64's range), 1.24 and 1.24,
// as at 1; a vector-Jacobian product 13.4, 5.5 and 13.3 ms, now 3.6 to 3.7.
struct OneTarget {
    int t;
    float x, y, z, wa, wb;   // relative to the centre of the cloud's cube; the window

    __device__ __forceinline__ OneTarget(const WalkArgs& a, int t_, int cloud) : t(t_)
    {
        const Cube& cube = a.cubes[cloud];
        x = (float)(a.x[t] - cube.c[0]);
        y = (float)(a.y[t] - cube.c[1]);
        z = (float)(a.z[t] - cube.c[2]);
        const float b = 5e-7f * fmaxf(fabsf(x), fmaxf(fabsf(y), fabsf(z)));
        wa = fmaf(b, (float)(16.0 / 2097152.0 * cube.kscale), 4e-6f);   // kscale = 2^21 / side
        wb = fmaf(b, (float)cube.L * (1.f / 64.f), 1e-37f);
    }

    // does it accept the box of record h?
    __device__ __forceinline__ bool accepts(const WalkArgs& a, int box, const float4 h) const
    {
        const float rx = x + h.x, ry = y + h.y, rz = z + h.z;
        const float d2 = fmaf(rx, rx, fmaf(ry, ry, rz * rz));
        const float dm = d2 - fabsf(h.w);
        if (fabsf(dm) > fmaf(wa, d2, wb)) return dm > 0.f;
        return accepts_fp64(a.t.mom + (size_t)box * kMom, a.x + t, a.y + t, a.z + t);
    }
};

constexpr int kStage = 32;           // accepted boxes evaluated per batch
constexpr int kStageStride = 36;     // floats per staged pair of boxes (32 used; 16-byte aligned)

struct __align__(16) WalkWarp {
    float stage[kStage / 2 * kStageStride];
    int2 stack[kStack];              // {twig, mask}
    int2 acc[2 * kStage];            // {accepted box, mask}
    int2 leaf[64];                   // {opened leaf, mask}
};

__device__ __forceinline__ float warp_min(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

__device__ __forceinline__ float2 splat(float v) { return make_float2(v, v); }

// One target of a chunk (t < 0: an idle lane) and the chunk's bounds.
struct ChunkTarget {
    int t;
    // target as an unevaluated float pair x = xh + xl, relative to the centre of
    // the cloud's cube like the box centroids, so that the FP32 errors scale with
    // the cloud's size and not with its distance from the origin
    float xh, yh, zh, xl, yl, zl;
    // window of the FP32 criterion (see walk_lists): |dm| <= wa d2 + wb bounds the FP32
    // error of d2 - rcrit2 for this target, given |x_t - xh| <= 2^-24 |x_t| and the
    // same for the centroid
    float wa, wb;
    // bounding box of the chunk's targets (centre, half extents), and four times the
    // widest window of its targets: the centre and extents are rounded too
    float gx, gy, gz, ex, ey, ez, gwa, gwb;

    __device__ __forceinline__ ChunkTarget(const WalkArgs& a, int t_, int cloud) : t(t_)
    {
        xh = yh = zh = xl = yl = zl = 0.f;
        const bool valid = t >= 0;
        if (valid) {
            const double* cc = a.cubes[cloud].c;
            const double X = a.x[t] - cc[0], Y = a.y[t] - cc[1], Z = a.z[t] - cc[2];
            xh = (float)X; yh = (float)Y; zh = (float)Z;
            xl = (float)(X - (double)xh); yl = (float)(Y - (double)yh); zl = (float)(Z - (double)zh);
        }
        const float bt = 5e-7f * fmaxf(fabsf(xh), fmaxf(fabsf(yh), fabsf(zh)));
        wa = fmaf(0.5f, bt, 4e-6f);
        wb = 0.5f * bt;
        const float xa = warp_min(valid ? xh : INFINITY), xb = -warp_min(valid ? -xh : INFINITY);
        const float ya = warp_min(valid ? yh : INFINITY), yb = -warp_min(valid ? -yh : INFINITY);
        const float za = warp_min(valid ? zh : INFINITY), zb = -warp_min(valid ? -zh : INFINITY);
        gx = 0.5f * (xa + xb);
        gy = 0.5f * (ya + yb);
        gz = 0.5f * (za + zb);
        ex = fmaxf(xb - gx, gx - xa);
        ey = fmaxf(yb - gy, gy - ya);
        ez = fmaxf(zb - gz, gz - za);
        gwb = 4.f * -warp_min(-wb);
        gwa = gwb + 1.6e-5f;
    }
};

// The targets of `mask` that accept this lane's box (box < 0: none), h its record; called
// by the whole warp.
__device__ __forceinline__ unsigned int accept_mask(const WalkArgs& a, float* stage,
                                                    const ChunkTarget& tg, int box,
                                                    unsigned int mask, const float4 h)
{
    const int lane = threadIdx.x & 31;
    const unsigned int lt = (1u << lane) - 1u, me = 1u << lane;
    const bool has = box >= 0;
    const float rc2 = fabsf(h.w);
    const float dx = fabsf(tg.gx + h.x), dy = fabsf(tg.gy + h.y), dz = fabsf(tg.gz + h.z);
    const float nx = fmaxf(dx - tg.ex, 0.f), ny = fmaxf(dy - tg.ey, 0.f), nz = fmaxf(dz - tg.ez, 0.f);
    const float fx = dx + tg.ex, fy = dy + tg.ey, fz = dz + tg.ez;
    const float near2 = fmaf(nx, nx, fmaf(ny, ny, nz * nz));
    const float far2 = fmaf(fx, fx, fmaf(fy, fy, fz * fz));
    const bool all_acc = near2 - rc2 > fmaf(tg.gwa, near2, tg.gwb);
    const bool all_opn = rc2 - far2 > fmaf(tg.gwa, far2, tg.gwb);
    unsigned int am = has && all_acc ? mask : 0u;   // targets that accept the box
    const bool some = has && !all_acc && !all_opn;
    const unsigned int between = __ballot_sync(0xffffffffu, some);
    if (between) {
        // decided target by target, two boxes per packed operation: pairs of
        // {-c} x, y, z, {-rcrit2}, {box, mask}, side by side
        const int slot = some ? __popc(between & lt) : -1;
        const int cnt = __popc(between);
        if (some) {
            float* d = stage + (slot >> 1) * 12 + (slot & 1);
            d[0] = h.x;
            d[2] = h.y;
            d[4] = h.z;
            d[6] = -rc2;
            d[8] = __int_as_float(box);
            d[10] = __int_as_float((int)mask);
        }
        if (lane == 0 && (cnt & 1)) {
            float* d = stage + (cnt >> 1) * 12 + 1;
            d[0] = d[2] = d[4] = d[6] = d[8] = d[10] = 0.f;
        }
        __syncwarp();
        const float2 x2 = splat(tg.xh), y2 = splat(tg.yh), z2 = splat(tg.zh);
        for (int p = 0; 2 * p < cnt; ++p) {
            const float4* P = reinterpret_cast<const float4*>(stage + p * 12);
            const float4 f0 = P[0], f1 = P[1], f2 = P[2];
            const float2 rx = __fadd2_rn(x2, make_float2(f0.x, f0.y));
            const float2 ry = __fadd2_rn(y2, make_float2(f0.z, f0.w));
            const float2 rz = __fadd2_rn(z2, make_float2(f1.x, f1.y));
            const float2 d2 = __ffma2_rn(rx, rx, __ffma2_rn(ry, ry, __fmul2_rn(rz, rz)));
            const float2 dm = __fadd2_rn(d2, make_float2(f1.z, f1.w));
            const float2 win = __ffma2_rn(splat(tg.wa), d2, splat(tg.wb));
            const bool in0 = (__float_as_int(f2.z) & me) != 0;
            const bool in1 = (__float_as_int(f2.w) & me) != 0;
            bool acc0 = in0 && dm.x > 0.f, acc1 = in1 && dm.y > 0.f;
            // Within the FP32 error of d2 - rcrit2 the decision is taken again in
            // FP64 exactly as the FP64 walk takes it, so both precisions open the
            // same boxes.  Per axis R is off by at most 2^-23 (|x_t| + |R|), so
            // |error| <= 2^-22 sqrt(3) X_t d + 2^-21 d2 (rcrit2's rounding
            // included) with X_t the target's largest coordinate; with
            // d <= (d2 + 1) / 2 that lies inside wa d2 + wb (rare: a few tests in
            // a million at the bench size).  Where d2 overflows it is taken there too.
            const bool again0 = in0 && !(fabsf(dm.x) > win.x);
            const bool again1 = in1 && !(fabsf(dm.y) > win.y);
            if (again0)
                acc0 = accepts_fp64(a.t.mom + (size_t)__float_as_int(f2.x) * kCentre, a.x + tg.t,
                                    a.y + tg.t, a.z + tg.t);
            if (again1)
                acc1 = accepts_fp64(a.t.mom + (size_t)__float_as_int(f2.y) * kCentre, a.x + tg.t,
                                    a.y + tg.t, a.z + tg.t);
            const unsigned int am0 = __ballot_sync(0xffffffffu, acc0);
            const unsigned int am1 = __ballot_sync(0xffffffffu, acc1);
            if (slot == 2 * p) am = am0;
            if (slot == 2 * p + 1) am = am1;
        }
        __syncwarp();
    }
    return am;
}

// Walks targets, a bit each of `targets`, through their cloud's tree with the lanes over
// boxes: accept(box, mask, h) gives the targets of mask that accept a lane's box (< 0: none)
// of record h; multipoles(list, cnt) takes cnt <= 32 accepted boxes {box, mask of the
// targets that accept it}, pairs(list, cnt) cnt <= 32 opened leaves {leaf, mask of the
// targets that open it}; all are called by the whole warp and may use W.stage, the last two
// their part of the list.
template <class Accept, class Boxes, class Pairs>
__device__ __forceinline__ void walk_lists(const WalkArgs& a, int gave_up, WalkWarp& W,
                                           unsigned int targets, int cloud, Accept accept, Boxes& multipoles,
                                           Pairs& direct_pairs)
{
    const int lane = threadIdx.x & 31;
    const unsigned int lt = (1u << lane) - 1u;
    int top = 0, na = 0, nl = 0;
    // the first step tests the root for every target
    int box = first_box(a, gave_up, cloud, lane);
    unsigned int mask = targets;
    while (true) {
        const bool has = box >= 0;
        const float4 h = has ? __ldg(a.t.hdr + box) : make_float4(0.f, 0.f, 0.f, 0.f);
        const bool leaf = __float_as_int(h.w) < 0;
        // targets that accept the box
        const unsigned int am = accept(box, mask, h);
        const unsigned int om = has ? mask & ~am : 0u;  // targets that open it
        const unsigned int A = __ballot_sync(0xffffffffu, am != 0u);
        const unsigned int OL = __ballot_sync(0xffffffffu, om != 0u && leaf);
        const unsigned int OT = __ballot_sync(0xffffffffu, om != 0u && !leaf);
        if (am) W.acc[na + __popc(A & lt)] = make_int2(box, (int)am);
        if (om) {
            if (leaf) W.leaf[nl + __popc(OL & lt)] = make_int2(box, (int)om);
            else W.stack[top + __popc(OT & lt)] = make_int2(box, (int)om);
        }
        na += __popc(A);
        nl += __popc(OL);
        top += __popc(OT);
        __syncwarp();
        const bool done = top == 0;
        while (na >= kStage || (done && na > 0)) {
            const int cnt = min(na, kStage);
            na -= cnt;
            multipoles(W.acc + na, cnt);
        }
        while (nl >= 32 || (done && nl > 0)) {
            const int cnt = min(nl, 32);
            nl -= cnt;
            direct_pairs(W.leaf + nl, cnt);
        }
        if (done) break;
        const int pop = top > kPopWide ? 1 : min(top, 4);
        box = -1;
        mask = 0u;
        if ((lane >> 3) < pop) {
            const int2 e = W.stack[top - 1 - (lane >> 3)];
            box = __ldg(a.t.child8 + (size_t)e.x * 8 + (lane & 7));
            if (box <= e.x) box = -1;   // a child comes after its parent: the walk ends
            mask = (unsigned int)e.y;
        }
        top -= pop;
        __syncwarp();
    }
}

// The same for a chunk's targets, one per lane.
template <class Boxes, class Pairs>
__device__ __forceinline__ void walk_lists(const WalkArgs& a, int gave_up, WalkWarp& W,
                                           const ChunkTarget& tg, int cloud, Boxes& multipoles,
                                           Pairs& direct_pairs)
{
    walk_lists(a, gave_up, W, __ballot_sync(0xffffffffu, tg.t >= 0), cloud,
               [&](int box, unsigned int mask, const float4 h) {
                   return accept_mask(a, W.stage, tg, box, mask, h);
               },
               multipoles, direct_pairs);
}

// The particles of up to 32 opened leaves {leaf, mask} as one run over the lanes.
struct LeafRun {
    int total, end, first;       // end: of this lane's leaf in the run; first: begin - start
    int begin;                   // of this lane's leaf
    int2 lm;

    __device__ __forceinline__ LeafRun(const WalkArgs& a, const int2* leaves, int cnt)
    {
        const int lane = threadIdx.x & 31;
        int2 be = make_int2(0, 0);
        lm = make_int2(0, 0);
        if (lane < cnt) {
            lm = leaves[lane];
            be = __ldg(reinterpret_cast<const int2*>(a.t.info + lm.x));
        }
        end = be.y - be.x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, end, o);
            if (lane >= o) end += v;
        }
        total = __shfl_sync(0xffffffffu, end, 31);
        first = be.y - end;
        begin = be.x;
    }

    // particle f of the run: its slot, its leaf, that leaf's first slot and its mask (0
    // past the end)
    __device__ __forceinline__ void at(int f, int& j, int& leaf, int& leaf_begin,
                                       unsigned int& mask) const
    {
        int owner = 0;           // leaves that end at or before f
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            if (__shfl_sync(0xffffffffu, end, owner + o - 1) <= f) owner += o;
        j = __shfl_sync(0xffffffffu, first, owner) + f;
        leaf = __shfl_sync(0xffffffffu, lm.x, owner);
        leaf_begin = __shfl_sync(0xffffffffu, begin, owner);
        mask = (unsigned int)__shfl_sync(0xffffffffu, lm.y, owner);
        if (f >= total) mask = 0u;
    }
};

}  // namespace ucp
