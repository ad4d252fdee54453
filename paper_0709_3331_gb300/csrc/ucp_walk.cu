// ucp_walk.cu -- particle-TREE interaction of Sec. 3 (arXiv 0709.3331): for
// every target, boxes are visited from the root in pre-order; a box that
// satisfies the opening criterion of Eq. 5, s/theta + delta < d, acts through
// its expansion about its centroid (monopole, dipole, second moment of the
// softened kernel); an opened leaf is summed pair by pair.
//
// FP64 contexts walk one target per warp (k_walk_fp64), FP32C contexts 32
// key-consecutive targets per warp (k_walk_fp32c); each is described at its kernel.
// In both, each target's sums are taken in a fixed order, so results do not depend
// on scheduling.
#include "ucp_box.cuh"
#include "ucp_lists.cuh"

#include <math.h>

namespace ucp {

namespace {

// Error-free sum (Knuth's TwoSum) folded into a running correction.
__device__ __forceinline__ void two_sum_acc2(float2& s, float2& c, float2 v)
{
    const float2 n = make_float2(-1.f, -1.f);
    const float2 t = __fadd2_rn(s, v);
    const float2 bp = __ffma2_rn(n, s, t);
    const float2 ap = __ffma2_rn(n, bp, t);
    c = __fadd2_rn(c, __fadd2_rn(__ffma2_rn(n, ap, s), __ffma2_rn(n, bp, v)));
    s = t;
}

// ------------------------------------------------------------------ FP64
// One warp walks one target; its lanes are boxes and sources.  A step of the
// traversal pops up to four opened twigs from a stack and tests their children, one
// per lane; accepted boxes and the particles of opened leaves wait in two lists and
// are evaluated 32 at a time, one per lane.  The criterion is taken in FP32 on the
// traversal records and again in FP64 within its rounding window (see the FP32C
// walk), so the decisions are those of FP64.
//
// What bounds it: the FP64 pipe, which takes a warp instruction for 16 cycles
// however many of its lanes are active (2 multiply-adds per clock and SM).  One
// target per warp keeps all lanes at work in both lists (of 32 targets in a warp
// 65 % took part in a multipole and 35 % in a direct pair) and the FP32 criterion
// leaves the pipe to the interactions: a walk over N = 131,072 particles takes 12.7 ms
// (31.0 with 32 targets per warp, the criterion in FP64 and the library's root), over
// 2,048 0.10 ms (1.85).  A target's sums
// are over its own boxes and sources in an order set by the tree alone, so they do
// not depend on the launch.
//
// Expansion of a box at R = x_t - c, r2 = R.R + eps^2, g = r2^-1/2, u = g^2,
// w = D.R - tr(Q)/2, h = u R.Q.R:
//   phi = g (M + u (w + (3/2) h))
//   E   = g^3 [(M + 3u (w + (5/2) h)) R - (D + 3u Q R)]
// (the Taylor expansion of the softened kernel through second order, with the
// terms of each power of u collected).
template <bool kKelbg, bool kPhi>
__global__ void __launch_bounds__(32, 16)
k_walk_fp64(WalkArgs a)
{
    follow();
    __shared__ int stack[kStack], acc[64], src[64];
    const int lane = threadIdx.x;
    const unsigned int lt = (1u << lane) - 1u;
    const double q0 = a.qsp[0], q1 = a.qsp[1];
    const int gave_up = *a.err;
    const float4* __restrict__ H = a.t.hdr;
    const double* __restrict__ X = a.x;
    const double* __restrict__ Y = a.y;
    const double* __restrict__ Z = a.z;
    const int8_t* __restrict__ SP = a.sp;
    unsigned long long sum_p = 0, sum_m = 0;

    while (true) {
        const unsigned int item = (unsigned int)next_chunk(a.work, lane);
        if ((item >> 5) >= (unsigned int)a.nchunks) break;
        const int4 ck = a.chunks[item >> 5];
        const int place = (int)(item & 31u);
        if (place >= ck.y) continue;
        const int ti = ck.x + place;
        const int t = a.targets ? a.targets[ti] : ti;
        const double xt = X[t], yt = Y[t], zt = Z[t];
        const int8_t st = SP[t];
        const OneTarget tg(a, t, ck.z);
        double ex = 0.0, ey = 0.0, ez = 0.0, ph = 0.0;
        int top = 0, na = 0, nq = 0, np = 0, nm = 0;

        // the last cnt <= 32 accepted boxes
        auto multipoles = [&](int cnt) {
            na -= cnt;
            if (lane < cnt) {
                const double2* m =
                    reinterpret_cast<const double2*>(a.t.mom + (size_t)acc[na + lane] * kMom);
                const double2 m0 = m[0], m1 = m[1], m2 = m[2], m3 = m[3], m4 = m[4], m5 = m[5],
                              m6 = m[6], m7 = m[7];
                const double rx = xt - m0.x, ry = yt - m0.y, rz = zt - m1.x;
                const double r2 = rx * rx + (ry * ry + (rz * rz + a.eps2));
                const double M = m2.x;
                const double g = rsqrt_fp64(r2);
                const double u = g * g;
                const double g3 = g * u;
                const double qx = m4.x * rx + m4.y * ry + m5.x * rz;
                const double qy = m4.y * rx + m5.y * ry + m6.x * rz;
                const double qz = m5.x * rx + m6.x * ry + m6.y * rz;
                const double rqr = rx * qx + ry * qy + rz * qz;
                const double w = m2.y * rx + (m3.x * ry + (m3.y * rz + m7.y));
                const double h = u * rqr;
                const double s3 = 3.0 * u;
                const double k = M + s3 * (w + 2.5 * h);
                ex += g3 * (k * rx - (m2.y + s3 * qx));
                ey += g3 * (k * ry - (m3.x + s3 * qy));
                ez += g3 * (k * rz - (m3.y + s3 * qz));
                if (kPhi) ph += g * (M + u * (w + 1.5 * h));
            }
            __syncwarp();
        };
        // the last cnt <= 32 sources
        auto direct_pairs = [&](int cnt) {
            nq -= cnt;
            const int j = lane < cnt ? src[nq + lane] : t;
            if (j != t) {
                const double qj = SP[j] ? q1 : q0;
                const double dx = xt - X[j], dy = yt - Y[j], dz = zt - Z[j];
                if (kKelbg && SP[j] != st) {
                    // Sec. 2.1 Eq. 3: qj (1 - e)/r, e = exp(-r/lambda);
                    // E = qj r_vec [(1 - e)/r^3 - e/(lambda r^2)]
                    const double r = sqrt(dx * dx + dy * dy + dz * dz);
                    if (r == 0.0) {
                        ph += qj / a.lambda;
                    } else {
                        const double u = r / a.lambda;
                        const double e = exp(-u), ome = -expm1(-u);
                        const double f = ome / (r * r * r) - e / (a.lambda * r * r);
                        ex += qj * dx * f;
                        ey += qj * dy * f;
                        ez += qj * dz * f;
                        ph += qj * ome / r;
                    }
                } else {
                    const double ri = rsqrt_fp64(dx * dx + (dy * dy + (dz * dz + a.eps2)));
                    const double qi = qj * ri;
                    const double qr3 = qi * (ri * ri);
                    ex += qr3 * dx;
                    ey += qr3 * dy;
                    ez += qr3 * dz;
                    if (kPhi) ph += qi;
                }
            }
            np += __popc(__ballot_sync(0xffffffffu, j != t));
        };

        int box = first_box(a, gave_up, ck.z, lane);
        while (true) {
            const bool has = box >= 0;
            const float4 h = has ? __ldg(H + box) : make_float4(0.f, 0.f, 0.f, 0.f);
            const bool leaf = __float_as_int(h.w) < 0;
            const bool ok = has && tg.accepts(a, box, h);
            const unsigned int A = __ballot_sync(0xffffffffu, ok);
            const unsigned int OL = __ballot_sync(0xffffffffu, has && !ok && leaf);
            const unsigned int OT = __ballot_sync(0xffffffffu, has && !ok && !leaf);
            if (ok) acc[na + __popc(A & lt)] = box;
            if (has && !ok && !leaf) stack[top + __popc(OT & lt)] = box;
            na += __popc(A);
            nm += __popc(A);
            top += __popc(OT);
            __syncwarp();
            const bool done = top == 0;
            while (na >= 32 || (done && na > 0)) multipoles(min(na, 32));
            if (OL) {
                // the opened leaves' particles, in one run over the lanes
                int2 be = make_int2(0, 0);
                if ((OL >> lane) & 1u) be = __ldg(reinterpret_cast<const int2*>(a.t.info + box));
                int end = be.y - be.x;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int v = __shfl_up_sync(0xffffffffu, end, o);
                    if (lane >= o) end += v;
                }
                const int total = __shfl_sync(0xffffffffu, end, 31);
                const int first = be.y - end;      // particle f of the run in this leaf: first + f
                for (int base = 0; base < total; base += 32) {
                    const int f = base + lane;
                    int owner = 0;                 // lanes whose leaf ends at or before f
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1)
                        if (__shfl_sync(0xffffffffu, end, owner + o - 1) <= f) owner += o;
                    const int j = __shfl_sync(0xffffffffu, first, owner) + f;
                    if (f < total) src[nq + lane] = j;
                    nq += min(32, total - base);
                    __syncwarp();
                    if (nq >= 32) direct_pairs(32);
                    __syncwarp();
                }
            }
            if (done) {
                if (nq > 0) direct_pairs(nq);
                break;
            }
            const int pop = top > kPopWide ? 1 : min(top, 4);
            box = -1;
            if ((lane >> 3) < pop) {
                const int twig = stack[top - 1 - (lane >> 3)];
                box = __ldg(a.t.child8 + (size_t)twig * 8 + (lane & 7));
                if (box <= twig) box = -1;   // a child comes after its parent: the walk ends
            }
            top -= pop;
            __syncwarp();
        }
        __syncwarp();
        // sums over the lanes by halving exchanges (six additions for the four values):
        // lanes 0, 8, 16 and 24 end with x, y, z and the potential
        {
            const bool hi = lane & 16;
            const double k0 = hi ? ez : ex, k1 = hi ? ph : ey;
            const double s0 = hi ? ex : ez, s1 = hi ? ey : ph;
            const double v0 = k0 + __shfl_xor_sync(0xffffffffu, s0, 16);
            const double v1 = k1 + __shfl_xor_sync(0xffffffffu, s1, 16);
            const bool odd = lane & 8;
            double v = (odd ? v1 : v0) + __shfl_xor_sync(0xffffffffu, odd ? v0 : v1, 8);
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if ((lane & 7) == 0) {
                if (lane == 24) {
                    if (kPhi && a.phi) a.phi[t] = v;
                } else {
                    double* out = lane == 0 ? a.ax : lane == 8 ? a.ay : a.az;
                    out[t] = a.msp[2 + st] * v;
                }
            }
        }
        if (lane == 0) {
            a.cnt_p2p[t] = np;
            a.cnt_m2p[t] = nm;
        }
        sum_p += (unsigned long long)np;
        sum_m += (unsigned long long)nm;
    }
    if (lane == 0) {
        atomicAdd(&a.stats[0], sum_p);
        atomicAdd(&a.stats[1], sum_m);
    }
}

// ------------------------------------------------------------------ FP32C
// Kelbg factors of an unlike pair, u = r/lambda: its potential is q ri fp and its field
// q ri^3 fg r_vec, with fp = 1 - e^-u and fg = 1 - (1 + u) e^-u from u = 1/2 on.  Below, ri
// becomes 1/lambda and the factors fp / u and fg / u^3 follow from Taylor series (no
// cancellation, and no power of 1/r: the field of a close pair tends to q / (2 lambda^2),
// where r^-3 overflows from r = 1.5e-13 down).  ri comes in as rsqrt_ftz of d2 and is taken
// again where that flushed d2.  A pair at r = 0 takes the limits, potential 1/lambda and no
// field.
__device__ __forceinline__ void kelbg_factors(float d2, float& ri, float inv_lambda, float& fp,
                                              float& fg)
{
    if (d2 < 1.17549435e-38f) {      // the smallest normal float
        if (d2 == 0.f) {
            ri = inv_lambda;
            fp = 1.f;
            fg = 0.f;
            return;
        }
        ri = rsqrtf(d2);
    }
    const float u = d2 * ri * inv_lambda;
    if (u >= 0.5f) {
        const float e = __expf(-u);
        fp = 1.f - e;
        fg = 1.f - (1.f + u) * e;
    } else {
        fp = fmaf(u, fmaf(u, fmaf(u, fmaf(u, fmaf(u, fmaf(u, 1.f / 5040.f, -1.f / 720.f),
                                                 1.f / 120.f), -1.f / 24.f), 1.f / 6.f),
                          -0.5f), 1.f);
        const float poly = fmaf(u, fmaf(u, fmaf(u, fmaf(u, fmaf(u, 1.f / 5760.f, -1.f / 840.f),
                                                        1.f / 144.f), -1.f / 30.f), 0.125f),
                                -1.f / 3.f);
        fg = __fdividef(0.5f, u) + poly;
        ri = inv_lambda;
    }
}

// A target of the FP32C walk as the sums see it.
struct LaneTarget {
    int t, tmin, tmax;              // slots: its own, the chunk's lowest and highest
    float xh, yh, zh, xl, yl, zl, q, eps2, inv_lambda;
};

template <bool kKelbg>
__device__ __forceinline__ LaneTarget lane_target(const WalkArgs& a, const ChunkTarget& tg, int n)
{
    LaneTarget g;
    g.t = tg.t;
    // slots of the chunk's targets are ascending
    g.tmin = __shfl_sync(0xffffffffu, tg.t, 0);
    g.tmax = __shfl_sync(0xffffffffu, tg.t, n - 1);
    g.xh = tg.xh; g.yh = tg.yh; g.zh = tg.zh;
    g.xl = tg.xl; g.yl = tg.yl; g.zl = tg.zl;
    g.q = tg.t >= 0 ? (float)a.qsp[a.sp[tg.t] ? 1 : 0] : 0.f;
    g.eps2 = (float)a.eps2;
    g.inv_lambda = kKelbg ? (float)(1.0 / a.lambda) : 0.f;
    return g;
}

// The records of cnt <= 32 boxes into shared memory, the fields of two side by side, the
// last of them the box's mask (0 past the end).
__device__ __forceinline__ void stage_boxes(const WalkArgs& a, float* stage, const int2* boxes,
                                            int cnt)
{
    const int lane = threadIdx.x & 31;
    const int part = lane & 3;
#pragma unroll
    for (int it = 0; it < kStage / 8; ++it) {
        const int e = it * 8 + (lane >> 2);
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (e < cnt) v = __ldg(a.t.rec + (size_t)boxes[e].x * kRec + part);
        if (part == 3) v.w = __int_as_float(e < cnt ? boxes[e].y : 0);
        float* d = stage + (e >> 1) * kStageStride + part * 8 + (e & 1);
        d[0] = v.x;
        d[2] = v.y;
        d[4] = v.z;
        d[6] = v.w;
    }
}

// Multipoles, lanes over targets: the sums {x, y}, {z, potential} of cnt <= 32 accepted
// boxes (zeros outside their masks), staged two boxes side by side; nm counts them.
template <bool kPhi>
__device__ __forceinline__ void box_batch(const WalkArgs& a, float* stage, const int2* boxes, int cnt,
                                          const LaneTarget& g_, int& nm, float2& fxy, float2& fzp)
{
    const unsigned int me = 1u << (threadIdx.x & 31);
    const float xh = g_.xh, yh = g_.yh, zh = g_.zh, eps2 = g_.eps2;
    stage_boxes(a, stage, boxes, cnt);
    __syncwarp();
    // With g = (R.R + eps^2)^-1/2, u = g^2, q = Q R / 2, y = D + 5 u q:
    //   E   = -g^3 [y + u q - (M + 3 u (T + y.R)) R]
    //   phi = g (M + u (T + y.R - 2 u q.R)),   T = -tr(Q)/2
    float2 bx = splat(0.f), by = bx, bz = bx, bp = bx;
    const float2 x2 = splat(xh), y2 = splat(yh), z2 = splat(zh), e2 = splat(eps2);
    const int pairs = (cnt + 1) >> 1;
#pragma unroll 2
    for (int p = 0; p < pairs; ++p) {
        const float4* P = reinterpret_cast<const float4*>(stage + p * kStageStride);
        const float4 f0 = P[0], f1 = P[1], f2 = P[2], f3 = P[3], f4 = P[4], f5 = P[5],
                     f6 = P[6], f7 = P[7];
        const float2 rx = __fadd2_rn(x2, make_float2(f0.x, f0.y));
        const float2 ry = __fadd2_rn(y2, make_float2(f0.z, f0.w));
        const float2 rz = __fadd2_rn(z2, make_float2(f1.x, f1.y));
        const float2 r2 = __ffma2_rn(rx, rx, __ffma2_rn(ry, ry, __ffma2_rn(rz, rz, e2)));
        const bool in0 = (__float_as_int(f7.z) & me) != 0;
        const bool in1 = (__float_as_int(f7.w) & me) != 0;
        const float2 g = make_float2(in0 ? rsqrt_ftz(r2.x) : 0.f,
                                     in1 ? rsqrt_ftz(r2.y) : 0.f);
        nm += in0;
        nm += in1;
        const float2 u = __fmul2_rn(g, g);
        const float2 g3 = __fmul2_rn(g, u);
        const float2 qxx = make_float2(f4.x, f4.y), qxy = make_float2(f4.z, f4.w),
                     qxz = make_float2(f5.x, f5.y), qyy = make_float2(f5.z, f5.w),
                     qyz = make_float2(f6.x, f6.y), qzz = make_float2(f6.z, f6.w);
        const float2 qx = __ffma2_rn(qxx, rx, __ffma2_rn(qxy, ry, __fmul2_rn(qxz, rz)));
        const float2 qy = __ffma2_rn(qxy, rx, __ffma2_rn(qyy, ry, __fmul2_rn(qyz, rz)));
        const float2 qz = __ffma2_rn(qxz, rx, __ffma2_rn(qyz, ry, __fmul2_rn(qzz, rz)));
        const float2 u5 = __fmul2_rn(splat(5.f), u);
        const float2 yx = __ffma2_rn(u5, qx, make_float2(f2.x, f2.y));
        const float2 yy = __ffma2_rn(u5, qy, make_float2(f2.z, f2.w));
        const float2 yz = __ffma2_rn(u5, qz, make_float2(f3.x, f3.y));
        const float2 w = __ffma2_rn(yx, rx, __ffma2_rn(yy, ry, __ffma2_rn(yz, rz,
                                    make_float2(f3.z, f3.w))));
        const float2 nk = __ffma2_rn(__fmul2_rn(splat(-3.f), u), w,
                                     make_float2(f7.x, f7.y));
        bx = __ffma2_rn(g3, __ffma2_rn(nk, rx, __ffma2_rn(u, qx, yx)), bx);
        by = __ffma2_rn(g3, __ffma2_rn(nk, ry, __ffma2_rn(u, qy, yy)), by);
        bz = __ffma2_rn(g3, __ffma2_rn(nk, rz, __ffma2_rn(u, qz, yz)), bz);
        if (kPhi) {
            const float2 qr = __ffma2_rn(qx, rx, __ffma2_rn(qy, ry, __fmul2_rn(qz, rz)));
            const float2 v = __ffma2_rn(__fmul2_rn(splat(-2.f), u), qr, w);
            bp = __ffma2_rn(g, __ffma2_rn(u, v, make_float2(f1.z, f1.w)), bp);
        }
    }
    fxy = make_float2(-(bx.x + bx.y), -(by.x + by.y));
    fzp = make_float2(-(bz.x + bz.y), kPhi ? bp.x + bp.y : 0.f);
    __syncwarp();
}

// One pair of sources {nx0, nx1, ny0, ny1}, {nz0, nz1, q0, q1} on a target at r from their
// leaf's centroid, added to p (two sums side by side); ok: not the target itself.
struct PairSums {
    float2 x = splat(0.f), y = x, z = x, p = x;
};

template <bool kKelbg, bool kPhi>
__device__ __forceinline__ void add_pair(const float4 F, const float4 Q, float2 rx, float2 ry, float2 rz,
                                         const LaneTarget& g, bool ok0, bool ok1, PairSums& s)
{
    const float2 dx = __fadd2_rn(rx, make_float2(F.x, F.y));
    const float2 dy = __fadd2_rn(ry, make_float2(F.z, F.w));
    const float2 dz = __fadd2_rn(rz, make_float2(Q.x, Q.y));
    const float2 q = make_float2(Q.z, Q.w);
    if (kKelbg) {
        // unlike charges (electron-ion) take the Kelbg form, unsoftened
        const bool un0 = q.x != g.q, un1 = q.y != g.q;
        const float2 d2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
        const float2 r2 = __fadd2_rn(d2, make_float2(un0 ? 0.f : g.eps2,
                                                     un1 ? 0.f : g.eps2));
        float2 ri = make_float2(ok0 ? rsqrt_ftz(r2.x) : 0.f,
                                ok1 ? rsqrt_ftz(r2.y) : 0.f);
        float2 fp = splat(1.f), fg = fp;
        if (un0 && ok0) kelbg_factors(d2.x, ri.x, g.inv_lambda, fp.x, fg.x);
        if (un1 && ok1) kelbg_factors(d2.y, ri.y, g.inv_lambda, fp.y, fg.y);
        const float2 qi = __fmul2_rn(q, ri);
        const float2 qr3 = __fmul2_rn(__fmul2_rn(__fmul2_rn(qi, ri), ri), fg);
        s.x = __ffma2_rn(qr3, dx, s.x);
        s.y = __ffma2_rn(qr3, dy, s.y);
        s.z = __ffma2_rn(qr3, dz, s.z);
        s.p = __ffma2_rn(qi, fp, s.p);
    } else {
        const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __ffma2_rn(dz, dz, splat(g.eps2))));
        const float2 ri = make_float2(ok0 ? rsqrt_ftz(r2.x) : 0.f,
                                      ok1 ? rsqrt_ftz(r2.y) : 0.f);
        const float2 qi = __fmul2_rn(q, ri);
        const float2 qr3 = __fmul2_rn(__fmul2_rn(qi, ri), ri);
        s.x = __ffma2_rn(qr3, dx, s.x);
        s.y = __ffma2_rn(qr3, dy, s.y);
        s.z = __ffma2_rn(qr3, dz, s.z);
        if (kPhi) s.p = __fadd2_rn(s.p, qi);
    }
}

// A leaf of more than 32 sources, part by part: 16 pairs at a time from F through the buffer P
// (which holds the first) by the whole warp; mine: this lane's target opens it.  Out of line,
// so that the walks over shorter leaves do not pay for its registers (N = 524,288, leaves of
// 32, no potential: 2.28 ms, in line 2.32).  Straight from memory, pair by pair, a walk over
// 131,072 particles in leaves of 300 took 2.08 ms, now 1.26; over 524,288 with 52,428 of them
// at one place 6.4, now 4.2.
template <bool kKelbg, bool kPhi>
static __device__ __noinline__ PairSums long_leaf(const float4* F, float4* P, int pairs, float3 r,
                                                  float q, float eps2, float inv_lambda, int tp,
                                                  bool mine)
{
    const int lane = threadIdx.x & 31;
    LaneTarget g;
    g.q = q;
    g.eps2 = eps2;
    g.inv_lambda = inv_lambda;
    const float2 rx = splat(r.x), ry = splat(r.y), rz = splat(r.z);
    PairSums sum;
#pragma unroll 1
    for (int p0 = 0; p0 < pairs; p0 += 16) {
        float4 u = make_float4(0.f, 0.f, 0.f, 0.f);
        if (p0 + 16 < pairs) u = __ldg(F + 2 * (p0 + 16) + lane);
        if (mine) {
            const int last = min(16, pairs - p0);
#pragma unroll 2
            for (int p = 0; p < last; ++p)
                add_pair<kKelbg, kPhi>(P[2 * p], P[2 * p + 1], rx, ry, rz, g, 2 * (p0 + p) != tp,
                                       2 * (p0 + p) + 1 != tp, sum);
        }
        __syncwarp();
        P[lane] = u;
        __syncwarp();
    }
    return sum;
}

// Direct pairs, lanes over targets: cnt <= 32 opened leaves, each one's sources brought
// into shared memory (32 float4 at a time) while the leaf or the part before is summed;
// add(e, {x, y}, {z, potential}) takes leaf e's sums in the lanes of its mask.  kParts: leaves
// of more than 32 sources come in parts (long_leaf), else straight from memory (walks that
// would pay for it with shorter leaves: the Kelbg law's 1.5 %, and see below).
template <bool kKelbg, bool kPhi, bool kParts, class Add>
__device__ __forceinline__ void leaf_batch(const WalkArgs& a, float* stage, int2* leaves, int cnt,
                                           const LaneTarget& g_, int& np, Add add)
{
    const int lane = threadIdx.x & 31;
    const unsigned int me = 1u << lane;
    const float4* __restrict__ H = a.t.hdr;
    const float4* __restrict__ S = a.src32;
    const float xh = g_.xh, yh = g_.yh, zh = g_.zh, xl = g_.xl, yl = g_.yl, zl = g_.zl;
    const float qt = g_.q, eps2 = g_.eps2, inv_lambda = g_.inv_lambda;
    const int t = g_.t, tmin = g_.tmin, tmax = g_.tmax;
    float4* meta = reinterpret_cast<float4*>(stage);   // {-ch, place}, {-cl, begin}
    float4* buf = meta + 64;                             // 2 x 32 float4
    if (lane < cnt) {
        const int nd = leaves[lane].x;
        float4 A = __ldg(H + nd), B = __ldg(a.t.lo + nd);
        const int2 be = __ldg(reinterpret_cast<const int2*>(a.t.info + nd));
        A.w = __int_as_float(src_place(be.x, nd));
        B.w = __int_as_float(be.x);
        meta[2 * lane] = A;
        meta[2 * lane + 1] = B;
        leaves[lane].x = be.y - be.x;                    // {particles, mask}
    }
    __syncwarp();
    const float2 e2 = splat(eps2);
    float4 v = __ldg(S + __float_as_int(meta[0].w) + lane);
    for (int e = 0; e < cnt; ++e) {
        float4* P = buf + (e & 1) * 32;
        P[lane] = v;
        if (e + 1 < cnt) v = __ldg(S + __float_as_int(meta[2 * e + 2].w) + lane);
        __syncwarp();
        const int2 nm1 = leaves[e];
        if (kParts && nm1.x > 32) {
            const float4 A = meta[2 * e], B = meta[2 * e + 1];
            const int begin = __float_as_int(B.w), num = nm1.x;
            const bool mine = (nm1.y & me) != 0;
            const bool self = (unsigned int)(t - begin) < (unsigned int)num;
            const PairSums sum = long_leaf<kKelbg, kPhi>(
                S + __float_as_int(A.w), P, ((begin & 1) + num + 1) >> 1,
                make_float3((xh + A.x) + (xl + B.x), (yh + A.y) + (yl + B.y),
                            (zh + A.z) + (zl + B.z)),
                qt, eps2, inv_lambda, self ? t - (begin & ~1) : -1, mine);
            if (mine) {
                np += num - (self ? 1 : 0);
                add(e, make_float2(sum.x.x + sum.x.y, sum.y.x + sum.y.y),
                    make_float2(sum.z.x + sum.z.y, kPhi ? sum.p.x + sum.p.y : 0.f));
            }
            continue;
        }
        if (!(nm1.y & me)) continue;
        const float4 A = meta[2 * e], B = meta[2 * e + 1];
        const float2 rx = splat((xh + A.x) + (xl + B.x));
        const float2 ry = splat((yh + A.y) + (yl + B.y));
        const float2 rz = splat((zh + A.z) + (zl + B.z));
        const int begin = __float_as_int(B.w), num = nm1.x;
        const int pairs = ((begin & 1) + num + 1) >> 1;
        const bool self = (unsigned int)(t - begin) < (unsigned int)num;
        np += num - (self ? 1 : 0);
        // place of the target's own particle among the leaf's halves, or none
        const int tp = self ? t - (begin & ~1) : -1;
        PairSums sum;
        auto pair = [&](const float4 F, const float4 Q, bool ok0, bool ok1) {
            add_pair<kKelbg, kPhi>(F, Q, rx, ry, rz, g_, ok0, ok1, sum);
        };
        if (pairs > 16) {
            // one pair more than the buffer (32 sources from an odd place), or a long leaf
            // without parts: straight from memory
            const float4* F = S + __float_as_int(A.w);
#pragma unroll 1
            for (int p = 0; p < pairs; ++p)
                pair(__ldg(F + 2 * p), __ldg(F + 2 * p + 1), 2 * p != tp, 2 * p + 1 != tp);
        } else if (begin <= tmax && begin + num > tmin) {
            // may hold targets of the chunk
#pragma unroll 1
            for (int p = 0; p < pairs; ++p)
                pair(P[2 * p], P[2 * p + 1], 2 * p != tp, 2 * p + 1 != tp);
        } else {
#pragma unroll 2
            for (int p = 0; p < pairs; ++p) pair(P[2 * p], P[2 * p + 1], true, true);
        }
        add(e, make_float2(sum.x.x + sum.x.y, sum.y.x + sum.y.y),
            make_float2(sum.z.x + sum.z.y, kPhi ? sum.p.x + sum.p.y : 0.f));
    }
    __syncwarp();
}

// A target's results from its compensated sums, and the chunk's interaction counts.
template <bool kPhi>
__device__ __forceinline__ void write_target(const WalkArgs& a, int t, float2 sxy, float2 cxy,
                                             float2 szp, float2 czp, int np, int nm)
{
    if (t >= 0) {
        const int s = a.sp[t];
        const double qm = a.msp[2 + s];
        a.ax[t] = qm * ((double)sxy.x + (double)cxy.x);
        a.ay[t] = qm * ((double)sxy.y + (double)cxy.y);
        a.az[t] = qm * ((double)szp.x + (double)czp.x);
        if (kPhi && a.phi) a.phi[t] = (double)szp.y + (double)czp.y;
        a.cnt_p2p[t] = np;
        a.cnt_m2p[t] = nm;
    }
    unsigned long long sp2 = (unsigned long long)np, sm2 = (unsigned long long)nm;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        sp2 += __shfl_xor_sync(0xffffffffu, sp2, o);
        sm2 += __shfl_xor_sync(0xffffffffu, sm2, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&a.stats[0], sp2);
        atomicAdd(&a.stats[1], sm2);
    }
}

// One warp walks a chunk of up to 32 key-consecutive targets of one cloud, one per
// lane, in three parts that alternate:
//
// Traversal, lanes over boxes.  A stack holds opened twigs with the mask of the
// targets that opened them; a step pops up to four and tests their children, one
// per lane, against the bounding box of the chunk's targets: a child is accepted
// or opened by every target of its mask when the nearest or the farthest point of
// that bounding box decides it beyond the criterion's rounding window (four of five
// children at N = 524,288, theta 0.5), and only the children in between are decided
// target by target, two per packed operation.  The interaction sets are those of
// the per-target criterion.
//
// Multipoles, lanes over targets.  Accepted boxes wait in a list; 32 at a time their
// records are brought into shared memory (four lanes per 64-byte record) with the
// fields of two boxes side by side, and each lane evaluates two boxes per packed
// FP32x2 instruction (35 of them per pair of boxes).  A lane outside a box's mask
// takes a zero inverse distance.
//
// Direct pairs, lanes over targets: the opened leaves in lists of up to 63, each
// leaf's sources brought into shared memory while the leaf before it is summed.
//
// What bounds it (N = 524,288, theta 0.5, leaves of 32, no potential): per chunk
// 1,950 children tested in about 70 steps, 1,775 boxes evaluated (68 % of the lanes
// take part, the others accepted an ancestor) and 162 leaves of 11 sources summed
// (44 %); of the 2.28 ms of a walk over every particle the multipoles take 1.1 (the
// FP32 pipe: an FFMA2 holds it for two cycles; 61 % busy over the whole walk), the pairs
// 0.7 and the traversal 0.4.  A depth-first walk that tested one box per visit in all
// lanes and evaluated it one box at a time took 3.75 ms (1.81e5 against 1.12e5 warp
// instructions per chunk); with the potential 4.1 against 2.45 ms, over the electrons
// 2.25 against 1.38.  Blocks of one warp keep the shared arrays at constant
// addresses: 8 % faster than blocks of two to eight warps at the same occupancy.
//
// Register budget for kBlocks resident blocks (of one warp) per SM.  kPhi = false (walks whose potential nobody reads, e.g. the electron
// substeps): the potential terms and their sums are left out; the field is computed
// by the same operations in the same order, so accelerations are bit-identical.
template <bool kKelbg, int kBlocks, bool kPhi>
__global__ void __launch_bounds__(32, kBlocks)
k_walk_fp32c(WalkArgs a)
{
    follow();
    __shared__ WalkWarp W;
    const int lane = threadIdx.x;
    const int gave_up = *a.err;

    for (int item = next_chunk(a.work, lane); item < a.nchunks;
         item = next_chunk(a.work, lane)) {
        const long long began = clock64();
        const int chunk = a.ord.order[item];
        const int4 ck = a.chunks[chunk];
        const int ti = ck.x + lane;
        const int t = lane < ck.y ? (a.targets ? a.targets[ti] : ti) : -1;
        const ChunkTarget tg(a, t, ck.z);
        const LaneTarget lt = lane_target<kKelbg>(a, tg, ck.y);
        // compensated totals (sum, correction)
        float2 sxy = splat(0.f), szp = sxy, cxy = sxy, czp = sxy;   // {x, y}, {z, potential}
        int np = 0, nm = 0;
        auto multipoles = [&](const int2* boxes, int cnt) {
            float2 fxy, fzp;
            box_batch<kPhi>(a, W.stage, boxes, cnt, lt, nm, fxy, fzp);
            two_sum_acc2(sxy, cxy, fxy);
            two_sum_acc2(szp, czp, fzp);
        };
        // a leaf's pairs are summed in FP32 and enter the total by a compensated add
        // (folding every fourth leaf only is 1.5 % faster and 1 % less exact)
        auto direct_pairs = [&](int2* leaves, int cnt) {
            leaf_batch<kKelbg, kPhi, !kKelbg>(a, W.stage, leaves, cnt, lt, np,
                                     [&](int, const float2 fxy, const float2 fzp) {
                                         two_sum_acc2(sxy, cxy, fxy);
                                         two_sum_acc2(szp, czp, fzp);
                                     });
        };

        walk_lists(a, gave_up, W, tg, ck.z, multipoles, direct_pairs);

        write_target<kPhi>(a, t, sxy, cxy, szp, czp, np, nm);
        if (lane == 0) {
            const float cost = (float)(clock64() - began);
            a.ord.cost[chunk] = cost;
            atomicAdd(&a.ord.bins[cost_bin(cost)], 1);
        }
    }
}

// The same walk with kWays warps to a chunk, for systems too small to fill the SMs with a
// warp per chunk, whose walks take as long as one chunk does (its chain of box records,
// and one warp's rate of issue).  Every warp runs the whole traversal (they agree on it,
// reading the same boxes), and warp w evaluates every kWays-th batch of multipoles or of
// kSplitLeaves leaves into a slot of shared memory; one more warp adds the slots to the
// totals in the order in which k_walk_fp32c adds them, a round of kWays slots behind, so
// that the results are those of k_walk_fp32c bit for bit, whatever splits them.  N = 4099:
// 187 -> 88 us (Kelbg law 321 -> 118); 16384: 242 -> 143 us; 50,000: 399 -> 383 us; one
// warp per chunk again from 1520 chunks on (walk_fp32c_few).
constexpr int kSplitLeaves = 4;

struct SplitSlot {
    float4 v[kSplitLeaves][32];          // {x, y, z, potential} of a batch or leaf, per lane
    unsigned int mask[kSplitLeaves];     // lanes that add it; 0 ends the slot
};

template <int kWays>
struct SplitShared {
    WalkWarp warp[kWays];
    SplitSlot slot[2][kWays];
    int2 counts[kWays][32];              // {pairs, boxes} per lane
    int filled[2];                       // slots of a round; ~slots: the last round
};

//
// kParts (of contexts with leaf_cap > 32): long leaves in parts, 2.2 times as fast (30,000
// particles in leaves of 300: 960 -> 430 us), which costs walks over shorter leaves 5 to 12 %
// here (20,000 particles: 172 -> 192 us).
template <bool kKelbg, bool kPhi, int kWays, int kBlocks, bool kParts>
__global__ void __launch_bounds__((kWays + 1) * 32, kBlocks)
k_walk_fp32c_split(WalkArgs a)
{
    follow();
    extern __shared__ __align__(16) unsigned char split_bytes[];
    SplitShared<kWays>& sh = *reinterpret_cast<SplitShared<kWays>*>(split_bytes);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int gave_up = *a.err;
    const long long began = clock64();
    const int chunk = a.ord.order[blockIdx.x];
    const int4 ck = a.chunks[chunk];
    const int t = lane < ck.y ? (a.targets ? a.targets[ck.x + lane] : ck.x + lane) : -1;
    // all warps meet once per round
    auto meet = [] { asm volatile("bar.sync 1, %0;" ::"n"((kWays + 1) * 32) : "memory"); };
    if (w < kWays) {
        WalkWarp& W = sh.warp[w];
        const ChunkTarget tg(a, t, ck.z);
        const LaneTarget lt = lane_target<kKelbg>(a, tg, ck.y);
        int np = 0, nm = 0, task = 0, round = 0;
        auto turn = [&](auto fill) {
            if ((task & (kWays - 1)) == w) fill(sh.slot[round & 1][w]);
            if ((++task & (kWays - 1)) == 0) {
                if (threadIdx.x == 0) sh.filled[round & 1] = kWays;
                meet();
                ++round;
            }
        };
        auto multipoles = [&](const int2* boxes, int cnt) {
            turn([&](SplitSlot& s) {
                float2 fxy, fzp;
                box_batch<kPhi>(a, W.stage, boxes, cnt, lt, nm, fxy, fzp);
                s.v[0][lane] = make_float4(fxy.x, fxy.y, fzp.x, fzp.y);
                if (lane < kSplitLeaves) s.mask[lane] = lane == 0 ? 0xffffffffu : 0u;
            });
        };
        auto direct_pairs = [&](int2* leaves, int cnt) {
            for (int e0 = 0; e0 < cnt; e0 += kSplitLeaves)
                turn([&](SplitSlot& s) {
                    const int c = min(kSplitLeaves, cnt - e0);
                    if (lane < kSplitLeaves)
                        s.mask[lane] = lane < c ? (unsigned int)leaves[e0 + lane].y : 0u;
                    leaf_batch<kKelbg, kPhi, kParts>(a, W.stage, leaves + e0, c, lt, np,
                                             [&](int e, const float2 fxy, const float2 fzp) {
                                                 s.v[e][lane] = make_float4(fxy.x, fxy.y, fzp.x, fzp.y);
                                             });
                });
        };
        walk_lists(a, gave_up, W, tg, ck.z, multipoles, direct_pairs);
        sh.counts[w][lane] = make_int2(np, nm);
        if (threadIdx.x == 0) sh.filled[round & 1] = ~(task & (kWays - 1));
        meet();
    } else {
        float2 sxy = splat(0.f), szp = sxy, cxy = sxy, czp = sxy;
        int filled = 0;
        for (int round = 0; filled >= 0; ++round) {
            meet();
            filled = sh.filled[round & 1];
            const int slots = filled < 0 ? ~filled : filled;
            for (int k = 0; k < slots; ++k) {
                const SplitSlot& s = sh.slot[round & 1][k];
#pragma unroll
                for (int e = 0; e < kSplitLeaves; ++e) {
                    const unsigned int mask = s.mask[e];
                    if (!mask) break;
                    if (!(mask >> lane & 1u)) continue;
                    const float4 v = s.v[e][lane];
                    two_sum_acc2(sxy, cxy, make_float2(v.x, v.y));
                    two_sum_acc2(szp, czp, make_float2(v.z, v.w));
                }
            }
        }
        int np = 0, nm = 0;
        for (int k = 0; k < kWays; ++k) {
            np += sh.counts[k][lane].x;
            nm += sh.counts[k][lane].y;
        }
        write_target<kPhi>(a, t, sxy, cxy, szp, czp, np, nm);
        if (lane == 0) {
            const float cost = (float)(clock64() - began);
            a.ord.cost[chunk] = cost;
            atomicAdd(&a.ord.bins[cost_bin(cost)], 1);
        }
    }
}

// ---- The FP32C walk of ucp_grad_ke_electrons' forward runs: a chunk's targets visit
// boxes in pre-order, one box per step in all lanes, and multipoles are summed box by
// box, 32 visits to a compensated add; opened leaves wait in lists of 64.  Its forces
// agree with k_walk_fp32c's to about 2e-8, but the gradient of an unresolved run
// amplifies such a difference to 1e-3 of single components within 20 electron steps
// (close electron-ion encounters), and this order of sums is the one whose gradients the
// library has always returned.
//
// The traversal has its lanes over boxes, as walk_lists has, but opens one twig at a time:
// a stack holds the boxes to come, tested when their parent was opened, first on top; a
// step lists the visits up to the next opened twig and tests that twig's children.  After
// every 32 visits the round's leaves are summed as in k_walk_fp32c, then its accepted
// boxes, two to a packed operation but added one after the other.  With one box tested
// and evaluated per visit in all lanes the walk took 1.60 ms over the electrons at N =
// 262,144; this one takes 1.1 ms, a gradient of 20 steps 98.6 ms for 114.1.
//
// kTwo: a second warp does the sums, a round behind the first.  Where chunks are few it
// shortens the chain that such a walk waits for (20,000 particles: gradient 28.4 for
// 30.6 ms); from 60,000 on (938 chunks) the warps are better used on chunks.
constexpr int kVisitList = 64;      // opened leaves to a list
constexpr int kVisitBatch = 32;     // visits summed in FP32 before a compensated add
constexpr int kVisitRing = 256;     // leaves listed and not yet summed: < 64 + 2 (64 + 32)
constexpr int visit_blocks(bool two) { return two ? 12 : 24; }   // per SM
constexpr int kVisitStack = 7 * kMaxDepth + 8;

struct __align__(16) VisitShared {
    float stage[kStage / 2 * kStageStride];
    int2 box[2][kVisitBatch];       // {accepted box, mask} of a round
    int2 ring[kVisitRing];          // {opened leaf, mask}
    int2 leaf[32];
    int4 stack[kVisitStack];        // visits to come
    float test[16 * 12];            // of accept_mask, when stage is the other warp's
    int boxes[2], leaves[2];        // of a round: its boxes, the end of its leaves
    int last[2];
    int item;
};

// The accepted boxes of a round, added to b in order: cnt <= 32 as box_batch stages them.
// q is Q R / 2 and s6 = 6 u, exact doubles or halves of the terms of
//   E = -g^3 (3 u Q R + D) + g^3 (3 u (5/2 u R.Q R + D.R - tr(Q)/2) + M) R.
__device__ __forceinline__ void box_batch_in_order(const WalkArgs& a, float* stage,
                                                   const int2* boxes, int cnt,
                                                   const ChunkTarget& tg, float eps2, int& nm,
                                                   float& bx, float& by, float& bz)
{
    const unsigned int me = 1u << (threadIdx.x & 31);
    stage_boxes(a, stage, boxes, cnt);
    __syncwarp();
    const float2 x2 = splat(tg.xh), y2 = splat(tg.yh), z2 = splat(tg.zh), e2 = splat(eps2);
    const int pairs = (cnt + 1) >> 1;
#pragma unroll 2
    for (int p = 0; p < pairs; ++p) {
        const float4* P = reinterpret_cast<const float4*>(stage + p * kStageStride);
        const float4 f0 = P[0], f1 = P[1], f2 = P[2], f3 = P[3], f4 = P[4], f5 = P[5], f6 = P[6],
                     f7 = P[7];
        const float2 rx = __fadd2_rn(x2, make_float2(f0.x, f0.y));
        const float2 ry = __fadd2_rn(y2, make_float2(f0.z, f0.w));
        const float2 rz = __fadd2_rn(z2, make_float2(f1.x, f1.y));
        const float2 d2 = __ffma2_rn(rx, rx, __ffma2_rn(ry, ry, __fmul2_rn(rz, rz)));
        const float2 r2 = __fadd2_rn(d2, e2);
        const bool in0 = (__float_as_int(f7.z) & me) != 0;
        const bool in1 = (__float_as_int(f7.w) & me) != 0;
        const float2 g = make_float2(in0 ? rsqrt_ftz(r2.x) : 0.f, in1 ? rsqrt_ftz(r2.y) : 0.f);
        nm += in0;
        nm += in1;
        const float2 u = __fmul2_rn(g, g);
        const float2 g3 = __fmul2_rn(g, u);
        const float2 qxx = make_float2(f4.x, f4.y), qxy = make_float2(f4.z, f4.w),
                     qxz = make_float2(f5.x, f5.y), qyy = make_float2(f5.z, f5.w),
                     qyz = make_float2(f6.x, f6.y), qzz = make_float2(f6.z, f6.w);
        const float2 qx = __ffma2_rn(qxx, rx, __ffma2_rn(qxy, ry, __fmul2_rn(qxz, rz)));
        const float2 qy = __ffma2_rn(qxy, rx, __ffma2_rn(qyy, ry, __fmul2_rn(qyz, rz)));
        const float2 qz = __ffma2_rn(qxz, rx, __ffma2_rn(qyz, ry, __fmul2_rn(qzz, rz)));
        const float2 rqr = __ffma2_rn(rx, qx, __ffma2_rn(ry, qy, __fmul2_rn(rz, qz)));
        const float2 dx = make_float2(f2.x, f2.y), dy = make_float2(f2.z, f2.w),
                     dz = make_float2(f3.x, f3.y);
        const float2 w = __ffma2_rn(dx, rx, __ffma2_rn(dy, ry, __ffma2_rn(dz, rz,
                                    make_float2(f3.z, f3.w))));
        const float2 s3 = __fmul2_rn(splat(3.f), u), s6 = __fadd2_rn(s3, s3);
        const float2 aa = __fmul2_rn(g3, __ffma2_rn(s3, __ffma2_rn(splat(5.f), __fmul2_rn(u, rqr), w),
                                                    make_float2(f1.z, f1.w)));
        const float2 ex = __ffma2_rn(s6, qx, dx), ey = __ffma2_rn(s6, qy, dy),
                     ez = __ffma2_rn(s6, qz, dz);
        bx = fmaf(-g3.x, ex.x, fmaf(aa.x, rx.x, bx));
        by = fmaf(-g3.x, ey.x, fmaf(aa.x, ry.x, by));
        bz = fmaf(-g3.x, ez.x, fmaf(aa.x, rz.x, bz));
        bx = fmaf(-g3.y, ex.y, fmaf(aa.y, rx.y, bx));
        by = fmaf(-g3.y, ey.y, fmaf(aa.y, ry.y, by));
        bz = fmaf(-g3.y, ez.y, fmaf(aa.y, rz.y, bz));
    }
    __syncwarp();
}

template <bool kTwo, bool kParts>
__global__ void __launch_bounds__(kTwo ? 64 : 32, visit_blocks(kTwo))
k_walk_fp32c_visits(WalkArgs a)
{
    follow();
    __shared__ __align__(16) VisitShared sh;
    const int lane = threadIdx.x & 31;
    const unsigned int lt = (1u << lane) - 1u;
    const bool traverses = threadIdx.x < 32, sums = !kTwo || threadIdx.x >= 32;
    const float4* __restrict__ H = a.t.hdr;
    const float eps2 = (float)a.eps2;
    const int gave_up = *a.err;

    while (true) {
        if (threadIdx.x == 0) sh.item = atomicAdd(a.work, 1);
        __syncthreads();
        const int item = sh.item;
        if (item >= a.nchunks) break;
        const long long began = clock64();
        const int chunk = a.ord.order[item];
        const int4 ck = a.chunks[chunk];
        const int t = lane < ck.y ? (a.targets ? a.targets[ck.x + lane] : ck.x + lane) : -1;
        const ChunkTarget tg(a, t, ck.z);
        float2 sxy = splat(0.f), sz0 = sxy, cxy = sxy, cz0 = sxy;
        int np = 0, nm = 0, done = 0;
        // a round: its leaves, then its boxes
        auto sum_round = [&](int r) {
            const int cnt = sh.boxes[r], upto = sh.leaves[r];
            if (done < upto) {
                LaneTarget lt;
                lt.t = t;
                lt.tmin = __shfl_sync(0xffffffffu, t, 0);
                lt.tmax = __shfl_sync(0xffffffffu, t, ck.y - 1);
                lt.xh = tg.xh; lt.yh = tg.yh; lt.zh = tg.zh;
                lt.xl = tg.xl; lt.yl = tg.yl; lt.zl = tg.zl;
                lt.q = lt.inv_lambda = 0.f;
                lt.eps2 = eps2;
                while (done < upto) {
                    const int m = min(32, upto - done);
                    if (lane < m) sh.leaf[lane] = sh.ring[(done + lane) & (kVisitRing - 1)];
                    __syncwarp();
                    leaf_batch<false, false, kParts>(a, sh.stage, sh.leaf, m, lt, np,
                                             [&](int, const float2 fxy, const float2 fzp) {
                                                 two_sum_acc2(sxy, cxy, fxy);
                                                 two_sum_acc2(sz0, cz0, fzp);
                                             });
                    done += m;
                }
            }
            float bx = 0.f, by = 0.f, bz = 0.f;
            if (cnt) box_batch_in_order(a, sh.stage, sh.box[r], cnt, tg, eps2, nm, bx, by, bz);
            two_sum_acc2(sxy, cxy, make_float2(bx, by));
            two_sum_acc2(sz0, cz0, make_float2(bz, 0.f));
        };
        // the two warps meet once per round
        auto meet = [] { asm volatile("bar.sync 1, 64;" ::: "memory"); };
        if (traverses) {
            int vis = 0, r = 0, nb = 0, listed = 0, given = 0;   // leaves listed, given on
            auto close = [&](bool last) {
                if (lane == 0) {
                    sh.boxes[r] = nb;
                    sh.leaves[r] = given;
                    sh.last[r] = last;
                }
                nb = 0;
                if (kTwo) {
                    meet();
                    r ^= 1;
                } else {
                    __syncwarp();
                    sum_round(0);
                    __syncwarp();
                }
            };
            // lists the visits of lanes [from, to) of a window, in order; ends: the last of
            // them is the last of its round
            auto list = [&](const int4 e, int from, int to, bool ends) {
                const bool mine = lane >= from && lane < to;
                const unsigned int am = __ballot_sync(0xffffffffu, mine && e.y != 0);
                if (mine && e.y) sh.box[r][nb + __popc(am & lt)] = make_int2(e.x, e.y);
                nb += __popc(am);
                const unsigned int ol = __ballot_sync(0xffffffffu, mine && e.z != 0 && e.w != 0);
                if (mine && e.z && e.w)
                    sh.ring[(listed + __popc(ol & lt)) & (kVisitRing - 1)] = make_int2(e.x, e.z);
                listed += __popc(ol);
                // a full list is summed before the boxes of the visit after its last leaf
                const bool full = listed - given >= kVisitList;
                const bool late = full && ends && listed - given == kVisitList && (ol >> (to - 1) & 1u);
                if (full && !late) given += kVisitList;
                if (ends) close(false);
                if (late) given += kVisitList;
            };
            int top = 0;
            int box = first_box(a, gave_up, ck.z, lane);
            unsigned int mask = __ballot_sync(0xffffffffu, t >= 0);
            while (true) {
                // the boxes that follow, first on top: {box, accepting, opening targets, leaf}
                const float4 h = box >= 0 ? __ldg(H + box) : make_float4(0.f, 0.f, 0.f, 0.f);
                const unsigned int am = accept_mask(a, sh.test, tg, box, mask, h);
                const unsigned int follow_up = __ballot_sync(0xffffffffu, box >= 0);
                if (box >= 0)
                    sh.stack[top + __popc(follow_up & ~lt) - 1] =
                        make_int4(box, (int)am, (int)(mask & ~am), __float_as_int(h.w) < 0);
                top += __popc(follow_up);
                __syncwarp();
                // visits up to the next opened twig
                int4 e;
                unsigned int twigs;
                int n;
                do {
                    const int cnt = min(top, 32);
                    e = lane < cnt ? sh.stack[top - 1 - lane] : make_int4(-1, 0, 0, 0);
                    twigs = __ballot_sync(0xffffffffu, e.z != 0 && e.w == 0);
                    n = twigs ? __ffs(twigs) : cnt;
                    const int room = kVisitBatch - (vis & (kVisitBatch - 1));
                    list(e, 0, min(n, room), n >= room);
                    if (n > room) list(e, room, n, false);
                    vis += n;
                    top -= n;
                } while (!twigs && top > 0);
                if (!twigs) break;
                const int twig = __shfl_sync(0xffffffffu, e.x, n - 1);
                mask = (unsigned int)__shfl_sync(0xffffffffu, e.z, n - 1);
                __syncwarp();
                box = lane < 8 ? __ldg(a.t.child8 + (size_t)twig * 8 + lane) : -1;
                if (box <= twig) box = -1;      // a child comes after its parent: the walk ends
            }
            given = listed;
            close(true);
        } else {
            int r = 0;
            bool last = false;
            while (!last) {
                meet();
                last = sh.last[r];
                sum_round(r);
                r ^= 1;
            }
        }
        if (sums) {
            write_target<false>(a, t, sxy, cxy, sz0, cz0, np, nm);
            if (lane == 0) {
                const float cost = (float)(clock64() - began);
                a.ord.cost[chunk] = cost;
                atomicAdd(&a.ord.bins[cost_bin(cost)], 1);
            }
        }
        __syncthreads();
    }
}

// Per walk: rcrit2 = (s/theta + delta)^2 of every box in FP64 (theta = 0:
// +inf, nothing accepted), and the FP32C box records.  In an FP64 context (kFp64) the
// moments and delta of every box that still holds the sums its build left are made from
// them first, one box per lane: nearly all FP64 work, so its blocks are small and spread
// over the SMs.
constexpr int prep_threads(bool fp64) { return fp64 ? 64 : 256; }

template <bool kFp64>
__global__ void __launch_bounds__(prep_threads(kFp64))
k_mac_prepare(Tree t, const Cube* __restrict__ cube, double theta, int* work, int* bins)
{
    follow();
    if (blockIdx.x == 0) {
        if (threadIdx.x == 0) *work = 0;
        if (bins)
            for (int i = threadIdx.x; i < 2 * kCostBins; i += blockDim.x) bins[i] = 0;
    }
    const int nn = *t.nnodes;
    for (int nd = blockIdx.x * blockDim.x + threadIdx.x; nd < nn; nd += gridDim.x * blockDim.x) {
        double* m = t.mom + (size_t)nd * (kFp64 ? kMom : kCentre);
        int dl = t.depth_leaf[nd];
        const Cube& cb = cube[t.cloud ? t.cloud[t.info[nd].x] : 0];
        const double L = cb.L;
        double s = ldexp(L, -(dl & 255));
        // (everything loaded before the test, so that no load waits for another)
        double a[14], delta = t.delta[nd], c[3] = {m[MC], m[MC + 1], m[MC + 2]};
        if (kFp64) {
            const double2* r = reinterpret_cast<const double2*>(m);
#pragma unroll
            for (int k = 0; k < 7; ++k) {
                const double2 v = r[k];
                a[2 * k] = v.x;
                a[2 * k + 1] = v.y;
            }
        }
        if (kFp64 && delta == kSumsDelta) {
            double z[3], rho[3], rec[kMom];
            box_centre_exact(cb, t.cell[nd], dl & 255, z, rho);
            finish_box(a, z, rho, rec, &delta);
            t.delta[nd] = delta;
#pragma unroll
            for (int k = 0; k < 3; ++k) c[k] = rec[MC + k];
#pragma unroll
            for (int k = 0; k < kMom; ++k)
                if (k != MR2) m[k] = rec[k];
        }
        double r2;
        if (theta > 0.0) {
            double rc = __dadd_rn(__ddiv_rn(s, theta), delta);
            r2 = __dmul_rn(rc, rc);
        } else {
            r2 = INFINITY;
        }
        m[MR2] = r2;
        // the centroid, relative to the cube's centre as the walk's targets are,
        // enters negated (x_t - c as a sum); the trace term of the expansion as
        // one value
        const double ux = c[0] - cb.c[0], uy = c[1] - cb.c[1], uz = c[2] - cb.c[2];
        const float chx = (float)ux, chy = (float)uy, chz = (float)uz;
        // finite as r2 is: past the range of FP32 it stands for "larger", and a box as far
        // away is decided in FP64
        const float rc2 = theta > 0.0 ? fminf((float)r2, 3.40282347e38f) : (float)r2;
        t.hdr[nd] = make_float4(-chx, -chy, -chz, (dl & 256) ? -rc2 : rc2);
        if (!kFp64) {
            t.lo[nd] = make_float4((float)((double)chx - ux), (float)((double)chy - uy),
                                   (float)((double)chz - uz), 0.f);
            const float4* m32 = reinterpret_cast<const float4*>(t.mom32 + (size_t)nd * 16);
            const float4 f1 = m32[1], f2 = m32[2], f3 = m32[3];   // {M, D}, {Q..}, {Q.., 0, 0}
            const float M = f1.x, qxx = f2.x, qyy = f2.w, qzz = f3.y;
            float4* r = t.rec + (size_t)nd * kRec;
            r[0] = make_float4(-chx, -chy, -chz, M);
            r[1] = make_float4(f1.y, f1.z, f1.w, -0.5f * ((qxx + qyy) + qzz));
            r[2] = make_float4(0.5f * qxx, 0.5f * f2.y, 0.5f * f2.z, 0.5f * qyy);
            r[3] = make_float4(0.5f * f3.x, 0.5f * qzz, -M, 0.f);
        }
    }
}

}  // namespace

void launch_mac_prepare(Tree t, const Cube* cube, double theta, int want_f32, int* work, int* bins,
                        Queue s)
{
    count_launch(1);
    if (want_f32)
        launch(k_mac_prepare<false>, 4 * 152, prep_threads(false), s, t, cube, theta, work, bins);
    else
        launch(k_mac_prepare<true>, 16 * 152, prep_threads(true), s, t, cube, theta, work, bins);
}

// blocks of one warp: per_sm on every SM, or one per work item
static int walk_blocks(int64_t items, int nsm, int per_sm)
{
    const int blocks = nsm * per_sm < items ? nsm * per_sm : (int)items;
    return blocks < 1 ? 1 : blocks;
}

void launch_walk_fp64(const WalkArgs& a, int nsm, Queue s)
{
    count_launch(1);
    const int b = walk_blocks((int64_t)a.nchunks * 32, nsm, 16);
    // the potential is computed only when the caller reads it
    if (a.kelbg && a.phi) launch(k_walk_fp64<true, true>, b, 32, s.whole(), a);
    else if (a.kelbg) launch(k_walk_fp64<true, false>, b, 32, s.whole(), a);
    else if (a.phi) launch(k_walk_fp64<false, true>, b, 32, s.whole(), a);
    else launch(k_walk_fp64<false, false>, b, 32, s.whole(), a);
}

// Launch shapes of the FP32C walk that the autotuner chooses from: blocks of one
// warp, and how many of them are resident per SM, which sets the register budget,
// {threads, blocks, 0}.  The persistent grid takes 32-target chunks from a counter,
// so the shape changes the schedule, never a result.  (Of walks with more than 10 chunks
// per SM; smaller ones take the block that suits their size, see walk_fp32c_few.)
static const int kShapes[][3] = {{32, 24, 0}, {32, 20, 0}, {32, 28, 0}, {32, 32, 0},
                                 {32, 16, 0}, {32, 18, 0}, {32, 22, 0}, {32, 26, 0},
                                 {32, 14, 0}, {32, 12, 0}};
int walk_shape_count() { return (int)(sizeof(kShapes) / sizeof(kShapes[0])); }

template <bool kKelbg, bool kPhi>
static void walk_fp32c_shape(const WalkArgs& a, int per_sm, int b, Queue s)
{
    switch (per_sm) {
    case 12: launch(k_walk_fp32c<kKelbg, 12, kPhi>, b, 32, s.whole(), a); break;
    case 14: launch(k_walk_fp32c<kKelbg, 14, kPhi>, b, 32, s.whole(), a); break;
    case 16: launch(k_walk_fp32c<kKelbg, 16, kPhi>, b, 32, s.whole(), a); break;
    case 18: launch(k_walk_fp32c<kKelbg, 18, kPhi>, b, 32, s.whole(), a); break;
    case 20: launch(k_walk_fp32c<kKelbg, 20, kPhi>, b, 32, s.whole(), a); break;
    case 22: launch(k_walk_fp32c<kKelbg, 22, kPhi>, b, 32, s.whole(), a); break;
    case 26: launch(k_walk_fp32c<kKelbg, 26, kPhi>, b, 32, s.whole(), a); break;
    case 28: launch(k_walk_fp32c<kKelbg, 28, kPhi>, b, 32, s.whole(), a); break;
    case 32: launch(k_walk_fp32c<kKelbg, 32, kPhi>, b, 32, s.whole(), a); break;
    default: launch(k_walk_fp32c<kKelbg, 24, kPhi>, b, 32, s.whole(), a); break;
    }
}

template <bool kKelbg, bool kPhi, int kWays, int kBlocks, bool kParts>
static void walk_fp32c_split_form(const WalkArgs& a, Queue s)
{
    const int bytes = (int)sizeof(SplitShared<kWays>);
    cudaFuncSetAttribute(k_walk_fp32c_split<kKelbg, kPhi, kWays, kBlocks, kParts>,
                         cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    launch_shared(k_walk_fp32c_split<kKelbg, kPhi, kWays, kBlocks, kParts>, a.nchunks,
                  (kWays + 1) * 32, bytes, s.whole(), a);
}

template <bool kKelbg, bool kPhi, int kWays, int kBlocks>
static void walk_fp32c_split(const WalkArgs& a, Queue s)
{
    if (!kKelbg && a.leaf_cap > 32)
        walk_fp32c_split_form<kKelbg, kPhi, kWays, kBlocks, !kKelbg>(a, s);
    else walk_fp32c_split_form<kKelbg, kPhi, kWays, kBlocks, false>(a, s);
}

// Walks whose chunks are few enough for several warps each: a block per chunk, all of them
// resident at once (the last rule: nearly), with the register budget that this number of
// blocks per SM leaves.  The lines lie where the next rule is as fast, in us for 8, 4 (3
// blocks per SM), 4 (5 blocks), 2 warps and 1 warp to a chunk, theta 0.5, with potential:
//   256 chunks 116 126 140 188 225     512 chunks 170 143 163 207 242
//   750 chunks 244 206 177 226 281    1024 chunks 335 280 256 256 310
//  1563 chunks 537 433 378 383 399    2048 chunks 697 567 482 461 444
template <bool kKelbg, bool kPhi>
static bool walk_fp32c_few(const WalkArgs& a, int nsm, Queue s)
{
    if (a.nchunks <= 2 * nsm) walk_fp32c_split<kKelbg, kPhi, 8, 2>(a, s);
    else if (a.nchunks <= 4 * nsm) walk_fp32c_split<kKelbg, kPhi, 4, 3>(a, s);
    else if (a.nchunks <= 5 * nsm) walk_fp32c_split<kKelbg, kPhi, 4, 5>(a, s);
    else if (a.nchunks <= 10 * nsm) walk_fp32c_split<kKelbg, kPhi, 2, 8>(a, s);
    else return false;
    return true;
}

void launch_walk_fp32c(const WalkArgs& a, int nsm, Queue s, int shape)
{
    count_launch(1);
    if (a.kelbg ? walk_fp32c_few<true, true>(a, nsm, s)
                : a.phi ? walk_fp32c_few<false, true>(a, nsm, s)
                        : walk_fp32c_few<false, false>(a, nsm, s))
        return;
    if (shape < 0 || shape >= walk_shape_count()) shape = 0;
    const int per_sm = kShapes[shape][1];
    const int b = walk_blocks(a.nchunks, nsm, per_sm);
    // the potential is computed only when the caller reads it (the Kelbg form
    // always computes it)
    if (a.kelbg) walk_fp32c_shape<true, true>(a, per_sm, b, s);
    else if (a.phi) walk_fp32c_shape<false, true>(a, per_sm, b, s);
    else walk_fp32c_shape<false, false>(a, per_sm, b, s);
}

template <bool kTwo>
static void walk_fp32c_visits(const WalkArgs& a, int nsm, Queue s)
{
    const int b = walk_blocks(a.nchunks, nsm, visit_blocks(kTwo)), threads = kTwo ? 64 : 32;
    // (long leaves in parts: gradients of 30,000 and 131,072 particles in leaves of 300 11.2 and
    // 19.6 -> 7.9 and 16.0 ms; the form costs a gradient at 262,144 in leaves of 32 1.7 %)
    if (a.leaf_cap > 32) launch(k_walk_fp32c_visits<kTwo, true>, b, threads, s.whole(), a);
    else launch(k_walk_fp32c_visits<kTwo, false>, b, threads, s.whole(), a);
}

void launch_walk_fp32c_visits(const WalkArgs& a, int nsm, Queue s)
{
    count_launch(1);
    if (a.nchunks <= 4 * nsm) walk_fp32c_visits<true>(a, nsm, s);
    else walk_fp32c_visits<false>(a, nsm, s);
}

}  // namespace ucp
