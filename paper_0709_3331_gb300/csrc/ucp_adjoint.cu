// ucp_adjoint.cu -- reverse-mode derivative of the TREE force of Sec. 3
// (arXiv 0709.3331): mu = (da/dx)^T lambda for a = q E / m with the tree held
// fixed (the boxes every target opens or accepts do not move under an
// infinitesimal displacement).  FP64.
//
// The walk visits exactly the boxes of the forward walk (the same decisions).  Per
// target:
//   direct pair j:    mu_t += (q_t q_j / m_t) J(r) lambda_t,  J = g^3 I - 3 g^5 r r^T
//                     mu_j -= q_j J(r) w_t,  w_t = q_t lambda_t / m_t
//   accepted box n:   mu_t -= (q_t/m_t) (M d2g lambda - sum_bc lambda_b D_c d3g_abc
//                                        + 1/2 sum_bcd lambda_b Q_cd d4g_abcd)
//                     alpha_n += d2g w, Gamma_n += w_a d3g_a.., kappa_n += 1/2 d4g[w,.,Q]
// and afterwards every particle s of box n receives
//   q_s (alpha_n - Gamma_n (x_s - c_n)) + (|q_s| / S0_n) kappa_n
// (the source side through the dipole and second moment at fixed centre, and
// through the |q|-weighted centre the expansion is taken about).
// Source-side sums over targets are summed per group of targets and then by atomic
// adds, so their order (and last bits) may vary from run to run.
#include "ucp_lists.cuh"

#include <math.h>

#include <type_traits>

namespace ucp {

namespace {

__device__ __forceinline__ void qmul(const double* Q, const double* v, double* o)
{
    o[0] = Q[0] * v[0] + Q[1] * v[1] + Q[2] * v[2];
    o[1] = Q[1] * v[0] + Q[3] * v[1] + Q[4] * v[2];
    o[2] = Q[2] * v[0] + Q[4] * v[1] + Q[5] * v[2];
}

__device__ __forceinline__ double dot3(const double* a, const double* b)
{
    return a[0] * b[0] + a[1] * b[1] + a[2] * b[2];
}

// ---- FP64 form: one warp per target, the traversal of the FP32C walk with the FP64 walk's
// decisions.  The lanes are the sources, 32 accepted boxes or 32 particles of opened
// leaves.  A box's or source's own terms are added to memory as they come; the target's
// partial sums stay in the lanes' registers until the end.  All terms are linear in the
// target's weight w = (q/m) lambda.
//
// What bounds it: the FP64 pipe (about 120 operations per box, 16 cycles per warp
// instruction however many lanes are active) and the box terms' additions in memory.  One
// target per warp keeps every lane at work and fills the SMs from a few hundred targets
// on; eight targets per warp, with their sums in shared memory and a quarter of the
// additions, left 15 % of the lanes idle: a vector-Jacobian product 870 against 543 us at
// N = 4,096, 43.9 against 33.8 ms at 131,072.  Eight warps per SM are as fast as twelve and
// 2 % faster at the smallest sizes.
__global__ void __launch_bounds__(32, 8)
k_walk_adjoint(WalkArgs a, const double* __restrict__ lam, double* __restrict__ mu,
               double* __restrict__ adj)
{
    follow();
    __shared__ WalkWarp W;
    const int lane = threadIdx.x;
    const double q0 = a.qsp[0], q1 = a.qsp[1];
    const int gave_up = *a.err;

    while (true) {
        const unsigned int item = (unsigned int)next_chunk(a.work, lane);
        if (item / 32 >= (unsigned int)a.nchunks) break;
        const int4 ck = a.chunks[item / 32];
        if ((int)(item % 32) >= ck.y) continue;
        const int ti = ck.x + (int)(item % 32);
        const int t = a.targets ? a.targets[ti] : ti;
        const OneTarget tg(a, t, ck.z);
        const double X[3] = {a.x[t], a.y[t], a.z[t]};
        const double qm = a.msp[2 + a.sp[t]];
        const double w[3] = {qm * lam[3 * (size_t)t], qm * lam[3 * (size_t)t + 1],
                             qm * lam[3 * (size_t)t + 2]};
        double mt[3] = {0.0, 0.0, 0.0};

        // The same terms as the FP32 form below: the target takes -H, the box alpha,
        // Gamma and kappa.
        auto multipoles = [&](const int2* boxes, int cnt) {
            if (lane < cnt) {
                const int box = boxes[lane].x;
                const double* m = a.t.mom + (size_t)box * kMom;
                const double R[3] = {X[0] - m[MC], X[1] - m[MC + 1], X[2] - m[MC + 2]};
                const double M = m[MM], D[3] = {m[MD], m[MD + 1], m[MD + 2]};
                const double Q[6] = {m[MQ], m[MQ + 1], m[MQ + 2], m[MQ + 3], m[MQ + 4], m[MQ + 5]};
                const double T = m[MT];                       // -tr(Q)/2
                const double gi = rsqrt_fp64(dot3(R, R) + a.eps2);
                const double u = gi * gi, g3 = gi * u, g5 = g3 * u, g7 = g5 * u, g9 = g7 * u;
                const double rw = dot3(R, w), rd = dot3(R, D), wd = dot3(w, D);
                double q[3], qw[3];
                qmul(Q, R, q);
                qmul(Q, w, qw);
                const double rqr = dot3(R, q), wqr = dot3(w, q);
                const double p5 = 3.0 * (g5 * rw), p7 = 15.0 * (g7 * rw), g53 = 3.0 * g5;
                // k = 1/2 T4(w) = kr R - p7 q + kw w + 3 g^5 Q w
                const double kw = -(7.5 * (g7 * rqr) + g53 * T);
                const double kr = 52.5 * (g9 * rw) * rqr - 15.0 * (g7 * wqr) + p7 * T;
                const double aR = g53 * (M * rw - wd) + p7 * rd;
                const double aw = -(M * g3 + g53 * rd);
                const double h7 = 0.5 * p7;
                double* d = adj + (size_t)box * 12;
                double b[3];
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const double kk = kr * R[k] + (kw * w[k] + (g53 * qw[k] - p7 * q[k]));
                    atomicAdd(d + 9 + k, kk);
                    mt[k] -= aR * R[k] + (aw * w[k] + (kk - p5 * D[k]));
                    atomicAdd(d + k, p5 * R[k] - g3 * w[k]);
                    b[k] = g53 * w[k] - h7 * R[k];
                }
                atomicAdd(d + 3, 2.0 * (b[0] * R[0]) + p5);
                atomicAdd(d + 4, b[0] * R[1] + b[1] * R[0]);
                atomicAdd(d + 5, b[0] * R[2] + b[2] * R[0]);
                atomicAdd(d + 6, 2.0 * (b[1] * R[1]) + p5);
                atomicAdd(d + 7, b[1] * R[2] + b[2] * R[1]);
                atomicAdd(d + 8, 2.0 * (b[2] * R[2]) + p5);
            }
            __syncwarp();
        };

        auto direct_pairs = [&](const int2* leaves, int cnt) {
            const LeafRun run(a, leaves, cnt);
            for (int base = 0; base < run.total; base += 32) {
                int j, nd, first;
                unsigned int mask;
                run.at(base + lane, j, nd, first, mask);
                if (!mask || j == t) continue;
                const double R[3] = {X[0] - a.x[j], X[1] - a.y[j], X[2] - a.z[j]};
                const double qj = a.sp[j] ? q1 : q0;
                const double gi = rsqrt_fp64(dot3(R, R) + a.eps2);
                const double u = gi * gi, cw = qj * (gi * u);
                const double cr = -3.0 * (cw * u) * dot3(R, w);
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const double tv = cr * R[k] + cw * w[k];
                    mt[k] += tv;
                    atomicAdd(&mu[3 * (size_t)j + k], -tv);
                }
            }
            __syncwarp();
        };

        walk_lists(a, gave_up, W, 1u, ck.z,
                   [&](int box, unsigned int, const float4 h) {
                       return box >= 0 && tg.accepts(a, box, h) ? 1u : 0u;
                   },
                   multipoles, direct_pairs);

#pragma unroll
        for (int k = 0; k < 3; ++k) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) mt[k] += __shfl_xor_sync(0xffffffffu, mt[k], o);
            if (lane == k) atomicAdd(&mu[3 * (size_t)t + k], mt[k]);
        }
        __syncwarp();
    }
}

// ---- FP32 form (FP32C contexts): one warp per group of up to 16 targets, the
// traversal of the FP32C walk (the same decisions).  Both parts of the derivative
// run with the lanes over the sources: 32 accepted boxes, or 32 particles of opened
// leaves, one per lane, against the group's targets two at a time in packed FP32x2.
// A lane then holds its source's own sums (12 box terms, or 3 components) in
// registers and adds them to memory once per batch; the targets' sums are three
// values per target summed over the lanes by halving exchanges, four targets at a
// time.  All terms are linear in the target's weight w = (q/m) lambda.  A pair's
// separation is formed from the leaf's centroid and the particle's offset, as in the
// forward walks.
//
// Groups are taken longest chunk first, by the costs that the forward walks noted.
//
// What bounds it: the FP32 pipe (61 % busy), by the box part's 113 packed operations
// per box and pair of targets.  The form before took the lanes over targets and summed
// each box's 12 values over the warp (70 instructions beside 110 of arithmetic,
// unpacked) and each pair's three: 6.1 ms over every particle at N = 262,144 against
// 2.9, over the electrons 4.1 against 1.65 (whole chunks in list order: 3.1 and 1.95).

// Warp sums of 16 values by halving exchanges: at each xor step a lane keeps half of
// its values and adds the partner's copy of that half, so 16 values take 16
// exchanges instead of 80; lane L ends with value L / 2 (both lanes of a pair).
__device__ __forceinline__ float warp_sum16(float (&v)[16], int lane)
{
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const bool hi = (lane & 16) != 0;
        const float keep = hi ? v[i + 8] : v[i], send = hi ? v[i] : v[i + 8];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const bool hi = (lane & 8) != 0;
        const float keep = hi ? v[i + 4] : v[i], send = hi ? v[i] : v[i + 4];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const bool hi = (lane & 4) != 0;
        const float keep = hi ? v[i + 2] : v[i], send = hi ? v[i] : v[i + 2];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
    }
    {
        const bool hi = (lane & 2) != 0;
        const float keep = hi ? v[1] : v[0], send = hi ? v[0] : v[1];
        v[0] = keep + __shfl_xor_sync(0xffffffffu, send, 2);
    }
    return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 dot2(const float2* a, const float2* b)
{
    return fma2(a[0], b[0], fma2(a[1], b[1], mul2(a[2], b[2])));
}

// four floats added to 16-byte aligned memory
__device__ __forceinline__ void red_add4(float* p, float x, float y, float z, float w)
{
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};"
                 :: "l"(p), "f"(x), "f"(y), "f"(z), "f"(w) : "memory");
}

constexpr int kTargets = 16;

struct __align__(16) AdjWarp {
    WalkWarp walk;
    // two targets: relative to the chunk's centre and weights {x, y}, {z, wx}, {wy, wz};
    // relative to the cube's centre as float pairs {xh, yh}, {zh, xl}, {yl, zl}
    float4 tgt[kTargets / 2][6];
    float mt[kTargets / 4][32];         // four targets' sums: lane L holds value L / 2
    int slot[kTargets];      // the targets' slots
};

__global__ void __launch_bounds__(32, 16)
k_walk_adjoint_f32(WalkArgs a, int group, const double* __restrict__ lam,
                   double* __restrict__ mu, float* __restrict__ adj)
{
    follow();
    __shared__ AdjWarp shared;
    AdjWarp& W = shared;
    const int lane = threadIdx.x;
    const float4* __restrict__ S = a.src32;
    const float2 e2 = splat((float)a.eps2);

    const int per = 32 / group;
    const int gave_up = *a.err;
    while (true) {
        const unsigned int item = (unsigned int)next_chunk(a.work, lane);
        if (item >= (unsigned int)a.nchunks * per) break;
        int4 ck = a.chunks[a.ord.order[item / per]];
        ck.x += (int)(item % per) * group;
        ck.y = min(group, ck.y - (int)(item % per) * group);
        if (ck.y <= 0) continue;
        const int t = lane < ck.y ? (a.targets ? a.targets[ck.x + lane] : ck.x + lane) : -1;
        const ChunkTarget tg(a, t, ck.z);
        {
            float w[3] = {0.f, 0.f, 0.f};
            if (t >= 0) {
                const int s = a.sp[t];
                const double qm = a.msp[2 + s];
#pragma unroll
                for (int k = 0; k < 3; ++k) w[k] = (float)(qm * lam[3 * (size_t)t + k]);
            }
            if (lane < kTargets) {
                float* d = reinterpret_cast<float*>(W.tgt[lane >> 1]) + (lane & 1);
                d[0] = (tg.xh - tg.gx) + tg.xl;
                d[2] = (tg.yh - tg.gy) + tg.yl;
                d[4] = (tg.zh - tg.gz) + tg.zl;
                d[6] = w[0];
                d[8] = w[1];
                d[10] = w[2];
                d[12] = tg.xh;
                d[14] = tg.yh;
                d[16] = tg.zh;
                d[18] = tg.xl;
                d[20] = tg.yl;
                d[22] = tg.zl;
                W.slot[lane] = t >= 0 ? t : 0x7fffffff;
            }
#pragma unroll
            for (int g = 0; g < kTargets / 4; ++g) W.mt[g][lane] = 0.f;
            __syncwarp();
        }
        const int groups = (ck.y + 3) >> 2;
        // Targets relative to the middle of the group keep a box's distance to as many bits as
        // the group is larger than that distance.  Where most neighbours in the group lie
        // within an eighth of its extent (a group over the gap between two clusters), the boxes
        // near them are taken from float pairs, as the direct pairs are.
        bool wide;
        {
            const float ext = 2.f * fmaxf(tg.ex, fmaxf(tg.ey, tg.ez));
            const float gap = fmaxf(fabsf(__shfl_down_sync(0xffffffffu, tg.xh, 1) - tg.xh),
                                    fmaxf(fabsf(__shfl_down_sync(0xffffffffu, tg.yh, 1) - tg.yh),
                                          fabsf(__shfl_down_sync(0xffffffffu, tg.zh, 1) - tg.zh)));
            const bool near = lane + 1 < ck.y && gap < 0.125f * ext;
            wide = 2 * __popc(__ballot_sync(0xffffffffu, near)) > ck.y - 1;
        }

        // Accepted boxes, one per lane.  With g = (R.R + eps^2)^-1/2 and every l replaced
        // by w:  H = aR R + al w + aD D + k,  k = 1/2 T4(w),
        //   aR = 3 g^5 (M R.w - w.D) + 15 g^7 (R.w)(R.D),  al = -(M g^3 + 3 g^5 R.D),
        //   aD = -3 g^5 R.w;
        // the target takes -H; the box 3 g^5 (R.w) R - g^3 w (alpha), k (kappa) and
        // b R^T + R b^T + 3 g^5 (R.w) I, b = 3 g^5 w - (15/2) g^7 (R.w) R (Gamma).
        auto multipoles = [&](const int2* boxes, int cnt) {
            const int2 bm = lane < cnt ? boxes[lane] : make_int2(0, 0);
            const unsigned int mask = (unsigned int)bm.y;
            const float4* r = a.t.rec + (size_t)bm.x * kRec;
            const float4 r0 = __ldg(r), r1 = __ldg(r + 1), r2 = __ldg(r + 2), r3 = __ldg(r + 3),
                         lo = __ldg(a.t.lo + bm.x);
            const float2 cx = splat((r0.x + tg.gx) + lo.x), cy = splat((r0.y + tg.gy) + lo.y),
                         cz = splat((r0.z + tg.gz) + lo.z);
            const float2 M3 = splat(3.f * r0.w), nM = splat(-r0.w);
            const float2 nD[3] = {splat(-3.f * r1.x), splat(-3.f * r1.y), splat(-3.f * r1.z)};
            const float2 qxx = splat(r2.x), qxy = splat(r2.y), qxz = splat(r2.z), qyy = splat(r2.w),
                         qyz = splat(r3.x), qzz = splat(r3.y);                 // Q / 2
            const float2 t3 = splat(-3.f * r1.w), t15 = splat(15.f * r1.w);    // 3/2, -15/2 tr Q
            float2 al[3], ga[6], ka[3], tr;
#pragma unroll
            for (int k = 0; k < 3; ++k) al[k] = ka[k] = splat(0.f);
#pragma unroll
            for (int k = 0; k < 6; ++k) ga[k] = splat(0.f);
            tr = splat(0.f);
            auto targets = [&](auto from_pairs) {
#pragma unroll 1
                for (int g4 = 0; g4 < groups; ++g4) {
                    float v[16];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const float4* T = W.tgt[2 * g4 + h];
                        const float4 f0 = T[0], f1 = T[1], f2 = T[2];
                        float2 R[3];
                        if (decltype(from_pairs)::value) {
                            const float4 f3 = T[3], f4 = T[4], f5 = T[5];
                            R[0] = add2(add2(splat(r0.x), make_float2(f3.x, f3.y)),
                                        add2(splat(lo.x), make_float2(f4.z, f4.w)));
                            R[1] = add2(add2(splat(r0.y), make_float2(f3.z, f3.w)),
                                        add2(splat(lo.y), make_float2(f5.x, f5.y)));
                            R[2] = add2(add2(splat(r0.z), make_float2(f4.x, f4.y)),
                                        add2(splat(lo.z), make_float2(f5.z, f5.w)));
                        } else {
                            R[0] = add2(cx, make_float2(f0.x, f0.y));
                            R[1] = add2(cy, make_float2(f0.z, f0.w));
                            R[2] = add2(cz, make_float2(f1.x, f1.y));
                        }
                        const float2 w[3] = {make_float2(f1.z, f1.w), make_float2(f2.x, f2.y),
                                             make_float2(f2.z, f2.w)};
                        const float2 rr = fma2(R[0], R[0], fma2(R[1], R[1], fma2(R[2], R[2], e2)));
                        const unsigned int in = mask >> (4 * g4 + 2 * h);
                        const float2 g = make_float2((in & 1u) ? rsqrt_ftz(rr.x) : 0.f,
                                                     (in & 2u) ? rsqrt_ftz(rr.y) : 0.f);
                        const float2 u = mul2(g, g), g3 = mul2(g, u), g5 = mul2(g3, u),
                                     g7 = mul2(g5, u), g9 = mul2(g7, u);
                        const float2 rw = dot2(R, w), rd = dot2(R, nD), wd = dot2(w, nD);
                        const float2 q[3] = {
                            fma2(qxx, R[0], fma2(qxy, R[1], mul2(qxz, R[2]))),
                            fma2(qxy, R[0], fma2(qyy, R[1], mul2(qyz, R[2]))),
                            fma2(qxz, R[0], fma2(qyz, R[1], mul2(qzz, R[2])))};
                        const float2 qw[3] = {
                            fma2(qxx, w[0], fma2(qxy, w[1], mul2(qxz, w[2]))),
                            fma2(qxy, w[0], fma2(qyy, w[1], mul2(qyz, w[2]))),
                            fma2(qxz, w[0], fma2(qyz, w[1], mul2(qzz, w[2])))};
                        const float2 rqr = dot2(R, q), wqr = dot2(w, q);
                        const float2 p5 = mul2(g5, rw), p7 = mul2(g7, rw);
                        // k = kr R + kq q + kw w + 6 g^5 (Q/2) w
                        const float2 kw = fma2(g7, mul2(splat(-15.f), rqr), mul2(g5, t3));
                        const float2 kr = fma2(mul2(splat(105.f), rqr), mul2(g9, rw),
                                               fma2(g7, mul2(splat(-30.f), wqr), mul2(t15, p7)));
                        const float2 kq = mul2(splat(-30.f), p7), k6 = mul2(splat(6.f), g5);
                        const float2 aR = fma2(mul2(splat(-5.f), p7), rd, mul2(g5, fma2(M3, rw, wd)));
                        const float2 aw = fma2(g5, rd, mul2(nM, g3));
                        const float2 p53 = mul2(splat(3.f), p5), g53 = mul2(splat(3.f), g5),
                                     ng3 = mul2(splat(-1.f), g3), p75 = mul2(splat(-7.5f), p7);
                        float2 b[3];
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            const float2 kk = fma2(kr, R[k], fma2(kq, q[k], fma2(kw, w[k], mul2(k6, qw[k]))));
                            const float2 hh = fma2(aR, R[k], fma2(aw, w[k], fma2(p5, nD[k], kk)));
                            v[6 * h + k] = hh.x;
                            v[6 * h + 3 + k] = hh.y;
                            ka[k] = add2(ka[k], kk);
                            al[k] = fma2(p53, R[k], fma2(ng3, w[k], al[k]));
                            b[k] = fma2(g53, w[k], mul2(p75, R[k]));
                        }
                        tr = add2(tr, p53);
                        ga[0] = fma2(b[0], R[0], ga[0]);
                        ga[1] = fma2(b[0], R[1], fma2(b[1], R[0], ga[1]));
                        ga[2] = fma2(b[0], R[2], fma2(b[2], R[0], ga[2]));
                        ga[3] = fma2(b[1], R[1], ga[3]);
                        ga[4] = fma2(b[1], R[2], fma2(b[2], R[1], ga[4]));
                        ga[5] = fma2(b[2], R[2], ga[5]);
                    }
                    v[12] = v[13] = v[14] = v[15] = 0.f;
                    const float tot = warp_sum16(v, lane);
                    W.mt[g4][lane] -= tot;
                }
            };
            if (wide) targets(std::true_type{});
            else targets(std::false_type{});
            if (mask) {
                float* d = adj + (size_t)bm.x * 12;
                const float T = tr.x + tr.y;
                red_add4(d, al[0].x + al[0].y, al[1].x + al[1].y, al[2].x + al[2].y,
                         2.f * (ga[0].x + ga[0].y) + T);
                red_add4(d + 4, ga[1].x + ga[1].y, ga[2].x + ga[2].y,
                         2.f * (ga[3].x + ga[3].y) + T, ga[4].x + ga[4].y);
                red_add4(d + 8, 2.f * (ga[5].x + ga[5].y) + T, ka[0].x + ka[0].y,
                         ka[1].x + ka[1].y, ka[2].x + ka[2].y);
            }
            __syncwarp();
        };

        // Opened leaves: their particles in one run over the lanes.  A pair's term on
        // the target is q_j (g^3 w - 3 g^5 (r.w) r); the source takes its negative.
        auto direct_pairs = [&](const int2* leaves, int cnt) {
            const LeafRun run(a, leaves, cnt);
            for (int base = 0; base < run.total; base += 32) {
                int j, nd, first;
                unsigned int mask;
                run.at(base + lane, j, nd, first, mask);
                float4 A = make_float4(0.f, 0.f, 0.f, 0.f), B = A;
                float nx = 0.f, ny = 0.f, nz = 0.f, qj = 0.f;
                if (mask) {
                    // r = (x_t - c_leaf) + (c_leaf - x_j), the first from float pairs
                    A = __ldg(a.t.hdr + nd);
                    B = __ldg(a.t.lo + nd);
                    const int at = src_place(first, nd) + (j & ~1) - (first & ~1);
                    const float4 P = __ldg(S + at), Q = __ldg(S + at + 1);
                    const bool odd = j & 1;
                    nx = odd ? P.y : P.x;
                    ny = odd ? P.w : P.z;
                    nz = odd ? Q.y : Q.x;
                    qj = odd ? Q.w : Q.z;
                    // the particle's own place among the targets, if it has one
                    int pos = 0;
#pragma unroll
                    for (int o = kTargets / 2; o > 0; o >>= 1)
                        if (W.slot[pos + o - 1] < j) pos += o;
                    if (W.slot[pos] == j) mask &= ~(1u << pos);
                }
                const float2 cx = splat(A.x), cy = splat(A.y), cz = splat(A.z);
                const float2 lx = splat(B.x), ly = splat(B.y), lz = splat(B.z);
                const float2 px = splat(nx), py = splat(ny), pz = splat(nz);
                const float2 q2 = splat(qj), nq3 = splat(-3.f * qj);
                float2 s3[3] = {splat(0.f), splat(0.f), splat(0.f)};
#pragma unroll 1
                for (int g4 = 0; g4 < groups; ++g4) {
                    float v[16];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const float4* T = W.tgt[2 * g4 + h];
                        const float4 f1 = T[1], f2 = T[2], f3 = T[3], f4 = T[4], f5 = T[5];
                        const float2 R[3] = {
                            add2(add2(add2(cx, make_float2(f3.x, f3.y)),
                                      add2(lx, make_float2(f4.z, f4.w))), px),
                            add2(add2(add2(cy, make_float2(f3.z, f3.w)),
                                      add2(ly, make_float2(f5.x, f5.y))), py),
                            add2(add2(add2(cz, make_float2(f4.x, f4.y)),
                                      add2(lz, make_float2(f5.z, f5.w))), pz)};
                        const float2 w[3] = {make_float2(f1.z, f1.w), make_float2(f2.x, f2.y),
                                             make_float2(f2.z, f2.w)};
                        const float2 rr = fma2(R[0], R[0], fma2(R[1], R[1], fma2(R[2], R[2], e2)));
                        const unsigned int in = mask >> (4 * g4 + 2 * h);
                        const float2 g = make_float2((in & 1u) ? rsqrt_ftz(rr.x) : 0.f,
                                                     (in & 2u) ? rsqrt_ftz(rr.y) : 0.f);
                        const float2 u = mul2(g, g), g3 = mul2(g, u), g5 = mul2(g3, u);
                        const float2 cr = mul2(mul2(nq3, g5), dot2(R, w)), cw = mul2(q2, g3);
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            const float2 tv = fma2(cr, R[k], mul2(cw, w[k]));
                            v[6 * h + k] = tv.x;
                            v[6 * h + 3 + k] = tv.y;
                            s3[k] = add2(s3[k], tv);
                        }
                    }
                    v[12] = v[13] = v[14] = v[15] = 0.f;
                    const float tot = warp_sum16(v, lane);
                    W.mt[g4][lane] += tot;
                }
                if (mask)
#pragma unroll
                    for (int k = 0; k < 3; ++k)
                        atomicAdd(&mu[3 * (size_t)j + k], -(double)(s3[k].x + s3[k].y));
            }
            __syncwarp();
        };

        walk_lists(a, gave_up, W.walk, tg, ck.z, multipoles, direct_pairs);

        // value L / 2 of a group: components of target (L / 2) / 3 of its four
        const int term = lane >> 1;
        if ((lane & 1) == 0 && term < 12)
            for (int g4 = 0; g4 < groups; ++g4) {
                const int k = 4 * g4 + term / 3;
                if (k < ck.y)
                    atomicAdd(&mu[3 * (size_t)W.slot[k] + term % 3], (double)W.mt[g4][lane]);
            }
        __syncwarp();
    }
}

// Every particle of a leaf receives the source-side terms of the leaf and of
// all its ancestors: q_s (sum alpha - sum Gamma (x_s - c)) + |q_s| sum kappa / S0.
// One thread per leaf, in blocks of one warp: the FP64 pipe bounds it (55 operations per
// leaf and ancestor, 25 per particle), and so its few warps spread evenly over the SMs (a
// gradient of 20 steps at 20,000 particles 22.7 -> 22.0 ms against blocks of eight warps).
template <class TA>
__global__ void k_adjoint_push(const double* __restrict__ x, const double* __restrict__ y,
                               const double* __restrict__ z, const int8_t* __restrict__ sp,
                               const double* __restrict__ qsp, Tree t,
                               const TA* __restrict__ adj, double* __restrict__ mu)
{
    follow();
    constexpr bool kFp32 = sizeof(TA) == sizeof(float);     // FP32C contexts
    const int nn = *t.nnodes;
    for (int leaf = blockIdx.x * blockDim.x + threadIdx.x; leaf < nn;
         leaf += gridDim.x * blockDim.x) {
        if (!(t.depth_leaf[leaf] & 256)) continue;
        double A[3] = {0, 0, 0}, G[6] = {0, 0, 0, 0, 0, 0}, Cc[3] = {0, 0, 0}, K[3] = {0, 0, 0};
        for (int nd = leaf, up; nd >= 0; nd = up) {
            up = t.info[nd].w;
            if (up >= nd) up = -1;      // a parent comes before its child: the loop ends
            double r[12];
            for (int k = 0; k < 12; ++k) r[k] = (double)adj[(size_t)nd * 12 + k];
            const double* m = t.mom + (size_t)nd * (kFp32 ? kCentre : kMom);
            double c[3] = {m[MC], m[MC + 1], m[MC + 2]};
            double Gc[3];
            qmul(r + 3, c, Gc);
            const double S0 = kFp32 ? (double)t.mom32[(size_t)nd * 16 + 3] : m[MS0];
            const double inv = S0 > 0.0 ? 1.0 / S0 : 0.0;
            for (int k = 0; k < 3; ++k) {
                A[k] += r[k];
                Cc[k] += Gc[k];
                K[k] += r[9 + k] * inv;
            }
            for (int k = 0; k < 6; ++k) G[k] += r[3 + k];
        }
        const int4 inf = t.info[leaf];
        for (int s = inf.x; s < inf.y; ++s) {
            const double qs = sp[s] ? qsp[1] : qsp[0];
            const double xs[3] = {x[s], y[s], z[s]};
            double Gx[3];
            qmul(G, xs, Gx);
            for (int k = 0; k < 3; ++k)
                mu[3 * (size_t)s + k] += qs * (A[k] - Gx[k] + Cc[k]) + fabs(qs) * K[k];
        }
    }
}

template <class TA>
__global__ void k_zero_adj(const int* __restrict__ nnodes, TA* __restrict__ adj)
{
    follow();
    const size_t total = (size_t)*nnodes * 12;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total;
         i += (size_t)gridDim.x * blockDim.x)
        adj[i] = (TA)0;
}

// dst[t] = src[id[t]] for N x 3 arrays (caller order -> key order)
__global__ void k_gather3(const double* __restrict__ src, const unsigned int* __restrict__ id, int n,
                          double* __restrict__ dst)
{
    follow();
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    size_t j = id[t];
    dst[3 * (size_t)t] = src[3 * j];
    dst[3 * (size_t)t + 1] = src[3 * j + 1];
    dst[3 * (size_t)t + 2] = src[3 * j + 2];
}

// dst[id[t]] += src[t] for N x 3 arrays (key order -> caller order)
__global__ void k_scatter_add3(const double* __restrict__ src, const unsigned int* __restrict__ id,
                               int n, double* __restrict__ dst)
{
    follow();
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    size_t j = id[t];
    dst[3 * j] += src[3 * (size_t)t];
    dst[3 * j + 1] += src[3 * (size_t)t + 1];
    dst[3 * j + 2] += src[3 * (size_t)t + 2];
}

// out = coefficient(species) * lam_v: electrons ce, ions ci
__global__ void k_kick_lambda(const double* __restrict__ lam_v, const int8_t* __restrict__ sp, int n,
                              double ce, double ci, double* __restrict__ out)
{
    follow();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double f = sp[i] ? ce : ci;
    for (int k = 0; k < 3; ++k) out[3 * (size_t)i + k] = f * lam_v[3 * (size_t)i + k];
}

// y += a x over n x 3
__global__ void k_axpy3(double* __restrict__ y, const double* __restrict__ x, double a, int n)
{
    follow();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 3 * n) return;
    y[i] += a * x[i];
}

// lam_v = m_e v on electrons, 0 on ions; part = the blocks' sums of 1/2 m_e v^2, added
// in block order by the second kernel (deterministic)
constexpr int kSeedBlocks = 304;

__global__ void __launch_bounds__(256)
k_ke_seed(const double* __restrict__ v, const int8_t* __restrict__ sp, int n, double me,
          double* __restrict__ lam_v, double* __restrict__ part)
{
    follow();
    double acc = 0.0;
    for (int i = blockIdx.x * 256 + threadIdx.x; i < n; i += gridDim.x * 256) {
        const bool e = sp[i] != 0;
        for (int k = 0; k < 3; ++k) {
            const double vv = v[3 * (size_t)i + k];
            lam_v[3 * (size_t)i + k] = e ? me * vv : 0.0;
            if (e) acc += 0.5 * me * vv * vv;
        }
    }
    __shared__ double sh[256];
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int st = 128; st > 0; st >>= 1) {
        if ((int)threadIdx.x < st) sh[threadIdx.x] += sh[threadIdx.x + st];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

__global__ void k_ke_sum(const double* __restrict__ part, int nblk, double* __restrict__ loss)
{
    follow();
    const int lane = threadIdx.x;
    double acc = 0.0;
    for (int b = lane; b < nblk; b += 32) acc += part[b];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) *loss = acc;
}

// dst[id[t]] = src[t] for N x 3 arrays (key order -> caller order)
__global__ void k_scatter_rows3(const double* __restrict__ src, const unsigned int* __restrict__ id,
                                int n, double* __restrict__ dst)
{
    follow();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const size_t j = id[t];
    dst[3 * j] = src[3 * (size_t)t];
    dst[3 * j + 1] = src[3 * (size_t)t + 1];
    dst[3 * j + 2] = src[3 * (size_t)t + 2];
}

}  // namespace

void launch_gather3(const double* src, const unsigned int* id, int n, double* dst, Queue s)
{
    count_launch(1);
    launch(k_gather3, (n + 255) / 256, 256, s, src, id, n, dst);
}

void launch_scatter_add3(const double* src, const unsigned int* id, int n, double* dst,
                         Queue s)
{
    count_launch(1);
    launch(k_scatter_add3, (n + 255) / 256, 256, s, src, id, n, dst);
}

void launch_kick_lambda(const double* lam_v, const int8_t* sp, int n, double ce, double ci,
                        double* out, Queue s)
{
    count_launch(1);
    launch(k_kick_lambda, (n + 255) / 256, 256, s, lam_v, sp, n, ce, ci, out);
}

void launch_axpy3(double* y, const double* x, double a, int n, Queue s)
{
    count_launch(1);
    launch(k_axpy3, (3 * n + 255) / 256, 256, s, y, x, a, n);
}

size_t ke_seed_words() { return 1 + kSeedBlocks; }

void launch_ke_seed(const double* v, const int8_t* sp, int n, double me, double* lam_v,
                    double* loss, Queue s)
{
    count_launch(2);
    const int b = n < 256 * kSeedBlocks ? (n + 255) / 256 : kSeedBlocks;
    launch(k_ke_seed, b, 256, s, v, sp, n, me, lam_v, loss + 1);
    launch(k_ke_sum, 1, 32, s, loss + 1, b, loss);
}

void launch_scatter_rows3(const double* src, const unsigned int* id, int n, double* dst,
                          Queue s)
{
    count_launch(1);
    launch(k_scatter_rows3, (n + 255) / 256, 256, s, src, id, n, dst);
}

void launch_walk_adjoint(const WalkArgs& a, const double* lam, double* mu, double* adj, int n,
                         int nsm, Queue s)
{
    count_launch(3);
    cudaMemsetAsync(mu, 0, sizeof(double) * 3 * (size_t)n, s);
    if (a.src32) {
        // 16 targets to a warp, fewer where chunks are few.  A gradient of 20 steps with 4,
        // 8 and 16: 13.4 14.0 15.2 ms at 4000 particles (63 and 125 chunks), 33.4 (8) 34.5
        // at 40,000, 52.5 51.8 at 120,000 (1875 and 3750)
        const int group = a.nchunks < nsm ? 4 : a.nchunks < 10 * nsm ? 8 : kTargets;
        const int64_t items = (int64_t)a.nchunks * (32 / group);
        const int blocks = items < 1 ? 1 : items < 16 * nsm ? (int)items : 16 * nsm;
        // FP32C context: FP32 walk, FP32 box accumulators (in the same buffer)
        float* adjf = reinterpret_cast<float*>(adj);
        launch(k_zero_adj<float>, 2 * 152, 256, s, a.t.nnodes, adjf);
        launch(k_walk_adjoint_f32, blocks, 32, s.whole(), a, group, lam, mu, adjf);
        launch(k_adjoint_push<float>, 32 * 152, 32, s, a.x, a.y, a.z, a.sp, a.qsp, a.t, adjf, mu);
    } else {
        launch(k_zero_adj<double>, 2 * 152, 256, s, a.t.nnodes, adj);
        const int64_t items = (int64_t)a.nchunks * 32;
        const int blocks = items < 1 ? 1 : items < 8 * nsm ? (int)items : 8 * nsm;
        launch(k_walk_adjoint, blocks, 32, s.whole(), a, lam, mu, adj);
        launch(k_adjoint_push<double>, 32 * 152, 32, s, a.x, a.y, a.z, a.sp, a.qsp, a.t, adj, mu);
    }
}

}  // namespace ucp
