// ucp_push.cu -- velocity Verlet kicks and drifts (Sec. 2 of arXiv 0709.3331),
// energy and momentum reductions (Sec. 5), and layout conversions at the boundary.
#include "ucp_internal.cuh"

#include <math.h>

namespace ucp {

namespace {

constexpr int kT = 256;

__global__ void k_kick(double* __restrict__ vx, double* __restrict__ vy, double* __restrict__ vz,
                       const double* __restrict__ ax, const double* __restrict__ ay,
                       const double* __restrict__ az, const int8_t* __restrict__ sp, int species,
                       double h, int n, int times)
{
    follow();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n || sp[i] != species) return;
    double ux = vx[i], uy = vy[i], uz = vz[i];
    double gx = ax[i], gy = ay[i], gz = az[i];
    // consecutive half kicks, each rounded on its own, each one fused
    // multiply-add (one FP64 operation per component: GB300's FP64 rate is 1/64
    // of FP32); written out so that every kernel that kicks gives the same bits
    for (int k = 0; k < times; ++k) {
        ux = __fma_rn(h, gx, ux);
        uy = __fma_rn(h, gy, uy);
        uz = __fma_rn(h, gz, uz);
    }
    vx[i] = ux;
    vy[i] = uy;
    vz[i] = uz;
}

__global__ void k_drift(double* __restrict__ x, double* __restrict__ y, double* __restrict__ z,
                        const double* __restrict__ vx, const double* __restrict__ vy,
                        const double* __restrict__ vz, double dt, int n)
{
    follow();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    x[i] = __fma_rn(dt, vx[i], x[i]);  // one rounding, as the kicks
    y[i] = __fma_rn(dt, vy[i], y[i]);
    z[i] = __fma_rn(dt, vz[i], z[i]);
}

// Deterministic two-level reduction: fixed per-thread strides, fixed tree in
// the block, partials summed in block order by one thread.
// out[6 c ..] = {KE_ion, KE_electron, PE, px, py, pz} of cloud c = blockIdx.y (cloud_start
// NULL: of everything).
__global__ void k_energy_partial(const double* __restrict__ vx, const double* __restrict__ vy,
                                 const double* __restrict__ vz, const double* __restrict__ phi,
                                 const int8_t* __restrict__ sp, const double* __restrict__ qsp,
                                 const double* __restrict__ msp, int n,
                                 const int* __restrict__ cloud_start, double* __restrict__ part)
{
    follow();
    const int c = blockIdx.y, end = cloud_start ? cloud_start[c + 1] : n;
    part += (size_t)c * gridDim.x * 6;
    double acc[6] = {0, 0, 0, 0, 0, 0};
    for (int i = (cloud_start ? cloud_start[c] : 0) + blockIdx.x * blockDim.x + threadIdx.x; i < end;
         i += gridDim.x * blockDim.x) {
        int s = sp[i];
        double m = msp[s];
        double ux = vx[i], uy = vy[i], uz = vz[i];
        double ke = 0.5 * m * (ux * ux + uy * uy + uz * uz);
        acc[s] += ke;
        acc[2] += 0.5 * qsp[s] * phi[i];
        acc[3] += m * ux;
        acc[4] += m * uy;
        acc[5] += m * uz;
    }
    __shared__ double sh[kT][6];
    for (int k = 0; k < 6; ++k) sh[threadIdx.x][k] = acc[k];
    __syncthreads();
    for (int st = kT / 2; st > 0; st >>= 1) {
        if ((int)threadIdx.x < st)
            for (int k = 0; k < 6; ++k) sh[threadIdx.x][k] += sh[threadIdx.x + st][k];
        __syncthreads();
    }
    if (threadIdx.x == 0)
        for (int k = 0; k < 6; ++k) part[blockIdx.x * 6 + k] = sh[0][k];
}

// Six warps, one per observable: lane l adds partials l, l + 32, ..., then the
// lanes are added by a fixed butterfly (a deterministic order).
__global__ void __launch_bounds__(192)
k_energy_final(const double* __restrict__ part, int nblk, double* __restrict__ out)
{
    follow();
    const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
    part += (size_t)blockIdx.x * nblk * 6;
    double acc = 0.0;
    for (int b = lane; b < nblk; b += 32) acc += part[6 * b + k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) out[6 * blockIdx.x + k] = acc;
}

__global__ void k_scatter3(const double* __restrict__ ax, const double* __restrict__ ay,
                           const double* __restrict__ az, const unsigned int* __restrict__ id,
                           int n, double* __restrict__ out)
{
    follow();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    unsigned int j = id[i];
    out[3 * (size_t)j] = ax[i];
    out[3 * (size_t)j + 1] = ay[i];
    out[3 * (size_t)j + 2] = az[i];
}

__global__ void k_scatter1(const double* __restrict__ a, const unsigned int* __restrict__ id, int n,
                           double* __restrict__ out)
{
    follow();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[id[i]] = a[i];
}

__global__ void k_scatter_int(const int* __restrict__ a, const unsigned int* __restrict__ id, int n,
                              int* __restrict__ out)
{
    follow();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[id[i]] = a[i];
}

// Caller-order state (N x 3 arrays, vel may be NULL: zeros) into the context's
// arrays: six streams, species (twice: in the slots' order and in the caller's) and
// the identity as caller indices.
__global__ void k_load_state(const double* __restrict__ pos, const double* __restrict__ vel,
                             const int8_t* __restrict__ sp, int n, double* __restrict__ x,
                             double* __restrict__ y, double* __restrict__ z,
                             double* __restrict__ vx, double* __restrict__ vy,
                             double* __restrict__ vz, int8_t* __restrict__ sp_slot,
                             int8_t* __restrict__ sp_caller, unsigned int* __restrict__ id)
{
    follow();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const size_t b = 3 * (size_t)i;
    x[i] = pos[b];
    y[i] = pos[b + 1];
    z[i] = pos[b + 2];
    vx[i] = vel ? vel[b] : 0.0;
    vy[i] = vel ? vel[b + 1] : 0.0;
    vz[i] = vel ? vel[b + 2] : 0.0;
    const int8_t s = sp[i];
    sp_slot[i] = s;
    if (sp_caller) sp_caller[i] = s;
    id[i] = (unsigned int)i;
}

// flags[0] |= 1 on a non-finite position or velocity, flags[1] |= 1 on a
// species code other than 0 or 1, flags[2 + c] += electrons of cloud c.
__global__ void k_check_state(const double* __restrict__ pos, const double* __restrict__ vel,
                              const int8_t* __restrict__ sp, int n,
                              const unsigned char* __restrict__ cloud, int* __restrict__ flags)
{
    follow();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31;
    bool bad = false, wrong = false, electron = false;
    int c = 0;
    if (i < n) {
        for (int a = 0; a < 3; ++a)
            bad |= !isfinite(pos[3 * (size_t)i + a]) || !isfinite(vel[3 * (size_t)i + a]);
        wrong = sp[i] != 0 && sp[i] != 1;
        electron = sp[i] == 1;
        if (cloud) c = cloud[i];
    }
    if (bad) atomicOr(&flags[0], 1);
    if (wrong) atomicOr(&flags[1], 1);
    // electrons: one count per warp and cloud
    const unsigned int e = __ballot_sync(0xffffffffu, electron);
    const unsigned int peers = __match_any_sync(0xffffffffu, c) & e;
    if (electron && lane == __ffs(peers) - 1) atomicAdd(&flags[2 + c], __popc(peers));
}

// Walk chunks of up to `width` consecutive targets, cloud by cloud: cloud c's run of
// targets is [first[c], first[c + 1]), its chunks start at place[c]; taken in list order, as
// are the first n_other of another list (whose chunks stay).
__global__ void k_chunks(const int* __restrict__ first, const int* __restrict__ place, int n_clouds,
                         int width, int nchunks, int4* __restrict__ chunks,
                         int* __restrict__ order, int n_other, int* __restrict__ other)
{
    follow();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n_other) other[i] = i;
    if (i >= nchunks) return;
    int lo = 0, hi = n_clouds;          // the cloud whose chunks hold i
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (place[mid] <= i) lo = mid;
        else hi = mid;
    }
    const int b = first[lo] + (i - place[lo]) * width;
    chunks[i] = make_int4(b, min(width, first[lo + 1] - b), lo, 0);
    order[i] = i;
}

inline int nb(int n) { return (n + kT - 1) / kT > 0 ? (n + kT - 1) / kT : 1; }

}  // namespace

void launch_kick(double* vx, double* vy, double* vz, const double* ax, const double* ay,
                 const double* az, const int8_t* sp, int species, double h, int n, int times,
                 Queue s)
{
    count_launch(1);
    launch(k_kick, nb(n), kT, s, vx, vy, vz, ax, ay, az, sp, species, h, n, times);
}

void launch_drift(double* x, double* y, double* z, const double* vx, const double* vy,
                  const double* vz, double dt, int n, Queue s)
{
    count_launch(1);
    launch(k_drift, nb(n), kT, s, x, y, z, vx, vy, vz, dt, n);
}

void launch_energy(const double* vx, const double* vy, const double* vz, const double* phi,
                   const int8_t* sp, const double* qsp, const double* msp, int n,
                   const int* cloud_start, int n_clouds, double* partials, int nblk, double* out,
                   Queue s)
{
    count_launch(2);
    launch(k_energy_partial, dim3(nblk, n_clouds), kT, s, vx, vy, vz, phi, sp, qsp, msp, n,
           cloud_start, partials);
    launch(k_energy_final, n_clouds, 192, s, partials, nblk, out);
}

void launch_scatter3(const double* ax, const double* ay, const double* az, const unsigned int* id,
                     int n, double* out, Queue s)
{
    count_launch(1);
    launch(k_scatter3, nb(n), kT, s, ax, ay, az, id, n, out);
}

void launch_scatter1(const double* a, const unsigned int* id, int n, double* out, Queue s)
{
    count_launch(1);
    launch(k_scatter1, nb(n), kT, s, a, id, n, out);
}

void launch_scatter_int(const int* a, const unsigned int* id, int n, int* out, Queue s)
{
    count_launch(1);
    launch(k_scatter_int, nb(n), kT, s, a, id, n, out);
}

void launch_load_state(const double* pos, const double* vel, const int8_t* sp, int n,
                       double* const* st6, int8_t* sp_slot, int8_t* sp_caller, unsigned int* id,
                       Queue s)
{
    count_launch(1);
    launch(k_load_state, nb(n), kT, s, pos, vel, sp, n, st6[0], st6[1], st6[2], st6[3], st6[4],
                                      st6[5], sp_slot, sp_caller, id);
}

void launch_check_state(const double* pos, const double* vel, const int8_t* sp, int n,
                        const unsigned char* cloud, int* flags, Queue s)
{
    count_launch(1);
    launch(k_check_state, nb(n), kT, s, pos, vel, sp, n, cloud, flags);
}

void launch_chunks(const int* first, const int* place, int n_clouds, int width, int nchunks,
                   int4* chunks, int* order, int n_other, int* other, Queue s)
{
    const int most = nchunks > n_other ? nchunks : n_other;
    if (most < 1) return;
    count_launch(1);
    launch(k_chunks, nb(most), kT, s, first, place, n_clouds, width, nchunks, chunks, order, n_other,
           other);
}

}  // namespace ucp
