// ucp_internal.cuh -- device data layout and kernel entry points shared by the
// translation units of libucp (TREE method of arXiv 0709.3331, Sec. 3).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

namespace ucp {

constexpr int kMaxDepth = 21;        // 21 bits per axis, 63-bit keys
constexpr int kWarp = 32;

// Order-preserving integer image of a double (larger double, larger image; -0 below
// +0; a NaN with the sign bit clear above every number, with it set below), so
// min/max reductions are exact, order-independent integer operations.
__device__ __forceinline__ unsigned long long ord64(double v)
{
    unsigned long long b = (unsigned long long)__double_as_longlong(v);
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__device__ __forceinline__ double unord64(unsigned long long u)
{
    return __longlong_as_double((long long)((u >> 63) ? (u & 0x7fffffffffffffffull) : ~u));
}

// Approximate reciprocal square root of the special-function unit (the
// approximation rsqrtf uses) with subnormal inputs and outputs flushed to zero,
// which spares the subnormal handling around it.  The walks call it on r^2 + eps^2
// or on |x_t - c|^2 + eps^2: below 2^-126 only for particles closer than 1e-19, whose
// FP32 field overflows in any case; for every normal input the result is rsqrtf's.
__device__ __forceinline__ float rsqrt_ftz(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Kernels launched by this process (read by ucp_stats).
extern std::atomic<unsigned long long> g_launches;
inline void count_launch(int k) { g_launches.fetch_add((unsigned long long)k, std::memory_order_relaxed); }

// The stream of a context's launches.  chained: a kernel is launched as a programmatic
// dependent of the one before it, so that its blocks are placed while that one drains
// (they wait in follow() until it has finished): 1-2 us off each of the ~25 kernels of a
// substep.  Force call at 8192 particles, FP32C, 244 -> 227 us; 11 substeps at N = 2048,
// FP64, 2.28 -> 2.04 ms.
struct Queue {
    cudaStream_t s = nullptr;
    bool chained = true;
    operator cudaStream_t() const { return s; }
    // for the walks: their blocks, a few to every SM, would be dealt out unevenly around
    // those of the kernel ahead (FP64 walk at N = 131,072: 7.2 -> 8.3 ms; force call at
    // 4099 particles, FP32C: 0.35 -> 0.41 ms)
    Queue whole() const { return {s, false}; }
};

template <class... P, class... A>
inline void launch_shared(void (*kernel)(P...), dim3 grid, dim3 block, int dynamic_bytes,
                          const Queue& q, A... args)
{
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = dynamic_bytes;
    cfg.stream = q.s;
    cfg.attrs = &attr;
    cfg.numAttrs = q.chained ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

template <class... P, class... A>
inline void launch(void (*kernel)(P...), dim3 grid, dim3 block, const Queue& q, A... args)
{
    launch_shared(kernel, grid, block, 0, q, args...);
}

// First statement of every kernel that launch() starts, by every thread: the next
// kernel of the stream may be placed as soon as every block of this one is (it waits
// here in its turn), and nothing of global memory is read or written before the
// kernel ahead has finished and its writes are visible.
__device__ __forceinline__ void follow()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// One FP64 box record, 16 doubles (128 B), read by the FP64 walk.
// {c.x, c.y, c.z, rcrit2, M, D.x, D.y, D.z, Qxx, Qxy, Qxz, Qyy, Qyz, Qzz, S0, -tr(Q)/2}
// FP32C contexts: the first kCentre of them, c and rcrit2 (the rest is in mom32).
// rcrit2 = (s/theta + delta)^2 is filled per walk (it depends on theta).  Until its first
// walk an FP64 tree holds in the same place each box's sums about its geometric centre,
// {S0, M, sum|q|y (3), sum q y (3), sum q y y^T (6)}, and kSumsDelta as the box's delta.
// The mark is the record's own, on the device, so that a captured sequence of launches
// finds the records as they are whenever it is replayed.
constexpr int kMom = 16, kCentre = 4;
constexpr double kSumsDelta = -1.0;
enum MomIdx { MC = 0, MR2 = 3, MM = 4, MD = 5, MQ = 8, MS0 = 14, MT = 15 };

// FP32 box records, written per walk (they hold rcrit2, which depends on theta):
//   hdr = {-ch.x, -ch.y, -ch.z, +-rcrit2}   ch = fp32(c) relative to the cube's centre;
//                                           the sign bit of rcrit2 marks a leaf
// and, in FP32C contexts, read only for boxes that act or are opened,
//   lo  = {-cl.x, -cl.y, -cl.z, 0}          cl = fp32(c - ch)
//   rec = {-ch.x, -ch.y, -ch.z, M}, {D.x, D.y, D.z, -tr(Q)/2}, {Qxx, Qxy, Qxz, Qyy} / 2,
//         {Qyz / 2, Qzz / 2, -M, 0}         64 B: four lanes load one box
constexpr int kRec = 4;

// FP32C sources: offsets n = c_leaf - x and charges in pairs of particles, two float4
// per pair {nx0, nx1, ny0, ny1}, {nz0, nz1, q0, q1}, particle j in the half j & 1.
// Every leaf starts at a place of its own, so that its pairs hold no other leaf's
// particles: an empty half (before an odd first particle, after an odd last one) is far
// away and has no charge.  src_place: float4 index of the first pair of the leaf `box`
// whose first particle is `begin` (two leaves never overlap: a later one has a later
// box, which moves it two places on).
__host__ __device__ __forceinline__ int src_place(int begin, int box)
{
    return (begin & ~1) + 2 * box;
}
constexpr int kSrcSlack = 64;        // float4 read (not used) past the last leaf
constexpr float kFarAway = 1e18f;

// Box topology {begin, end, next, parent}; depth and leaf flag separately.
struct Tree {
    int cap;                 // box capacity
    int* nnodes;             // device scalar
    int* maxdepth;           // device scalar
    int4* info;              // {begin, end, next, parent}
    int* depth_leaf;         // depth | leaf << 8
    unsigned long long* cell;// key prefix of the box at its depth
    double* mom;             // kMom doubles per box (FP32C contexts: kCentre)
    double* delta;           // |centroid - geometric centre| per box
    float4* hdr;             // traversal record per box
    float4* lo;              // FP32C contexts: low part of the centroid
    float4* rec;             // FP32C contexts: kRec float4 per box
    float* mom32;            // FP32C contexts: 16 floats per box {e xyz, S0, M, D, Q, 0, 0}
    int* child8;             // 8 child slots per box (octant order), -1 = empty
    int* arrive;             // finished children per box (moments' bottom-up sweep)
    // clouds: cloud[i] = cloud of key-sorted position i, whose segment is
    // [cloud_start[c], cloud_start[c + 1]); NULL cloud = one cloud over [0, n)
    const unsigned char* cloud;
    const int* cloud_start;
};

struct Cube {                // enclosing cube: centre, side, lower corner, 2^21 / side
    double c[3];
    double L;
    double lo[3];
    double kscale;
};

// ---- build (ucp_build.cu, ucp_sort.cu) ----
constexpr int kKeyBits = 63;
constexpr int kRadix = 256;
constexpr int kSortPassesMax = 4;        // passes over the key's top digits (sort_passes)
// Counters of one build, cleared together at its start.
enum CtlIdx {
    kCtlHist = 0,                                  // digit counts of every pass
    kCtlTile = kCtlHist + kSortPassesMax * kRadix, // tile counters: passes, then the clouds' pass
    kCtlLong = kCtlTile + kSortPassesMax + 1,      // raised: a run too long for the run sort
    kCtlBarrier,                                   // arrivals at the full sort's barrier
    kCtlTopoTile,                                  // tiles of the topology's scan
    kCtlMaxDepth,
    kCtlWords
};
struct BuildCtl {
    int* words;              // kCtlWords
    unsigned int* epoch;     // tag of the published words, advanced every build
};
// One cloud of up to this many particles is sorted by one block (ucp_sort.cu).
constexpr int kBlockSort = 6144, kBlockThreads = 1024;
inline bool block_sorted(int n, int n_clouds) { return n_clouds == 1 && n <= kBlockSort; }

void launch_bbox(const double* x, const double* y, const double* z, int n, double* partials,
                 int nblk, Cube* cubes, const int* cloud_start, int n_clouds, BuildCtl ctl,
                 Queue s);
void launch_keys(const double* x, const double* y, const double* z, int n, const Cube* cubes,
                 const unsigned char* cloud, unsigned long long* key, int passes, BuildCtl ctl,
                 Queue s);
struct SortScratch {
    unsigned long long* status;    // passes x tiles x 256 published words
    int* err;                      // raised by a wait that gave up
    int* full_counts;              // full sort: digit counts of its eight passes
    unsigned int* test_epoch;      // tag used by the bounded-wait self-test (1)
    int* test_ctl;                 // its tile counter and 256 zero offsets
    unsigned long long* test_keys; // 4 tiles, for the bounded-wait self-test
    unsigned int* test_vals;
};
int sort_passes(int64_t largest_cloud);
size_t sort_status_words(int n);
size_t sort_test_words();
size_t sort_full_words();
// Particle state of one order: six streams, species, caller index.
struct StateRef {
    double* f[6];
    int8_t* sp;
    unsigned int* id;
};
// Particle at sorted place i: its state, species and caller index from slot p.
__device__ __forceinline__ void move_state(const StateRef& in, const StateRef& out, int i,
                                           unsigned int p)
{
#pragma unroll
    for (int a = 0; a < 6; ++a) out.f[a][i] = in.f[a][p];
    out.sp[i] = in.sp[p];
    out.id[i] = in.id[p];
}

// Sorts key[0] (unsorted keys of the slots of `in`) and moves the state into key order
// (`out`), or leaves that to launch_topology (block_sorted), with the slots in order in
// val[1]; returns the buffer (0 or 1) that holds the sorted keys.
int launch_sort(unsigned long long* key[2], unsigned int* val[2], int n, int passes,
                const SortScratch& sc, BuildCtl ctl, const StateRef& in, const StateRef& out,
                const unsigned char* cloud, const int* cloud_start, int n_clouds, int nsm,
                Queue s);
int sort_selftest_timeout(const SortScratch& sc, Queue s);
void launch_topology(const unsigned long long* key, int n, int leaf_cap, int* pos_cnt,
                     int* pos_off, Tree t, BuildCtl ctl, unsigned long long* status, int* err,
                     const StateRef& in,
                     const StateRef& out, const unsigned int* from, Queue s);
size_t topo_status_words(int n);
void launch_moments(const double* x, const double* y, const double* z, const int8_t* sp,
                    const double* qsp, int n, int leaf_cap, const int* pos_cnt,
                    const int* pos_off, const Cube* cube, Tree t, float4* src32, int want_f32,
                    Queue s);

// ---- walk (ucp_walk.cu, ucp_schedule.cu) ----
// Order in which a walk takes its chunks, and the costs it notes for the next order (of the
// same state's next substep or walk: a new state starts from list order).
constexpr int kCostBins = 256;
struct WalkOrder {
    int* order;             // chunk of every work item
    float* cost;            // cycles per chunk of the last walk
    int* bins;              // chunks per cost bin, then the rewrite's cursors (2 x kCostBins)
};
// bin of a cost, longest first: 16 bins per factor of two from 2^8 cycles up
__device__ __forceinline__ int cost_bin(float c)
{
    const int b = (__float_as_int(c) >> 19) - ((127 + 8) << 4);
    return kCostBins - 1 - (b < 0 ? 0 : (b > kCostBins - 1 ? kCostBins - 1 : b));
}

struct WalkArgs {
    const double* x; const double* y; const double* z;
    const int8_t* sp;
    const double* qsp;      // charge per species (device, 2)
    const double* msp;      // mass, then charge over mass, per species (device, 4)
    const float4* src32;    // FP32C sources (src_place)
    Tree t;
    const int* targets;     // key-order slots of the targets, or NULL = all
    int ntargets;
    const int4* chunks;     // {first target index, count <= 32, cloud, 0}, one cloud each
    int nchunks;
    WalkOrder ord;          // FP32C forward walks only
    const int* pos_off;     // first box started at each sorted position (the roots)
    const Cube* cubes;      // per cloud: FP32C coordinates are taken relative to the centre
    double eps2;
    int leaf_cap;           // of the context
    int kelbg;              // electron-ion pairs use the Kelbg form (Sec. 2.1 Eq. 3)
    double lambda;          // its fixed lambda_ei
    double* ax; double* ay; double* az; double* phi;  // key order; phi may be NULL
    int* cnt_p2p; int* cnt_m2p;                        // key order
    int* work;              // dynamic work counter (zeroed before launch)
    const int* err;         // raised by a bounded wait that gave up: the tree is not walked
    unsigned long long* stats; // {p2p, m2p}
};
// per walk: box records (in an FP64 context also the moments, where they are still the sums
// launch_moments left), and the work counter and cost bins (may be NULL) cleared
void launch_mac_prepare(Tree t, const Cube* cube, double theta, int want_f32, int* work, int* bins,
                        Queue s);
void launch_walk_fp64(const WalkArgs& a, int nsm, Queue s);
void launch_walk_fp32c(const WalkArgs& a, int nsm, Queue s, int shape);
void launch_walk_fp32c_visits(const WalkArgs& a, int nsm, Queue s);  // no potential
int walk_shape_count();
// rewrites o.order longest-first by the costs of the walk just finished
void launch_chunk_order(const WalkOrder& o, int nchunks, Queue s);

// ---- adjoint (ucp_adjoint.cu) ----
// mu (n particles, key order) = (d a / d x)^T lam over the targets of a (all
// particles when a.targets is NULL; the others must have lam = 0)
void launch_walk_adjoint(const WalkArgs& a, const double* lam, double* mu, double* adj, int n,
                         int nsm, Queue s);
void launch_gather3(const double* src, const unsigned int* id, int n, double* dst, Queue s);
void launch_scatter_add3(const double* src, const unsigned int* id, int n, double* dst,
                         Queue s);
void launch_kick_lambda(const double* lam_v, const int8_t* sp, int n, double ce, double ci,
                        double* out, Queue s);
void launch_axpy3(double* y, const double* x, double a, int n, Queue s);
void launch_scatter_rows3(const double* src, const unsigned int* id, int n, double* dst,
                          Queue s);
size_t ke_seed_words();  // doubles at loss: the sum and the blocks' partial sums
void launch_ke_seed(const double* v, const int8_t* sp, int n, double me, double* lam_v,
                    double* loss, Queue s);

// ---- push and reductions (ucp_push.cu) ----
void launch_kick(double* vx, double* vy, double* vz, const double* ax, const double* ay,
                 const double* az, const int8_t* sp, int species, double h, int n, int times,
                 Queue s);
// list = the slots whose species is `species`, in slot order; partials holds
// select_words(n) ints; cnt0 and cnt1 (n ints, may be NULL) are cleared
size_t select_words(int n);
void launch_select(const int8_t* sp, int species, int n, int* list, int* partials, int* cnt0,
                   int* cnt1, Queue s);
void launch_drift(double* x, double* y, double* z, const double* vx, const double* vy,
                  const double* vz, double dt, int n, Queue s);
// out[6 c ..]: observables of cloud c (cloud_start NULL: one cloud over [0, n)); partials
// holds 6 n_clouds nblk doubles
void launch_energy(const double* vx, const double* vy, const double* vz, const double* phi,
                   const int8_t* sp, const double* qsp, const double* msp, int n,
                   const int* cloud_start, int n_clouds, double* partials, int nblk, double* out,
                   Queue s);
void launch_scatter3(const double* ax, const double* ay, const double* az, const unsigned int* id,
                     int n, double* out, Queue s);
void launch_scatter1(const double* a, const unsigned int* id, int n, double* out, Queue s);
void launch_scatter_int(const int* a, const unsigned int* id, int n, int* out, Queue s);
void launch_load_state(const double* pos, const double* vel, const int8_t* sp, int n,
                       double* const* st6, int8_t* sp_slot, int8_t* sp_caller, unsigned int* id,
                       Queue s);
// flags: {non-finite, bad species, electrons of cloud 0, 1, ...}, zeroed before
void launch_check_state(const double* pos, const double* vel, const int8_t* sp, int n,
                        const unsigned char* cloud, int* flags, Queue s);
void launch_chunks(const int* first, const int* place, int n_clouds, int width, int nchunks,
                   int4* chunks, int* order, int n_other, int* other, Queue s);

}  // namespace ucp
