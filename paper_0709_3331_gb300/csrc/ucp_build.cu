// ucp_build.cu -- TREE construction of Sec. 3 (arXiv 0709.3331) on the GPU:
// enclosing cube, Morton keys, stable radix sort, box topology as key
// prefixes in pre-order, and box moments bottom-up.
//
// Arithmetic that decides an integer (cube, cell coordinates, box centre) is
// written with explicit round-to-nearest intrinsics in the order of the
// definition, so that no multiply-add contraction changes a cell.
#include "ucp_box.cuh"
#include "ucp_scan.cuh"

#include <math.h>

namespace ucp {

namespace {

// ---------------------------------------------------------------- cube
// Ordered integer image of a finite double: comparing the images compares the
// values, so min/max run on the integer ALU instead of the (scarce) FP64 pipe.
// Partial min/max of cloud blockIdx.y over its segment (the whole array when
// cloud_start is NULL); block x of the cloud strides the segment.
__global__ void k_bbox_partial(const double* __restrict__ x, const double* __restrict__ y,
                               const double* __restrict__ z, int n, double* __restrict__ part,
                               const int* __restrict__ cloud_start)
{
    follow();
    const int c = blockIdx.y;
    const int lo_i = cloud_start ? cloud_start[c] : 0, hi_i = cloud_start ? cloud_start[c + 1] : n;
    unsigned long long lo[3] = {~0ull, ~0ull, ~0ull}, hi[3] = {0ull, 0ull, 0ull};
    for (int i = lo_i + blockIdx.x * blockDim.x + threadIdx.x; i < hi_i;
         i += gridDim.x * blockDim.x) {
        unsigned long long v[3] = {ord64(x[i]), ord64(y[i]), ord64(z[i])};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            lo[a] = min(lo[a], v[a]);
            hi[a] = max(hi[a], v[a]);
        }
    }
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lo[a] = min(lo[a], __shfl_xor_sync(0xffffffffu, lo[a], o));
            hi[a] = max(hi[a], __shfl_xor_sync(0xffffffffu, hi[a], o));
        }
    __shared__ unsigned long long s[32][6];
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0)
        for (int a = 0; a < 3; ++a) {
            s[w][a] = lo[a];
            s[w][3 + a] = hi[a];
        }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int ww = 1; ww < (int)(blockDim.x >> 5); ++ww)
            for (int a = 0; a < 3; ++a) {
                s[0][a] = min(s[0][a], s[ww][a]);
                s[0][3 + a] = max(s[0][3 + a], s[ww][3 + a]);
            }
        // an empty partial (more blocks than particles) keeps +/-inf
        double* pp = part + ((size_t)c * gridDim.x + blockIdx.x) * 6;
        for (int a = 0; a < 3; ++a) {
            pp[a] = s[0][a] == ~0ull ? INFINITY : unord64(s[0][a]);
            pp[3 + a] = s[0][3 + a] == 0ull ? -INFINITY : unord64(s[0][3 + a]);
        }
    }
}

// Sec. 3: the cube that encloses every particle, from the images of the lowest and the
// highest coordinates.  Centre = (min + max) / 2 per axis; side = largest extent *
// (1 + 2^-20) so that the maximum falls inside; side 1 when all particles coincide.
__device__ __forceinline__ void enclosing_cube(const unsigned long long* s, Cube* cube)
{
    double ext = 0.0;
    for (int a = 0; a < 3; ++a) {
        const double mn = unord64(s[a]), mx = unord64(s[3 + a]);
        cube->c[a] = __dmul_rn(__dadd_rn(mn, mx), 0.5);
        double e = __dsub_rn(mx, mn);
        if (e > ext) ext = e;
    }
    double L = ext > 0.0 ? __dmul_rn(ext, 1.0 + 0x1p-20) : 1.0;
    cube->L = L;
    for (int a = 0; a < 3; ++a) cube->lo[a] = __dsub_rn(cube->c[a], __dmul_rn(L, 0.5));
    cube->kscale = __ddiv_rn(2097152.0, L);
}

// Clears a build's counters and advances the tag of the published words, by one block.
// Every build's published words carry a tag 16 above the previous build's, kept on the
// device so that a captured graph replays with fresh tags (every word of a region is
// rewritten each build, so a stale word always carries an older tag, also across 30-bit
// wrap-around).
__device__ __forceinline__ void clear_build(const BuildCtl& ctl)
{
    for (int i = threadIdx.x; i < kCtlWords; i += blockDim.x) ctl.words[i] = 0;
    if (threadIdx.x == 0) *ctl.epoch = (*ctl.epoch + 16u) & 0x3fffffffu;
}

// The cubes from the partial extents.
__global__ void k_bbox_final(const double* __restrict__ part, int nblk, Cube* cubes, BuildCtl ctl)
{
    follow();
    if (blockIdx.x == 0) clear_build(ctl);
    part += (size_t)blockIdx.x * nblk * 6;  // cloud blockIdx.x
    Cube* cube = cubes + blockIdx.x;
    // min and max taken on the ordered integer images, as in k_bbox_partial
    __shared__ unsigned long long s[256][6];
    unsigned long long lo[3] = {~0ull, ~0ull, ~0ull}, hi[3] = {0ull, 0ull, 0ull};
    for (int b = threadIdx.x; b < nblk; b += blockDim.x)
        for (int a = 0; a < 3; ++a) {
            lo[a] = min(lo[a], ord64(part[6 * b + a]));
            hi[a] = max(hi[a], ord64(part[6 * b + 3 + a]));
        }
    for (int a = 0; a < 3; ++a) {
        s[threadIdx.x][a] = lo[a];
        s[threadIdx.x][3 + a] = hi[a];
    }
    __syncthreads();
    for (int st = 128; st > 0; st >>= 1) {
        if ((int)threadIdx.x < st)
            for (int a = 0; a < 3; ++a) {
                s[threadIdx.x][a] = min(s[threadIdx.x][a], s[threadIdx.x + st][a]);
                s[threadIdx.x][3 + a] = max(s[threadIdx.x][3 + a], s[threadIdx.x + st][3 + a]);
            }
        __syncthreads();
    }
    if (threadIdx.x == 0) enclosing_cube(s[0], cube);
}

// The same for one cloud of up to kBlockSort particles by one block, in one launch: at
// N = 2048 5 us for 8 + 4.5.
__global__ void __launch_bounds__(kBlockThreads)
k_bbox_block(const double* __restrict__ x, const double* __restrict__ y,
             const double* __restrict__ z, int n, Cube* cube, BuildCtl ctl)
{
    follow();
    clear_build(ctl);
    unsigned long long lo[3] = {~0ull, ~0ull, ~0ull}, hi[3] = {0ull, 0ull, 0ull};
#pragma unroll 4
    for (int i = threadIdx.x; i < n; i += kBlockThreads) {
        const unsigned long long v[3] = {ord64(x[i]), ord64(y[i]), ord64(z[i])};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            lo[a] = min(lo[a], v[a]);
            hi[a] = max(hi[a], v[a]);
        }
    }
    __shared__ unsigned long long s[6][kBlockThreads / 32], r[6];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lo[a] = min(lo[a], __shfl_xor_sync(0xffffffffu, lo[a], o));
            hi[a] = max(hi[a], __shfl_xor_sync(0xffffffffu, hi[a], o));
        }
        if (lane == 0) {
            s[a][w] = lo[a];
            s[3 + a][w] = hi[a];
        }
    }
    __syncthreads();
    if (w < 6) {
        unsigned long long v = s[w][lane];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long u = __shfl_xor_sync(0xffffffffu, v, o);
            v = w < 3 ? min(v, u) : max(v, u);
        }
        if (lane == 0) r[w] = v;
    }
    __syncthreads();
    if (threadIdx.x == 0) enclosing_cube(r, cube);
}

// ---------------------------------------------------------------- keys
__device__ __forceinline__ unsigned long long spread3(unsigned int v)
{
    unsigned long long x = v & 0x1fffffu;
    x = (x | (x << 32)) & 0x001f00000000ffffull;
    x = (x | (x << 16)) & 0x001f0000ff0000ffull;
    x = (x | (x << 8)) & 0x100f00f00f00f00full;
    x = (x | (x << 4)) & 0x10c30c30c30c30c3ull;
    x = (x | (x << 2)) & 0x1249249249249249ull;
    return x;
}

// cell coordinate k = floor((x - lo) * (2^21 / L)), clamped to [0, 2^21 - 1].
// Truncation toward zero equals floor wherever the clamp keeps the value (it
// differs only below 0, which clamps to 0 either way), and the saturating
// conversion keeps values past the int range above the upper clamp: three FP64
// operations per axis, the clamps on the integer ALU.
__device__ __forceinline__ unsigned int cell_coord(double x, double lo, double kscale)
{
    const int k = __double2int_rz(__dmul_rn(__dsub_rn(x, lo), kscale));
    return (unsigned int)min(max(k, 0), 2097151);
}

__device__ __forceinline__ unsigned long long morton_key(double x, double y, double z,
                                                         const Cube* __restrict__ cube)
{
    const double ks = cube->kscale;
    return spread3(cell_coord(x, cube->lo[0], ks)) | (spread3(cell_coord(y, cube->lo[1], ks)) << 1) |
           (spread3(cell_coord(z, cube->lo[2], ks)) << 2);
}

// Keys, and the digit counts of every pass of the sort (the passes' digits are the
// key's top 8 passes bits).
constexpr int kKeyThreads = 256;
__global__ void __launch_bounds__(kKeyThreads)
k_keys(const double* __restrict__ x, const double* __restrict__ y, const double* __restrict__ z,
       int n, const Cube* __restrict__ cubes, const unsigned char* __restrict__ cloud,
       unsigned long long* __restrict__ key, int passes, int* __restrict__ hist)
{
    follow();
    __shared__ int h[kSortPassesMax][kRadix];
    for (int i = threadIdx.x; i < passes * kRadix; i += kKeyThreads) (&h[0][0])[i] = 0;
    __syncthreads();
    const int low = kKeyBits - 8 * passes;
    for (int i = blockIdx.x * kKeyThreads + threadIdx.x; i < n; i += gridDim.x * kKeyThreads) {
        const unsigned long long k = morton_key(x[i], y[i], z[i], cubes + (cloud ? cloud[i] : 0));
        key[i] = k;
        for (int p = 0; p < passes; ++p)
            atomicAdd(&h[p][(unsigned int)(k >> (low + 8 * p)) & 0xffu], 1);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < passes * kRadix; i += kKeyThreads) {
        const int v = (&h[0][0])[i];
        if (v) atomicAdd(&hist[i], v);
    }
}

// ---------------------------------------------------------------- topology
__device__ __forceinline__ unsigned long long prefix_at(unsigned long long k, int d)
{
    return d == 0 ? 0ull : (k >> (3 * (kMaxDepth - d)));
}

// Boxes never span two clouds: every cloud occupies a fixed segment
// [seg_lo, seg_hi) of the key-sorted order (its own root, its own cube).

// first j > i in the segment whose depth-d prefix differs from key[i]'s (or seg_hi)
__device__ int box_end(const unsigned long long* __restrict__ K, int seg_hi, int i, int d)
{
    if (d == 0) return seg_hi;
    unsigned long long p = prefix_at(K[i], d);
    int lo = i, step = 1, hi = i + 1;
    while (hi < seg_hi && prefix_at(K[hi], d) == p) {
        lo = hi;
        step <<= 1;
        hi = i + step;
    }
    if (hi > seg_hi) hi = seg_hi;
    while (hi - lo > 1) {
        int mid = lo + ((hi - lo) >> 1);
        if (prefix_at(K[mid], d) == p) lo = mid;
        else hi = mid;
    }
    return hi;
}

// first j <= i in the segment whose depth-d prefix equals key[i]'s
__device__ int box_begin(const unsigned long long* __restrict__ K, int seg_lo, int i, int d)
{
    if (d == 0) return seg_lo;
    unsigned long long p = prefix_at(K[i], d);
    int hi = i, step = 1, lo = i - 1;
    while (lo >= seg_lo && prefix_at(K[lo], d) == p) {
        hi = lo;
        step <<= 1;
        lo = i - step;
    }
    if (lo < seg_lo - 1) lo = seg_lo - 1;
    while (hi - lo > 1) {
        int mid = lo + ((hi - lo) >> 1);
        if (prefix_at(K[mid], d) == p) hi = mid;
        else lo = mid;
    }
    return hi;
}

// depth of the first box that starts at sorted position i (22 = none)
__device__ __forceinline__ int first_depth(const unsigned long long* __restrict__ K, int seg_lo,
                                           int i)
{
    if (i == seg_lo) return 0;
    unsigned long long x = K[i] ^ K[i - 1];
    if (x == 0ull) return kMaxDepth + 1;
    return (__clzll((long long)x) - 1) / 3 + 1;
}

__device__ __forceinline__ void segment_of(const Tree& t, int n, int i, int& lo, int& hi)
{
    if (t.cloud) {
        const int c = t.cloud[i];
        lo = t.cloud_start[c];
        hi = t.cloud_start[c + 1];
    } else {
        lo = 0;
        hi = n;
    }
}

// Every box is a key prefix; the boxes that start at sorted position i are
// those of depth >= first_depth(i) down to the first leaf.  A box exists iff
// its parent holds more than leaf_cap particles.  Emitting boxes in order of
// (start position, depth) gives pre-order with children in octant order.
__device__ int count_by_search(const unsigned long long* __restrict__ K, int lo, int hi, int i,
                               int leaf_cap)
{
    const int d0 = first_depth(K, lo, i);
    if (d0 > kMaxDepth) return 0;
    if (d0 > 0 && box_end(K, hi, i, d0 - 1) - box_begin(K, lo, i, d0 - 1) <= leaf_cap) return 0;
    int c = 0;
    for (int d = d0; d <= kMaxDepth; ++d) {
        const int e = box_end(K, hi, i, d);
        ++c;
        if (e - i <= leaf_cap || d == kMaxDepth) break;
    }
    return c;
}

// ---- the same counts by a window of sorted positions (leaf_cap <= kTopoWin).
// fd[j] = first_depth(j): the box of depth d that holds position i ends at the
// first j > i with fd[j] <= d and starts at the last j <= i with fd[j] <= d.  It
// holds at most leaf_cap particles iff those two lie within leaf_cap of each
// other, so the depth of the leaf that holds i is
//   min over m = 0 .. leaf_cap - 1 of max(min fd[i - m .. i], min fd[i + 1 .. i + leaf_cap - m])
// (capped at kMaxDepth): a fixed window of shared memory instead of searches.
// Outside [0, n) and at every segment start fd is 0, which closes every box.
constexpr int kTopoThreads = 256;
constexpr int kTopoWin = 32;

__device__ __forceinline__ int fd_at(const unsigned long long* __restrict__ K, const Tree& t,
                                     int n, int j)
{
    if (j <= 0 || j >= n) return 0;
    int lo, hi;
    segment_of(t, n, j, lo, hi);
    return first_depth(K, lo, j);
}

// fd over [base - kTopoWin, base + kTopoThreads + kTopoWin) into smem
__device__ __forceinline__ void load_fd_window(const unsigned long long* __restrict__ K,
                                               const Tree& t, int n, int base,
                                               unsigned char* fd)
{
    for (int k = threadIdx.x; k < kTopoThreads + 2 * kTopoWin; k += kTopoThreads)
        fd[k] = (unsigned char)fd_at(K, t, n, base - kTopoWin + k);
}

// depth of the leaf that holds the position in slot li (see above); the
// backward running minima stay in registers (fully unrolled over the window)
__device__ __forceinline__ int leaf_depth_win(const unsigned char* fd, int li, int w)
{
    int bmin[kTopoWin];
    int bm = 255;
#pragma unroll
    for (int m = 0; m < kTopoWin; ++m) {
        if (m < w) bm = min(bm, (int)fd[li - m]);
        bmin[m] = bm;
    }
    int fm = 255, best = 255;
#pragma unroll
    for (int m = kTopoWin - 1; m >= 0; --m) {
        if (m < w) {
            fm = min(fm, (int)fd[li + (w - m)]);
            best = min(best, max(bmin[m], fm));
        }
    }
    return min(best, kMaxDepth);
}

// Box counts of every position and their exclusive prefix sums in one kernel
// (decoupled look-back over tiles taken from a counter, as in the key sort; waits
// bounded), which gives every box its place; a tile also clears the child slots and
// arrival counters of the boxes that start in it, and, when the sort left that to it (from
// = the slots in key order), moves the state of its positions.
constexpr int kTopoSpinLimit = 1 << 20;

template <bool kWin>
__global__ void __launch_bounds__(kTopoThreads)
k_topo_scan(const unsigned long long* __restrict__ K, int n, int leaf_cap, int* __restrict__ cnt,
            int* __restrict__ off, Tree t, BuildCtl ctl, unsigned long long* status, int* err,
            StateRef in, StateRef out, const unsigned int* __restrict__ from)
{
    follow();
    __shared__ unsigned char fd[kWin ? kTopoThreads + 2 * kTopoWin : 1];
    __shared__ int s_tile, s_tot, s_prefix;
    if (threadIdx.x == 0) s_tile = atomicAdd(&ctl.words[kCtlTopoTile], 1);
    __syncthreads();
    const int tile = s_tile, base = tile * kTopoThreads;
    const int i = base + threadIdx.x;
    if (from && i < n) move_state(in, out, i, from[i]);
    int c = 0;
    if (kWin) {
        load_fd_window(K, t, n, base, fd);
        __syncthreads();
        const int li = threadIdx.x + kTopoWin;
        const int d0 = fd[li];
        if (i < n && d0 <= kMaxDepth) {
            const int lv = leaf_depth_win(fd, li, leaf_cap);
            if (lv >= d0) c = lv - d0 + 1;
        }
    } else if (i < n) {
        int lo, hi;
        segment_of(t, n, i, lo, hi);
        c = count_by_search(K, lo, hi, i, leaf_cap);
    }
    const int before = block_excl_scan(c, &s_tot);
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        const unsigned int epoch = (*ctl.epoch + 15u) & 0x3fffffffu;
        const unsigned long long tag = (unsigned long long)epoch << 34;
        if (lane == 0 && tile > 0)
            atomicExch(status + tile, tag | (1ull << 32) | (unsigned int)s_tot);
        unsigned int prefix = 0;
        int spins = 0;
        for (int j = tile - 1; j >= 0;) {
            // lane l reads the word of tile j - l (past the first tile: nothing, final)
            const unsigned long long v = j - lane >= 0 ? __ldcv(status + (j - lane)) : tag | (2ull << 32);
            const unsigned int flag = (v >> 34) == (unsigned long long)epoch
                                          ? (unsigned int)(v >> 32) & 3u : 0u;
            const unsigned int fin = __ballot_sync(0xffffffffu, flag == 2u);
            const unsigned int none = __ballot_sync(0xffffffffu, flag == 0u);
            // the lanes up to the first final word, all published?
            const int last = fin ? __ffs(fin) - 1 : 31;
            if (none & (0xffffffffu >> (31 - last))) {
                if (++spins > kTopoSpinLimit) {
                    if (lane == 0) atomicOr(err, 1);
                    break;
                }
                __nanosleep(32);
                continue;
            }
            unsigned int sum = lane <= last ? (unsigned int)v : 0u;
            prefix += __reduce_add_sync(0xffffffffu, sum);
            if (fin) break;
            j -= 32;
        }
        if (lane == 0) {
            atomicExch(status + tile, tag | (2ull << 32) | (prefix + (unsigned int)s_tot));
            s_prefix = (int)prefix;
        }
    }
    __syncthreads();
    const int first = s_prefix, tot = s_tot;
    if (i < n) {
        cnt[i] = c;
        off[i] = first + before;
    }
    // the capacity bounds the box count of sorted keys; clamp in case it ever did not
    if (threadIdx.x == 0 && base + kTopoThreads >= n) *t.nnodes = min(first + tot, t.cap);
    const int lim = min(first + tot, t.cap);
    for (int b = first + threadIdx.x; b < lim; b += kTopoThreads) t.arrive[b] = 0;
    int4* rows = reinterpret_cast<int4*>(t.child8);
    for (int r = 2 * first + threadIdx.x; r < 2 * lim; r += kTopoThreads)
        rows[r] = make_int4(-1, -1, -1, -1);
}

// The boxes that start at each position, with their parents.  The parent of the first
// one, of depth d0 - 1, starts at the last earlier position whose first box is no
// deeper: found in a table of minima of the first depths over 1, 2, 4, .. 256 positions
// (nine steps in shared memory, 256 positions back), else by search.  A leaf ends where
// the next box starts and skips to the next box; twigs take their end and skip from
// their last child (the moments' bottom-up sweep).
constexpr int kTopoLevels = 9;

__global__ void __launch_bounds__(kTopoThreads)
k_topo_emit(const unsigned long long* __restrict__ K, int n, const int* __restrict__ cnt,
            const int* __restrict__ off, Tree t)
{
    follow();
    __shared__ unsigned char mn[kTopoLevels][2 * kTopoThreads];
    __shared__ unsigned int starts[kTopoThreads / 32];
    __shared__ int s_depth;
    const int base = blockIdx.x * kTopoThreads, i = base + threadIdx.x;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int k = threadIdx.x; k < 2 * kTopoThreads; k += kTopoThreads)
        mn[0][k] = (unsigned char)fd_at(K, t, n, base - kTopoThreads + k);
    const int c = i < n ? cnt[i] : 0;
    const unsigned int sb = __ballot_sync(0xffffffffu, c > 0);
    if (lane == 0) starts[w] = sb;
    if (threadIdx.x == 0) s_depth = 0;
    for (int v = 1; v < kTopoLevels; ++v) {
        __syncthreads();
        const int h = 1 << (v - 1);
        for (int k = threadIdx.x; k < 2 * kTopoThreads; k += kTopoThreads)
            mn[v][k] = min(mn[v - 1][k], k >= h ? mn[v - 1][k - h] : (unsigned char)255);
    }
    __syncthreads();
    if (c > 0) {
        int lo, hi;
        segment_of(t, n, i, lo, hi);
        const int d0 = i == lo ? 0 : mn[0][kTopoThreads + threadIdx.x];
        int parent = -1;
        if (d0 > 0) {
            int k = kTopoThreads + (int)threadIdx.x - 1;
#pragma unroll
            for (int v = kTopoLevels - 1; v >= 0; --v)
                if (k - (1 << v) + 1 >= 0 && mn[v][k] >= d0) k -= 1 << v;
            int pb, dp;
            if (k >= 0) {
                pb = base - kTopoThreads + k;
                dp = pb == lo ? 0 : mn[0][k];
            } else {
                pb = box_begin(K, lo, i, d0 - 1);
                dp = first_depth(K, lo, pb);
            }
            parent = off[pb] + (d0 - 1 - dp);
        }
        // the next start: in this warp, in a later warp of the block, or by search
        int e = -1;
        const unsigned int later = lane < 31 ? sb >> (lane + 1) : 0u;
        if (later) e = i + __ffs(later);
        for (int ww = w + 1; ww < kTopoThreads / 32 && e < 0; ++ww)
            if (starts[ww]) e = base + ww * 32 + __ffs(starts[ww]) - 1;
        if (e < 0) e = box_end(K, hi, i, d0 + c - 1);
        int node = off[i];
        for (int j = 0; j < c; ++j) {
            if (node >= t.cap || parent >= t.cap) break;  // cannot happen: the capacity bounds the box count
            const int d = d0 + j;
            const bool leaf = j == c - 1;
            const unsigned long long pre = prefix_at(K[i], d);
            t.info[node] = make_int4(i, leaf ? e : -1, leaf ? node + 1 : -1, parent);
            t.depth_leaf[node] = d | (leaf ? 256 : 0);
            t.cell[node] = pre;
            if (parent >= 0) t.child8[(size_t)parent * 8 + (int)(pre & 7ull)] = node;
            parent = node;
            ++node;
        }
        atomicMax(&s_depth, d0 + c - 1);
    }
    __syncthreads();
    if (threadIdx.x == 0 && s_depth > 0) atomicMax(t.maxdepth, s_depth);
}

// ---------------------------------------------------------------- moments
// Sum over the eight lanes of a group by an xor butterfly, in every lane:
// ((s0 + s4) + (s2 + s6)) + ((s1 + s5) + (s3 + s7)).
template <class T>
__device__ __forceinline__ T sum8(T v)
{
    v += __shfl_xor_sync(0xffffffffu, v, 4);
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    return v;
}

// A twig of the bottom-up sweep (id < 0: none).
struct Twig {
    int id, parent, first, depth;       // first: particle
    unsigned long long cell;
    int nch, last;                      // children, and the last of them
};

__device__ __forceinline__ Twig load_twig(const Tree& t, int p)
{
    Twig w = {p, -1, 0, 0, 0ull, 0, -1};
    if (p < 0) return w;
    const int4* row = reinterpret_cast<const int4*>(t.child8 + (size_t)p * 8);
    const int4 r0 = row[0], r1 = row[1];
    w.first = t.info[p].x;
    w.parent = t.info[p].w;
    w.depth = t.depth_leaf[p] & 255;
    w.cell = t.cell[p];
    const int ch[8] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w};
#pragma unroll
    for (int o = 0; o < 8; ++o) {
        w.nch += ch[o] >= 0;
        if (ch[o] >= 0) w.last = ch[o];
    }
    return w;
}

// One step of a sum by halving exchanges: lanes with the bit set keep b and send a, the
// others keep a and send b.
__device__ __forceinline__ double halve(bool bit, double a, double b, int mask)
{
    return (bit ? b : a) + __shfl_xor_sync(0xffffffffu, bit ? a : b, mask);
}

// Sums of child ch, in slot o of a twig, about the twig's geometric centre: shifted by the
// difference of the centres, h = a quarter of the twig's side along each axis, signed by the
// octant bit.  The child was written by another thread of the same launch: its record is
// read through L2 (__ldcg) after the acquire of the bottom-up sweep.
__device__ __forceinline__ void child_sums_f64(const Tree& t, int ch, int o, double h, double* a)
{
    const double2* r = reinterpret_cast<const double2*>(t.mom + (size_t)ch * kMom);
#pragma unroll
    for (int k = 0; k < 7; ++k) {
        const double2 v = __ldcg(r + k);
        a[2 * k] = v.x;
        a[2 * k + 1] = v.y;
    }
    const double e[3] = {o & 1 ? h : -h, o & 2 ? h : -h, o & 4 ? h : -h};
    const double me[3] = {a[1] * e[0], a[1] * e[1], a[1] * e[2]};
    // P + d e^T + e d^T + M e e^T
    a[8] += (2.0 * a[5] + me[0]) * e[0];
    a[9] += a[5] * e[1] + (a[6] + me[1]) * e[0];
    a[10] += a[5] * e[2] + (a[7] + me[2]) * e[0];
    a[11] += (2.0 * a[6] + me[1]) * e[1];
    a[12] += a[6] * e[2] + (a[7] + me[2]) * e[1];
    a[13] += (2.0 * a[7] + me[2]) * e[2];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        a[2 + k] += a[0] * e[k];
        a[5 + k] += me[k];
    }
}

// Sums of a twig with one or two children by one lane (the same bits as by eight: the other
// slots add zeros).  The first child follows the twig.
__device__ __forceinline__ void narrow_sums_f64(const Cube* __restrict__ cube, const Tree& t,
                                                const Twig& w)
{
    const double h = ldexp(cube_of(cube, t, w.first).L, -(w.depth + 2));
    double a[14];
#pragma unroll
    for (int k = 0; k < 14; ++k) a[k] = 0.0;
#pragma unroll 1
    for (int c = 0; c < w.nch; ++c) {
        const int ch = c ? w.last : w.id + 1;
        double b[14];
        child_sums_f64(t, ch, (int)(t.cell[ch] & 7ull), h, b);
#pragma unroll
        for (int k = 0; k < 14; ++k) a[k] += b[k];
    }
    double2* r = reinterpret_cast<double2*>(t.mom + (size_t)w.id * kMom);
#pragma unroll
    for (int k = 0; k < 7; ++k) r[k] = make_double2(a[2 * k], a[2 * k + 1]);
    t.delta[w.id] = kSumsDelta;
}

// Sums of a twig about its geometric centre by a group of eight lanes, one child slot o
// each (ch < 0: empty).  A level costs its latency and the
// FP64 pipe's 16 cycles per warp instruction, so nothing but the sums goes up the tree
// (moments follow from them with the walk's records, one box per lane), and they are
// added by halving exchanges, 14 additions for 14 values instead of 42, which leave sums
// o and 8 + o in lane o.  With the centroid, division and root of every level in the
// chain, and 256 positions to a block, this kernel took 58 us at N = 2048 and 89 at
// 131,072; now 33 and 63, and the moments 3 us of the walk's preparation.
__device__ __forceinline__ void twig_sums_f64(const Cube* __restrict__ cube, const Tree& t,
                                              const Twig& w, int o, int ch)
{
    double a[14];
#pragma unroll
    for (int k = 0; k < 14; ++k) a[k] = 0.0;
    if (ch >= 0) child_sums_f64(t, ch, o, ldexp(cube_of(cube, t, w.first).L, -(w.depth + 2)), a);
    // ((s0 + s4) + (s2 + s6)) + ((s1 + s5) + (s3 + s7)) of each value
    const bool b4 = o & 4, b2 = o & 2, b1 = o & 1;
    double u[8];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        u[k] = halve(b4, a[k], a[4 + k], 4);
        u[4 + k] = halve(b4, a[8 + k], k < 2 ? a[12 + k] : 0.0, 4);
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        u[k] = halve(b2, u[k], u[2 + k], 2);
        u[4 + k] = halve(b2, u[4 + k], u[6 + k], 2);
    }
    const double lo = halve(b1, u[0], u[1], 1), hi = halve(b1, u[4], u[5], 1);
    if (w.id >= 0) {
        double* r = t.mom + (size_t)w.id * kMom;
        r[o] = lo;
        if (o < 6) r[8 + o] = hi;
        if (o == 7) t.delta[w.id] = kSumsDelta;
    }
}

// atomicAdd with acquire-release semantics at device scope: the caller's
// earlier writes are visible to whoever reads the counter after it (release),
// and the writes released by every earlier increment of the counter are
// visible to the caller after it (acquire: the increments form one release
// sequence).  One ordered atomic in place of a fence on either side.
__device__ __forceinline__ int atomic_add_acq_rel(int* ctr, int v)
{
    int old;
    asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], %2;"
                 : "=r"(old) : "l"(ctr), "r"(v) : "memory");
    return old;
}

// Bottom-up sweep from the finished boxes of a warp's lanes (node < 0: none): each box
// counts its finished children (t.arrive, cleared with the topology); the lane that
// finishes the last child has the parent combined, four parents at a time by groups of
// eight lanes, and carries on upwards.  No thread waits for another, and every twig is
// combined once, from all its children, whichever warp does it.  Where more than eight of a
// warp's twigs have one or two children, each of those lanes combines its own, narrow(twig),
// in the time of two rounds of the groups: close pairs in small leaves hang on chains of up to
// 20 boxes with a single child, and particles on a line have two to a box.  A build of 131,072
// particles in pairs 1e-6 apart with leaves of 1: FP64 1.64 -> 0.45 ms, FP32C 1.33 -> 0.46.
template <bool kNarrow, class Combine, class Narrow>
__device__ __forceinline__ void sweep_up(const Tree& t, int node, Combine combine, Narrow narrow)
{
    const int lane = threadIdx.x & 31;
    // (a parent comes before its child: the sweep ends, also in tables that are no tree since
    // a wait gave up)
    int p = node >= 0 ? t.info[node].w : -1;
    Twig w = load_twig(t, p < node ? p : -1);
    while (__any_sync(0xffffffffu, w.id >= 0)) {
        // this box's records (written by any lane of the warp) are published with its
        // arrival; the last arrival sees every sibling's
        __syncwarp();
        const bool ready = w.id >= 0 && atomic_add_acq_rel(&t.arrive[w.id], 1) + 1 >= w.nch;
        unsigned int todo = __ballot_sync(0xffffffffu, ready);
        // what the acquiring lanes see, every lane sees.  The next twig's records come in
        // while this one is combined.
        __syncwarp();
        const Twig up = load_twig(t, ready && w.parent < w.id ? w.parent : -1);
        int4 lc;
        if (ready) lc = __ldcg(&t.info[max(w.last, 0)]);
        if (kNarrow && __popc(todo) > 8) {
            const unsigned int few = __ballot_sync(0xffffffffu, ready && w.nch <= 2);
            if (__popc(few) > 8) {
                if (ready && w.nch <= 2) narrow(w);
                todo &= ~few;
            }
        }
        while (todo) {
            // the (lane / 8)-th of the lanes that are left
            unsigned int m = todo;
            for (int g = 0; g < (lane >> 3) && m; ++g) m &= m - 1u;
            const int src = m ? __ffs(m) - 1 : 0;
            Twig q;
            q.id = __shfl_sync(0xffffffffu, w.id, src);
            q.first = __shfl_sync(0xffffffffu, w.first, src);
            q.depth = __shfl_sync(0xffffffffu, w.depth, src);
            q.cell = __shfl_sync(0xffffffffu, w.cell, src);
            if (!m) q.id = -1;
            const int o = lane & 7;
            const int ch = q.id >= 0 ? t.child8[(size_t)q.id * 8 + o] : -1;
            combine(q, o, ch);
            for (int g = 0; g < 4 && todo; ++g) todo &= todo - 1u;
        }
        if (ready) {
            // a twig ends where its last child (in octant order, so last in pre-order)
            // ends, and skips to where that child skips
            int* ip = reinterpret_cast<int*>(&t.info[w.id]);
            ip[1] = lc.y;
            ip[2] = lc.z;
        }
        w = up;
    }
}

// A block's leaves: those that start among its kPos positions, compacted in position
// order; returns their number.
constexpr int mom_threads(int pos) { return pos >= 256 ? 128 : 32; }
constexpr int kMomHalo = 32;       // largest leaf that is summed from shared memory
constexpr unsigned short kNoOwner = 0xffff;

template <int kPos>
__device__ __forceinline__ int block_leaves(const int* __restrict__ cnt, int base, int n,
                                            int* list)
{
    constexpr int kThreads = mom_threads(kPos);
    __shared__ int s_tot;
    int total = 0;
    for (int part = 0; part < kPos; part += kThreads) {
        const int i = base + part + threadIdx.x;
        const bool start = i < n && cnt[i] > 0;
        const int at = block_excl_scan(start ? 1 : 0, &s_tot);
        if (start) list[total + at] = i;
        total += s_tot;
        __syncthreads();
    }
    return total;
}

// FP64 sums of every leaf from its particles, one thread per leaf, summed about
// the leaf's geometric centre in key order, then the twigs (sweep_up).  Twigs shift by exactly
// a quarter of their side, so all sums are about exact centres: about the rounded ones, which
// are off by 2^-53 of the cube's side, a centroid was off by as much however near the box lies
// to the origin (rms error of the forces of a Gaussian cloud's cubes 1.6e-14, now 5e-16; of
// pairs 1e-6 apart in leaves of 1 9.4e-12, now 9.8e-15).
template <int kPos>
__global__ void __launch_bounds__(mom_threads(kPos))
k_moments(const double* __restrict__ x, const double* __restrict__ y,
          const double* __restrict__ z, const int8_t* __restrict__ sp,
          const double* __restrict__ qsp, int n, const int* __restrict__ cnt,
          const int* __restrict__ off, const Cube* __restrict__ cube, Tree t)
{
    follow();
    constexpr int kThreads = mom_threads(kPos);
    __shared__ int list[kPos];
    const int nl = block_leaves<kPos>(cnt, blockIdx.x * kPos, n, list);
    const double q0 = qsp[0], q1 = qsp[1];
    for (int l0 = threadIdx.x & ~31; l0 < nl; l0 += kThreads) {
        const int l = l0 + (threadIdx.x & 31);
        int node = -1;
        if (l < nl) {
            const int i = list[l];
            node = min(off[i] + cnt[i] - 1, t.cap - 1);
            const int4 inf = t.info[node];
            double zc[3], rho[3];
            box_centre_exact(cube_of(cube, t, inf.x), t.cell[node], t.depth_leaf[node] & 255, zc, rho);
            double a[14];
#pragma unroll
            for (int k = 0; k < 14; ++k) a[k] = 0.0;
#pragma unroll 4
            for (int j = inf.x; j < inf.y; ++j) {
                double qj = sp[j] ? q1 : q0;
                double aq = fabs(qj);
                double yv[3] = {x[j] - zc[0], y[j] - zc[1], z[j] - zc[2]};
                a[0] += aq;
                a[1] += qj;
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    a[2 + k] += aq * yv[k];
                    a[5 + k] += qj * yv[k];
                }
                double qy0 = qj * yv[0], qy1 = qj * yv[1];
                a[8] += qy0 * yv[0];
                a[9] += qy0 * yv[1];
                a[10] += qy0 * yv[2];
                a[11] += qy1 * yv[1];
                a[12] += qy1 * yv[2];
                a[13] += qj * yv[2] * yv[2];
            }
            // to the exact centre, on which the twigs' shifts rest
            a[8] -= 2.0 * (a[5] * rho[0]);
            a[9] -= a[5] * rho[1] + a[6] * rho[0];
            a[10] -= a[5] * rho[2] + a[7] * rho[0];
            a[11] -= 2.0 * (a[6] * rho[1]);
            a[12] -= a[6] * rho[2] + a[7] * rho[1];
            a[13] -= 2.0 * (a[7] * rho[2]);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                a[2 + k] -= a[0] * rho[k];
                a[5 + k] -= a[1] * rho[k];
            }
            double2* r = reinterpret_cast<double2*>(t.mom + (size_t)node * kMom);
#pragma unroll
            for (int k = 0; k < 7; ++k) r[k] = make_double2(a[2 * k], a[2 * k + 1]);
            t.delta[node] = kSumsDelta;
        }
        // (a small system's blocks of 32 positions gain less by it than its test costs)
        sweep_up<(kPos > 32)>(
            t, node, [&](const Twig& w, int o, int ch) { twig_sums_f64(cube, t, w, o, ch); },
            [&](const Twig& w) { narrow_sums_f64(cube, t, w); });
    }
}

// ---- FP32 moments (FP32C contexts).  Offsets from a box's geometric centre z
// are at most one box side, so they are formed in FP64 once and summed in FP32;
// the expansion centre is c = z + e exactly as stored (FP64), and D, Q are taken
// about that same point; the FP64 record of such a box holds its centre only.  Compact
// per-box record mom32 = {e xyz, S0, M, D xyz,
// Q xx xy xz yy yz zz, 0, 0} feeds the twig combine.
__device__ __forceinline__ void finish_box_f32(const float* a, const double z[3], float* m32,
                                               double* __restrict__ m64,
                                               double* __restrict__ delta)
{
    float S0 = a[0], M = a[1];
    float inv = S0 > 0.f ? 1.f / S0 : 0.f;
    float e[3] = {a[2] * inv, a[3] * inv, a[4] * inv};
    float d[3];
    for (int k = 0; k < 3; ++k) d[k] = fmaf(-M, e[k], a[5 + k]);
    const int ia[6] = {0, 0, 0, 1, 1, 2}, ib[6] = {0, 1, 2, 1, 2, 2};
    float q[6];
    for (int k = 0; k < 6; ++k)
        q[k] = a[8 + k] - a[5 + ia[k]] * e[ib[k]] - e[ia[k]] * a[5 + ib[k]] +
               M * e[ia[k]] * e[ib[k]];
    m32[0] = e[0];
    m32[1] = e[1];
    m32[2] = e[2];
    m32[3] = S0;
    m32[4] = M;
    for (int k = 0; k < 3; ++k) m32[5 + k] = d[k];
    for (int k = 0; k < 6; ++k) m32[8 + k] = q[k];
    m32[14] = 0.f;
    m32[15] = 0.f;
    for (int k = 0; k < 3; ++k) m64[MC + k] = z[k] + (double)e[k];
    *delta = sqrtf(fmaf(e[0], e[0], fmaf(e[1], e[1], e[2] * e[2])));
}

// Child slot o of a twig shifted to the twig's centre (zeros for an empty slot).
// The child's expansion centre lies at its own geometric centre plus its FP32
// offset e_child (mom32), and its geometric centre at the twig's plus q = side/4
// along each axis, signed by the octant bit (x bit 0, y bit 1, z bit 2): the shift
// is q +/- e_child, formed in FP32 without touching the FP64 unit.
__device__ __forceinline__ void twig_child_f32(const Tree& t, int ch, int o, float q, float* a)
{
#pragma unroll
    for (int k = 0; k < 14; ++k) a[k] = 0.f;
    if (ch < 0) return;
    const float4* r32 = reinterpret_cast<const float4*>(t.mom32 + (size_t)ch * 16);
    const float4 R0 = __ldcg(r32), R1 = __ldcg(r32 + 1), R2 = __ldcg(r32 + 2),
                 R3 = __ldcg(r32 + 3);
    const float S0k = R0.w, Mk = R1.x;
    const float dk[3] = {R1.y, R1.z, R1.w};
    const float qk[6] = {R2.x, R2.y, R2.z, R2.w, R3.x, R3.y};
    const float ec[3] = {R0.x, R0.y, R0.z};
    float e[3];
    for (int k = 0; k < 3; ++k) e[k] = ((o >> k) & 1 ? q : -q) + ec[k];
    a[0] = S0k;
    a[1] = Mk;
    for (int k = 0; k < 3; ++k) {
        a[2 + k] = S0k * e[k];
        a[5 + k] = fmaf(Mk, e[k], dk[k]);
    }
    float me0 = Mk * e[0], me1 = Mk * e[1], me2 = Mk * e[2];
    a[8] = qk[0] + (2.f * dk[0] + me0) * e[0];
    a[9] = qk[1] + dk[0] * e[1] + (dk[1] + me1) * e[0];
    a[10] = qk[2] + dk[0] * e[2] + (dk[2] + me2) * e[0];
    a[11] = qk[3] + (2.f * dk[1] + me1) * e[1];
    a[12] = qk[4] + dk[1] * e[2] + (dk[2] + me2) * e[1];
    a[13] = qk[5] + (2.f * dk[2] + me2) * e[2];
}

// A twig's records from its sums.
__device__ __forceinline__ void put_twig_f32(const Tree& t, const Twig& w, const float* a,
                                             const double zp[3])
{
    float m32[16];
    finish_box_f32(a, zp, m32, t.mom + (size_t)w.id * kCentre, t.delta + w.id);
    float4* w32 = reinterpret_cast<float4*>(t.mom32 + (size_t)w.id * 16);
    for (int k = 0; k < 4; ++k)
        w32[k] = make_float4(m32[4 * k], m32[4 * k + 1], m32[4 * k + 2], m32[4 * k + 3]);
}

// FP32 moments of a twig by a group of eight lanes, one child
// slot each, summed by an xor butterfly over the slots.
__device__ __forceinline__ void twig_combine_f32(const Cube* __restrict__ cube, const Tree& t,
                                                 const Twig& w, int o, int ch)
{
    double zp[3] = {0, 0, 0}, ps = 0.0;
    if (w.id >= 0) box_centre(cube_of(cube, t, w.first), w.cell, w.depth, zp, &ps);
    float a[14];
    twig_child_f32(t, ch, o, (float)(0.25 * ps), a);
#pragma unroll
    for (int k = 0; k < 14; ++k) a[k] = sum8(a[k]);
    if (w.id >= 0 && o == 0) put_twig_f32(t, w, a, zp);
}

// The same for a twig with one or two children, by one lane (the same bits: the other slots
// add zeros).  The first child follows the twig.
__device__ __forceinline__ void narrow_combine_f32(const Cube* __restrict__ cube, const Tree& t,
                                                   const Twig& w)
{
    double zp[3], ps;
    box_centre(cube_of(cube, t, w.first), w.cell, w.depth, zp, &ps);
    float a[14];
#pragma unroll
    for (int k = 0; k < 14; ++k) a[k] = 0.f;
#pragma unroll 1
    for (int c = 0; c < w.nch; ++c) {
        const int ch = c ? w.last : w.id + 1;
        float b[14];
        twig_child_f32(t, ch, (int)(t.cell[ch] & 7ull), (float)(0.25 * ps), b);
#pragma unroll
        for (int k = 0; k < 14; ++k) a[k] += b[k];
    }
    put_twig_f32(t, w, a, zp);
}

// One particle's source record, and the empty halves of its leaf's pairs.
__device__ __forceinline__ void put_source(float* f, int place, int begin, int j, float nx, float ny,
                                           float nz, float q)
{
    float* d = f + (size_t)(place + (j & ~1) - (begin & ~1)) * 4 + (j & 1);
    d[0] = nx;
    d[2] = ny;
    d[4] = nz;
    d[6] = q;
}
__device__ __forceinline__ void put_empty_halves(float* f, int place, int begin, int end)
{
    if (begin & 1) put_source(f, place, begin, begin - 1, kFarAway, 0.f, 0.f, 0.f);
    if (end & 1) put_source(f, place, begin, end, kFarAway, 0.f, 0.f, 0.f);
}

// FP32C contexts: a block takes the leaves that start among its kPos positions.
// kTile (leaves of up to kMomHalo particles): the particles' offsets from their leaf's
// geometric centre are formed with one particle per lane (the FP64 pipe takes a warp
// instruction for 16 cycles however many lanes are active) and kept in shared memory,
// where each leaf's thread sums them in key order; the source records are written one
// particle per lane again.  Larger leaves: one thread per leaf does all of it.  Then
// the twigs (sweep_up).
template <bool kTile, int kPos>
__global__ void __launch_bounds__(mom_threads(kPos))
k_moments_f32(const double* __restrict__ x, const double* __restrict__ y,
              const double* __restrict__ z, const int8_t* __restrict__ sp,
              const double* __restrict__ qsp, int n, const int* __restrict__ cnt,
              const int* __restrict__ off, const Cube* __restrict__ cube, Tree t,
              float4* __restrict__ src32)
{
    follow();
    constexpr int kThreads = mom_threads(kPos);
    __shared__ int list[kPos];
    __shared__ double ctr[kTile ? kPos : 1][3];                  // geometric centre, then c
    __shared__ float4 ys[kTile ? kPos + kMomHalo : 1];           // offset, charge
    __shared__ unsigned short owner[kTile ? kPos + kMomHalo : 1];
    __shared__ int place[kTile ? kPos : 1];
    const int base = blockIdx.x * kPos;
    const int nl = block_leaves<kPos>(cnt, base, n, list);
    const float q0 = (float)qsp[0], q1 = (float)qsp[1];
    float* f = reinterpret_cast<float*>(src32);
    if (kTile) {
        for (int l = threadIdx.x; l < nl; l += kThreads) {
            const int i = list[l];
            const int node = min(off[i] + cnt[i] - 1, t.cap - 1);
            const int4 inf = t.info[node];
            double side;
            box_centre(cube_of(cube, t, inf.x), t.cell[node], t.depth_leaf[node] & 255, ctr[l], &side);
            const int e = min(inf.y - base, kPos + kMomHalo);
            const bool fat = inf.y - inf.x > kMomHalo;   // a depth-cap box: its thread does it all
            place[l] = src_place(i, node);
            if (!fat) put_empty_halves(f, place[l], i, inf.y);
            for (int k = i - base; k < e; ++k) owner[k] = fat ? kNoOwner : (unsigned short)l;
        }
        __syncthreads();
        const int first = nl > 0 ? list[0] - base : kPos;
        const int end = nl > 0 ? min(t.info[min(off[list[nl - 1]] + cnt[list[nl - 1]] - 1, t.cap - 1)].y - base,
                                     kPos + kMomHalo) : 0;
        for (int k = first + threadIdx.x; k < end; k += kThreads) {
            const int j = base + k;
            if (owner[k] >= nl) continue;    // none, or a place that no leaf of the block covers
            const double* zc = ctr[owner[k]];
            ys[k] = make_float4((float)(x[j] - zc[0]), (float)(y[j] - zc[1]), (float)(z[j] - zc[2]),
                                sp[j] ? q1 : q0);
        }
        __syncthreads();
        for (int l = threadIdx.x; l < nl; l += kThreads) {
            const int i = list[l];
            const int node = min(off[i] + cnt[i] - 1, t.cap - 1);
            const int e = t.info[node].y - base;
            if (e - (i - base) > kMomHalo) continue;
            float a[14];
#pragma unroll
            for (int k = 0; k < 14; ++k) a[k] = 0.f;
#pragma unroll 4
            for (int k = i - base; k < e; ++k) {
                const float4 v = ys[k];
                const float qj = v.w, aq = fabsf(qj);
                const float yv[3] = {v.x, v.y, v.z};
                a[0] += aq;
                a[1] += qj;
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    a[2 + c] = fmaf(aq, yv[c], a[2 + c]);
                    a[5 + c] = fmaf(qj, yv[c], a[5 + c]);
                }
                float qy0 = qj * yv[0], qy1 = qj * yv[1];
                a[8] = fmaf(qy0, yv[0], a[8]);
                a[9] = fmaf(qy0, yv[1], a[9]);
                a[10] = fmaf(qy0, yv[2], a[10]);
                a[11] = fmaf(qy1, yv[1], a[11]);
                a[12] = fmaf(qy1, yv[2], a[12]);
                a[13] = fmaf(qj * yv[2], yv[2], a[13]);
            }
            float m32[16];
            double* m = t.mom + (size_t)node * kCentre;
            double zc[3] = {ctr[l][0], ctr[l][1], ctr[l][2]};
            double c64[3];
            finish_box_f32(a, zc, m32, c64, t.delta + node);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                m[MC + c] = c64[c];
                ctr[l][c] = c64[c];
            }
            float4* r32 = reinterpret_cast<float4*>(t.mom32 + (size_t)node * 16);
            for (int k = 0; k < 4; ++k)
                r32[k] = make_float4(m32[4 * k], m32[4 * k + 1], m32[4 * k + 2], m32[4 * k + 3]);
        }
        __syncthreads();
        for (int k = first + threadIdx.x; k < end; k += kThreads) {
            const int j = base + k, l = owner[k];
            if (l >= nl) continue;
            const double* c = ctr[l];
            put_source(f, place[l], list[l], j, (float)(c[0] - x[j]), (float)(c[1] - y[j]),
                       (float)(c[2] - z[j]), ys[k].w);
        }
    }
    for (int l0 = threadIdx.x & ~31; l0 < nl; l0 += kThreads) {
        const int l = l0 + (threadIdx.x & 31);
        int node = -1;
        if (l < nl) {
            const int i = list[l];
            node = min(off[i] + cnt[i] - 1, t.cap - 1);
            const int4 inf = t.info[node];
            if (!kTile || inf.y - inf.x > kMomHalo) {
                double zc[3], side;
                box_centre(cube_of(cube, t, inf.x), t.cell[node], t.depth_leaf[node] & 255, zc, &side);
                float a[14];
#pragma unroll
                for (int k = 0; k < 14; ++k) a[k] = 0.f;
                for (int j = inf.x; j < inf.y; ++j) {
                    float qj = sp[j] ? q1 : q0;
                    float aq = fabsf(qj);
                    float yv[3] = {(float)(x[j] - zc[0]), (float)(y[j] - zc[1]),
                                   (float)(z[j] - zc[2])};
                    a[0] += aq;
                    a[1] += qj;
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        a[2 + k] = fmaf(aq, yv[k], a[2 + k]);
                        a[5 + k] = fmaf(qj, yv[k], a[5 + k]);
                    }
                    float qy0 = qj * yv[0], qy1 = qj * yv[1];
                    a[8] = fmaf(qy0, yv[0], a[8]);
                    a[9] = fmaf(qy0, yv[1], a[9]);
                    a[10] = fmaf(qy0, yv[2], a[10]);
                    a[11] = fmaf(qy1, yv[1], a[11]);
                    a[12] = fmaf(qy1, yv[2], a[12]);
                    a[13] = fmaf(qj * yv[2], yv[2], a[13]);
                }
                float m32[16];
                double* m = t.mom + (size_t)node * kCentre;
                finish_box_f32(a, zc, m32, m, t.delta + node);
                float4* r32 = reinterpret_cast<float4*>(t.mom32 + (size_t)node * 16);
                for (int k = 0; k < 4; ++k)
                    r32[k] = make_float4(m32[4 * k], m32[4 * k + 1], m32[4 * k + 2], m32[4 * k + 3]);
                const double cx = m[MC], cy = m[MC + 1], cz = m[MC + 2];
                const int at = src_place(inf.x, node);
                put_empty_halves(f, at, inf.x, inf.y);
                for (int j = inf.x; j < inf.y; ++j)
                    put_source(f, at, inf.x, j, (float)(cx - x[j]), (float)(cy - y[j]),
                               (float)(cz - z[j]), sp[j] ? q1 : q0);
            }
        }
        sweep_up<true>(
            t, node, [&](const Twig& w, int o, int ch) { twig_combine_f32(cube, t, w, o, ch); },
            [&](const Twig& w) { narrow_combine_f32(cube, t, w); });
    }
}

}  // namespace

// ---------------------------------------------------------------- launchers
void launch_bbox(const double* x, const double* y, const double* z, int n, double* partials,
                 int nblk, Cube* cubes, const int* cloud_start, int n_clouds, BuildCtl ctl,
                 Queue s)
{
    if (block_sorted(n, n_clouds)) {
        count_launch(1);
        launch(k_bbox_block, 1, kBlockThreads, s, x, y, z, n, cubes, ctl);
        return;
    }
    count_launch(2);
    launch(k_bbox_partial, dim3(nblk, n_clouds), 256, s, x, y, z, n, partials, cloud_start);
    launch(k_bbox_final, n_clouds, 256, s, partials, nblk, cubes, ctl);
}

void launch_keys(const double* x, const double* y, const double* z, int n, const Cube* cubes,
                 const unsigned char* cloud, unsigned long long* key, int passes, BuildCtl ctl,
                 Queue s)
{
    count_launch(1);
    int nb = (n + kKeyThreads - 1) / kKeyThreads;
    if (nb > 8 * 152) nb = 8 * 152;
    launch(k_keys, nb, kKeyThreads, s, x, y, z, n, cubes, cloud, key, passes, ctl.words + kCtlHist);
}

void launch_topology(const unsigned long long* key, int n, int leaf_cap, int* pos_cnt,
                     int* pos_off, Tree t, BuildCtl ctl, unsigned long long* status, int* err,
                     const StateRef& in,
                     const StateRef& out, const unsigned int* from, Queue s)
{
    count_launch(2);
    const int nb = (n + kTopoThreads - 1) / kTopoThreads;
    if (leaf_cap <= kTopoWin)
        launch(k_topo_scan<true>, nb, kTopoThreads, s, key, n, leaf_cap, pos_cnt, pos_off, t, ctl,
               status, err, in, out, from);
    else
        launch(k_topo_scan<false>, nb, kTopoThreads, s, key, n, leaf_cap, pos_cnt, pos_off, t, ctl,
               status, err, in, out, from);
    launch(k_topo_emit, nb, kTopoThreads, s, key, n, pos_cnt, pos_off, t);
}

size_t topo_status_words(int n) { return (size_t)((n + kTopoThreads - 1) / kTopoThreads) + 1; }

template <int kPos>
static void moments(const double* x, const double* y, const double* z, const int8_t* sp,
                    const double* qsp, int n, int leaf_cap, const int* pos_cnt,
                    const int* pos_off, const Cube* cube, Tree t, float4* src32, int want_f32,
                    Queue s)
{
    constexpr int kThreads = mom_threads(kPos);
    const int nb = (n + kPos - 1) / kPos;
    if (!want_f32)
        launch(k_moments<kPos>, nb, kThreads, s, x, y, z, sp, qsp, n, pos_cnt, pos_off, cube, t);
    else if (leaf_cap <= kMomHalo)
        launch(k_moments_f32<true, kPos>, nb, kThreads, s, x, y, z, sp, qsp, n, pos_cnt, pos_off,
               cube, t, src32);
    else
        launch(k_moments_f32<false, kPos>, nb, kThreads, s, x, y, z, sp, qsp, n, pos_cnt, pos_off,
               cube, t, src32);
}

// Up to these sizes a block takes 32 positions instead of 256: the sweep is a chain of
// levels whose FP64 (centres in FP32C contexts) then runs on more SMs at once.  Larger
// systems fill the SMs either way, and the leaves of 256 positions fill a warp better.
// FP64: 30 against 34 us at N = 2048, 45 against 51 at 16384, 59 against 56 at 32768;
// FP32C: 22 against 27, 24 against 27, and at 65536 and 131072 31 against 32, 37 against 34.
constexpr int kMomSmallF64 = 16384, kMomSmallF32 = 65536;

void launch_moments(const double* x, const double* y, const double* z, const int8_t* sp,
                    const double* qsp, int n, int leaf_cap, const int* pos_cnt,
                    const int* pos_off, const Cube* cube, Tree t, float4* src32, int want_f32,
                    Queue s)
{
    // leaves from their particles, then every twig as its last child finishes
    // (bottom-up sweep with arrival counters), in one launch
    count_launch(1);
    if (n <= (want_f32 ? kMomSmallF32 : kMomSmallF64))
        moments<32>(x, y, z, sp, qsp, n, leaf_cap, pos_cnt, pos_off, cube, t, src32, want_f32, s);
    else
        moments<256>(x, y, z, sp, qsp, n, leaf_cap, pos_cnt, pos_off, cube, t, src32, want_f32, s);
}

}  // namespace ucp
