// ucp_sort.cu -- the key order of Sec. 3's TREE (arXiv 0709.3331) on the GPU: a stable
// radix sort of the Morton keys and the permutation of the particle state into that
// order, and the selection of the walk's targets.
//
// Only the key's top digits are sorted by radix passes: with 2^(8 passes) cells a run
// of particles whose keys share those digits is short (two on average in the densest
// part of a Gaussian cloud of 524,288 with three passes), and the kernel that moves
// the state orders each run of its tile by the rest of the key in shared memory.  A
// run longer than kRun raises a flag on the device, on which one further kernel,
// otherwise empty, sorts the whole key.  Three passes take 53 us at N = 524,288, eight
// took 165.
#include "ucp_scan.cuh"

namespace ucp {

namespace {

constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kSortChunks = 8;                              // 32-key chunks per warp
constexpr int kSortTile = kSortThreads * kSortChunks;       // 2048 keys per block
constexpr int kSortSpinLimit = 1 << 20;  // polls of a predecessor's word before giving up
constexpr int kLook = 8;                  // predecessors read per look-back round trip
constexpr int kRun = 32;                  // longest run ordered in shared memory

// Stable ranks of a tile's keys by digit: each warp owns a contiguous part and ranks it
// chunk by chunk with match_any; cnt[w][d] counts warp w's keys of digit d before.
struct TileRanks {
    unsigned long long kk[kSortChunks];
    unsigned int vv[kSortChunks];
    int dig[kSortChunks], rank[kSortChunks];
};

__device__ __forceinline__ void rank_chunk(TileRanks& r, int c, bool ok, int digit, int* cnt,
                                           int lane)
{
    const int d = ok ? digit : kRadix + lane;  // invalid lanes unique
    r.dig[c] = d;
    const unsigned int peers = __match_any_sync(0xffffffffu, d);
    const int leader = __ffs(peers) - 1;
    int before = 0;
    if (ok && lane == leader) {
        before = cnt[d];
        cnt[d] = before + __popc(peers);
    }
    before = __shfl_sync(0xffffffffu, before, leader);
    r.rank[c] = before + __popc(peers & ((1u << lane) - 1u));
    __syncwarp();
}

// Shared memory of a pass: keys of a digit in each warp, and whether a wait gave up.
struct PassShared {
    int cnt[kSortWarps][kRadix];
    int fail;
};

// A tile of one stable LSD pass (decoupled look-back): ranks the tile's keys r stably and
// publishes the per-digit count; the digit offset of the tile is the sum of the counts of
// all earlier tiles, read back through their published words {epoch, flag (1 = count of the
// tile, 2 = inclusive prefix), value}, on top of the digit's first place (thread d: digit
// d's).  A block waits only on earlier tiles, whose blocks are running, and every wait is
// bounded: past spin_limit polls it raises *err and leaves its keys where they are (the host
// reports UCP_ETIMEOUT).  sh.cnt is zero at the start.  kL2: another block of the same launch
// reads what this one writes.
template <bool kL2, class Digit>
__device__ __forceinline__ void place_tile(TileRanks& r, int n, int tile, Digit digit, int first,
                                           unsigned long long* status, unsigned int epoch, int* err,
                                           int spin_limit, PassShared& sh,
                                           unsigned long long* kout, unsigned int* vout)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int base = tile * kSortTile + w * (kSortTile / kSortWarps);
#pragma unroll
    for (int c = 0; c < kSortChunks; ++c) {
        const bool ok = base + c * 32 + lane < n;
        rank_chunk(r, c, ok, ok ? digit(r.kk[c], r.vv[c]) : 0, sh.cnt[w], lane);
    }
    __syncthreads();
    {
        const int d = threadIdx.x;
        int total = 0;
        for (int ww = 0; ww < kSortWarps; ++ww) {
            int t = sh.cnt[ww][d];
            sh.cnt[ww][d] = total;
            total += t;
        }
        const unsigned long long tag = (unsigned long long)epoch << 34;
        unsigned long long* mine = status + (size_t)tile * kRadix + d;
        unsigned int prefix = 0;
        if (tile > 0) {
            atomicExch(mine, tag | (1ull << 32) | (unsigned int)total);
            // kLook predecessors' words per round trip (independent loads), taken in
            // order j, j - 1, ... up to the first inclusive prefix or the first word
            // not yet published, which is polled again
            int j = tile - 1, spins = 0;
            bool done = false;
            while (!done) {
                unsigned long long v[kLook];
#pragma unroll
                for (int u = 0; u < kLook; ++u)
                    v[u] = j - u >= 0 ? __ldcv(status + (size_t)(j - u) * kRadix + d) : 0ull;
                int used = 0;
                bool blocked = false;
#pragma unroll
                for (int u = 0; u < kLook; ++u) {
                    if (done || blocked || j - u < 0) continue;
                    const unsigned int flag = (unsigned int)(v[u] >> 32) & 3u;
                    if ((v[u] >> 34) != (unsigned long long)epoch || flag == 0u) {
                        blocked = true;
                        continue;
                    }
                    prefix += (unsigned int)v[u];
                    ++used;
                    if (flag == 2u) done = true;
                }
                j -= used;
                if (done || j < 0) break;  // (tile 0 publishes an inclusive prefix)
                if (blocked) {
                    if (++spins > spin_limit) {
                        atomicOr(err, 1);
                        sh.fail = 1;
                        break;
                    }
                    __nanosleep(64);
                }
            }
        }
        atomicExch(mine, tag | (2ull << 32) | (prefix + (unsigned int)total));
        const int off = first + (int)prefix;
        for (int ww = 0; ww < kSortWarps; ++ww) sh.cnt[ww][d] += off;
    }
    __syncthreads();
    const bool fail = sh.fail != 0;
#pragma unroll
    for (int c = 0; c < kSortChunks; ++c) {
        const int i = base + c * 32 + lane;
        if (i < n) {
            const int p = fail ? i : sh.cnt[w][r.dig[c]] + r.rank[c];
            if (kL2) {
                __stcg(kout + p, r.kk[c]);
                __stcg(vout + p, r.vv[c]);
            } else {
                kout[p] = r.kk[c];
                vout[p] = r.vv[c];
            }
        }
    }
}

// One pass: a block takes the next tile from a counter.  A digit's first place is the scan of
// the digit counts `digits`, or (scan = 0) `digits` itself, its first ndigits valid.
__global__ void __launch_bounds__(kSortThreads)
k_onesweep(const unsigned long long* __restrict__ kin, const unsigned int* __restrict__ vin,
           unsigned long long* __restrict__ kout, unsigned int* __restrict__ vout, int n,
           int shift, const int* __restrict__ digits, int scan, int ndigits,
           unsigned long long* status, int* tile_ctr, const unsigned int* __restrict__ epoch_dev,
           unsigned int pass, int* err, int spin_limit,
           const unsigned char* __restrict__ digit_of_val)
{
    follow();
    const unsigned int epoch = (*epoch_dev + pass) & 0x3fffffffu;
    __shared__ PassShared sh;
    __shared__ int s_tile, s_tot;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        s_tile = atomicAdd(tile_ctr, 1);
        sh.fail = 0;
    }
    for (int d = lane; d < kRadix; d += 32) sh.cnt[w][d] = 0;
    const int dv = (int)threadIdx.x < ndigits ? digits[threadIdx.x] : 0;  // kSortThreads == kRadix
    __syncthreads();
    const int tile = s_tile;
    const int base = tile * kSortTile + w * (kSortTile / kSortWarps);
    TileRanks r;
#pragma unroll
    for (int c = 0; c < kSortChunks; ++c) {
        const int i = base + c * 32 + lane;
        const bool ok = i < n;
        r.kk[c] = ok ? kin[i] : 0ull;
        r.vv[c] = ok ? (vin ? vin[i] : (unsigned int)i) : 0u;
    }
    const int first = scan ? block_excl_scan(dv, &s_tot) : dv;
    // digit: 8 key bits, or (cloud pass) the cloud of the element's previous slot
    place_tile<false>(r, n, tile,
                      [&](unsigned long long k, unsigned int v) {
                          return digit_of_val ? (int)digit_of_val[v] : (int)((k >> shift) & 0xffu);
                      },
                      first, status, epoch, err, spin_limit, sh, kout, vout);
}

// Orders the runs of equal top digits by (key, caller index) and moves the state.  A
// block owns kFinish places and also sees the kRun places on either side, so that
// every run that touches its places and is no longer than kRun lies in its window;
// neighbouring blocks order a shared run each for itself.  Reads the passes' result,
// writes the sorted keys to another buffer.
constexpr int kFinish = 256;
constexpr int kWindow = kFinish + 2 * kRun;

__global__ void __launch_bounds__(kFinish)
k_finish_sort(const unsigned long long* __restrict__ kin, const unsigned int* __restrict__ vin,
              unsigned long long* __restrict__ kout, int n, int low, StateRef in, StateRef out,
              const unsigned char* __restrict__ cloud, int* __restrict__ long_run)
{
    follow();
    __shared__ unsigned long long sk[kWindow + 1];   // place l - 1 of the window
    __shared__ unsigned int sv[kWindow + 1];
    __shared__ unsigned char sc[kWindow + 1];
    const int base = blockIdx.x * kFinish;
    for (int l = threadIdx.x; l <= kWindow; l += kFinish) {
        const int i = base - kRun - 1 + l;
        const bool ok = i >= 0 && i < n;
        sk[l] = ok ? kin[i] : 0ull;
        sv[l] = ok ? vin[i] : 0u;
        sc[l] = ok && cloud ? cloud[i] : 0;
    }
    __syncthreads();
    // place l of the window continues the run of place l - 1
    auto follows = [&](int l) {
        const int i = base - kRun - 1 + l;
        return i > 0 && i < n && l <= kWindow && (sk[l] >> low) == (sk[l - 1] >> low) &&
               sc[l] == sc[l - 1];
    };
    // the first places of the runs (decided before any run is reordered; the top
    // digits of a place do not change)
    for (int l = 1 + threadIdx.x; l < 1 + kRun + kFinish; l += kFinish) {
        if (follows(l) || !follows(l + 1)) continue;
        int e = l + 1;
        while (e - l <= kRun && follows(e)) ++e;
        if (e - l > kRun) {
            *long_run = 1;
            continue;
        }
        for (int a = l + 1; a < e; ++a) {
            const unsigned long long k = sk[a];
            const unsigned int v = sv[a];
            int b = a - 1;
            while (b >= l && (sk[b] > k || (sk[b] == k && in.id[sv[b]] > in.id[v]))) {
                sk[b + 1] = sk[b];
                sv[b + 1] = sv[b];
                --b;
            }
            sk[b + 1] = k;
            sv[b + 1] = v;
        }
    }
    __syncthreads();
    const int i = base + threadIdx.x;
    if (i < n) {
        const int l = 1 + kRun + threadIdx.x;
        kout[i] = sk[l];
        move_state(in, out, i, sv[l]);
    }
}

// One cloud of up to kBlockSort particles by one block of 32 warps, all in shared
// memory: the same passes over the top digits and the same ordering of runs, or, when a
// run is too long, passes over the caller index and the whole key.  The state is moved by
// the topology's blocks (one SM would take longer for its traffic than for the sort).
// A chain of barriers and shared-memory latencies, about 3 us for every 1024 particles:
// in place of two or three passes of one to four blocks, the run kernel and the empty
// full sort it takes 11.5 for 27 us at N = 2048 and 22 for 40 at 4099 (a build of such a
// cloud 111 -> 96 and 128 -> 112 us, with the extents also by one block); at 6000 a build
// still gains 8 us, at 8192 it would lose 2.
constexpr int kBlockItems = kBlockSort / kBlockThreads;
constexpr int kBlockWarps = kBlockThreads / 32;

struct BlockSortShared {
    unsigned long long key[kBlockSort];
    unsigned short val[kBlockSort];
    int cnt[kBlockWarps][kRadix];    // keys of a digit in warp w before, then its first place
    int part[4][kRadix];             // the same for each eight warps
    int sums[kRadix / 32];
};

__global__ void __launch_bounds__(kBlockThreads)
k_sort_block(const unsigned long long* __restrict__ kin, unsigned long long* __restrict__ kout,
             unsigned int* __restrict__ vout, int n, const unsigned int* __restrict__ id)
{
    follow();
    extern __shared__ __align__(16) unsigned char sort_bytes[];
    BlockSortShared& sh = *reinterpret_cast<BlockSortShared*>(sort_bytes);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int items = (n + kBlockThreads - 1) / kBlockThreads;
    const int first = w * 32 * items + lane;        // a warp owns a contiguous part
    unsigned long long kk[kBlockItems];
    unsigned int vv[kBlockItems];
#pragma unroll
    for (int j = 0; j < kBlockItems; ++j) {
        const int i = first + 32 * j;
        const bool ok = j < items && i < n;
        kk[j] = ok ? kin[i] : 0ull;
        vv[j] = ok ? (unsigned int)i : 0u;
    }
    // one stable pass by digit(key, slot) < kRadix
    auto pass = [&](auto digit) {
        for (int i = threadIdx.x; i < kBlockWarps * kRadix; i += kBlockThreads) (&sh.cnt[0][0])[i] = 0;
        __syncthreads();
        unsigned int place[kBlockItems];            // digit << 16 | rank in the warp
#pragma unroll
        for (int j = 0; j < kBlockItems; ++j) {
            if (j >= items) break;
            const bool ok = first + 32 * j < n;
            const int d = ok ? (int)digit(kk[j], vv[j]) : kRadix + lane;   // invalid lanes unique
            const unsigned int peers = __match_any_sync(0xffffffffu, d);
            const int leader = __ffs(peers) - 1;
            int before = 0;
            if (ok && lane == leader) {
                before = sh.cnt[w][d];
                sh.cnt[w][d] = before + __popc(peers);
            }
            before = __shfl_sync(0xffffffffu, before, leader);
            place[j] = (unsigned int)d << 16 | (unsigned int)(before + __popc(peers & ((1u << lane) - 1u)));
            __syncwarp();
        }
        __syncthreads();
        const int d = threadIdx.x & (kRadix - 1), q = threadIdx.x / kRadix;
        int sum = 0;
#pragma unroll
        for (int k = 0; k < kBlockWarps / 4; ++k) {
            const int c = sh.cnt[q * (kBlockWarps / 4) + k][d];
            sh.cnt[q * (kBlockWarps / 4) + k][d] = sum;
            sum += c;
        }
        sh.part[q][d] = sum;
        __syncthreads();
        int total = 0, upto = 0;
        if (w < kRadix / 32) {
#pragma unroll
            for (int k = 0; k < 4; ++k) total += sh.part[k][d];
            upto = warp_incl_scan(total, lane);
            if (lane == 31) sh.sums[w] = upto;
        }
        __syncthreads();
        if (w < kRadix / 32) {
            int at = upto - total;
            for (int k = 0; k < w; ++k) at += sh.sums[k];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int c = sh.part[k][d];
                sh.part[k][d] = at;
                at += c;
            }
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kBlockItems; ++j) {
            if (j >= items || first + 32 * j >= n) break;
            const int dj = place[j] >> 16;
            const int p = sh.part[w / (kBlockWarps / 4)][dj] + sh.cnt[w][dj] + (int)(place[j] & 0xffffu);
            sh.key[p] = kk[j];
            sh.val[p] = (unsigned short)vv[j];
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kBlockItems; ++j) {
            const int i = first + 32 * j;
            if (j >= items || i >= n) break;
            kk[j] = sh.key[i];
            vv[j] = sh.val[i];
        }
    };
    auto by_key = [&](int shift) {
        pass([&](unsigned long long k, unsigned int) { return (unsigned int)(k >> shift) & 0xffu; });
    };
    constexpr int low = kKeyBits - 16;      // two passes: runs of 4 in the densest part at 6144
    by_key(low);
    by_key(low + 8);
    // each particle's place in its run of equal top digits, by (key, caller index)
    int place[kBlockItems];
    bool too_long = false;
#pragma unroll
    for (int j = 0; j < kBlockItems; ++j) {
        const int i = first + 32 * j;
        place[j] = i;
        if (j >= items || i >= n) break;
        const unsigned long long k = kk[j], top = k >> low;
        int b = i, e = i + 1;
        while (b > 0 && i - b <= kRun && sh.key[b - 1] >> low == top) --b;
        while (e < n && e - b <= kRun && sh.key[e] >> low == top) ++e;
        if (e - b > kRun) {
            too_long = true;
            continue;
        }
        int at = b;
        for (int o = b; o < e; ++o) {
            const unsigned long long ko = sh.key[o];
            at += ko < k || (ko == k && o != i && id[sh.val[o]] < id[vv[j]]);
        }
        place[j] = at;
    }
    if (__syncthreads_or(too_long)) {
        static_assert(kBlockSort <= kRadix * kRadix, "two digits of the caller index");
        pass([&](unsigned long long, unsigned int v) { return id[v] & 0xffu; });
        pass([&](unsigned long long, unsigned int v) { return id[v] >> 8; });
        for (int shift = 0; shift < kKeyBits; shift += 8) by_key(shift);
#pragma unroll
        for (int j = 0; j < kBlockItems; ++j) place[j] = first + 32 * j;
    }
#pragma unroll
    for (int j = 0; j < kBlockItems; ++j) {
        if (j >= items || first + 32 * j >= n) break;
        kout[place[j]] = kk[j];
        vout[place[j]] = vv[j];
    }
}

// The whole key, when a run was too long, by resident blocks that meet at a barrier after
// every pass (a cooperative launch; its waits are bounded).  Every particle goes to the place
// of its caller index first, so that equal keys, however many, come out in that order of the
// stable passes, and all passes' digits are counted on the way; then eight LSD passes (a
// ninth by cloud) as in k_onesweep, a block taking every gridDim-th tile, and the state.
// Returns at once when no run was.  A build with a particle at 100, 1000 and 1e5 sigma takes
// 385, 348 and 342 us at N = 524,288 and 2.58, 2.45 and 2.08 ms at 4,194,304 (204 us and 1.41
// ms without it); with a block per SM, a pass over the keys for each digit's counts and runs
// of equal keys ordered by one thread each it took 433, 391 and 575 us, 3.15, 3.07 and 5.13
// ms, and sorting every key by eight passes in each build 410, 430 and 447 us, 2.27, 2.50
// and 2.33 ms (396 us and 2.42 ms without the particle).
constexpr int kFullPasses = 8;
constexpr int kFullPerSM = 2;        // resident blocks, which the register budget allows

__global__ void __launch_bounds__(kSortThreads, kFullPerSM)
k_sort_full(unsigned long long* k0, unsigned long long* k1, unsigned int* v0, unsigned int* v1,
            int n, int n_clouds, int* ctl, const unsigned int* __restrict__ epoch_dev, int* counts,
            unsigned long long* status, int* err, StateRef in, StateRef out,
            const unsigned char* __restrict__ cloud, const int* __restrict__ cloud_start)
{
    follow();
    if (ctl[kCtlLong] == 0) return;
    __shared__ PassShared sh;
    __shared__ int s_tot;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int stride = gridDim.x * kSortThreads, at = blockIdx.x * kSortThreads + threadIdx.x;
    int met = 0;
    bool lost = false;
    auto barrier = [&]() {
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            atomicAdd(&ctl[kCtlBarrier], 1);
            ++met;
            int spins = 0;
            while (*(volatile int*)&ctl[kCtlBarrier] < met * (int)gridDim.x) {
                if (++spins > (kSortSpinLimit << 3)) {
                    atomicOr(err, 1);
                    break;
                }
                __nanosleep(64);
            }
            __threadfence();
            s_tot = *(volatile int*)err;
        }
        __syncthreads();
        lost = s_tot != 0;
        __syncthreads();
    };
    if (threadIdx.x == 0) sh.fail = 0;
    for (int i = at; i < kFullPasses * kRadix; i += stride) __stcg(counts + i, 0);
    barrier();
    if (lost) return;
    // caller indices are a permutation (after a wait that gave up they may repeat, and leave
    // a place as it was)
    static_assert(kFullPasses == kSortWarps, "sh.cnt holds the counts of every pass");
    for (int d = lane; d < kRadix; d += 32) sh.cnt[w][d] = 0;
    __syncthreads();
    for (int i = at; i < n; i += stride) {
        const unsigned long long k = k0[i];
        const unsigned int v = v0[i], d = in.id[v];
        __stcg(k1 + d, k);
        __stcg(v1 + d, v);
#pragma unroll
        for (int p = 0; p < kFullPasses; ++p) atomicAdd(&sh.cnt[p][(unsigned int)(k >> (8 * p)) & 0xffu], 1);
    }
    __syncthreads();
    for (int p = 0; p < kFullPasses; ++p) {
        const int c = sh.cnt[p][threadIdx.x];
        if (c) atomicAdd(counts + p * kRadix + threadIdx.x, c);
    }
    barrier();
    unsigned long long *ka = k1, *kb = k0;
    unsigned int *va = v1, *vb = v0;
    const int tiles = (n + kSortTile - 1) / kSortTile;
    const int passes = kFullPasses + (n_clouds > 1 ? 1 : 0);
    for (int p = 0; p < passes && !lost; ++p) {
        // tags of their own, after those of the passes over the top digits
        const unsigned int epoch = (*epoch_dev + kSortPassesMax + 1 + p) & 0x3fffffffu;
        const int first = p < kFullPasses
                              ? block_excl_scan(__ldcg(counts + p * kRadix + threadIdx.x), &s_tot)
                              : (int)threadIdx.x < n_clouds ? cloud_start[threadIdx.x] : 0;
        for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
            for (int d = lane; d < kRadix; d += 32) sh.cnt[w][d] = 0;
            const int base = tile * kSortTile + w * (kSortTile / kSortWarps);
            TileRanks r;
#pragma unroll
            for (int c = 0; c < kSortChunks; ++c) {
                const int i = base + c * 32 + lane;
                const bool ok = i < n;
                r.kk[c] = ok ? __ldcg(ka + i) : 0ull;
                r.vv[c] = ok ? __ldcg(va + i) : 0u;
            }
            __syncwarp();
            place_tile<true>(r, n, tile,
                             [&](unsigned long long k, unsigned int v) {
                                 return p == kFullPasses ? (int)cloud[v]
                                                         : (int)((k >> (8 * p)) & 0xffu);
                             },
                             first, status, epoch, err, kSortSpinLimit, sh, kb, vb);
            __syncthreads();
        }
        barrier();
        unsigned long long* tk = ka;
        ka = kb;
        kb = tk;
        unsigned int* tv = va;
        va = vb;
        vb = tv;
    }
    if (lost) return;
    // the sorted keys end in k1 whatever the number of passes
    for (int i = at; i < n; i += stride) {
        if (ka != k1) k1[i] = __ldcg(ka + i);
        move_state(in, out, i, __ldcg(va + i));
    }
}

}  // namespace

// Passes over the top digits: a run of equal digits should stay a few particles where
// the cloud is densest (a Gaussian cloud's centre holds 63 times the mean over its
// cube: 4 particles per cell at 2^12 with two passes and at 2^20 with three).
int sort_passes(int64_t largest_cloud)
{
    return largest_cloud <= (1 << 12) ? 2 : largest_cloud <= (1 << 20) ? 3 : 4;
}

size_t sort_test_words() { return 4 * (size_t)kSortTile; }
size_t sort_full_words() { return (size_t)kFullPasses * kRadix; }

size_t sort_status_words(int n)
{
    int nb = (n + kSortTile - 1) / kSortTile;
    return (size_t)(kSortPassesMax + 1) * kRadix * (size_t)(nb > 0 ? nb : 1);
}

int launch_sort(unsigned long long* key[2], unsigned int* val[2], int n, int passes,
                const SortScratch& sc, BuildCtl ctl, const StateRef& in, const StateRef& out,
                const unsigned char* cloud, const int* cloud_start, int n_clouds, int nsm,
                Queue s)
{
    const bool clouds = n_clouds > 1;
    if (block_sorted(n, n_clouds)) {
        count_launch(1);
        const int bytes = (int)sizeof(BlockSortShared);
        cudaFuncSetAttribute(k_sort_block, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        launch_shared(k_sort_block, 1, kBlockThreads, bytes, s, key[0], key[1], val[1], n,
                      in.id);
        return 1;
    }
    count_launch(passes + 2 + (clouds ? 1 : 0));
    const int nb = (n + kSortTile - 1) / kSortTile;
    const int low = kKeyBits - 8 * passes;
    int cur = 0;
    for (int p = 0; p < passes; ++p) {
        launch(k_onesweep, nb, kSortThreads, s, key[cur],
               p == 0 ? static_cast<unsigned int*>(nullptr) : val[cur], key[cur ^ 1],
               val[cur ^ 1], n, low + 8 * p,
            ctl.words + kCtlHist + p * kRadix, 1, kRadix, sc.status + (size_t)p * nb * kRadix,
            ctl.words + kCtlTile + p, ctl.epoch, (unsigned int)p, sc.err, kSortSpinLimit, nullptr);
        cur ^= 1;
    }
    if (clouds) {
        // a stable pass by cloud: (cloud, key) order, each cloud back in its fixed
        // segment; a cloud's first place is its segment's start
        launch(k_onesweep, nb, kSortThreads, s, key[cur], val[cur], key[cur ^ 1],
               val[cur ^ 1], n, 0, cloud_start, 0, n_clouds,
            sc.status + (size_t)passes * nb * kRadix, ctl.words + kCtlTile + passes, ctl.epoch,
            (unsigned int)passes, sc.err, kSortSpinLimit, cloud);
        cur ^= 1;
    }
    const int fin = cur ^ 1;
    launch(k_finish_sort, (n + kFinish - 1) / kFinish, kFinish, s, key[cur], val[cur],
           key[fin], n, low, in, out, cloud, ctl.words + kCtlLong);
    unsigned long long *k0 = key[cur], *k1 = key[fin], *status = sc.status;
    unsigned int *v0 = val[cur], *v1 = val[fin], *epoch = ctl.epoch;
    int* words = ctl.words;
    int *counts = sc.full_counts, *err = sc.err;
    StateRef si = in, so = out;
    void* args[] = {&k0, &k1, &v0, &v1, &n, &n_clouds, &words, &epoch, &counts,
                    &status, &err, &si, &so, &cloud, &cloud_start};
    const int blocks = nb < kFullPerSM * nsm ? nb : kFullPerSM * nsm;
    cudaLaunchCooperativeKernel(reinterpret_cast<void*>(k_sort_full), dim3(blocks),
                                dim3(kSortThreads), args, 0, s);
    return fin;
}

int sort_selftest_timeout(const SortScratch& sc, Queue s)
{
    // a lone block that takes tile 1 while tile 0 never publishes: its bounded
    // wait must run out, raise *err and leave the keys where they are
    count_launch(1);
    static const int one = 1;
    if (cudaMemsetAsync(sc.status, 0, sizeof(unsigned long long) * 2 * kRadix, s) != cudaSuccess ||
        cudaMemsetAsync(sc.test_ctl, 0, sizeof(int) * (1 + kRadix), s) != cudaSuccess ||
        cudaMemcpyAsync(sc.test_ctl, &one, sizeof(int), cudaMemcpyHostToDevice, s) != cudaSuccess ||
        cudaMemcpyAsync(sc.test_epoch, &one, sizeof(int), cudaMemcpyHostToDevice, s) != cudaSuccess ||
        cudaMemsetAsync(sc.test_keys, 0, sizeof(unsigned long long) * 4 * kSortTile, s) != cudaSuccess ||
        cudaMemsetAsync(sc.test_vals, 0, sizeof(unsigned int) * 4 * kSortTile, s) != cudaSuccess)
        return -1;
    // input: tiles 0-1 of the test buffers; output: tiles 2-3
    launch(k_onesweep, 1, kSortThreads, s, sc.test_keys, sc.test_vals, sc.test_keys + 2 * kSortTile,
                                          sc.test_vals + 2 * kSortTile, 2 * kSortTile, 0,
                                          sc.test_ctl + 1, 1, kRadix, sc.status, sc.test_ctl,
                                          sc.test_epoch, 0u, sc.err, 2000, nullptr);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// ---- target selection: the slots whose species is `species`, in slot order
namespace {

constexpr int kSelThreads = 1024;
constexpr int kSelItems = 4;
constexpr int kSelTile = kSelThreads * kSelItems;

__global__ void __launch_bounds__(kSelThreads)
k_select_count(const int8_t* __restrict__ sp, int species, int n, int* __restrict__ part)
{
    follow();
    const int base = blockIdx.x * kSelTile;
    int s = 0;
#pragma unroll
    for (int k = 0; k < kSelItems; ++k) {
        const int i = base + threadIdx.x * kSelItems + k;
        if (i < n) s += sp[i] == species;
    }
    __shared__ int tot;
    block_excl_scan(s, &tot);
    if (threadIdx.x == 0) part[blockIdx.x] = tot;
}

// Every block sums the counts of the tiles before its own; the interaction counts of
// every slot (if given) are cleared on the way (the walk writes those of its targets).
__global__ void __launch_bounds__(kSelThreads)
k_select_write(const int8_t* __restrict__ sp, int species, int n, const int* __restrict__ part,
               int* __restrict__ list, int* __restrict__ cnt0, int* __restrict__ cnt1)
{
    follow();
    __shared__ int tot, before;
    int b = 0;
    for (int i = threadIdx.x; i < (int)blockIdx.x; i += kSelThreads) b += part[i];
    block_excl_scan(b, &before);
    const int base = blockIdx.x * kSelTile;
    int v[kSelItems];
    int s = 0;
#pragma unroll
    for (int k = 0; k < kSelItems; ++k) {
        const int i = base + threadIdx.x * kSelItems + k;
        v[k] = i < n && sp[i] == species;
        s += v[k];
        if (i < n && cnt0) {
            cnt0[i] = 0;
            cnt1[i] = 0;
        }
    }
    int off = block_excl_scan(s, &tot) + before;
#pragma unroll
    for (int k = 0; k < kSelItems; ++k) {
        const int i = base + threadIdx.x * kSelItems + k;
        if (v[k]) list[off++] = i;
    }
}

}  // namespace

size_t select_words(int n) { return (size_t)((n + kSelTile - 1) / kSelTile) + 1; }

void launch_select(const int8_t* sp, int species, int n, int* list, int* partials, int* cnt0,
                   int* cnt1, Queue s)
{
    count_launch(2);
    const int nb = (n + kSelTile - 1) / kSelTile;
    launch(k_select_count, nb, kSelThreads, s, sp, species, n, partials);
    launch(k_select_write, nb, kSelThreads, s, sp, species, n, partials, list, cnt0, cnt1);
}

}  // namespace ucp
