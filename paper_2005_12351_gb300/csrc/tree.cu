// tree.cu -- octree and interaction lists on the GPU (paper §3.2).
//
// Root box: lo = per-axis minimum; side = the smallest power of two not below
// the largest extent.  Integer coordinates q = min(floor((x - lo) * 2^21 /
// side), 2^21 - 1) are interleaved (x highest) into 63-bit Morton keys and
// sorted stably.  Cells are built breadth-first: a cell splits while it holds
// more than n_crit particles and its level is below 21; empty octants are
// not created, so cells come out in (level, Morton prefix) order.
//
// Lists come from the dual-tree traversal of §3.2 run as a breadth-first
// frontier of cell pairs.  MAC (Eq. (13)) with r = half the cell side,
// evaluated exactly in integer units of the finest half-cell; when it fails:
// two leaves -> P2P, one leaf -> open the other, else open the larger cell
// (the target on a tie); a self pair opens into all ordered child pairs.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "fmm_internal.cuh"

namespace fmm {

namespace {

__device__ __forceinline__ unsigned long long ordered_bits(double x)
{
    unsigned long long b = (unsigned long long)__double_as_longlong(x);
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__device__ __forceinline__ double from_ordered_bits(unsigned long long b)
{
    b = (b >> 63) ? (b & 0x7fffffffffffffffull) : ~b;
    return __longlong_as_double((long long)b);
}

// the running box and the head words of the sort's scratch, one block
__global__ void k_sort_init(unsigned long long *box, uint32_t *hist)
{
    const int i = threadIdx.x;
    if (i < 3) box[i] = ~0ull;            // running minimum
    else if (i < 6) box[i] = 0ull;        // running maximum
    for (int w = i; w < kRadixHead; w += blockDim.x) hist[w] = 0u;
}

__global__ void k_bbox(const double *pos, int64_t n, unsigned long long *box, int *err)
{
    pdl_wait();
    unsigned long long mn[3] = {~0ull, ~0ull, ~0ull}, mx[3] = {0ull, 0ull, 0ull};
    bool bad = false;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            double x = pos[3 * i + d];
            if (!isfinite(x)) bad = true;
            unsigned long long b = ordered_bits(x);
            mn[d] = b < mn[d] ? b : mn[d];
            mx[d] = b > mx[d] ? b : mx[d];
        }
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            unsigned long long a = __shfl_xor_sync(0xffffffffu, mn[d], o);
            unsigned long long b = __shfl_xor_sync(0xffffffffu, mx[d], o);
            mn[d] = a < mn[d] ? a : mn[d];
            mx[d] = b > mx[d] ? b : mx[d];
        }
    }
    // the block's warps through shared memory, then six atomics per block
    __shared__ unsigned long long s_mm[6][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (lane == 0) {
#pragma unroll
        for (int d = 0; d < 3; ++d) { s_mm[d][warp] = mn[d]; s_mm[3 + d][warp] = mx[d]; }
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        const int d = threadIdx.x;
        unsigned long long v = s_mm[d][0];
        for (int w = 1; w < nw; ++w) v = d < 3 ? (s_mm[d][w] < v ? s_mm[d][w] : v) : (s_mm[d][w] > v ? s_mm[d][w] : v);
        if (d < 3) atomicMin(&box[d], v); else atomicMax(&box[d], v);
    }
    if (bad) atomicOr(err, kErrNonFinite);
}

// (lo_x, lo_y, lo_z, side) of the ordered bits of the minima and maxima
__device__ __forceinline__ void box_final(const unsigned long long *box, double *out)
{
    double lo[3], ext = 0.0;
    for (int d = 0; d < 3; ++d) {
        lo[d] = from_ordered_bits(box[d]);
        double e = __dsub_rn(from_ordered_bits(box[3 + d]), lo[d]);
        ext = e > ext ? e : ext;
    }
    double side = 1.0;
    if (ext > 0.0 && isfinite(ext)) {
        int e2;
        double m = frexp(ext, &e2);        // ext = m 2^e2, m in [0.5, 1)
        side = ldexp(1.0, m == 0.5 ? e2 - 1 : e2);
    }
    out[0] = lo[0]; out[1] = lo[1]; out[2] = lo[2]; out[3] = side;
}

__device__ __forceinline__ uint64_t spread3(uint64_t x)
{
    x &= 0x1fffffull;
    x = (x | x << 32) & 0x1f00000000ffffull;
    x = (x | x << 16) & 0x1f0000ff0000ffull;
    x = (x | x << 8) & 0x100f00f00f00f00full;
    x = (x | x << 4) & 0x10c30c30c30c30c3ull;
    x = (x | x << 2) & 0x1249249249249249ull;
    return x;
}

// floor(d 2^k) for a double d >= 0 and 2^k a power of two, clamped to the
// grid (the product is exact, so this is floor((x - lo) scale) of the
// definition), from d's bits: one FP64 operation per coordinate, the rest
// integer arithmetic.
__device__ __forceinline__ uint64_t grid_coord(double d, int k)
{
    const uint64_t b = (uint64_t)__double_as_longlong(d);
    const int ef = (int)((b >> 52) & 0x7ff);
    // d = m 2^(e - 1075), subnormals with e = 1 and no implicit bit
    const uint64_t m = (b & ((1ull << 52) - 1)) | (ef ? (1ull << 52) : 0ull);
    const int sh = (ef ? ef : 1) - 1075 + k;        // d 2^k = m 2^sh
    const uint64_t top = (uint64_t)((1 << kLevels) - 1);
    if (sh >= 0) return sh > 11 ? top : ((m << sh) > top ? top : (m << sh));
    return sh <= -64 ? 0 : ((m >> -sh) > top ? top : (m >> -sh));
}

// The keys, and for the radix sort that follows the counts of the 8-bit digits
// p0 .. 7 of them (per block in shared memory, then one atomic per digit and
// block) and the zeroed status words of its first pass.  Every block forms the
// box from its six words (the first one stores it), which saves a launch.
__global__ void __launch_bounds__(256)
k_keys(const double *pos, int64_t n, const unsigned long long *raw_box, double *box_out, uint64_t *keys,
       uint32_t *idx, int p0, uint32_t *ghist, uint64_t *status0, int64_t nstatus)
{
    pdl_wait();
    __shared__ uint32_t h[kRadixMaxPasses][256];
    __shared__ double box[4];
    for (int p = p0; p < kRadixMaxPasses; ++p) h[p][threadIdx.x] = 0;
    for (int64_t w = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; w < nstatus;
         w += (int64_t)gridDim.x * blockDim.x)
        status0[w] = 0ull;
    if (threadIdx.x == 0) box_final(raw_box, box);
    __syncthreads();
    if (blockIdx.x == 0 && threadIdx.x < 4) box_out[threadIdx.x] = box[threadIdx.x];
    const int k = kLevels - ilogb(box[3]);          // scale = 2^kLevels / side = 2^k
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        uint64_t q[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) q[d] = grid_coord(__dsub_rn(pos[3 * i + d], box[d]), k);
        const uint64_t key = spread3(q[0]) << 2 | spread3(q[1]) << 1 | spread3(q[2]);
        keys[i] = key;
        idx[i] = (uint32_t)i;
        for (int p = p0; p < kRadixMaxPasses; ++p) atomicAdd(&h[p][(unsigned)(key >> (8 * p)) & 255u], 1u);
    }
    __syncthreads();
    for (int p = p0; p < kRadixMaxPasses; ++p)
        if (h[p][threadIdx.x]) atomicAdd(&ghist[p * 256 + threadIdx.x], h[p][threadIdx.x]);
}

// The first radix pass of a set of n Morton keys.  Sorting by the leading bits
// alone leaves runs of equal leading bits, which k_tie_sort puts in order; at
// these depths (23 bits up to 2^14 points, 31 up to 2^22, 39 up to 2^30) a
// uniform set has hardly any and the core of a Plummer sphere of scale radius
// a twentieth of the box some four points to a run.  Each pass saved is a
// launch and 24 bytes a key: 8 -> 4 passes and the tie sort, 0.230 -> 0.130 ms
// at 1M points, 0.072 -> 0.037 ms at 2,000.
inline int first_pass(int64_t n) { return n <= (1 << 14) ? 5 : (n <= (1 << 22) ? 4 : (n <= (1 << 30) ? 3 : 2)); }

// Keys in order of their bits from `shift` up -> keys in order, stable: within
// a run of equal leading bits an element goes behind the smaller keys and the
// equal ones before it.  A run of more than kTieRun keys stays as it is (each
// of its elements sees at least kTieRun neighbours, so they agree) and sets
// kErrTieRun: the caller sorts by all bits instead.  GATHER: the particle
// arrays in the new order too.
constexpr int kTieRun = 256;

// The elements of the run of `top` next to element i on one side, at most
// kTieRun: one by one up to kTieNear, then by doubling and halving steps (the run
// is contiguous).  move: of the first kTieNear, those out of order with `key`.
constexpr int kTieNear = 8;
template <int DIR>
__device__ __forceinline__ int run_reach(const uint64_t *keys, int64_t i, int64_t n, int shift, uint64_t key, int &move)
{
    auto at = [&](int q, uint64_t &o) {
        const int64_t j = i + DIR * q;
        if (DIR < 0 ? j < 0 : j >= n) return false;
        o = keys[j];
        return o >> shift == key >> shift;
    };
    uint64_t o;
    int lo = 0;
    for (; lo < kTieNear && at(lo + 1, o); ++lo) move += DIR < 0 ? -(int)(o > key) : (int)(o < key);
    if (lo < kTieNear) return lo;
    int hi = 2 * kTieNear;                  // lo is in the run
    while (hi <= kTieRun && at(hi, o)) {
        lo = hi;
        hi *= 2;
    }
    hi = min(hi, kTieRun + 1);              // hi is not, or does not matter
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (at(mid, o)) lo = mid; else hi = mid;
    }
    return lo;
}

template <bool GATHER>
__global__ void __launch_bounds__(256)
k_tie_sort(const uint64_t *keys, const uint32_t *idx, int64_t n, int shift, uint64_t *okeys, uint32_t *oidx, int *err,
           const double *pos, const double *mom, int nS, double *px, double *py, double *pz, double *S,
           int32_t *perm_out)
{
    pdl_wait();
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint64_t key = keys[i];
    const uint32_t id = idx[i];
    int move = 0;
    const int left = run_reach<-1>(keys, i, n, shift, key, move), right = run_reach<1>(keys, i, n, shift, key, move);
    if (left + right + 1 > kTieRun) {
        move = 0;
        if ((*(volatile int *)err & kErrTieRun) == 0) atomicOr(err, kErrTieRun);
    } else {
#pragma unroll 4
        for (int q = kTieNear + 1; q <= left; ++q) move -= keys[i - q] > key;
#pragma unroll 4
        for (int q = kTieNear + 1; q <= right; ++q) move += keys[i + q] < key;
    }
    const int64_t k = i + move;
    okeys[k] = key;
    oidx[k] = id;
    if (GATHER) {
        const int64_t o = id;
        px[k] = pos[3 * o];
        py[k] = pos[3 * o + 1];
        pz[k] = pos[3 * o + 2];
        for (int a = 0; a < nS; ++a) S[k * nS + a] = mom[o * nS + a];
        perm_out[k] = (int32_t)o;
    }
}

__global__ void k_sys_of(const int64_t *off, int nsys, int64_t n, int32_t *sys_of)
{
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    int lo = 0, hi = nsys - 1;                 // last system whose start is <= i
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (off[mid] <= i) lo = mid; else hi = mid - 1;
    }
    sys_of[i] = lo;
}

__global__ void k_box_init_seg(unsigned long long *box, int nsys)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 6 * nsys) return;
    box[i] = (i % 6) < 3 ? ~0ull : 0ull;
}

// Per-system min/max.  A warp whose particles all belong to one system
// reduces with shuffles first; mixed warps fall back to per-lane atomics.
__global__ void k_bbox_seg(const double *pos, int64_t n, const int32_t *sys_of,
                           unsigned long long *box, int *err)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const bool valid = i < n;
    const int s = valid ? sys_of[i] : -1;
    unsigned long long mn[3] = {~0ull, ~0ull, ~0ull}, mx[3] = {0ull, 0ull, 0ull};
    bool bad = false;
    if (valid) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const double x = pos[3 * i + d];
            if (!isfinite(x)) bad = true;
            mn[d] = mx[d] = ordered_bits(x);
        }
    }
    const int s0 = __shfl_sync(0xffffffffu, s, 0);
    const bool uniform = __all_sync(0xffffffffu, s == s0);
    if (uniform) {
#pragma unroll
        for (int d = 0; d < 3; ++d)
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                unsigned long long a = __shfl_xor_sync(0xffffffffu, mn[d], o);
                unsigned long long b = __shfl_xor_sync(0xffffffffu, mx[d], o);
                mn[d] = a < mn[d] ? a : mn[d];
                mx[d] = b > mx[d] ? b : mx[d];
            }
        if ((threadIdx.x & 31) == 0 && s0 >= 0)
            for (int d = 0; d < 3; ++d) {
                atomicMin(&box[6 * s0 + d], mn[d]);
                atomicMax(&box[6 * s0 + 3 + d], mx[d]);
            }
    } else if (valid) {
        for (int d = 0; d < 3; ++d) {
            atomicMin(&box[6 * s + d], mn[d]);
            atomicMax(&box[6 * s + 3 + d], mx[d]);
        }
    }
    if (bad) atomicOr(err, kErrNonFinite);
}

// box_out[4 s .. 4 s + 3] = (lo_x, lo_y, lo_z, side) of system s; empty systems get side 1
__global__ void k_box_final_seg(const unsigned long long *box, int nsys, double *box_out)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= nsys) return;
    const unsigned long long *b = box + 6 * s;
    if (b[0] == ~0ull) {                       // no particles
        box_out[4 * s] = box_out[4 * s + 1] = box_out[4 * s + 2] = 0.0;
        box_out[4 * s + 3] = 1.0;
        return;
    }
    double lo[3], ext = 0.0;
    for (int d = 0; d < 3; ++d) {
        lo[d] = from_ordered_bits(b[d]);
        const double e = __dsub_rn(from_ordered_bits(b[3 + d]), lo[d]);
        ext = e > ext ? e : ext;
    }
    double side = 1.0;
    if (ext > 0.0 && isfinite(ext)) {
        int e2;
        const double m = frexp(ext, &e2);
        side = ldexp(1.0, m == 0.5 ? e2 - 1 : e2);
    }
    box_out[4 * s] = lo[0]; box_out[4 * s + 1] = lo[1]; box_out[4 * s + 2] = lo[2];
    box_out[4 * s + 3] = side;
}

__global__ void k_keys_seg(const double *pos, int64_t n, const int32_t *sys_of,
                           const double *box, uint64_t *keys, uint32_t *idx)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double *bx = box + 4 * sys_of[i];
    const double scale = ldexp(1.0, kLevels) / bx[3];
    uint64_t q[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        double u = floor(__dmul_rn(__dsub_rn(pos[3 * i + d], bx[d]), scale));
        uint64_t v = (uint64_t)u;
        q[d] = v > (uint64_t)((1 << kLevels) - 1) ? (uint64_t)((1 << kLevels) - 1) : v;
    }
    keys[i] = spread3(q[0]) << 2 | spread3(q[1]) << 1 | spread3(q[2]);
    idx[i] = (uint32_t)i;
}

// after the key sort: secondary key = system of each element, and a copy of
// the sorted keys by original index for the final re-gather
__global__ void k_sys_keys(const uint64_t *keys, const uint32_t *idx, const int32_t *sys_of,
                           int64_t n, uint64_t *skeys, uint64_t *key_of)
{
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= n) return;
    skeys[k] = (uint64_t)sys_of[idx[k]];
    key_of[idx[k]] = keys[k];
}

__global__ void k_regather_keys(const uint64_t *key_of, const uint32_t *idx, int64_t n,
                                uint64_t *keys)
{
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k < n) keys[k] = key_of[idx[k]];
}

// keys (or NULL): sorted; a run of more than kTieRun equal ones from bit `shift` up sets kErrLongTies
__global__ void k_gather(const double *pos, const double *mom, int nS, const uint32_t *perm,
                         int64_t n, double *px, double *py, double *pz, double *S, int32_t *perm_out,
                         const uint64_t *keys, int shift, int *err)
{
    pdl_wait();
    int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= n) return;
    if (keys && k + kTieRun < n && keys[k] >> shift == keys[k + kTieRun] >> shift &&
        (*(volatile int *)err & kErrLongTies) == 0)
        atomicOr(err, kErrLongTies);
    const int64_t o = perm[k];
    px[k] = pos[3 * o];
    py[k] = pos[3 * o + 1];
    pz[k] = pos[3 * o + 2];
    for (int a = 0; a < nS; ++a) S[k * nS + a] = mom[o * nS + a];
    perm_out[k] = (int32_t)o;
}

struct CellArrays {
    int32_t *level, *parent, *child, *nchild, *begin, *end, *cx, *cy, *cz, *sys;
};

// the traversal's start: counters and row counts zero, one (root, root) pair per system
__global__ void k_list_init(unsigned *cnt, int ncnt, unsigned *rows, int64_t nrows, int2 *front, int nsys, int nf0)
{
    pdl_wait();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x, i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    for (int64_t i = i0; i < ncnt; i += stride) cnt[i] = i == nf0 ? (unsigned)nsys : 0u;
    for (int64_t i = i0; i < nrows; i += stride) rows[i] = 0u;
    for (int64_t i = i0; i < nsys; i += stride) front[i] = make_int2((int)i, (int)i);
}

__device__ __forceinline__ int digit_at(uint64_t key, int level)
{
    return (int)((key >> (3 * (kLevels - level))) & 7ull);
}

// ---- cells, all levels in one launch by one thread-block cluster.
// A level's cells need the level above and a scan of its child counts: three
// small launches a level, or one cluster barrier and a few block barriers.  A
// cluster of eight blocks is co-scheduled, so its barriers need no host and no
// bounded waits; eight SMs are enough for the work (a binary search per cell
// and octant) of a level that is a chain of memory latencies whatever the width.
// Cells phase, before (26 launches, two host syncs) and now: 0.165 -> 0.054 ms at 2,000 points,
// 0.22 -> 0.12 ms at 1M, 0.43 -> 0.34 ms at 4M.
// A level of more than kWideLevel cells ends it: from there on two launches a
// level over the whole chip (k_wide_count, k_wide_write).  Such trees took longer
// in the cluster than in three launches a level, now less than either: 4M points,
// leaves of 4 (2.5M cells) 1.13 and 2.37, now 0.59 ms; leaves of 16 (1.0M) 0.54 and
// 0.89, now 0.44; 1M points, leaves of 8 (318k) 0.30, 0.32, 0.31.
//
// ctl: [0] overflow (more cells than cap), [1 + l] first cell of level l, then
// the leaf count, the error word, the tie flag (a run the tie sort left: no
// cells, the host sorts again), one more than the level where the whole chip
// takes over (0: none), the particles of the longest leaf past n_crit (deepest
// level), and the first system's box as four doubles; behind the words that go to
// the host the blocks' totals, and per level the leaves and the cells with children
// before it.
constexpr int kCtlOverflow = 0, kCtlLevel = 1, kCtlLeaves = 26, kCtlErr = 27, kCtlTie = 28, kCtlWide = 29,
              kCtlLong = 30, kCtlBox = 32, kCtlHost = 40, kCtlTot = 40, kCtlBefore = 40 + 4 * 16,
              kCtlWords = kCtlBefore + 2 * (kLevels + 2);             // words [0, kCtlHost) go to the host
constexpr int kCellBlocks = 8, kCellThreads = 1024;
constexpr int kWideLevel = 1 << 16;

__device__ __forceinline__ void cluster_sync_all()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// first index in [L, R) whose octant at this level is >= o
__device__ __forceinline__ int first_digit_ge(const uint64_t *keys, int L, int R, int level, int o)
{
    while (L < R) {
        const int mid = (L + R) >> 1;
        if (digit_at(keys[mid], level) < o) L = mid + 1; else R = mid;
    }
    return L;
}

// The same by the four lanes of a group (g = lane / 4), four probes a step.
__device__ __forceinline__ int first_digit_ge4(const uint64_t *keys, int L, int R, int level, int o, int lane)
{
    const int q = lane & 3;
    const unsigned gm = 0xfu << (lane & ~3);
    while (R - L > 4) {
        const int len = R - L;
        const bool lt = digit_at(keys[L + (int)(((int64_t)(q + 1) * len) / 5)], level) < o;
        const int k = __popc(__ballot_sync(gm, lt) & gm);
        const int nL = k > 0 ? L + (int)(((int64_t)k * len) / 5) + 1 : L;
        const int nR = k < 4 ? L + (int)(((int64_t)(k + 1) * len) / 5) : R;
        L = nL;
        R = nR;
    }
    const bool lt = q < R - L && digit_at(keys[L + q], level) < o;
    return L + __popc(__ballot_sync(gm, lt) & gm);
}

// Exclusive prefix of v over the block's threads; *total = the block's sum.
__device__ __forceinline__ unsigned cells_scan(unsigned v, unsigned *wsum, unsigned *total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[warp] = x;
    __syncthreads();
    const unsigned w = wsum[lane];                 // kCellThreads / 32 = 32 warps
    unsigned s = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, s, o);
        if (lane >= o) s += y;
    }
    *total = __shfl_sync(0xffffffffu, s, 31);
    const unsigned before = __shfl_sync(0xffffffffu, s - w, warp);
    __syncthreads();                               // wsum is free again
    return before + x - v;
}

// Each block takes a contiguous part of the level's cells.  It lists the cells
// to split (a thread per cell), finds their octants' first particles (eight
// lanes per cell, or a warp with four lanes to a search while there are few)
// and counts their children; the blocks' totals meet over the cluster barrier;
// then the children are written, and each cell's rank among the leaves or
// among the cells with children.  c.nchild holds a split cell's children
// before it until its children are written.
__global__ void __cluster_dims__(kCellBlocks, 1, 1) __launch_bounds__(kCellThreads)
k_cells(CellArrays c, const int64_t *off, int nsys, const double *box, const int *err, int ncrit,
        const uint64_t *keys, int64_t cap, int32_t *cb, int32_t *ce, uint32_t *list, uint32_t *rank,
        unsigned *ctl)
{
    __shared__ unsigned s_w[kCellThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = kCellThreads / 32;
    const int blk = blockIdx.x;
    const unsigned e = *(volatile const int *)err;
    const bool tie = (e & kErrTieRun) != 0;
    for (int s = blk * kCellThreads + tid; s < nsys; s += kCellBlocks * kCellThreads) {
        c.level[s] = 0; c.parent[s] = -1; c.begin[s] = (int32_t)off[s]; c.end[s] = (int32_t)off[s + 1];
        c.cx[s] = c.cy[s] = c.cz[s] = 0;
        c.sys[s] = s;
    }
    if (blk == 0 && tid == 0) ctl[kCtlLong] = 0u;
    cluster_sync_all();
    int lb = 0, le = tie ? 0 : nsys;
    unsigned leaves = 0, inner = 0;            // before this level
    bool over = (int64_t)le > cap;
    int level = 0;
    for (; level <= kLevels && le > lb && le - lb <= kWideLevel && !over; ++level) {
        const int ncl = le - lb;
        const int chunk = (ncl + kCellBlocks - 1) / kCellBlocks;
        const int i0 = min(ncl, blk * chunk), i1 = min(ncl, i0 + chunk);
        uint32_t *mylist = list + i0;
        // the cells to split
        unsigned np = 0;
        for (int base = i0; base < i1; base += kCellThreads) {
            const int i = base + tid;
            const bool split = i < i1 && level < kLevels &&
                               __ldcg(c.end + lb + i) - __ldcg(c.begin + lb + i) > ncrit;
            unsigned tot;
            const unsigned k = np + cells_scan(split, s_w, &tot);
            if (i < i1) rank[lb + i] = k;                      // cells to split before it
            if (split) mylist[k] = (uint32_t)(lb + i);
            np += tot;
        }
        __syncthreads();
        // their octants
        const bool wide = np <= (unsigned)nw;                  // a warp per cell
        const int per = wide ? nw : kCellThreads / 8;
        unsigned nch = 0;
        for (unsigned base = 0; base < np; base += per) {
            const unsigned k = base + (wide ? warp : tid >> 3);
            const int o = lane & 7;
            int lo_i = 0, hi_i = 0, cell = 0;
            if (k < np) {                                      // uniform in a warp (8 lanes) that shares a cell
                cell = (int)mylist[k];
                const int b = __ldcg(c.begin + cell), en = __ldcg(c.end + cell);
                if (wide) {
                    const int g = lane >> 2;                   // the first particle of octant g
                    const int bnd = g ? first_digit_ge4(keys, b, en, level + 1, g, lane) : b;
                    lo_i = __shfl_sync(0xffffffffu, bnd, 4 * o);
                    hi_i = __shfl_sync(0xffffffffu, bnd, (4 * o + 4) & 31);
                } else {
                    lo_i = o ? first_digit_ge(keys, b, en, level + 1, o) : b;
                    hi_i = __shfl_down_sync(0xffu << (lane & ~7), lo_i, 1, 8);
                }
                if (o == 7) hi_i = en;
            }
            const bool flag = hi_i > lo_i && (!wide || lane < 8);
            const unsigned m = (__ballot_sync(0xffffffffu, flag) >> (lane & ~7)) & 0xffu;
            const bool first = k < np && o == 0 && (!wide || lane == 0);
            unsigned tot;
            const unsigned before = nch + cells_scan(first ? __popc(m) : 0u, s_w, &tot);
            if (k < np && (!wide || lane < 8)) {
                const int64_t at = 8 * ((int64_t)i0 + k) + o;
                cb[at] = lo_i;
                ce[at] = hi_i;
            }
            if (first) c.nchild[cell] = (int)before;
            nch += tot;
        }
        unsigned *tot = ctl + kCtlTot + (level & 1) * 2 * kCellBlocks;
        if (tid == 0) { __stcg(tot + 2 * blk, nch); __stcg(tot + 2 * blk + 1, np); }
        cluster_sync_all();
        unsigned c0 = 0, p0 = 0, ca = 0, pa = 0;
        for (int k = 0; k < kCellBlocks; ++k) {
            const unsigned x = __ldcg(tot + 2 * k), y = __ldcg(tot + 2 * k + 1);
            if (k < blk) { c0 += x; p0 += y; }
            ca += x;
            pa += y;
        }
        over = (int64_t)le + ca > cap;
        if (!over) {
            for (unsigned t = tid; t < 8 * np; t += kCellThreads) {      // eight lanes per split cell
                const unsigned k = t >> 3;
                const int o = (int)(t & 7), cell = (int)mylist[k];
                const int64_t at = 8 * ((int64_t)i0 + k) + o;
                const int beg = cb[at], en = ce[at];
                const unsigned gm = 0xffu << (lane & ~7);
                const unsigned m = (__ballot_sync(gm, en > beg) >> (lane & ~7)) & 0xffu;
                const int ch0 = le + (int)(c0 + (unsigned)c.nchild[cell]);
                __syncwarp(gm);                                // every lane has read the count before the cell
                if (o == 0) {
                    c.nchild[cell] = __popc(m);
                    c.child[cell] = ch0;
                    rank[cell] = inner + p0 + k;
                }
                if (en > beg) {
                    const int ch = ch0 + __popc(m & ((1u << o) - 1u));
                    c.level[ch] = level + 1;
                    c.parent[ch] = cell;
                    c.begin[ch] = beg;
                    c.end[ch] = en;
                    c.cx[ch] = 2 * __ldcg(c.cx + cell) + ((o >> 2) & 1);
                    c.cy[ch] = 2 * __ldcg(c.cy + cell) + ((o >> 1) & 1);
                    c.cz[ch] = 2 * __ldcg(c.cz + cell) + (o & 1);
                    c.sys[ch] = __ldcg(c.sys + cell);
                }
            }
            for (int i = i0 + tid; i < i1; i += kCellThreads) {
                const int cell = lb + i, held = __ldcg(c.end + cell) - __ldcg(c.begin + cell);
                if (held > ncrit) {
                    if (level < kLevels) continue;
                    atomicMax(ctl + kCtlLong, (unsigned)held);
                }
                c.nchild[cell] = 0;
                c.child[cell] = -1;
                rank[cell] = leaves + (unsigned)i - (p0 + rank[cell]);
            }
        }
        if (blk == 0 && tid == 0) ctl[kCtlLevel + level] = (unsigned)lb;
        leaves += (unsigned)ncl - pa;
        inner += pa;
        lb = le;
        le += (int)ca;
        cluster_sync_all();
    }
    const bool wide_next = level <= kLevels && le > lb && !over;       // levels are left
    if (blk == 0) {
        for (int l = level + tid; l <= kLevels + 2; l += kCellThreads)
            ctl[kCtlLevel + l] = (unsigned)(wide_next && l > level ? le : lb);
        if (tid == 0) {
            ctl[kCtlWide] = wide_next ? (unsigned)level + 1u : 0u;
            if (wide_next) {
                ctl[kCtlBefore + 2 * level] = leaves;
                ctl[kCtlBefore + 2 * level + 1] = inner;
            }
            ctl[kCtlOverflow] = over;
            ctl[kCtlLeaves] = leaves;
            ctl[kCtlErr] = e;
            ctl[kCtlTie] = tie;
        }
        if (tid < 4) ((double *)(ctl + kCtlBox))[tid] = box[tid];
    }
}

// ---- the cells of one wide level, part of it per block (the same part in both kernels).
constexpr int kWideThreads = 256, kWideBlocksPerSM = 8;
struct WidePart {
    int lb, ncl, i0, i1;                     // the level's first cell and cells; the block's part
};
__device__ __forceinline__ WidePart wide_part(const unsigned *ctl, int level)
{
    WidePart w;
    w.lb = (int)ctl[kCtlLevel + level];
    w.ncl = (int)ctl[kCtlLevel + level + 1] - w.lb;
    const int chunk = (w.ncl + (int)gridDim.x - 1) / (int)gridDim.x;
    w.i0 = min(w.ncl, (int)blockIdx.x * chunk);
    w.i1 = min(w.ncl, w.i0 + chunk);
    return w;
}

// Children of every cell of the level (0 for a leaf) into c.nchild, the
// octants' particle ranges of cell lb + i at cb, ce [8 i + o], and the block's
// children and split cells into tot.  Eight lanes a cell.
__global__ void __launch_bounds__(kWideThreads)
k_wide_count(CellArrays c, int level, int ncrit, const uint64_t *keys, int32_t *cb, int32_t *ce, uint32_t *tot,
             unsigned *ctl)
{
    pdl_wait();
    __shared__ unsigned s_ch[kWideThreads / 32], s_sp[kWideThreads / 32];
    const WidePart p = wide_part(ctl, level);
    if (p.ncl == 0) return;
    const int tid = threadIdx.x, lane = tid & 31, o = lane & 7;
    const unsigned gm = 0xffu << (lane & ~7);
    unsigned nch = 0, nsp = 0;
    for (int i = p.i0 + (tid >> 3); i < p.i1; i += kWideThreads / 8) {
        const int cell = p.lb + i, b = c.begin[cell], en = c.end[cell];
        if (level >= kLevels || en - b <= ncrit) {
            if (o == 0) {
                c.nchild[cell] = 0;
                if (en - b > ncrit) atomicMax(ctl + kCtlLong, (unsigned)(en - b));
            }
            continue;
        }
        const int lo = o ? first_digit_ge(keys, b, en, level + 1, o) : b;
        int hi = __shfl_down_sync(gm, lo, 1, 8);
        if (o == 7) hi = en;
        const int m = __popc((__ballot_sync(gm, hi > lo) >> (lane & ~7)) & 0xffu);
        cb[8 * (int64_t)i + o] = lo;
        ce[8 * (int64_t)i + o] = hi;
        if (o == 0) {
            c.nchild[cell] = m;
            nch += (unsigned)m;
            ++nsp;
        }
    }
    nch = __reduce_add_sync(0xffffffffu, nch);
    nsp = __reduce_add_sync(0xffffffffu, nsp);
    if (lane == 0) {
        s_ch[tid >> 5] = nch;
        s_sp[tid >> 5] = nsp;
    }
    __syncthreads();
    if (tid == 0) {
        for (int w = 1; w < kWideThreads / 32; ++w) {
            nch += s_ch[w];
            nsp += s_sp[w];
        }
        tot[2 * blockIdx.x] = nch;
        tot[2 * blockIdx.x + 1] = nsp;
    }
}

// The children of the level's cells and each cell's rank, after the totals of
// the blocks before this one; the first block leaves the next level's bounds
// (an empty level where the cells would pass the capacity, so that the launches behind do nothing).
__global__ void __launch_bounds__(kWideThreads)
k_wide_write(CellArrays c, int level, int64_t cap, const int32_t *cb, const int32_t *ce, const uint32_t *tot,
             uint32_t *rank, unsigned *ctl)
{
    pdl_wait();
    constexpr int kW = kWideThreads / 32;
    __shared__ unsigned s_t[4], s_w[kW];
    __shared__ int s_ch0[kWideThreads];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const WidePart p = wide_part(ctl, level);
    if (p.ncl == 0) {
        if (blockIdx.x == 0 && tid == 0) ctl[kCtlLevel + level + 2] = ctl[kCtlLevel + level + 1];
        return;
    }
    const unsigned leaves = ctl[kCtlBefore + 2 * level], inner = ctl[kCtlBefore + 2 * level + 1];
    if (tid < 4) s_t[tid] = 0;
    __syncthreads();
    {
        unsigned v[4] = {0, 0, 0, 0};        // children and split cells: of the blocks before, of all
        for (unsigned k = tid; k < gridDim.x; k += kWideThreads) {
            const unsigned x = tot[2 * k], y = tot[2 * k + 1];
            if (k < blockIdx.x) {
                v[0] += x;
                v[1] += y;
            }
            v[2] += x;
            v[3] += y;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            v[q] = __reduce_add_sync(0xffffffffu, v[q]);
            if (lane == 0 && v[q]) atomicAdd(&s_t[q], v[q]);
        }
    }
    __syncthreads();
    const int le = p.lb + p.ncl;
    unsigned ch = s_t[0], sp = s_t[1];       // children and split cells before the next one
    const bool over = (int64_t)le + s_t[2] > cap;
    if (blockIdx.x == 0 && tid == 0) {
        ctl[kCtlLevel + level + 2] = (unsigned)le + (over ? 0u : s_t[2]);
        ctl[kCtlBefore + 2 * level + 2] = leaves + (unsigned)p.ncl - s_t[3];
        ctl[kCtlBefore + 2 * level + 3] = inner + s_t[3];
        ctl[kCtlLeaves] = leaves + (unsigned)p.ncl - s_t[3];
        if (over) ctl[kCtlOverflow] = 1u;
    }
    if (over) return;
    for (int base = p.i0; base < p.i1; base += kWideThreads) {
        const int i = base + tid, cell = p.lb + i;
        const unsigned n = i < p.i1 ? (unsigned)c.nchild[cell] : 0u;
        // children and split cells in one scan: up to 2,048 and 256
        unsigned x = n | (n ? 1u << 16 : 0u);
        const unsigned v = x;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, x, d);
            if (lane >= d) x += y;
        }
        if (lane == 31) s_w[warp] = x;
        __syncthreads();
        unsigned before = x - v, all = 0;
#pragma unroll
        for (int w = 0; w < kW; ++w) {
            if (w < warp) before += s_w[w];
            all += s_w[w];
        }
        const int ch0 = le + (int)(ch + (before & 0xffffu));
        const unsigned k = sp + (before >> 16);
        s_ch0[tid] = n ? ch0 : -1;
        if (i < p.i1) {
            c.child[cell] = n ? ch0 : -1;
            rank[cell] = n ? inner + k : leaves + (unsigned)i - k;
        }
        __syncthreads();
        for (int t = tid; t < 8 * kWideThreads; t += kWideThreads) {         // eight lanes per cell
            const int q = t >> 3, o = t & 7, first = s_ch0[q];
            if (first < 0) continue;
            const int64_t at = 8 * (int64_t)(base + q) + o;
            const int beg = cb[at], en = ce[at], pa = p.lb + base + q;
            const unsigned gm = 0xffu << (lane & ~7);
            const unsigned m = (__ballot_sync(gm, en > beg) >> (lane & ~7)) & 0xffu;
            if (en > beg) {
                const int to = first + __popc(m & ((1u << o) - 1u));
                c.level[to] = level + 1;
                c.parent[to] = pa;
                c.begin[to] = beg;
                c.end[to] = en;
                c.cx[to] = 2 * c.cx[pa] + ((o >> 2) & 1);
                c.cy[to] = 2 * c.cy[pa] + ((o >> 1) & 1);
                c.cz[to] = 2 * c.cz[pa] + (o & 1);
                c.sys[to] = c.sys[pa];
            }
        }
        ch += all & 0xffffu;
        sp += all >> 16;
        __syncthreads();                     // s_w and s_ch0 are free again
    }
}

// Besides the geometry, each cell gets its place among the leaves or the cells
// with children (rank: k_cells) and the packed record the traversal reads with
// one 16-byte load: {cx | level << 21, cy | nchild << 21, cz, child}.
__global__ void k_cell_geometry(CellArrays c, int64_t ncells, int64_t nleaves, const uint32_t *rank,
                                const double *box, int nsys, double *centre, double *half, int32_t *leaves,
                                int *eside, int4 *tcell)
{
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= ncells) return;
    if (i < nsys) eside[i] = ilogb(box[4 * i + 3]);        // the first cells are the roots
    const double *bx = box + 4 * c.sys[i];
    const double h = ldexp(bx[3], -(c.level[i] + 1));
    half[i] = h;
    centre[3 * i] = __dadd_rn(bx[0], __dmul_rn((double)(2 * c.cx[i] + 1), h));
    centre[3 * i + 1] = __dadd_rn(bx[1], __dmul_rn((double)(2 * c.cy[i] + 1), h));
    centre[3 * i + 2] = __dadd_rn(bx[2], __dmul_rn((double)(2 * c.cz[i] + 1), h));
    // leaves[0, nleaves): the leaves in index order; leaves[nleaves, ncells): the
    // cells with children in index (so breadth-first) order, for the downward pass
    const int nch = c.nchild[i];
    leaves[nch ? nleaves + rank[i] : rank[i]] = (int32_t)i;
    tcell[i] = make_int4(c.cx[i] | c.level[i] << kLevels, c.cy[i] | nch << kLevels, c.cz[i], c.child[i]);
}

// ----------------------------------------------------------- traversal
// MAC of Eq. (13), exact: centres (2c+1) 2^(21-l) and radii 2^(21-l) in units
// of the finest half-cell; (rA + rB)^2 < (theta*theta) |dc|^2.  The cells come
// as the packed records of k_cell_geometry.
constexpr int kCoordMask = (1 << kLevels) - 1;
__device__ __forceinline__ bool mac_accept(const int4 A, const int4 B, double theta2)
{
    const int la = A.x >> kLevels, lb = B.x >> kLevels;
    const long long ra = 1ll << (kLevels - la), rb = 1ll << (kLevels - lb);
    const long long dx = (2ll * (A.x & kCoordMask) + 1) * ra - (2ll * (B.x & kCoordMask) + 1) * rb;
    const long long dy = (2ll * (A.y & kCoordMask) + 1) * ra - (2ll * (B.y & kCoordMask) + 1) * rb;
    const long long dz = (2ll * A.z + 1) * ra - (2ll * B.z + 1) * rb;
    const long long d2 = dx * dx + dy * dy + dz * dz;
    const double lhs = (double)((ra + rb) * (ra + rb));
    return lhs < __dmul_rn(theta2, (double)d2);
}

// Position of a pair inside its target's row: the lanes that emit a pair of
// the same list for the same target share one atomic on that row's count.
// All lanes of the warp call it; lanes with want == false get 0.
__device__ __forceinline__ unsigned row_slot(unsigned *rows, int a, bool want)
{
    const int lane = threadIdx.x & 31;
    const unsigned act = __ballot_sync(0xffffffffu, want);
    unsigned slot = 0;
    if (want) {
        const unsigned peers = __match_any_sync(act, a);
        const int leader = __ffs(peers) - 1;
        unsigned base = 0;
        if (lane == leader) base = atomicAdd(&rows[a], (unsigned)__popc(peers));
        base = __shfl_sync(peers, base, leader);
        slot = base + __popc(peers & ((1u << lane) - 1u));
    }
    return slot;
}

// One round of the breadth-first dual traversal.  The rounds are launched
// back to back without the host: round r reads its frontier size from
// counters[kTravFront + r] and adds the next round's to the word after it.
// counters: 0 = m2l, 1 = p2p, kTravOverflow = a frontier exceeded front_cap
// (every later round then does nothing).  Outputs beyond a list's capacity
// are counted but not written; the host grows what overflowed and reruns
// the whole traversal.  Each emitted pair also takes the next position in
// its target's row (rows_m2l / rows_p2p count the pairs of every target),
// kept in slot_m2l / slot_p2p beside the pair, so that the lists can be laid
// out by target without a sort by target.
constexpr int kTravOverflow = 16, kTravFront = 32, kTravMaxRounds = 960;
// blocks of a traversal round: 8 resident blocks of 256 threads per SM
constexpr int kTravBlocksPerSM = 8;
constexpr int kTravWarps = 8;            // warps of a traversal block (256 threads)

__global__ void __launch_bounds__(256)
k_traverse_round(const int4 *__restrict__ tc, int round, double theta2, const int2 *front,
                 unsigned front_cap, int2 *m2l, uint32_t *slot_m2l, unsigned *rows_m2l, unsigned m2l_cap,
                 int2 *p2p, uint32_t *slot_p2p, unsigned *rows_p2p, unsigned p2p_cap, int2 *next,
                 unsigned *counters)
{
    pdl_wait();
    // the frontier size and the overflow flag, read once per block so that the
    // whole block takes the same way (the loop below has block barriers)
    __shared__ unsigned s_nf, s_stop;
    if (threadIdx.x == 0) {
        s_nf = counters[kTravFront + round];
        s_stop = s_nf == 0 || counters[kTravOverflow] != 0u;
    }
    __syncthreads();
    const unsigned nf = s_nf;
    if (s_stop) return;
    if (nf > front_cap) {
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&counters[kTravOverflow], 1u);
        return;
    }
    unsigned *next_count = &counters[kTravFront + round + 1];
    // per-warp totals and block bases of the reservation, two sets used in turn
    __shared__ unsigned s_wsum[2][3][kTravWarps], s_base[2][3];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int par = 0;
    const unsigned stride = gridDim.x * blockDim.x;
    for (unsigned base = blockIdx.x * blockDim.x; base < nf; base += stride) {
        const unsigned t = base + threadIdx.x;
        const bool valid = t < nf;
        int a = 0, b = 0, na = 0, nb = 0;
        int4 A = make_int4(0, 0, 0, 0), B = A;
        if (valid) {
            const int2 pr = front[t];
            a = pr.x; b = pr.y;
            A = __ldg(tc + a);
            B = a == b ? A : __ldg(tc + b);
            na = A.y >> kLevels; nb = B.y >> kLevels;
        }
        // classify: kind 0 = M2L, 1 = P2P, 2 = open a (all children against b,
        // or all child pairs for a self pair), 3 = open b
        int kind = -1;
        if (valid) {
            if (a == b) kind = na == 0 ? 1 : 2;
            else if (mac_accept(A, B, theta2)) kind = 0;
            else if (na == 0 && nb == 0) kind = 1;
            else if (na == 0) kind = 3;
            else if (nb == 0) kind = 2;
            else kind = (A.x >> kLevels) <= (B.x >> kLevels) ? 2 : 3;
        }
        const unsigned n_next = kind == 2 ? (a == b ? (unsigned)(na * na) : (unsigned)na)
                                          : (kind == 3 ? (unsigned)nb : 0u);
        // slots in the three outputs: one atomic per block and output (the
        // counters are shared by the whole grid), lanes in thread order
        const unsigned want[3] = {kind == 0 ? 1u : 0u, kind == 1 ? 1u : 0u, n_next};
        unsigned incl[3];
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            incl[l] = want[l];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned y = __shfl_up_sync(0xffffffffu, incl[l], o);
                if (lane >= o) incl[l] += y;
            }
        }
        unsigned (*wsum)[kTravWarps] = s_wsum[par];
        if (lane == 31) {
#pragma unroll
            for (int l = 0; l < 3; ++l) wsum[l][warp] = incl[l];
        }
        __syncthreads();
        if (threadIdx.x < 3) {
            const int l = threadIdx.x;
            unsigned run = 0;
            for (int w = 0; w < kTravWarps; ++w) {
                const unsigned v = wsum[l][w];
                wsum[l][w] = run;
                run += v;
            }
            s_base[par][l] = run ? atomicAdd(l == 0 ? &counters[0] : (l == 1 ? &counters[1] : next_count), run) : 0u;
        }
        __syncthreads();
        const unsigned o_m2l = s_base[par][0] + wsum[0][warp] + incl[0] - want[0];
        const unsigned o_p2p = s_base[par][1] + wsum[1][warp] + incl[1] - want[1];
        const unsigned o_next = s_base[par][2] + wsum[2][warp] + incl[2] - want[2];
        par ^= 1;
        const unsigned r_m2l = row_slot(rows_m2l, a, kind == 0);
        const unsigned r_p2p = row_slot(rows_p2p, a, kind == 1);
        if (kind == 0) {
            if (o_m2l < m2l_cap) { m2l[o_m2l] = make_int2(a, b); slot_m2l[o_m2l] = r_m2l; }
        } else if (kind == 1) {
            if (o_p2p < p2p_cap) { p2p[o_p2p] = make_int2(a, b); slot_p2p[o_p2p] = r_p2p; }
        }
        // the next frontier: a self pair opens into up to 64 child pairs, far
        // more than other entries, so a warp holding one writes its lanes'
        // children together (entry q of the warp's run goes to the lane whose
        // range holds it); otherwise each lane writes its own
        const int fc = kind == 2 ? A.w : B.w;
        if (__any_sync(0xffffffffu, n_next > 16)) {
            const unsigned wtot = __shfl_sync(0xffffffffu, incl[2], 31);
            const unsigned wbase = o_next - (incl[2] - want[2]);
            for (unsigned q0 = 0; q0 < wtot; q0 += 32) {
                const unsigned q = q0 + lane;
                // owner: the first lane whose inclusive end exceeds q
                int lo = 0;
#pragma unroll
                for (int st = 16; st > 0; st >>= 1) {
                    const unsigned e = __shfl_sync(0xffffffffu, incl[2], lo + st - 1);
                    if (e <= q) lo += st;
                }
                const unsigned ex = __shfl_sync(0xffffffffu, incl[2] - want[2], lo);
                const int oa = __shfl_sync(0xffffffffu, a, lo), ob = __shfl_sync(0xffffffffu, b, lo);
                const int of = __shfl_sync(0xffffffffu, fc, lo), ok = __shfl_sync(0xffffffffu, kind, lo);
                const int on = __shfl_sync(0xffffffffu, na, lo);
                if (q < wtot && wbase + q < front_cap) {
                    const int k = (int)(q - ex);
                    int2 v;
                    if (ok == 3) v = make_int2(oa, of + k);
                    else if (oa == ob) v = make_int2(of + k / on, of + k % on);
                    else v = make_int2(of + k, ob);
                    next[wbase + q] = v;
                }
            }
        } else if (kind == 2 && a == b) {
            for (int i = 0; i < na; ++i)
                for (int j = 0; j < na; ++j) {
                    const unsigned k = o_next + (unsigned)(i * na + j);
                    if (k < front_cap) next[k] = make_int2(fc + i, fc + j);
                }
        } else if (kind == 2) {
            for (int i = 0; i < na; ++i)
                if (o_next + i < front_cap) next[o_next + i] = make_int2(fc + i, b);
        } else if (kind == 3) {
            for (int j = 0; j < nb; ++j)
                if (o_next + j < front_cap) next[o_next + j] = make_int2(a, fc + j);
        }
    }
}

// ------------------------------------------------- lists laid out by target
// A pair goes to its row at the position the traversal gave it.
struct ListArgs {
    const int2 *pairs;
    const uint32_t *slot;
    int64_t np;
    const uint32_t *off;
    int32_t *src;
};
__global__ void k_list_scatter(const ListArgs m, const ListArgs p)
{
    pdl_wait();
    int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const bool second = k >= m.np;
    const ListArgs &l = second ? p : m;
    if (second) k -= m.np;
    if (k >= l.np) return;
    const int2 q = l.pairs[k];
    l.src[l.off[q.x] + l.slot[k]] = q.y;
}

// The exclusive scans of both lists' row counts, a block each (rows and off:
// two arrays of n words one after the other).  One launch for up to kScanRows
// cells; larger trees take the general scan, three launches a list.
constexpr int kScanRows = 1 << 16;
__global__ void __launch_bounds__(1024)
k_scan_rows(const unsigned *rows, int n, uint32_t *off_a, uint32_t *off_b)
{
    __shared__ unsigned s_w[32];
    const unsigned *in = rows + (int64_t)blockIdx.x * n;
    uint32_t *out = blockIdx.x ? off_b : off_a;
    unsigned carry = 0;
    for (int base = 0; base < n; base += 4096) {
        const int i = base + 4 * (int)threadIdx.x;
        unsigned v[4], sum = 0, tot;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[k] = i + k < n ? in[i + k] : 0u;
            sum += v[k];
        }
        unsigned x = carry + cells_scan(sum, s_w, &tot);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (i + k < n) out[i + k] = x;
            x += v[k];
        }
        carry += tot;
    }
}

// Rows of a list sorted by source, in place, so that every build gives the
// same lists in the same order whatever order the traversal's atomics took.
// One warp per row: up to 32 entries in registers, up to kRowWarpMax in the
// warp's slice of shared memory (bitonic network, padded with ~0); longer rows
// are queued for k_row_sort_long.  With COUNT, the P2P interactions of every
// pair (targets x sources) are summed into *inter.
constexpr int kRowWarpMax = 1024, kRowBlockMax = 8192;

__device__ __forceinline__ void bitonic_smem(uint32_t *v, int n, int tid, int nthreads, bool warp)
{
    for (int k = 2; k <= n; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = tid; i < (n >> 1); i += nthreads) {
                const int lo = 2 * i - (i & (j - 1)), hi = lo + j;
                const bool up = (lo & k) == 0;
                const uint32_t x = v[lo], y = v[hi];
                if ((x > y) == up) { v[lo] = y; v[hi] = x; }
            }
            if (warp) __syncwarp(); else __syncthreads();
        }
}

template <bool COUNT>
__device__ __forceinline__ void
row_sort(uint32_t (*buf)[kRowWarpMax], const uint32_t *off, int32_t *src, int64_t nrows, const int32_t *cbeg,
         const int32_t *cend, unsigned long long *inter, uint32_t *long_rows, unsigned *n_long, int warp_max)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t nwarps = (int64_t)gridDim.x * 8;
    unsigned long long acc = 0;
    for (int64_t r = blockIdx.x * 8ll + w; r < nrows; r += nwarps) {
        const uint32_t b0 = off[r], L = off[r + 1] - b0;
        if (L == 0) continue;
        if (COUNT) {
            unsigned long long s = 0;
            for (uint32_t k = lane; k < L; k += 32) {
                const int j = src[b0 + k];
                s += (unsigned long long)(cend[j] - cbeg[j]);
            }
            acc += s * (unsigned long long)(cend[r] - cbeg[r]);
        }
        if (L == 1) continue;
        if (L > (uint32_t)warp_max) {
            if (lane == 0) long_rows[atomicAdd(n_long, 1u)] = (uint32_t)r;
        } else if (L <= 32) {
            uint32_t v = lane < (int)L ? (uint32_t)src[b0 + lane] : ~0u;
#pragma unroll
            for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
                for (int j = k >> 1; j > 0; j >>= 1) {
                    const uint32_t o = __shfl_xor_sync(0xffffffffu, v, j);
                    const bool up = (lane & k) == 0, lower = (lane & j) == 0;
                    v = (lower == up) ? min(v, o) : max(v, o);
                }
            if (lane < (int)L) src[b0 + lane] = (int32_t)v;
        } else {
            int n = 64;
            while (n < (int)L) n <<= 1;
            uint32_t *v = buf[w];
            for (int k = lane; k < n; k += 32) v[k] = k < (int)L ? (uint32_t)src[b0 + k] : ~0u;
            __syncwarp();
            bitonic_smem(v, n, lane, 32, true);
            for (int k = lane; k < (int)L; k += 32) src[b0 + k] = (int32_t)v[k];
            __syncwarp();
        }
    }
    if (COUNT) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lane == 0 && acc) atomicAdd(inter, acc);
    }
}

// both lists in one launch: blockIdx.y 0 the M2L rows, 1 the P2P rows
__global__ void __launch_bounds__(256)
k_row_sort(const uint32_t *m2l_off, int32_t *m2l_src, const uint32_t *p2p_off, int32_t *p2p_src, int64_t nrows,
           const int32_t *cbeg, const int32_t *cend, unsigned long long *inter, uint32_t *long_rows,
           unsigned *n_long, int warp_max)
{
    pdl_wait();
    __shared__ uint32_t buf[8][kRowWarpMax];
    if (blockIdx.y == 0)
        row_sort<false>(buf, m2l_off, m2l_src, nrows, cbeg, cend, nullptr, long_rows, n_long, warp_max);
    else
        row_sort<true>(buf, p2p_off, p2p_src, nrows, cbeg, cend, inter, long_rows + nrows + 1, n_long + 1, warp_max);
}

// The queued long rows, one block each; a row longer than block_max (at most
// kRowBlockMax) sets kErrLongRow in *err and is left for the host, which
// then sorts the whole list by (target, source) with the radix sort.
__global__ void __launch_bounds__(1024)
k_row_sort_long(const uint32_t *m2l_off, int32_t *m2l_src, const uint32_t *p2p_off, int32_t *p2p_src,
                int64_t nrows, const uint32_t *long_rows, const unsigned *n_long, int *err, int block_max)
{
    pdl_wait();
    __shared__ uint32_t v[kRowBlockMax];
    const uint32_t *off = blockIdx.y ? p2p_off : m2l_off;
    int32_t *src = blockIdx.y ? p2p_src : m2l_src;
    if (blockIdx.y) long_rows += nrows + 1;
    const unsigned nl = n_long[blockIdx.y];
    for (unsigned q = blockIdx.x; q < nl; q += gridDim.x) {
        const uint32_t r = long_rows[q], b0 = off[r], L = off[r + 1] - b0;
        if (L > (uint32_t)block_max) {
            if (threadIdx.x == 0) atomicOr(err, kErrLongRow);
            continue;
        }
        int n = 64;
        while (n < (int)L) n <<= 1;
        for (int k = threadIdx.x; k < n; k += blockDim.x) v[k] = k < (int)L ? (uint32_t)src[b0 + k] : ~0u;
        __syncthreads();
        bitonic_smem(v, n, threadIdx.x, blockDim.x, false);
        for (int k = threadIdx.x; k < (int)L; k += blockDim.x) src[b0 + k] = (int32_t)v[k];
        __syncthreads();
    }
}

__global__ void k_pack_pairs(const int2 *pairs, int64_t np, int cbits, uint64_t *keys,
                             uint32_t *vals)
{
    int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= np) return;
    keys[k] = ((uint64_t)(uint32_t)pairs[k].x << cbits) | (uint32_t)pairs[k].y;
    vals[k] = (uint32_t)k;
}

// CSR offsets: off[c] = first sorted pair whose target is >= c.
__global__ void k_row_offsets(const uint64_t *keys, int64_t np, int cbits, int64_t ncells,
                              int32_t *off)
{
    int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (c > ncells) return;
    int64_t L = 0, R = np;
    while (L < R) {
        int64_t mid = (L + R) >> 1;
        if ((int64_t)(keys[mid] >> cbits) < c) L = mid + 1; else R = mid;
    }
    off[c] = (int32_t)L;
}

__global__ void k_unpack_src(const uint64_t *keys, int64_t np, int cbits, int32_t *src)
{
    int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k < np) src[k] = (int32_t)(keys[k] & ((1ull << cbits) - 1ull));
}

__global__ void k_p2p_interactions(const uint64_t *keys, int64_t np, int cbits, CellArrays c,
                                   unsigned long long *total)
{
    int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    unsigned long long v = 0;
    if (k < np) {
        const int a = (int)(keys[k] >> cbits), b = (int)(keys[k] & ((1ull << cbits) - 1ull));
        v = (unsigned long long)(c.end[a] - c.begin[a]) * (unsigned long long)(c.end[b] - c.begin[b]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0 && v) atomicAdd(total, v);
}

// --------------------------------------------------- D-table offset keys
// key = level gap (5 bits) | target-is-finer (1 bit) | three 17-bit biased
// offsets v in units of the finer cell's half side u.  D rows are stored for
// the unit-free offset v; a pair's real offset is u v with u = side / 2^(lf+1)
// a power of two, so one row serves every level and every system.
__device__ __forceinline__ uint64_t hash64(uint64_t x)
{
    x ^= x >> 33; x *= 0xff51afd7ed558ccdull; x ^= x >> 33; x *= 0xc4ceb9fe1a85ec53ull;
    x ^= x >> 33;
    return x;
}

// Probes before the table counts as full: a table under half full needs fewer
// than a hundred, and walking all of a full one for every pair would take seconds.
constexpr int kMaxProbes = 256;

// Offset keys of the M2L pairs, one warp per target row (CSR order): the
// key of a pair is its level gap, which side is finer and the centre offset
// in finer half-cells; equal keys share one derivative row.
__global__ void k_offset_keys(CellArrays c, const int32_t *off, const int32_t *src, int64_t nrows,
                              unsigned long long *table, uint32_t hmask, uint32_t *slot_of,
                              uint64_t *new_key, uint32_t *new_slot, unsigned *n_new, int *err,
                              unsigned *max_gap)
{
    pdl_wait();
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t a = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; a < nrows; a += nwarps) {
        const int k0 = off[a], k1 = off[a + 1];
        if (k0 == k1) continue;
        const int la = c.level[a];
        const long long ax = 2ll * c.cx[a] + 1, ay = 2ll * c.cy[a] + 1, az = 2ll * c.cz[a] + 1;
        unsigned gmax = 0;
        for (int k = k0 + lane; k < k1; k += 32) {
            const int b = src[k];
            const int lb = c.level[b], lf = la > lb ? la : lb;
            const long long sa = 1ll << (lf - la), sb = 1ll << (lf - lb);
            long long d[3] = {ax * sa - (2ll * c.cx[b] + 1) * sb, ay * sa - (2ll * c.cy[b] + 1) * sb,
                              az * sa - (2ll * c.cz[b] + 1) * sb};
            const int gap = la > lb ? la - lb : lb - la;
            gmax = gap > (int)gmax ? (unsigned)gap : gmax;
            uint64_t key = (uint64_t)gap << 52 | (uint64_t)(la > lb) << 51;
            bool bad = false;
            for (int i = 0; i < 3; ++i) {
                if (d[i] < -kKeyBias || d[i] >= kKeyBias) { bad = true; break; }
                key |= (uint64_t)(d[i] + kKeyBias) << (34 - 17 * i);
            }
            if (bad) { atomicOr(err, kErrKeyRange); slot_of[k] = 0; continue; }
            uint32_t h = (uint32_t)hash64(key) & hmask;
            bool placed = false;
            for (int probe = 0; probe < kMaxProbes; ++probe) {
                unsigned long long cur = table[h];
                if (cur == key) { placed = true; break; }
                if (cur == ~0ull) {
                    unsigned long long prev = atomicCAS(&table[h], ~0ull, (unsigned long long)key);
                    if (prev == ~0ull) {                     // a key seen first here joins the list
                        const unsigned k = atomicAdd(n_new, 1u);
                        new_key[k] = key;
                        new_slot[k] = h;
                    }
                    if (prev == ~0ull || prev == key) { placed = true; break; }
                }
                h = (h + 1) & hmask;
            }
            if (!placed) { atomicOr(err, kErrHashFull); h = 0; }
            slot_of[k] = h;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) gmax = max(gmax, __shfl_xor_sync(0xffffffffu, gmax, o));
        if (lane == 0 && gmax) atomicMax(max_gap, gmax);
    }
}

// Which colliding key wins a hash slot depends on timing, so neither the slots
// nor the list's order are reproducible: the distinct keys are sorted by value
// and a pair's D row is the rank of its key.
// A key's rank is the number of smaller keys among the n distinct ones: a warp
// per key up to kRankSmall keys (the radix sort beyond).  keys_out[rank] = key,
// rank_of[slot of the key in the table] = rank.
constexpr unsigned kRankSmall = 4096;
__global__ void __launch_bounds__(256)
k_rank_keys(const uint64_t *key, const uint32_t *slot, const unsigned *n_keys, uint64_t *keys_out, uint32_t *rank_of)
{
    pdl_wait();
    const unsigned n = *n_keys;
    if (n > kRankSmall) return;
    const unsigned lane = threadIdx.x & 31, nw = gridDim.x * (blockDim.x >> 5);
    for (unsigned i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < n; i += nw) {
        const uint64_t v = key[i];
        unsigned r = 0;
        for (unsigned j = lane; j < n; j += 32) r += key[j] < v;
        r = __reduce_add_sync(0xffffffffu, r);
        if (lane == 0) {
            keys_out[r] = v;
            rank_of[slot[i]] = r;
        }
    }
}

// the sorted list's ranks (more than kRankSmall keys)
__global__ void k_rank_sorted(const uint32_t *slot, int64_t n, uint32_t *rank_of)
{
    const int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (r < n) rank_of[slot[r]] = (uint32_t)r;
}

// table slots -> ranks, once rank_of is known (max_keys: up to how many keys it is)
__global__ void k_slot_to_rank(int32_t *didx, int64_t np, const uint32_t *rank_of, const unsigned *n_keys,
                               unsigned max_keys)
{
    pdl_wait();
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (*n_keys <= max_keys && k < np) didx[k] = (int32_t)rank_of[didx[k]];
}

inline unsigned grid(int64_t n, int bs) { return (unsigned)((n + bs - 1) / bs); }

CellArrays cells_of(fmm_tree *t)
{
    CellArrays c;
    c.level = (int32_t *)t->b_level.ptr; c.parent = (int32_t *)t->b_parent.ptr;
    c.child = (int32_t *)t->b_child.ptr; c.nchild = (int32_t *)t->b_nchild.ptr;
    c.begin = (int32_t *)t->b_begin.ptr; c.end = (int32_t *)t->b_end.ptr;
    c.cx = (int32_t *)t->b_cx.ptr; c.cy = (int32_t *)t->b_cy.ptr; c.cz = (int32_t *)t->b_cz.ptr;
    c.sys = (int32_t *)t->b_sys.ptr;
    return c;
}

// Grow a buffer, keeping its first keep_bytes.
fmm_status grow_keep(fmm_tree *t, DevBuf &b, size_t bytes, size_t keep_bytes)
{
    if (b.bytes >= bytes) return FMM_OK;
    DevBuf nb;
    size_t want = std::max(bytes, b.bytes + b.bytes / 2);
    FMM_TRY(ensure(t, nb, want));
    if (keep_bytes && b.ptr)
        FMM_TRY(cuda_check(t, cudaMemcpyAsync(nb.ptr, b.ptr, keep_bytes, cudaMemcpyDeviceToDevice,
                                              t->stream), "grow copy"));
    release(t, b);
    b = nb;
    return FMM_OK;
}

fmm_status check_err(fmm_tree *t, int e)
{
    if (e & kErrNonFinite) { t->err = "non-finite particle position"; return FMM_EINVAL; }
    if (e & kErrKeyRange) {
        t->err = "an accepted M2L offset exceeds 2^16 finer half-cells (theta too small for the tree)";
        return FMM_EINVAL;
    }
    if (e & kErrSortWait) { t->err = "a bounded wait of the radix sort gave up"; return FMM_ETIMEOUT; }
    return FMM_OK;
}

void record(fmm_tree *t, int i)
{
    if (t->profiling) cudaEventRecord(t->ev[i], t->stream);
}

}  // namespace

// ---------------------------------------------------------------------------
// keys of one system, with the counts of their digits p0 .. 7 (hist: the sort's
// scratch, its head zeroed here)
static void morton_keys(cudaStream_t st, const double *pos, int64_t n, int p0, uint64_t *keys, uint32_t *idx,
                        unsigned long long *box_scratch, double *box_out, int *err, uint32_t *hist,
                        int64_t *launches)
{
    const unsigned g = (unsigned)std::min<int64_t>(grid(n, 256), 4 * (int64_t)sm_count());
    k_sort_init<<<1, 256, 0, st>>>(box_scratch, hist);
    launch_next(st, k_bbox, g, 256, 0, pos, n, box_scratch, err);
    const int64_t ntiles = (n + kRadixTile - 1) / kRadixTile;
    launch_next(st, k_keys, g, 256, 0, pos, n, box_scratch, box_out, keys, idx, p0, hist, (uint64_t *)(hist + kRadixHead),
                              ntiles * 256);
    *launches += 3;
}

void morton_order_prepare()
{
    cudaFuncAttributes fa;
    const void *kerns[] = {(const void *)k_sort_init, (const void *)k_bbox, (const void *)k_keys,
                           (const void *)k_tie_sort<false>};
    for (const void *k : kerns)
        if (cudaFuncGetAttributes(&fa, k) != cudaSuccess) cudaGetLastError();
    radix_sort_prepare();
}

fmm_status morton_order_raw(cudaStream_t st, const double *pos, int64_t n, uint64_t *keys,
                            uint32_t *idx, uint64_t *keys2, uint32_t *idx2, uint32_t *hist,
                            unsigned long long *box_scratch, double *box_out, int *err)
{
    int64_t launches = 0;
    int herr = 0;
    const int p0 = first_pass(n);
    // the passes end in (keys2, idx2), the tie sort in (keys, idx)
    const bool even = (kRadixMaxPasses - p0) % 2 == 0;
    uint64_t *ka = even ? keys2 : keys, *kb = even ? keys : keys2;
    uint32_t *va = even ? idx2 : idx, *vb = even ? idx : idx2;
    if (cudaMemsetAsync(err, 0, sizeof(int), st) != cudaSuccess) {
        cudaGetLastError();
        return FMM_ECUDA;
    }
    morton_keys(st, pos, n, p0, ka, va, box_scratch, box_out, err, hist, &launches);
    radix_sort_top(ka, va, kb, vb, n, p0, hist, err, st, &launches);
    launch_next(st, k_tie_sort<false>, grid(n, 256), 256, 0, keys2, idx2, n, 8 * p0, keys, idx, err, nullptr, nullptr, 0,
                                                     nullptr, nullptr, nullptr, nullptr, nullptr);
    cudaError_t e = cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e == cudaSuccess && (herr & kErrTieRun)) {
        // every pass, over the keys as they stand (each key still carries its index)
        radix_sort_pairs(keys, idx, keys2, idx2, n, 3 * kLevels, hist, err, st, &launches);
        e = cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        return FMM_ECUDA;
    }
    if (herr & kErrNonFinite) return FMM_EINVAL;
    return (herr & kErrSortWait) ? FMM_ETIMEOUT : FMM_OK;
}

fmm_status build_tree(fmm_tree *t, const double *pos, const double *mom)
{
    const int64_t n = t->n;
    const int nsys = (int)t->sys_off.size() - 1;
    cudaStream_t st = t->stream;
    t->have_lists = false;
    t->ncells = t->nleaves = 0;
    t->long_leaf = 0;
    t->nlevels = 0;
    t->level_begin.clear();
    if (n == 0) return FMM_OK;

    FMM_TRY(ensure(t, t->b_keys, 8 * n));
    FMM_TRY(ensure(t, t->b_keys2, 8 * n));
    FMM_TRY(ensure(t, t->b_idx, 4 * n));
    FMM_TRY(ensure(t, t->b_idx2, 4 * n));
    FMM_TRY(ensure(t, t->b_hist, radix_hist_bytes(n)));
    FMM_TRY(ensure(t, t->b_scan_tmp, scan_scratch_bytes(std::max<int64_t>(n, 1 << 20) * 8)));
    FMM_TRY(ensure(t, t->b_px, 8 * n));
    FMM_TRY(ensure(t, t->b_py, 8 * n));
    FMM_TRY(ensure(t, t->b_pz, 8 * n));
    FMM_TRY(ensure(t, t->b_S, 8 * n * t->nS));
    FMM_TRY(ensure(t, t->b_perm, 4 * n));
    FMM_TRY(ensure(t, t->b_sysoff, 8 * (size_t)(nsys + 1)));
    FMM_TRY(ensure(t, t->b_sysbox, 32 * (size_t)nsys + 48 * (size_t)nsys));
    uint64_t *keys = (uint64_t *)t->b_keys.ptr;
    uint32_t *idx = (uint32_t *)t->b_idx.ptr;
    int64_t *off = (int64_t *)t->b_sysoff.ptr;
    double *sbox = (double *)t->b_sysbox.ptr;                               // [nsys][4]
    unsigned long long *sbox_raw = (unsigned long long *)(sbox + 4 * nsys); // [nsys][6]

    record(t, 0);
    cudaMemsetAsync(t->b_err.ptr, 0, sizeof(int), st);
    FMM_TRY(cuda_check(t, cudaMemcpyAsync(off, t->sys_off.data(), 8 * (size_t)(nsys + 1),
                                          cudaMemcpyHostToDevice, st), "system offsets"));
    // one system: by the leading key bits and the tie sort, by all bits where the
    // last set of this handle (or, below, this one) had a long run of ties
    auto sort_one = [&](bool full) {
        uint64_t *keys2 = (uint64_t *)t->b_keys2.ptr;
        uint32_t *idx2 = (uint32_t *)t->b_idx2.ptr, *hist = (uint32_t *)t->b_hist.ptr;
        int *err = (int *)t->b_err.ptr;
        double *px = (double *)t->b_px.ptr, *py = (double *)t->b_py.ptr, *pz = (double *)t->b_pz.ptr,
               *S = (double *)t->b_S.ptr;
        int32_t *perm = (int32_t *)t->b_perm.ptr;
        const int p0 = full ? 0 : first_pass(n);
        const bool swap = !full && (kRadixMaxPasses - p0) % 2 == 0;      // the passes end in (keys2, idx2)
        uint64_t *ka = swap ? keys2 : keys, *kb = swap ? keys : keys2;
        uint32_t *va = swap ? idx2 : idx, *vb = swap ? idx : idx2;
        morton_keys(st, pos, n, p0, ka, va, sbox_raw, sbox, err, hist, &t->launches);
        record(t, 1);
        radix_sort_top(ka, va, kb, vb, n, p0, hist, err, st, &t->launches);
        if (full)
            launch_next(st, k_gather, grid(n, 256), 256, 0, pos, mom, t->nS, idx, n, px, py, pz, S, perm, keys,
                        8 * first_pass(n), err);
        else
            launch_next(st, k_tie_sort<true>, grid(n, 256), 256, 0, keys2, idx2, n, 8 * p0, keys, idx, err, pos, mom, t->nS,
                                                            px, py, pz, S, perm);
        ++t->launches;
        record(t, 2);
    };
    bool full = t->sort_full;
    if (nsys == 1) {
        sort_one(full);
    } else {
        // particle -> system (kept in b_idx2 until the sort needs it)
        FMM_TRY(ensure(t, t->b_lval2, 4 * n));
        int32_t *sys_of = (int32_t *)t->b_lval2.ptr;
        k_sys_of<<<grid(n, 256), 256, 0, st>>>(off, nsys, n, sys_of);
        k_box_init_seg<<<grid(6 * nsys, 256), 256, 0, st>>>(sbox_raw, nsys);
        k_bbox_seg<<<grid(n, 256), 256, 0, st>>>(pos, n, sys_of, sbox_raw, (int *)t->b_err.ptr);
        k_box_final_seg<<<grid(nsys, 128), 128, 0, st>>>(sbox_raw, nsys, sbox);
        k_keys_seg<<<grid(n, 256), 256, 0, st>>>(pos, n, sys_of, sbox, keys, idx);
        t->launches += 5;
        record(t, 1);
        radix_sort_pairs(keys, idx, (uint64_t *)t->b_keys2.ptr, (uint32_t *)t->b_idx2.ptr, n,
                         3 * kLevels, (uint32_t *)t->b_hist.ptr, (int *)t->b_err.ptr, st, &t->launches);
        // stable second pass by system: order = (system, key, original index)
        FMM_TRY(ensure(t, t->b_lkeys, 8 * n));
        FMM_TRY(ensure(t, t->b_lkeys2, 8 * n));
        uint64_t *skeys = (uint64_t *)t->b_lkeys.ptr, *key_of = (uint64_t *)t->b_lkeys2.ptr;
        k_sys_keys<<<grid(n, 256), 256, 0, st>>>(keys, idx, (const int32_t *)t->b_lval2.ptr, n,
                                                 skeys, key_of);
        int sbits = 1;
        while ((1 << sbits) < nsys) ++sbits;
        radix_sort_pairs(skeys, idx, (uint64_t *)t->b_keys2.ptr, (uint32_t *)t->b_idx2.ptr, n,
                         sbits, (uint32_t *)t->b_hist.ptr, (int *)t->b_err.ptr, st, &t->launches);
        k_regather_keys<<<grid(n, 256), 256, 0, st>>>(key_of, idx, n, keys);
        launch_next(st, k_gather, grid(n, 256), 256, 0, pos, mom, t->nS, idx, n, (double *)t->b_px.ptr,
                                               (double *)t->b_py.ptr, (double *)t->b_pz.ptr,
                                               (double *)t->b_S.ptr, (int32_t *)t->b_perm.ptr, nullptr, 0, nullptr);
        t->launches += 3;
        record(t, 2);
    }

    // ---- cells: one launch, one host sync (again with more room where they overflow)
    FMM_TRY(ensure(t, t->b_ctl, 4 * kCtlWords));
    unsigned *ctl = (unsigned *)t->b_ctl.ptr;
    DevBuf *cb[10] = {&t->b_level, &t->b_parent, &t->b_child, &t->b_nchild, &t->b_begin,
                      &t->b_end, &t->b_cx, &t->b_cy, &t->b_cz, &t->b_sys};
    int64_t cap = std::max<int64_t>(t->b_level.bytes / 4,
                                    std::max<int64_t>(1024, 5 * (n / std::max(1, t->max_leaf)) + 64 + 2 * nsys));
    unsigned hc[kCtlHost];
    t->sys_box.assign(4 * (size_t)nsys, 0.0);
    for (;;) {
        for (DevBuf *b : cb) FMM_TRY(ensure(t, *b, 4 * cap));
        FMM_TRY(ensure(t, t->b_flags, 4 * cap));
        FMM_TRY(ensure(t, t->b_scan, 4 * cap));
        FMM_TRY(ensure(t, t->b_front, 8 * 8 * cap));      // child begin/end of every octant
        int32_t *cbeg = (int32_t *)t->b_front.ptr, *cend = cbeg + 8 * cap;
        k_cells<<<kCellBlocks, kCellThreads, 0, st>>>(cells_of(t), off, nsys, sbox, (const int *)t->b_err.ptr,
                                                      t->max_leaf, keys, cap, cbeg, cend, (uint32_t *)t->b_scan.ptr,
                                                      (uint32_t *)t->b_flags.ptr, ctl);
        ++t->launches;
        FMM_TRY(cuda_check(t, cudaGetLastError(), "cells"));
        FMM_TRY(cuda_check(t, cudaMemcpyAsync(hc, ctl, sizeof(hc), cudaMemcpyDeviceToHost, st), "level counts"));
        if (nsys > 1)
            FMM_TRY(cuda_check(t, cudaMemcpyAsync(t->sys_box.data(), sbox, 32 * (size_t)nsys,
                                                  cudaMemcpyDeviceToHost, st), "box"));
        FMM_TRY(cuda_check(t, cudaStreamSynchronize(st), "sync"));
        if (hc[kCtlTie]) {                  // a long run of ties: by all bits
            full = true;
            cudaMemsetAsync(t->b_err.ptr, 0, sizeof(int), st);
            sort_one(full);
            continue;
        }
        // wide levels: four at a time, then a look whether any are left
        const unsigned wide = hc[kCtlWide];
        for (int l = (int)wide - 1; wide && !hc[kCtlOverflow] && l <= kLevels &&
                                    hc[kCtlLevel + l + 1] > hc[kCtlLevel + l];) {
            const unsigned g = (unsigned)(kWideBlocksPerSM * std::max(1, sm_count()));   // totals: 2 g <= cap words
            for (const int to = std::min(l + 4, kLevels + 1); l < to; ++l) {
                launch_next(st, k_wide_count, g, kWideThreads, 0, cells_of(t), l, t->max_leaf, keys, cbeg, cend,
                            (uint32_t *)t->b_scan.ptr, ctl);
                launch_next(st, k_wide_write, g, kWideThreads, 0, cells_of(t), l, cap, cbeg, cend,
                            (const uint32_t *)t->b_scan.ptr, (uint32_t *)t->b_flags.ptr, ctl);
                t->launches += 2;
            }
            FMM_TRY(cuda_check(t, cudaGetLastError(), "wide levels"));
            FMM_TRY(cuda_check(t, cudaMemcpyAsync(hc, ctl, sizeof(hc), cudaMemcpyDeviceToHost, st), "level counts"));
            FMM_TRY(cuda_check(t, cudaStreamSynchronize(st), "sync"));
        }
        if (!hc[kCtlOverflow]) break;
        cap *= 2;
    }
    FMM_TRY(check_err(t, (int)hc[kCtlErr]));
    t->sort_full = nsys == 1 && full && (hc[kCtlErr] & kErrLongTies);
    if (nsys == 1) std::memcpy(t->sys_box.data(), hc + kCtlBox, 32);
    // levels 0 .. nlev - 1 hold cells
    int nlev = 1;
    while (nlev <= kLevels && hc[kCtlLevel + nlev + 1] > hc[kCtlLevel + nlev]) ++nlev;
    t->level_begin.assign(hc + kCtlLevel, hc + kCtlLevel + nlev + 1);
    t->ncells = t->level_begin.back();
    t->nlevels = nlev;
    t->nleaves = hc[kCtlLeaves];
    t->long_leaf = (int)hc[kCtlLong];
    t->lo[0] = t->sys_box[0]; t->lo[1] = t->sys_box[1]; t->lo[2] = t->sys_box[2];
    t->side = t->sys_box[3];
    const int64_t nc = t->ncells;
    FMM_TRY(ensure(t, t->b_centre, 8 * 3 * nc));
    FMM_TRY(ensure(t, t->b_half, 8 * nc));
    FMM_TRY(ensure(t, t->b_tcell, 16 * nc));
    FMM_TRY(ensure(t, t->b_leaves, 4 * (size_t)nc));
    FMM_TRY(ensure(t, t->b_syseside, 4 * (size_t)nsys));
    k_cell_geometry<<<grid(nc, 256), 256, 0, st>>>(cells_of(t), nc, t->nleaves, (const uint32_t *)t->b_flags.ptr, sbox,
                                                    nsys, (double *)t->b_centre.ptr, (double *)t->b_half.ptr,
                                                    (int32_t *)t->b_leaves.ptr, (int *)t->b_syseside.ptr,
                                                    (int4 *)t->b_tcell.ptr);
    ++t->launches;
    record(t, 3);
    return cuda_check(t, cudaGetLastError(), "cell geometry");
}

fmm_status build_lists(fmm_tree *t, double theta)
{
    cudaStream_t st = t->stream;
    t->have_lists = false;
    t->tc_plan = false;
    t->fx_off = false;
    t->sym_plan = false;
    t->n_m2l = t->n_p2p = t->n_p2p_inter = t->n_doff = 0;
    t->d_p = -1;
    if (t->n == 0) { t->theta = theta; t->have_lists = true; return FMM_OK; }
    const int64_t nc = t->ncells;
    CellArrays c = cells_of(t);
    const double theta2 = theta * theta;

    // ---- breadth-first dual traversal: a pair's two levels add up to at
    // least its round, so 2 * nlevels rounds empty the frontier; they run as
    // one batch of launches with one host sync (more batches if not)
    FMM_TRY(ensure(t, t->b_counters, 4 * (kTravFront + kTravMaxRounds + 64)));
    unsigned *cnt = (unsigned *)t->b_counters.ptr;
    // row counts of both lists: [0, nc] M2L, [nc + 1, 2 nc + 1] P2P (the last
    // word of each stays 0 and becomes the total under the exclusive scan)
    FMM_TRY(ensure(t, t->b_rows, 8 * (size_t)(nc + 1)));
    unsigned *rows = (unsigned *)t->b_rows.ptr;
    const int nsys = (int)t->sys_off.size() - 1;
    size_t m2l_cap = std::max<size_t>(4096, t->m2l_cap_hint), p2p_cap = std::max<size_t>(4096, 40 * (size_t)t->nleaves);
    size_t front_cap = std::max<size_t>({(size_t)4096, (size_t)nsys, 16 * (size_t)t->nleaves,
                                         t->b_front.bytes / 8, t->b_front2.bytes / 8});
    std::vector<unsigned> hc((size_t)kTravFront + kTravMaxRounds + 1);
    const int batch = 2 * std::max(t->nlevels, 1) + 1;
    for (;;) {
        FMM_TRY(grow_keep(t, t->b_m2l_raw, 8 * m2l_cap, 0));
        FMM_TRY(grow_keep(t, t->b_p2p_raw, 8 * p2p_cap, 0));
        FMM_TRY(grow_keep(t, t->b_m2l_slot, 4 * (t->b_m2l_raw.bytes / 8), 0));
        FMM_TRY(grow_keep(t, t->b_p2p_slot, 4 * (t->b_p2p_raw.bytes / 8), 0));
        FMM_TRY(grow_keep(t, t->b_front, 8 * front_cap, 0));
        FMM_TRY(grow_keep(t, t->b_front2, 8 * front_cap, 0));
        m2l_cap = t->b_m2l_raw.bytes / 8;
        p2p_cap = t->b_p2p_raw.bytes / 8;
        front_cap = std::min(t->b_front.bytes, t->b_front2.bytes) / 8;
        int2 *fr[2] = {(int2 *)t->b_front.ptr, (int2 *)t->b_front2.ptr};
        launch_next(st, k_list_init, (unsigned)std::min<int64_t>(grid(std::max<int64_t>(2 * (nc + 1), nsys), 256), 2 * (int64_t)sm_count()), 256, 0, cnt, kTravFront + kTravMaxRounds + 1, rows, 2 * (nc + 1), fr[0], nsys, kTravFront);
        ++t->launches;
        int r = 0;
        bool retry = false;
        const unsigned trav_blocks = (unsigned)(kTravBlocksPerSM * sm_count());
        for (;;) {
            const int end = std::min(r + batch, kTravMaxRounds);
            for (; r < end; ++r) {
                launch_next(st, k_traverse_round, trav_blocks, 256, 0,
                    (const int4 *)t->b_tcell.ptr, r, theta2, fr[r & 1], (unsigned)front_cap,
                    (int2 *)t->b_m2l_raw.ptr, (uint32_t *)t->b_m2l_slot.ptr, rows, (unsigned)m2l_cap,
                    (int2 *)t->b_p2p_raw.ptr, (uint32_t *)t->b_p2p_slot.ptr, rows + nc + 1,
                    (unsigned)p2p_cap, fr[(r + 1) & 1], cnt);
                ++t->launches;
            }
            FMM_TRY(cuda_check(t, cudaMemcpyAsync(hc.data(), cnt, 4 * (size_t)(kTravFront + r + 1),
                                                  cudaMemcpyDeviceToHost, st), "counters"));
            FMM_TRY(cuda_check(t, cudaStreamSynchronize(st), "sync"));
            unsigned fmax = 0;
            for (int k = 0; k <= r; ++k) fmax = std::max(fmax, hc[kTravFront + k]);
            if (hc[kTravOverflow] || fmax > front_cap) {
                front_cap = std::max<size_t>(2 * front_cap, 2 * (size_t)fmax);
                retry = true;
            }
            if (hc[0] > m2l_cap) { m2l_cap = 2 * (size_t)hc[0]; retry = true; }
            if (hc[1] > p2p_cap) { p2p_cap = 2 * (size_t)hc[1]; retry = true; }
            if (retry || hc[kTravFront + r] == 0) break;
            if (r >= kTravMaxRounds) {
                t->err = "the dual traversal did not end within its round limit";
                return FMM_EINVAL;
            }
        }
        if (!retry) break;
    }
    const unsigned host_cnt[2] = {hc[0], hc[1]};
    const int64_t nm2l = host_cnt[0], np2p = host_cnt[1];
    t->m2l_cap_hint = (size_t)nm2l + nm2l / 8;

    // ---- both lists laid out by target (CSR).  Normally: offsets from the
    // row counts of the traversal, each pair to the position it was given,
    // rows sorted by source.  A row too long for the row sort (flag in
    // counter word 6, seen at the next host sync) sends both lists through
    // the radix sort of (target, source) keys instead; both give the same
    // lists.  The sorts report a wait that gave up in counter word 14.
    FMM_TRY(ensure(t, t->b_scan_tmp, scan_scratch_bytes(std::max<int64_t>(nc + 1, 1 << 20) * 8)));
    FMM_TRY(ensure(t, t->b_m2l_src, 4 * std::max<int64_t>(nm2l, 1)));
    FMM_TRY(ensure(t, t->b_m2l_didx, 4 * std::max<int64_t>(nm2l, 1)));
    FMM_TRY(ensure(t, t->b_m2l_off, 4 * (nc + 1)));
    FMM_TRY(ensure(t, t->b_p2p_src, 4 * std::max<int64_t>(np2p, 1)));
    FMM_TRY(ensure(t, t->b_p2p_off, 4 * (nc + 1)));
    FMM_TRY(ensure(t, t->b_long, 8 * (size_t)(nc + 1)));
    // counter words (zero since k_list_init): 4, 5 long rows of each list, 6 their
    // flag, 8-9 P2P interactions, 10 errors of the offset hash, 12 largest level
    // gap, 13 distinct offsets, 14 sort status; one copy brings them to the host
    int *sort_err = (int *)(cnt + 14), *long_err = (int *)(cnt + 6);
    unsigned *n_long = cnt + 4;
    unsigned long long *inter_d = (unsigned long long *)(cnt + 8);
    struct Words {
        unsigned pad0[4], n_long[2];
        int le;
        unsigned pad1;
        unsigned long long inter;
        int he;
        unsigned pad2, gmax, nd;
        int serr;
        unsigned pad3;
    } hw;
    static_assert(sizeof(Words) == 64, "counter words 0 .. 15");
    auto read_words = [&]() -> fmm_status {
        FMM_TRY(cuda_check(t, cudaMemcpyAsync(&hw, cnt, sizeof(hw), cudaMemcpyDeviceToHost, st), "list counters"));
        return cuda_check(t, cudaStreamSynchronize(st), "sync");
    };
    int32_t *m2l_off = (int32_t *)t->b_m2l_off.ptr, *p2p_off = (int32_t *)t->b_p2p_off.ptr;
    int32_t *m2l_src = (int32_t *)t->b_m2l_src.ptr, *p2p_src = (int32_t *)t->b_p2p_src.ptr;
    int cbits = 1;
    while ((1ll << cbits) < nc) ++cbits;
    // FMM_ROW_SORT_LIMIT (tests) lowers the longest row the row sorts take
    int row_lim = kRowBlockMax;
    if (const char *env = getenv("FMM_ROW_SORT_LIMIT")) row_lim = std::min(std::max(2, atoi(env)), kRowBlockMax);
    auto layout_rows = [&]() {
        if (nc + 1 <= kScanRows) {
            k_scan_rows<<<2, 1024, 0, st>>>(rows, (int)(nc + 1), (uint32_t *)m2l_off, (uint32_t *)p2p_off);
            ++t->launches;
        } else {
            exclusive_scan_u32(rows, (uint32_t *)m2l_off, nc + 1, (uint32_t *)t->b_scan_tmp.ptr, st, &t->launches);
            exclusive_scan_u32(rows + nc + 1, (uint32_t *)p2p_off, nc + 1, (uint32_t *)t->b_scan_tmp.ptr, st,
                               &t->launches);
        }
        const ListArgs lm = {(const int2 *)t->b_m2l_raw.ptr, (const uint32_t *)t->b_m2l_slot.ptr, nm2l,
                             (const uint32_t *)m2l_off, m2l_src};
        const ListArgs lp = {(const int2 *)t->b_p2p_raw.ptr, (const uint32_t *)t->b_p2p_slot.ptr, np2p,
                             (const uint32_t *)p2p_off, p2p_src};
        if (nm2l + np2p > 0) launch_next(st, k_list_scatter, grid(nm2l + np2p, 256), 256, 0, lm, lp);
        uint32_t *lq = (uint32_t *)t->b_long.ptr;
        const unsigned rgrid = (unsigned)std::min<int64_t>((nc + 7) / 8, 6 * (int64_t)sm_count());
        launch_next(st, k_row_sort, dim3(rgrid, 2), 256, 0, (const uint32_t *)m2l_off, m2l_src, (const uint32_t *)p2p_off,
                                                    p2p_src, nc, c.begin, c.end, inter_d, lq, n_long,
                                                    std::min(row_lim, kRowWarpMax));
        launch_next(st, k_row_sort_long, dim3((unsigned)sm_count(), 2), 1024, 0, (const uint32_t *)m2l_off, m2l_src,
                                                                         (const uint32_t *)p2p_off, p2p_src, nc, lq,
                                                                         n_long, long_err, row_lim);
        t->launches += 3;
    };
    auto layout_radix = [&]() -> fmm_status {
        const int64_t nmax = std::max<int64_t>({nm2l, np2p, 1});
        FMM_TRY(ensure(t, t->b_lkeys, 8 * nmax));
        FMM_TRY(ensure(t, t->b_lkeys2, 8 * nmax));
        FMM_TRY(ensure(t, t->b_lval, 4 * nmax));
        FMM_TRY(ensure(t, t->b_lval2, 4 * nmax));
        FMM_TRY(ensure(t, t->b_hist, radix_hist_bytes(nmax)));
        uint64_t *lk = (uint64_t *)t->b_lkeys.ptr, *lk2 = (uint64_t *)t->b_lkeys2.ptr;
        uint32_t *lv = (uint32_t *)t->b_lval.ptr, *lv2 = (uint32_t *)t->b_lval2.ptr;
        cudaMemsetAsync(cnt + 6, 0, 4 * 4, st);          // words 6 .. 9: flag, P2P count
        k_pack_pairs<<<grid(np2p, 256), 256, 0, st>>>((const int2 *)t->b_p2p_raw.ptr, np2p, cbits, lk, lv);
        radix_sort_pairs(lk, lv, lk2, lv2, np2p, 2 * cbits, (uint32_t *)t->b_hist.ptr, sort_err, st,
                         &t->launches);
        k_row_offsets<<<grid(nc + 1, 256), 256, 0, st>>>(lk, np2p, cbits, nc, p2p_off);
        k_unpack_src<<<grid(np2p, 256), 256, 0, st>>>(lk, np2p, cbits, p2p_src);
        k_p2p_interactions<<<grid(np2p, 256), 256, 0, st>>>(lk, np2p, cbits, c, inter_d);
        t->launches += 4;
        if (nm2l > 0) {
            k_pack_pairs<<<grid(nm2l, 256), 256, 0, st>>>((const int2 *)t->b_m2l_raw.ptr, nm2l, cbits, lk, lv);
            radix_sort_pairs(lk, lv, lk2, lv2, nm2l, 2 * cbits, (uint32_t *)t->b_hist.ptr, sort_err,
                             st, &t->launches);
            k_unpack_src<<<grid(nm2l, 256), 256, 0, st>>>(lk, nm2l, cbits, m2l_src);
            t->launches += 2;
        }
        k_row_offsets<<<grid(nc + 1, 256), 256, 0, st>>>(lk, nm2l, cbits, nc, m2l_off);
        ++t->launches;
        return FMM_OK;
    };
    layout_rows();

    // ---- distinct M2L offsets (rows of the derivative table), numbered by value.
    // The ranks and the pairs' rows are formed before the host knows the count;
    // one host sync then reads everything at once: the hash status, the long-row
    // flag, the distinct count, the largest level gap and the P2P interaction
    // count.  A full hash table, a long row or more than kRankSmall offsets
    // (rare) redo the part concerned.  The table starts at 64k slots whatever the
    // list's length: even deep adaptive trees have a few thousand offsets.
    int64_t ndoff = 0;
    if (nm2l > 0) {
        uint32_t H = 1u << 16;
        size_t dcap = 0;
        for (bool again = false;; again = true) {
            FMM_TRY(ensure(t, t->b_hash, 8 * (size_t)H));
            dcap = (size_t)std::min<int64_t>(H, nm2l);            // distinct keys, at most
            FMM_TRY(ensure(t, t->b_dsort, 12 * dcap));            // the list: keys, then slots
            FMM_TRY(ensure(t, t->b_scan, 4 * (size_t)H));         // slot -> rank
            FMM_TRY(ensure(t, t->b_dkeys, 8 * (size_t)kRankSmall));
            uint64_t *lkey = (uint64_t *)t->b_dsort.ptr;
            uint32_t *lslot = (uint32_t *)(lkey + dcap), *rank_of = (uint32_t *)t->b_scan.ptr;
            cudaMemsetAsync(t->b_hash.ptr, 0xff, 8 * (size_t)H, st);
            if (again) cudaMemsetAsync(cnt + 10, 0, 4 * 4, st);   // errors, gap, count
            launch_next(st, k_offset_keys, (unsigned)std::min<int64_t>((nc + 7) / 8, 8 * (int64_t)sm_count()), 256, 0,
                c, m2l_off, m2l_src, nc, (unsigned long long *)t->b_hash.ptr, H - 1,
                (uint32_t *)t->b_m2l_didx.ptr, lkey, lslot, cnt + 13, (int *)(cnt + 10), cnt + 12);
            launch_next(st, k_rank_keys, (unsigned)sm_count(), 256, 0, lkey, lslot, cnt + 13, (uint64_t *)t->b_dkeys.ptr,
                                                              rank_of);
            launch_next(st, k_slot_to_rank, grid(nm2l, 256), 256, 0, (int32_t *)t->b_m2l_didx.ptr, nm2l, rank_of, cnt + 13,
                                                            kRankSmall);
            t->launches += 3;
            FMM_TRY(read_words());
            if (hw.le) {
                FMM_TRY(layout_radix());
                hw.le = 0;
                continue;
            }
            if (hw.he & kErrKeyRange) {
                t->err = "an accepted M2L offset exceeds 2^16 finer half-cells (theta too small for the tree)";
                return FMM_EINVAL;
            }
            if (!(hw.he & kErrHashFull)) break;
            H <<= 1;
        }
        t->max_gap = (int)hw.gmax;
        ndoff = hw.nd;
        if (ndoff > (int64_t)kRankSmall) {
            uint64_t *lkey = (uint64_t *)t->b_dsort.ptr;
            uint32_t *lslot = (uint32_t *)(lkey + dcap), *rank_of = (uint32_t *)t->b_scan.ptr;
            FMM_TRY(ensure(t, t->b_dkeys, 8 * (size_t)ndoff));
            FMM_TRY(ensure(t, t->b_lkeys2, 8 * (size_t)ndoff));
            FMM_TRY(ensure(t, t->b_lval2, 4 * (size_t)ndoff));
            FMM_TRY(ensure(t, t->b_dsort_h, radix_hist_bytes(ndoff)));
            radix_sort_pairs(lkey, lslot, (uint64_t *)t->b_lkeys2.ptr, (uint32_t *)t->b_lval2.ptr, ndoff, 57,
                             (uint32_t *)t->b_dsort_h.ptr, sort_err, st, &t->launches);
            k_rank_sorted<<<grid(ndoff, 256), 256, 0, st>>>(lslot, ndoff, rank_of);
            launch_next(st, k_slot_to_rank, grid(nm2l, 256), 256, 0, (int32_t *)t->b_m2l_didx.ptr, nm2l, rank_of, cnt + 13, ~0u);
            t->launches += 2;
            FMM_TRY(cuda_check(t, cudaMemcpyAsync(t->b_dkeys.ptr, lkey, 8 * (size_t)ndoff, cudaMemcpyDeviceToDevice, st),
                               "offset keys"));
            FMM_TRY(read_words());                                // the sort's status
        }
    } else {
        FMM_TRY(read_words());
        while (hw.le) {                     // a long P2P row with no M2L list to catch it earlier
            FMM_TRY(layout_radix());
            FMM_TRY(read_words());
        }
    }
    const int serr = hw.serr;
    const unsigned long long inter = hw.inter;
    if (serr & kErrSortWait) {
        t->err = "a bounded wait of the radix sort gave up";
        return FMM_ETIMEOUT;
    }
    t->n_m2l = nm2l;
    t->n_p2p = np2p;
    t->n_p2p_inter = (int64_t)inter;
    t->n_doff = ndoff;
    t->theta = theta;
    t->have_lists = true;
    return FMM_OK;
}

}  // namespace fmm
