// m2l_fx.cu -- the FP64 form's M2L in 64-bit fixed point over the target tiles
// of the plan (m2l_tc.cu).
//
// The per-cell FP64 kernel (k_m2l) is bound by the FP64 pipe: one warp
// instruction per 64 clocks and scheduler, 812 multiply-adds a pair at p = 6,
// 5.0 of its 5.6 ms at 1M dipoles.  Three 32 x 32 + 64 bit integer
// multiply-adds (5.6 clocks each) carry the same product to 57 bits, provided
// both factors have a common scale per sum.  The plan gives it: the 128
// targets of a tile share the operator of a row's key, so the operator is
// scaled once per key, a multipole once per cell, and the sums of a target in
// a unit that holds all of its list.
//
// Scaling (powers of two throughout, so exact).  With h_t, h_s the half sides,
//   M'_m = M_m h_s^(s-|m|) 2^(a_m),   a_m = round(log2 m!) - (|m| - s),
//   T'_nm = D_{n+m} (level factors) 2^(-a_m - b_n),   b_n = round(log2 n!),
//   L_n = h_t^(-|n|-1-s) 2^(b_n) sum_pairs sum_m T'_nm M'_m.
// a_m and b_n level the magnitudes over the orders: for particles spread over
// a cell, or bunched in its corner, at theta 0.5, 1 <= p <= 12, max |M'| times the
// largest row sum of |T'| is 1.2 to 7 times the sum of the absolute values of the
// terms of a first-order component, so that 57 bits of the product of those
// bounds are more than the 53 of each FP64 rounding (wider angles: below).
//   per cell  e_s:  |M'| < 2^e_s;  M' = (Mh 2^26 + Ml) 2^(e_s - B), B = 57 (56 for nM > 126)
//   per key   e_k:  sum_m |T'_nm| < 2^e_k for every n; T' likewise at 2^(e_k - 57)
//   per target e_t: sum over its list of 2^(e_s + e_k) <= 2^e_t
// both for every class of n: n = 0 alone, then the groups of four columns by their
// lowest order.  The row sums grow with the order where cells are close (theta 0.7,
// p = 9: a hundred times those of n = 0) and fall by 2^-g an order where the source is g
// levels coarser: in one unit for all n the field was off by 9e-15 of the magnitudes of
// its terms there, 5e-13 at p = 12, 4e-12 on small sets of 22 levels; FP64 1e-16.
// With their own units it is within 4e-16 up to p = 10 at theta 0.6 and p = 9 at 0.7;
// beyond (1e-15 to 1e-14: the multipoles share one unit a cell) the per-cell kernel stays.
// A row's sum A1 + A0 / 2^26, A1 = sum Th Mh, A0 = sum (Th Ml + Tl Mh), stays
// below 2^(B + 5) (the row sums of T' bound it) and A0 below 2^63 (nM 2^(B - 1)
// and 2^56); it is shifted right by e_t - e_s - e_k into a 64-bit sum that
// cannot pass 2^(B + 5) either.
// Integer sums do not depend on their order: the chunks add theirs with
// 64-bit reductions to one array, and a target's result does not depend on
// the other targets of its tile.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "fmm_internal.cuh"
#include "fx64.cuh"
#include "umma.cuh"

namespace fmm {

using namespace umma;
using namespace fx;

namespace {

constexpr int kFxThreads = 128;
// rows of a block: a part of a chunk (1M dipoles, p = 6: 1.84 ms with 8 rows,
// 1.86 with 16, 1.91 with 32; 200k: 0.25, 0.275, 0.33: the last blocks' wait)
constexpr int kFxRows = 8;
constexpr int kFxMaxK = 13;          // classes: orders up to 12
constexpr int kFxMaxNM = 253;        // A0 stays below 2^63
constexpr int kFxSmemMax = 216 * 1024;
constexpr int kFxPad = 33;           // 16-byte pieces per line of 32 targets: staging by rows without conflicts
constexpr int kZeroExp = -(1 << 20); // exponent of an all-zero row
constexpr int kBadExp = 1 << 24;     // a row that holds an infinity or a NaN

// What turns a target's sums into its row of L
struct FxOut {
    const int32_t *tile_tgt, *col, *cls, *level, *sys, *rn;      // rn: full index of each stored component
    const int *e_side;
    double *L;
    int s, ncol, nL, nLh, unit;
};

struct FxArgs {
    const int32_t *chunk_rb, *chunk_re, *row_key, *slot;
    const uint32_t *tile_chunk;          // [tiles + 1] first chunk of each tile
    const int4 *M;                       // [cells][nq]: two limb pairs (h, l, h, l) each
    const int *eM;
    const int *ekey, *etgt;              // [key][K], [target][K] exponents of the classes
    const int2 *img;                     // [keys][E] limb pairs
    u64 *acc;                            // [tile][4][ncolp][32]
    unsigned *arrive;                    // [tile][4] blocks done, from 0
    FxOut out;
    int K, with0;                        // classes; column 0 is n = 0
    int parts, tiles, nq, E, ncolp;      // parts: blocks of kFxRows rows a chunk can take
    // the column groups (4 columns each) dealt to the four warps: image offset
    // (elements), pairs of multipoles, first column
    int ng[4];
    int g_off[4][kFxMaxGroups], g_mq[4][kFxMaxGroups], g_col[4][kFxMaxGroups], g_cls[4][kFxMaxGroups];
};

struct Sum {
    s64 a1, a0;
};

__device__ __forceinline__ void mac(Sum &s, int th, int tl, int mh, int ml)
{
    s.a1 = madp(th, mh, s.a1);
    s.a0 = madp(th, ml, s.a0);
    s.a0 = madp(tl, mh, s.a0);
}

// The sums of 32 targets back to FP64 rows, by the block that arrives last: a
// column's sums read side by side and turned in shared memory.
__device__ __noinline__ void fx_finish(const FxArgs &a, int slot0, s64 *fs)
{
    __shared__ int s_pos[kMaxTot];                   // full index -> column
    const FxOut &o = a.out;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int k = threadIdx.x; k < o.nL; k += kFxThreads) s_pos[k] = -1;
    const u64 *acc = a.acc + (size_t)slot0 * a.ncolp;
    for (int k = threadIdx.x; k < a.ncolp * 32; k += kFxThreads)
        fs[(k >> 5) * kFxPad + (k & 31)] = (s64)__ldcg(acc + k);
    __syncthreads();
    for (int k = threadIdx.x; k < o.ncol; k += kFxThreads) s_pos[o.col[k] & 511] = k;
    __syncthreads();
    for (int t = w; t < 32; t += 4) {
        const int c = o.tile_tgt[slot0 + t];
        if (c < 0) continue;
        const int *et = a.etgt + (size_t)(slot0 + t) * a.K;
        const int hl = o.e_side[o.sys[c]] - o.level[c] - 1;
        for (int r = lane; r < o.nLh; r += 32) {
            const int k = s_pos[o.rn[r]];
            double v = 0.0;
            if (k >= 0) {
                const int cv = o.col[k], nn = (cv >> 9) & 15, bn = cv >> 13, e = et[nn ? o.cls[k >> 2] : 0];
                v = ldexp((double)fs[k * kFxPad + t], e - o.unit + bn - (nn + 1 + o.s) * hl);
                if (e >= kBadExp / 2) v = __longlong_as_double(0x7ff8000000000000ll);
            }
            o.L[(size_t)c * o.nLh + r] = v;
        }
    }
}

// One block per (part of a chunk, 32 targets of the tile): lane = target, the
// four warps share the staged multipoles and divide the columns.  Shared
// memory: [nq][33] 16-byte multipole pieces and E limb pairs of the operator of
// one row; the other blocks of the SM compute while one waits for its row.  Bound
// by the integer pipes, 3 multiply-adds a product: M2L phase (this kernel; the
// per-cell k_m2l before) 5.59 -> 1.73 ms at 1M dipoles, p = 6 (32 targets 87 %
// full); 3.30 -> 1.54 ms at 262k Plummer, p = 8 (47 % full); 0.57 -> 0.23 ms at
// 200k charges and dipoles, p = 6; 125k dipoles, p = 6: 0.68 -> 0.28 ms.  (Two stages with the next
// row's copies in flight halve the blocks an SM holds: 1M dipoles, p = 6, 1.96
// instead of 1.86 ms; 262k Plummer, p = 8, 1.99 instead of 1.67.)
template <int NG>
__global__ void __launch_bounds__(kFxThreads, NG <= 4 ? 5 : (NG <= 8 ? 4 : 2)) k_m2l_fx(const __grid_constant__ FxArgs a)
{
    pdl_wait();
    extern __shared__ int4 sm4[];
    __shared__ int s_src[kFxRows][32], s_es[kFxRows][32], s_ek[kFxRows][kFxMaxK], s_key[kFxRows],
        s_act[kFxRows], s_tile, s_last;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int qt = blockIdx.x & 3, chunk = (blockIdx.x >> 2) / a.parts, part = (blockIdx.x >> 2) - chunk * a.parts;
    const int rb = a.chunk_rb[chunk] + part * kFxRows, n = min(a.chunk_re[chunk] - rb, kFxRows);
    for (int i = tid; i < a.tiles; i += kFxThreads)
        if ((int)a.tile_chunk[i] <= chunk && chunk < (int)a.tile_chunk[i + 1]) s_tile = i;
    __syncthreads();
    const int slot0 = s_tile * 128 + 32 * qt;
    int4 *Ts = sm4 + a.nq * kFxPad;
    int *Es = (int *)(Ts + (a.E >> 1));              // [K][32] exponents of the targets
    for (int k = w; k < a.K; k += 4) Es[32 * k + lane] = a.etgt[(size_t)(slot0 + lane) * a.K + k];
    int any = 0;
    for (int r = w; r < n; r += 4) {
        const int src = a.slot[(size_t)(rb + r) * 128 + 32 * qt + lane], key = a.row_key[rb + r];
        s_src[r][lane] = src;
        s_es[r][lane] = src >= 0 ? a.eM[src] : 0;
        if (lane < a.K) s_ek[r][lane] = a.ekey[(size_t)key * a.K + lane];
        const int act = __any_sync(0xffffffffu, src >= 0);
        any |= act;
        if (lane == 0) {
            s_key[r] = key;
            s_act[r] = act;
        }
    }
    any = __syncthreads_or(any);
    auto stage = [&](int r) {
        for (int k = tid, t = tid / a.nq, q = tid - t * a.nq; k < 32 * a.nq; k += kFxThreads) {
            const int src = s_src[r][t];
            cp_async16(smem_u32(sm4 + q * kFxPad + t), a.M + (size_t)max(src, 0) * a.nq + q, src < 0 ? 0 : 16);
            q += kFxThreads;
            while (q >= a.nq) {
                q -= a.nq;
                ++t;
            }
        }
        const int4 *ti = (const int4 *)(a.img + (size_t)s_key[r] * a.E);
        for (int e = tid; e < (a.E >> 1); e += kFxThreads) cp_async16(smem_u32(Ts + e), ti + e, 16);
        cp_async_commit();
    };
    s64 P[NG][4];
#pragma unroll
    for (int g = 0; g < NG; ++g)
#pragma unroll
        for (int c = 0; c < 4; ++c) P[g][c] = 0;
    const int ng = any ? a.ng[w] : 0;
    for (int r = 0; r < n; ++r) {
        if (!s_act[r]) continue;                     // no pair of these 32 targets
        stage(r);
        cp_async_wait<0>();
        __syncthreads();
        const int4 *Ms = sm4 + lane;
        const int es = s_es[r][lane];
        // 0..62: a pair 2^62 below its target's unit adds nothing
        auto shift = [&](int k) { return min(max(Es[32 * k + lane] - es - s_ek[r][k], 0), 62); };
#pragma unroll
        for (int g = 0; g < NG; ++g) {
            if (g < ng) {
                const int4 *T4 = Ts + (a.g_off[w][g] >> 1);
                const int mq = a.g_mq[w][g], sh = shift(a.g_cls[w][g]);
                const int sh0 = g == 0 && w == 0 && a.with0 ? shift(0) : sh;
                const s64 half = (1ll << sh) >> 1, half0 = (1ll << sh0) >> 1;
                Sum s[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) s[c] = {g + c ? half : half0, 1ll << 25};    // both shifts round
#pragma unroll 4
                for (int q = 0; q < mq; ++q) {
                    const int4 m = Ms[q * kFxPad];
                    const int4 t0 = T4[4 * q], t1 = T4[4 * q + 1], t2 = T4[4 * q + 2], t3 = T4[4 * q + 3];
                    mac(s[0], t0.x, t0.y, m.x, m.y);
                    mac(s[1], t0.z, t0.w, m.x, m.y);
                    mac(s[2], t1.x, t1.y, m.x, m.y);
                    mac(s[3], t1.z, t1.w, m.x, m.y);
                    mac(s[0], t2.x, t2.y, m.z, m.w);
                    mac(s[1], t2.z, t2.w, m.z, m.w);
                    mac(s[2], t3.x, t3.y, m.z, m.w);
                    mac(s[3], t3.z, t3.w, m.z, m.w);
                }
#pragma unroll
                for (int c = 0; c < 4; ++c) P[g][c] += (s[c].a1 + (s[c].a0 >> 26)) >> (g + c ? sh : sh0);
            }
        }
        __syncthreads();                             // before the next row is staged
    }
    u64 *acc = a.acc + (size_t)slot0 * a.ncolp + lane;
#pragma unroll
    for (int g = 0; g < NG; ++g)
        if (g < ng)
#pragma unroll
            for (int c = 0; c < 4; ++c) atomicAdd(acc + (size_t)(a.g_col[w][g] + c) * 32, (u64)P[g][c]);
    __threadfence();                                 // the sums are added before the block counts as done
    __syncthreads();
    if (tid == 0) {
        const unsigned blocks = (a.tile_chunk[s_tile + 1] - a.tile_chunk[s_tile]) * a.parts;
        s_last = atomicAdd(a.arrive + s_tile * 4 + qt, 1u) + 1u == blocks;
        __threadfence();
    }
    __syncthreads();
    if (s_last) fx_finish(a, slot0, (s64 *)sm4);
}

// The cells' multipoles as limbs, then the exponents of the plan's targets.  One
// warp per cell: the row folded as in k_fold_m, its exponent, the limbs.  One warp
// per target: e_t from its list.  Blocks claim their work in order, the cells
// first, so that every cell is with a running block when the first targets' block
// waits for them: the wait ends whatever else holds the rest of the chip (as
// blocks of a cooperative launch that met at a grid barrier, it could run into its
// bound).  per: cells or targets of a block; four where all blocks fit the chip at
// once or nearly (one for each warp), eight beyond, as each claim is an atomic on one
// word (125k and 1M dipoles, us: 4 30, 102; 8 34, 87; 16 43, 90; as blocks that met at
// a barrier 29, 80; with an exponent for every order since, 125k 25, 1M 120).  ctl: [0] claimed, [1] blocks of cells done, from 0.
constexpr int kExpSmall = 1 << 15;                   // cells and targets up to which a block takes four
__global__ void __launch_bounds__(128)
k_fx_exps(const double *M, int64_t nc, DevTables tb, const int32_t *am, const int32_t *level, const int32_t *sys,
          const int *e_side, int nq, int bits, int2 *Mx, int *eM, int slots, const int32_t *tile_tgt,
          const int32_t *off, const int32_t *src, const int32_t *didx, int k0, int K, const int *ekey, int *etgt, unsigned *ctl,
          int per)
{
    extern __shared__ double fsm[];
    __shared__ unsigned s_id;
    __shared__ int s_ok;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned ncb = (unsigned)((nc + per - 1) / per);
    if (threadIdx.x == 0) s_id = atomicAdd(ctl, 1u);
    __syncthreads();
    if (s_id < ncb) {
        double *v = fsm + w * tb.nM;
        const int64_t c0 = (int64_t)s_id * per, c1 = min(nc, c0 + per);
        for (int64_t c = c0 + w; c < c1; c += 4) {
            for (int m = lane; m < tb.nM; m += 32) v[m] = M[c * tb.nM + m];
            __syncwarp();
            for (int l = 0; l < tb.h_fold_lev; ++l) {
                for (int q = tb.h_fold_off[l] + lane; q < tb.h_fold_off[l + 1]; q += 32) {
                    const int i = tb.h_fold[3 * q], a = tb.h_fold[3 * q + 1], b = tb.h_fold[3 * q + 2];
                    double x = v[i];
                    if (a >= 0) x -= v[a];
                    if (b >= 0) x -= v[b];
                    v[i] = x;
                }
                __syncwarp();
            }
            const int hl = e_side[sys[c]] - level[c] - 1;        // log2 of the half side
            int e = kZeroExp;
            for (int r = lane; r < tb.nMh; r += 32) {
                const int k = am[r], wr = (k >> 8) - (k & 255) * hl;
                const u64 b = (u64)__double_as_longlong(v[tb.h_rm[r]]) & 0x7fffffffffffffffull;
                if (b >= 0x7ff0000000000000ull) e = kBadExp;
                // a value within 2^-29 of the next power of two would round to it: Mh < 2^31
                else if (b) e = max(e, (int)((b + (1ull << 23)) >> 52) - 1022 + wr);
            }
            e = __reduce_max_sync(0xffffffffu, e);
            if (lane == 0) eM[c] = e;
            for (int r = lane; r < 2 * nq; r += 32) {
                s64 x = 0;
                if (r < tb.nMh && e != kBadExp) {
                    const int k = am[r], wr = (k >> 8) - (k & 255) * hl;
                    x = fix64(v[tb.h_rm[r]], wr + bits - e);
                }
                const int h = (int)((x + (1ll << 25)) >> 26);
                Mx[c * 2 * nq + r] = make_int2(h, (int)(x - ((s64)h << 26)));
            }
            __syncwarp();
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            atomicAdd(ctl + 1, 1u);
        }
        return;
    }
    if (threadIdx.x == 0) {
        const volatile unsigned *done = ctl + 1;
        const long long t0 = clock64();
        while (*done < ncb && clock64() - t0 < (1ll << 31)) __nanosleep(32);
        s_ok = *done >= ncb;
        __threadfence();
    }
    __syncthreads();
    const int q0 = (int)(s_id - ncb) * per, q1 = min(slots, q0 + per);
    for (int q = q0 + w; q < q1; q += 4) {
        const int c = tile_tgt[q];
        constexpr int kK = kFxMaxK;
        int e[kK];
#pragma unroll
        for (int k = 0; k < kK; ++k) e[k] = kZeroExp;
        if (c >= 0 && s_ok) {
            const int b = off[c], en = off[c + 1];
            float f[kK];
            for (int q2 = b + lane; q2 < en; q2 += 32) {
                const int es = __ldcg(eM + src[q2]), *ek = ekey + (size_t)didx[q2] * K;
#pragma unroll
                for (int k = 0; k < kK; ++k)
                    if (k >= k0 && k < K) e[k] = max(e[k], es + ek[k]);
            }
#pragma unroll
            for (int k = 0; k < kK; ++k) {
                f[k] = 0.0f;
                if (k >= k0 && k < K) e[k] = __reduce_max_sync(0xffffffffu, e[k]);
            }
            for (int q2 = b + lane; q2 < en; q2 += 32) {
                const int es = __ldcg(eM + src[q2]), *ek = ekey + (size_t)didx[q2] * K;
#pragma unroll
                for (int k = 0; k < kK; ++k)
                    if (k >= k0 && k < K) f[k] += __int_as_float((127 + max(es + ek[k] - e[k], -100)) << 23);   // 2 to that
            }
#pragma unroll
            for (int k = 0; k < kK; ++k)
                if (k >= k0 && k < K) {
                    for (int o = 16; o > 0; o >>= 1) f[k] += __shfl_xor_sync(0xffffffffu, f[k], o);
                    e[k] += ilogbf(f[k] * 1.01f) + 1;
                }
        }
        if (lane == 0)
#pragma unroll
            for (int k = 0; k < kK; ++k)
                if (k < K) etgt[(size_t)q * K + k] = s_ok ? e[k] : kBadExp;      // a wait that gave up shows as NaN
    }
}

// Operator images, a block per key (17 us at 346 keys, p = 6): T'_nm of every element, the key's exponent
// from the largest row sum, the limbs.
__device__ __forceinline__ double fx_element(int el, const double *D, int esc, int dl)
{
    if (el < 0) return 0.0;
    const int k = el & 511, nm = (el >> 9) & 15, msh = (el >> 13) & 15, sh = (el >> 17) - 64;
    return ldexp(D[k], (nm + 1) * esc + dl * msh - sh);
}

__global__ void __launch_bounds__(128)
k_fx_images(const uint64_t *dkeys, const double *D, int nD, int E, int ngroups, const int32_t *g_first,
            const int32_t *g_cls, const int32_t *el, int with0, int K, int2 *img, int *ekey)
{
    __shared__ u64 s_big[kFxMaxK];             // largest row sum of each class, its bits
    __shared__ int s_ek[kFxMaxK];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t r = blockIdx.x;
    const uint64_t key = dkeys[r];
    const int gap = (int)((key >> 52) & 31), tfiner = (int)((key >> 51) & 1);
    const int esc = tfiner ? 0 : gap, dl = tfiner ? gap : -gap;
    const double *Dr = D + r * nD;
    if (threadIdx.x < K) s_big[threadIdx.x] = 0;
    __syncthreads();
    for (int g = w; g < ngroups; g += 4) {
        double v = 0.0;                              // lanes of equal (lane & 3) share a column
        for (int e = g_first[g] + lane; e < g_first[g + 1]; e += 32) v += fabs(fx_element(el[e], Dr, esc, dl));
        v += __shfl_xor_sync(0xffffffffu, v, 4);
        v += __shfl_xor_sync(0xffffffffu, v, 8);
        v += __shfl_xor_sync(0xffffffffu, v, 16);
        if (lane < 4) atomicMax(&s_big[with0 && g + lane == 0 ? 0 : g_cls[g]], (u64)__double_as_longlong(v));
    }
    __syncthreads();
    // row sums below 2^ek less a margin for their own rounding: Th < 2^31
    if (threadIdx.x < K) {
        const double big = __longlong_as_double((long long)s_big[threadIdx.x]);
        s_ek[threadIdx.x] = big > 0.0 ? ilogb(big * 1.004) + 1 : 0;
        ekey[r * K + threadIdx.x] = s_ek[threadIdx.x];
    }
    __syncthreads();
    for (int g = w; g < ngroups; g += 4)
        for (int e = g_first[g] + lane; e < g_first[g + 1]; e += 32) {
            const int ek = s_ek[with0 && g + (lane & 3) == 0 ? 0 : g_cls[g]];
            const s64 x = __double2ll_rn(ldexp(fx_element(el[e], Dr, esc, dl), 57 - ek));
            const int h = (int)((x + (1ll << 25)) >> 26);
            img[r * E + e] = make_int2(h, (int)(x - ((s64)h << 26)));
        }
}

int log2_factorial(const MultiIndex &I, int k)
{
    double v = 1.0;
    for (int q : {I.nx[k], I.ny[k], I.nz[k]})
        for (int j = 2; j <= q; ++j) v *= j;
    return (int)std::lround(std::log2(v));
}

void build_layout_fx(FxLayout &Ly, int s, int p, int h, int n_lo)
{
    const MultiIndex &I = multi_index();
    auto shell = [&](int k) { return I.nx[k] + I.ny[k] + I.nz[k]; };
    std::vector<int> ms, ns;
    for (int k = ntot(s - 1); k < ntot(p + s); ++k)
        if (!h || I.nz[k] <= 1) ms.push_back(k);
    for (int n = 0; n < ntot(p); ++n)
        if (shell(n) >= n_lo && (!h || I.nz[n] <= 1)) ns.push_back(n);
    Ly.s = s;
    Ly.p = p;
    Ly.h = h;
    Ly.n_lo = n_lo;
    Ly.nM = (int)ms.size();
    Ly.nq = (Ly.nM + 1) / 2;
    Ly.bits = Ly.nM <= 126 ? 57 : 56;
    Ly.ncol = (int)ns.size();
    Ly.groups = (Ly.ncol + 3) / 4;
    auto a_of = [&](int gm) { return log2_factorial(I, gm) - (shell(gm) - s); };
    Ly.am.clear();
    for (int gm : ms) Ly.am.push_back(a_of(gm) * 256 + (shell(gm) - s));
    Ly.col.clear();
    for (int n : ns) Ly.col.push_back(n | shell(n) << 9 | log2_factorial(I, n) << 13);
    Ly.cls.clear();
    Ly.K = std::max(p, 1) + 1;
    Ly.first.assign(1, 0);
    Ly.el.clear();
    Ly.products = 0;
    for (int g = 0; g < Ly.groups; ++g) {
        const int reach = p + s - shell(ns[4 * g]);      // graded: the group's lowest order comes first
        int cnt = 0;
        while (cnt < Ly.nM && shell(ms[cnt]) <= reach) ++cnt;
        cnt = (cnt + 1) & ~1;
        for (int m = 0; m < cnt; ++m)
            for (int j = 0; j < 4; ++j) {
                const int c = 4 * g + j;
                int v = -1;
                if (c < Ly.ncol && m < Ly.nM) {
                    const int n = ns[c], gm = ms[m], tot = shell(n) + shell(gm);
                    if (tot <= p + s) {
                        const int d = I(I.nx[n] + I.nx[gm], I.ny[n] + I.ny[gm], I.nz[n] + I.nz[gm]);
                        const int sh = a_of(gm) + log2_factorial(I, n);
                        // the shift may be negative: kept in the upper bits with the sign
                        // bit clear (offset by 64)
                        ++Ly.products;
                        v = d | tot << 9 | (shell(gm) - s) << 13 | (sh + 64) << 17;
                    }
                }
                Ly.el.push_back(v);
            }
        Ly.first.push_back((int)Ly.el.size());
        Ly.cls.push_back(std::max(shell(ns[4 * g]), 1));
    }
    Ly.E = (int)Ly.el.size();
    // columns to warps: the longest group to the least loaded warp, at most cap
    // groups to a warp; the smallest cap within a tenth of the best balance
    Ly.cap = 0;
    int best = 0;
    for (int cap : {16, 12, 8, 6, 4}) {
        if (4 * cap < Ly.groups) break;
        int load[4] = {0, 0, 0, 0}, cnt[4] = {0, 0, 0, 0};
        std::vector<int> owner(Ly.groups);
        for (int g = 0; g < Ly.groups; ++g) {            // lengths fall with g
            int w = -1;
            for (int k = 0; k < 4; ++k)
                if (cnt[k] < cap && (w < 0 || load[k] < load[w])) w = k;
            owner[g] = w;
            load[w] += Ly.first[g + 1] - Ly.first[g];
            ++cnt[w];
        }
        const int span = std::max(std::max(load[0], load[1]), std::max(load[2], load[3]));
        if (!Ly.cap) best = span;
        if (!Ly.cap || 10 * span <= 11 * best) {
            Ly.cap = cap;
            Ly.owner = owner;
        }
    }
}

inline size_t fx_smem(const FxLayout &Ly)
{
    return 16 * (size_t)Ly.nq * kFxPad + 8 * (size_t)Ly.E + 128 * (size_t)Ly.K;
}

inline unsigned gridn(int64_t n, int bs) { return (unsigned)((n + bs - 1) / bs); }

}  // namespace

// The line between this form and the per-cell k_m2l: the list's products a
// system, and its pairs per distinct offset, on which depends how full the plan's
// rows are (a row holds a tile's pairs of one offset; an adaptive tree has six times
// the offsets of a uniform one).  Evaluates with new lists, per cell -> here, ms:
//   uniform          1 6 (source order, p) 419k pairs, 3.4e8 products   1.76 -> 1.30
//                    0 3 419k pairs, 0.4e8 products                     no difference
//                    1 11 38k pairs, 2.0e8 (110 pairs an offset)        2.09 -> 1.44
//   Plummer          2 8 91k pairs, 2.3e8 (44)                          2.09 -> 2.18
//                    2 8 143k, 3.6e8 (60)                               2.51 -> 2.48
//                    1 10 61k, 2.4e8 (29)                               2.09 -> 2.40
//                    1 10 129k, 5.1e8 (55)                              2.92 -> 2.94
//                    1 6 272k, 2.2e8 (126)                              1.94 -> 1.88
//   theta 0.4        1 7 286k, 3.7e8 (37)                               3.36 -> 3.65
// Past p + s = 11 of charges and dipoles the per-cell kernel falls off and the line
// lies lower: Plummer 1 11 49k pairs (25) 2.65 -> 2.71, 68k (33) 3.24 -> 2.94; 0 12 the same.
// Lists that stay (loops) gain 0.1 to 0.3 ms more than these, the plan's time.
// Handles with a memory budget keep the per-cell kernel, so that a served request's
// bits do not depend on its slot's memory.
constexpr double kFxMinWork = 2.0e8;
constexpr int64_t kFxMinFill = 56, kFxMinFillHigh = 30;    // pairs an offset
constexpr int kFxHighProducts = 5000;

bool fx_usable(fmm_tree *t, int s, int p, int harmonic, int n_lo)
{
    if (!t->m2l_tiled || t->budget) return false;
    FxLayout &Ly = t->fx_lay;
    const int h = harmonic ? 1 : 0;
    if (Ly.s != s || Ly.p != p || Ly.h != h || Ly.n_lo != n_lo) {
        build_layout_fx(Ly, s, p, h, n_lo);
        t->fx_img_p = -1;                     // images and maps of the old layout
        t->fx_off = false;
    }
    if (t->fx_off || (p >= 11 && t->theta > 0.5) || (p >= 10 && t->theta > 0.6)) return false;
    const double nsys = (double)std::max<int64_t>(1, (int64_t)t->sys_off.size() - 1);
    const double fill = (double)(Ly.products > kFxHighProducts ? kFxMinFillHigh : kFxMinFill) * t->n_doff;
    return (double)t->n_m2l * Ly.products >= kFxMinWork * nsys && (double)t->n_m2l >= fill * nsys && Ly.cap > 0 &&
           Ly.nM <= kFxMaxNM && fx_smem(Ly) <= (size_t)kFxSmemMax;
}

fmm_status fx_prepare(fmm_tree *t, int p)
{
    cudaStream_t st = t->stream;
    const FxLayout &Ly = t->fx_lay;
    if (!t->tc_plan) FMM_TRY(tc_build_plan(t));
    if (t->tc_chunks == 0) return FMM_OK;
    const size_t slots = (size_t)t->tc_tiles * 128;
    if (t->fx_img_p != p) {
        const size_t n1 = (size_t)Ly.E, n2 = Ly.first.size(), n3 = Ly.am.size(), n4 = Ly.col.size(),
                     n5 = Ly.cls.size();
        FMM_TRY(ensure(t, t->b_fx_el, 4 * (n1 + n2 + n3 + n4 + n5)));
        int32_t *d = (int32_t *)t->b_fx_el.ptr;
        auto up = [&](const std::vector<int> &v) {
            const cudaError_t e = cudaMemcpyAsync(d, v.data(), 4 * v.size(), cudaMemcpyHostToDevice, st);
            d += v.size();
            return cuda_check(t, e, "upload");
        };
        FMM_TRY(up(Ly.el));
        FMM_TRY(up(Ly.first));
        FMM_TRY(up(Ly.am));
        FMM_TRY(up(Ly.col));
        FMM_TRY(up(Ly.cls));
        FMM_TRY(ensure(t, t->b_fx_img, 8 * (size_t)t->n_doff * Ly.E));
        FMM_TRY(ensure(t, t->b_fx_ekey, 4 * (size_t)t->n_doff * Ly.K));
        d = (int32_t *)t->b_fx_el.ptr;
        k_fx_images<<<(unsigned)t->n_doff, 128, 0, st>>>(
            (const uint64_t *)t->b_dkeys.ptr, (const double *)t->b_D.ptr, ntot(p + t->s), Ly.E, Ly.groups, d + n1,
            d + n1 + n2 + n3 + n4, d, Ly.n_lo == 0, Ly.K, (int2 *)t->b_fx_img.ptr, (int *)t->b_fx_ekey.ptr);
        ++t->launches;
        t->fx_img_p = p;
    }
    FMM_TRY(ensure(t, t->b_fx_em, 4 * (size_t)t->ncells));
    FMM_TRY(ensure(t, t->b_fx_et, 4 * slots * Ly.K));
    // the sums, the blocks done per 32 targets, k_fx_exps' counters
    FMM_TRY(ensure(t, t->b_fx_acc, 32 * slots * Ly.groups + slots / 8 + 16));
    // the limbs take the place of the folded multipoles
    return ensure(t, t->b_Mh, 16 * (size_t)t->ncells * Ly.nq);
}

fmm_status run_fx_exps(fmm_tree *t, const double *M, const DevTables &tb)
{
    cudaStream_t st = t->stream;
    const FxLayout &Ly = t->fx_lay;
    if (Ly.nM != tb.nMh || (Ly.h == 1) != (tb.harmonic == 1)) {
        t->err = "fixed-point M2L: layout and tables disagree";
        return FMM_EINVAL;                   // not reachable: both follow the handle's flag
    }
    if (t->tc_chunks == 0) return FMM_OK;
    const int slots = (int)t->tc_tiles * 128;
    const size_t acc = 32 * (size_t)slots * Ly.groups;
    FMM_TRY(cuda_check(t, cudaMemsetAsync(t->b_fx_acc.ptr, 0, acc + slots / 8 + 16, st), "memset"));
    const int32_t *am = (const int32_t *)t->b_fx_el.ptr + Ly.E + Ly.first.size();
    const int per = t->ncells + slots <= kExpSmall ? 4 : 8;
    k_fx_exps<<<gridn(t->ncells, per) + gridn(slots, per), 128, 32 * (size_t)tb.nM, st>>>(
        M, t->ncells, tb, am, (const int32_t *)t->b_level.ptr, (const int32_t *)t->b_sys.ptr, t->sys_eside_dev(), Ly.nq,
        Ly.bits, (int2 *)t->b_Mh.ptr, (int *)t->b_fx_em.ptr, slots, (const int32_t *)t->b_tc_tgt.ptr,
        (const int32_t *)t->b_m2l_off.ptr, (const int32_t *)t->b_m2l_src.ptr, (const int32_t *)t->b_m2l_didx.ptr,
        Ly.n_lo, Ly.K, (const int *)t->b_fx_ekey.ptr, (int *)t->b_fx_et.ptr,
        (unsigned *)((char *)t->b_fx_acc.ptr + acc + slots / 8), per);
    ++t->launches;
    return cuda_check(t, cudaGetLastError(), "fixed-point multipoles");
}

fmm_status run_m2l_fx(fmm_tree *t, const DevTables &tb, double *L)
{
    cudaStream_t st = t->stream;
    const FxLayout &Ly = t->fx_lay;
    if (t->tc_chunks == 0) return FMM_OK;
    const int slots = (int)t->tc_tiles * 128, ncolp = 4 * Ly.groups;
    FxArgs a;
    std::memset(&a, 0, sizeof(a));
    a.chunk_rb = (const int32_t *)t->b_tc_crb.ptr;
    a.chunk_re = (const int32_t *)t->b_tc_cre.ptr;
    a.row_key = (const int32_t *)t->b_tc_rowkey.ptr;
    a.slot = (const int32_t *)t->b_tc_slot.ptr;
    a.tile_chunk = (const uint32_t *)t->b_tc_coff.ptr;
    a.M = (const int4 *)t->b_Mh.ptr;
    a.eM = (const int *)t->b_fx_em.ptr;
    a.ekey = (const int *)t->b_fx_ekey.ptr;
    a.etgt = (const int *)t->b_fx_et.ptr;
    a.img = (const int2 *)t->b_fx_img.ptr;
    a.acc = (u64 *)t->b_fx_acc.ptr;
    a.arrive = (unsigned *)(a.acc + (size_t)slots * ncolp);
    a.out.tile_tgt = (const int32_t *)t->b_tc_tgt.ptr;
    a.out.col = (const int32_t *)t->b_fx_el.ptr + Ly.E + Ly.first.size() + Ly.am.size();
    a.out.cls = a.out.col + Ly.col.size();
    a.out.level = (const int32_t *)t->b_level.ptr;
    a.out.sys = (const int32_t *)t->b_sys.ptr;
    a.out.rn = tb.h_rn;
    a.out.e_side = t->sys_eside_dev();
    a.out.L = L;
    a.out.s = t->s;
    a.out.ncol = Ly.ncol;
    a.out.nL = tb.nL;
    a.out.nLh = tb.nLh;
    a.out.unit = Ly.bits + 5;
    a.tiles = (int)t->tc_tiles;
    a.parts = (t->tc_G + kFxRows - 1) / kFxRows;
    a.K = Ly.K;
    a.with0 = Ly.n_lo == 0;
    a.nq = Ly.nq;
    a.E = Ly.E;
    a.ncolp = ncolp;
    for (int g = 0; g < Ly.groups; ++g) {
        const int w = Ly.owner[g], k = a.ng[w]++;
        a.g_off[w][k] = Ly.first[g];
        a.g_mq[w][k] = (Ly.first[g + 1] - Ly.first[g]) / 8;
        a.g_col[w][k] = 4 * g;
        a.g_cls[w][k] = Ly.cls[g];
    }
    const size_t smem = std::max(fx_smem(Ly), 32 * (size_t)Ly.groups * kFxPad);   // the last block's turn
    auto go = [&](auto kern) {
        allow_max_dynamic_smem(kern);
        launch_next(st, kern, (unsigned)(4 * t->tc_chunks * a.parts), kFxThreads, smem, a);
    };
    switch (Ly.cap) {
    case 4: go(k_m2l_fx<4>); break;
    case 6: go(k_m2l_fx<6>); break;
    case 8: go(k_m2l_fx<8>); break;
    case 12: go(k_m2l_fx<12>); break;
    default: go(k_m2l_fx<16>); break;
    }
    ++t->launches;
    return cuda_check(t, cudaGetLastError(), "fixed-point M2L");
}

}  // namespace fmm
