// operators.cu -- derivative tables and the expansion operators (FP64).
//
// Conventions (paper §2, read as stated in the header):
//   P2M  M_m(z)   = sum_j sum_{|a|=s, a<=m} (z - x_j)^(m-a)/(m-a)! S_{j,a}   (Eq. (5))
//   M2M  M_n(z')  = sum_{k<=n} (z' - z)^k/k! M_{n-k}(z)                        (Eq. (4))
//   M2L  L_n(zt)  = sum_{m, |n|+|m|<=p+s} D_{n+m}(zt - zs) M_m(zs)            (Eq. (8))
//   L2L  L_n(z')  = sum_{|n+k|<=p} (z' - z)^k/k! L_{n+k}(z)
//   L2P  phi = sum_n (x-z)^n/n! L_n,  d_k phi = sum_{n>=e_k} (x-z)^(n-e_k)/(n-e_k)! L_n
//                                                                             (Eqs. (9), (10))
// D_n(R) = grad^n (1/|R|) is generated once per distinct M2L offset.
#include <algorithm>
#include <cstring>
#include <stdexcept>
#include <mutex>

#include "fmm_internal.cuh"
#include "fx64.cuh"

namespace fmm {

MultiIndex::MultiIndex()
{
    std::memset(lut, 0xff, sizeof(lut));
    int i = 0;
    for (int k = 0; k <= kMaxOrder; ++k)
        for (int a = 0; a <= k; ++a)          // a = ny + nz
            for (int z = 0; z <= a; ++z) {
                nx[i] = k - a; ny[i] = a - z; nz[i] = z;
                lut[k - a][a - z][z] = (int16_t)i;
                ++i;
            }
}

const MultiIndex &multi_index()
{
    static MultiIndex mi;
    return mi;
}

void build_tables(OpTables &T, int s, int s_hi, int p, int n_lo, int m2l_threads, bool harmonic)
{
    const MultiIndex &I = multi_index();
    T.s = s; T.p = p; T.n_lo = n_lo; T.harmonic = harmonic;
    // source terms a: the orders s..s_hi, graded indices from ntot(s - 1) on
    T.nS = ntot(s_hi) - ntot(s - 1); T.m0 = ntot(s - 1); T.nM = ntot(p + s) - T.m0; T.nL = ntot(p);
    T.nD = ntot(p + s);
    const int nK = ntot(p);                   // shift / particle monomials |k| <= p

    T.p2m_terms.assign((size_t)T.nM * T.nS, -1);
    for (int mi = 0; mi < T.nM; ++mi) {
        const int m = mi + T.m0;
        for (int ai = 0; ai < T.nS; ++ai) {
            const int a = ai + T.m0;
            int kx = I.nx[m] - I.nx[a], ky = I.ny[m] - I.ny[a], kz = I.nz[m] - I.nz[a];
            if (kx >= 0 && ky >= 0 && kz >= 0) T.p2m_terms[(size_t)mi * T.nS + ai] = I(kx, ky, kz);
        }
    }

    T.m2m_off.assign(1, 0); T.m2m_kq.clear();
    for (int ni = 0; ni < T.nM; ++ni) {
        const int n = ni + T.m0;
        for (int qi = 0; qi < T.nM; ++qi) {
            const int q = qi + T.m0;
            int kx = I.nx[n] - I.nx[q], ky = I.ny[n] - I.ny[q], kz = I.nz[n] - I.nz[q];
            if (kx < 0 || ky < 0 || kz < 0) continue;
            T.m2m_kq.push_back(I(kx, ky, kz) | qi << 16);
        }
        T.m2m_off.push_back((int)T.m2m_kq.size());
    }
    const int nG = ntot(p - 1);
    T.l2p_grad.assign((size_t)3 * std::max(nG, 0), 0);
    for (int k = 0; k < nG; ++k) {
        T.l2p_grad[3 * k + 0] = I(I.nx[k] + 1, I.ny[k], I.nz[k]);
        T.l2p_grad[3 * k + 1] = I(I.nx[k], I.ny[k] + 1, I.nz[k]);
        T.l2p_grad[3 * k + 2] = I(I.nx[k], I.ny[k], I.nz[k] + 1);
    }

    // L2P: the k of |k| <= p, then of |k| <= p - 1, in the order of nested loops
    // over k_x, k_y, k_z
    T.l2p_ord.clear();
    for (int q : {p, p - 1})
        for (int x = 0; x <= q; ++x)
            for (int y = 0; y <= q - x; ++y)
                for (int z = 0; z <= q - x - y; ++z) T.l2p_ord.push_back(I(x, y, z));

    // ---- harmonic M2L (§3.1 harmonic derivatives).  Since D_{k+2x} + D_{k+2y}
    // + D_{k+2z} = 0 for every k, a term D_{n+m} M_m with m_z >= 2 equals
    // -(D_{n+m-2z+2x} + D_{n+m-2z+2y}) M_m, a pair of terms of the same degree
    // |m|, hence inside the same truncation |n| + |m| <= p + s: moving M_m onto
    // those two m (in decreasing m_z) leaves the m with m_z <= 1 only, 2k+1
    // per degree k.  Likewise L_n with n_z >= 2 is -L_{n+2x-2z} - L_{n+2y-2z}
    // (same degree, same m range).  The same sums, mathematically.
    T.h_rm.clear();
    for (int mi = 0; mi < T.nM; ++mi)
        if (!harmonic || I.nz[mi + T.m0] <= 1) T.h_rm.push_back(mi);
    T.nMh = (int)T.h_rm.size();
    std::vector<int> r_of(T.nM, -1);
    for (int r = 0; r < T.nMh; ++r) r_of[T.h_rm[r]] = r;
    T.h_fold.clear(); T.h_fold_off.assign(1, 0);
    T.h_unfold.clear(); T.h_unfold_off.assign(1, 0);
    if (harmonic) {
        for (int z = p + s - 2; z >= 0; --z) {
            for (int mi = 0; mi < T.nM; ++mi) {
                const int m = mi + T.m0;
                if (I.nz[m] != z) continue;
                const int a = I.nx[m] >= 2 ? I(I.nx[m] - 2, I.ny[m], I.nz[m] + 2) - T.m0 : -1;
                const int b = I.ny[m] >= 2 ? I(I.nx[m], I.ny[m] - 2, I.nz[m] + 2) - T.m0 : -1;
                if (a < 0 && b < 0) continue;
                T.h_fold.insert(T.h_fold.end(), {mi, a, b});
            }
            T.h_fold_off.push_back((int)T.h_fold.size() / 3);
        }
        for (int z = 2; z <= p; ++z) {
            for (int n = 0; n < T.nL; ++n) {
                if (I.nz[n] != z) continue;
                T.h_unfold.insert(T.h_unfold.end(), {n, I(I.nx[n] + 2, I.ny[n], z - 2),
                                                     I(I.nx[n], I.ny[n] + 2, z - 2)});
            }
            T.h_unfold_off.push_back((int)T.h_unfold.size() / 3);
        }
    }
    // stored locals: the n with n_z <= 1 when harmonic (the others follow from
    // the identity wherever the full expansion is needed), all of them otherwise
    T.h_rn.clear();
    for (int n = 0; n < T.nL; ++n)
        if (!harmonic || I.nz[n] <= 1) T.h_rn.push_back(n);
    T.nLh = (int)T.h_rn.size();

    T.l2l_ix.assign(2 * (size_t)((nK + 3) / 4) * T.nLh, T.nL | T.nL << 16);
    for (int r = 0; r < T.nLh; ++r) {
        const int n = T.h_rn[r];
        for (int k = 0, t = 0; k < nK; ++k) {                 // the k that fit come first
            const int x = I.nx[n] + I.nx[k], y = I.ny[n] + I.ny[k], z = I.nz[n] + I.nz[k];
            if (x + y + z > p) continue;
            int &w = T.l2l_ix[2 * ((size_t)(t / 4) * T.nLh + r) + (t % 4) / 2];
            w = t & 1 ? (w & 0xffff) | I(x, y, z) << 16 : (w & ~0xffff) | I(x, y, z);
            ++t;
        }
    }

    // ---- M2L: flat (n, m) term list in n order, cut into equal per-thread
    // chunks; each maximal same-n run inside a chunk owns one partial slot.
    // m is the position r in the kept list h_rm (all m when not harmonic).
    struct Term { int n, m, d; };
    std::vector<Term> terms;
    for (int n = 0; n < T.nL; ++n) {
        const int kn = I.nx[n] + I.ny[n] + I.nz[n];
        if (kn < n_lo || (harmonic && I.nz[n] > 1)) continue;
        for (int r = 0; r < T.nMh; ++r) {
            const int m = T.h_rm[r] + T.m0;
            if (kn + I.nx[m] + I.ny[m] + I.nz[m] > p + s) continue;
            terms.push_back({n, r, I(I.nx[n] + I.nx[m], I.ny[n] + I.ny[m], I.nz[n] + I.nz[m])});
        }
    }
    const int W = (int)terms.size(), Tn = m2l_threads;
    const int cap = std::max(1, (W + Tn - 1) / Tn);
    T.m2l_threads = Tn; T.m2l_T = cap;
    T.m2l_desc.assign((size_t)cap * Tn, 0xffffffffu);
    std::vector<std::vector<int>> red(T.nL);
    int max_slots = 0;
    for (int j = 0; j < Tn; ++j) {
        const int b = j * cap, e = std::min(W, b + cap);
        int slot = -1;
        for (int i = b; i < e; ++i) {
            if (i == b || terms[i].n != terms[i - 1].n) {
                ++slot;
                red[terms[i].n].push_back(slot * Tn + j);
            }
            const bool flush = (i + 1 == e) || terms[i + 1].n != terms[i].n;
            T.m2l_desc[(size_t)(i - b) * Tn + j] =
                (uint32_t)terms[i].m | ((uint32_t)terms[i].d << 9) | ((uint32_t)flush << 18) |
                ((uint32_t)slot << 19);
        }
        max_slots = std::max(max_slots, slot + 1);
    }
    T.m2l_slots = max_slots;
    T.m2l_red_off.assign(1, 0); T.m2l_red_src.clear();
    for (int n = 0; n < T.nL; ++n) {
        for (int v : red[n]) T.m2l_red_src.push_back(v);
        T.m2l_red_off.push_back((int)T.m2l_red_src.size());
    }
}

namespace {

constexpr int kM2LThreads = 128;
constexpr int kM2LBatch = 16;
constexpr size_t kM2LSmemMax = 226 * 1024;   // next to the kernel's static shared memory

__constant__ int8_t c_nx[kMaxTot], c_ny[kMaxTot], c_nz[kMaxTot];


// ---------------------------------------------------- derivative tables
// r^2 D_n = -(2 n_i - 1) R_i D_{n-e_i} - (n_i - 1)^2 D_{n-2e_i}
//           - sum_{j != i} [ 2 n_j R_j D_{n-e_j} + n_j (n_j - 1) D_{n-2e_j} ],
// i = first axis with n_i >= 1 (Leibniz' rule on r^2 d_i(1/r) = -R_i / r).
// Rows are unit-free: D_k(v) at the integer offset v of the key; a pair with
// finer half-cell u uses u^-(|k|+1) D_k(v), applied exactly as an exponent shift.
// One warp per distinct offset: the row is built shell by shell in the warp's
// shared memory (an entry of shell |n| reads shells |n| - 1 and |n| - 2 only,
// so a shell's entries are independent and the lanes take them side by side),
// then stored.  Each entry is the same arithmetic as a one-thread recurrence.
__global__ void k_dtables(const uint64_t *dkeys, int64_t ndoff, int nD, const int32_t *lut,
                          double *D)
{
    extern __shared__ double dsm[];
    const int lane = threadIdx.x & 31;
    const int64_t r = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (r >= ndoff) return;
    double *Dr = dsm + (threadIdx.x >> 5) * (int64_t)nD;
    const uint64_t key = dkeys[r];
    double R[3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
        R[i] = (double)((long long)((key >> (34 - 17 * i)) & 0x1ffffull) - kKeyBias);
    const double r2 = R[0] * R[0] + R[1] * R[1] + R[2] * R[2];
    const double inv_r2 = 1.0 / r2;
    if (lane == 0) Dr[0] = rsqrt(r2);
    __syncwarp();
    const int L = kMaxOrder + 1;
    for (int sh = 1, s0 = 1; s0 < nD; ++sh) {
        const int s1 = min(nD, (sh + 1) * (sh + 2) * (sh + 3) / 6);      // shell sh: [s0, s1)
        for (int idx = s0 + lane; idx < s1; idx += 32) {
            const int n[3] = {c_nx[idx], c_ny[idx], c_nz[idx]};
            const int i = n[0] ? 0 : (n[1] ? 1 : 2);
            int m[3] = {n[0], n[1], n[2]};
            m[i] -= 1;
            double acc = -(2.0 * n[i] - 1.0) * R[i] * Dr[lut[(m[0] * L + m[1]) * L + m[2]]];
            if (n[i] >= 2) {
                int q[3] = {m[0], m[1], m[2]};
                q[i] -= 1;
                acc -= (double)((n[i] - 1) * (n[i] - 1)) * Dr[lut[(q[0] * L + q[1]) * L + q[2]]];
            }
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                if (j == i || n[j] == 0) continue;
                int q[3] = {n[0], n[1], n[2]};
                q[j] -= 1;
                acc -= 2.0 * n[j] * R[j] * Dr[lut[(q[0] * L + q[1]) * L + q[2]]];
                if (n[j] >= 2) {
                    q[j] -= 1;
                    acc -= (double)(n[j] * (n[j] - 1)) * Dr[lut[(q[0] * L + q[1]) * L + q[2]]];
                }
            }
            Dr[idx] = acc * inv_r2;
        }
        __syncwarp();
        s0 = s1;
    }
    for (int k = lane; k < nD; k += 32) D[r * nD + k] = Dr[k];
}

// per-axis scaled powers d^j / j!, j <= P, then monomials d^k / k! = ax[kx] ay[ky] az[kz]
__constant__ double c_invint[kMaxOrder + 2];     // 1/j

__device__ __forceinline__ void axis_powers(double d, int P, double *out)
{
    double v = 1.0;
    out[0] = 1.0;
    for (int j = 1; j <= P; ++j) {
        v = v * d * c_invint[j];
        out[j] = v;
    }
}

// ------------------------------------------------------------------ P2M
constexpr int kP2MThreads = 128;
constexpr int kP2MChunk = 32;             // particles staged at a time
constexpr int kP2MRun = 16 * kP2MChunk;   // particles whose sums share 64 bits
// source terms of one particle: the kernel is instantiated for 3, 6 and 10 (one
// order up to a dipole, a quadrupole, mixed orders) and takes the smallest that fits

// Fixed point at the particles (P2M, L2P).  The FP64 pipe (64 clocks a warp
// instruction) bound both; inside a leaf the displacements have a common range,
// so their powers and the sums run on the integer pipes (fx64.cuh).
//   displacement d = u 2^re, |u| <= 1 + 2^-10: u and the monomials u^k at 2^60
//   monomials in the sums at 2^56 (error below 2^-56), as limbs h 2^26 + l
//   moments at 2^53 of a power of two above the largest, so that the sum over a
//   chunk of 32 particles stays below 2^63; the chunks' sums are shifted right,
//   rounded, by the bits their number needs: at most four, as after 16 chunks they
//   go to the FP64 row and start again (leaves of any size: deep ones of coincident
//   points, or a large max_leaf)
//   L_n rho^k / k! at 2^56 of a power of two above the sum of their magnitudes,
//   so that the sum over them stays below 2^61
using fx::I2;
using fx::s64;
using fx::madp;

constexpr int kNoExp = -100000, kBadExp = 1 << 24;        // all zero; an infinity or a NaN

// |x| < 2^e
__device__ __forceinline__ int mag_exp(double x)
{
    const int hi = __double2hiint(x) & 0x7fffffff;
    return (hi | __double2loint(x)) ? (hi < 0x7ff00000 ? (hi >> 20) - 1022 : kBadExp) : kNoExp;
}
// |d| <= 2^e (1 + 2^-10): a particle on its cell's face, with its rounding, is
// within the half side, so that u^k keeps all of its bits
__device__ __forceinline__ int disp_exp(double d)
{
    const int hi = __double2hiint(d) & 0x7fffffff;
    return (hi | __double2loint(d)) ? max(hi - 1024, 0) / (1 << 20) - 1022 : kNoExp;
}
// A bound of a sum of magnitudes without FP64 operations: the leading 21 bits
// of each, rounded up, in units of 2^(top - 21), top = mag_exp of the largest
__device__ __forceinline__ unsigned long long mag_units(double x, int up, int top)
{
    const int hi = __double2hiint(x) & 0x7fffffff, ex = hi >> 20, sh = top - up - (ex - 1022);
    return (hi | __double2loint(x)) ? ((sh < 22 ? (unsigned)(hi & 0xfffff | 1 << 20) >> sh : 0u) + 1u) : 0u;
}
struct MagSum {
    int top;                              // kNoExp: no term; kBadExp: one is not finite
    unsigned long long units;
};
// the power of two above the sums of several parts
__device__ __forceinline__ int mag_sum_exp(const MagSum *m, int parts, int stride)
{
    int top = kNoExp;
    for (int i = 0; i < parts; ++i) top = max(top, m[i * stride].top);
    if (top == kNoExp || top >= kBadExp / 2) return top == kNoExp ? kNoExp : kBadExp;
    unsigned long long u = 0;
    for (int i = 0; i < parts; ++i) {
        const int sh = top - m[i * stride].top;
        u += (sh < 64 ? m[i * stride].units >> sh : 0ull) + (sh > 0);
    }
    return top - 21 + (64 - __clzll((long long)u));
}
__device__ __forceinline__ MagSum warp_mag_sum(unsigned long long u, int top)
{
    for (int o = 16; o > 0; o >>= 1) u += __shfl_xor_sync(0xffffffffu, u, o);
    return {top, u};
}
// x 2^e for a normal x, FP64 multiplications only where the result is not normal
__device__ __forceinline__ double scale2(double x, int e)
{
    const int hi = __double2hiint(x), ex = ((hi >> 20) & 0x7ff) + e;
    if (ex > 0 && ex < 0x7ff) return __hiloint2double(hi + (e << 20), __double2loint(x));
    return ldexp(x, e);
}
__device__ __forceinline__ I2 bal_of(int2 v) { return {v.x, v.y}; }
// a b / 2^60 for |a|, |b| < 2^60.1 (error below 2^-57 of the range)
__device__ __forceinline__ s64 mul60(I2 a, I2 b)
{
    const s64 c = madp(a.h, b.l, madp(a.l, b.h, 1ll << 27));
    return (madp(a.h, b.h, 0) << 4) + (c >> 28);
}
// 2^60 -> limbs at 2^56
__device__ __forceinline__ I2 limbs60(s64 m)
{
    const int h = (int)((m + (1ll << 29)) >> 30);
    return {h, (int)((m - ((s64)h << 30)) >> 4)};
}
// x 2^sc as limbs (|x 2^sc| < 2^56.5)
__device__ __forceinline__ int2 limbs_of(double x, int sc)
{
    const s64 v = fx::fix64(x, sc);
    const int h = (int)((v + (1ll << 25)) >> 26);
    return make_int2(h, (int)(v - ((s64)h << 26)));
}
__device__ __forceinline__ void axis_powers_fx(double d, int re, int P, int2 *out)
{
    const I2 u = fx::bal(fx::fix64(d, 60 - re));
    I2 v = fx::bal(1ll << 60);
    out[0] = make_int2(v.h, v.l);
    for (int j = 1; j <= P; ++j) {
        v = fx::bal(mul60(v, u));
        out[j] = make_int2(v.h, v.l);
    }
}

// 1 / (k_x! k_y! k_z!)
__device__ __forceinline__ double inv_factorial(const DevTables &tb, int k)
{
    return __hiloint2double(__ldg(tb.inv_fact + 2 * k + 1), __ldg(tb.inv_fact + 2 * k));
}

// The sums of a run that is not its leaf's last, as doubles into the leaf's row, and cleared
__device__ __noinline__ void p2m_run_end(s64 *G, int nK, int nS, const int *s_es, int re, int room, const int *mis,
                                         const int *inv_fact, const int *terms, int nM, bool first, double *M)
{
    double *Gd = (double *)G;
    for (int k = threadIdx.x; k < nK; k += kP2MThreads) {
        const int ek = mi_shell(mi_at(mis, k)) * re;
        const double f = __hiloint2double(__ldg(inv_fact + 2 * k + 1), __ldg(inv_fact + 2 * k));
        for (int a = 0; a < nS; ++a) {
            const s64 g = G[k * nS + a];
            Gd[k * nS + a] = g ? scale2((double)g * f, s_es[a] + ek + room - 57) : 0.0;
        }
    }
    __syncthreads();
    for (int m = threadIdx.x; m < nM; m += kP2MThreads) {
        double acc = first ? 0.0 : M[m];
        for (int a = 0; a < nS; ++a) {
            const int k = terms[m * nS + a];
            if (k >= 0) acc += Gd[k * nS + a];
        }
        M[m] = acc;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < nK * nS; k += kP2MThreads) G[k] = 0;      // the staging's barrier comes next
}

// One block per leaf.  A thread owns monomials k and sums u^k S_a over the
// particles for every source term a (a moment's limbs read by all lanes at
// once); the multipole m is then the sum over a of the terms m - a.  Per
// particle 84 monomials (p = 6) of two products and nS sums of three
// multiply-adds each, where the FP64 form issued 570 operations: upward pass
// (with the M2M of the time) 1.69 -> 0.81 ms at 1M dipoles, p = 6; 0.50 -> 0.26 ms
// at 200k charges and dipoles, p = 6; 2.22 -> 0.79 ms at 96 quadrupole systems, p = 5.
template <int kMaxSrc>
__device__ __forceinline__ void p2m_leaf(int c, const int32_t *begin, const int32_t *end,
                                         const double *centre, const double *px, const double *py,
                                         const double *pz, const double *S, const DevTables &tb,
                                         double *M, double *sm)
{
    __shared__ int s_re[kP2MThreads / 32], s_es[10];
    const int P = tb.p, P1 = tb.p + 1, nK = tb.nK, nS = tb.nS;
    s64 *G = (s64 *)sm;                                 // [nK][nS] sums, then their doubles
    int2 *pw = (int2 *)(G + nK * nS);                   // [chunk][3][P+1] powers at 2^60, balanced halves
    int2 *Sx = pw + kP2MChunk * 3 * P1;                 // [chunk][nS] moments
    const int b = begin[c], e = end[c], n = e - b;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const double z0 = centre[3 * c], z1 = centre[3 * c + 1], z2 = centre[3 * c + 2];
    auto disp = [&](int j, int ax) {
        return ax == 0 ? z0 - px[j] : (ax == 1 ? z1 - py[j] : z2 - pz[j]);
    };
    // exponents: the largest displacement, the largest of each moment
    int re = kNoExp;
    double d0 = 0.0;                                    // the thread's displacement of the first chunk
    for (int t = threadIdx.x; t < 3 * n; t += kP2MThreads) {
        const double d = disp(b + t / 3, t % 3);
        if (t == threadIdx.x) d0 = d;
        re = max(re, disp_exp(d));
    }
    re = __reduce_max_sync(0xffffffffu, re);
    if (lane == 0) s_re[w] = re;
    for (int a = w; a < nS; a += kP2MThreads / 32) {
        int top = kNoExp;
        for (int j = b + lane; j < e; j += 32) top = max(top, mag_exp(S[(int64_t)j * nS + a]));
        top = __reduce_max_sync(0xffffffffu, top);
        if (lane == 0) s_es[a] = top;
    }
    for (int k = threadIdx.x; k < nK * nS; k += kP2MThreads) G[k] = 0;
    __syncthreads();
    re = max(max(s_re[0], s_re[1]), max(s_re[2], s_re[3]));
    const int room = 32 - __clz((min(n, kP2MRun) - 1) / kP2MChunk);      // 2^room > chunks of a run - 1
    const int half = (1 << room) >> 1;
    for (int j0 = b; j0 < e; j0 += kP2MChunk) {
        const int nj = min(kP2MChunk, e - j0);
        for (int t = threadIdx.x; t < 3 * nj; t += kP2MThreads)
            axis_powers_fx(j0 == b ? d0 : disp(j0 + t / 3, t % 3), re, P, pw + t * P1);
        for (int t = threadIdx.x; t < nj * nS; t += kP2MThreads) {
            const int es = s_es[t % nS];
            Sx[t] = es == kBadExp ? make_int2(0, 0) : limbs_of(S[(int64_t)j0 * nS + t], 53 - es);
        }
        __syncthreads();
        for (int k = threadIdx.x; k < nK; k += kP2MThreads) {
            const int v = mi_at(tb.mi, k);
            const int2 *x = pw + mi_nx(v), *y = pw + P1 + mi_ny(v), *z = pw + 2 * P1 + mi_nz(v);
            s64 a1[kMaxSrc], a0[kMaxSrc];
#pragma unroll
            for (int a = 0; a < kMaxSrc; ++a) {
                a1[a] = half;
                a0[a] = 1ll << 25;
            }
            for (int j = 0; j < nj; ++j) {
                const int o = 3 * P1 * j;
                const I2 m = limbs60(mul60(fx::bal(mul60(bal_of(x[o]), bal_of(y[o]))), bal_of(z[o])));
#pragma unroll
                for (int a = 0; a < kMaxSrc; ++a)
                    if (a < nS) {
                        const int2 q = Sx[j * nS + a];
                        a1[a] = madp(m.h, q.x, a1[a]);
                        a0[a] = madp(m.h, q.y, a0[a]);
                        a0[a] = madp(m.l, q.x, a0[a]);
                    }
            }
#pragma unroll
            for (int a = 0; a < kMaxSrc; ++a)
                if (a < nS) G[k * nS + a] += (a1[a] + (a0[a] >> 26)) >> room;
        }
        __syncthreads();
        if ((j0 - b) % kP2MRun == kP2MRun - kP2MChunk && j0 + kP2MChunk < e)
            p2m_run_end(G, nK, nS, s_es, re, room, tb.mi, tb.inv_fact, tb.p2m_terms, tb.nM, j0 - b < kP2MRun,
                        M + (int64_t)c * tb.nM);
    }
    // the sums as doubles: u^k S_a 2^(57 - room) -> (z - x)^k / k! S_a
    double *Gd = (double *)G;
    for (int k = threadIdx.x; k < nK; k += kP2MThreads) {
        const int ek = mi_shell(mi_at(tb.mi, k)) * re;
        const double f = inv_factorial(tb, k);
        for (int a = 0; a < nS; ++a) {
            const int es = s_es[a];
            const s64 g = G[k * nS + a];
            Gd[k * nS + a] = es == kBadExp ? __longlong_as_double(0x7ff8000000000000ll)
                                           : (g ? scale2((double)g * f, es + ek + room - 57) : 0.0);
        }
    }
    __syncthreads();
    for (int mi = threadIdx.x; mi < tb.nM; mi += kP2MThreads) {
        double acc = n > kP2MRun ? M[(int64_t)c * tb.nM + mi] : 0.0;     // the runs before, by the same thread
        for (int a = 0; a < nS; ++a) {
            const int k = tb.p2m_terms[mi * nS + a];
            if (k >= 0) acc += Gd[k * nS + a];
        }
        M[(int64_t)c * tb.nM + mi] = acc;
    }
}

// ------------------------------------------------------------------ M2M
// The multipole of parent cell c from its children (Eq. (4) with the sign of
// R2), one axis at a time: the children's centres differ along an axis only by
// the child's bit, so the two of each pair are shifted along x and added, then
// the four sums along y, then along z.  14 axis shifts of some three terms a
// component in place of 8 shifts of (n_x+1)(n_y+1)(n_z+1), and sums of 8 terms
// in a row in place of 8 x 40: upward pass 0.81 -> 0.48 ms at 1M dipoles, p = 6;
// 1.08 -> 0.53 ms at 262k Plummer, p = 8; 0.33 -> 0.14 ms at 125k, p = 6.  ldcg:
// the children's rows may have been written by other blocks of the same launch.
__device__ __forceinline__ void m2m_cell(int c, const int32_t *child, const int32_t *nchild,
                                         const int32_t *cx, const int32_t *cy, const int32_t *cz,
                                         const double *centre, const DevTables &tb, double *M,
                                         double *sm)
{
    const int P1 = tb.p + 1, nM = tb.nM, nch = nchild[c], ch0 = child[c];
    double *pw = sm;                    // [3][2][P+1]: (z'_d - z_d)^j / j! of the lower and upper children
    double *A = pw + 6 * P1;            // [8][nM] children by bits x + 2 y + 4 z, then [2][nM]
    double *B = A + 8 * nM;             // [4][nM]
    unsigned have = 0, done = 0;        // bits of the children there are; powers formed
    for (int i = 0; i < nch; ++i) {
        const int ch = ch0 + i, slot = (cx[ch] & 1) | (cy[ch] & 1) << 1 | (cz[ch] & 1) << 2;
        have |= 1u << slot;
        if (threadIdx.x < 3) {
            const int up = (slot >> threadIdx.x) & 1;
            if (!(done >> up & 1u))
                axis_powers(centre[3 * c + threadIdx.x] - centre[3 * ch + threadIdx.x], tb.p,
                            pw + (2 * threadIdx.x + up) * P1);
            done |= 1u << up;
        }
        for (int t = threadIdx.x; t < nM; t += blockDim.x) A[slot * nM + t] = __ldcg(M + (int64_t)ch * nM + t);
    }
    __syncthreads();
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        const int outs = 4 >> ax;
        const double *in = ax == 1 ? B : A;
        double *out = ax == 0 ? B : (ax == 1 ? A : M + (int64_t)c * nM);
        for (int t = threadIdx.x; t < outs * nM; t += blockDim.x) {
            const int g = t / nM, ni = t - g * nM;
            const int v = mi_at(tb.mi, ni + tb.m0), sh0 = mi_shell(v);
            const int na = ax == 0 ? mi_nx(v) : (ax == 1 ? mi_ny(v) : mi_nz(v));
            const int js = min(na, sh0 - tb.s);
            double acc = 0.0;
#pragma unroll
            for (int up = 0; up < 2; ++up) {
                if (!(have >> (2 * g + up) & 1u)) continue;
                const double *p = pw + (2 * ax + up) * P1, *x = in + (2 * g + up) * nM + ni;
                // n - j e: one shell lower, at the same place in it (x), a row up
                // (y), a row and a place (z)
                int sh = sh0, a = mi_ny(v) + mi_nz(v);
                for (int j = 0; j <= js; ++j) {
                    acc = fma(p[j], *x, acc);
                    x -= sh * (sh + 1) / 2 + (ax == 0 ? 0 : (ax == 1 ? a : a + 1));
                    --sh;
                    --a;
                }
            }
            out[t] = acc;
        }
        have = (have | have >> 1) & 0x55u;          // pairs with a child
        have = (have | have >> 1) & 0x33u;
        have = (have | have >> 2) & 0x0fu;
        if (ax < 2) __syncthreads();
    }
}

// The upward pass in one launch: block b forms the multipole of leaf b (P2M,
// Eq. (3)), then climbs -- the block whose child arrives last at a parent
// (a counter per cell) forms that parent's multipole (M2M), and so on up to
// the root.  No block waits on another; every parent is formed exactly once,
// from its finished children, in the same order as a level-by-level pass.
// arrive[] starts at zero and is left at zero (the winner resets it).
template <int kMaxSrc>
__global__ void __launch_bounds__(kP2MThreads)
k_upward(const int32_t *leaves, const int32_t *begin, const int32_t *end, const int32_t *parent,
         const int32_t *child, const int32_t *nchild, const int32_t *cx, const int32_t *cy,
         const int32_t *cz, const double *centre, const double *px, const double *py,
         const double *pz, const double *S, DevTables tb, double *M, unsigned *arrive)
{
    pdl_wait();
    extern __shared__ double sm[];
    __shared__ int s_go;
    int c = leaves[blockIdx.x];
    p2m_leaf<kMaxSrc>(c, begin, end, centre, px, py, pz, S, tb, M, sm);
    for (;;) {
        const int pa = parent[c];
        if (pa < 0) break;
        __syncthreads();                       // every thread's row of c is written
        if (threadIdx.x == 0) {
            __threadfence();                   // ... and visible before the arrival counts
            const unsigned n = atomicAdd(&arrive[pa], 1u) + 1u;
            const bool last = n == (unsigned)nchild[pa];
            if (last) {
                arrive[pa] = 0u;
                __threadfence();               // the other children's rows are visible now
            }
            s_go = last;
        }
        __syncthreads();
        if (!s_go) break;
        m2m_cell(pa, child, nchild, cx, cy, cz, centre, tb, M, sm);
        c = pa;
    }
}

// ------------------------------------------------------------------ M2L
// One block per target cell.  Sources are taken `batch` at a time (16; 8 where the full
// Cartesian sums of p + s = 12 leave no shared memory for more): their
// multipoles and derivative-table rows are staged in shared memory, then
// each thread walks its fixed chunk of (n, m) terms, accumulating
// D_{n+m} M_m over the staged sources, and flushes each finished n-run to its
// partial slot.  Partials are summed per n in a fixed order at the end.
// x * 2^e for normal x (exponent field arithmetic; zeros stay zero)
__device__ __forceinline__ double scale_pow2(double x, int e)
{
    const long long b = __double_as_longlong(x);
    return (b & 0x7ff0000000000000ll) ? __longlong_as_double(b + ((long long)e << 52)) : x;
}

// One warp per cell: the row of M in shared memory (FP64), the fold levels of
// the harmonic M2L in order (an entry reads only entries of the level two
// z-steps up, final by then), the kept entries written in graded order.
template <typename Tm>
__global__ void __launch_bounds__(128)
k_fold_m(const Tm *M, int ldM, int64_t nc, DevTables tb, Tm *Mh, int ldH)
{
    pdl_wait();
    extern __shared__ double fsm[];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t c = blockIdx.x * 4ll + w;
    if (c >= nc) return;                 // whole warps; no block barrier below
    double *v = fsm + w * tb.nM;
    for (int m = lane; m < tb.nM; m += 32) v[m] = (double)M[c * ldM + m];
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
    for (int r = lane; r < tb.nMh; r += 32) Mh[c * ldH + r] = (Tm)v[tb.h_rm[r]];
}

__global__ void __launch_bounds__(kM2LThreads)
k_m2l(const int32_t *off, const int32_t *src, const int32_t *didx, const int32_t *level,
      const int32_t *sys, const int *e_side, const double *M, const double *D, DevTables tb,
      double *L, int batch)
{
    pdl_wait();
    extern __shared__ double sm[];
    const int c = blockIdx.x;
    const int b = off[c], e = off[c + 1];
    if (b == e) return;
    // M: the kept (folded, when harmonic) multipole rows, nMh per cell
    const int nM = tb.nMh, nD = tb.nD, T = tb.m2l_T, Tn = kM2LThreads;
    const int ldM = nM | 1, ldD = nD | 1;              // odd strides spread banks
    double *Msm = sm;                                  // [batch][ldM]
    double *Dsm = Msm + batch * ldM;                   // [batch][ldD]
    double *part = Dsm + batch * ldD;                  // [slots][Tn]
    uint32_t *desc = (uint32_t *)(part + tb.m2l_slots * Tn);   // [T][Tn]
    const int tid = threadIdx.x;
    const int lt = level[c], es = e_side[sys[c]];
    __shared__ int bsrc[kM2LBatch], bdidx[kM2LBatch], beu[kM2LBatch];
    for (int i = tid; i < T * Tn; i += Tn) desc[i] = tb.m2l_desc[i];
    for (int i = tid; i < tb.m2l_slots * Tn; i += Tn) part[i] = 0.0;
    for (int k0 = b; k0 < e; k0 += batch) {
        const int kb = min(batch, e - k0);
        __syncthreads();
        if (tid < kb) {                    // batch metadata, loaded in parallel
            const int s = src[k0 + tid];
            bsrc[tid] = s;
            bdidx[tid] = didx[k0 + tid];
            // u = side / 2^(lf+1): D_k(u v) = 2^(-(|k|+1) log2 u) D_k(v)
            beu[tid] = es - max(lt, level[s]) - 1;
        }
        __syncthreads();
        for (int k = 0; k < kb; ++k) {
            const double *Ms = M + (int64_t)bsrc[k] * nM;
            for (int m = tid; m < nM; m += Tn) Msm[k * ldM + m] = Ms[m];
            const double *Dk = D + (int64_t)bdidx[k] * nD;
            const int eu = beu[k];
            for (int d = tid; d < nD; d += Tn)
                Dsm[k * ldD + d] = scale_pow2(Dk[d], -(mi_shell(mi_at(tb.mi, d)) + 1) * eu);
        }
        __syncthreads();
        double acc = 0.0;
        for (int t = 0; t < T; ++t) {
            const uint32_t u = desc[t * Tn + tid];
            if (u == 0xffffffffu) break;
            const double *Mp = Msm + (u & 511u);
            const double *Dp = Dsm + ((u >> 9) & 511u);
            int k = 0;
            for (; k + 4 <= kb; k += 4) {
                acc = fma(Dp[k * ldD], Mp[k * ldM], acc);
                acc = fma(Dp[(k + 1) * ldD], Mp[(k + 1) * ldM], acc);
                acc = fma(Dp[(k + 2) * ldD], Mp[(k + 2) * ldM], acc);
                acc = fma(Dp[(k + 3) * ldD], Mp[(k + 3) * ldM], acc);
            }
            for (; k < kb; ++k) acc = fma(Dp[k * ldD], Mp[k * ldM], acc);
            if (u & (1u << 18)) {
                part[(u >> 19) * Tn + tid] += acc;
                acc = 0.0;
            }
        }
    }
    __syncthreads();
    // the stored components (n_z <= 1 when harmonic, the traceless form)
    for (int r = tid; r < tb.nLh; r += Tn) {
        const int n = tb.h_rn[r];
        double v = 0.0;
        for (int q = tb.m2l_red_off[n]; q < tb.m2l_red_off[n + 1]; ++q) v += part[tb.m2l_red_src[q]];
        L[(int64_t)c * tb.nLh + r] = v;
    }
}

// ------------------------------------------------------------------ L2L
// The local expansion of cell c shifted from its parent's (Eq. (9)-type Taylor
// shift), added to c's stored components; one axis at a time, three stages of at
// most p + 1 terms in a row in place of (p + 1)(p + 2)(p + 3) / 6: L2L 0.285 ->
// 0.177 ms at 1M dipoles, p = 6; 0.217 -> 0.102 ms at 262k Plummer, p = 8.
__device__ __forceinline__ void l2l_cell(int c, int pa, const double *centre, const DevTables &tb,
                                         double *L, double *sm)
{
    const int p = tb.p, P1 = p + 1, nL = tb.nL;
    double *pw = sm;                    // [3][P+1]: (z_d - z'_d)^j / j!
    double *A = pw + 3 * P1;            // [nL]
    double *B = A + nL;                 // [nL]
    if (threadIdx.x < 3)
        axis_powers(centre[3 * c + threadIdx.x] - centre[3 * pa + threadIdx.x], p, pw + threadIdx.x * P1);
    expand_local_cg(L + (int64_t)pa * tb.nLh, tb, A);         // the parent's full expansion
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        const double *in = ax == 1 ? B : A, *w = pw + ax * P1;
        // the last stage forms the child's stored components only (the shift keeps
        // the expansion harmonic)
        const int outs = ax == 2 ? tb.nLh : nL;
        for (int t = threadIdx.x; t < outs; t += blockDim.x) {
            const int n = ax == 2 ? tb.h_rn[t] : t;
            const int v = mi_at(tb.mi, n);
            int sh = mi_shell(v), a = mi_ny(v) + mi_nz(v);
            if (ax == 2 && sh < tb.n_lo) continue;
            const int js = p - sh;
            const double *x = in + n;
            double acc = 0.0;
            for (int j = 0; j <= js; ++j) {
                acc = fma(w[j], *x, acc);
                // n + j e: one shell up, at the same place in it (x), a row up (y),
                // a row and a place (z)
                x += (sh + 1) * (sh + 2) / 2 + (ax == 0 ? 0 : (ax == 1 ? a + 1 : a + 2));
                ++sh;
                ++a;
            }
            if (ax == 2) L[(int64_t)c * tb.nLh + t] += acc;
            else (ax == 0 ? B : A)[t] = acc;
        }
        if (ax < 2) __syncthreads();
    }
}

// ------------------------------------------------------------------ L2P
constexpr int kL2PThreads = 128;

// Leaf c: the far-field part of phi and E = -grad phi at its particles (Eqs.
// (9), (10)), one thread per particle, in sorted particle order; fixed point as
// in the P2M.  The coefficients L_n rho^k / k! (n = k, k + e_d) lie in shared
// memory in the order of the nested loops over k, so a monomial is one product
// from the one before it: with the three sums 70 multiply-adds' time where the
// FP64 form spent five operations of 64 clocks: L2P
// 0.84 -> 0.27 ms at 1M dipoles, p = 6; 0.79 -> 0.20 ms at 262k, p = 8.
template <bool PHI, bool FIELD>
__global__ void __launch_bounds__(kL2PThreads)
k_l2p(const int32_t *leaves, const int32_t *begin, const int32_t *end, const double *centre,
      const double *px, const double *py, const double *pz, const double *L, DevTables tb,
      double *phi, double *E)
{
    pdl_wait();
    extern __shared__ int4 lsm4[];
    constexpr int D0 = FIELD ? 0 : 3, D1 = PHI ? 4 : 3;     // components wanted
    __shared__ int s_re[kL2PThreads / 32];
    __shared__ MagSum s_ms[kL2PThreads / 32][4];
    const int c = leaves[blockIdx.x], b = begin[c], e = end[c];
    const int P = PHI ? tb.p : tb.p - 1, nst = PHI ? tb.nL : tb.nG;
    const int *ord = PHI ? tb.l2p_ord : tb.l2p_ord + tb.nL;     // k of each step
    int4 *C4 = lsm4;                                        // [steps][2]: limbs of d/dx, d/dy | d/dz, phi
    double *C = (double *)lsm4;                             // the same as doubles over rho^k, first
    double *Lsm = C + 4 * nst;                              // [nL]
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const double z0 = centre[3 * c], z1 = centre[3 * c + 1], z2 = centre[3 * c + 2];
    int re = kNoExp;
    double dx = 0.0, dy = 0.0, dz = 0.0;                    // of the thread's first particle
    const int jt = b + threadIdx.x;
    for (int j = jt; j < e; j += kL2PThreads) {
        const double x = px[j] - z0, y = py[j] - z1, z = pz[j] - z2;
        if (j == jt) {
            dx = x;
            dy = y;
            dz = z;
        }
        re = max(re, max(disp_exp(x), max(disp_exp(y), disp_exp(z))));
    }
    re = __reduce_max_sync(0xffffffffu, re);
    if (lane == 0) s_re[w] = re;
    expand_local_cg(L + (int64_t)c * tb.nLh, tb, Lsm);      // ends with a barrier
    re = max(max(s_re[0], s_re[1]), max(s_re[2], s_re[3]));
    // every particle at the centre: a radius below FP64's range leaves the coefficients
    // of k = 0 their scale (at a radius of 1 the others set it, and those lost their bits)
    if (re == kNoExp) re = -2200;
    int top[4] = {kNoExp, kNoExp, kNoExp, kNoExp};
    for (int i = threadIdx.x; i < nst; i += kL2PThreads) {
        const int k = ord[i], up = mi_shell(mi_at(tb.mi, k)) * re;
        const double f = inv_factorial(tb, k);
#pragma unroll
        for (int d = D0; d < D1; ++d) {
            const double x = d == 3 ? Lsm[k] * f : (k < tb.nG ? Lsm[tb.l2p_grad[3 * k + d]] * f : 0.0);
            C[4 * i + d] = x;
            const int me = mag_exp(x);
            if (me != kNoExp) top[d] = max(top[d], me + up);
        }
    }
    unsigned long long u[4] = {0, 0, 0, 0};
#pragma unroll
    for (int d = D0; d < D1; ++d) top[d] = __reduce_max_sync(0xffffffffu, top[d]);
    for (int i = threadIdx.x; i < nst; i += kL2PThreads) {
        const int up = mi_shell(mi_at(tb.mi, ord[i])) * re;
#pragma unroll
        for (int d = D0; d < D1; ++d) u[d] += mag_units(C[4 * i + d], up, top[d]);
    }
#pragma unroll
    for (int d = D0; d < D1; ++d) {
        const MagSum ms = warp_mag_sum(u[d], top[d]);
        if (lane == 0) s_ms[w][d] = ms;
    }
    __syncthreads();
    int es[4];
#pragma unroll
    for (int d = D0; d < D1; ++d) es[d] = mag_sum_exp(&s_ms[0][d], kL2PThreads / 32, 4);
    for (int i = threadIdx.x; i < nst; i += kL2PThreads) {
        const int up = mi_shell(mi_at(tb.mi, ord[i])) * re;
#pragma unroll
        for (int d = D0; d < D1; ++d)
            ((int2 *)C)[4 * i + d] = es[d] == kBadExp ? make_int2(0, 0) : limbs_of(C[4 * i + d], 56 - es[d] + up);
    }
    __syncthreads();
    for (int j = jt; j < e; j += kL2PThreads) {
        if (j != jt) {
            dx = px[j] - z0;
            dy = py[j] - z1;
            dz = pz[j] - z2;
        }
        const I2 ux = fx::bal(fx::fix64(dx, 60 - re)), uy = fx::bal(fx::fix64(dy, 60 - re)),
                 uz = fx::bal(fx::fix64(dz, 60 - re));
        s64 a1[4] = {0, 0, 0, 0}, X = 1ll << 60;
        const int4 *Cp = C4;
        for (int kx = 0; kx <= P; ++kx) {
            s64 a0[4] = {1ll << 25, 1ll << 25, 1ll << 25, 1ll << 25}, Y = X;
            for (int ky = 0; ky <= P - kx; ++ky) {
                s64 Z = Y;
                for (int kz = P - kx - ky;; --kz) {
                    const I2 m = limbs60(Z);
                    const int4 t0 = Cp[0], t1 = Cp[1];
                    Cp += 2;
                    if (FIELD) {
                        a1[0] = madp(m.h, t0.x, a1[0]);
                        a0[0] = madp(m.h, t0.y, a0[0]);
                        a0[0] = madp(m.l, t0.x, a0[0]);
                        a1[1] = madp(m.h, t0.z, a1[1]);
                        a0[1] = madp(m.h, t0.w, a0[1]);
                        a0[1] = madp(m.l, t0.z, a0[1]);
                        a1[2] = madp(m.h, t1.x, a1[2]);
                        a0[2] = madp(m.h, t1.y, a0[2]);
                        a0[2] = madp(m.l, t1.x, a0[2]);
                    }
                    if (PHI) {
                        a1[3] = madp(m.h, t1.z, a1[3]);
                        a0[3] = madp(m.h, t1.w, a0[3]);
                        a0[3] = madp(m.l, t1.z, a0[3]);
                    }
                    if (kz == 0) break;
                    Z = mul60(fx::bal(Z), uz);
                }
                if (ky < P - kx) Y = mul60(fx::bal(Y), uy);
            }
            if (kx < P) X = mul60(fx::bal(X), ux);
            // at most 91 steps of 2^55 since the last carry
#pragma unroll
            for (int d = 0; d < 4; ++d) a1[d] += a0[d] >> 26;
        }
        auto value = [&](int d) {
            return es[d] == kBadExp ? __longlong_as_double(0x7ff8000000000000ll) : (a1[d] ? scale2((double)a1[d], es[d] - 60) : 0.0);
        };
        if (PHI) phi[j] = value(3);
        if (FIELD) {
            E[3 * (int64_t)j] = -value(0);
            E[3 * (int64_t)j + 1] = -value(1);
            E[3 * (int64_t)j + 2] = -value(2);
        }
    }
}

// The L2L shifts of all levels in one launch.  Blocks claim cells in
// breadth-first order (a counter), so a cell's parent was claimed earlier by a
// block that is running or done and waits on nothing later: the block waits
// (bounded) for the parent's flag, shifts the parent's local expansion into the
// cell and publishes its own flag.  A wait that gives up fills the cell's
// expansion with NaN, so the failure shows in the output.  ctl[0] (the claim
// counter) and the flags ctl[1 + c] start at zero.
__global__ void __launch_bounds__(128)
k_downward(int64_t nc, const int32_t *parent, const double *centre, DevTables tb, double *L,
           unsigned *ctl)
{
    pdl_wait();
    extern __shared__ double sm[];
    __shared__ int s_c, s_ok;
    if (threadIdx.x == 0) s_c = (int)atomicAdd(&ctl[0], 1u);
    __syncthreads();
    const int c = s_c;
    if (c >= nc) return;
    const int pa = parent[c];
    if (pa >= 0) {
        if (threadIdx.x == 0) {
            s_ok = wait_flag(ctl + 1 + pa);
            __threadfence();
        }
        __syncthreads();
        if (s_ok) {
            l2l_cell(c, pa, centre, tb, L, sm);
        } else {
            for (int r = threadIdx.x; r < tb.nLh; r += blockDim.x)
                L[(int64_t)c * tb.nLh + r] = __longlong_as_double(0x7ff8000000000000ll);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicExch(ctl + 1 + c, 1u);
    }
}

}  // namespace

inline unsigned grid(int64_t n, int bs) { return (unsigned)((n + bs - 1) / bs); }

// 1/(k_x! k_y! k_z!) of every index, a double as two words; the same for all
// handles and orders, formed once (every evaluate assembles the tables)
static const std::vector<int> &inv_factorial_words()
{
    static const std::vector<int> words = [] {
        const MultiIndex &I = multi_index();
        std::vector<int> v(2 * (size_t)kMaxTot);
        for (int i = 0; i < kMaxTot; ++i) {
            double f = 1.0;                      // exact: at most 12!
            for (int q : {I.nx[i], I.ny[i], I.nz[i]})
                for (int j = 2; j <= q; ++j) f *= j;
            f = 1.0 / f;
            std::memcpy(&v[2 * i], &f, 8);
        }
        return v;
    }();
    return words;
}

// Table buffer layout (int32): lut | p2m | m2m_off | m2m_kq | l2p_grad | red_off |
// red_src | l2l_ix | l2p_ord | 1/k! | harmonic maps | packed indices
fmm_status upload_tables(fmm_tree *t, int s, int p, int n_lo, DevTables *dt, const int32_t **lut)
{
    static int consts_ready[64] = {0};
    static std::mutex consts_mu;
    std::lock_guard<std::mutex> consts_lock(consts_mu);
    if (t->device < 64 && !consts_ready[t->device]) {
        const MultiIndex &I = multi_index();
        int8_t x[kMaxTot], y[kMaxTot], z[kMaxTot];
        for (int i = 0; i < kMaxTot; ++i) { x[i] = (int8_t)I.nx[i]; y[i] = (int8_t)I.ny[i]; z[i] = (int8_t)I.nz[i]; }
        FMM_TRY(cuda_check(t, cudaMemcpyToSymbol(c_nx, x, sizeof(x)), "constants"));
        FMM_TRY(cuda_check(t, cudaMemcpyToSymbol(c_ny, y, sizeof(y)), "constants"));
        FMM_TRY(cuda_check(t, cudaMemcpyToSymbol(c_nz, z, sizeof(z)), "constants"));
        double inv[kMaxOrder + 2];
        inv[0] = 0.0;
        for (int q = 1; q < kMaxOrder + 2; ++q) inv[q] = 1.0 / q;
        FMM_TRY(cuda_check(t, cudaMemcpyToSymbol(c_invint, inv, sizeof(inv)), "constants"));
        consts_ready[t->device] = 1;
    }
    OpTables &T = t->tab;
    std::vector<int32_t> buf;
    size_t o_lut, o_p2m, o_m2m_off, o_m2m_kq, o_grad, o_roff, o_rsrc;
    auto put = [&](const std::vector<int> &v) {
        size_t o = buf.size();
        buf.insert(buf.end(), v.begin(), v.end());
        buf.push_back(0);
        return o;
    };
    const int h = t->m2l_harmonic ? 1 : 0;
    const int s_hi = std::max(s, t->s_hi);
    const bool rebuild = !(t->tab_key_s == s && t->tab_key_p == p && t->tab_key_nlo == n_lo &&
                           t->tab_key_h == h && t->tab_key_shi == s_hi);
    if (rebuild) build_tables(T, s, s_hi, p, n_lo, kM2LThreadsShared, h != 0);
    {
        const MultiIndex &I = multi_index();
        std::vector<int> lutv((kMaxOrder + 1) * (kMaxOrder + 1) * (kMaxOrder + 1));
        for (int i = 0; i < (int)lutv.size(); ++i) lutv[i] = ((const int16_t *)I.lut)[i];
        o_lut = put(lutv);
    }
    o_p2m = put(T.p2m_terms); o_m2m_off = put(T.m2m_off); o_m2m_kq = put(T.m2m_kq);
    o_grad = put(T.l2p_grad); o_roff = put(T.m2l_red_off);
    if (buf.size() & 1) buf.push_back(0);                 // read in pairs of words
    const size_t o_ix = put(T.l2l_ix);
    const size_t o_ord = put(T.l2p_ord);
    const size_t o_if = put(inv_factorial_words());
    o_rsrc = put(T.m2l_red_src);
    const size_t o_hrm = put(T.h_rm), o_hf = put(T.h_fold), o_hfo = put(T.h_fold_off);
    const size_t o_hu = put(T.h_unfold), o_huo = put(T.h_unfold_off), o_hrn = put(T.h_rn);
    size_t o_mi;
    {
        const MultiIndex &I = multi_index();
        std::vector<int> mi(kMaxTot);
        for (int i = 0; i < kMaxTot; ++i)
            mi[i] = I.nx[i] | I.ny[i] << 5 | I.nz[i] << 10 | (I.nx[i] + I.ny[i] + I.nz[i]) << 15;
        o_mi = put(mi);
    }
    FMM_TRY(ensure(t, t->b_tab_i32, 4 * buf.size()));
    FMM_TRY(ensure(t, t->b_tab_u32, 4 * (T.m2l_desc.size() + 2)));
    if (rebuild) {
        FMM_TRY(cuda_check(t, cudaMemcpyAsync(t->b_tab_i32.ptr, buf.data(), 4 * buf.size(),
                                              cudaMemcpyHostToDevice, t->stream), "tables"));
        FMM_TRY(cuda_check(t, cudaMemcpyAsync(t->b_tab_u32.ptr, T.m2l_desc.data(),
                                              4 * T.m2l_desc.size(), cudaMemcpyHostToDevice,
                                              t->stream), "tables"));
        t->tab_key_s = s; t->tab_key_p = p; t->tab_key_nlo = n_lo; t->tab_key_h = h;
        t->tab_key_shi = s_hi;
    }
    const int32_t *B = (const int32_t *)t->b_tab_i32.ptr;
    dt->s = s; dt->p = p; dt->n_lo = n_lo; dt->nS = T.nS; dt->nM = T.nM; dt->nL = T.nL;
    dt->nD = T.nD; dt->m0 = T.m0; dt->nK = ntot(p); dt->nG = ntot(p - 1);
    dt->p2m_terms = B + o_p2m; dt->m2m_off = B + o_m2m_off; dt->m2m_kq = B + o_m2m_kq;
    dt->l2p_grad = B + o_grad; dt->l2p_ord = B + o_ord; dt->l2l_ix = B + o_ix; dt->inv_fact = B + o_if; dt->m2l_red_off = B + o_roff;
    dt->m2l_red_src = B + o_rsrc;
    dt->m2l_desc = (const uint32_t *)t->b_tab_u32.ptr;
    dt->m2l_T = T.m2l_T; dt->m2l_slots = T.m2l_slots;
    dt->mi = B + o_mi;
    dt->harmonic = T.harmonic ? 1 : 0;
    dt->nMh = T.nMh;
    dt->h_fold_lev = (int)T.h_fold_off.size() - 1;
    dt->h_unfold_lev = (int)T.h_unfold_off.size() - 1;
    dt->h_rm = B + o_hrm; dt->h_fold = B + o_hf; dt->h_fold_off = B + o_hfo;
    dt->h_unfold = B + o_hu; dt->h_unfold_off = B + o_huo;
    dt->nLh = T.nLh; dt->h_rn = B + o_hrn;
    *lut = B + o_lut;
    return FMM_OK;
}

namespace {

void record(fmm_tree *t, int i)
{
    if (t->profiling) cudaEventRecord(t->ev[i], t->stream);
}

}  // namespace

void launch_fold_m(cudaStream_t st, const double *M, int ldM, int64_t nc, const DevTables &tb,
                   double *Mh, int ldH, bool dependent)
{
    if (nc > 0)
        launch_next_if(dependent, st, k_fold_m<double>, (unsigned)((nc + 3) / 4), 128, 32 * (size_t)tb.nM, M, ldM, nc, tb, Mh, ldH);
}

void launch_fold_m(cudaStream_t st, const float *M, int ldM, int64_t nc, const DevTables &tb,
                   float *Mh, int ldH)
{
    if (nc > 0)
        launch_next(st, k_fold_m<float>, (unsigned)((nc + 3) / 4), 128, 32 * (size_t)tb.nM, M, ldM, nc, tb, Mh, ldH);
}

// derivative tables, one FP64 row per distinct M2L offset key
fmm_status build_dtables(fmm_tree *t, int p, const DevTables &tb, const int32_t *lut)
{
    if (t->d_p != p && t->n_doff > 0) {
        FMM_TRY(ensure(t, t->b_D, 8 * (size_t)t->n_doff * tb.nD));
        // warps per block: as many rows of nD doubles as fit in 48 KB, at most 8
        const int wpb = (int)std::max<int64_t>(1, std::min<int64_t>(8, 49152 / (8 * (int64_t)tb.nD)));
        k_dtables<<<(unsigned)((t->n_doff + wpb - 1) / wpb), 32 * wpb, 8 * (size_t)wpb * tb.nD,
                    t->stream>>>((const uint64_t *)t->b_dkeys.ptr, t->n_doff, tb.nD, lut,
                                 (double *)t->b_D.ptr);
        ++t->launches;
        t->d_p = p;
        t->d32_p = -1;
        t->tc_img_p = -1;
        t->m32_img_p = -1;
        t->fx_img_p = -1;
    }
    return FMM_OK;
}

// P2M at the leaves and M2M upward, level by level, into b_M (FP64, tb.nM per cell)
fmm_status run_upward(fmm_tree *t, const DevTables &tb, bool rec)
{
    cudaStream_t st = t->stream;
    const int64_t nc = t->ncells;
    const int P1 = tb.p + 1;
    FMM_TRY(ensure(t, t->b_M, 8 * (size_t)nc * tb.nM));
    FMM_TRY(ensure(t, t->b_ud, 8 * (size_t)(nc + 1)));
    t->m_cells = nc;
    double *M = (double *)t->b_M.ptr;
    const double *centre = (const double *)t->b_centre.ptr;
    // P2M and M2M in one launch; the arrival counters start (and end) at zero
    cudaMemsetAsync(t->b_ud.ptr, 0, 8 * (size_t)(nc + 1), st);     // with the downward pass's flags behind them
    const size_t smem = 8 * std::max<size_t>(
        (size_t)tb.nK * tb.nS + (size_t)kP2MChunk * 3 * P1 + (size_t)kP2MChunk * tb.nS,
        6 * (size_t)P1 + 12 * (size_t)tb.nM);
    auto go = [&](auto kern) {
        allow_max_dynamic_smem(kern);
        launch_next(st, kern, (unsigned)t->nleaves, kP2MThreads, smem,
            (const int32_t *)t->b_leaves.ptr, (const int32_t *)t->b_begin.ptr,
            (const int32_t *)t->b_end.ptr, (const int32_t *)t->b_parent.ptr,
            (const int32_t *)t->b_child.ptr, (const int32_t *)t->b_nchild.ptr, (const int32_t *)t->b_cx.ptr,
            (const int32_t *)t->b_cy.ptr, (const int32_t *)t->b_cz.ptr, centre,
            (const double *)t->b_px.ptr, (const double *)t->b_py.ptr, (const double *)t->b_pz.ptr,
            (const double *)t->b_S.ptr, tb, M, (unsigned *)t->b_ud.ptr);
    };
    if (tb.nS <= 3) go(k_upward<3>);
    else if (tb.nS <= 6) go(k_upward<6>);
    else go(k_upward<10>);
    ++t->launches;
    if (rec) record(t, 7);
    return FMM_OK;
}

fmm_status run_expansions(fmm_tree *t, int p, int want_phi, int want_field)
{
    cudaStream_t st = t->stream;
    const int s = t->s;
    const int n_lo = want_phi ? 0 : 1;
    DevTables tb;
    const int32_t *lut;
    FMM_TRY(upload_tables(t, s, p, n_lo, &tb, &lut));
    const int64_t nc = t->ncells, n = t->n;
    const int P1 = p + 1;

    FMM_TRY(build_dtables(t, p, tb, lut));
    record(t, 6);
    FMM_TRY(ensure(t, t->b_L, 8 * (size_t)nc * tb.nLh));
    FMM_TRY(ensure(t, t->b_phi, 8 * (size_t)n));
    FMM_TRY(ensure(t, t->b_E, 24 * (size_t)n));
    // The M2L: in fixed point over the tiles of a plan (m2l_fx.cu) where the
    // lists are long enough, else one block per target cell.  A plan that has to
    // be built (new lists or p: two host syncs) is built on the handle's side
    // stream while the upward pass runs; not while the stream is being captured
    // (the graph's evaluate follows an ordinary one, which built it).  Where the
    // device has no memory for it, the per-cell kernel serves these lists and
    // orders from then on (fx_off), in later evaluates and captures too.
    bool fx = t->n_m2l > 0 && fx_usable(t, s, p, tb.harmonic, tb.n_lo);
    const bool stale = fx && (!t->tc_plan || t->fx_img_p != p);
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (stale) FMM_TRY(cuda_check(t, cudaStreamIsCapturing(st, &cap), "capture status"));
    const bool side = stale && cap == cudaStreamCaptureStatusNone;
    if (stale && !side) fx = false;           // nothing may be allocated or waited for in a capture
    if (side) {
        FMM_TRY(side_stream(t));
        FMM_TRY(cuda_check(t, cudaEventRecord(t->ev_lists, st), "event"));
    }
    cudaMemsetAsync(t->b_L.ptr, 0, 8 * (size_t)nc * tb.nLh, st);   // here, so that the kernels follow one another
    FMM_TRY(run_upward(t, tb, true));
    double *M = (double *)t->b_M.ptr, *L = (double *)t->b_L.ptr;
    const int32_t *leaves = (const int32_t *)t->b_leaves.ptr;
    const int32_t *begin = (const int32_t *)t->b_begin.ptr, *end = (const int32_t *)t->b_end.ptr;
    const double *centre = (const double *)t->b_centre.ptr;
    const double *px = (const double *)t->b_px.ptr, *py = (const double *)t->b_py.ptr,
                 *pz = (const double *)t->b_pz.ptr;
    if (fx) {
        if (side) {
            cudaStreamWaitEvent(t->side_st, t->ev_lists, 0);
            t->stream = t->side_st;
        }
        t->soft_alloc = true;                 // no memory for the plan: the per-cell kernel needs none
        const fmm_status ps = fx_prepare(t, p);
        t->soft_alloc = false;
        t->stream = st;
        if (side) {
            cudaEventRecord(t->ev_plan, t->side_st);
            cudaStreamWaitEvent(st, t->ev_plan, 0);
        }
        if (ps == FMM_EBUDGET) {
            tc_release(t);
            t->err.clear();
            fx = false;
            t->fx_off = true;
        } else {
            FMM_TRY(ps);
        }
    }
    // M2L over the stored lists (harmonic: on the folded multipoles)
    const double *Ms = M;
    if (fx) {
        FMM_TRY(run_fx_exps(t, M, tb));
    } else if (t->n_m2l > 0 && tb.harmonic) {
        FMM_TRY(ensure(t, t->b_Mh, 8 * (size_t)nc * tb.nMh));
        launch_fold_m(st, M, tb.nM, nc, tb, (double *)t->b_Mh.ptr, tb.nMh, !side);
        ++t->launches;
        Ms = (const double *)t->b_Mh.ptr;
    }
    record(t, 8);
    if (fx) {
        FMM_TRY(run_m2l_fx(t, tb, L));
    } else if (t->n_m2l > 0) {
        const int ldM = tb.nMh | 1, ldD = tb.nD | 1;
        size_t fixed = 8 * (size_t)tb.m2l_slots * kM2LThreads + 4 * (size_t)tb.m2l_T * kM2LThreads;
        const size_t row = 8 * (size_t)(ldM + ldD);
        const int batch = fixed + kM2LBatch * row <= kM2LSmemMax ? kM2LBatch : kM2LBatch / 2;
        const size_t smem = fixed + batch * row;
        allow_max_dynamic_smem(k_m2l);
        launch_next_if(!side || Ms != M, st, k_m2l, (unsigned)nc, kM2LThreads, smem,
            (const int32_t *)t->b_m2l_off.ptr, (const int32_t *)t->b_m2l_src.ptr,
            (const int32_t *)t->b_m2l_didx.ptr, (const int32_t *)t->b_level.ptr,
            (const int32_t *)t->b_sys.ptr, t->sys_eside_dev(), Ms, (const double *)t->b_D.ptr, tb, L, batch);
        ++t->launches;
    }
    record(t, 9);
    // L2L downward, all levels in one launch (flags and claim counter start at zero)
    if (t->nlevels > 1) {
        unsigned *ctl = (unsigned *)t->b_ud.ptr + nc + 1;
        size_t smem = 8 * (size_t)(3 * P1 + 2 * tb.nL);
        launch_next(st, k_downward, (unsigned)nc, 128, smem, nc, (const int32_t *)t->b_parent.ptr, centre, tb, L, ctl);
        ++t->launches;
    }
    record(t, 10);
    // L2P
    {
        const size_t smem = 32 * (size_t)(want_phi ? tb.nL : tb.nG) + 8 * (size_t)tb.nL;
        auto go = [&](auto kern) {
            launch_next(st, kern, (unsigned)t->nleaves, kL2PThreads, smem, leaves, begin, end, centre, px, py, pz, L, tb,
                                                                  (double *)t->b_phi.ptr, (double *)t->b_E.ptr);
        };
        if (want_phi && want_field) go(k_l2p<true, true>);
        else if (want_phi) go(k_l2p<true, false>);
        else go(k_l2p<false, true>);
        ++t->launches;
    }
    record(t, 11);
    return cuda_check(t, cudaGetLastError(), "expansion kernels");
}

}  // namespace fmm
