// p2p_fx.cu -- the FP64 near field (P2P) in fixed-point arithmetic.
//
// The pair terms of the P2P (p2p.cu's header has the formulas) need about 24
// FP64 instructions per directed interaction (17 with both directions of a pair
// shared), and GB300 issues one FP64 warp instruction per 64 clocks and
// scheduler: 1,100 clocks or more per warp step.  The same dipole terms in
// 64-bit fixed point (fx64.cuh) take about 60 integer multiply-adds and 130
// other instructions, some 390 clocks.  Inside one leaf's near field every
// quantity has a known range, so fixed point carries 55 to 60 significant bits
// per factor: a pair term's error is at or below an FP64 evaluation's (about
// ten roundings of 2^-53), and the sums over pairs are exact integers.
// Measured, one million dipoles, field, 946 M interactions: 36.3 ms with the
// symmetric FP64 kernel -> 10.4 ms; error against long double at or below the
// FP64 kernels' (a set of 700: 1e-16 to 4e-16 against 2e-16 to 1e-15).
// Bound: the integer multiply pipe and the ALU together; 16 or 32 warps per SM
// run alike.  Measured and not better: cross products by IMAD.HI, sums by
// shifts and carries in place of the two multiply-adds by a power of two, the
// cross products' upper half added by a multiply-add, 64 to 104 registers for
// more warps.  The sums as the factor's four limbs times the term's two (seven
// multiply-adds a component, nothing rounded) took 11.0 ms; 262k Plummer
// dipoles 6.9 instead of 6.0, 200k charges and dipoles 5.9 instead of 5.1,
// 96 quadrupole systems 32.0 instead of 29.1.
//
//   R    separation, source minus target: exact differences of coordinates
//        rounded to 2^-58 of the coarser leaf's half side, shifted left by sh
//        so that |R|^2 is in [1/4, 1) (the shift from an FP32 estimate)
//   y    1/|R|: FP32 hardware seed y0 (21 bits kept), e = 1 - |R|^2 y0^2, one
//        third-order step y = y0 (1 + e/2 + 3/8 e^2) (error 5/16 e^3 < 2^-60)
//   M    a source's moments times a power of two of its own
//   sums the term as one 59-bit integer (rounded at 2^-52 of the moment over the
//        normalised distance's power, which is at least 1), times a power of two
//        into 28-bit limbs of four 64-bit sums.  The scale leaves room for the
//        row's largest moments at the closest fixed-point separation; a term
//        keeps all its bits down to 2^-56 of the largest possible, and some down
//        to 2^-84
//
// Pairs closer than 2^-7 of the coordinate range (a sixteenth of a half side;
// a few in a million of a uniform set's) and coincident points take the FP64
// formulas, as do whole rows that hold a non-finite moment.  So do targets whose
// sum is so small beside the row's scale that what its terms can have lost (counted
// while the sources are staged) passes 2^-54 of it: a target that holds the row's
// largest moment itself, coincides with it or sees none of its field, from ratios
// to the others of about 2^42 (charges), 2^35 (dipoles) and 2^28 (quadrupoles) on.
// That costs about 0.6 % of the P2P at 1M dipoles, 1 % at 262k Plummer and 200k
// charges and dipoles (the count in the staging; the pairs' loop is the same).
// Keeping every bit in the loop instead cost 2 to 5 %.
#include <algorithm>
#include <type_traits>

#include "fmm_internal.cuh"
#include "fx64.cuh"
#include "pair.cuh"

namespace fmm {

namespace {

using namespace fx;

constexpr int kShMax = 7;                  // largest normalising shift a pair may take
constexpr int kFxGroups = 32;              // partner leaves of a staging round
constexpr uint32_t kM28 = 0x0fffffffu;

// A staged source: 32-bit words in int4 columns.  Words 0..5 the position
// (three 64-bit), 6 the particle index, then per shell its shift bases and
// moment words.
__host__ __device__ constexpr int fx_shell_words(int s, bool phi, bool field)
{
    const int b = (phi ? 1 : 0) + (field ? 1 : 0);
    return b + (s == 0 ? (phi ? 2 : 0) + (field ? 2 : 0) : (s == 1 ? 6 + (field ? 6 : 0) : 14));
}
__host__ __device__ constexpr int fx_off(int slo, int s, bool phi, bool field)
{
    return s <= slo ? 7 : fx_off(slo, s - 1, phi, field) + fx_shell_words(s - 1, phi, field);
}
template <int SLO, int SHI, bool PHI, bool FIELD>
struct FxRec {
    static constexpr int words = fx_off(SLO, SHI + 1, PHI, FIELD);
    static constexpr int nw = (words + 3) / 4;             // int4s per source
    static constexpr int ch = nw <= 6 ? 256 : 128;         // sources staged per round
};

// A term T Y (T the bracket, Y the power of y) enters as t = T Y / 2^K, |t| <
// 2^59, times 2^(56 - shift).  The shells' terms stand at different powers of
// two; these adjust their shifts to the sums' common unit, 2^(base - kUnit).
__host__ __device__ constexpr int fx_off_e(int s) { return s == 2 ? -4 : 0; }
__host__ __device__ constexpr int fx_off_p(int s) { return s == 0 ? 2 : (s == 2 ? -2 : 0); }
constexpr int kUnitE = 108, kUnitP = 111;

// the shift amount that stands for "contributes nothing"
constexpr int kFar = 160;
constexpr int kWhole = 56;                 // a term of a larger shift loses bits

// the two forms of a multiply-add (fx64.cuh): the quadrupoles' sums run faster
// fused, the others' with the addend in the instruction
template <bool Q>
__device__ __forceinline__ s64 mac(int a, int b, s64 c)
{
    return Q ? madp(a, b, c) : madw(a, b, c);
}
// N terms of one shift s: t 2^(56 - s) in limbs of 28 bits.  Nearly every pair
// has s <= 28 and takes two multiply-adds by 2^(28 - s); beyond, a limb (two)
// further down; past 84 nothing.
template <int N, bool Q>
__device__ __forceinline__ void fx_add(const s64 (&t)[N], int s, s64 (*P)[4])
{
    int h[N], l[N];
    const int m = (int)shl32(1u, (uint32_t)(28 - s));
#pragma unroll
    for (int c = 0; c < N; ++c) {
        h[c] = (int)(t[c] >> 28);
        l[c] = (int)((uint32_t)t[c] & kM28);
        P[c][2] = mac<Q>(h[c], m, P[c][2]);
        P[c][1] = mac<Q>(l[c], m, P[c][1]);
    }
    if (s > 28 && s <= 84) {
        const int m1 = (int)shl32(1u, (uint32_t)(56 - s)), m0 = s > 56 ? (int)shl32(1u, (uint32_t)(84 - s)) : 0;
#pragma unroll
        for (int c = 0; c < N; ++c) {
            P[c][1] = mac<Q>(h[c], m1, P[c][1]);
            P[c][0] = mac<Q>(h[c], m0, mac<Q>(l[c], m1, P[c][0]));
        }
    }
}
// carries: afterwards the lower three sums are in [0, 2^28)
__device__ __forceinline__ void fx_carry(s64 *P)
{
#pragma unroll
    for (int l = 0; l < 3; ++l) {
        P[l + 1] += P[l] >> 28;
        P[l] &= kM28;
    }
}
// the sums' value as a double: magnitude first, so that no leading limb cancels
__device__ __forceinline__ double fx_value(s64 *P, int e)
{
    fx_carry(P);
    const bool neg = P[3] < 0;
    if (neg) {
#pragma unroll
        for (int l = 0; l < 4; ++l) P[l] = -P[l];
        fx_carry(P);
    }
    const double d = scalbn((double)P[3] * 0x1p84 + (double)((P[2] << 28) | P[1]) * 0x1p28 + (double)P[0], e);
    return neg ? -d : d;
}

struct FxGeo {
    I2 x, y, z;            // R 2^62
    u64 y1, y2, y3;        // 1/|R| 2^62, 1/|R|^2 2^60, 1/|R|^3 2^58
    int sh;
};

__device__ __forceinline__ float rsqrt_seed(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ s64 shl_any(s64 v, int n)
{
    s64 d;
    asm("shl.b64 %0, %1, %2;" : "=l"(d) : "l"(v), "r"(n));
    return d;
}

// |d| components below 2^61 and their norm below 2^62
__device__ __forceinline__ FxGeo fx_geo(s64 dx, s64 dy, s64 dz)
{
    FxGeo g;
    const float ax = (float)hi32(dx), ay = (float)hi32(dy), az = (float)hi32(dz);
    const int rb = __float_as_int(fmaf(ax, ax, fmaf(ay, ay, az * az)));  // |d|^2 2^-64
    // sh = floor((59 - log2) / 2), so that the shifted |R|^2 is in [1/4, 1); the
    // 2^11 (2^-12 of the estimate) keeps it above 1/4, y below 2, whatever the
    // estimate's rounding
    const int t = (187 << 23) - 1 + (1 << 11) - rb;
    g.sh = t >> 24;
    const float r2n = __int_as_float(rb + (t & (int)0xff000000) - (60 << 23));     // |R|^2
    // y0 2^30: the 23 fraction bits of y0 + 4, the bits above shifted out
    const uint32_t n0 = (uint32_t)__float_as_int(rsqrt_seed(r2n) + 4.0f) << 9;
    g.x = bal(shl_any(dx, g.sh));
    g.y = bal(shl_any(dy, g.sh));
    g.z = bal(shl_any(dz, g.sh));
    const s64 c = madp(g.z.h, g.z.l, madp(g.y.h, g.y.l, madp(g.x.h, g.x.l, kHalfUlp / 2)));
    const u64 r2 = (u64)madp(g.z.h, g.z.h, madp(g.y.h, g.y.h, madp(g.x.h, g.x.h, c >> 31)));   // |R|^2 2^60
    const s64 en = (s64)mulhi_u(r2, madu(n0, n0, 0), -(1ull << 56));            // -e 2^56, |e| < 2^-19
    const int es = (int)(en >> 6);
    const int e2 = hi32(madp(es, es, 0)) >> 12;                          // e^2 2^56
    const s64 h = ((s64)(e2 - (e2 >> 2)) - en) << 7;                     // (e/2 + 3/8 e^2) 2^64
    const u64 u = madu(n0, (uint32_t)h, 0);
    g.y1 = (u64)madp((int)n0, hi32(h), (s64)(((u64)n0 << 32) | (u >> 32)));
    g.y2 = mulhi_u(g.y1, g.y1);
    g.y3 = mulhi_u(g.y2, g.y1);
    return g;
}

__device__ __forceinline__ s64 word64(const int *r, int i)
{
    return (s64)(((u64)(uint32_t)r[i + 1] << 32) | (uint32_t)r[i]);
}
__device__ __forceinline__ I2 word_bal(const int *r, int i) { return {r[i + 1], r[i]}; }

// One shell's terms of a pair (R = source - target, so the odd powers change
// sign against p2p.cu's formulas).  r: the shell's words; dead: contributes
// nothing.
template <int S, bool PHI, bool FIELD>
__device__ __forceinline__ void fx_pair(const FxGeo &g, const int *r, bool dead, s64 (*P)[4])
{
    constexpr int e = PHI ? 1 : 0;                 // first field component
    constexpr int nb = (PHI ? 1 : 0) + (FIELD ? 1 : 0);
    int sp = 0, se = 0;
    if (PHI) sp = dead ? kFar : r[0] - (S + 1) * g.sh;
    if (FIELD) se = dead ? kFar : r[e] - (S + 2) * g.sh;
    const int *m = r + nb;
    if constexpr (S == 0) {
        if (PHI) {
            const s64 t[1] = {mulhi(word_bal(m, 0), bal((s64)g.y1))};      // q y 2^57
            fx_add<1, S == 2>(t, sp, P);
        }
        if (FIELD) {
            const I2 q = word_bal(m, PHI ? 2 : 0), y = bal((s64)(g.y3 >> 1));      // -q 2^61
            // -q R 2^59, times y^3 2^57
            const s64 t[3] = {mulhi(bal_biased(mulhi(q, g.x, kBias)), y), mulhi(bal_biased(mulhi(q, g.y, kBias)), y),
                              mulhi(bal_biased(mulhi(q, g.z, kBias)), y)};
            fx_add<3, S == 2>(t, se, P + e);
        }
    } else if constexpr (S == 1) {
        // M.R 2^59
        const I2 sr = bal_biased(dot3hi(word_bal(m, 0), g.x, word_bal(m, 2), g.y, word_bal(m, 4), g.z, kBias));
        const I2 y3 = bal((s64)(g.y3 << 2));
        if (PHI) {
            const s64 t[1] = {mulhi(sr, y3)};                              // (M.R) y^3
            fx_add<1, S == 2>(t, sp, P);
        }
        if (FIELD) {
            const I2 v1 = bal_biased(mulhi(sr, bal((s64)g.y2), kBias));    // (M.R) y^2 2^55
            // -3 (M.R) y^2 2^58: the factor -24
            const s64 vb = madw(v1.l, -24, kBias);
            const I2 v = {hi32(vb) + v1.h * -24, lo32(vb) ^ (int)0x80000000};
            // (M - 3 (M.R) y^2 R) 2^56 (the words of M hold the bias), times y^3 2^60
            const s64 t[3] = {mulhi(bal_biased(mulhi(v, g.x, word64(m, 6))), y3),
                              mulhi(bal_biased(mulhi(v, g.y, word64(m, 8))), y3),
                              mulhi(bal_biased(mulhi(v, g.z, word64(m, 10))), y3)};
            fx_add<3, S == 2>(t, se, P + e);
        }
    } else {
        // grad q and 2 q(R) of q(R) = sum S_a R^a; the words are 2 S_200, S_110,
        // S_101, 2 S_020, S_011, 2 S_002 (2^62: the doubled ones below 1, the
        // others below 1/2, so a row's cross products sum below 2^63) and the trace (2^58)
        const I2 m0 = word_bal(m, 0), m1 = word_bal(m, 2), m2 = word_bal(m, 4), m3 = word_bal(m, 6),
                 m4 = word_bal(m, 8), m5 = word_bal(m, 10);
        const s64 tr = word64(m, 12);
        // grad q 2^60, each plus 2^31
        const s64 G[3] = {dot3hi(m0, g.x, m1, g.y, m2, g.z, kBias), dot3hi(m1, g.x, m3, g.y, m4, g.z, kBias),
                          dot3hi(m2, g.x, m4, g.y, m5, g.z, kBias)};
        const s64 q2 = dot3hi(bal_biased(G[0]), g.x, bal_biased(G[1]), g.y, bal_biased(G[2]), g.z);   // 2 q 2^58
        const s64 p = mulhi_62(bal(q2 << 2), bal((s64)g.y2));              // 2 q y^2 2^58
        if (PHI) {
            const s64 t[1] = {mulhi(bal(p + (p >> 1) - tr), bal((s64)(g.y3 << 1)))};       // (3 q y^2 - tr) y^3
            fx_add<1, S == 2>(t, sp, P);
        }
        if (FIELD) {
            // 3 y^5 (grad q - (5 q y^2 - tr) R)
            const I2 n = bal(tr - 2 * p - (p >> 1));                       // (tr - 5 q y^2) 2^58
            const u64 y5 = mulhi_u(g.y3 << 2, g.y2);                       // 2^56
            const I2 y = bal((s64)((y5 - (y5 >> 2)) << 2));                // 3 y^5 2^56
            constexpr s64 b = kBias - (kBias >> 4);
            const s64 t[3] = {mulhi(bal_biased(mulhi(n, g.x, (G[0] >> 4) + b)), y),        // 2^56
                              mulhi(bal_biased(mulhi(n, g.y, (G[1] >> 4) + b)), y),
                              mulhi(bal_biased(mulhi(n, g.z, (G[2] >> 4) + b)), y)};
            fx_add<3, S == 2>(t, se, P + e);
        }
    }
}

template <int S, int SLO, int SHI, bool PHI, bool FIELD>
__device__ __forceinline__ void fx_pair_orders(const FxGeo &g, const int *r, bool dead, s64 (*P)[4])
{
    fx_pair<S, PHI, FIELD>(g, r + fx_off(SLO, S, PHI, FIELD), dead, P);
    if constexpr (S < SHI) fx_pair_orders<S + 1, SLO, SHI, PHI, FIELD>(g, r, dead, P);
}

// power of two above the moments of a shell (the largest |S_a| < 2^em), or
// kNone when they are all zero; 5000 for a non-finite one
constexpr int kNone = -20000, kBad = 5000;
__device__ __forceinline__ int fx_moment_exp(const double *S, int n)
{
    int top = 0, any = 0;
    for (int a = 0; a < n; ++a) {
        const s64 b = __double_as_longlong(S[a]) & 0x7fffffffffffffffll;
        any |= b != 0;
        top = max(top, (int)(b >> 52));
    }
    if (top == 0x7ff) return kBad;
    return any ? max(top, 1) - 1022 : kNone;
}
// quadrupoles: 2 S_a stay below 2^em too
__host__ __device__ constexpr int fx_exp_room(int s) { return s == 2 ? 1 : 0; }

__device__ __forceinline__ void put64(int *r, int i, s64 v)
{
    r[i] = (int)v;
    r[i + 1] = (int)(v >> 32);
}
__device__ __forceinline__ void put_bal(int *r, int i, s64 v)
{
    const I2 b = bal(v);
    r[i] = b.l;
    r[i + 1] = b.h;
}

// a shell's words of one source: base_e, base_p = the target leaf's bases plus
// (S + 2) or (S + 1) times the round's unit exponent.  True if its terms can lose
// bits in fx_add.
template <int S, bool PHI, bool FIELD>
__device__ __forceinline__ bool fx_stage_shell(const double *Sj, int base_p, int base_e, int *r)
{
    constexpr int e = PHI ? 1 : 0;
    constexpr int nb = (PHI ? 1 : 0) + (FIELD ? 1 : 0);
    int em = fx_moment_exp(Sj, (S + 1) * (S + 2) / 2);
    const bool none = em == kNone;
    em = none ? 0 : em + fx_exp_room(S);
    if (PHI) r[0] = none ? kFar : min(kFar, base_p - em);
    if (FIELD) r[e] = none ? kFar : min(kFar, base_e - em);
    int *m = r + nb;
    if constexpr (S == 0) {
        if (PHI) put_bal(m, 0, fix64(Sj[0], 59 - em));
        if (FIELD) put_bal(m, PHI ? 2 : 0, -fix64(Sj[0], 61 - em));
    } else if constexpr (S == 1) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const s64 v = fix64(Sj[a], 61 - em);
            put_bal(m, 2 * a, v);
            if (FIELD) put64(m, 6 + 2 * a, ((v + 16) >> 5) + kBias);
        }
    } else {
#pragma unroll
        for (int a = 0; a < 6; ++a)
            put_bal(m, 2 * a, fix64(Sj[a], (a == 0 || a == 3 || a == 5 ? 63 : 62) - em));
        put64(m, 12, fix64(Sj[0], 58 - em) + fix64(Sj[3], 58 - em) + fix64(Sj[5], 58 - em));
    }
    return !none && max(PHI ? r[0] : 0, FIELD ? r[e] : 0) > kWhole;
}

template <int S, int SLO, int SHI, bool PHI, bool FIELD>
__device__ __forceinline__ bool fx_stage_orders(const double *Sj, int bp, int be, int lu, int *r)
{
    bool lose = fx_stage_shell<S, PHI, FIELD>(Sj, bp + fx_off_p(S) + (S + 1) * lu, be + fx_off_e(S) + (S + 2) * lu,
                                              r + fx_off(SLO, S, PHI, FIELD));
    if constexpr (S < SHI)
        lose |= fx_stage_orders<S + 1, SLO, SHI, PHI, FIELD>(Sj + (S + 1) * (S + 2) / 2, bp, be, lu, r);
    return lose;
}

// What a term of base b can lose in fx_add, in units of the sums, when its shift is
// b less up to k sh: nothing down to 56, the lower limb (below 2^(84 - shift)) down
// to 84, all of it (below 2^(115 - shift)) beyond.  At least one unit, a whole
// number, so that the count does not depend on the order of its atomics (as a float
// it did in its last bits, and with it which sums a set at the line forms again).
__device__ __forceinline__ u64 fx_loss(int b, int k, int sh)
{
    const int lo = max(b - k * sh, kWhole + 1);            // the smallest shift that loses anything
    return 1ull << (lo > 84 ? max(115 - lo, 0) : (b > 84 ? 30 : 84 - lo));
}
// The same of all terms of one source, added to lost[0] (potential) and lost[1]
// (field).  gap: a target of the leaf is at least so far away along some axis.
template <int SLO, int SHI, bool PHI, bool FIELD>
__device__ __noinline__ void fx_count_loss(const double *Sj, int bp, int be, int lu, s64 gap, u64 *lost)
{
    const int sh = gap > 0 ? min(kShMax, __clzll(gap) - 1) : kShMax;     // the largest normalising shift
    int o = 0;
    for (int s = SLO; s <= SHI; ++s) {
        const int n = (s + 1) * (s + 2) / 2, em = fx_moment_exp(Sj + o, n) + fx_exp_room(s);
        o += n;
        if (em < kNone / 2) continue;
        const int ap = bp + fx_off_p(s) + (s + 1) * lu - em, ae = be + fx_off_e(s) + (s + 2) * lu - em;
        if (PHI && ap > kWhole) atomicAdd(lost, fx_loss(ap, s + 1, sh));
        if (FIELD && ae > kWhole) atomicAdd(lost + 1, fx_loss(ae, s + 2, sh));
    }
}

// The FP64 terms of one pair, added to the thread's sums in shared memory:
// the few pairs too close for the fixed-point range.
template <int SLO, int SHI, bool PHI, bool FIELD>
__device__ __noinline__ void fx_close(int i, int j, const double *px, const double *py, const double *pz,
                                      const double *Sm, double *acc, int stride)
{
    constexpr int nS = Orders<SLO, SHI>::n;
    double f = 0.0, e0 = 0.0, e1 = 0.0, e2 = 0.0;
    pair_orders<SLO, SHI, PHI, FIELD>(px[i] - px[j], py[i] - py[j], pz[i] - pz[j], Sm + (int64_t)j * nS, f, e0,
                                      e1, e2);
    if (PHI) acc[0] += f;
    if (FIELD) {
        constexpr int e = PHI ? 1 : 0;
        acc[e * stride] += e0;
        acc[(e + 1) * stride] += e1;
        acc[(e + 2) * stride] += e2;
    }
}

// What the terms of a row can have lost against 2^-54 of a target's sums: 1 the
// potential, 2 the field.  Out of line, like the next one: rare, and written into
// k_p2p_fx the two took 1.5 % of its time (200k Plummer charges 3.33 instead of 3.28
// ms an evaluate).
template <bool PHI, bool FIELD>
__device__ __noinline__ int fx_lost(const u64 *lost, int bp, int be, double f, double e0, double e1, double e2)
{
    int redo = 0;
    if (PHI && lost[0] && scalbn((double)lost[0], bp - kUnitP + 54) > fabs(f)) redo = 1;
    if (FIELD && lost[1] && scalbn((double)lost[1], be - kUnitE + 54) > fmax(fabs(e0), fmax(fabs(e1), fabs(e2)))) redo |= 2;
    return redo;
}
// The marked targets' rows in FP64, the block's threads side by side
template <int SLO, int SHI, bool PHI, bool FIELD>
__device__ __noinline__ void fx_redo(const unsigned char *redo, int cnt, int i0, int q0, int q1, const int32_t *src,
                                     const int32_t *begin, const int32_t *end, const double *px, const double *py,
                                     const double *pz, const double *Sm, double *accd, const double *phi_far,
                                     const double *E_far, const int32_t *perm, double *phi_out, double *E_out)
{
    constexpr int NC = (PHI ? 1 : 0) + (FIELD ? 3 : 0), ef = PHI ? 1 : 0;
    const int nthr = blockDim.x, tid = threadIdx.x;
    for (int u = 0; u < cnt; ++u) {
        const int which = redo[u], iu = i0 + u;
        if (which == 0) continue;
        for (int c = 0; c < NC; ++c) accd[c * nthr + tid] = 0.0;
        for (int q = q0; q < q1; ++q) {
            const int B = src[q], je = end[B];
            for (int j = begin[B] + tid; j < je; j += nthr)
                fx_close<SLO, SHI, PHI, FIELD>(iu, j, px, py, pz, Sm, accd + tid, nthr);
        }
        __syncthreads();
        if (tid < NC && (which >> (tid >= ef) & 1)) {
            double d = 0.0;
            for (int w = 0; w < nthr; ++w) d += accd[tid * nthr + w];
            const int64_t o = perm[iu];
            if (tid < ef) phi_out[o] = phi_far[iu] + d;
            else E_out[3 * o + tid - ef] = E_far[3 * (int64_t)iu + tid - ef] + d;
        }
        __syncthreads();
    }
}

// One block per target leaf, several (blockIdx.y) where a leaf of the deepest level
// holds more than max_leaf: one block took its tiles in turn (3,000 coincident
// dipoles among 50,000 others 200 -> 35 ms, most of it the FP64 sums of those
// targets; 3,000 within 1e-9 of each other 86 -> 15.5 ms).  That is the LONG form: the
// kernel without it is faster (262k Plummer dipoles 8.43 instead of 8.58 ms an
// evaluate).  The leaf's targets are cut into m tiles of t (the cut that leaves the
// fewest threads without work), each covered k = floor(threads / t) times; copy c
// takes the staged sources c, c + k, ...
// Sources are staged already in fixed point and in the target leaf's frame: a
// thread converts one source, about 3 % of the work of the pairs it serves.
// A round holds sources of one coordinate unit (the coarser of the two leaves'
// half sides): partner leaves come in order of level, so units change only
// between rounds.
// The charges' potential fits 64 registers, which holds it at 16 blocks of 128 an SM
// (500k charges: 6.16 ms, 6.5 with 111 registers); the others need all 128.
template <int SLO, int SHI, bool PHI, bool FIELD, bool LONG>
__global__ void __launch_bounds__(512, SHI == 0 && !FIELD ? 2 : 1)
k_p2p_fx(const int32_t *leaves, const int32_t *begin, const int32_t *end, const int32_t *off,
         const int32_t *src, const int32_t *level, const int32_t *cx, const int32_t *cy, const int32_t *cz,
         const int32_t *sys, const double *sys_box, const double *px, const double *py, const double *pz,
         const double *Sm, const double *phi_far, const double *E_far, const int32_t *perm, double *phi_out,
         double *E_out)
{
    pdl_wait();
    using Rec = FxRec<SLO, SHI, PHI, FIELD>;
    constexpr int nS = Orders<SLO, SHI>::n;
    constexpr int NC = (PHI ? 1 : 0) + (FIELD ? 3 : 0);
    constexpr int CH = Rec::ch, NW = Rec::nw;
    constexpr int kCarry = 16 >> (SHI - SLO);              // steps between carries
    constexpr int ef = PHI ? 1 : 0;
    extern __shared__ __align__(16) int fxsm[];
    const int nthr = blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarp = nthr >> 5;
    double *accd = (double *)fxsm;                         // [NC][nthr]
    int4 *stage = (int4 *)(accd + NC * nthr);              // [NW][CH]
    s64 *red = (s64 *)stage;                               // [4 NC][nthr], after the last round
    __shared__ int gbeg[kFxGroups], gpre[kFxGroups + 1];
    __shared__ int s_next_q, s_next_j, s_ng, s_key;
    __shared__ int s_g, s_mx[3];
    __shared__ u64 s_lost[2];                              // what the row's terms can lose, units of the sums
    __shared__ unsigned char s_redo[512];
    const int A = leaves[blockIdx.x];
    const int b = begin[A], nt = end[A] - b;
    const int parts = LONG && nt > 2 * nthr ? (int)gridDim.y : 1;     // blocks that share the leaf
    if (nt == 0 || (LONG && (int)blockIdx.y >= parts)) return;
    const int q0 = off[A], q1 = off[A + 1];
    const int lA = level[A], sy = sys[A];
    const int lside = ilogb(sys_box[4 * sy + 3]);
    // the row: range of the separations in half sides of the coarser leaf,
    // sources, largest moment exponent per shell
    if (tid < 3) s_mx[tid] = kNone;
    if (tid == 3) s_g = 1;
    if (tid >= 4 && tid < 6) s_lost[tid - 4] = 0;
    __syncthreads();
    {
        const s64 rA = 1ll << (kLevels - lA);
        const s64 zx = (2ll * cx[A] + 1) * rA, zy = (2ll * cy[A] + 1) * rA, zz = (2ll * cz[A] + 1) * rA;
        int g = 1, mx[3] = {kNone, kNone, kNone};
        for (int q = q0 + warp; q < q1; q += nwarp) {      // a warp per partner leaf
            const int B = src[q], lB = level[B], key = min(lA, lB);
            const s64 rB = 1ll << (kLevels - lB);
            const s64 ax = llabs((2ll * cx[B] + 1) * rB - zx), ay = llabs((2ll * cy[B] + 1) * rB - zy),
                      az = llabs((2ll * cz[B] + 1) * rB - zz);
            const s64 ext = max(ax, max(ay, az)) + rA + rB;
            g = max(g, (64 - __clzll(ext - 1)) - (kLevels - key));
            const int jb = begin[B], je = end[B];
            const int lu = lside - key - 1;
            for (int j = jb + lane; j < je; j += 32) {
                const double *Sj = Sm + (int64_t)j * nS;
                int o = 0;
#pragma unroll
                for (int s = SLO; s <= SHI; ++s) {
                    const int em = fx_moment_exp(Sj + o, (s + 1) * (s + 2) / 2);
                    o += (s + 1) * (s + 2) / 2;
                    if (em == kBad) mx[s] = 1 << 20;
                    else if (em != kNone) mx[s] = max(mx[s], em + fx_exp_room(s) - (s + 2) * lu);
                }
            }
        }
#pragma unroll
        for (int s = SLO; s <= SHI; ++s) {
            const int v = (int)__reduce_max_sync(0xffffffffu, mx[s]);
            if (lane == 0) atomicMax(&s_mx[s], v);
        }
        if (lane == 0) atomicMax(&s_g, g);
    }
    __syncthreads();
    const int g1 = s_g + 1, F = 61 - s_g;
    // bases: the shift of a pair's factor is base - (exponent of its term)
    int be = kNone, bp = kNone;
    bool bad = false;
#pragma unroll
    for (int s = SLO; s <= SHI; ++s) {
        const int mx = s_mx[s];
        bad |= mx == 1 << 20;
        if (mx == kNone) continue;
        be = max(be, mx + (s + 2) * (kShMax - g1) - fx_off_e(s));
        bp = max(bp, mx + (s + 1) * (kShMax - g1) - fx_off_p(s));
    }
    if (be == kNone) be = bp = 0;
    // mx holds em - (s + 2) lu, the potential's terms go with em - (s + 1) lu:
    // at most the row's coarsest unit (its first partner's) more
    bp += lside - 1 - min(lA, q1 > q0 ? level[src[q0]] : lA);
    for (int c = 0; c < NC; ++c) accd[c * nthr + tid] = 0.0;

    // tiles: m passes over the sources with k copies each, m / k smallest
    int tile = nt, best = 1 << 30;
    {
        const int m0 = (nt + nthr - 1) / nthr;
        for (int m = m0; m < m0 + 4; ++m) {
            const int t = (nt + m - 1) / m, cost = m * (1000 / (nthr / t)) + 12 * m;
            if (cost < best) { best = cost; tile = t; }
        }
    }
    const int stride = parts * tile;
    for (int t0 = LONG ? (int)blockIdx.y * tile : 0; t0 < nt; t0 += stride) {
        const int cnt = min(tile, nt - t0), k = nthr / cnt;
        const int ti = tid % cnt, sp = tid / cnt;
        const bool act = sp < k;
        const int i = b + t0 + ti;
        s64 P[NC][4];
#pragma unroll
        for (int c = 0; c < NC; ++c) P[c][0] = P[c][1] = P[c][2] = P[c][3] = 0;
        if (bad) {
            // a non-finite moment in the row: FP64 throughout
            if (act) {
                int n = 0;
                for (int q = q0; q < q1; ++q) {
                    const int B = src[q];
                    for (int j = begin[B]; j < end[B]; ++j, ++n)
                        if (n % k == sp) fx_close<SLO, SHI, PHI, FIELD>(i, j, px, py, pz, Sm, accd + tid, nthr);
                }
            }
        } else {
            s64 tx = 0, ty = 0, tz = 0;
            int key_t = -1;
            int q = q0, j_in = 0;
            if (tid < 2) s_lost[tid] = 0;                  // the round's barriers come first
            while (q < q1) {
                __syncthreads();
                if (tid < 32) {
                    // up to 32 partner leaves of one unit, as many as fit CH sources (the
                    // last one possibly in part)
                    const int qq = q + lane;
                    int lb = 0, take = 0, sl = 0, key = -1;
                    if (qq < q1) {
                        sl = src[qq];
                        key = min(level[sl], lA);
                        lb = begin[sl] + (lane == 0 ? j_in : 0);
                        take = end[sl] - lb;
                    }
                    const int key0 = __shfl_sync(0xffffffffu, key, 0);
                    int incl = take;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int y = __shfl_up_sync(0xffffffffu, incl, o);
                        if (lane >= o) incl += y;
                    }
                    const int excl = incl - take;
                    const bool in = qq < q1 && excl < CH && key == key0;
                    const int tk = in ? min(take, CH - excl) : 0;
                    if (in) {
                        gbeg[lane] = lb;
                        gpre[lane] = excl;
                    }
                    const int ng = __popc(__ballot_sync(0xffffffffu, in));
                    if (lane == ng - 1) {
                        const bool whole = tk == take;
                        gpre[ng] = excl + tk;
                        s_ng = ng;
                        s_key = key0;
                        s_next_q = whole ? qq + 1 : qq;
                        s_next_j = whole ? 0 : (lb - begin[sl]) + tk;
                    }
                }
                __syncthreads();
                const int ng = s_ng, used = gpre[ng], key = s_key;
                // coordinates in 2^-F of the unit 2^lU, from the target leaf's centre
                const int lU = lside - key - 1, sc = F - lU;
                const int fa = F - (lA - key);
                const s64 zx = fix64(sys_box[4 * sy], sc) + (s64)((u64)(2ll * cx[A] + 1) << fa);
                const s64 zy = fix64(sys_box[4 * sy + 1], sc) + (s64)((u64)(2ll * cy[A] + 1) << fa);
                const s64 zz = fix64(sys_box[4 * sy + 2], sc) + (s64)((u64)(2ll * cz[A] + 1) << fa);
                for (int d = tid; d < used; d += nthr) {
                    int lo = 0, hi = ng - 1;
                    while (lo < hi) {
                        const int mid = (lo + hi + 1) >> 1;
                        if (gpre[mid] <= d) lo = mid; else hi = mid - 1;
                    }
                    const int j = gbeg[lo] + (d - gpre[lo]);
                    int r[4 * NW];
                    put64(r, 0, fix64(px[j], sc) - zx);
                    put64(r, 2, fix64(py[j], sc) - zy);
                    put64(r, 4, fix64(pz[j], sc) - zz);
                    r[6] = j;
#pragma unroll
                    for (int w = Rec::words; w < 4 * NW; ++w) r[w] = 0;
                    if (fx_stage_orders<SLO, SLO, SHI, PHI, FIELD>(Sm + (int64_t)j * nS, bp, be, g1 + lU, r))
                        fx_count_loss<SLO, SHI, PHI, FIELD>(
                            Sm + (int64_t)j * nS, bp, be, g1 + lU,
                            max(max(llabs(word64(r, 0)), llabs(word64(r, 2))), llabs(word64(r, 4))) - (1ll << fa), s_lost);
#pragma unroll
                    for (int w = 0; w < NW; ++w)
                        stage[w * CH + d] = make_int4(r[4 * w], r[4 * w + 1], r[4 * w + 2], r[4 * w + 3]);
                }
                if (act && key != key_t) {                 // the target in this round's unit
                    tx = fix64(px[i], sc) - zx;
                    ty = fix64(py[i], sc) - zy;
                    tz = fix64(pz[i], sc) - zz;
                    key_t = key;
                }
                __syncthreads();
                if (act) {
                    int until = kCarry;
                    for (int jj = sp; jj < used; jj += k) {
                        int r[4 * NW];
#pragma unroll
                        for (int w = 0; w < NW; ++w) {
                            const int4 v = stage[w * CH + jj];
                            r[4 * w] = v.x; r[4 * w + 1] = v.y; r[4 * w + 2] = v.z; r[4 * w + 3] = v.w;
                        }
                        const FxGeo g = fx_geo(word64(r, 0) - tx, word64(r, 2) - ty, word64(r, 4) - tz);
                        const bool close = g.sh > kShMax;
                        fx_pair_orders<SLO, SLO, SHI, PHI, FIELD>(g, r, close, P);
                        if (close && r[6] != i)
                            fx_close<SLO, SHI, PHI, FIELD>(i, r[6], px, py, pz, Sm, accd + tid, nthr);
                        if (--until == 0) {
                            until = kCarry;
#pragma unroll
                            for (int c = 0; c < NC; ++c) fx_carry(P[c]);
                        }
                    }
#pragma unroll
                    for (int c = 0; c < NC; ++c) fx_carry(P[c]);
                }
                q = s_next_q;
                j_in = s_next_j;
            }
        }
        __syncthreads();
#pragma unroll
        for (int c = 0; c < NC; ++c)
#pragma unroll
            for (int l = 0; l < 4; ++l) red[(4 * c + l) * nthr + tid] = P[c][l];
        __syncthreads();
        int redo = 0;                                      // 1 the potential, 2 the field
        if (tid < cnt) {
            // the copies' integers, exact in any order, then the FP64 pairs in copy order
            double v[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                s64 p[4] = {0, 0, 0, 0};
                double d = 0.0;
                for (int u = 0; u < k; ++u) {
                    const int o = u * cnt + tid;
#pragma unroll
                    for (int l = 0; l < 4; ++l) p[l] += red[(4 * c + l) * nthr + o];
                    d += accd[c * nthr + o];
                }
                v[c] = fx_value(p, PHI && c == 0 ? bp - kUnitP : be - kUnitE) + d;
            }
            const int64_t o = perm[i];
            if (PHI) phi_out[o] = phi_far[i] + v[0];
            if (FIELD) {
#pragma unroll
                for (int a = 0; a < 3; ++a) E_out[3 * o + a] = E_far[3 * (int64_t)i + a] + v[ef + a];
            }
            if (s_lost[0] | s_lost[1])
                redo = fx_lost<PHI, FIELD>(s_lost, bp, be, v[0], v[FIELD ? ef : 0], v[FIELD ? ef + 1 : 0], v[FIELD ? ef + 2 : 0]);
        }
        if (__syncthreads_or(redo)) {
            if (tid < cnt) s_redo[tid] = (unsigned char)redo;
            __syncthreads();
            fx_redo<SLO, SHI, PHI, FIELD>(s_redo, cnt, b + t0, q0, q1, src, begin, end, px, py, pz, Sm, accd, phi_far, E_far,
                                          perm, phi_out, E_out);
        }
        if (t0 + stride < nt)
            for (int c = 0; c < NC; ++c) accd[c * nthr + tid] = 0.0;
    }
}

template <int SLO, int SHI>
void launch_fx(fmm_tree *t, int want_phi, int want_field, double *phi, double *E)
{
    // 128 threads a leaf; where the leaves would leave the chip idle, more copies of each
    const int64_t sms = std::max(1, sm_count());
    const int nthr = t->nleaves >= 4 * sms ? 128 : (t->nleaves >= 2 * sms ? 256 : 512);
    // blocks a leaf: two tiles or so each, and not many millions of blocks with nothing to do
    const int64_t want = t->long_leaf ? (t->long_leaf + 2 * nthr - 1) / (2 * nthr) : 1;
    const unsigned parts = (unsigned)std::min<int64_t>({want, 256, std::max<int64_t>(8, (1 << 20) / t->nleaves)});
    auto go = [&](auto kern, int nw, int ch, int nc) {
        const size_t smem = 8 * (size_t)nc * nthr +
                            std::max<size_t>(16 * (size_t)nw * ch, 32 * (size_t)nc * nthr);
        allow_max_dynamic_smem(kern);
        launch_next(t->stream, kern, dim3((unsigned)t->nleaves, parts), nthr, smem,
            (const int32_t *)t->b_leaves.ptr, (const int32_t *)t->b_begin.ptr, (const int32_t *)t->b_end.ptr,
            (const int32_t *)t->b_p2p_off.ptr, (const int32_t *)t->b_p2p_src.ptr, (const int32_t *)t->b_level.ptr,
            (const int32_t *)t->b_cx.ptr, (const int32_t *)t->b_cy.ptr, (const int32_t *)t->b_cz.ptr,
            (const int32_t *)t->b_sys.ptr, (const double *)t->b_sysbox.ptr, (const double *)t->b_px.ptr,
            (const double *)t->b_py.ptr, (const double *)t->b_pz.ptr, (const double *)t->b_S.ptr,
            (const double *)t->b_phi.ptr, (const double *)t->b_E.ptr, (const int32_t *)t->b_perm.ptr, phi, E);
    };
    auto pick = [&](auto phi_t, auto field_t) {
        constexpr bool PHI = decltype(phi_t)::value, FIELD = decltype(field_t)::value;
        using Rec = FxRec<SLO, SHI, PHI, FIELD>;
        constexpr int nc = (PHI ? 1 : 0) + (FIELD ? 3 : 0);
        if (parts > 1) go(k_p2p_fx<SLO, SHI, PHI, FIELD, true>, Rec::nw, Rec::ch, nc);
        else go(k_p2p_fx<SLO, SHI, PHI, FIELD, false>, Rec::nw, Rec::ch, nc);
    };
    if (want_phi && want_field) pick(std::true_type(), std::true_type());
    else if (want_phi) pick(std::true_type(), std::false_type());
    else pick(std::false_type(), std::true_type());
}

}  // namespace

void launch_p2p_fx(fmm_tree *t, int want_phi, int want_field, double *phi, double *E)
{
    switch (t->s * 3 + t->s_hi) {
    case 0: launch_fx<0, 0>(t, want_phi, want_field, phi, E); break;
    case 1: launch_fx<0, 1>(t, want_phi, want_field, phi, E); break;
    case 2: launch_fx<0, 2>(t, want_phi, want_field, phi, E); break;
    case 4: launch_fx<1, 1>(t, want_phi, want_field, phi, E); break;
    case 5: launch_fx<1, 2>(t, want_phi, want_field, phi, E); break;
    default: launch_fx<2, 2>(t, want_phi, want_field, phi, E); break;
    }
    ++t->launches;
}

}  // namespace fmm
