// bh.cu -- multipolar Barnes-Hut (§2 multipole potential; §3.2 Methods), FP64.
//
// Multipoles of order p (s <= |m| <= p: the P2M/M2M of the FMM storage at
// order p - s), then for every target a walk from its system's root: a cell
// with r_cell^2 < theta^2 |x - x_c|^2 (r_cell = half side, strict) is taken by
// M2P, phi += sum_m M_m D_m(x - z_c), E -= sum_m M_m D_{m+e_k}(x - z_c); a
// failing leaf by P2P with its particles; a failing inner cell is opened.
//
// One warp walks 32 consecutive targets of the sorted order (neighbours in
// space) together: a shared stack of (cell, lanes) entries, where "lanes" are
// the targets for which the cell is reached (their walks opened its parent).
// Each lane takes its own MAC decision, so every target sees exactly its own
// walk; a cell is visited once for all the lanes that reach it.  The MAC is
// evaluated with explicitly rounded operations (no contraction), in the order
// ((dx dx + dy dy) + dz dz), so the decisions are those of a plain FP64 program.
//
// M2P evaluates the cell's potential in solid harmonics.  With eta = d_x + i d_y
// and H_l^m = d_z^(l-m) eta^m (1/r), m = 0..l, every D_k = grad^k (1/r) of
// degree l is a combination of the Re and Im of those 2l + 1 functions: d_x =
// (eta + eta*)/2, d_y = (eta - eta*)/(2i) and, 1/r being harmonic, eta eta* =
// -d_z^2.  So each cell's Cartesian multipole becomes (p + 1)^2 coefficients
// c_l^m once (k_bh_coef; the map's entries are binomials over powers of two),
// phi = Re sum c_l^m H_l^m, and with d_x H_l^m = (H_{l+1}^{m+1} -
// H_{l+1}^{m-1})/2, d_y H_l^m = (H_{l+1}^{m+1} + H_{l+1}^{m-1})/(2i), d_z H_l^m
// = H_{l+1}^m the field takes the same coefficients.  The H follow row by row
// from H_0^0 = 1/r,
//   H_{l+1}^m = -((2l + 1) z H_l^m + (l^2 - m^2) H_{l-1}^m) / r^2,
//   H_{l+1}^{l+1} = -(2l + 1) (x + iy) H_l^l / r^2,
// about 250 FP64 operations per M2P at p = 4 with the field, against 560 for the
// Cartesian D recurrence and contraction.  The walk is bound by the FP64 pipe.
//
// An accepted cell goes into its target's queue, a failing leaf into another.
// When a queue is full, and at the end, the warp deals all queued (target, cell)
// tasks to its 32 lanes, first entries first, whichever lane owns them, and the
// owners add the results in the order of their walks, the M2P and the P2P sums
// apart, so that a target's result does not depend on the warp's other targets.
// (The targets of a warp agree on half of their cells and a quarter of their
// leaves: evaluated as the walk meets them, two FP64 lanes of three were idle.)
// A block is one warp and 8, 16 or 32 targets: fewer where there are few, so
// that the chip fills and the last blocks end together.  One Barnes-Hut step of
// 100,000 charges, p = 4, theta = 0.5, potential and field: 17.6 -> 5.6 ms.
#include <cstring>
#include <algorithm>
#include <utility>
#include <vector>

#include "fmm_internal.cuh"
#include "pair.cuh"

namespace fmm {

namespace {

// pending roots (<= 31) + 7 per level (pop one, push <= 8) over 21 levels + 8
constexpr int kBHStack = 256;
constexpr int kBHQueue = 32;               // accepted cells a lane holds
constexpr int kBHLeaves = 8;               // failing leaves a lane holds

struct BHArgs {
    int64_t n;
    int nsys, p, l0, tpw;    // degrees l0 .. p; targets per warp
    double theta2;
    const int32_t *nchild, *child, *begin, *end;
    const double *centre, *half;
    const double *px, *py, *pz, *Sm;
    const int32_t *perm;
    const double *C;         // per cell and degree l: Re c_l^0, then Re c_l^m, -Im c_l^m, m = 1..l
    unsigned long long *count;   // [M2P evaluations, P2P pairs], added per warp
    double *phi_out, *E_out;
};

// Coefficients of every cell: C[cell][q] = sum over the map's entries of row q
// (multipole index, factor).  One warp per cell.
__global__ void __launch_bounds__(128)
k_bh_coef(const double *M, int nM, int64_t nc, int nC, const int *off, const int *idx, const double *fac, double *C)
{
    const int64_t c = blockIdx.x * 4ll + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (c >= nc) return;
    const double *Mc = M + c * nM;
    for (int q = lane; q < nC; q += 32) {
        double v = 0.0;
        for (int k = off[q]; k < off[q + 1]; ++k) v = fma(fac[k], Mc[idx[k]], v);
        C[c * nC + q] = v;
    }
}

__constant__ double b_odd[kMaxOrder + 2];      // -(2 l + 1)
__constant__ double b_sq[kMaxOrder + 2];       // l^2

// The M2P of one cell for this lane: R = x - z_c, h0, h1 = this lane's columns of
// two rows of H (Re at [64 m], Im at [64 m + 32]).
template <bool PHI, bool FIELD>
__device__ __forceinline__ void m2p(double X, double Y, double Z, const double *C, int l0, int p, double *h0,
                                    double *h1, double &f, double &e0, double &e1, double &e2)
{
    const double r2 = fma(X, X, fma(Y, Y, Z * Z));
    const double y = rsqrt_hh(r2);
    const double w = y * y;                                    // 1/r^2
    const double zw = Z * w, xw = X * w, yw = Y * w;
    double *h = h0, *hp = h1;                                  // row l, row l - 1
    h[0] = y;
    h[32] = 0.0;
    double sr = y, si = 0.0;                                   // H_l^l
    double pf = 0.0, g0 = 0.0, g1 = 0.0, g2 = 0.0;
    const double *c = C;
    for (int l = 0; l <= p; ++l) {
        // row l + 1 over row l - 1 (needed for the field, and for the next degree)
        const bool next = FIELD || l < p;
        double *hn = hp;
        if (next) {
            const double t1 = b_odd[l] * zw, ll = b_sq[l];
            hn[0] = l ? fma(t1, h[0], -(ll * w) * hp[0]) : t1 * h[0];
            for (int m = 1; m <= l; ++m) {
                const double re = t1 * h[64 * m], im = t1 * h[64 * m + 32];
                if (m < l) {
                    const double t2 = (b_sq[m] - ll) * w;
                    hn[64 * m] = fma(t2, hp[64 * m], re);
                    hn[64 * m + 32] = fma(t2, hp[64 * m + 32], im);
                } else {
                    hn[64 * m] = re;
                    hn[64 * m + 32] = im;
                }
            }
            const double ur = b_odd[l] * xw, ui = b_odd[l] * yw;
            const double nr = fma(ur, sr, -(ui * si));
            si = fma(ur, si, ui * sr);
            sr = nr;
            hn[64 * (l + 1)] = sr;
            hn[64 * (l + 1) + 32] = si;
        }
        if (l >= l0) {
            const double a = __ldg(c);
            if (PHI) pf = fma(a, h[0], pf);
            if (FIELD) {
                g0 = fma(a, hn[64], g0);
                g1 = fma(a, hn[96], g1);
                g2 = fma(a, hn[0], g2);
            }
            double lr = FIELD ? hn[0] : 0.0, li = 0.0;         // H_{l+1}^{m-1}
            double mr = FIELD ? hn[64] : 0.0, mi = FIELD ? hn[96] : 0.0;   // H_{l+1}^m
            for (int m = 1; m <= l; ++m) {
                const double A = __ldg(c + 2 * m - 1), B = __ldg(c + 2 * m);
                if (PHI) pf = fma(A, h[64 * m], fma(B, h[64 * m + 32], pf));
                if (FIELD) {
                    const double ur = hn[64 * (m + 1)], ui = hn[64 * (m + 1) + 32];
                    const double A2 = 0.5 * A, B2 = 0.5 * B;
                    g0 = fma(A2, ur - lr, fma(B2, ui - li, g0));
                    g1 = fma(A2, ui + li, fma(-B2, ur + lr, g1));
                    g2 = fma(A, mr, fma(B, mi, g2));
                    lr = mr; li = mi;
                    mr = ur; mi = ui;
                }
            }
            c += 2 * l + 1;
        }
        hp = h;
        h = hn;
    }
    if (PHI) f += pf;
    if (FIELD) { e0 -= g0; e1 -= g1; e2 -= g2; }
}

// SHI > S: every particle carries the orders S..SHI (mixed systems)
template <int S, bool PHI, bool FIELD, int SHI = S>
__global__ void __launch_bounds__(32)
k_bh(BHArgs a)
{
    constexpr int nS = Orders<S, SHI>::n;
    constexpr unsigned kAll = 0xffffffffu;
    extern __shared__ double bsm[];
    __shared__ int st_c[kBHStack];
    __shared__ unsigned st_m[kBHStack];
    __shared__ int queue[kBHQueue][32], lqueue[kBHLeaves][32], task[32];
    __shared__ double res[4][32];
    const int lane = threadIdx.x;
    const int row = 64 * (a.p + 1 + (FIELD ? 1 : 0));                // doubles of a row of H for a warp
    double *hl = bsm + lane;
    const int nC = (a.p + 1) * (a.p + 1) - a.l0 * a.l0;
    const int64_t i = (int64_t)blockIdx.x * a.tpw + lane;
    const bool valid = lane < a.tpw && i < a.n;
    const double x = valid ? a.px[i] : 0.0, y = valid ? a.py[i] : 0.0, z = valid ? a.pz[i] : 0.0;
    double f = 0.0, e0 = 0.0, e1 = 0.0, e2 = 0.0;              // P2P
    double mf = 0.0, m0 = 0.0, m1 = 0.0, m2 = 0.0;             // M2P
    int qn = 0, ln = 0;                    // entries of this lane's queues
    // Deals the queued tasks (cnt per lane, cells in q[slot][lane]) to the lanes in
    // order of slot, then lane: eval(cell, target's x, y, z) gives a task's four
    // values; its owner adds them to s0..s3.
    auto deal = [&](int &cnt, const int (*q)[32], auto eval, double &s0, double &s1, double &s2, double &s3) {
        const unsigned below = (1u << lane) - 1u;
        int j = 0, skip = 0;               // the next task: the skip-th one of slot j
        __syncwarp();
        for (;;) {
            int base = -skip, jj = j;
            for (; base < 32; ++jj) {
                const unsigned m = __ballot_sync(kAll, cnt > jj);
                if (m == 0) break;
                const int pos = base + __popc(m & below);
                if (cnt > jj && pos >= 0 && pos < 32) task[pos] = lane | jj << 8;
                base += __popc(m);
            }
            const int nb = min(base, 32);
            if (nb <= 0) break;
            __syncwarp();
            const int tk = lane < nb ? task[lane] : lane, owner = tk & 255;
            const double tx = __shfl_sync(kAll, x, owner), ty = __shfl_sync(kAll, y, owner),
                         tz = __shfl_sync(kAll, z, owner);
            double v0 = 0.0, v1 = 0.0, v2 = 0.0, v3 = 0.0;
            if (lane < nb) eval(q[tk >> 8][owner], tx, ty, tz, v0, v1, v2, v3);
            if (PHI) res[0][lane] = v0;
            if (FIELD) { res[1][lane] = v1; res[2][lane] = v2; res[3][lane] = v3; }
            __syncwarp();
            int left = -skip, last = 0;
            for (int k = j; k < jj; ++k) {
                const unsigned m = __ballot_sync(kAll, cnt > k);
                const int pos = left + __popc(m & below);
                if (cnt > k && pos >= 0 && pos < 32) {
                    if (PHI) s0 += res[0][pos];
                    if (FIELD) { s1 += res[1][pos]; s2 += res[2][pos]; s3 += res[3][pos]; }
                }
                last = __popc(m);
                left += last;
            }
            __syncwarp();
            // the last slot may be taken in part
            skip = left > 32 ? last - (left - 32) : 0;
            j = left > 32 ? jj - 1 : jj;
        }
        cnt = 0;
    };
    auto take_cells = [&]() {
        deal(qn, queue,
             [&](int c, double tx, double ty, double tz, double &v0, double &v1, double &v2, double &v3) {
                 m2p<PHI, FIELD>(tx - a.centre[3 * c], ty - a.centre[3 * c + 1], tz - a.centre[3 * c + 2],
                                 a.C + (int64_t)c * nC, a.l0, a.p, hl, hl + row, v0, v1, v2, v3);
             },
             mf, m0, m1, m2);
    };
    auto take_leaves = [&]() {
        deal(ln, lqueue,
             [&](int c, double tx, double ty, double tz, double &v0, double &v1, double &v2, double &v3) {
                 const int je = a.end[c];
                 for (int j = a.begin[c]; j < je; ++j)
                     pair_orders<S, SHI, PHI, FIELD>(tx - a.px[j], ty - a.py[j], tz - a.pz[j],
                                                     a.Sm + (int64_t)j * nS, v0, v1, v2, v3);
             },
             f, e0, e1, e2);
    };
    // FP32 copies for the MAC: most cells pass or fail it by far more than the
    // rounding of the copies, which spares them the ten FP64 operations (squares
    // near FP32's smallest, whose rounding is not relative, take the FP64 test)
    const float xf = (float)x, yf = (float)y, zf = (float)z, t2f = (float)a.theta2;
    const float af = fmaxf(fabsf(xf), fmaxf(fabsf(yf), fabsf(zf)));
    unsigned long long n_m2p = 0, n_p2p = 0;
    int root = 0;
    if (valid) {                          // the last root whose particle range starts at or before i
        int lo = 0, hi = a.nsys - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (a.begin[mid] <= i) lo = mid; else hi = mid - 1;
        }
        root = lo;
    }
    int top = 0;
    for (unsigned rem = __ballot_sync(kAll, valid); rem;) {
        const int r = __shfl_sync(kAll, root, __ffs(rem) - 1);
        const unsigned m = __ballot_sync(kAll, valid && root == r);
        if (lane == 0) {
            st_c[top] = r;
            st_m[top] = m;
        }
        ++top;
        rem &= ~m;
    }
    __syncwarp();
    while (top > 0) {
        --top;
        const int c = st_c[top];
        const unsigned m = st_m[top];
        __syncwarp();                     // read by every lane before a push overwrites it
        bool acc = false;
        if ((m >> lane) & 1u) {
            const double cx = a.centre[3 * c], cy = a.centre[3 * c + 1], cz = a.centre[3 * c + 2], h = a.half[c];
            // |d| and its error: each coordinate is off by at most 2^-23 (|x| + |d|)
            const float fx = xf - (float)cx, fy = yf - (float)cy, fz = zf - (float)cz, hf = (float)h;
            const float dd = fmaf(fx, fx, fmaf(fy, fy, fz * fz)), d1 = fabsf(fx) + fabsf(fy) + fabsf(fz);
            const float m = fmaf(4.8e-7f * (af + d1), d1 + af * 2.4e-7f, 2e-6f * dd), hh = hf * hf;
            if (dd > 1e-30f && dd < 1e30f && hh > 1e-30f && hh < 1e30f && hh * 1.000002f < t2f * (dd - m) * 0.999998f) {
                acc = true;
            } else if (!(dd > 1e-30f && dd < 1e30f && hh > 1e-30f && hh * 0.999998f > t2f * (dd + m) * 1.000002f)) {
                const double dx = __dsub_rn(x, cx), dy = __dsub_rn(y, cy), dz = __dsub_rn(z, cz);
                const double d2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
                acc = __dmul_rn(h, h) < __dmul_rn(a.theta2, d2);
            }
        }
        if (acc) {
            queue[qn++][lane] = c;
            ++n_m2p;
        }
        if (__any_sync(kAll, qn == kBHQueue)) take_cells();
        const unsigned om = m & ~__ballot_sync(kAll, acc);    // lanes for which c failed
        if (om == 0) continue;
        const int nch = a.nchild[c];
        if (nch == 0) {                   // P2P with the leaf's particles
            if ((om >> lane) & 1u) {
                n_p2p += (unsigned long long)(a.end[c] - a.begin[c]);
                lqueue[ln++][lane] = c;
            }
            if (__any_sync(kAll, ln == kBHLeaves)) take_leaves();
        } else {                          // open: children pushed last-first, taken in order
            const int ch0 = a.child[c];
            if (lane == 0)
                for (int k = 0; k < nch; ++k) {
                    st_c[top + k] = ch0 + nch - 1 - k;
                    st_m[top + k] = om;
                }
            top += nch;
            __syncwarp();
        }
    }
    take_cells();
    take_leaves();
    f += mf;
    e0 += m0; e1 += m1; e2 += m2;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        n_m2p += __shfl_xor_sync(kAll, n_m2p, o);
        n_p2p += __shfl_xor_sync(kAll, n_p2p, o);
    }
    if (lane == 0) {
        atomicAdd(a.count, n_m2p);
        atomicAdd(a.count + 1, n_p2p);
    }
    if (valid) {
        const int64_t o = a.perm[i];
        if (PHI) a.phi_out[o] = f;
        if (FIELD) {
            a.E_out[3 * o] = e0;
            a.E_out[3 * o + 1] = e1;
            a.E_out[3 * o + 2] = e2;
        }
    }
}

template <int S, int SHI = S>
void launch_bh_s(const BHArgs &a, int want_phi, int want_field, unsigned grid, int threads, size_t smem,
                 cudaStream_t st)
{
    auto go = [&](auto kern) {
        allow_max_dynamic_smem(kern);
        kern<<<grid, threads, smem, st>>>(a);
    };
    if (want_phi && want_field) go(k_bh<S, true, true, SHI>);
    else if (want_phi) go(k_bh<S, true, false, SHI>);
    else go(k_bh<S, false, true, SHI>);
}

// The map from a Cartesian multipole to the coefficients c_l^m (see the file
// header): rows in the order of BHArgs::C, entries (multipole index, factor).
struct BHMap {
    std::vector<int> off, idx;
    std::vector<double> fac;
};

BHMap bh_map(int l0, int p)
{
    const MultiIndex &I = multi_index();
    std::vector<std::vector<std::pair<int, double>>> rows((size_t)((p + 1) * (p + 1) - l0 * l0));
    const int first = ntot(l0 - 1);
    for (int k = first; k < ntot(p); ++k) {
        const int a = I.nx[k], b = I.ny[k], l = a + b + I.nz[k], N = a + b;
        // ((eta + eta*)/2)^a ((eta - eta*)/(2i))^b: g[j] = the factor of eta^j eta*^(N-j)
        // without i^-b; products of small integers over 2^N, exact
        std::vector<double> g(1, 1.0);
        for (int f = 0; f < N; ++f) {
            std::vector<double> h(g.size() + 1, 0.0);
            const double sg = f < a ? 1.0 : -1.0;
            for (size_t j = 0; j < g.size(); ++j) {
                h[j + 1] += 0.5 * g[j];
                h[j] += sg * 0.5 * g[j];
            }
            g = h;
        }
        const int base = l * l - l0 * l0;
        for (int j = 0; j <= N; ++j) {
            const int m = std::abs(2 * j - N), lo = std::min(j, N - j);
            double v = g[j] * (lo & 1 ? -1.0 : 1.0);       // eta eta* = -d_z^2
            if (v == 0.0) continue;
            // times i^-b: real (b even, sign (-1)^(b/2)) or imaginary (-i (-1)^((b-1)/2))
            if (b % 4 == 2 || b % 4 == 3) v = -v;
            if (b % 2 == 0) {
                rows[(size_t)(base + (m ? 2 * m - 1 : 0))].push_back({k - first, v});     // v Re H
            } else if (m) {
                // -i v H or -i v H*: the real part is v Im H, or -v Im H for the conjugate
                rows[(size_t)(base + 2 * m)].push_back({k - first, 2 * j > N ? v : -v});
            }
        }
    }
    BHMap M;
    M.off.push_back(0);
    for (auto &r : rows) {
        // one entry per multipole term (j and N - j meet in the same row)
        for (size_t q = 0; q < r.size(); ++q) {
            if (q && M.idx.size() > (size_t)M.off.back() && M.idx.back() == r[q].first) M.fac.back() += r[q].second;
            else { M.idx.push_back(r[q].first); M.fac.push_back(r[q].second); }
        }
        M.off.push_back((int)M.idx.size());
    }
    return M;
}

}  // namespace

fmm_status run_bh(fmm_tree *t, int p, double theta, int want_phi, int want_field, double *phi_out,
                  double *E_out)
{
    cudaStream_t st = t->stream;
    const int s = t->s;
    DevTables tb;
    const int32_t *lut;
    FMM_TRY(upload_tables(t, s, p - s, 0, &tb, &lut));
    FMM_TRY(run_upward(t, tb, false));
    const int nC = (p + 1) * (p + 1) - s * s;
    FMM_TRY(ensure(t, t->b_Mh, 8 * (size_t)t->ncells * nC));
    const int key = s | p << 4;
    if (t->bh_key_s != key) {
        const BHMap g = bh_map(s, p);
        // one buffer: factors (double) | offsets | indices
        const size_t b_f = 8 * g.fac.size(), b_o = 4 * g.off.size(), b_i = 4 * g.idx.size();
        std::vector<uint8_t> host(b_f + b_o + b_i);
        std::memcpy(host.data(), g.fac.data(), b_f);
        std::memcpy(host.data() + b_f, g.off.data(), b_o);
        std::memcpy(host.data() + b_f + b_o, g.idx.data(), b_i);
        double odd[kMaxOrder + 2], sq[kMaxOrder + 2];
        for (int l = 0; l < kMaxOrder + 2; ++l) { odd[l] = -(2.0 * l + 1.0); sq[l] = (double)(l * l); }
        t->bh_key_s = -1;
        FMM_TRY(cuda_check(t, cudaMemcpyToSymbolAsync(b_odd, odd, sizeof(odd), 0, cudaMemcpyHostToDevice, st), "constants"));
        FMM_TRY(cuda_check(t, cudaMemcpyToSymbolAsync(b_sq, sq, sizeof(sq), 0, cudaMemcpyHostToDevice, st), "constants"));
        FMM_TRY(ensure(t, t->b_bh_mt, host.size()));
        FMM_TRY(cuda_check(t, cudaMemcpyAsync(t->b_bh_mt.ptr, host.data(), host.size(), cudaMemcpyHostToDevice,
                                              st), "Barnes-Hut map"));
        t->bh_key_s = key;
        t->bh_nfac = (int)g.fac.size();
    }
    {
        const double *fac = (const double *)t->b_bh_mt.ptr;
        const int *off = (const int *)(fac + t->bh_nfac);
        k_bh_coef<<<(unsigned)((t->ncells + 3) / 4), 128, 0, st>>>((const double *)t->b_M.ptr, tb.nM, t->ncells, nC, off,
                                                                    off + nC + 1, fac, (double *)t->b_Mh.ptr);
        ++t->launches;
    }
    FMM_TRY(ensure(t, t->b_bh_cnt, 16));
    FMM_TRY(cuda_check(t, cudaMemsetAsync(t->b_bh_cnt.ptr, 0, 16, st), "memset"));
    BHArgs a;
    a.count = (unsigned long long *)t->b_bh_cnt.ptr;
    a.n = t->n;
    a.nsys = std::max(1, (int)t->sys_off.size() - 1);
    a.p = p;
    a.l0 = s;
    a.theta2 = theta * theta;
    a.nchild = (const int32_t *)t->b_nchild.ptr;
    a.child = (const int32_t *)t->b_child.ptr;
    a.begin = (const int32_t *)t->b_begin.ptr;
    a.end = (const int32_t *)t->b_end.ptr;
    a.centre = (const double *)t->b_centre.ptr;
    a.half = (const double *)t->b_half.ptr;
    a.px = (const double *)t->b_px.ptr;
    a.py = (const double *)t->b_py.ptr;
    a.pz = (const double *)t->b_pz.ptr;
    a.Sm = (const double *)t->b_S.ptr;
    a.perm = (const int32_t *)t->b_perm.ptr;
    a.C = (const double *)t->b_Mh.ptr;
    a.phi_out = phi_out;
    a.E_out = E_out;
    // two rows of H: 32 lanes x (degrees + 1) complex doubles
    const size_t smem = 2 * 512 * (size_t)(p + 1 + (want_field ? 1 : 0));
    // targets per warp: about three waves of sixteen warps per SM or more
    const int64_t warps = 48 * (int64_t)sm_count();
    a.tpw = t->n >= 32 * warps ? 32 : (t->n >= 16 * warps / 2 ? 16 : 8);
    const unsigned grid = (unsigned)((t->n + a.tpw - 1) / a.tpw);
    switch (s * 3 + t->s_hi) {
    case 0: launch_bh_s<0>(a, want_phi, want_field, grid, 32, smem, st); break;
    case 1: launch_bh_s<0, 1>(a, want_phi, want_field, grid, 32, smem, st); break;
    case 2: launch_bh_s<0, 2>(a, want_phi, want_field, grid, 32, smem, st); break;
    case 4: launch_bh_s<1>(a, want_phi, want_field, grid, 32, smem, st); break;
    case 5: launch_bh_s<1, 2>(a, want_phi, want_field, grid, 32, smem, st); break;
    default: launch_bh_s<2>(a, want_phi, want_field, grid, 32, smem, st); break;
    }
    ++t->launches;
    t->bh_ran = true;
    return cuda_check(t, cudaGetLastError(), "Barnes-Hut walk");
}

}  // namespace fmm
