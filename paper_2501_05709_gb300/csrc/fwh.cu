// FW-H acoustic pressure at far-field observers from a stationary permeable
// data surface in a uniformly moving medium (Appendix B, Eqs. B.2-B.14),
// advanced-time (source-time-dominant) form, in double precision.
//
//   k_fwh_delays : the smallest and largest delay R/c0 of each observer, from
//                  which the host takes its unified window (Eq. B.13).
//   k_fwh_series : per panel and source time, the thickness and loading
//                  sources Q (Eq. A.5) and L_i (Eqs. A.7-A.8, sigma_ij
//                  omitted), with u_i the disturbance velocity V - U_inf,
//                  and their 4th-order finite-difference tau-derivatives.
//   k_fwh_fix    : the series in 60-bit fixed point, one exponent per series.
//   k_fwh_accum  : per (panel, spanwise copy) the radii R*, R and their
//                  gradients (Eqs. B.8-B.12) give the integrand coefficients
//                  of Eqs. B.2-B.3; each observer time t* (unified window,
//                  step dtau) interpolates the panel integrand at
//                  tau = t* - R/c0 (Eq. B.13) with a 4-point cubic Lagrange
//                  stencil and sums (Eq. B.14), on the integer pipe; one
//                  partial row per panel group.
//   k_fwh_accum64: the same sums in double, for the observers whose records the
//                  fixed point would hold with fewer bits than a double does.
//   k_fwh_reduce : sums the partial rows in a fixed order, divides by 4 pi.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstddef>
#include <cstring>
#include <string>
#include <vector>

#include "fr.h"
#include "fr_pool.h"

namespace {

constexpr int NSER = 8;  // Q, L1, L2, L3, dQ, dL1, dL2, dL3
constexpr int kFwhGroup = 32;   // panel copies per row of partial sums

struct FwhConst {
    double M[3];
    double c0, rho0, p0, dtau, tau0;
    double b2;  // Prandtl-Glauert factor squared, 1 / (1 - |M|^2)
};

// The sources of one panel sample h = (rho, V1, V2, V3, p): n its normal, U = c0 M
// the mean flow and Un = U.n.  rho (V.n) is formed from the disturbance u = V - U as
// rho (u.n + Un), so that the rounding of Un, the same in both terms, leaves their
// difference Q (with V.n Q is off by a rounding of |U| even on panels along the flow,
// where Un is small).
__device__ __forceinline__ void sources(const double* h, const double* n, const double* U, double Un,
                                        const FwhConst& k, double* out) {
    const double u[3] = {h[1] - U[0], h[2] - U[1], h[3] - U[2]};
    const double rv = h[0] * ((u[0] * n[0] + u[1] * n[1] + u[2] * n[2]) + Un);
    out[0] = rv - k.rho0 * Un;
    const double dp = h[4] - k.p0;
    for (int i = 0; i < 3; ++i) out[1 + i] = dp * n[i] + rv * u[i];
}

// The source series of a batch of panels: layout of one panel [nt places][4 pairs]
// [2 series], pair 0 = (Q, L1), 1 = (L2, L3), 2 = (dQ, dL1), 3 = (dL2, dL3); pair v
// of place a sits at v ^ ((a >> 1) & 3), so that 8 lanes reading the same pair of
// neighbouring places touch every bank group once.  Places along time are ordered by t mod KO, then t / KO, so that
// lanes of k_fwh_accum, which are KO samples apart, read neighbouring 16-byte
// places whatever the delay.
constexpr int KO = 4;   // consecutive samples of a lane of k_fwh_accum
__host__ __device__ __forceinline__ int fwh_place(int t, int nt) {
    const int r = t & (KO - 1);
    return r * (nt / KO) + min(r, nt & (KO - 1)) + (t - r) / KO;   // t - r is a multiple of KO, also for t < 0
}
// 16-byte slot of pair v of place a within a panel
__host__ __device__ __forceinline__ unsigned fwh_slot(unsigned a, unsigned v) { return 4 * a + (v ^ ((a >> 1) & 3)); }

// k_fwh_series: a block takes 8 panels x 256 source times.  It evaluates the
// four sources once per panel and time (4 more on each side for the stencil)
// into shared memory, then warp w writes panel w's eight series, 32 neighbouring
// places per store, and keeps each series' largest magnitude (high word of the
// double, a total order on magnitudes) for the fixed-point form.  Bound by the FP64
// pipe (32 operations a panel and time).  At 18,840 panels x 1000 times 1.45 ms;
// one thread per (panel, time) with six source evaluations each and stores 64 kB
// apart took 4.93 ms.
constexpr int SER_P = 8, SER_T = 256, SER_H = 4, SER_W = SER_T + 2 * SER_H;
constexpr size_t SER_SMEM = sizeof(double) * 4 * SER_P * SER_W;

__global__ void __launch_bounds__(256) k_fwh_series(const double* __restrict__ hist, int nt, int npts, int p0, int np,
                                                    const double* __restrict__ nrm, FwhConst k,
                                                    double* __restrict__ X, int* __restrict__ hw) {
    extern __shared__ double sq[];   // [4][SER_P][SER_W]
    const int pb = blockIdx.x * SER_P, tb = blockIdx.y * SER_T;
    {
        const int lp = threadIdx.x % SER_P;
        const int p = p0 + min(pb + lp, np - 1);
        const double n[3] = {nrm[p * 3 + 0], nrm[p * 3 + 1], nrm[p * 3 + 2]};
        // rounded products: fused into V - U they would leave U's rounding in u
        const double U[3] = {__dmul_rn(k.c0, k.M[0]), __dmul_rn(k.c0, k.M[1]), __dmul_rn(k.c0, k.M[2])};
        const double Un = U[0] * n[0] + U[1] * n[1] + U[2] * n[2];
        for (int i = threadIdx.x / SER_P; i < SER_W; i += 256 / SER_P) {
            const int t = min(max(tb - SER_H + i, 0), nt - 1);
            double q[4];
            sources(hist + (int64_t(t) * npts + p) * 5, n, U, Un, k, q);
#pragma unroll
            for (int v = 0; v < 4; ++v) sq[(v * SER_P + lp) * SER_W + i] = q[v];
        }
    }
    __syncthreads();
    const int lp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (pb + lp >= np) return;
    double2* xp = reinterpret_cast<double2*>(X) + int64_t(pb + lp) * 4 * nt;
    const double s = 1.0 / (12.0 * k.dtau);
    int top[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    for (int r = 0; r < SER_T / 32; ++r) {
        const int t = tb + 32 * KO * (r / KO) + KO * lane + r % KO;
        if (t >= nt) continue;
        double x[8];
        if (t >= 2 && t <= nt - 3) {
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const double* q = sq + (v * SER_P + lp) * SER_W + (t - tb + SER_H);
                x[v] = q[0];
                x[4 + v] = ((q[-2] - q[2]) + 8.0 * (q[1] - q[-1])) * s;
            }
        } else {
            // one-sided 4th-order stencils at both ends
            const double c[4][5] = {{-25, 48, -36, 16, -3}, {-3, -10, 18, -6, 1}, {-1, 6, -18, 10, 3},
                                    {3, -16, 36, -48, 25}};
            const int j0 = t < 2 ? 0 : nt - 5, w = t < 2 ? t : t - nt + 4;
            for (int v = 0; v < 4; ++v) {
                const double* q = sq + (v * SER_P + lp) * SER_W + (SER_H - tb);
                double der = 0.0;
                for (int m = 0; m < 5; ++m) der += c[w][m] * q[j0 + m];
                x[v] = q[t];
                x[4 + v] = der * s;
            }
        }
        const int at = fwh_place(t, nt);
#pragma unroll
        for (int w = 0; w < 4; ++w) xp[fwh_slot(at, w)] = make_double2(x[2 * w], x[2 * w + 1]);
#pragma unroll
        for (int v = 0; v < 8; ++v) top[v] = max(top[v], __double2hiint(x[v]) & 0x7fffffff);
    }
#pragma unroll
    for (int v = 0; v < 8; ++v) {
        const int m = __reduce_max_sync(0xffffffffu, top[v]);
        if (lane == 0) atomicMax(hw + (pb + lp) * 8 + v, m);
    }
}

// Fixed-point form of a number: N = x 2^(60 - e) for |x| < 2^e, as two limbs
// N = h 2^30 + l with -2^29 <= l < 2^29.  e follows from the largest high word H
// of the series.  A series of zeros has H = 0; a record with an infinity, a NaN or
// a series of magnitudes beyond 2^500 either way is summed in double.
__device__ __forceinline__ bool fwh_wide(int hi) {
    const int ex = (hi >> 20) & 0x7ff;
    return (hi & 0x7fffffff) != 0 && (ex < 523 || ex > 1523);
}
// mantissa of |x| as an integer < 2^53 (x normal or 0), shifted left by s and
// right by d with rounding
__device__ __forceinline__ long long fwh_fix(double x, int s, int d) {
    const unsigned long long u = static_cast<unsigned long long>(__double_as_longlong(x));
    const int ex = int(u >> 52) & 0x7ff;
    if (ex == 0 || d > 62) return 0;
    long long m = static_cast<long long>((u & 0xfffffffffffffull) | 0x10000000000000ull) << s;
    if (d > 0) m = (m + (1ll << (d - 1))) >> d;
    return (u >> 63) ? -m : m;
}
__device__ __forceinline__ int2 fwh_limbs(long long N) {
    const int h = int((N + (1ll << 29)) >> 30);
    return make_int2(h, int(N - (static_cast<long long>(h) << 30)));
}

// the series of a batch to fixed point, in place (16 bytes, two series, a thread);
// *wide is set if one has no fixed-point form
__global__ void k_fwh_fix(double* __restrict__ X, const int* __restrict__ hw, int nt, int np, int* __restrict__ wide) {
    const int64_t n = int64_t(np) * 4 * nt;
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
        const int64_t p = i / (4 * int64_t(nt));
        const unsigned at = unsigned(i - p * 4 * nt);
        const int* H = hw + p * 8;
        const int v = 2 * ((at ^ (at >> 3)) & 3);   // the series of this slot (fwh_slot)
        if (fwh_wide(H[v]) || fwh_wide(H[v + 1])) {
            *wide = 1;
            continue;
        }
        const double2 x = reinterpret_cast<const double2*>(X)[i];
        auto conv = [](double x, int H) {
            const int ex = (__double2hiint(x) >> 20) & 0x7ff;
            return fwh_limbs(fwh_fix(x, 7, (H >> 20) - ex));
        };
        const int2 a = conv(x.x, H[v]), b = conv(x.y, H[v + 1]);
        reinterpret_cast<int4*>(X)[i] = make_int4(a.x, a.y, b.x, b.y);
    }
}

// Geometry of one (panel, copy): integrand coefficients and delay.
__device__ void panel_coefs(const double* y, double dS, const double* obs, const FwhConst& k, double* cf,
                            double* delay) {
    double r[3];
    for (int i = 0; i < 3; ++i) r[i] = obs[i] - y[i];
    double Mr = 0, rr = 0;
    for (int i = 0; i < 3; ++i) {
        Mr += k.M[i] * r[i];
        rr += r[i] * r[i];
    }
    const double b2 = k.b2;
    const double Rs = sqrt(rr + b2 * Mr * Mr) / sqrt(b2);          // Eq. B.8
    const double R = b2 * (Rs - Mr);                               // Eq. B.9
    double Rts[3], Rt[3];
    double MRs = 0, MR = 0;
    for (int i = 0; i < 3; ++i) {
        Rts[i] = (r[i] + b2 * Mr * k.M[i]) / (b2 * Rs);            // Eq. B.11
        Rt[i] = b2 * (Rts[i] - k.M[i]);                            // Eq. B.12
        MRs += k.M[i] * Rts[i];
        MR += k.M[i] * Rt[i];
    }
    // I = a dQ + b Q + sum_i (d_i dL_i + e_i L_i)   (Eqs. B.2-B.7, times dS)
    cf[4] = (1.0 - MR) * dS / Rs;
    cf[0] = -k.c0 * MRs * dS / (Rs * Rs);
    for (int i = 0; i < 3; ++i) {
        cf[5 + i] = Rt[i] * dS / (k.c0 * Rs);
        cf[1 + i] = Rts[i] * dS / (Rs * Rs);
    }
    *delay = R / k.c0;
}

// One observer of a launch: position, first time and length of its window, and its
// row of the output.
struct FwhObs {
    double x[3], tstart;
    int T, row;
};

// the delay R / c0 of a panel copy at y (Eqs. B.8, B.9)
__device__ __forceinline__ double panel_delay(const double* y, const double* obs, const FwhConst& k) {
    double Mr = 0, rr = 0;
    for (int i = 0; i < 3; ++i) {
        const double r = obs[i] - y[i];
        Mr += k.M[i] * r;
        rr += r * r;
    }
    const double Rs = sqrt(rr + k.b2 * Mr * Mr) / sqrt(k.b2);
    return k.b2 * (Rs - Mr) / k.c0;
}

// ext[2 o], ext[2 o + 1]: largest delay of observer o and the complement of the
// smallest, as bits of non-negative doubles (0 at the start).  One thread a panel
// copy; the host loop this takes the place of took 8 ms for 2.0 million of them.
__global__ void k_fwh_delays(const double* __restrict__ y, int npts, FwhConst k, const FwhObs* __restrict__ obs,
                             int ncopies, double Lspan, unsigned long long* __restrict__ ext) {
    const int o = blockIdx.y, K = (ncopies - 1) / 2;
    const double ob[3] = {obs[o].x[0], obs[o].x[1], obs[o].x[2]};
    unsigned long long hi = 0, lo = 0;
    for (int64_t w = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; w < int64_t(npts) * ncopies;
         w += int64_t(gridDim.x) * blockDim.x) {
        const int64_t p = w / ncopies;
        const double yy[3] = {y[p * 3 + 0], y[p * 3 + 1], y[p * 3 + 2] + (int(w - p * ncopies) - K) * Lspan};
        const double d = panel_delay(yy, ob, k);
        if (!(d >= 0.0)) continue;   // NaN: left out, as by a comparison
        const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(d + 0.0));
        hi = max(hi, b);
        lo = max(lo, ~b);
    }
    for (int s = 16; s > 0; s >>= 1) {
        hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, s));
        lo = max(lo, __shfl_xor_sync(0xffffffffu, lo, s));
    }
    if ((threadIdx.x & 31) == 0) {
        atomicMax(ext + 2 * o, hi);
        atomicMax(ext + 2 * o + 1, lo);
    }
}

__device__ __forceinline__ void cubic_weights(double x, double (&wt)[4]) {
    wt[0] = -(x - 1.0) * (x - 2.0) * (x - 3.0) / 6.0;
    wt[1] = x * (x - 2.0) * (x - 3.0) / 2.0;
    wt[2] = -x * (x - 1.0) * (x - 3.0) / 2.0;
    wt[3] = x * (x - 1.0) * (x - 2.0) / 6.0;
}
// start j of the stencil of source index s = i + off, clamped to the record (its
// position in the stencil is (i - j) + off: s itself rounds off's last bits away)
__device__ __forceinline__ int fwh_stencil(double s, int nt) {
    return int(fmin(fmax(floor(s) - 1.0, 0.0), double(nt - 4)));
}

// Coefficients and source index of sample 0 of panel copy (p, cc)
__device__ void fwh_panel(const double* y, const double* dS, int p, int cc, double Lspan, const FwhObs& ob,
                          const FwhConst& k, double* cf, double* off) {
    const double yy[3] = {y[p * 3 + 0], y[p * 3 + 1], y[p * 3 + 2] + cc * Lspan};
    double delay;
    panel_coefs(yy, dS[p], ob.x, k, cf, &delay);
    *off = (ob.tstart - k.tau0 - delay) / k.dtau;
}
// Sum over panel copies of the interpolated integrand (Eqs. B.2, B.13, B.14), in
// fixed point on the integer pipe: this GPU multiplies 32-bit integers 32 times
// as fast as it does FP64, and 18 FP64 operations a panel copy and sample bound
// the sum in double (18,840 panels, 36 observers, 3 copies, 690 samples: 72 ms in
// double at 0.6 of the FP64 rate, 14 ms here).
//   I = sum_v cf_v x_v(j) with |x_v| <= m_v < 2^e_v over the record and
//   sum_v |cf_v| m_v < 2^E: x_v, cf_v 2^e_v / 2^E and I have 60 bits below 2^e_v, 1
//   and 2^E, products of limbs h h' + ((h l' + l h') >> 30) drop only l l', 2^-62 of
//   the bound; then p += sum_m w_m I(j + m) with the cubic weights scaled by
//   2^(E - top - r) (top the largest E of the block's copies, 2^(r + 3) twice their
//   number), kept as the two sums hh and mid of 64 bits, with which a sum over a
//   block is exact; it becomes a double once, at the block's end.
// One exponent holds for the whole record and for all copies of a block, so what is
// lost is relative to the largest of them: at 32 copies about 2^-55 of 2^top (2-norm
// of dropped l l' and rounded weights), where double loses about 2^-51 of the largest
// |I| at that sample.  A sample at which no copy's integrand reaches 2^-12 of 2^top (a
// transient's rise or decay, the quiet part of a record with one large outlier) is not
// left to fixed point: what it loses is then above 1e-13 of the largest |I|, the size of
// the sources' own errors.  The kernel takes the largest |I| of each sample's stencils,
// over those points that count (weight at least 1/32), over some of the block's copies,
// and marks the observer where that is too small (fwh_loud); a marked observer is summed
// again in double (k_fwh_accum64).  At 2^-10 the common zero of a block's 32 copies marked
// an observer in 2 of 12 records of sinusoids (18,840 panels, 36 observers: 18.8 ms for
// 16.0), at 2^-12 in none.
// Error against a reference in another order of summation, 2-norm: 1.3e-13 to 1.5e-12
// here, 1.5e-13 to 1.8e-12 in double (it comes from the sources).
// A block: one group of panels and one observer; a warp takes 124 samples of one of
// ns slices of its copies (a few observers leave too few warps otherwise; the integer
// sums of the slices add up exactly, whatever ns), a lane 4 consecutive ones (31
// lanes; lane 31 only supplies the integrands that lane 30's stencils need).  Each
// integrand is formed once and passed to the lane
// before it by shuffles: 24 + 12 products of limb pairs, 4 loads of 16 bytes and
// 1.5 shuffles a sample.  Issue and latency bound it: at 18,840 panels, 36 observers and
// 3 copies the products need 5.1 of 13.8 ms (at 32 wide multiply-adds a clock and SM),
// the rest goes to limbs, loads and shuffles at 24 warps an SM.  With 8 samples a lane
// and 128 registers 1.80 ms against 1.51 ms at 2,198 panels.
constexpr int ACC_PC = 96;        // panel copies set up at a time
constexpr int ACC_LANES = 31;     // lanes with samples of their own
constexpr int ACC_WARPS = 8;      // warps (sample chunks) of a block at most
constexpr int ACC_S = KO * ACC_LANES;

constexpr int SILENT = -100000;    // exponent of a copy without a contribution (no branch: that cost 1.5%)
constexpr int ACC_QUIET = 19;      // bits of a top limb of 2^-12 of the bound (2^18)

struct __align__(16) FwhPc {   // read in 16-byte pieces
    int c[2 * NSER];   // coefficient limbs (h, l)
    int w[8];          // weight limbs
    int count[4];      // -1: this point of the stencil counts for how loud a sample is, 0: not
    int at[KO];        // place of t = jb + m, m < KO
    double off;        // source index of sample 0
    int E, sc;         // exponent E (SILENT: all coefficients and weights are 0); weights are scaled by 2^sc
    int jb;
};
static_assert(sizeof(FwhPc) % 16 == 0 && offsetof(FwhPc, w) % 16 == 0 && offsetof(FwhPc, count) % 16 == 0, "");

// top limb of one integrand (by the top limbs of its factors alone)
__device__ __forceinline__ int fwh_top(const int* c, const int4* xp, unsigned at) {
    long long a = 0;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        const int4 q = xp[fwh_slot(at, v)];
        a += static_cast<long long>(c[4 * v]) * q.x;
        a += static_cast<long long>(c[4 * v + 2]) * q.z;
    }
    return abs(int(a >> 30));
}
// one integrand, N = I 2^60 / 2^E, of a panel's series at place `at`
__device__ __forceinline__ long long fwh_integrand(const int (&c)[2 * NSER], const int4* xp, unsigned at) {
    long long a = 0, b = 0;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        const int4 q = xp[fwh_slot(at, v)];
        a += static_cast<long long>(c[4 * v]) * q.x;
        b += static_cast<long long>(c[4 * v]) * q.y;
        b += static_cast<long long>(c[4 * v + 1]) * q.x;
        a += static_cast<long long>(c[4 * v + 2]) * q.z;
        b += static_cast<long long>(c[4 * v + 2]) * q.w;
        b += static_cast<long long>(c[4 * v + 3]) * q.z;
    }
    return a + (b >> 30);
}
// sample i of a panel copy whose stencil runs over an end of the record: the
// stencil is clamped to the record and its weights are the sample's own
__device__ __noinline__ void fwh_end(const FwhPc* rc, const int4* xp, int nt, int i, long long* hh, long long* mid) {
    int c[2 * NSER];
#pragma unroll
    for (int v = 0; v < 2 * NSER; v += 4) *reinterpret_cast<int4*>(c + v) = *reinterpret_cast<const int4*>(rc->c + v);
    const int j = fwh_stencil(double(i) + rc->off, nt);
    double wt[4];
    cubic_weights(double(i - j) + rc->off, wt);
    long long a = 0, b = 0;
    for (int m = 0; m < 4; ++m) {
        const int2 q = fwh_limbs(fwh_integrand(c, xp, fwh_place(j + m, nt)));
        const int2 w = fwh_limbs(__double2ll_rn(scalbn(wt[m], rc->sc)));
        a += static_cast<long long>(w.x) * q.x;
        b += static_cast<long long>(w.x) * q.y;
        b += static_cast<long long>(w.y) * q.x;
    }
    *hh = a + (b >> 30);
    *mid = b & ((1ll << 30) - 1);
}

// How loud a lane's samples are: for each the bits of the largest top limb, in units
// of 2^top, over the points of its stencils that count (4 x 8 bits; or-ed, so that one
// bit too many is possible), over those of the copies w0..w1 - 1 of rec that are
// multiples of step.  A loop of its own: inside k_fwh_accum's it took registers, and 1.1
// ms of 14.2 (18,840 panels, 36 observers, 3 copies) instead of 0.3.
__device__ __noinline__ unsigned fwh_loud(const FwhPc* rec, int w0, int w1, int step, int top, const int4* X, int first,
                                          int c0, int ncopies, int nt, int unit, int samples) {
    int loud[KO] = {};
    for (int w = (w0 + step - 1) / step * step; w < w1; w += step) {
        const FwhPc& rc = rec[w];
        const int4* xp = X + int64_t(first + (c0 + w) / ncopies) * 4 * nt;
        const int down = min(31, top - rc.E), t0 = KO * unit + rc.jb;
        int ih[KO + 3];
#pragma unroll
        for (int m = 0; m < KO; ++m) ih[m] = fwh_top(rc.c, xp, min(unsigned(rc.at[m] + unit), unsigned(nt - 1)));
#pragma unroll
        for (int m = 0; m < 3; ++m) ih[KO + m] = __shfl_down_sync(0xffffffffu, ih[m], 1);
#pragma unroll
        for (int q = 0; q < KO; ++q) {
            if (t0 + q >= 0 && t0 + q + 3 < nt) {
                loud[q] |= ((ih[q] & rc.count[0]) | (ih[q + 1] & rc.count[1]) | (ih[q + 2] & rc.count[2]) |
                            (ih[q + 3] & rc.count[3])) >> down;
            } else if (q < samples) {   // over an end of the record: the sample's own stencil
                const int i = KO * unit + q, j = fwh_stencil(double(i) + rc.off, nt);
                double wt[4];
                cubic_weights(double(i - j) + rc.off, wt);
                for (int m = 0; m < 4; ++m)
                    if (fabs(wt[m]) >= 0.03125) loud[q] |= fwh_top(rc.c, xp, fwh_place(j + m, nt)) >> down;
            }
        }
    }
    unsigned bits = 0;
#pragma unroll
    for (int q = 0; q < KO; ++q) bits |= unsigned(32 - __clz(loud[q])) << (8 * q);
    return bits;
}

template <bool SLICED>   // false: ns = 1
__global__ void __launch_bounds__(32 * ACC_WARPS, 3)
    k_fwh_accum(const int4* __restrict__ X, const int* __restrict__ hwb, int nt, int p0, int np, int nrows,
                const double* __restrict__ y, const double* __restrict__ dS, const __grid_constant__ FwhConst k,
                const FwhObs* __restrict__ obs, int Tmax, int ncopies, double Lspan, int group,
                double* __restrict__ partial, int ns, volatile int* flag, volatile int* wide) {
    __shared__ __align__(16) FwhPc rec[ACC_PC];
    __shared__ long long s_sum[SLICED ? 2 * KO : 1][32 * ACC_WARPS];
    __shared__ unsigned s_bits[32 * ACC_WARPS];
    __shared__ int s_top, s_double;
    const int o = blockIdx.x, row = blockIdx.y;
    const int lane = threadIdx.x & 31;
    const int T = obs[o].T;
    const int bw = int(blockDim.x >> 5) / (SLICED ? ns : 1), slice = SLICED ? int(threadIdx.x >> 5) / bw : 0;
    const int unit = lane + ACC_LANES * (int(blockIdx.z) * bw + int(threadIdx.x >> 5) - slice * bw);
    const int i0 = KO * unit;
    const bool mine = lane < ACC_LANES && i0 < T;              // samples i0.. are this lane's
    const bool idle = __shfl_sync(0xffffffffu, i0, 0) >= T;    // no lane of this warp does
    const int gp0 = row * group, gnp = min(group, np - gp0);   // panels of this block, within the batch
    const int npc = gnp * ncopies, K = (ncopies - 1) / 2;
    double* out = partial + (int64_t(o) * nrows + row) * Tmax;   // adds up over the batches of panels
    const int room = max(0, 30 - __clz(min(npc, ACC_PC)));     // r
    if (threadIdx.x == 0) s_double = *wide | flag[o];
    __syncthreads();
    if (s_double) return;   // this observer is summed in double anyway
    for (int c0 = 0; c0 < npc; c0 += ACC_PC) {
        const int n = min(ACC_PC, npc - c0);
        __syncthreads();
        if (threadIdx.x == 0) s_top = INT_MIN;
        __syncthreads();
        // coefficients and weights of this chunk's panel copies
        for (int w = threadIdx.x; w < n; w += blockDim.x) {
            FwhPc& rc = rec[w];
            const int pl = gp0 + (c0 + w) / ncopies, cc = (c0 + w) % ncopies - K;
            const int* hw = hwb + pl * 8;
            double cf[NSER], off, S = 0.0;
            fwh_panel(y, dS, p0 + pl, cc, Lspan, obs[o], k, cf, &off);
            bool fixed = fabs(off) < 1e9;
#pragma unroll
            for (int v = 0; v < NSER; ++v) {
                fixed = fixed && !fwh_wide(__double2hiint(cf[v]));
                if (hw[v]) S += fabs(cf[v]) * __hiloint2double(hw[v], -1);
            }
            if (!fixed) flag[o] = 1;
            fixed = fixed && S != 0.0;
            int E = SILENT;
            const int jb = fixed ? int(floor(off)) - 1 : 0;
#pragma unroll
            for (int m = 0; m < KO; ++m) rc.at[m] = fwh_place(jb + m, nt);
            rc.jb = jb;
#pragma unroll
            for (int v = 0; v < 2 * NSER; ++v) rc.c[v] = 0;
            if (fixed) {
                E = ((__double2hiint(S * (1.0 + 1e-15)) >> 20) & 0x7ff) - 1022;   // S < 2^E
#pragma unroll
                for (int v = 0; v < NSER; ++v) {
                    // cf 2^e / 2^E, below 2 since 2^e is at most twice the series' largest value
                    const int ex = (__double2hiint(cf[v]) >> 20) & 0x7ff;
                    const int2 q = hw[v] == 0 ? make_int2(0, 0) : fwh_limbs(fwh_fix(cf[v], 8, 2045 + E - ex - (hw[v] >> 20)));
                    rc.c[2 * v] = q.x;
                    rc.c[2 * v + 1] = q.y;
                }
                atomicMax(&s_top, E);
            }
            rc.E = E;
            rc.off = off;
        }
        __syncthreads();
        const int top = s_top;
        for (int w = threadIdx.x; w < n; w += blockDim.x) {
            FwhPc& rc = rec[w];
            const int sc = rc.E == SILENT ? -200 : max(-200, 60 - room + rc.E - top);
            rc.sc = sc;
            double wt[4];
            cubic_weights(rc.off - floor(rc.off) + 1.0, wt);   // position in the stencil, [1, 2)
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const int2 q = fwh_limbs(__double2ll_rn(scalbn(wt[m], sc)));
                rc.w[2 * m] = q.x;
                rc.w[2 * m + 1] = q.y;
                rc.count[m] = fabs(wt[m]) >= 0.03125 ? -1 : 0;
            }
        }
        __syncthreads();
        if (!SLICED && idle) continue;
        long long hh[KO], mid[KO];
#pragma unroll
        for (int q = 0; q < KO; ++q) hh[q] = mid[q] = 0;
        const int w0 = SLICED ? n * slice / ns : 0, w1 = !SLICED ? n : idle ? w0 : n * (slice + 1) / ns;
        bool carry = (w1 - w0) & 1;   // the last copy's sums are carried over
        int pl = gp0 + (c0 + w0) / ncopies, copy = (c0 + w0) % ncopies;   // of w (uniform: one base address for all lanes)
        for (int w = w0; w < w1; ++w) {
            const FwhPc& rc = rec[w];
            const int4* xp = X + int64_t(pl) * 4 * nt;
            if (++copy == ncopies) {
                copy = 0;
                ++pl;
            }
            int ih[KO + 3], il[KO + 3];
            {
                int c[2 * NSER];
#pragma unroll
                for (int v = 0; v < 2 * NSER; v += 4)
                    *reinterpret_cast<int4*>(c + v) = *reinterpret_cast<const int4*>(rc.c + v);
#pragma unroll
                for (int m = 0; m < KO; ++m) {
                    // a place outside the record (a lane without samples there) reads the last one
                    const unsigned at = min(unsigned(rc.at[m] + unit), unsigned(nt - 1));
                    const int2 q = fwh_limbs(fwh_integrand(c, xp, at));
                    ih[m] = q.x;
                    il[m] = q.y;
                }
            }
#pragma unroll
            for (int m = 0; m < 3; ++m) {
                ih[KO + m] = __shfl_down_sync(0xffffffffu, ih[m], 1);
                il[KO + m] = __shfl_down_sync(0xffffffffu, il[m], 1);
            }
            const int t0 = i0 + rc.jb;
            int wt[8];
            *reinterpret_cast<int4*>(wt) = *reinterpret_cast<const int4*>(rc.w);
            *reinterpret_cast<int4*>(wt + 4) = *reinterpret_cast<const int4*>(rc.w + 4);
            auto add = [&](int q) {
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    hh[q] += static_cast<long long>(wt[2 * m]) * ih[q + m];
                    mid[q] += static_cast<long long>(wt[2 * m]) * il[q + m];
                    mid[q] += static_cast<long long>(wt[2 * m + 1]) * ih[q + m];
                }
            };
            if (__all_sync(0xffffffffu, !mine || (t0 >= 0 && t0 + min(KO, T - i0) + 2 < nt))) {
                // lanes without samples, and samples past T, add what is never stored
#pragma unroll
                for (int q = 0; q < KO; ++q) add(q);
            } else if (mine) {
#pragma unroll
                for (int q = 0; q < KO; ++q)
                    if (t0 + q >= 0 && t0 + q + 3 < nt) {
                        add(q);
                    } else if (i0 + q < T) {
                        long long a, b;
                        fwh_end(&rc, xp, nt, i0 + q, &a, &b);
                        hh[q] += a;
                        mid[q] += b;
                    }
            }
            // a copy adds at most 2^61 to mid: carry it over every second time
            carry = !carry;
            if (!carry)
#pragma unroll
                for (int q = 0; q < KO; ++q) {
                    hh[q] += mid[q] >> 30;
                    mid[q] &= (1ll << 30) - 1;
                }
        }
        // every 32nd copy looked at (fewer copies: every eighth, or all)
        unsigned bits = top == INT_MIN ? 0xffffffffu
                                       : fwh_loud(rec, w0, w1, n >= 64 ? 32 : n >= 16 ? 8 : 1, top, X, gp0, c0, ncopies, nt,
                                                  unit, mine ? T - i0 : 0);
        if constexpr (SLICED) {
#pragma unroll
            for (int q = 0; q < KO; ++q) {
                s_sum[q][threadIdx.x] = hh[q];
                s_sum[KO + q][threadIdx.x] = mid[q];
            }
            s_bits[threadIdx.x] = bits;
            __syncthreads();
            if (slice > 0) continue;
            for (int t = threadIdx.x + 32 * bw; t < blockDim.x; t += 32 * bw) {
#pragma unroll
                for (int q = 0; q < KO; ++q) {
                    hh[q] += s_sum[q][t];
                    mid[q] += s_sum[KO + q][t];
                }
                bits = __vmaxu4(bits, s_bits[t]);
            }
#pragma unroll
            for (int q = 0; q < KO; ++q) {
                hh[q] += mid[q] >> 30;
                mid[q] &= (1ll << 30) - 1;
            }
        }
        if (mine && slice == 0)
#pragma unroll
            for (int q = 0; q < KO; ++q)
                if (i0 + q < T) {
                    if (int((bits >> (8 * q)) & 255) < ACC_QUIET) flag[o] = 1;
                    const double v = top == INT_MIN ? 0.0
                                                    : scalbn(double(hh[q]) + double(mid[q]) * (1.0 / 1073741824.0),
                                                             top + room - 60);
                    out[i0 + q] = p0 + c0 == 0 ? v : out[i0 + q] + v;
                }
    }
}

// The sums in double, with the lanes and shared integrands of k_fwh_accum: 12 FP64
// operations a panel copy and sample (18 where a thread formed 7 integrands for 4
// samples of its own), bound by the FP64 pipe.  Always in D_NS slices of a block's
// copies, added in order.
constexpr int D_NS = 4;
struct __align__(16) FwhPc64 {
    double c[NSER], w[4], off;
    int at[KO];
    int jb, pad;
};
// sample i of a panel copy whose stencil runs over an end of the record
__device__ __noinline__ double fwh_end64(const FwhPc64* rc, const double2* xp, int nt, int i) {
    const int j = fwh_stencil(double(i) + rc->off, nt);
    double wt[4], sum = 0.0;
    cubic_weights(double(i - j) + rc->off, wt);
    for (int m = 0; m < 4; ++m) {
        double I = 0.0;
        for (int v = 0; v < 4; ++v) {
            const double2 q = xp[fwh_slot(fwh_place(j + m, nt), v)];
            I += rc->c[2 * v] * q.x;
            I += rc->c[2 * v + 1] * q.y;
        }
        sum += wt[m] * I;
    }
    return sum;
}
__global__ void __launch_bounds__(32 * ACC_WARPS, 3)
    k_fwh_accum64(const double2* __restrict__ X, int nt, int p0, int np, int nrows, const double* __restrict__ y,
                  const double* __restrict__ dS, const __grid_constant__ FwhConst k, const FwhObs* __restrict__ obs,
                  int Tmax, int ncopies, double Lspan, int group, double* __restrict__ partial, int z0) {
    __shared__ __align__(16) FwhPc64 rec[ACC_PC];
    __shared__ double s_sum[KO][32 * ACC_WARPS];
    const int o = blockIdx.x, row = blockIdx.y;
    const int lane = threadIdx.x & 31;
    const int T = obs[o].T;
    const int bw = int(blockDim.x >> 5) / D_NS, slice = int(threadIdx.x >> 5) / bw;
    const int unit = lane + ACC_LANES * ((z0 + int(blockIdx.z)) * bw + int(threadIdx.x >> 5) - slice * bw);
    const int i0 = KO * unit;
    const bool mine = lane < ACC_LANES && i0 < T;
    const bool idle = __shfl_sync(0xffffffffu, i0, 0) >= T;
    const int gp0 = row * group, npc = min(group, np - gp0) * ncopies, K = (ncopies - 1) / 2;
    double* out = partial + (int64_t(o) * nrows + row) * Tmax;
    for (int c0 = 0; c0 < npc; c0 += ACC_PC) {
        const int n = min(ACC_PC, npc - c0);
        __syncthreads();
        for (int w = threadIdx.x; w < n; w += blockDim.x) {
            FwhPc64& rc = rec[w];
            const int pl = gp0 + (c0 + w) / ncopies, cc = (c0 + w) % ncopies - K;
            fwh_panel(y, dS, p0 + pl, cc, Lspan, obs[o], k, rc.c, &rc.off);
            cubic_weights(rc.off - floor(rc.off) + 1.0, rc.w);   // position in the stencil, [1, 2)
            // (no such offset: every sample takes its own stencil)
            const int jb = fabs(rc.off) < 1e9 ? int(floor(rc.off)) - 1 : INT_MIN / 2;
#pragma unroll
            for (int m = 0; m < KO; ++m) rc.at[m] = fwh_place(jb + m, nt);
            rc.jb = jb;
        }
        __syncthreads();
        double acc[KO] = {};
        const int w1 = idle ? 0 : n * (slice + 1) / D_NS;
        for (int w = n * slice / D_NS; w < w1; ++w) {
            const FwhPc64& rc = rec[w];
            const double2* xp = X + int64_t(gp0 + (c0 + w) / ncopies) * 4 * nt;
            double I[KO + 3];
#pragma unroll
            for (int m = 0; m < KO; ++m) {
                // a place outside the record (a lane without samples there) reads the last one
                const unsigned at = min(unsigned(rc.at[m] + unit), unsigned(nt - 1));
                I[m] = 0.0;
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    const double2 q = xp[fwh_slot(at, v)];
                    I[m] += rc.c[2 * v] * q.x;
                    I[m] += rc.c[2 * v + 1] * q.y;
                }
            }
#pragma unroll
            for (int m = 0; m < 3; ++m) I[KO + m] = __shfl_down_sync(0xffffffffu, I[m], 1);
            const int t0 = i0 + rc.jb;
#pragma unroll
            for (int q = 0; q < KO; ++q) {
                if (!mine || i0 + q >= T) continue;
                double sum = 0.0;
                if (t0 + q >= 0 && t0 + q + 3 < nt) {
#pragma unroll
                    for (int m = 0; m < 4; ++m) sum += rc.w[m] * I[q + m];
                } else {
                    sum = fwh_end64(&rc, xp, nt, i0 + q);
                }
                acc[q] += sum;
            }
        }
#pragma unroll
        for (int q = 0; q < KO; ++q) s_sum[q][threadIdx.x] = acc[q];
        __syncthreads();
        if (mine && slice == 0)
#pragma unroll
            for (int q = 0; q < KO; ++q)
                if (i0 + q < T) {
                    for (int t = threadIdx.x + 32 * bw; t < blockDim.x; t += 32 * bw) acc[q] += s_sum[q][t];
                    out[i0 + q] = p0 + c0 == 0 ? acc[q] : out[i0 + q] + acc[q];
                }
    }
}

// p'(t_i) = (1/4 pi) sum over panel groups of the partial sums: 32 samples x
// 32 group slices per block, each slice summing groups g = slice (mod 32) in
// order, then a fixed-order tree over the slices (the same order every call).
// Observers marked in `flag` (null: none) are left out.
__global__ void k_fwh_reduce(const double* __restrict__ partial, int ngroups, int Tmax,
                             const FwhObs* __restrict__ obs, double* __restrict__ p_out, int cap,
                             const int* __restrict__ flag, const int* __restrict__ wide) {
    __shared__ double red[32][33];
    const int i = blockIdx.x * 32 + threadIdx.x, o = blockIdx.y, T = obs[o].T;
    const double* row = partial + int64_t(o) * ngroups * Tmax;
    if (flag && (flag[o] | *wide)) return;
    double* out = p_out + int64_t(obs[o].row) * cap;
    double s = 0.0;
    if (i < T)
        for (int g = threadIdx.y; g < ngroups; g += 32) s += row[int64_t(g) * Tmax + i];
    red[threadIdx.y][threadIdx.x] = s;
    __syncthreads();
    for (int st = 16; st > 0; st >>= 1) {
        if (threadIdx.y < st) red[threadIdx.y][threadIdx.x] += red[threadIdx.y + st][threadIdx.x];
        __syncthreads();
    }
    if (threadIdx.y == 0 && i < T) out[i] = red[0][threadIdx.x] / (4.0 * M_PI);
}

}  // namespace

// records the message returned by fr_last_error (defined with the context code)
int fr_set_error_from_fwh(int code, const char* msg);

namespace {

// Host-side plan of one FW-H integration: the constants of Eqs. B.8-B.12,
// every observer's unified window (Eq. B.13 and the text after it: from the
// latest first arrival to the earliest last arrival over all panel copies),
// and the panel grouping of the accumulation kernel.
struct FwhPlan {
    FwhConst k;
    std::vector<FwhObs> obs;   // position, first unified time and samples per observer
    int group = 1, ngroups = 1, Tmax = 0;
};

// Device scratch of one integration: the source series of a batch of panels X
// [nbatch][4][nt][2] doubles, their largest high words hw [nbatch][8], partial
// sums [observers of a launch][groups][Tmax] (npartial doubles), and the
// observer table of a launch (up to OBS_MAX observers) with its delay bounds, whose
// place the marks of the observers to be summed in double take afterwards (the last
// one of them: all).
constexpr int OBS_MAX = 2048;
struct FwhScratch {
    double* X = nullptr;
    int* hw = nullptr;
    int nbatch = 0;
    double* partial = nullptr;
    size_t npartial = 0;
    FwhObs* obs = nullptr;
    unsigned long long* ext = nullptr;
    int* flag() const { return reinterpret_cast<int*>(ext); }   // [OBS_MAX + 1], after the plan is made
};
constexpr size_t OBS_BYTES = OBS_MAX * (sizeof(FwhObs) + 2 * sizeof(unsigned long long));

int fwh_plan(int nt, int npts, const double* y, double dtau, double tau0, const double* obs, int nobs,
             const double Minf[3], double c0, double rho0, double p0, double Lspan, int ncopies, int cap,
             cudaStream_t s, const FwhScratch& sc, FwhPlan& pl) {
    const double MM = Minf[0] * Minf[0] + Minf[1] * Minf[1] + Minf[2] * Minf[2];
    FwhConst& k = pl.k;
    for (int i = 0; i < 3; ++i) k.M[i] = Minf[i];
    k.c0 = c0;
    k.rho0 = rho0;
    k.p0 = p0;
    k.dtau = dtau;
    k.tau0 = tau0;
    k.b2 = 1.0 / (1.0 - MM);
    pl.obs.assign(nobs, FwhObs{});
    for (int o = 0; o < nobs; ++o) {
        for (int i = 0; i < 3; ++i) pl.obs[o].x[i] = obs[o * 3 + i];
        pl.obs[o].row = o;
    }
    // unified observer windows from the delay bounds
    std::vector<unsigned long long> ext(2 * size_t(std::min(nobs, OBS_MAX)));
    for (int o0 = 0; o0 < nobs; o0 += OBS_MAX) {
        const int no = std::min(OBS_MAX, nobs - o0);
        cudaError_t e = cudaMemcpyAsync(sc.obs, pl.obs.data() + o0, sizeof(FwhObs) * no, cudaMemcpyHostToDevice, s);
        if (e == cudaSuccess) e = cudaMemsetAsync(sc.ext, 0, 16 * size_t(no), s);
        if (e == cudaSuccess) {
            const int64_t pcs = int64_t(npts) * ncopies;
            k_fwh_delays<<<dim3(unsigned(std::min<int64_t>((pcs + 255) / 256, 1024)), no), 256, 0, s>>>(
                y, npts, k, sc.obs, ncopies, Lspan, sc.ext);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) e = cudaMemcpyAsync(ext.data(), sc.ext, 16 * size_t(no), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return fr_set_error_from_fwh(FR_ECUDA, "cannot read panel positions");
        for (int o = 0; o < no; ++o) {
            if (ext[2 * o + 1] == 0) return fr_set_error_from_fwh(FR_EWINDOW, "empty observer window");   // NaN panels
            double dmax, dmin;
            const unsigned long long lo = ~ext[2 * o + 1];
            std::memcpy(&dmax, &ext[2 * o], 8);
            std::memcpy(&dmin, &lo, 8);
            const double ts = tau0 + dmax;
            const double te = tau0 + (nt - 1) * dtau + dmin;
            if (!(te >= ts)) return fr_set_error_from_fwh(FR_EWINDOW, "empty observer window");
            const double len = std::floor((te - ts) / dtau + 1e-9) + 1.0;
            if (!(len <= double(cap)))
                return fr_set_error_from_fwh(FR_EWINDOW, "observer window longer than the output capacity");
            pl.obs[o0 + o].tstart = ts;
            pl.obs[o0 + o].T = int(len);
            pl.Tmax = std::max(pl.Tmax, int(len));
        }
    }
    pl.group = std::max(1, kFwhGroup / ncopies);
    pl.ngroups = (npts + pl.group - 1) / pl.group;
    return FR_OK;
}

// the argument checks of an integration (before any device work)
int fwh_check(const double* hist, int nt, int npts, const double* y, const double* n, const double* dS, double dtau,
              const double* obs, int nobs, const double* Minf, double c0, int ncopies, const double* p_out, int cap,
              const int* nt_out, const double* t0_out) {
    if (!hist || !y || !n || !dS || !obs || !Minf || !p_out || !nt_out || !t0_out)
        return fr_set_error_from_fwh(FR_EINVAL, "null argument");
    if (nt < 5 || npts < 1 || nobs < 1 || cap < 1 || ncopies < 1 || ncopies % 2 == 0 || !(dtau > 0.0) ||
        !(c0 > 0.0))
        return fr_set_error_from_fwh(FR_EINVAL, "bad sizes (nt >= 5, odd ncopies, dtau > 0, c0 > 0 required)");
    const double MM = Minf[0] * Minf[0] + Minf[1] * Minf[1] + Minf[2] * Minf[2];
    if (!(MM < 1.0)) return fr_set_error_from_fwh(FR_EINVAL, "|Minf| must be below 1");
    if (ncopies > 2003) return fr_set_error_from_fwh(FR_ECUDA, "too many span copies (at most 2003)");
    if ((cap + 512 - 1) / 512 > 65535)
        return fr_set_error_from_fwh(FR_EINVAL, "observer window too long for one launch");
    return FR_OK;
}

// Scratch that fwh_integrate_noalloc counts against its fixed array, in
// doubles: the source series of all panels and one row of partial sums per
// group of kFwhGroup panel copies.
size_t fwh_series_doubles(int npts, int nt) { return size_t(npts) * NSER * nt; }
size_t fwh_partial_doubles(const FwhPlan& pl) { return size_t(pl.ngroups) * pl.Tmax; }

// Panels of a block (a row of partial sums) and of a batch, and a batch's rows.  The
// order of summation, and the exponent that a block's copies share, follow from the
// panels, copies and record alone: an observer's p' has the same bits whichever other
// observers are in the call.  kFwhGroup copies a block (18,840 panels, 36 observers, 3
// copies: k_fwh_accum 13.6 ms, with 96 a block 13.8).  At one observer, 752 panels and
// 2,400 samples it takes 54 us in 8 slices, without slices 113; blocks of few panels,
// chosen by the number of observers, took 49.
struct FwhSplit {
    int group, batch, rows;
    FwhSplit(int npts, int ncopies, int nbatch) {
        group = std::max(1, kFwhGroup / ncopies);
        const int nb = std::min(npts, nbatch);
        if (nb == npts) {   // rows of even length
            const int n = (npts + group - 1) / group;
            group = (npts + n - 1) / n;
        }
        batch = nb == npts && npts <= 65535 * int64_t(group) ? npts : std::min(nb / group, 65535) * group;
        rows = (batch + group - 1) / group;
    }
};

// The kernels of one integration (all scratch is fully written before it is
// read), then a synchronisation of the stream.  Panels go in batches of
// sc.nbatch, whose series are formed once for all observers of a launch.
// Observers that the fixed point marks are summed again in double.
// Warps of a block: time chunks and slices of copies, as many slices as it takes to
// have 24 warps for every SM.
int fwh_run(const FwhPlan& pl, const double* hist, int nt, int npts, const double* y, const double* n,
            const double* dS, const double* obs, int nobs, double Lspan, int ncopies, double* p_out, int cap,
            int* nt_out, double* t0_out, const FwhScratch& sc, cudaStream_t s) {
    const FwhSplit sp(npts, ncopies, sc.nbatch);
    const int group = sp.group, batch = sp.batch, ngroups = sp.rows;
    const int obs_fit = int(std::min<size_t>(OBS_MAX, sc.npartial / (size_t(ngroups) * pl.Tmax)));
    int dev = 0, nsm = 1;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return fr_set_error_from_fwh(FR_ECUDA, "no device");
    const int warps = (pl.Tmax + ACC_S - 1) / ACC_S;
    int ns = 1;
    while (ns < ACC_WARPS && int64_t(ngroups) * std::min(nobs, obs_fit) * warps * ns < 24 * int64_t(nsm)) ns *= 2;
    // time chunks of a block (even) and blocks in time, in ns slices
    auto chunks = [warps](int ns) { return (warps + ACC_WARPS / ns - 1) / (ACC_WARPS / ns); };
    auto threads = [warps, chunks](int ns) { return 32 * ns * ((warps + chunks(ns) - 1) / chunks(ns)); };
    cudaError_t err = cudaFuncSetAttribute(k_fwh_series, cudaFuncAttributeMaxDynamicSharedMemorySize, int(SER_SMEM));
    int *flag = sc.flag(), *wide = flag + OBS_MAX;
    // the panels of a launch of `no` observers, in fixed point or in double
    auto sums = [&](const FwhObs* table, int no, bool fixed, bool series) {
        err = cudaMemcpyAsync(sc.obs, table, sizeof(FwhObs) * no, cudaMemcpyHostToDevice, s);
        if (err == cudaSuccess && fixed) err = cudaMemsetAsync(flag, 0, sizeof(int) * (OBS_MAX + 1), s);
        for (int p0 = 0; p0 < npts && err == cudaSuccess; p0 += batch) {
            const int np = std::min(batch, npts - p0);
            if (series || batch < npts) {
                err = cudaMemsetAsync(sc.hw, 0, sizeof(int) * 8 * size_t(np), s);
                if (err != cudaSuccess) return;
                k_fwh_series<<<dim3((np + SER_P - 1) / SER_P, (nt + SER_T - 1) / SER_T), 256, SER_SMEM, s>>>(
                    hist, nt, npts, p0, np, n, pl.k, sc.X, sc.hw);
                const int64_t places = int64_t(np) * 4 * nt;
                if (fixed)
                    k_fwh_fix<<<unsigned(std::min<int64_t>((places + 255) / 256, nsm * 32)), 256, 0, s>>>(
                        sc.X, sc.hw, nt, np, wide);
            }
            const unsigned rows = unsigned((np + group - 1) / group);
            if (fixed)
                (ns > 1 ? k_fwh_accum<true> : k_fwh_accum<false>)<<<dim3(no, rows, chunks(ns)), threads(ns), 0, s>>>(
                    reinterpret_cast<const int4*>(sc.X), sc.hw, nt, p0, np, ngroups, y, dS, pl.k, sc.obs, pl.Tmax, ncopies,
                    Lspan, group, sc.partial, ns, flag, wide);
            else   // (windows above 16 million samples have more chunks than a grid's z)
                for (int z0 = 0; z0 < chunks(D_NS); z0 += 65535)
                    k_fwh_accum64<<<dim3(no, rows, std::min(65535, chunks(D_NS) - z0)), threads(D_NS), 0, s>>>(
                        reinterpret_cast<const double2*>(sc.X), nt, p0, np, ngroups, y, dS, pl.k, sc.obs, pl.Tmax, ncopies,
                        Lspan, group, sc.partial, z0);
            err = cudaGetLastError();
        }
        if (err != cudaSuccess) return;
        k_fwh_reduce<<<dim3((pl.Tmax + 31) / 32, no), dim3(32, 32), 0, s>>>(
            sc.partial, ngroups, pl.Tmax, sc.obs, p_out, cap, fixed ? flag : nullptr, wide);
        err = cudaGetLastError();
    };
    std::vector<FwhObs> again;   // observers to be summed in double
    std::vector<int> mark(OBS_MAX + 1, 0);
    for (int o0 = 0; o0 < nobs && err == cudaSuccess; o0 += obs_fit) {
        const int no = std::min(obs_fit, nobs - o0);
        if (!mark[OBS_MAX]) {   // (a record without a fixed-point form: all that are left)
            sums(pl.obs.data() + o0, no, true, o0 == 0);
            if (err == cudaSuccess) err = cudaMemcpyAsync(mark.data(), flag, sizeof(int) * (OBS_MAX + 1), cudaMemcpyDeviceToHost, s);
            if (err == cudaSuccess) err = cudaStreamSynchronize(s);
        }
        for (int o = 0; o < no; ++o)
            if (mark[OBS_MAX] || mark[o]) again.push_back(pl.obs[o0 + o]);
    }
    for (size_t o0 = 0; o0 < again.size() && err == cudaSuccess; o0 += obs_fit)
        sums(again.data() + o0, int(std::min<size_t>(obs_fit, again.size() - o0)), false, o0 == 0);
    for (int o = 0; o < nobs; ++o) {
        nt_out[o] = pl.obs[o].T;
        t0_out[o] = pl.obs[o].tstart;
    }
    if (err == cudaSuccess) err = cudaStreamSynchronize(s);
    if (err != cudaSuccess) return fr_set_error_from_fwh(FR_ECUDA, cudaGetErrorString(err));
    return FR_OK;
}

}  // namespace

extern "C" int fwh_integrate(const double* hist, int nt, int npts, const double* y, const double* n,
                             const double* dS, double dtau, double tau0, const double* obs, int nobs,
                             const double Minf[3], double c0, double rho0, double p0, double Lspan,
                             int ncopies, double* p_out, int cap, int* nt_out, double* t0_out, void* stream) {
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int rc = fwh_check(hist, nt, npts, y, n, dS, dtau, obs, nobs, Minf, c0, ncopies, p_out, cap, nt_out, t0_out);
    if (rc != FR_OK) return rc;
    FwhScratch sc;
    // scratch from the pool, or (no pool) by cudaMalloc
    auto get = [s](void** p, size_t bytes, bool* pooled) {
        *pooled = fr_pool_alloc(p, bytes, s);
        return *pooled || cudaMalloc(p, bytes) == cudaSuccess;
    };
    auto put = [s](void* p, bool pooled) {
        if (pooled) fr_pool_free(p, s);
        else cudaFree(p);
    };
    void *tab = nullptr, *buf = nullptr;
    bool tab_pooled = false, buf_pooled = false;
    if (!get(&tab, OBS_BYTES, &tab_pooled))
        return fr_set_error_from_fwh(FR_ENOMEM, "cannot allocate FW-H scratch");
    sc.obs = static_cast<FwhObs*>(tab);
    sc.ext = reinterpret_cast<unsigned long long*>(sc.obs + OBS_MAX);
    FwhPlan pl;
    rc = fwh_plan(nt, npts, y, dtau, tau0, obs, nobs, Minf, c0, rho0, p0, Lspan, ncopies, cap, s, sc, pl);
    if (rc == FR_OK) {
        // up to 160 MiB of series at a time and 64 MiB of partial sums (never
        // less than the panels of one block and the rows of one observer)
        const size_t per = sizeof(double) * NSER * size_t(nt);
        sc.nbatch = int(std::min<size_t>(size_t(npts), std::max<size_t>(ACC_PC, (size_t(160) << 20) / per)));
        const size_t one = size_t(FwhSplit(npts, ncopies, sc.nbatch).rows) * pl.Tmax;
        sc.npartial = std::min(one * nobs, std::max(one, size_t(8) << 20));
        const size_t nx = fwh_series_doubles(sc.nbatch, nt);
        if (!get(&buf, sizeof(double) * (nx + sc.npartial) + 32 * size_t(sc.nbatch), &buf_pooled)) {
            put(tab, tab_pooled);
            return fr_set_error_from_fwh(FR_ENOMEM, "cannot allocate FW-H scratch");
        }
        sc.X = static_cast<double*>(buf);
        sc.hw = reinterpret_cast<int*>(sc.X + nx);
        sc.partial = sc.X + nx + 4 * size_t(sc.nbatch);
        rc = fwh_run(pl, hist, nt, npts, y, n, dS, obs, nobs, Lspan, ncopies, p_out, cap, nt_out, t0_out, sc, s);
        put(buf, buf_pooled);
    }
    put(tab, tab_pooled);
    return rc;
}

// ---------------------------------------------------------------------------
// fwh_integrate_noalloc: the same computation with its scratch (the source
// series and the partial sums) in a fixed file-scope device array, for callers
// that cannot call cudaMalloc/cudaFree.  On the host the arrays' names are only
// stand-ins, never device addresses: every call looks the addresses up on the
// current device with cudaGetSymbolAddress (which allocates nothing), so they
// always belong to the context the kernels run in.

namespace {

constexpr size_t kNoallocScratchDoubles = size_t(1) << 22;  // 32 MiB per device
__device__ __align__(256) double g_fwh_scratch[kNoallocScratchDoubles];
// the high words of the series' panels (at most 2^22 / (8 * 5) panels fit the
// scratch) and the observer table
constexpr size_t kNoallocPanels = kNoallocScratchDoubles / (NSER * 5) + 1;
__device__ __align__(256) int g_fwh_hw[kNoallocPanels * 8];
__device__ __align__(256) unsigned char g_fwh_tab[OBS_BYTES];

// Device addresses of the fixed arrays in the current device's context.
int noalloc_scratch(FwhScratch* sc) {
    void *p = nullptr, *h = nullptr, *t = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_fwh_scratch);
    if (e == cudaSuccess) e = cudaGetSymbolAddress(&h, g_fwh_hw);
    if (e == cudaSuccess) e = cudaGetSymbolAddress(&t, g_fwh_tab);
    if (e != cudaSuccess || !p || !h || !t)
        return fr_set_error_from_fwh(FR_ECUDA, (std::string("cudaGetSymbolAddress of the FW-H scratch: ") +
                                                cudaGetErrorString(e)).c_str());
    sc->X = static_cast<double*>(p);
    sc->hw = static_cast<int*>(h);
    sc->obs = static_cast<FwhObs*>(t);
    sc->ext = reinterpret_cast<unsigned long long*>(sc->obs + OBS_MAX);
    return FR_OK;
}

}  // namespace

extern "C" int fwh_integrate_noalloc(const double* hist, int nt, int npts, const double* y, const double* n,
                                     const double* dS, double dtau, double tau0, const double* obs, int nobs,
                                     const double Minf[3], double c0, double rho0, double p0, double Lspan,
                                     int ncopies, double* p_out, int cap, int* nt_out, double* t0_out,
                                     void* stream) {
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int rc = fwh_check(hist, nt, npts, y, n, dS, dtau, obs, nobs, Minf, c0, ncopies, p_out, cap, nt_out, t0_out);
    if (rc != FR_OK) return rc;
    FwhScratch sc;
    rc = noalloc_scratch(&sc);
    if (rc != FR_OK) return rc;
    FwhPlan pl;
    rc = fwh_plan(nt, npts, y, dtau, tau0, obs, nobs, Minf, c0, rho0, p0, Lspan, ncopies, cap, s, sc, pl);
    if (rc != FR_OK) return rc;
    // the series and the partial rows must fit the fixed scratch
    const size_t need = fwh_series_doubles(npts, nt) + fwh_partial_doubles(pl);
    if (need > kNoallocScratchDoubles)
        return fr_set_error_from_fwh(
            FR_EINVAL, ("fwh_integrate_noalloc: needs " + std::to_string(need) + " doubles of scratch, the fixed "
                        "maximum is " + std::to_string(kNoallocScratchDoubles) +
                        " (8*npts*nt + ceil(npts/max(1,32/ncopies))*window); use fwh_integrate").c_str());
    sc.nbatch = npts;
    sc.partial = sc.X + fwh_series_doubles(npts, nt);
    sc.npartial = kNoallocScratchDoubles - fwh_series_doubles(npts, nt);
    return fwh_run(pl, hist, nt, npts, y, n, dS, obs, nobs, Lspan, ncopies, p_out, cap, nt_out, t0_out, sc, s);
}
