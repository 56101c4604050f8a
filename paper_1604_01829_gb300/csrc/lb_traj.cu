// Trajectory analysis of rigid raspberries on the GPU (Ustach & Faller,
// arXiv:1604.01829, Sec. 2.4-2.7 and the SI sections "Body-frame
// translational displacement" and "Body-frame angular displacement").
//
// Input: per body, nrec recorded centres X_k and orientations q_k (unit
// quaternions, Hamilton convention, lab = R(q) body) at a fixed interval.
// Per body and lag l (in records) the kernels average over all time origins
//   0-2  (X_{t+l} - X_t)_a^2 per lab axis                      Eq. (dt_lab)
//   3-5  (X^b_{t+l} - X^b_t)_a^2 per body axis, with the body-frame trajectory
//        X^b_n = sum_{k<=n} R(q_{k-1})^T (X_k - X_{k-1})       Eqs. (labdisp),
//        (quat), (bodyframedisplacement), (bodyframetrajectory), (dt_body)
//   6    Theta^2, Theta the angle between p(t) and p(t+l), p = R(q) p_ref
//                                                                Eq. (delta_theta)
//   7-9  (Theta_a(t+l) - Theta_a(t))^2, Theta_a the summed body-frame angular
//        displacements about body axis a by the projection method of the SI
//                                     Eqs. (bodyframerotdisplacement),
//                                     (bodyframerottrajectory), (dr_body)
// Readings: the body-frame displacement over an interval uses the
// orientation at its start; the angle of the projected axis is taken with
// atan2, equal to the printed arctangent of the component ratio for
// rotations below 90 degrees per interval; the lab-frame angle is computed
// as atan2(|p x p'|, p . p'), the same angle as the printed arccosine of the
// dot product of the unit vectors without its loss of precision at small
// angles.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <type_traits>
#include <vector>

#include "../../include/lb.h"
#include "lb_fix64.cuh"
#include "lb_rigid.cuh"

namespace lbk {

namespace {

// Work per body, columns of nrec values each (SoA): p-hat (3), body-frame
// trajectory (3), body-frame angles (3).
constexpr int kW = 9;

__device__ __forceinline__ double dot3(const double *a, const double *b) {
    return a[0] * b[0] + a[1] * b[1] + a[2] * b[2];
}

__device__ __forceinline__ void axes_of(const double *q, double ax[3][3]) {
    double R[9];
    quat_to_R(q, R);
    for (int c = 0; c < 3; ++c)            // body axis c in the lab frame: column c of R
        for (int r = 0; r < 3; ++r) ax[c][r] = R[3 * r + c];
}

// one thread per (body, record): unit reference vector, increments of the
// body-frame trajectory and of the body-frame angles over [k-1, k]
__global__ void k_msd_prep(const double *X, const double *q, int nrec, int nb, const double *p_ref, double *work) {
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (t >= (long long)nrec * nb) return;
    const int b = (int)(t / nrec), k = (int)(t % nrec);
    const double *qk = q + ((long long)b * nrec + k) * 4;
    double ak[3][3];
    axes_of(qk, ak);
    double *w = work + (long long)b * nrec * kW + k;
    const double pn = sqrt(dot3(p_ref, p_ref));
    double p[3];
    for (int r = 0; r < 3; ++r) p[r] = (ak[0][r] * p_ref[0] + ak[1][r] * p_ref[1] + ak[2][r] * p_ref[2]) / pn;
    // a quaternion that is not a unit one to rounding: the length is taken out
    // (the squared chord of k_msd_angle scales with it), unless it has none in
    // FP64 (the vector is 0, or its square under- or overflows)
    const double off = fma(p[0], p[0], fma(p[1], p[1], fma(p[2], p[2], -1.0))), n2 = dot3(p, p);
    const double len = fabs(off) > 0x1p-50 && n2 > 0.0 && n2 < 0x1p1023 ? sqrt(n2) : 1.0;
    for (int r = 0; r < 3; ++r) w[(long long)r * nrec] = p[r] / len;
    if (k == 0) {
        for (int c = 3; c < kW; ++c) w[(long long)c * nrec] = 0.0;
        return;
    }
    double ap[3][3];
    axes_of(qk - 4, ap);
    const double *Xk = X + ((long long)b * nrec + k) * 3;
    const double d[3] = {Xk[0] - Xk[-3], Xk[1] - Xk[-2], Xk[2] - Xk[-1]};
    for (int c = 0; c < 3; ++c) w[(long long)(3 + c) * nrec] = dot3(ap[c], d);
    // i, j, k of step k against those of step k-1 (projection method)
    w[6LL * nrec] = atan2(dot3(ak[2], ap[1]), dot3(ak[2], ap[2]));
    w[7LL * nrec] = atan2(dot3(ak[0], ap[2]), dot3(ak[0], ap[0]));
    w[8LL * nrec] = atan2(dot3(ak[1], ap[0]), dot3(ak[1], ap[1]));
}

constexpr int kThreads = 256;

// one block per (column 3..8, body): running sums over the records; each
// thread a contiguous run, the runs' totals by warp scans
__global__ void __launch_bounds__(kThreads) k_msd_scan(int nrec, double *work) {
    double *w = work + ((long long)blockIdx.y * kW + 3 + blockIdx.x) * nrec;
    const int per = (nrec + kThreads - 1) / kThreads;
    const int k0 = min(nrec, (int)threadIdx.x * per), k1 = min(nrec, k0 + per);
    double s = 0.0;
    for (int k = k0; k < k1; ++k) s += w[k];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double v = s;
    for (int o = 1; o < 32; o <<= 1) {
        const double u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    __shared__ double tot[kThreads / 32];
    if (lane == 31) tot[warp] = v;
    __syncthreads();
    double base = __shfl_up_sync(0xffffffffu, v, 1);
    if (lane == 0) base = 0.0;
    double before = 0.0;
    for (int u = 0; u < warp; ++u) before += tot[u];
    base += before;
    for (int k = k0; k < k1; ++k) {
        base += w[k];
        w[k] = base;
    }
}

// The averages over time origins in integers. GB300 issues FP64 at 2 lanes
// per SM and clock; a pair of records takes 85 FP64 instructions (9 squared
// differences and an arctangent), which bound the FP64 kernel below at 15.0
// ms for 64 bodies x 4000 records x 400 lags. As 57-bit integers the
// differences are exact, the squares are three 32-bit products summed in 64
// and then 128 bits, and the squared angle is a power series: integer work at
// 64 times the rate. Measured for that case: 0.55 ms (k_msd_disp, 9 warp
// instructions per 32 pairs and column) and 1.70 ms (k_msd_angle, bound by
// its ~350, the polynomial mostly), the whole call 15.8 -> 2.87 ms.
// The integer columns take the place of what they come from: X's three that of
// the quaternions (read last by k_msd_prep), the others that of the work
// columns, so the analysis needs no more memory than in FP64.
constexpr int kFixCols = 12;       // X (3), body-frame trajectory (3), angles (3), p-hat (3)
constexpr int kFixBits = 56;       // |value| < 2^56 about the middle of a column's range
constexpr int kRun = 15;           // consecutive origins per lane and tile (odd: no bank conflicts)
constexpr int kTile = 32 * kRun;   // origins per tile
constexpr int kTilesPerSum = 8;    // tiles until the 128-bit sums (< 2^114 a term, 3840 terms) are taken off
constexpr int kWarps = 8;
constexpr int kExact = -0x7FFFFFFF;    // a column of X that its integers hold exactly (k_msd_near)

// a value v of a column as h 2^29 + l, 0 <= l < 2^29: the difference of two is
// (h1 - h0) 2^29 + (l1 - l0), two subtractions without a carry
struct Limbs {
    int l, h;
};

// its two words as the bits of a double (of the column that it replaces)
__device__ __forceinline__ double limbs(long long v) {
    return __hiloint2double((int)(v >> 29), (int)((unsigned)v & 0x1FFFFFFFu));
}

// integer column c of body b (nrec values)
__device__ __forceinline__ double *fix_column(double *q, double *work, int b, int c, int nrec) {
    return c < 3 ? q + ((long long)b * 4 + c) * nrec : work + ((long long)b * kW + (c < 9 ? c : c - 9)) * nrec;
}
__device__ __forceinline__ const Limbs *fix_column(const double *q, const double *work, int b, int c, int nrec) {
    return reinterpret_cast<const Limbs *>(fix_column(const_cast<double *>(q), const_cast<double *>(work), b, c, nrec));
}

// One block per (column, body): the exponent of the column's largest value, its
// scale; bad[b] is set where a value is not finite, the scale is extreme or a
// reference vector has no length (the FP64 kernel then takes the body).
__global__ void __launch_bounds__(kThreads) k_msd_scale(const double *X, const double *work, int nrec, int *unit,
                                                      int *bad) {
    const int c = blockIdx.x, b = blockIdx.y;
    const double *src = c < 3 ? X + (long long)b * nrec * 3 + c
                              : work + ((long long)b * kW + (c < 9 ? c : c - 9)) * nrec;
    const long long st = c < 3 ? 3 : 1;
    __shared__ double smax[kThreads];
    const int t = threadIdx.x;
    double m = 0.0;
    bool fine = true;
#pragma unroll 4
    for (int k = t; k < nrec; k += kThreads) {
        const double v = fabs(src[k * st]);
        fine = fine && v < 0x1p400;
        if (c == 9) {                              // p-hat: a unit vector
            const double p1 = src[k + (long long)nrec], p2 = src[k + 2LL * nrec];
            fine = fine && fabs(fma(v, v, fma(p1, p1, fma(p2, p2, -1.0)))) < 0x1p-40;
        }
        if (v > m) m = v;
    }
    smax[t] = m;
    fine = __syncthreads_and(fine);
    for (int w = kThreads / 2; w > 0; w >>= 1) {
        if (t < w && smax[t + w] > smax[t]) smax[t] = smax[t + w];
        __syncthreads();
    }
    if (t != 0) return;
    m = smax[0];
    if (!fine || (m > 0.0 && m < 0x1p-400)) bad[b] = 1;
    int e = 0;
    frexp(m, &e);                                  // m < 2^e
    unit[b * kFixCols + c] = e;
}

// One block per (column, body), the last one per body all of p-hat: the column
// as integers about the middle of its range, value = fix 2^unit.
__global__ void __launch_bounds__(kThreads) k_msd_fix(const double *X, double *q, double *work, int nrec, int *unit,
                                                    const int *bad) {
    const int c = blockIdx.x, b = blockIdx.y, t = threadIdx.x;
    if (bad[b]) return;
    double *dst = fix_column(q, work, b, c, nrec);
    if (c >= 9) {
        // p-hat: components of a unit vector at 2^56, the last rounding errors
        // of its length taken out (p - p off / 2, off = |p|^2 - 1 exactly)
        for (int k = t; k < nrec; k += kThreads) {
            long long v[3];
            __int128 sum = -((__int128)1 << 112);
            for (int r = 0; r < 3; ++r) {
                v[r] = __double2ll_rn(dst[(long long)r * nrec + k] * 0x1p56);
                sum += (__int128)v[r] * v[r];
            }
            for (int r = 0; r < 3; ++r)
                dst[(long long)r * nrec + k] = limbs(v[r] - (long long)((__int128)v[r] * (long long)sum >> 113));
        }
        return;
    }
    const double *src = c < 3 ? X + (long long)b * nrec * 3 + c : dst;
    const long long st = c < 3 ? 3 : 1;
    __shared__ long long slo[kThreads], shi[kThreads];
    const int e = unit[b * kFixCols + c];
    const double up = ldexp(1.0, 61 - e);
    long long lo = 0x7FFFFFFFFFFFFFFFLL, hi = -0x7FFFFFFFFFFFFFFFLL;
#pragma unroll 4
    for (int k = t; k < nrec; k += kThreads) {
        const long long v = __double2ll_rn(src[k * st] * up);
        if (v < lo) lo = v;
        if (v > hi) hi = v;
    }
    slo[t] = lo;
    shi[t] = hi;
    __syncthreads();
    for (int w = kThreads / 2; w > 0; w >>= 1) {
        if (t < w) {
            if (slo[t + w] < slo[t]) slo[t] = slo[t + w];
            if (shi[t + w] > shi[t]) shi[t] = shi[t + w];
        }
        __syncthreads();
    }
    lo = slo[0];
    hi = shi[0];
    const long long half = (hi - lo) / 2 + 2;
    int sh = 0;
    while ((half >> sh) >= (1LL << kFixBits) - 3) ++sh;
    const long long low = (1LL << sh) - 1, mid = (lo / 2 + hi / 2) & ~low, rnd = (low + 1) >> 1;
    bool coarse = false;
    for (int k = t; k < nrec; k += kThreads) {
        const double v = src[k * st] * up;
        const long long r = __double2ll_rn(v);
        coarse |= v != rint(v) || (r & low);
        dst[k] = limbs((r - mid + rnd) >> sh);
    }
    coarse = __syncthreads_or(coarse);
    if (t != 0) return;
    unit[b * kFixCols + c] = e - 61 + sh;
    // X: the exponent of the column's range, where its grid is coarser than a value (p-hat has no use for the place)
    if (c < 3) unit[b * kFixCols + 9 + c] = coarse ? 64 - __clzll(hi - lo) + e - 61 : kExact;
}

typedef unsigned __int128 U128;

__device__ __forceinline__ U128 shfl_xor128(U128 v, int o) {
    unsigned long long lo = (unsigned long long)v, hi = (unsigned long long)(v >> 64);
    lo = __shfl_xor_sync(0xffffffffu, lo, o);
    hi = __shfl_xor_sync(0xffffffffu, hi, o);
    return ((U128)hi << 64) | lo;
}

// from the low end up, so that only the last addition rounds noticeably
__device__ __forceinline__ double to_double(U128 v) {
    const unsigned long long lo = (unsigned long long)v, hi = (unsigned long long)(v >> 64);
    const double c = fma((double)(unsigned)(lo >> 32), 0x1p32, (double)(unsigned)lo);
    return fma((double)(unsigned)(hi >> 32), 0x1p96, fma((double)(unsigned)hi, 0x1p64, c));
}

// Squared differences of one column (grid y) of one body (grid z): each warp
// takes 8 lags, each lane 15 consecutive origins per tile and a sliding
// window of 8 later records in registers (a quarter load per pair).
constexpr int kLags = 8;
__global__ void __launch_bounds__(32 * kWarps) k_msd_disp(const double *fq, const double *work, const int *unit,
                                                         const int *bad, int nrec, int max_lag, double *out) {
    const int c = blockIdx.y, b = blockIdx.z;
    if (bad[b]) return;
    const Limbs *x = fix_column(fq, work, b, c, nrec);
    __shared__ Limbs s0[kTile], s1[kTile + kLags * kWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int lb0 = blockIdx.x * kLags * kWarps + 1;      // first lag of the block
    const int l0 = lb0 + warp * kLags;                    // of the warp
    U128 acc[kLags];
#pragma unroll
    for (int q = 0; q < kLags; ++q) acc[q] = 0;
    double total = 0.0;                                   // lane q: of lag l0 + q
    auto take = [&]() {
#pragma unroll
        for (int q = 0; q < kLags; ++q) {
            for (int o = 16; o > 0; o >>= 1) acc[q] += shfl_xor128(acc[q], o);
        }
        U128 mine = acc[0];
#pragma unroll
        for (int q = 1; q < kLags; ++q)
            if (lane == q) mine = acc[q];
        total += to_double(mine);
#pragma unroll
        for (int q = 0; q < kLags; ++q) acc[q] = 0;
    };
    int tiles = 0;
    for (int t0 = 0; t0 + lb0 < nrec; t0 += kTile) {
        for (int i = threadIdx.x; i < kTile; i += 32 * kWarps) s0[i] = t0 + i < nrec ? x[t0 + i] : Limbs{0, 0};
        for (int i = threadIdx.x; i < kTile + kLags * kWarps; i += 32 * kWarps)
            s1[i] = t0 + lb0 + i < nrec ? x[t0 + lb0 + i] : Limbs{0, 0};
        __syncthreads();
        auto tile = [&](auto edge) {
            constexpr bool EDGE = decltype(edge)::value;
            const Limbs *p0 = s0 + lane * kRun, *p1 = s1 + warp * kLags + lane * kRun;
            Limbs w[kLags];
            long long A0[kLags], A1[kLags], A2[kLags];
#pragma unroll
            for (int q = 0; q < kLags; ++q) {
                w[q] = p1[q];
                A0[q] = A1[q] = A2[q] = 0;
            }
            const int room = nrec - (t0 + lane * kRun) - l0;      // pair (i, q) exists where i + q < room
#pragma unroll
            for (int i = 0; i < kRun; ++i) {
                const Limbs a = p0[i];
#pragma unroll
                for (int q = 0; q < kLags; ++q) {
                    // D = d1 2^29 + d0: |d1| <= 2^28, |d0| < 2^29
                    int d0 = w[(i + q) % kLags].l - a.l, d1 = w[(i + q) % kLags].h - a.h;
                    if (EDGE && i + q >= room) d0 = d1 = 0;
                    A0[q] += (long long)d0 * d0;
                    A1[q] += (long long)d1 * d0;
                    A2[q] += (long long)d1 * d1;
                }
                if (i + 1 < kRun) w[i % kLags] = p1[i + kLags];
            }
#pragma unroll
            for (int q = 0; q < kLags; ++q)
                acc[q] += (U128)(unsigned long long)A0[q] + ((U128)(__int128)A1[q] << 30) +
                          ((U128)(unsigned long long)A2[q] << 58);
        };
        if (l0 <= max_lag) {                              // warp-uniform
            if (t0 + kTile + l0 + kLags <= nrec) tile(std::false_type{});
            else tile(std::true_type{});
            if (++tiles == kTilesPerSum) {
                take();
                tiles = 0;
            }
        }
        __syncthreads();
    }
    if (l0 > max_lag) return;
    take();
    const int l = l0 + lane;
    if (lane < kLags && l <= max_lag) {
        const int col = c < 6 ? c : c + 1;
        out[((long long)b * max_lag + (l - 1)) * LB_MSD_COLS + col] =
            ldexp(total, 2 * unit[b * kFixCols + c]) / (double)(nrec - l);
    }
}

// The squared angle between unit vectors at distance d apart: with z = d^2 =
// 4 sin^2(theta/2), theta^2 = 4 asin^2(sqrt(z)/2) = sum_n 2 z^n / (n^2 C(2n, n))
// = z + z^2 k(z). k on [0, 2] (angles up to 90 degrees) as the polynomial in
// u = z/2 - 1/2 that interpolates its series at 19 Chebyshev nodes (error
// below 2^-55; powers 0-11 at 2^64, 12-18 at 2^kAsinSqBits).
constexpr int kAsinSqBits = 45;
__constant__ long long kAsinSq[12] = {
    1782374425807430006LL,
    588604380132131925LL,
    241213464260874337LL,
    110996215031437458LL,
    54884372548530884LL,
    28496654949892514LL,
    15326638144275224LL,
    8465569096850234LL,
    4774105254303728LL,
    2737667270170072LL,
    1591456043319638LL,
    935016549813558LL,
};
__constant__ int kAsinSq32[7] = {1058753029, 642436037, 387510425, 203554602, 123855014, 139058146, 85944151};

// LG lags per warp; block z of gridDim.z takes every gridDim.z-th tile and
// leaves its sums in part (one block: the average in out)
template <int LG>
__global__ void __launch_bounds__(32 * kWarps) k_msd_angle(const double *fq, const double *work, const int *bad,
                                                         int nrec, int max_lag, double *part, double *out) {
    const int b = blockIdx.y;
    if (bad[b]) return;
    const Limbs *x = fix_column(fq, work, b, 9, nrec);
    __shared__ Limbs s0[3][kTile], s1[3][kTile + LG * kWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int lb0 = blockIdx.x * LG * kWarps + 1, l0 = lb0 + warp * LG;
    U128 accz[LG], accr[LG];                              // sums of z at 2^112 and of z^2 k at 2^116
    double slow[LG];                                      // sums of the angles beyond 176 degrees (FP64)
#pragma unroll
    for (int q = 0; q < LG; ++q) {
        accz[q] = accr[q] = 0;
        slow[q] = 0.0;
    }
    double total = 0.0;
    auto take = [&]() {
#pragma unroll
        for (int q = 0; q < LG; ++q) {
            for (int o = 16; o > 0; o >>= 1) {
                accz[q] += shfl_xor128(accz[q], o);
                accr[q] += shfl_xor128(accr[q], o);
            }
            if (__any_sync(0xffffffffu, slow[q] != 0.0))
                for (int o = 16; o > 0; o >>= 1) slow[q] += __shfl_xor_sync(0xffffffffu, slow[q], o);
        }
        U128 mz = accz[0], mr = accr[0];
        double ms = slow[0];
#pragma unroll
        for (int q = 1; q < LG; ++q)
            if (lane == q) {
                mz = accz[q];
                mr = accr[q];
                ms = slow[q];
            }
        total += fma(to_double(mz + (mr >> 4)), 0x1p-112, ms);
#pragma unroll
        for (int q = 0; q < LG; ++q) {
            accz[q] = accr[q] = 0;
            slow[q] = 0.0;
        }
    };
    int tiles = 0;
    for (int t0 = blockIdx.z * kTile; t0 + lb0 < nrec; t0 += gridDim.z * kTile) {
        for (int c = 0; c < 3; ++c) {
            const Limbs *xc = x + (long long)c * nrec;
            for (int i = threadIdx.x; i < kTile; i += 32 * kWarps) s0[c][i] = t0 + i < nrec ? xc[t0 + i] : Limbs{0, 0};
            for (int i = threadIdx.x; i < kTile + LG * kWarps; i += 32 * kWarps)
                s1[c][i] = t0 + lb0 + i < nrec ? xc[t0 + lb0 + i] : Limbs{0, 0};
        }
        __syncthreads();
        if (l0 <= max_lag) {
            const int at0 = lane * kRun, at1 = warp * LG + lane * kRun;
            const int room = nrec - (t0 + lane * kRun) - l0;
            long long A0[LG], A1[LG], A2[LG];
#pragma unroll
            for (int q = 0; q < LG; ++q) A0[q] = A1[q] = A2[q] = 0;
            const int run = min(kRun, nrec - t0 - l0);        // of lane 0, which has the most pairs
            for (int i = 0; i < run; ++i) {
                const Limbs a[3] = {s0[0][at0 + i], s0[1][at0 + i], s0[2][at0 + i]};
#pragma unroll
                for (int q = 0; q < LG; ++q) {
                    const Limbs v[3] = {s1[0][at1 + i + q], s1[1][at1 + i + q], s1[2][at1 + i + q]};
                    long long a0 = 0, a1 = 0, a2 = 0;
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        const int d0 = v[c].l - a[c].l, d1 = v[c].h - a[c].h;     // |d1| <= 2^28
                        a0 += (long long)d0 * d0;
                        a1 += (long long)d1 * d0;
                        a2 += (long long)d1 * d1;
                    }
                    long long z = a2 + (a1 >> 28);                           // at 2^54
                    const bool in = i + q < room;
                    const bool far = in && z >= (1LL << 55);                 // beyond 90 degrees
                    if (!in || far) {
                        a0 = a1 = a2 = 0;
                        z = 0;
                    }
                    if (far) {                   // the supplement's squared chord, from the sum of the vectors
                        // to nearest: s = sqrt(z) passes z's error on over 2 s, and the low
                        // product left out would be 12 units
                        long long t0 = 0, t1 = 0, t2 = 0;
#pragma unroll
                        for (int c = 0; c < 3; ++c) {
                            const int e0 = v[c].l + a[c].l, e1 = v[c].h + a[c].h;    // e0 < 2^30
                            t0 += (long long)e0 * e0;
                            t1 += (long long)e1 * e0;
                            t2 += (long long)e1 * e1;
                        }
                        z = t2 + ((t1 + (t0 >> 30) + (1LL << 27)) >> 28);
                        if (z >= (1LL << 55)) z = (1LL << 55) - 1;           // a right angle: u stays below 1/2
                    }
                    if (z < 0) z = 0;
                    // k by Horner's rule in u = z/2 - 1/2, -1/2 <= u < 1/2: the inner seven
                    // steps (below 2^-14, and times u^12 at the end) in 32 bits
                    const long long half = z << 7;                           // z/2 at 2^62
                    const long long u = (z << 8) - (1LL << 62);              // at 2^63
                    const int u32 = (int)(u >> 31);                          // at 2^32
                    int ki = kAsinSq32[6];
#pragma unroll
                    for (int j = 5; j >= 0; --j) ki = kAsinSq32[j] + __mulhi(ki, u32);
                    long long k = (long long)ki << (64 - kAsinSqBits);
                    const FixPair up = fix_split(u);
#pragma unroll
                    for (int j = 11; j >= 0; --j) k = kAsinSq[j] + (fix_mul(fix_split(k), up) << 1);
                    const long long B = fix_mul(fix_split(k), fix_split(half)) << 1;   // z k at 2^62
                    if (!far) {
                        accr[q] += (U128)(unsigned long long)z * (unsigned long long)B;
                    } else if (z >= (1LL << 46)) {
                        // theta = pi - s, s^2 = z (1 + z k), s from an integer square root of
                        // 4^j s^2 in [1/4, 1.24): m = 7 + 2 j odd, z's top bit to bit 59 or 60
                        const int m = (__clzll(z) - 4) | 1;
                        const long long zz = z << m;                         // 4^j z at 2^61
                        const long long r = fix_sqrt(zz + (fix_mul(fix_split(zz), fix_split(B)) << 2));
                        // pi 2^61 less s at 2^61 (j = -1 from z = 1 on)
                        const FixPair th = fix_split(7244019458077122842LL - (m < 7 ? r << 1 : r >> ((m - 7) >> 1)));
                        a2 = (fix_mul(th, th) + 8) >> 4;                     // theta^2 at 2^54
                    } else {
                        auto val = [](Limbs x) { return fma((double)x.h, 0x1p29, (double)x.l); };
                        const double w0[3] = {val(a[0]), val(a[1]), val(a[2])};
                        const double w1[3] = {val(v[0]), val(v[1]), val(v[2])};
                        const double cr[3] = {w0[1] * w1[2] - w0[2] * w1[1], w0[2] * w1[0] - w0[0] * w1[2],
                                              w0[0] * w1[1] - w0[1] * w1[0]};
                        const double th = atan2(sqrt(dot3(cr, cr)), dot3(w0, w1));
                        slow[q] += th * th;
                    }
                    A0[q] += a0;
                    A1[q] += a1;
                    A2[q] += a2;
                }
            }
#pragma unroll
            for (int q = 0; q < LG; ++q)
                accz[q] += (U128)(unsigned long long)A0[q] + ((U128)(__int128)A1[q] << 30) +
                           ((U128)(unsigned long long)A2[q] << 58);
            if (++tiles == kTilesPerSum) {
                take();
                tiles = 0;
            }
        }
        __syncthreads();
    }
    if (l0 > max_lag) return;
    take();
    const int l = l0 + lane;
    if (lane < LG && l <= max_lag) {
        const long long at = (long long)b * max_lag + (l - 1);
        if (gridDim.z > 1) part[(long long)blockIdx.z * gridDim.y * max_lag + at] = total;
        else out[at * LB_MSD_COLS + 6] = total / (double)(nrec - l);
    }
}

// X's averages that a column's grid is too coarse for, again in FP64. The grid
// is 2^-57 of the column's range: where every record takes part in a lag, the
// average is at least 1/n of the range squared and the grid's errors (random,
// and summed over n pairs) stay below the rounding of an FP64 evaluation. A lag
// beyond half the trajectory leaves out the records in its middle, and the
// rest may have moved by far less than the range: an average below 2^(2 s - 8)
// / n, 2^s the range, is recomputed from the values themselves. (The other
// columns are running sums, whose own rounding in such a trajectory is larger
// than the grid.) Nothing to do where the integers are exact, as they are for
// values away from 0 by more than 1/8 of their range.
// Before that, the angle's average from the sums of `parts` blocks (parts > 1).
__global__ void __launch_bounds__(kThreads) k_msd_near(const double *X, int nrec, int max_lag, const int *unit,
                                                     const int *bad, const double *part, int parts, double *out) {
    const int b = blockIdx.y;
    const int *span = unit + b * kFixCols + 9;
    if (bad[b]) return;
    if (parts > 1)
        for (int l = 1 + blockIdx.x + gridDim.x * threadIdx.x; l <= max_lag; l += gridDim.x * kThreads) {
            const long long at = (long long)b * max_lag + (l - 1);
            double v = 0.0;
            for (int z = 0; z < parts; ++z) v += part[(long long)z * gridDim.y * max_lag + at];
            out[at * LB_MSD_COLS + 6] = v / (double)(nrec - l);
        }
    if (span[0] == kExact && span[1] == kExact && span[2] == kExact) return;
    const double *Xb = X + (long long)b * nrec * 3;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __shared__ double red[3][kThreads / 32];
    for (int l = blockIdx.x + 1; l <= max_lag; l += gridDim.x) {
        const int n = nrec - l;
        double *o = out + ((long long)b * max_lag + (l - 1)) * LB_MSD_COLS;
        int need = 0;                        // the same in every thread: written below, after a barrier
        for (int a = 0; a < 3; ++a)
            if (span[a] != kExact && o[a] < ldexp(1.0, 2 * span[a] - 8) / (double)n) need |= 1 << a;
        if (!need) continue;
        double acc[3] = {0.0, 0.0, 0.0};
        for (int t = threadIdx.x; t < n; t += kThreads) {
            const double *x0 = Xb + (long long)t * 3, *x1 = Xb + (long long)(t + l) * 3;
            for (int a = 0; a < 3; ++a) {
                const double d = x1[a] - x0[a];
                acc[a] += d * d;
            }
        }
        for (int a = 0; a < 3; ++a) {
            for (int k = 16; k > 0; k >>= 1) acc[a] += __shfl_down_sync(0xffffffffu, acc[a], k);
            if (lane == 0) red[a][warp] = acc[a];
        }
        __syncthreads();
        if (threadIdx.x < 3 && (need >> threadIdx.x & 1)) {
            double v = 0.0;
            for (int w = 0; w < kThreads / 32; ++w) v += red[threadIdx.x][w];
            o[threadIdx.x] = v / (double)n;
        }
        __syncthreads();                     // red is reused
    }
}

// The same averages in FP64 (blocks over lags and bodies), for the bodies
// that k_msd_scale marked: non-finite values spread to the lags they take part
// in.
__global__ void __launch_bounds__(kThreads) k_msd_lags(const double *X, int nrec, int max_lag, const double *work,
                                                     const int *bad, double *out) {
    const int b = blockIdx.y;
    if (!bad[b]) return;
    for (int l = blockIdx.x + 1; l <= max_lag; l += gridDim.x) {
        const int n = nrec - l;
        double acc[LB_MSD_COLS];
        for (int c = 0; c < LB_MSD_COLS; ++c) acc[c] = 0.0;
        const double *Xb = X + (long long)b * nrec * 3;
        const double *wb = work + (long long)b * nrec * kW;
        for (int t = threadIdx.x; t < n; t += kThreads) {
            const double *x0 = Xb + (long long)t * 3, *x1 = Xb + (long long)(t + l) * 3;
            auto w0 = [&](int c) { return wb[(long long)c * nrec + t]; };
            auto w1 = [&](int c) { return wb[(long long)c * nrec + t + l]; };
            for (int a = 0; a < 3; ++a) {
                const double dx = x1[a] - x0[a];
                acc[a] += dx * dx;
                const double db = w1(3 + a) - w0(3 + a);
                acc[3 + a] += db * db;
                const double dr = w1(6 + a) - w0(6 + a);
                acc[7 + a] += dr * dr;
            }
            const double p[3] = {w0(0), w0(1), w0(2)}, r[3] = {w1(0), w1(1), w1(2)};
            const double cr[3] = {p[1] * r[2] - p[2] * r[1], p[2] * r[0] - p[0] * r[2], p[0] * r[1] - p[1] * r[0]};
            const double th = atan2(sqrt(dot3(cr, cr)), dot3(p, r));
            acc[6] += th * th;
        }
        __shared__ double red[LB_MSD_COLS][kThreads / 32];
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        for (int c = 0; c < LB_MSD_COLS; ++c) {
            double v = acc[c];
            for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
            if (lane == 0) red[c][warp] = v;
        }
        __syncthreads();
        if (threadIdx.x < LB_MSD_COLS) {
            double v = 0.0;
            for (int w = 0; w < kThreads / 32; ++w) v += red[threadIdx.x][w];
            out[((long long)b * max_lag + (l - 1)) * LB_MSD_COLS + threadIdx.x] = v / (double)n;
        }
        __syncthreads();                     // red is reused
    }
}

}  // namespace

// k_msd_angle: four lags a warp (32 a block) and one block per body and lags
// when these fill the SMs twice; else one lag a warp and the tiles split over
// blocks until they do, so that few bodies or few lags are not a few blocks'
// serial work (one body: calls of 4000 records x 80 lags 716 -> 320 us, 606 in
// FP64; 500 x 10 305 -> 270, 271; 16 bodies 4000 x 400 1135 -> 932, 4426)
static int angle_parts(int nrec, int nbodies, int max_lag, bool &wide) {
    const long long want = 2LL * sm_count(), nb = nbodies;
    wide = nb * ((max_lag + 4 * kWarps - 1) / (4 * kWarps)) >= want;
    const long long blocks = nb * ((max_lag + kWarps - 1) / kWarps);
    const long long tiles = (nrec - 2) / kTile + 1;
    return wide ? 1 : (int)std::max(1LL, std::min(tiles, want / blocks));
}

// the sums that angle_parts' blocks leave: parts x 8 lags x blocks at most
static size_t part_doubles() { return 2 * (size_t)sm_count() * kWarps; }

size_t msd_work_bytes(int nrec, int nbodies) {
    return ((size_t)nrec * nbodies * kW + part_doubles()) * sizeof(double) +
           (size_t)nbodies * (kFixCols + 1) * sizeof(int);
}

cudaError_t launch_msd(const double *X, double *q, int nrec, int nbodies, int max_lag, const double *p_ref,
                       void *work, double *out, cudaStream_t s) {
    const size_t n = (size_t)nrec * nbodies;
    const unsigned nb = (unsigned)nbodies;
    double *w = static_cast<double *>(work);
    double *part = w + n * kW;
    int *unit = reinterpret_cast<int *>(part + part_doubles()), *bad = unit + (size_t)nbodies * kFixCols;
    cudaError_t e = cudaMemsetAsync(bad, 0, sizeof(int) * nbodies, s);
    if (e != cudaSuccess) return e;
    k_msd_prep<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(X, q, nrec, nbodies, p_ref, w);
    k_msd_scan<<<dim3(6, nb), kThreads, 0, s>>>(nrec, w);
    k_msd_scale<<<dim3(kFixCols, nb), kThreads, 0, s>>>(X, w, nrec, unit, bad);
    k_msd_fix<<<dim3(10, nb), kThreads, 0, s>>>(X, q, w, nrec, unit, bad);
    const unsigned gd = (unsigned)((max_lag + kLags * kWarps - 1) / (kLags * kWarps));
    k_msd_disp<<<dim3(gd, 9, nb), 32 * kWarps, 0, s>>>(q, w, unit, bad, nrec, max_lag, out);
    bool wide = false;
    const int parts = angle_parts(nrec, nbodies, max_lag, wide);
    const unsigned lags = wide ? 4 * kWarps : kWarps;
    const dim3 ga((max_lag + lags - 1) / lags, nb, (unsigned)parts);
    if (wide) k_msd_angle<4><<<ga, 32 * kWarps, 0, s>>>(q, w, bad, nrec, max_lag, part, out);
    else k_msd_angle<1><<<ga, 32 * kWarps, 0, s>>>(q, w, bad, nrec, max_lag, part, out);
    const dim3 gl((unsigned)std::min(max_lag, std::max(8, 2048 / nbodies)), nb);
    k_msd_near<<<gl, kThreads, 0, s>>>(X, nrec, max_lag, unit, bad, part, parts, out);
    k_msd_lags<<<gl, kThreads, 0, s>>>(X, nrec, max_lag, w, bad, out);
    return cudaGetLastError();
}

// Host side of the trajectory readers: the valid records of body `id` (of
// nb) in the ring, oldest first. Records k = k0 .. step / every exist;
// the ring keeps the last cap of them.
cudaError_t copy_records(const double *ring, int every, int cap, long long k0, long long step, int nb, int id,
                         int max_records, long long *steps, double *X, double *q, int *count, cudaStream_t s) {
    *count = 0;
    if (!ring || every <= 0) return cudaSuccess;
    const long long k_last = step / every;
    long long k_first = k_last - cap + 1;
    if (k_first < k0) k_first = k0;
    long long n = k_last - k_first + 1;
    if (n <= 0) return cudaSuccess;
    if (n > max_records) {                  // the most recent max_records
        k_first = k_last - max_records + 1;
        n = max_records;
    }
    // one strided 2-D copy per contiguous run of slots (at most two)
    std::vector<double> rec((size_t)n * 7);
    long long done = 0;
    while (done < n) {
        const long long slot = (k_first + done - 1) % cap;
        const long long run = std::min<long long>(n - done, cap - slot);
        cudaError_t e = cudaMemcpy2DAsync(rec.data() + done * 7, 7 * sizeof(double),
                                          ring + (slot * nb + id) * 7, (size_t)nb * 7 * sizeof(double),
                                          7 * sizeof(double), (size_t)run, cudaMemcpyDeviceToHost, s);
        if (e != cudaSuccess) return e;
        done += run;
    }
    cudaError_t e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return e;
    for (long long r = 0; r < n; ++r) {
        if (steps) steps[r] = (k_first + r) * every;
        if (X) std::memcpy(X + 3 * r, &rec[7 * r], 3 * sizeof(double));
        if (q) std::memcpy(q + 4 * r, &rec[7 * r + 3], 4 * sizeof(double));
    }
    *count = (int)n;
    return cudaSuccess;
}

}  // namespace lbk

extern "C" lb_status lb_msd_trajectory(const double *X, const double *q, int nrec, int nbodies, int max_lag,
                                       const double p_ref[3], double *out, void *cuda_stream, char *err,
                                       size_t err_len) {
    auto fail = [&](lb_status st, const std::string &m) {
        if (err && err_len) {
            std::strncpy(err, m.c_str(), err_len - 1);
            err[err_len - 1] = 0;
        }
        return st;
    };
    if (!X || !q || !p_ref || !out) return fail(LB_ERR_ARG, "null pointer");
    if (nbodies < 1 || nrec < 2 || max_lag < 1 || max_lag >= nrec || nbodies > 65535)
        return fail(LB_ERR_ARG, "need nbodies in [1, 65535], nrec >= 2 and 1 <= max_lag < nrec");
    if (!(p_ref[0] * p_ref[0] + p_ref[1] * p_ref[1] + p_ref[2] * p_ref[2] > 0.0))
        return fail(LB_ERR_ARG, "p_ref must be non-zero");
    cudaStream_t s = (cudaStream_t)cuda_stream;
    const size_t nX = (size_t)nrec * nbodies * 3, nq = (size_t)nrec * nbodies * 4;
    const size_t nw = (lbk::msd_work_bytes(nrec, nbodies) + 7) / 8, no = (size_t)max_lag * nbodies * LB_MSD_COLS;
    double *d = nullptr;
    const size_t total = nX + nq + nw + no + 3;
    cudaError_t e = cudaMalloc((void **)&d, total * sizeof(double));
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        return fail(LB_ERR_OOM, "device allocation for the trajectory failed");
    }
    if (e != cudaSuccess) return fail(LB_ERR_CUDA, std::string("cudaMalloc: ") + cudaGetErrorString(e));
    double *dX = d, *dq = dX + nX, *dw = dq + nq, *dout = dw + nw, *dp = dout + no;
    e = cudaMemcpyAsync(dX, X, nX * sizeof(double), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(dq, q, nq * sizeof(double), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(dp, p_ref, 3 * sizeof(double), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = lbk::launch_msd(dX, dq, nrec, nbodies, max_lag, dp, dw, dout, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(out, dout, no * sizeof(double), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(d);
    if (e != cudaSuccess) return fail(LB_ERR_CUDA, std::string("lb_msd_trajectory: ") + cudaGetErrorString(e));
    return LB_OK;
}

// --------------------------------------------------------------- pore frame
// Pore-frame analysis (Sec. 2.8 and the SI "Pore-frame coordinate
// determination"): centres relative to the pore axis (x^c, y^c across it, z
// along it); one interval's displacement rotated into the frame of its start
// (x^p radial, y^p azimuthal, z^p axial; cos and sin of theta as x^c / r and
// y^c / r) and summed; the MSD of the sub-trajectories binned by the radial
// coordinate of their first record.
namespace lbk {
namespace {

struct PoreFrame {
    int a1, a2, ax;
    double c1, c2;
};

__device__ __forceinline__ double radial(double xc, double yc) {
    return sqrt(__dadd_rn(__dmul_rn(xc, xc), __dmul_rn(yc, yc)));   // no contraction: bins depend on it
}

// one thread per record: increment over [k-1, k] (zero for k = 0) and r_k
__global__ void k_pore_prep(const double *X, int nrec, PoreFrame pf, double *work) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nrec) return;
    const double *x = X + 3ll * k;
    const double xc = x[pf.a1] - pf.c1, yc = x[pf.a2] - pf.c2;
    double *w = work + 4ll * k;
    w[3] = radial(xc, yc);
    if (k == 0) {
        w[0] = w[1] = w[2] = 0.0;
        return;
    }
    const double *xp = x - 3;
    const double xp1 = xp[pf.a1] - pf.c1, yp1 = xp[pf.a2] - pf.c2;
    const double r0 = radial(xp1, yp1);
    const double c = r0 > 0.0 ? xp1 / r0 : 1.0, s = r0 > 0.0 ? yp1 / r0 : 0.0;
    const double dx = xc - xp1, dy = yc - yp1, dz = x[pf.ax] - xp[pf.ax];
    w[0] = c * dx + s * dy;
    w[1] = -s * dx + c * dy;
    w[2] = dz;
}

__global__ void k_pore_scan(int nrec, double *work) {
    const int c = threadIdx.x;
    if (c >= 3) return;
    double acc = 0.0;
    for (int k = 0; k < nrec; ++k) {
        acc += work[4ll * k + c];
        work[4ll * k + c] = acc;
    }
}

// one block per lag: per-bin sums in shared memory
__global__ void k_pore_lags(int nrec, int nbins, double R, int max_lag, const double *work, double *out,
                            long long *counts) {
    extern __shared__ double sm[];
    double *acc = sm;                                            // [nbins][3]
    unsigned long long *cnt = reinterpret_cast<unsigned long long *>(sm + 3 * nbins);
    for (int i = threadIdx.x; i < 4 * nbins; i += blockDim.x) sm[i] = 0.0;
    __syncthreads();
    const int l = blockIdx.x + 1;
    for (int t = threadIdx.x; t < nrec - l; t += blockDim.x) {
        const double *w0 = work + 4ll * t, *w1 = work + 4ll * (t + l);
        const double fb = floor(__dmul_rn(w0[3] / R, (double)nbins));
        if (!(fb >= 0.0 && fb < (double)nbins)) continue;
        const int b = (int)fb;
        for (int c = 0; c < 3; ++c) {
            const double d = w1[c] - w0[c];
            atomicAdd(&acc[3 * b + c], d * d);
        }
        atomicAdd(&cnt[b], 1ull);
    }
    __syncthreads();
    for (int b = threadIdx.x; b < nbins; b += blockDim.x) {
        const unsigned long long n = cnt[b];
        for (int c = 0; c < 3; ++c)
            out[((long long)b * max_lag + (l - 1)) * 3 + c] = n ? acc[3 * b + c] / (double)n : 0.0;
        counts[(long long)b * max_lag + (l - 1)] = (long long)n;
    }
}

}  // namespace
}  // namespace lbk

extern "C" lb_status lb_pore_msd(const double *X, int nrec, int nx, int ny, int nz, int axis, double R_pore,
                                 int nbins, int max_lag, double *out, long long *counts, void *cuda_stream,
                                 char *err, size_t err_len) {
    auto fail = [&](lb_status st, const std::string &m) {
        if (err && err_len) {
            std::strncpy(err, m.c_str(), err_len - 1);
            err[err_len - 1] = 0;
        }
        return st;
    };
    if (!X || !out || !counts) return fail(LB_ERR_ARG, "null pointer");
    if (nrec < 2 || max_lag < 1 || max_lag >= nrec || nbins < 1 || nbins > 4096 || axis < 0 || axis > 2 ||
        !(R_pore > 0.0) || nx < 1 || ny < 1 || nz < 1)
        return fail(LB_ERR_ARG, "need nrec >= 2, 1 <= max_lag < nrec, 1 <= nbins <= 4096, axis 0-2, R_pore > 0");
    const int n[3] = {nx, ny, nz};
    lbk::PoreFrame pf;
    pf.ax = axis;
    pf.a1 = axis == 0 ? 1 : 0;
    pf.a2 = axis == 2 ? 1 : 2;
    pf.c1 = 0.5 * n[pf.a1];
    pf.c2 = 0.5 * n[pf.a2];
    cudaStream_t s = (cudaStream_t)cuda_stream;
    const size_t nX = 3ull * nrec, nw = 4ull * nrec, no = 3ull * nbins * max_lag, nc = (size_t)nbins * max_lag;
    double *d = nullptr;
    cudaError_t e = cudaMalloc((void **)&d, (nX + nw + no + nc) * sizeof(double));
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        return fail(LB_ERR_OOM, "device allocation for the trajectory failed");
    }
    if (e != cudaSuccess) return fail(LB_ERR_CUDA, std::string("cudaMalloc: ") + cudaGetErrorString(e));
    double *dX = d, *dw = dX + nX, *dout = dw + nw;
    long long *dcnt = reinterpret_cast<long long *>(dout + no);
    const size_t smem = 4ull * nbins * sizeof(double);
    e = cudaMemcpyAsync(dX, X, nX * sizeof(double), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) {
        lbk::k_pore_prep<<<(nrec + 255) / 256, 256, 0, s>>>(dX, nrec, pf, dw);
        lbk::k_pore_scan<<<1, 32, 0, s>>>(nrec, dw);
        if (smem > 48 * 1024)
            e = cudaFuncSetAttribute(lbk::k_pore_lags, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess) {
            lbk::k_pore_lags<<<max_lag, 256, smem, s>>>(nrec, nbins, R_pore, max_lag, dw, dout, dcnt);
            e = cudaGetLastError();
        }
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(out, dout, no * sizeof(double), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(counts, dcnt, nc * sizeof(long long), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(d);
    if (e != cudaSuccess) return fail(LB_ERR_CUDA, std::string("lb_pore_msd: ") + cudaGetErrorString(e));
    return LB_OK;
}
