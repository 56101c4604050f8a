// Raspberry shell construction on the GPU (Ustach & Faller, arXiv:1604.01829,
// Sec. 2.1 and the SI section "Details for ellipsoidal raspberry
// construction").
//
// Beads of one shell relax on an ellipsoid x^2/a^2 + y^2/b^2 + z^2/c^2 = 1
// under two forces: a harmonic pull -2k (r - r_s) towards the nearest surface
// point r_s, and pairwise WCA repulsion between the beads of the shell. The
// nearest point follows from the normal condition r - r_s = (t/2) grad S(r_s),
// i.e. r_s = (x a^2/(t + a^2), ...) (Eq. (xtoxs)), with t the root of
// F(t) = sum (x a/(t + a^2))^2 - 1 (Eq. (bisection) read without its printed
// "+1", which contradicts Eq. (xtoxs)). F decreases for t > -m^2 (m the
// smallest semi-axis); the root lies in [-m^2 + m |x_m|, a_max |r|], where the
// term of the smallest axis alone is 1 at the lower end and F <= 0 at the
// upper end. The paper stops its bisection at |F| < 1e-6; here the bracket is
// halved a fixed number of times (64 in FP64, 40 in FP32), which is tighter.
// Integration: damped leapfrog with unit mass, v <- (1 - eta dt) v + dt F,
// r <- r + dt v.
//
// Design: one thread block per shell; the automatic pair search keeps
// neighbour lists (k_relax_list). The explicit all-pairs and cell-list
// searches: the shell's positions and velocities in
// shared memory (structure of arrays, 6 n values: 192 KB for 4096 beads in
// FP64), each thread owning up to 4 beads. A step reads every position once per owned
// bead group (shared-memory broadcast: all lanes of a warp read the same j),
// then, after a barrier, each thread moves its beads. Shells are independent,
// so many of them fill the GPU in one launch.
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include <cuda_runtime.h>

#include "../../include/lb.h"
#include "lb_device.cuh"

namespace lbk {

namespace {

constexpr int kShellThreads = 1024;
constexpr int kMaxCells = 4096;                     // cells per shell at most
constexpr double kWcaCut = 1.122462048309373;      // 2^(1/6)

template <typename R>
struct ShellArgs {
    const double *axes;       // [nshells][3]
    const int *count;         // [nshells]
    const long long *offset;  // [nshells] first bead of each shell
    double *xyz;              // [total][3], in and out
    int max_count;            // largest shell (shared-memory extent)
    R k2;                     // 2k
    R sig2, rc2, eps24;       // sigma^2, (2^(1/6) sigma)^2, 24 epsilon
    R dt, damp;               // dt, 1 - eta dt
    long long steps;
    int project_final;
    // cell list (CELLS kernels): per shell the grid g[3] over the box
    // [-L, L) per axis (L = box[3 s + q]) with cells of size >= the WCA range
    const int *cgrid;         // [nshells][3]
    const double *cbox;       // [nshells][3] half-widths L
    int max_cells;            // largest grid (shared-memory extent)
    int *err;                 // index checks of checked builds (LB_CHECKS): bit 2 on failure
    R rl2, move2;             // neighbour lists: (range + skin)^2 and the squared move that outdates them
};

// Lists of crowded shells in device memory: [nshells][rows][max_count], and the
// longest list of each shell. Not among ShellArgs: the kernels without them keep
// their arguments' places (a small shell's step 1.61 -> 1.70 us otherwise).
template <bool LONG>
struct LongLists {};
template <>
struct LongLists<true> {
    uint16_t *list;
    const int *len;
    int rows;
};

__device__ __forceinline__ float rdiv(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ double rdiv(double a, double b) { return a / b; }

// Nearest surface point of (x, y, z): bisection for the root of F(t).
template <typename R>
__device__ __forceinline__ void surface_point(R x, R y, R z, R a, R b, R c, R &sx, R &sy, R &sz) {
    constexpr int H = sizeof(R) == 8 ? 64 : 40;
    const R m = fmin(a, fmin(b, c));
    R xm = R(0);
    if (a == m) xm = fmax(xm, fabs(x));
    if (b == m) xm = fmax(xm, fabs(y));
    if (c == m) xm = fmax(xm, fabs(z));
    R lo = -m * m + m * xm;
    R hi = fmax(a, fmax(b, c)) * sqrt(x * x + y * y + z * z);
    if (hi < lo) hi = lo;
    const R a2 = a * a, b2 = b * b, c2 = c * c, xa = x * a, yb = y * b, zc = z * c;
    for (int it = 0; it < H; ++it) {
        const R mid = R(0.5) * (lo + hi);
        const R u = rdiv(xa, mid + a2), v = rdiv(yb, mid + b2), w = rdiv(zc, mid + c2);
        if (u * u + v * v + w * w - R(1) > R(0)) lo = mid;
        else hi = mid;
    }
    const R t = R(0.5) * (lo + hi);
    const R da = t + a2, db = t + b2, dc = t + c2;
    // a denominator vanishes only when the bracket collapsed onto -m^2 (a bead
    // on the medial set inside, without a unique nearest point): component 0
    sx = da > R(0) ? rdiv(x * a2, da) : R(0);
    sy = db > R(0) ? rdiv(y * b2, db) : R(0);
    sz = dc > R(0) ? rdiv(z * c2, dc) : R(0);
}

// The same point by Newton's iteration from a guess t (the bead's root of the
// step before; updated). F is convex and falls on (-m^2, inf): from the left
// of the root the iteration climbs to it without passing, from the right one
// step leads to the left, and lo = -m^2 + m |x_m| (F(lo) >= 0) bounds it from
// below. It ends after a step shorter than `tol` times the distance to the
// nearest pole, whose square is below rounding: one step is usual where a
// bead has moved by little. A bead for which it does not end so (the root at
// the pole: no unique nearest point) takes the bisection.
template <typename R>
__device__ __forceinline__ void surface_point_near(R x, R y, R z, R a, R b, R c, R &t, R &sx, R &sy, R &sz) {
    constexpr R tol = sizeof(R) == 8 ? R(0x1p-28) : R(0x1p-13);
    const R a2 = a * a, b2 = b * b, c2 = c * c, xa = x * a, yb = y * b, zc = z * c;
    const R m = fmin(a, fmin(b, c)), m2 = m * m;
    R xm = R(0);
    if (a == m) xm = fmax(xm, fabs(x));
    if (b == m) xm = fmax(xm, fabs(y));
    if (c == m) xm = fmax(xm, fabs(z));
    const R lo = -m2 + m * xm;
    t = fmax(t, lo);
    for (int it = 0; it < 24; ++it) {
        const R ia = rdiv(R(1), t + a2), ib = rdiv(R(1), t + b2), ic = rdiv(R(1), t + c2);
        const R u = xa * ia, v = yb * ib, w = zc * ic;
        const R F = u * u + v * v + w * w - R(1), D = u * u * ia + v * v * ib + w * w * ic;
        const R d = rdiv(R(0.5) * F, D), tn = t + d;
        // a NaN (0/0 at the pole) never ends the loop
        if (fabs(d) <= tol * (t + m2) && tn > lo) {
            // 1/(t + d + a^2) from 1/(t + a^2): the next term, (d ia)^3, is below rounding
            const R ea = d * ia, eb = d * ib, ec = d * ic;
            t = tn;
            sx = x * a2 * (ia - ia * (ea - ea * ea));
            sy = y * b2 * (ib - ib * (eb - eb * eb));
            sz = z * c2 * (ic - ic * (ec - ec * ec));
            return;
        }
        t = fmax(tn, lo);
    }
    surface_point(x, y, z, a, b, c, sx, sy, sz);
    t = lo;
}

// Block-wide exclusive scan of cnt[0..C) into start[0..C] (start[C] = total),
// resetting cnt to 0 (it then serves as the fill cursor). wsum: 32 ints.
__device__ __forceinline__ void scan_cells(int *cnt, int *start, int C, int *wsum) {
    const int T = blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int per = (C + T - 1) / T;
    const int c0 = min(C, tid * per), c1 = min(C, c0 + per);
    int sum = 0;
    for (int c = c0; c < c1; ++c) sum += cnt[c];
    int v = sum;
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    if (lane == 31) wsum[warp] = v;
    __syncthreads();
    if (warp == 0) {
        int w = lane < ((T + 31) >> 5) ? wsum[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += u;
        }
        wsum[lane] = w;
    }
    __syncthreads();
    int base = v - sum + (warp > 0 ? wsum[warp - 1] : 0);
    for (int c = c0; c < c1; ++c) {
        start[c] = base;
        base += cnt[c];
        cnt[c] = 0;
    }
    if (tid == T - 1) start[C] = base;
}

// One block per shell. CELLS: pair search through a cell list rebuilt every
// step (counting sort by cell, beads of a cell in index order, so results do
// not depend on the order of the atomics); a step in which a bead lies
// outside the grid's box searches all pairs instead. Without CELLS every
// step tests all pairs, summed in index order.
template <typename R, int BPT, bool CELLS>
__global__ void __launch_bounds__(kShellThreads) k_relax_shells(const ShellArgs<R> a) {
    extern __shared__ unsigned char smem_raw[];
    R *px = reinterpret_cast<R *>(smem_raw);
    R *py = px + a.max_count;
    R *pz = py + a.max_count;
    R *vx = pz + a.max_count;              // velocities
    R *vy = vx + a.max_count;
    R *vz = vy + a.max_count;
    int *bcell = reinterpret_cast<int *>(vz + a.max_count);   // CELLS: cell of each bead
    int *sorted = bcell + a.max_count;                        // bead indices by cell
    int *cnt = sorted + a.max_count;                          // per cell count / cursor
    int *start = cnt + a.max_cells;                           // per cell first slot (+1)
    __shared__ int wsum[32];
    const int s = blockIdx.x;
    const int n = a.count[s];
    double *X = a.xyz + 3 * a.offset[s];
    const R ax = (R)a.axes[3 * s], ay = (R)a.axes[3 * s + 1], az = (R)a.axes[3 * s + 2];
    int gx = 1, gy = 1, gz = 1, C = 1;
    R Lx = R(0), Ly = R(0), Lz = R(0), ihx = R(0), ihy = R(0), ihz = R(0);
    if (CELLS) {
        gx = a.cgrid[3 * s]; gy = a.cgrid[3 * s + 1]; gz = a.cgrid[3 * s + 2];
        C = gx * gy * gz;
        Lx = (R)a.cbox[3 * s]; Ly = (R)a.cbox[3 * s + 1]; Lz = (R)a.cbox[3 * s + 2];
        ihx = (R)gx / (R(2) * Lx); ihy = (R)gy / (R(2) * Ly); ihz = (R)gz / (R(2) * Lz);
        for (int c = threadIdx.x; c < C; c += blockDim.x) cnt[c] = 0;
    }
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        px[i] = (R)X[3 * i];
        py[i] = (R)X[3 * i + 1];
        pz[i] = (R)X[3 * i + 2];
        vx[i] = vy[i] = vz[i] = R(0);
    }
    __syncthreads();

    for (long long step = 0; step < a.steps; ++step) {
        R xi[BPT], yi[BPT], zi[BPT], fx[BPT], fy[BPT], fz[BPT];
        int id[BPT];
        bool outside = false;
#pragma unroll
        for (int b = 0; b < BPT; ++b) {
            const int i = threadIdx.x + b * blockDim.x;
            id[b] = i < n ? i : -1;
            xi[b] = yi[b] = zi[b] = fx[b] = fy[b] = fz[b] = R(0);
            if (i < n) {
                xi[b] = px[i];
                yi[b] = py[i];
                zi[b] = pz[i];
                if (CELLS) {
                    const int cx = (int)floor((xi[b] + Lx) * ihx), cy = (int)floor((yi[b] + Ly) * ihy),
                              cz = (int)floor((zi[b] + Lz) * ihz);
                    if (cx < 0 || cx >= gx || cy < 0 || cy >= gy || cz < 0 || cz >= gz) {
                        outside = true;
                        bcell[i] = -1;
                    } else {
                        const int c = chk(cx + gx * (cy + gy * cz), C, a.err);
                        bcell[i] = c;
                        atomicAdd(&cnt[c], 1);
                    }
                }
                R sx, sy, sz;
                surface_point(xi[b], yi[b], zi[b], ax, ay, az, sx, sy, sz);
                fx[b] = -a.k2 * (xi[b] - sx);
                fy[b] = -a.k2 * (yi[b] - sy);
                fz[b] = -a.k2 * (zi[b] - sz);
            }
        }
        auto pair = [&](int b, int j) {
            const R dx = xi[b] - px[j], dy = yi[b] - py[j], dz = zi[b] - pz[j];
            const R r2 = dx * dx + dy * dy + dz * dz;
            if (r2 < a.rc2 && j != id[b]) {
                const R s2 = rdiv(a.sig2, r2);
                const R s6 = s2 * s2 * s2;
                const R fm = rdiv(a.eps24 * (R(2) * s6 * s6 - s6), r2);
                fx[b] += fm * dx;
                fy[b] += fm * dy;
                fz[b] += fm * dz;
            }
        };
        bool use_cells = false;
        if (CELLS) {
            use_cells = !__syncthreads_or(outside);
            if (use_cells) {
                scan_cells(cnt, start, C, wsum);
                __syncthreads();
                for (int i = threadIdx.x; i < n; i += blockDim.x)
                    sorted[chk(start[bcell[i]] + atomicAdd(&cnt[bcell[i]], 1), n, a.err)] = i;
                __syncthreads();
                // beads of each cell in index order (few per cell: insertion sort)
                for (int c = threadIdx.x; c < C; c += blockDim.x) {
                    for (int k = start[c] + 1; k < start[c + 1]; ++k) {
                        const int v = sorted[k];
                        int m = k - 1;
                        while (m >= start[c] && sorted[m] > v) {
                            sorted[m + 1] = sorted[m];
                            --m;
                        }
                        sorted[m + 1] = v;
                    }
                }
                __syncthreads();
            } else {
                for (int c = threadIdx.x; c < C; c += blockDim.x) cnt[c] = 0;
            }
        }
        if (use_cells) {
            // WCA over the 27 cells around each bead (cells are at least as wide as the range)
#pragma unroll
            for (int b = 0; b < BPT; ++b) {
                if (id[b] < 0) continue;
                const int c = bcell[id[b]];
                const int cx = c % gx, cy = (c / gx) % gy, cz = c / (gx * gy);
                for (int dz = -1; dz <= 1; ++dz) {
                    const int z = cz + dz;
                    if (z < 0 || z >= gz) continue;
                    for (int dy = -1; dy <= 1; ++dy) {
                        const int y = cy + dy;
                        if (y < 0 || y >= gy) continue;
                        for (int dx = -1; dx <= 1; ++dx) {
                            const int x = cx + dx;
                            if (x < 0 || x >= gx) continue;
                            const int cc = x + gx * (y + gy * z);
                            for (int k = start[cc]; k < start[cc + 1]; ++k) pair(b, chk(sorted[k], n, a.err));
                        }
                    }
                }
            }
        } else {
            // pairwise WCA, summed over j in index order (one read of j for all owned beads)
            for (int j = 0; j < n; ++j) {
                const R xj = px[j], yj = py[j], zj = pz[j];
#pragma unroll
                for (int b = 0; b < BPT; ++b) {
                    const R dx = xi[b] - xj, dy = yi[b] - yj, dz = zi[b] - zj;
                    const R r2 = dx * dx + dy * dy + dz * dz;
                    if (r2 < a.rc2 && j != id[b] && id[b] >= 0) {
                        const R s2 = rdiv(a.sig2, r2);
                        const R s6 = s2 * s2 * s2;
                        const R fm = rdiv(a.eps24 * (R(2) * s6 * s6 - s6), r2);
                        fx[b] += fm * dx;
                        fy[b] += fm * dy;
                        fz[b] += fm * dz;
                    }
                }
            }
        }
        __syncthreads();   // every thread has read every position of this step
#pragma unroll
        for (int b = 0; b < BPT; ++b) {
            const int i = id[b];
            if (i < 0) continue;
            const R ux = a.damp * vx[i] + a.dt * fx[b];
            const R uy = a.damp * vy[i] + a.dt * fy[b];
            const R uz = a.damp * vz[i] + a.dt * fz[b];
            vx[i] = ux;
            vy[i] = uy;
            vz[i] = uz;
            px[i] = xi[b] + a.dt * ux;
            py[i] = yi[b] + a.dt * uy;
            pz[i] = zi[b] + a.dt * uz;
        }
        if (CELLS && use_cells)
            for (int c = threadIdx.x; c < C; c += blockDim.x) cnt[c] = 0;
        __syncthreads();   // positions of the next step are complete
    }

    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        R x = px[i], y = py[i], z = pz[i];
        if (a.project_final) {
            R sx, sy, sz;
            surface_point(x, y, z, ax, ay, az, sx, sy, sz);
            x = sx;
            y = sy;
            z = sz;
        }
        X[3 * i] = (double)x;
        X[3 * i + 1] = (double)y;
        X[3 * i + 2] = (double)z;
    }
}

// Pair search through per-bead neighbour lists that last many steps: list
// column i holds the beads within rl = the WCA range + skin of bead i when it
// was built, in index order, and stays complete until some bead has moved by
// skin / 2; the pairs outside the range add nothing, so every step sums what
// the all-pairs search sums, in the same order. A list longer than kListLen
// is not kept: its bead tests all pairs. Crowded shells (LONG: more than
// kCrowded beads expected within rl of a bead) have longer lists in device
// memory, read through L1: at kListLen most of their beads would test all
// pairs. Per step, with short lists, long ones and the cell list: FP32 2000
// beads at three a unit area 279 / 18.7 / 117 us, 900 there 59 / 8.3 / 59, 200
// at six 18.6 / 7.4 / -; FP64 2000 at three 7204 / 724 / 4818. A shell that
// flies apart rebuilds its lists every step whatever their length (2000 at six,
// dt^2 times the forces ~0.01: 661 / 401 / 332).
//
// One block per shell, positions in two shared buffers (one barrier a step),
// velocities, list references and surface roots in registers. Bound by the
// latency of ~550 dependent instructions per warp and step and one barrier
// (ncu: issue 30 %, shared-memory pipe 9 %); the searches above spend 40
// halvings (three divisions each) and n pair tests per bead. Measured on
// GB300 per step, FP32: 203 shells of up to 344 beads 32.2 -> 2.9 us (all
// pairs before), one (15, 5, 5) raspberry 29.0 -> 3.0 us (cell list before),
// one shell of 2400 beads 117 -> 14.8 us (cell list); FP64, the 203 shells:
// 1134 -> 98 us (its divisions on the FP64 pipe).
constexpr int kListLen = 32;
constexpr double kCrowded = 24.0;
constexpr size_t kLongBytes = 1ull << 30;           // device memory for long lists at most
#ifndef LB_LIST_SKIN
#define LB_LIST_SKIN 0.15
#endif

// threads of a block at most: FP64 beads need twice the registers
template <typename R>
constexpr int list_threads() { return sizeof(R) == 8 ? 512 : 1024; }

template <typename R, int BPT, bool LONG>
__global__ void __launch_bounds__(list_threads<R>()) k_relax_list(const ShellArgs<R> a, const LongLists<LONG> ll) {
    extern __shared__ unsigned char smem_raw[];
    R *pos = reinterpret_cast<R *>(smem_raw);                          // [2][3][max_count]
    const int M = a.max_count;
    const int s = blockIdx.x;
    uint16_t *list = reinterpret_cast<uint16_t *>(pos + 6 * (size_t)M);   // [cap][max_count]
    int cap = kListLen;
    if constexpr (LONG) {
        list = ll.list + (size_t)s * ll.rows * M;
        cap = ll.len[s];
    }
    const int n = a.count[s];
    double *X = a.xyz + 3 * a.offset[s];
    const R ax = (R)a.axes[3 * s], ay = (R)a.axes[3 * s + 1], az = (R)a.axes[3 * s + 2];
    R xi[BPT], yi[BPT], zi[BPT], vx[BPT], vy[BPT], vz[BPT], rx[BPT], ry[BPT], rz[BPT], t[BPT];
    int len[BPT];
#pragma unroll
    for (int b = 0; b < BPT; ++b) {
        const int i = threadIdx.x + b * blockDim.x;
        xi[b] = yi[b] = zi[b] = vx[b] = vy[b] = vz[b] = rx[b] = ry[b] = rz[b] = t[b] = R(0);
        len[b] = 0;
        if (i < n) {
            xi[b] = (R)X[3 * i];
            yi[b] = (R)X[3 * i + 1];
            zi[b] = (R)X[3 * i + 2];
            pos[i] = xi[b];
            pos[M + i] = yi[b];
            pos[2 * M + i] = zi[b];
        }
    }
    bool rebuild = true;
    __syncthreads();
    for (long long step = 0; step < a.steps; ++step) {
        const R *px = pos + (step & 1) * 3 * (size_t)M, *py = px + M, *pz = py + M;
        R *nx = pos + ((step + 1) & 1) * 3 * (size_t)M, *ny = nx + M, *nz = ny + M;
        if (rebuild) {                       // each thread its own beads' columns: no barrier needed
#pragma unroll
            for (int b = 0; b < BPT; ++b) {
                const int i = threadIdx.x + b * blockDim.x;
                if (i >= n) continue;
                int k = 0;
                for (int j = 0; j < n; ++j) {
                    const R dx = xi[b] - px[j], dy = yi[b] - py[j], dz = zi[b] - pz[j];
                    if (dx * dx + dy * dy + dz * dz < a.rl2 && j != i) {
                        if (k < cap) list[(size_t)k * M + i] = (uint16_t)j;
                        ++k;
                    }
                }
                // padded to whole groups of four with the bead itself
                for (int q = k; q < ((k + 3) & ~3) && q < cap; ++q) list[(size_t)q * M + i] = (uint16_t)i;
                len[b] = k <= cap ? k : -1;
                rx[b] = xi[b];
                ry[b] = yi[b];
                rz[b] = zi[b];
            }
        }
        bool moved = false;
#pragma unroll
        for (int b = 0; b < BPT; ++b) {
            const int i = threadIdx.x + b * blockDim.x;
            if (i >= n) continue;
            const R x = xi[b], y = yi[b], z = zi[b];
            R sx, sy, sz;
            surface_point_near(x, y, z, ax, ay, az, t[b], sx, sy, sz);
            R fx = -a.k2 * (x - sx), fy = -a.k2 * (y - sy), fz = -a.k2 * (z - sz);
            auto pair = [&](int j) {
                const R dx = x - px[j], dy = y - py[j], dz = z - pz[j];
                const R r2 = dx * dx + dy * dy + dz * dz;
                if (r2 < a.rc2 && j != i) {
                    const R s2 = rdiv(a.sig2, r2);
                    const R s6 = s2 * s2 * s2;
                    const R fm = rdiv(a.eps24 * (R(2) * s6 * s6 - s6), r2);
                    fx += fm * dx;
                    fy += fm * dy;
                    fz += fm * dz;
                }
            };
            if (len[b] < 0) {
                for (int j = 0; j < n; ++j) pair(j);
            } else if constexpr (sizeof(R) == 8) {
                for (int k = 0; k < len[b]; ++k) pair(chk((int)list[(size_t)k * M + i], n, a.err));
            } else {
                // four at a time without a branch: their loads and divisions overlap
                for (int k = 0; k < len[b]; k += 4) {
                    R dx[4], dy[4], dz[4], fm[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int j = chk((int)list[(size_t)(k + q) * M + i], n, a.err);
                        dx[q] = x - px[j];
                        dy[q] = y - py[j];
                        dz[q] = z - pz[j];
                        const R r2 = dx[q] * dx[q] + dy[q] * dy[q] + dz[q] * dz[q];
                        const R ir2 = rdiv(R(1), r2), s2 = a.sig2 * ir2, s6 = s2 * s2 * s2;
                        fm[q] = r2 < a.rc2 && j != i ? a.eps24 * (R(2) * s6 * s6 - s6) * ir2 : R(0);
                    }
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        fx += fm[q] * dx[q];
                        fy += fm[q] * dy[q];
                        fz += fm[q] * dz[q];
                    }
                }
            }
            vx[b] = a.damp * vx[b] + a.dt * fx;
            vy[b] = a.damp * vy[b] + a.dt * fy;
            vz[b] = a.damp * vz[b] + a.dt * fz;
            xi[b] = x + a.dt * vx[b];
            yi[b] = y + a.dt * vy[b];
            zi[b] = z + a.dt * vz[b];
            nx[i] = xi[b];
            ny[i] = yi[b];
            nz[i] = zi[b];
            const R ux = xi[b] - rx[b], uy = yi[b] - ry[b], uz = zi[b] - rz[b];
            moved |= !(ux * ux + uy * uy + uz * uz < a.move2);
        }
        rebuild = __syncthreads_or(moved);   // the next step's positions are complete
    }
#pragma unroll
    for (int b = 0; b < BPT; ++b) {
        const int i = threadIdx.x + b * blockDim.x;
        if (i >= n) continue;
        R x = xi[b], y = yi[b], z = zi[b];
        if (a.project_final) surface_point(xi[b], yi[b], zi[b], ax, ay, az, x, y, z);
        X[3 * i] = (double)x;
        X[3 * i + 1] = (double)y;
        X[3 * i + 2] = (double)z;
    }
}

size_t list_smem(size_t rsize, int max_count) {
    return 6 * rsize * (size_t)max_count + sizeof(uint16_t) * kListLen * (size_t)max_count;
}

// The longest list to keep for a shell of n beads: a spherical cap of chord
// radius rl has the area pi rl^2, so n pi rl^2 / area beads lie within rl of an
// evenly spread bead, with 4 pi / 3 (ab + ac + bc) for the area (a sphere's; up
// to 15 % too small for a long ellipsoid); half as many again, and a few, for
// uneven spreads. A value of this shell alone: shells relaxed together are
// relaxed as each alone.
int list_rows(const double *a, int n, double sigma) {
    const double rl = (kWcaCut + LB_LIST_SKIN) * sigma;
    const double near = 0.75 * n * rl * rl / (a[0] * a[1] + a[0] * a[2] + a[1] * a[2]);
    if (n <= kListLen || !(near > kCrowded)) return kListLen;
    return (int)std::min((n + 3.0) / 4.0, 0.375 * near + 5.0) * 4;
}

template <typename R, int BPT, bool LONG>
cudaError_t launch_list_t(const ShellArgs<R> &a, const LongLists<LONG> &ll, int nshells, int threads, cudaStream_t s) {
    const size_t smem = LONG ? 6 * sizeof(R) * (size_t)a.max_count : list_smem(sizeof(R), a.max_count);
    cudaError_t e = cudaFuncSetAttribute(k_relax_list<R, BPT, LONG>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    k_relax_list<R, BPT, LONG><<<nshells, threads, smem, s>>>(a, ll);
    return cudaGetLastError();
}

template <typename R, bool LONG>
cudaError_t launch_list(const ShellArgs<R> &a, const LongLists<LONG> &ll, int bpt, int nshells, int threads,
                        cudaStream_t s) {
    if (bpt == 1) return launch_list_t<R, 1, LONG>(a, ll, nshells, threads, s);
    if (bpt == 2) return launch_list_t<R, 2, LONG>(a, ll, nshells, threads, s);
    return launch_list_t<R, 4, LONG>(a, ll, nshells, threads, s);
}

size_t shell_smem(size_t rsize, int max_count, int max_cells, bool cells) {
    return 6 * rsize * (size_t)max_count + (cells ? sizeof(int) * (2 * (size_t)max_count + 2 * (size_t)max_cells + 1) : 0);
}

template <typename R, int BPT, bool CELLS>
cudaError_t launch_shells_t(const ShellArgs<R> &a, int nshells, int threads, cudaStream_t s) {
    const size_t smem = shell_smem(sizeof(R), a.max_count, a.max_cells, CELLS);
    cudaError_t e = cudaFuncSetAttribute(k_relax_shells<R, BPT, CELLS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    k_relax_shells<R, BPT, CELLS><<<nshells, threads, smem, s>>>(a);
    return cudaGetLastError();
}

template <typename R>
cudaError_t launch_shells(ShellArgs<R> a, const lb_shell_params &p, int nshells, bool cells, bool lists,
                          const LongLists<true> &ll, cudaStream_t s) {
    a.k2 = (R)(2.0 * p.k_surface);
    a.sig2 = (R)(p.sigma * p.sigma);
    a.rc2 = (R)(kWcaCut * kWcaCut * p.sigma * p.sigma);
    a.eps24 = (R)(24.0 * p.epsilon);
    a.dt = (R)p.dt;
    a.damp = (R)(1.0 - p.eta * p.dt);
    a.steps = p.steps;
    a.project_final = p.project_final;
    // beads per thread: 1, 2 or 4; threads a multiple of the warp
    const int cap = lists ? list_threads<R>() : kShellThreads;
    const int bpt = a.max_count <= cap ? 1 : (a.max_count <= 2 * cap ? 2 : 4);
    int threads = (a.max_count + bpt - 1) / bpt;
    threads = ((threads + 31) / 32) * 32;
    if (lists) {
        // skin: 0.15 sigma (about 9 listed beads at one bead per unit area, a
        // few rebuilds in the first 1000 steps; 0.05 to 0.15 within 3 %, 2400
        // beads 22.8 / 16.6 / 14.8 us per step at 0.05 / 0.1 / 0.15); 0.98:
        // the margin of the rounding of distances and moves
        const double skin = LB_LIST_SKIN * p.sigma, rl = kWcaCut * p.sigma + skin;
        a.rl2 = (R)(rl * rl);
        a.move2 = (R)(0.98 * 0.25 * skin * skin);
        if (ll.list) return launch_list<R, true>(a, ll, bpt, nshells, threads, s);
        return launch_list<R, false>(a, {}, bpt, nshells, threads, s);
    }
    if (cells) {
        if (bpt == 1) return launch_shells_t<R, 1, true>(a, nshells, threads, s);
        if (bpt == 2) return launch_shells_t<R, 2, true>(a, nshells, threads, s);
        return launch_shells_t<R, 4, true>(a, nshells, threads, s);
    }
    if (bpt == 1) return launch_shells_t<R, 1, false>(a, nshells, threads, s);
    if (bpt == 2) return launch_shells_t<R, 2, false>(a, nshells, threads, s);
    return launch_shells_t<R, 4, false>(a, nshells, threads, s);
}

}  // namespace

}  // namespace lbk

extern "C" lb_status lb_relax_shells(int nshells, const double *axes, const int *counts, double *xyz,
                                     const lb_shell_params *p, void *cuda_stream, char *err, size_t err_len) {
    auto fail = [&](lb_status st, const std::string &m) {
        if (err && err_len) {
            std::strncpy(err, m.c_str(), err_len - 1);
            err[err_len - 1] = 0;
        }
        return st;
    };
    if (!axes || !counts || !xyz || !p) return fail(LB_ERR_ARG, "null pointer");
    if (nshells < 1 || nshells > 65535) return fail(LB_ERR_ARG, "nshells must be in [1, 65535]");
    if (p->precision != 32 && p->precision != 64) return fail(LB_ERR_ARG, "precision must be 32 or 64");
    if (!(p->k_surface > 0.0) || !(p->sigma > 0.0) || !(p->epsilon > 0.0) || !(p->dt > 0.0) || !(p->eta >= 0.0) ||
        !(p->eta * p->dt <= 2.0) || p->steps < 0 || !std::isfinite(p->k_surface) || !std::isfinite(p->sigma) ||
        !std::isfinite(p->epsilon) || !std::isfinite(p->dt) || !std::isfinite(p->eta))
        return fail(LB_ERR_ARG, "need k, sigma, epsilon, dt > 0, eta >= 0, eta dt <= 2 and steps >= 0");
    if (p->pair_search < 0 || p->pair_search > 2) return fail(LB_ERR_ARG, "pair_search must be 0, 1 or 2");
    std::vector<long long> off(nshells);
    long long total = 0;
    int max_count = 0;
    for (int s = 0; s < nshells; ++s) {
        if (counts[s] < 1 || counts[s] > LB_SHELL_MAX_BEADS)
            return fail(LB_ERR_ARG, "every shell needs 1 to LB_SHELL_MAX_BEADS (4096) beads");
        for (int q = 0; q < 3; ++q)
            if (!(axes[3 * s + q] > 0.0) || !std::isfinite(axes[3 * s + q]))
                return fail(LB_ERR_ARG, "semi-axes must be positive and finite");
        off[s] = total;
        total += counts[s];
        if (counts[s] > max_count) max_count = counts[s];
    }
    for (long long i = 0; i < 3 * total; ++i)
        if (!std::isfinite(xyz[i])) return fail(LB_ERR_ARG, "initial positions must be finite");

    // cell grids: per axis the box [-L, L), L = 1.25 a + 1, cut into cells at
    // least as wide as the WCA range, at most kMaxCells cells per shell
    const double rc = lbk::kWcaCut * p->sigma;
    std::vector<int> grid((size_t)3 * nshells);
    std::vector<double> box((size_t)3 * nshells);
    int max_cells = 1;
    for (int s = 0; s < nshells; ++s) {
        long long g[3];
        for (int q = 0; q < 3; ++q) {
            box[3 * s + q] = 1.25 * axes[3 * s + q] + 1.0;
            g[q] = std::max(1LL, (long long)std::floor(2.0 * box[3 * s + q] / rc));
            g[q] = std::min(g[q], 4096LL);
        }
        while (g[0] * g[1] * g[2] > lbk::kMaxCells) {
            const int q = g[0] >= g[1] && g[0] >= g[2] ? 0 : (g[1] >= g[2] ? 1 : 2);
            g[q] = std::max(1LL, (g[q] * 7) / 8);
        }
        for (int q = 0; q < 3; ++q) grid[3 * s + q] = (int)g[q];
        max_cells = std::max(max_cells, (int)(g[0] * g[1] * g[2]));
    }
    const size_t rsize = p->precision == 64 ? sizeof(double) : sizeof(float);
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return fail(LB_ERR_CUDA, std::string("device query: ") + cudaGetErrorString(e));
    const bool cells_fit = lbk::shell_smem(rsize, max_count, max_cells, true) <= (size_t)optin;
    if (p->pair_search == 2 && !cells_fit)
        return fail(LB_ERR_ARG, "the cell list does not fit in shared memory for this shell size and precision");
    if (lbk::shell_smem(rsize, max_count, 1, false) > (size_t)optin)
        return fail(LB_ERR_ARG, "the shell does not fit in shared memory at this precision");
    // automatic: neighbour lists wherever they fit (4 beads a thread at most);
    // the larger shells (2048 beads in FP64, about 2640 in FP32 and more) take
    // the cell list when it fits, 4 times faster there than all pairs
    const int list_cap = 4 * (p->precision == 64 ? lbk::list_threads<double>() : lbk::list_threads<float>());
    const bool lists = p->pair_search == 0 && max_count <= list_cap && lbk::list_smem(rsize, max_count) <= (size_t)optin;
    const bool cells = p->pair_search == 2 || (p->pair_search == 0 && !lists && cells_fit);

    // longer lists where a shell is crowded (without them, as without their
    // memory: lists of kListLen)
    std::vector<int> rows(nshells, lbk::kListLen);
    int max_rows = lbk::kListLen;
    if (lists)
        for (int s = 0; s < nshells; ++s) {
            rows[s] = lbk::list_rows(axes + 3 * s, counts[s], p->sigma);
            max_rows = std::max(max_rows, rows[s]);
        }
    const size_t long_bytes = sizeof(uint16_t) * (size_t)nshells * max_rows * max_count;
    bool longer = max_rows > lbk::kListLen && long_bytes <= lbk::kLongBytes;

    cudaStream_t st = (cudaStream_t)cuda_stream;
    const size_t nd = (size_t)3 * nshells + (size_t)3 * total + (size_t)3 * nshells;
    const size_t bytes = nd * sizeof(double) + (size_t)nshells * (sizeof(long long) + sizeof(int) + 4 * sizeof(int)) +
                         sizeof(int);
    void *d = nullptr;
    e = cudaMalloc(&d, bytes + (longer ? long_bytes : 0));
    if (e == cudaErrorMemoryAllocation && longer) {
        cudaGetLastError();
        longer = false;
        e = cudaMalloc(&d, bytes);
    }
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        return fail(LB_ERR_OOM, "device allocation for the shells failed");
    }
    if (e != cudaSuccess) return fail(LB_ERR_CUDA, std::string("cudaMalloc: ") + cudaGetErrorString(e));
    double *daxes = static_cast<double *>(d), *dxyz = daxes + 3 * nshells, *dbox = dxyz + 3 * total;
    long long *doff = reinterpret_cast<long long *>(dbox + 3 * nshells);
    int *dcount = reinterpret_cast<int *>(doff + nshells);
    int *dgrid = dcount + nshells;
    int *drows = dgrid + 3 * nshells;
    int *derr = drows + nshells;                 // index checks of checked builds
    uint16_t *dlong = longer ? reinterpret_cast<uint16_t *>(derr + 1) : nullptr;
    std::vector<double> out((size_t)3 * total);
    e = cudaMemcpyAsync(daxes, axes, 3 * nshells * sizeof(double), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(dxyz, xyz, 3 * total * sizeof(double), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(doff, off.data(), nshells * sizeof(long long), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(dcount, counts, nshells * sizeof(int), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(dbox, box.data(), 3 * nshells * sizeof(double), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(dgrid, grid.data(), 3 * nshells * sizeof(int), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess && longer)
        e = cudaMemcpyAsync(drows, rows.data(), nshells * sizeof(int), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(derr, 0, sizeof(int), st);
    if (e == cudaSuccess) {
        if (p->precision == 64) {
            lbk::ShellArgs<double> a{};
            a.axes = daxes; a.count = dcount; a.offset = doff; a.xyz = dxyz; a.max_count = max_count;
            a.cgrid = dgrid; a.cbox = dbox; a.max_cells = cells ? max_cells : 1; a.err = derr;
            e = lbk::launch_shells<double>(a, *p, nshells, cells, lists, {dlong, drows, max_rows}, st);
        } else {
            lbk::ShellArgs<float> a{};
            a.axes = daxes; a.count = dcount; a.offset = doff; a.xyz = dxyz; a.max_count = max_count;
            a.cgrid = dgrid; a.cbox = dbox; a.max_cells = cells ? max_cells : 1; a.err = derr;
            e = lbk::launch_shells<float>(a, *p, nshells, cells, lists, {dlong, drows, max_rows}, st);
        }
    }
    int herr = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(out.data(), dxyz, 3 * total * sizeof(double), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&herr, derr, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaFree(d);
    if (e != cudaSuccess) return fail(LB_ERR_CUDA, std::string("lb_relax_shells: ") + cudaGetErrorString(e));
    if (herr) return fail(LB_ERR_STATE, "an index check of the checked build failed (an index outside its array)");
    for (double v : out)
        if (!std::isfinite(v)) return fail(LB_ERR_UNSTABLE, "non-finite bead position: reduce dt or k");
    std::memcpy(xyz, out.data(), out.size() * sizeof(double));
    return LB_OK;
}
