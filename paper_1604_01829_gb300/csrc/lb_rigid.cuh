// Rigid raspberry bodies (Ustach & Faller, arXiv:1604.01829, Sec. 1.2 and
// Sec. 2.3): quaternion rotation, velocity-Verlet half kicks and drift. One
// warp per body, FP64; shared by the single-lattice and batched paths.
#pragma once

#include "lb_internal.h"

namespace lbk {

__device__ __forceinline__ void cross3(const double a[3], const double b[3], double o[3]) {
    o[0] = a[1] * b[2] - a[2] * b[1];
    o[1] = a[2] * b[0] - a[0] * b[2];
    o[2] = a[0] * b[1] - a[1] * b[0];
}

// lab = R body, Hamilton convention, q = (w, x, y, z)
__device__ __forceinline__ void quat_to_R(const double q[4], double R[9]) {
    const double w = q[0], x = q[1], y = q[2], z = q[3];
    R[0] = 1.0 - 2.0 * (y * y + z * z); R[1] = 2.0 * (x * y - z * w); R[2] = 2.0 * (x * z + y * w);
    R[3] = 2.0 * (x * y + z * w); R[4] = 1.0 - 2.0 * (x * x + z * z); R[5] = 2.0 * (y * z - x * w);
    R[6] = 2.0 * (x * z - y * w); R[7] = 2.0 * (y * z + x * w); R[8] = 1.0 - 2.0 * (x * x + y * y);
}

// entry (i, j) of quat_to_R
__device__ __forceinline__ double rot_entry(double qw, double qx, double qy, double qz, int i, int j) {
    if (i == j) {
        const double u = i == 0 ? qy : qx, v = i == 2 ? qy : qz;
        return 1.0 - 2.0 * (u * u + v * v);
    }
    const double u = i == 0 || j == 0 ? qx : qy, v = i == 2 || j == 2 ? qz : qy;
    const double o = i + j == 1 ? qz : (i + j == 2 ? qy : qx);              // the third axis
    const bool neg = j == i + 1 || (i == 2 && j == 0);                      // -w o for (0,1), (1,2), (2,0)
    return 2.0 * (u * v + (neg ? -(o * qw) : o * qw));
}

// One body's update by one warp: the second half kick of the (sub)step that
// has its coupling done (FINISH) and / or the first half kick and drift of the
// next (START), over dt (1 without MD substeps, 1/n with n per LB step). snap:
// receives what the adjoint reads of the body's state between the two.
//
// Second half kick: totals F = beads + external and torque, V += dt F/(2M),
// body-frame omega implicitly (6 fixed-point iterations), so that the two half
// kicks around a step boundary form the trapezoidal rule of Euler's equations
// I dw/dt = T - w x (I w): a second-order, time-symmetric rotation update like
// the velocity-Verlet rotation schemes of Sec. 2.3. First half kick with the
// last totals, omega explicitly, then X += dt V, q <- q (x) exp(omega dt / 2)
// with the half-step omega, normalised.
//
// The update lies on every step's critical path and is a chain of FP64
// instructions of ~50 clocks each (2 FP64 lanes per SM): lanes a = 0, 1, 2 of
// the warp carry the components (the others repeat them), lanes 0-3 the
// quaternion, 0-8 the rotation matrix, with the others' values by shuffles;
// no division, square root or sincos in the usual case (a rotation below
// 1 rad per step, a quaternion near unit length: power series, else the
// functions). ~60 dependent FP64 instructions instead of the ~450 of one
// thread. Measured on GB300 (ncu): the update
// between MD substeps 13.8 -> 6.2 us, the step prologue of a free body 14.0
// -> 8.1 us, the group's end 8.0 -> 4.2 us; steps: 48 x 48 x 96 pore with two
// substeps 54 -> 40 us, 64 boxes of 24^3 60 -> 47 us.
template <bool FINISH, bool START>
__device__ __forceinline__ void body_update(Body *B, int lane, double dt, const double *ext, int b, int nb,
                                            const Recorder &rec, Body *snap = nullptr) {
    constexpr unsigned FULL = 0xffffffffu;
    auto from = [&](double v, int src) { return __shfl_sync(FULL, v, src); };
    const int a = lane % 3, a1 = a == 2 ? 0 : a + 1, a2 = a == 0 ? 2 : a - 1;
    const int fixed = B->fixed;
    const double inv_mass = B->inv_mass, iI = B->inv_I[a], dI = B->I[a2] - B->I[a1];
    double V = B->V[a], w = B->w[a], Fl, Tl;
    if (FINISH) {
        const double F = B->acc[a] + B->F_ext[a], T = B->acc[3 + a] + B->T_ext[a];
        const double Tb = B->R[a] * from(T, 0) + B->R[3 + a] * from(T, 1) + B->R[6 + a] * from(T, 2);
        if (lane < 3) {
            B->F_tot[a] = F;
            B->T_tot[a] = T;
            B->F_last[a] = F;
            B->T_last[a] = Tb;
        }
        Fl = F;
        Tl = Tb;
        if (fixed != 1) V += 0.5 * dt * F * inv_mass;
        if (fixed == 0) {
            // w_a = w0_a + (dt / 2 I_a) (T_a - (I_a2 - I_a1) w_a1 w_a2)
            const double h = 0.5 * dt * iI, g = w + h * Tb, e = h * dI;
            for (int it = 0; it < 6; ++it) w = g - e * (from(w, a1) * from(w, a2));
        }
    } else {
        Fl = B->F_last[a];
        Tl = B->T_last[a];
    }
    if (!START) {
        if (lane < 3) {
            B->V[a] = V;
            B->w[a] = w;
        }
        return;
    }
    if (ext && lane < 3) {              // this step's external force and torque (host-written, mapped)
        B->F_ext[a] = ext[3 * b + a];
        B->T_ext[a] = ext[3 * nb + 3 * b + a];
    }
    double X = B->X[a], q = B->q[lane & 3];
    if (snap) {
        if (lane < 3) {
            snap->X[a] = X;
            snap->V[a] = V;
            snap->w[a] = w;
            snap->F_last[a] = Fl;
        }
        if (lane < 4) snap->q[lane] = q;
        if (lane == 0) {
            snap->mass = B->mass;
            snap->inv_mass = inv_mass;
            snap->fixed = fixed;
        }
    }
    if (fixed != 1) {
        V += 0.5 * dt * Fl * inv_mass;
        X += dt * V;
    }
    if (fixed == 2) w = 0.0;
    if (fixed == 0) {
        w += 0.5 * dt * iI * (Tl - dI * (from(w, a1) * from(w, a2)));
        const double w0 = from(w, 0), w1 = from(w, 1), w2 = from(w, 2);
        const double wn2 = w0 * w0 + w1 * w1 + w2 * w2;
        const double h2 = 0.25 * dt * dt * wn2;            // squared half angle
        double ch, sh;                                     // cos h and sin h / |w|
        if (h2 < 0.25) {
            // sin h / h and cos h by their Taylor series (next terms below 1e-18)
            double s = 1.0 / 355687428096000.0, c = 1.0 / 20922789888000.0;
            s = fma(s, -h2, 1.0 / 1307674368000.0);  c = fma(c, -h2, 1.0 / 87178291200.0);
            s = fma(s, -h2, 1.0 / 6227020800.0);     c = fma(c, -h2, 1.0 / 479001600.0);
            s = fma(s, -h2, 1.0 / 39916800.0);       c = fma(c, -h2, 1.0 / 3628800.0);
            s = fma(s, -h2, 1.0 / 362880.0);         c = fma(c, -h2, 1.0 / 40320.0);
            s = fma(s, -h2, 1.0 / 5040.0);           c = fma(c, -h2, 1.0 / 720.0);
            s = fma(s, -h2, 1.0 / 120.0);            c = fma(c, -h2, 1.0 / 24.0);
            s = fma(s, -h2, 1.0 / 6.0);              c = fma(c, -h2, 0.5);
            s = fma(s, -h2, 1.0);                    c = fma(c, -h2, 1.0);
            ch = c;
            sh = s * (0.5 * dt);
        } else {
            const double wn = sqrt(wn2);
            sincos(0.5 * wn * dt, &sh, &ch);
            sh /= wn;
        }
        // Hamilton product q (x) (ch, sh w), component `lane & 3`
        const double q0 = from(q, 0), q1 = from(q, 1), q2 = from(q, 2), q3 = from(q, 3);
        const double d1 = sh * w0, d2 = sh * w1, d3 = sh * w2;
        const int c4 = lane & 3;
        const double x = c4 == 0 ? -q1 : (c4 == 1 ? q0 : (c4 == 2 ? q3 : -q2));
        const double y = c4 == 0 ? -q2 : (c4 == 1 ? -q3 : (c4 == 2 ? q0 : q1));
        const double z = c4 == 0 ? -q3 : (c4 == 1 ? q2 : (c4 == 2 ? -q1 : q0));
        q = q * ch + x * d1 + y * d2 + z * d3;
        // 1 / |q|: |q|^2 = 1 + e, e of rounding size
        const double r0 = from(q, 0), r1 = from(q, 1), r2 = from(q, 2), r3 = from(q, 3);
        const double n2 = r0 * r0 + r1 * r1 + r2 * r2 + r3 * r3, e = n2 - 1.0;
        double inv;
        if (fabs(e) < 0x1p-11)
            inv = fma(e, fma(e, fma(e, fma(e, 35.0 / 128.0, -5.0 / 16.0), 0.375), -0.5), 1.0);
        else
            inv = rsqrt(n2);
        q *= inv;
    }
    // rotation, lab = R body: R_ij of lane 3 i + j
    const double qw = from(q, 0), qx = from(q, 1), qy = from(q, 2), qz = from(q, 3);
    const int l9 = lane < 9 ? lane : 0, i = l9 / 3, j = l9 - 3 * i;
    const double R = rot_entry(qw, qx, qy, qz, i, j);
    const double Rw = R * from(w, j);                       // lab omega: row sums of R_ij w_j
    const double wl = from(Rw, 3 * a) + from(Rw, 3 * a + 1) + from(Rw, 3 * a + 2);
    if (lane < 9) {
        B->R[lane] = R;
        B->Rf[lane] = (float)R;
    }
    if (lane < 6) B->acc[lane] = 0.0;
    if (lane < 4) B->q[lane] = q;
    if (lane < 3) {
        B->V[a] = V;
        B->X[a] = X;
        B->w[a] = w;
        B->wl[a] = wl;
        B->Vf[a] = (float)V;
        B->wlf[a] = (float)wl;
        const double h = X - 0.5, fl = floor(h);
        B->Xi[a] = (int)fl;
        B->Xf[a] = (float)(h - fl);
    }
    // trajectory record after the drift of step *step_base + step_off
    if (rec.ring) {
        const unsigned long long t1 = *rec.step_base + rec.step_off + 1ull;
        if (t1 % (unsigned long long)rec.every == 0) {
            const unsigned long long slot = (t1 / (unsigned long long)rec.every - 1ull) % (unsigned long long)rec.cap;
            double *o = rec.ring + (slot * (unsigned long long)nb + (unsigned long long)b) * 7ull;
            if (lane < 3) o[lane] = X;
            if (lane < 4) o[3 + lane] = q;
        }
    }
}

// The list of flagged tiles restarts empty once every block of the clearing
// kernel has read its length: the last block to arrive (count[1] is the
// ticket, left at 0) resets it, in place of a memset node in the step's chain
// (48 x 48 x 96 pore with two substeps 37 -> 28 us per step, 64^3 23 -> 17).
__device__ __forceinline__ void restart_list(int *count, int blocks) {
    __syncthreads();
    if (threadIdx.x != 0 || threadIdx.y != 0) return;
    __threadfence();
    if (atomicAdd(count + 1, 1) == blocks - 1) {
        count[0] = 0;
        count[1] = 0;
    }
}

// The end of a group of steps for body b (one warp): its second half kick and,
// with `out` (host-mapped), its totals (6 a body) and X, V, q, w (13 a body,
// after the totals and the error word); each lane writes what it holds itself.
__device__ __forceinline__ void finish_body(Body *bodies, int b, int nb, int lane, double dt, double *out) {
    const Recorder none{};
    body_update<true, false>(bodies + b, lane, dt, nullptr, b, nb, none);
    if (!out) return;
    const Body &B = bodies[b];           // X and q are the prologue's, the rest this lane's own
    double *st = out + 6 * nb + 1 + 13 * b;
    if (lane < 3) {
        out[6 * b + lane] = B.F_tot[lane];
        out[6 * b + 3 + lane] = B.T_tot[lane];
        st[lane] = B.X[lane];
        st[3 + lane] = B.V[lane];
        st[10 + lane] = B.w[lane];
    }
    if (lane < 4) st[6 + lane] = B.q[lane];
}

// Zeroes the force on the nodes of the listed tiles and drops their flags:
// thread t of n, one (tile, node of the tile) at a time.
template <typename T>
__device__ __forceinline__ void clear_tiles(const Geom &g, T *F, int *tiles, const int *tlist, const int *tcount,
                                            int ntx, int nty, long long t, long long n) {
    const long long total = 64LL * (*tcount);
    for (long long i = t; i < total; i += n) {
        const int tile = tlist[i >> 6];
        const int l = (int)(i & 63);
        const int tx = tile % ntx, ty = (tile / ntx) % nty, tz = tile / (ntx * nty);
        const int x = 4 * tx + (l & 3), y = 4 * ty + ((l >> 2) & 3), z = 4 * tz + (l >> 4);
        if (x < g.nx && y < g.ny && z < g.nz) {
            const long long m = nidx(g, x, y, z);
            F[m] = T(0);
            F[g.N + m] = T(0);
            F[2 * g.N + m] = T(0);
        }
        if (l == 0) tiles[tile] = 0;
    }
}

// Extra block eb of a chained fluid kernel (StepExtra).
template <typename T>
__device__ __noinline__ void step_extra(const StepExtra &e, const Geom &g, int eb) {
    const int n = blockDim.x * blockDim.y, t = threadIdx.x + blockDim.x * threadIdx.y;
    const int lane = t & 31, warp = t >> 5, warps = n >> 5;
    if (eb < e.body_blocks) {
        for (int b = eb + e.body_blocks * warp; b < e.nb; b += e.body_blocks * warps) {
            if (e.mode == 1) body_update<true, true>(e.bodies + b, lane, e.dt, e.ext, b, e.nb, e.rec);
            else finish_body(e.bodies, b, e.nb, lane, e.dt, e.out);
        }
        if (e.mode == 2 && eb == 0 && t == 0) {
            *e.step += e.by;
            if (e.out) e.out[6 * e.nb] = e.err ? (double)*e.err : 0.0;
        }
    } else {                                   // mode 1
        const int blocks = e.blocks - e.body_blocks;
        clear_tiles(g, static_cast<T *>(e.F), e.tiles, e.tlist, e.tcount, e.ntx, e.nty,
                    (long long)(eb - e.body_blocks) * n + t, (long long)blocks * n);
        restart_list(e.tcount, blocks);
    }
}

}  // namespace lbk
