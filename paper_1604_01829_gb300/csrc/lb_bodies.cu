// Raspberry kernels (Ustach & Faller, arXiv:1604.01829):
//  - rigid-body integration of the centre of mass by velocity Verlet and of
//    the orientation by a quaternion (Sec. 2.3), one warp per body in FP64;
//  - virtual sites r_b = X + R(q) s_b, v_b = V + omega x (r_b - X) (Sec. 1.2);
//  - friction coupling F_b = -gamma (v_b - u(r_b)) + f_s, Eq.
//    (latticeboltzmannfriction) in Sec. 1.1, with u trilinearly interpolated
//    from the 8 surrounding nodes and -F_b spread back onto the same nodes
//    with the same weights, so the exchange conserves momentum; bead forces
//    and torques summed onto the body (Sec. 2.3).
#include "lb_couple.cuh"

namespace lbk {

namespace {

// Step prologue in one launch: warp 0 of blocks [0, nb) finishes the
// previous step's body (second half kick) if asked and starts this step's
// (half kick, drift, rotation); every thread also clears nodes of the
// flagged 4x4x4 tiles of this step's spread-force buffer.
template <typename T>
__global__ void k_step_pre(Body *bodies, int nb, int finish_prev, T *F, int *tiles, const int *tlist,
                           int *tcount, Geom g, int ntx, int nty, Recorder rec, double dt, const double *ext, Body *snap,
                           unsigned long long *step) {
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    // one body per block, so the FP64 work of the bodies spreads over SMs
    if (threadIdx.x < 32 && blockIdx.x < nb) {
        Body *B = bodies + blockIdx.x;
        Body *sn = snap ? snap + blockIdx.x : nullptr;
        if (finish_prev) body_update<true, true>(B, threadIdx.x, dt, ext, blockIdx.x, nb, rec, sn);
        else body_update<false, true>(B, threadIdx.x, dt, ext, blockIdx.x, nb, rec, sn);
    }
    if (step && blockIdx.x == 0 && threadIdx.x == 0) step[1] = step[0];
    if (!tiles) return;
    clear_tiles(g, F, tiles, tlist, tcount, ntx, nty, t, (long long)gridDim.x * blockDim.x);
    restart_list(tcount, gridDim.x);
}

// The end of a group of steps in one launch: the last step's second half
// kick (one body per block) and the advance of the device step counter;
// with `out` (host-mapped) also every body's force and torque totals (6 a
// body), the device error word and every body's X, V, q, w (13 a body), so
// the host reads them without a copy.
__global__ void k_finish(Body *bodies, int nb, double dt, unsigned long long *step, unsigned int by, double *out,
                         const int *err) {
    const int b = blockIdx.x, lane = threadIdx.x;
    if (b < nb) finish_body(bodies, b, nb, lane, dt, out);
    if (b == 0 && lane == 0) {
        *step += by;
        if (out) out[6 * nb] = err ? (double)*err : 0.0;
    }
}

__global__ void k_error_word(double *out, const int *err) { *out = (double)*err; }

// Between two MD substeps of one LB step: the finished substep's second half
// kick, the next substep's first half kick and drift (and the trajectory
// record after the last substep's drift).
__global__ void k_substep(Body *bodies, int nb, double dt, Recorder rec) {
    const int b = blockIdx.x;
    if (b < nb) body_update<true, true>(bodies + b, threadIdx.x, dt, nullptr, b, nb, rec);
}

// threads per block of the body prologue when it runs beside a fluid kernel
#ifndef LB_PRE_BLOCK
#define LB_PRE_BLOCK 256
#endif

// register cap of the FP32 coupling kernel (resident CTAs of 128 per SM:
// 65536 / (128 x cap))
#ifndef LB_COUPLE_REGS
#define LB_COUPLE_REGS 64
#endif
template <typename T>
__global__ void __launch_bounds__(128) __maxnreg__(sizeof(T) == 4 ? LB_COUPLE_REGS : 255) k_couple(const __grid_constant__ CoupleArgs a) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int k = t >> 3;
    couple_bead<T>(a, k, k, t & 7, threadIdx.x & 31, k < a.nbeads);
    if (a.wall.on && k < a.nbeads)
        couple_wall(a.wall, a.bodies, chk(a.bead_body[k], a.nbodies, a.err), a.s, k, t & 7);
}

}  // namespace

int sm_count() {
    static const int sms = [] {     // initialised once, thread-safe
        int dev = 0, n = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) !=
                                                      cudaSuccess || n <= 0)
            n = 152;
        return n;
    }();
    return sms;
}

int couple_block(int nbeads) { return nbeads <= 16 * sm_count() ? 32 : 128; }

cudaError_t launch_step_pre(Body *b, int nbodies, bool finish_prev, void *F, bool fp32, int *tiles, const int *tlist,
                            int *tcount, int list_cap, const Geom &g, int ntx, int nty, const Recorder &rec,
                            cudaStream_t s, double dt, const double *ext, bool alone, Body *snap,
                            unsigned long long *step) {
    // one block per body, and for the tile clearing (grid-stride) at most a
    // quarter of the SMs' worth of blocks when the kernel runs beside the
    // fluid kernel of the previous step, whose blocks it would otherwise
    // displace (measured on GB300 at 256^3 with 64 bodies: fluid kernel
    // 0.4372 ms against 0.4392 with a full-GPU grid, the step 0.4620 against
    // 0.4641); 8 blocks per SM when nothing runs beside it (the first step of
    // a group, e.g. every step of a one-step-per-call control loop)
    const int sms = sm_count();
    long long n = 64LL * list_cap;
    const int bs = alone ? 256 : LB_PRE_BLOCK;
    const long long cap = (alone ? 8LL * sms : (long long)(sms + 3) / 4) * bs;
    if (n > cap) n = cap;
    unsigned grid = (unsigned)((n + bs - 1) / bs);
    if (grid < (unsigned)nbodies) grid = (unsigned)nbodies;
    if (fp32) k_step_pre<float><<<grid, bs, 0, s>>>(b, nbodies, finish_prev ? 1 : 0, (float *)F, tiles, tlist, tcount, g, ntx, nty, rec, dt, ext, snap, step);
    else k_step_pre<double><<<grid, bs, 0, s>>>(b, nbodies, finish_prev ? 1 : 0, (double *)F, tiles, tlist, tcount, g, ntx, nty, rec, dt, ext, snap, step);
    return cudaGetLastError();
}

cudaError_t launch_couple(const CoupleArgs &a, cudaStream_t s) {
    if (a.nbeads <= 0) return cudaSuccess;
    const int block = couple_block(a.nbeads);
    const unsigned grid = (unsigned)((8LL * a.nbeads + block - 1) / block);
    if (a.fp32) k_couple<float><<<grid, block, 0, s>>>(a);
    else k_couple<double><<<grid, block, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_finish(Body *b, int nbodies, double dt, unsigned long long *step, unsigned int by, cudaStream_t s,
                          double *out, const int *err) {
    k_finish<<<nbodies > 0 ? nbodies : 1, 32, 0, s>>>(b, nbodies > 0 ? nbodies : 0, dt, step, by, out, err);
    return cudaGetLastError();
}

cudaError_t launch_error_word(double *out, const int *err, cudaStream_t s) {
    k_error_word<<<1, 1, 0, s>>>(out, err);
    return cudaGetLastError();
}

cudaError_t launch_substep(Body *b, int nbodies, double dt, const Recorder &rec, cudaStream_t s) {
    if (nbodies <= 0) return cudaSuccess;
    k_substep<<<nbodies, 32, 0, s>>>(b, nbodies, dt, rec);
    return cudaGetLastError();
}

}  // namespace lbk
