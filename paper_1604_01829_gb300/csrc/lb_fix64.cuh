// The FP64 collision of one node in 64-bit fixed point.
//
// GB300 issues FP64 at 2 lanes per SM and clock, 64 times fewer than FP32 and
// 32-bit integer work, so the FP64 collide-and-stream kernel was bound by its
// ~300 FP64 instructions per node, an order of magnitude above its memory
// time. Here the same collision (lb_collide.cuh: the MRT moments, equilibrium,
// Guo source and noise; BGK is MRT with all rates equal) runs on the integer
// pipes: populations become 64-bit integers at 2^-61 of a power of two near
// rho0, the moments and the way back are exact integer sums, products keep the
// top 64 of 128 bits with rounding, and only the results are rounded to
// doubles (to nearest even). The conserved moments are not recomputed: a
// population changes by the relaxation of the 15 other moments and by its
// share of the force, so mass is exact before the final rounding.
//
// Error against the same runs in 80-bit arithmetic, this form and the FP64
// evaluation: populations (rms, in units of rho0) 1.4e-17 and 2.9e-15 after 200
// steps of a pulled sphere in 32^3, 1.4e-17 and 1.4e-15 after 100 in a driven
// 48 x 48 x 96 pore, 1.5e-17 and 6e-16 after 50 with noise; momentum of a pore
// driven by 1e-6 for 2000 steps 5e-14 and 1.2e-12 relative, by 1e-8 3e-12 and
// 9e-11 (the share of the force is rounded to 2^-61, for a node always the same
// way; FP64 rounds the sums that it is added to at 2^-58).
//
// Range: with rho0 scaled into [2/3, 4/3) the inputs must satisfy
// |f_0| < 1/2, |f_1..6| < 1/8, |f_7..18| < 1/16 (about twice the values at
// rest and below a flow speed of 0.3), rho > 1/4, |u| < 1/2, |F| < 1/2. Then
// every sum below stays under 4 and every post-collision population under 2
// (|m_k| <= 2.75; rows of the relaxation operator over all rates: 1.75 rest,
// 0.89 axis, 0.75 diagonal). collide_fix() returns false for any other node
// (also infinities and NaN) and the caller takes the FP64 evaluation.
#pragma once

#include <cmath>

#include "lb_collide.cuh"

namespace lbk {

#ifdef __CUDACC__
#define LB_FIX_FN __host__ __device__ __forceinline__
#else
#define LB_FIX_FN inline
#endif

// v = h 2^32 + l, l signed; v below 2^63 - 2^31 (from there on h would be 2^31)
LB_FIX_FN FixPair fix_split(long long v) {
    FixPair p;
    p.l = (int)v;
    p.h = (int)(v >> 32) - (p.l >> 31);
    return p;
}

// a b / 2^64, rounded; the low halves' product is left out (below 1/4)
LB_FIX_FN long long fix_mul(FixPair a, FixPair b) {
    long long t = (long long)a.h * b.l + 0x80000000LL;
    t = (long long)a.l * b.h + t;
    return (long long)a.h * b.h + (t >> 32);
}

LB_FIX_FN unsigned fix_clz(unsigned v) {
#ifdef __CUDA_ARCH__
    return (unsigned)__clz((int)v);
#else
    return v ? (unsigned)__builtin_clz(v) : 32u;
#endif
}

LB_FIX_FN unsigned long long fix_shr(unsigned long long v, int r) {
#ifdef __CUDA_ARCH__
    unsigned long long o;           // PTX clamps the shift: 0 from 64 on
    asm("shr.u64 %0, %1, %2;" : "=l"(o) : "l"(v), "r"(r));
    return o;
#else
    return (unsigned)r > 63u ? 0ull : v >> r;
#endif
}

LB_FIX_FN long long fix_bits(double v) {
#ifdef __CUDA_ARCH__
    return __double_as_longlong(v);
#else
    long long o;
    __builtin_memcpy(&o, &v, 8);
    return o;
#endif
}

LB_FIX_FN double fix_double(unsigned long long b) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)b);
#else
    double o;
    __builtin_memcpy(&o, &b, 8);
    return o;
#endif
}

// v 2^61 (of the scaled unit) of a double below 2^-B in magnitude, B >= 1:
// exact down to 2^-9, truncated below that. over: the sign bit is set when
// |v| >= 2^-B. cb = 1023 + k, k the exponent of the scaled unit.
template <int B>
LB_FIX_FN long long fix_in(double v, int cb, int &over) {
    const unsigned long long b = (unsigned long long)fix_bits(v);
    const unsigned hi = (unsigned)(b >> 32), lo = (unsigned)b;
    const int r = cb - 1 - B - (int)((hi >> 20) & 0x7FFu);
    over |= r;
    const unsigned mh = (hi & 0xFFFFFu) | 0x100000u;
    // mantissa at bit 52; the largest exponent allowed, -1 - B, puts it at bit 60 - B
    const unsigned long long m = (((unsigned long long)mh << 32) | lo) << (8 - B);
    const long long s = (long long)fix_shr(m, r);
    return (int)hi < 0 ? -s : s;
}

// The double nearest (even) to V 2^(k - 61), |V| < 2^62, by integer
// instructions (~18): shift to bit 62, round, shift back. small: the smallest
// upper half of |V| seen; 0: a value is too small for this form.
LB_FIX_FN double fix_out(long long V, const FixParams &P, unsigned &small) {
    const unsigned sgn = (unsigned)((unsigned long long)V >> 32) & 0x80000000u;
    const unsigned long long A = (unsigned long long)(V < 0 ? -V : V);
    const unsigned ah = (unsigned)(A >> 32);
    small = small < ah ? small : ah;
    const unsigned n = fix_clz(ah | 1u) - 1u;
    const unsigned long long w = A << n;
    const unsigned long long m = (w + (0x1FFu + (((unsigned)w >> 10) & 1u))) >> 10;
    const unsigned h = (unsigned)(m >> 32) + (unsigned)P.ce - (n << 20) + sgn;
    return fix_double(((unsigned long long)h << 32) | (unsigned)m);
}

// The same by two additions on the FP64 pipe: the halves of V + 2^63 as the
// low words of two doubles of fixed exponents, (2^84 + 2^32 (hi + 2^31)) and
// (2^52 + lo) times 2^(k - 61); what was added is taken from the first
// (exactly), and only the sum rounds. With every output by one form its pipe
// is the bound (integer 65 % busy, or FP64 75 %): LB_FIX_OUT64 of the 19 take
// this one.
LB_FIX_FN double fix_out64(long long V, const FixParams &P) {
    const unsigned hi = (unsigned)((unsigned long long)V >> 32) ^ 0x80000000u, lo = (unsigned)V;
    const double a = fix_double(((unsigned long long)(unsigned)P.eh << 32) | hi);
    const double b = fix_double(((unsigned long long)(unsigned)P.el << 32) | lo);
    return (a - P.out) + b;
}
#ifndef LB_FIX_OUT64
#define LB_FIX_OUT64 7
#endif

#ifdef __CUDACC__
LB_FIX_FN float fix_rcp(float x) {
#ifdef __CUDA_ARCH__
    return __fdividef(1.0f, x);
#else
    return 1.0f / x;
#endif
}
LB_FIX_FN float fix_rsqrt(float x) {
#ifdef __CUDA_ARCH__
    return rsqrtf(x);
#else
    return 1.0f / sqrtf(x);
#endif
}
#else
LB_FIX_FN float fix_rcp(float x) { return 1.0f / x; }
LB_FIX_FN float fix_rsqrt(float x) { return 1.0f / std::sqrt(x); }
#endif

// 1/rho at 2^61 of rho at 2^61, rho in (1/4, 2): a 23-bit estimate corrected
// by two terms of its geometric series (relative error below 2^-57)
LB_FIX_FN long long fix_reciprocal(long long rho) {
    const unsigned rh = (unsigned)(rho >> 32), rl = (unsigned)rho;       // rho = rh 2^-29
    const unsigned r0 = (unsigned)(fix_rcp((float)rh) * 0x1p58f);        // 1/rho at 2^29
    // e = 1 - rho r0 at 2^58, |e| < 2^-21
    const long long p = (long long)((unsigned long long)rh * r0 + (((unsigned long long)rl * r0) >> 32));
    long long e = (1LL << 58) - p;
    const int es = (int)(e >> 20);
    e += ((long long)es * es) >> 18;
    // r0 (1 + e) at 2^61: r0 2^32 + r0 e 2^-26
    const long long eh = e >> 32;
    const unsigned long long lo = ((unsigned long long)(unsigned)e * r0) >> 26;
    return (long long)(((unsigned long long)r0 << 32) + lo + (unsigned long long)((eh * (long long)r0) << 6));
}

// sqrt(rho) at 2^61 of rho at 2^61, rho in (1/4, 2): s = rho r with r a
// 22-bit estimate of 1/sqrt(rho), times 1 + e/2 + 3 e^2/8, e = 1 - s r
LB_FIX_FN long long fix_sqrt(long long rho) {
    const unsigned rh = (unsigned)(rho >> 32), rl = (unsigned)rho;
    const unsigned r0 = (unsigned)(fix_rsqrt((float)rh * 0x1p-29f) * 0x1p30f);
    const unsigned long long s = (unsigned long long)rh * r0 + (((unsigned long long)rl * r0) >> 32);    // 2^59
    const unsigned sh = (unsigned)(s >> 32), sl = (unsigned)s;
    const long long p = (long long)((unsigned long long)sh * r0 + (((unsigned long long)sl * r0) >> 32)); // 2^57
    long long e = (1LL << 57) - p;
    const int es = (int)(e >> 19);
    e = (e >> 1) + ((3 * (((long long)es * es) >> 19)) >> 3);
    const unsigned st = (unsigned)(s >> 28);                             // s at 2^31
    const long long eh = e >> 32;
    const long long c = (long long)(((unsigned long long)(unsigned)e * st) >> 29) + ((eh * (long long)st) << 3);
    return (long long)((s + (unsigned long long)c) << 2);
}

// Collision of one node: f the pre-collision populations, (Fx, Fy, Fz) the
// force, rnd the node's two Philox outputs (NOISE), node its index, o the
// post-collision populations. Returns false, o unspecified, outside the range
// above.
template <bool NOISE>
LB_FIX_FN bool collide_fix(const double (&f)[19], double (&o)[19], double Fx, double Fy, double Fz, const FixParams &P,
                           const unsigned (&rnd)[8], unsigned node) {
    typedef long long L;
    int over = 0;
    L v[19];
    v[0] = fix_in<1>(f[0], P.cb, over);
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int i = 1; i < 7; ++i) v[i] = fix_in<3>(f[i], P.cb, over);
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int i = 7; i < 19; ++i) v[i] = fix_in<4>(f[i], P.cb, over);

    const L s1 = v[1] + v[2], d1 = v[1] - v[2], s3 = v[3] + v[4], d3 = v[3] - v[4];
    const L s5 = v[5] + v[6], d5 = v[5] - v[6], s7 = v[7] + v[8], d7 = v[7] - v[8];
    const L s9 = v[9] + v[10], d9 = v[9] - v[10], s11 = v[11] + v[12], d11 = v[11] - v[12];
    const L s13 = v[13] + v[14], d13 = v[13] - v[14], s15 = v[15] + v[16], d15 = v[15] - v[16];
    const L s17 = v[17] + v[18], d17 = v[17] - v[18];
    const L Sax = s1 + s3 + s5, Sxy = s7 + s9, Sxz = s11 + s13, Syz = s15 + s17, Sd = Sxy + Sxz + Syz;
    const L rho = v[0] + Sax + Sd;
    const L tx = d7 + d9 + d11 + d13, ty = d7 - d9 + d15 + d17, tz = d11 - d13 + d15 - d17;

    // any component not 0 (tested as bits: no FP64 instruction)
    const bool forced = ((fix_bits(Fx) | fix_bits(Fy) | fix_bits(Fz)) << 1) != 0;
    L Fq[3] = {0, 0, 0}, cF[3] = {0, 0, 0};
    if (forced) {
        const double F[3] = {Fx, Fy, Fz};
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
        for (int a = 0; a < 3; ++a) {
            Fq[a] = fix_in<1>(F[a], P.cb, over);
            // F / 12, rounded up or down by a hash of the node: a constant
            // force far below 2^-61 of a population is right on average
            const unsigned h = (node ^ (0x9E3779B9u * (unsigned)a)) * 2654435761u;
            const double xi = fix_double(((unsigned long long)(0x3FF00000u | (h >> 12)) << 32)) - 1.0;
            const double t = (F[a] < 0.0 ? -F[a] : F[a]) * P.fs + xi;
            const unsigned long long b = (unsigned long long)fix_bits(t);
            const unsigned hi = (unsigned)(b >> 32);
            const unsigned long long m =
                (((unsigned long long)((hi & 0xFFFFFu) | 0x100000u) << 32) | (unsigned)b) << 10;
            const L q = (L)fix_shr(m, 1023 + 62 - (int)(hi >> 20));
            cF[a] = F[a] < 0.0 ? -q : q;
        }
    }
    // j + F/2
    const L gx = d1 + tx + (Fq[0] >> 1), gy = d3 + ty + (Fq[1] >> 1), gz = d5 + tz + (Fq[2] >> 1);
    {
        const int rh = (int)(rho >> 32);
        const int hx = (int)(gx >> 32), hy = (int)(gy >> 32), hz = (int)(gz >> 32);
        const int ax = hx < 0 ? -hx : hx, ay = hy < 0 ? -hy : hy, az = hz < 0 ? -hz : hz;
        const int am = ax > ay ? (ax > az ? ax : az) : (ay > az ? ay : az);
        // rho > 1/4, |g| < 1/2, |g| < rho / 2
        if (over < 0 || rh <= (1 << 27) || am >= (1 << 28) - 1 || 2 * am + 4 >= rh) return false;
    }
    const FixPair ir = fix_split(fix_reciprocal(rho));
    const FixPair Gx = fix_split(gx << 2), Gy = fix_split(gy << 2), Gz = fix_split(gz << 2);      // 2^63
    const FixPair ux = fix_split(fix_mul(Gx, ir) << 2), uy = fix_split(fix_mul(Gy, ir) << 2),     // 2^62
        uz = fix_split(fix_mul(Gz, ir) << 2);
    const L exx = fix_mul(Gx, ux), eyy = fix_mul(Gy, uy), ezz = fix_mul(Gz, uz);                  // 2^61
    const L eyz = eyy + ezz;

    const L A5 = 2 * s1 - s3 - s5, B5 = Sxy + Sxz - 2 * Syz, A6 = s3 - s5, B6 = Sxy - Sxz;
    L q4 = fix_mul(P.ke[0], fix_split(exx + eyz - (Sd - v[0])));
    L q5 = fix_mul(P.ke[1], fix_split(2 * exx - eyz - (A5 + B5)));
    L q6 = fix_mul(P.ke[2], fix_split(eyy - ezz - (A6 + B6)));
    L q7 = fix_mul(P.ke[3], fix_split(fix_mul(Gx, uy) - (s7 - s9)));
    L q8 = fix_mul(P.ke[4], fix_split(fix_mul(Gy, uz) - (s15 - s17)));
    L q9 = fix_mul(P.ke[5], fix_split(fix_mul(Gz, ux) - (s11 - s13)));
    if (forced) {
        const FixPair Hx = fix_split(Fq[0] << 2), Hy = fix_split(Fq[1] << 2), Hz = fix_split(Fq[2] << 2);   // 2^63
        const L fxx = fix_mul(ux, Hx), fyy = fix_mul(uy, Hy), fzz = fix_mul(uz, Hz);
        const L fyz = fyy + fzz;
        q4 += 2 * fix_mul(P.ks[0], fix_split(fxx + fyz));
        q5 += 2 * fix_mul(P.ks[1], fix_split(2 * fxx - fyz));
        q6 += 2 * fix_mul(P.ks[2], fix_split(fyy - fzz));
        q7 += fix_mul(P.ks[3], fix_split(fix_mul(ux, Hy) + fix_mul(uy, Hx)));
        q8 += fix_mul(P.ks[4], fix_split(fix_mul(uy, Hz) + fix_mul(uz, Hy)));
        q9 += fix_mul(P.ks[5], fix_split(fix_mul(uz, Hx) + fix_mul(ux, Hz)));
    }
    L q10 = -fix_mul(P.ke[6], fix_split(tx - 2 * d1));
    L q11 = -fix_mul(P.ke[7], fix_split(ty - 2 * d3));
    L q12 = -fix_mul(P.ke[8], fix_split(tz - 2 * d5));
    L q13 = -fix_mul(P.ke[9], fix_split(d7 + d9 - d11 - d13));
    L q14 = -fix_mul(P.ke[10], fix_split(d9 - d7 + d15 + d17));
    L q15 = -fix_mul(P.ke[11], fix_split(d11 - d13 - d15 + d17));
    L q16 = -fix_mul(P.ke[12], fix_split(v[0] - 2 * Sax + Sd));
    L q17 = -fix_mul(P.ke[13], fix_split(B5 - A5));
    L q18 = -fix_mul(P.ke[14], fix_split(B6 - A6));

    if (NOISE) {
        // the 16-bit variates of lb_collide.cuh as signed 2^-32 fractions;
        // amplitude sqrt(rho) kn at 2^61 (kn < 1 at 2^64, sqrt(rho) at 2^61)
        const FixPair sr = fix_split(fix_sqrt(rho));
        auto add = [&](L &q, int k, unsigned t) {
            const FixPair a = fix_split(fix_mul(sr, P.kn[k]));
            const int ti = (int)t;
            q += (L)ti * a.h + (((L)ti * a.l) >> 32);
        };
        auto hi = [&](L &q, int k, unsigned r) { add(q, k, (r & 0xFFFF0000u) ^ 0x80008000u); };
        auto lo = [&](L &q, int k, unsigned r) { add(q, k, (r << 16) ^ 0x80008000u); };
        hi(q4, 0, rnd[0]); lo(q5, 1, rnd[0]); hi(q6, 2, rnd[1]); lo(q7, 3, rnd[1]);
        hi(q8, 4, rnd[2]); lo(q9, 5, rnd[2]); hi(q10, 6, rnd[3]); lo(q11, 7, rnd[3]);
        hi(q12, 8, rnd[4]); lo(q13, 9, rnd[4]); hi(q14, 10, rnd[5]); lo(q15, 11, rnd[5]);
        hi(q16, 12, rnd[6]); lo(q17, 13, rnd[6]); hi(q18, 14, rnd[7]);
    }

    unsigned small = 0xFFFFFFFFu;
    auto put = [&](int i, L V) { o[i] = i < LB_FIX_OUT64 ? fix_out64(V, P) : fix_out(V, P, small); };
    put(0, v[0] + 12 * (q16 - q4));
    const L U = -2 * q16, V = q17 - q5, W = q6 - q18;
    auto pair2 = [&](int i, L E, L O) {
        put(i, v[i] + E + O);
        put(i + 1, v[i + 1] + E - O);
    };
    pair2(1, 2 * (U - 2 * V), 2 * (cF[0] - 2 * q10));
    pair2(3, 2 * (U + V + W), 2 * (cF[1] - 2 * q11));
    pair2(5, 2 * (U + V - W), 2 * (cF[2] - 2 * q12));
    const L Ed = q4 + q16, S5 = q5 + q17, S6 = q6 + q18;
    const L T1 = Ed + S5 + S6, T2 = Ed + S5 - S6, T3 = Ed - 2 * S5;
    const L X = cF[0] + q10, Y = cF[1] + q11, Z = cF[2] + q12;
    pair2(7, T1 + q7, X + Y + q13 - q14);
    pair2(9, T1 - q7, X - Y + q13 + q14);
    pair2(11, T2 + q9, X + Z - q13 + q15);
    pair2(13, T2 - q9, X - Z - q13 - q15);
    pair2(15, T3 + q8, Y + Z + q14 - q15);
    pair2(17, T3 - q8, Y - Z + q14 + q15);
    return small != 0u;
}

#ifdef __CUDACC__
// The FP64 evaluation, out of line: the few nodes outside the fixed-point
// range take it, and its registers stay out of the kernel's.
template <int COLL, bool NOISE>
__device__ __noinline__ void collide_f64(double *f, double Fx, double Fy, double Fz, const CollParams<double> &pd, uint2 key,
                                         uint32_t instance, uint32_t node, uint32_t step) {
    double v[19];
#pragma unroll
    for (int i = 0; i < 19; ++i) v[i] = f[i];
    collide<double, false, COLL, NOISE>(v, Fx, Fy, Fz, pd, key, instance, node, step);
#pragma unroll
    for (int i = 0; i < 19; ++i) f[i] = v[i];
}

// Collision of one FP64 node: in fixed point, or in FP64 from the populations
// that `reload` fetches again (nothing has been stored yet).
template <int COLL, bool NOISE, typename Reload>
__device__ __forceinline__ void collide_node_f64(double (&f)[19], double Fx, double Fy, double Fz, const FixParams &fx,
                                                 const CollParams<double> &pd, uint2 key, uint32_t instance,
                                                 uint32_t node, uint32_t step, Reload reload) {
    bool ok = false;
    double o[19];
    if (fx.on) {
        unsigned rnd[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        if (NOISE) {
            const uint4 r0 = philox4x32_10(make_uint4(node, step, instance, 0u), key);
            const uint4 r1 = philox4x32_10(make_uint4(node, step, instance, 1u), key);
            rnd[0] = r0.x; rnd[1] = r0.y; rnd[2] = r0.z; rnd[3] = r0.w;
            rnd[4] = r1.x; rnd[5] = r1.y; rnd[6] = r1.z; rnd[7] = r1.w;
        }
        ok = collide_fix<NOISE>(f, o, Fx, Fy, Fz, fx, rnd, node);
    }
    if (!ok) {
        asm volatile("" ::: "memory");         // fetched again, not kept in registers across the collision
        double g[19];
        reload(g);
        collide_f64<COLL, NOISE>(g, Fx, Fy, Fz, pd, key, instance, node, step);
#pragma unroll
        for (int i = 0; i < 19; ++i) o[i] = g[i];
    }
#pragma unroll
    for (int i = 0; i < 19; ++i) f[i] = o[i];
}
#endif

// The fixed-point constants of a parameter set. rate[k - 4]: the relaxation
// rate g_k of mode k = 4..18 (BGK: 1 - 1/tau for all). Not usable (on = 0)
// when the scaled exponents could leave the doubles', a factor of the
// equilibrium fix_split's, or too many nodes the range above by their noise:
// from kT = 0.002 rho0 on most warps hold a node that does, and pay for both
// evaluations. 94 x 81 x 103, us per step in fixed point (FP64: 462): 74 at kT
// = 5e-4, 98 at 1e-3 (0.1 % of the nodes leave), 239 at 1.5e-3, 421 at 2e-3
// (6 %), 485 from 3e-3 (20 %) on; 40^3 67.8 at 2e-3, 74-75 beyond (FP64: 69).
inline FixParams fix_params(double rho0, double kT, const double rate[15]) {
    FixParams P{};
    int e = 0;
    std::frexp(rho0 * 1.5, &e);
    const int k = e - 1;                       // rho0 2^-k in [2/3, 4/3)
    P.on = k > -600 && k < 600 && kT <= 0.002 * rho0 ? 1 : 0;
    P.cb = 1023 + k;
    P.ce = (1023 + k) * (1 << 20);
    P.eh = (0x453 - 61 + k) * (1 << 20);
    P.el = (0x433 - 61 + k) * (1 << 20);
    P.out = std::ldexp(0x1p84 + 0x1p63 + 0x1p52, k - 61);
    P.fs = std::ldexp(1.0, 61 - k) / 12.0;
    static const long double b[15] = {2.0L / 3, 4.0L / 3, 4.0L / 9, 1.0L / 9, 1.0L / 9, 1.0L / 9, 2.0L / 3, 2.0L / 3,
                                      2.0L / 3, 2.0L / 9, 2.0L / 9, 2.0L / 9, 2.0L,     4.0L / 3, 4.0L / 9};
    for (int q = 0; q < 15; ++q) {
        const long double c = 1.0L / 36 / b[q], g = rate[q], ke = std::ldexp(c * (1 - g), 64);
        if (ke >= 0x1p63L - 0x1p31L) {         // c = 1/4 and g within 2^-31 of -1: beyond fix_split's range
            P.on = 0;
            return P;
        }
        P.ke[q] = fix_split(std::llrint(ke));
        if (q < 6) P.ks[q] = fix_split(std::llrint(std::ldexp(c * (1 + g) / 2, 64)));
        if (P.on) {
            const long double kn = c * std::sqrt(36.0L * kT * b[q] * (1 - g * g));
            P.kn[q] = fix_split(std::llrint(std::ldexp(kn * std::exp2(-0.5L * k), 64)));
        }
    }
    return P;
}

}  // namespace lbk
