// Collision of one node (Sec. 1.1 of Ustach & Faller, arXiv:1604.01829),
// shared by the fused collide-and-stream kernels.
#pragma once

#include "lb_internal.h"

namespace lbk {

// ---------------------------------------------------------------- collision
// Post-collision populations of one node, in place. Force F = uniform + spread
// bead force; u = (j + F/2) / rho (Guo forcing); MRT in the orthogonal
// D3Q19 moment basis 1, c, c^2-1, 3cx^2-c^2, cy^2-cz^2, cxcy, cycz, czcx,
// (3c^2-5)c, (cy^2-cz^2)cx, (cz^2-cx^2)cy, (cx^2-cy^2)cz, 3c^4-6c^2+1,
// (2c^2-3)(3cx^2-c^2), (2c^2-3)(cy^2-cz^2), with norms b_k = sum w e_k^2.
template <typename R, bool DEV, int COLL, bool NOISE>
__device__ __forceinline__ void collide(R (&f)[19], R Fx, R Fy, R Fz, const CollParams<R> &a, uint2 key,
                                        uint32_t instance, uint32_t node, uint32_t step) {
    const R s1 = f[1] + f[2], d1 = f[1] - f[2];
    const R s3 = f[3] + f[4], d3 = f[3] - f[4];
    const R s5 = f[5] + f[6], d5 = f[5] - f[6];
    const R s7 = f[7] + f[8], d7 = f[7] - f[8];
    const R s9 = f[9] + f[10], d9 = f[9] - f[10];
    const R s11 = f[11] + f[12], d11 = f[11] - f[12];
    const R s13 = f[13] + f[14], d13 = f[13] - f[14];
    const R s15 = f[15] + f[16], d15 = f[15] - f[16];
    const R s17 = f[17] + f[18], d17 = f[17] - f[18];
    const R Sax = s1 + s3 + s5;
    const R Sxy = s7 + s9, Sxz = s11 + s13, Syz = s15 + s17;
    const R Sd = Sxy + Sxz + Syz;
    const R m0 = f[0] + Sax + Sd;                      // rho, or rho - rho0 for deviations
    const R rho = DEV ? a.rho0 + m0 : m0;
    const R jx = d1 + d7 + d9 + d11 + d13;
    const R jy = d3 + d7 - d9 + d15 + d17;
    const R jz = d5 + d11 - d13 + d15 - d17;
    R ir;
    if constexpr (sizeof(R) == 4) ir = __fdividef(1.0f, rho); else ir = R(1) / rho;
    const R ux = (jx + R(0.5) * Fx) * ir;
    const R uy = (jy + R(0.5) * Fy) * ir;
    const R uz = (jz + R(0.5) * Fz) * ir;
    const R uF = ux * Fx + uy * Fy + uz * Fz;
    const R uu = ux * ux + uy * uy + uz * uz;
    constexpr R w0 = R(1.0 / 3.0), w1 = R(1.0 / 18.0), w2 = R(1.0 / 36.0);

    if (COLL == 0) {
        // BGK: f* = f - (f - f_eq)/tau + (1 - 1/(2 tau)) w [3(c-u) + 9 (c.u) c].F
        const R om = a.omega, h = R(1) - R(0.5) * om;
        const R base = DEV ? m0 : rho;                 // w rho (or w (rho - rho0)) coefficient of '1'
        const R k2 = R(1.5) * uu;
        // rest population
        f[0] = f[0] - om * (f[0] - w0 * (base - rho * k2)) + h * w0 * (R(-3) * uF);
        auto pair = [&](int i, R cu, R cF, R w) {
            const R e = w * (base + rho * (R(4.5) * cu * cu - k2));
            const R o = w * rho * R(3) * cu;
            const R se = w * (R(9) * cu * cF - R(3) * uF);
            const R so = w * R(3) * cF;
            f[i] = f[i] - om * (f[i] - (e + o)) + h * (se + so);
            f[i + 1] = f[i + 1] - om * (f[i + 1] - (e - o)) + h * (se - so);
        };
        pair(1, ux, Fx, w1);
        pair(3, uy, Fy, w1);
        pair(5, uz, Fz, w1);
        pair(7, ux + uy, Fx + Fy, w2);
        pair(9, ux - uy, Fx - Fy, w2);
        pair(11, ux + uz, Fx + Fz, w2);
        pair(13, ux - uz, Fx - Fz, w2);
        pair(15, uy + uz, Fy + Fz, w2);
        pair(17, uy - uz, Fy - Fz, w2);
        return;
    }

    // MRT: non-conserved moments
    const R A5 = R(2) * s1 - s3 - s5, B5 = Sxy + Sxz - R(2) * Syz;
    const R A6 = s3 - s5, B6 = Sxy - Sxz;
    const R m4 = Sd - f[0];
    const R m5 = A5 + B5, m17 = B5 - A5;
    const R m6 = A6 + B6, m18 = B6 - A6;
    const R m7 = s7 - s9, m8 = s15 - s17, m9 = s11 - s13;
    const R m10 = R(-2) * d1 + d7 + d9 + d11 + d13;
    const R m11 = R(-2) * d3 + d7 - d9 + d15 + d17;
    const R m12 = R(-2) * d5 + d11 - d13 + d15 - d17;
    const R m13 = d7 + d9 - d11 - d13;
    const R m14 = -d7 + d9 + d15 + d17;
    const R m15 = d11 - d13 - d15 + d17;
    const R m16 = f[0] - R(2) * Sax + Sd;

    // Post-collision moments, each already multiplied by c_k = w_diag / b_k
    // (the host folds c_k into the rates): A_k = c_k ((1 - g_k) m_eq + g_k m
    // + (1 + g_k)/2 S_k + noise). Equilibrium stress moments rho u u and Guo
    // source moments (uF + Fu); ghost modes have zero equilibrium and source.
    const R ruu_x = rho * ux, ruu_y = rho * uy, ruu_z = rho * uz;
    const R e4 = ruu_x * ux + ruu_y * uy + ruu_z * uz;
    const R exx = ruu_x * ux, eyy = ruu_y * uy, ezz = ruu_z * uz;
    const R e5 = R(2) * exx - eyy - ezz, e6 = eyy - ezz;
    const R e7 = ruu_x * uy, e8 = ruu_y * uz, e9 = ruu_z * ux;
    const R uFx = ux * Fx, uFy = uy * Fy, uFz = uz * Fz;
    R q4 = a.ke[0] * e4 + a.km[0] * m4 + a.ks[0] * (R(2) * uF);
    R q5 = a.ke[1] * e5 + a.km[1] * m5 + a.ks[1] * (R(2) * (R(2) * uFx - uFy - uFz));
    R q6 = a.ke[2] * e6 + a.km[2] * m6 + a.ks[2] * (R(2) * (uFy - uFz));
    R q7 = a.ke[3] * e7 + a.km[3] * m7 + a.ks[3] * (ux * Fy + uy * Fx);
    R q8 = a.ke[4] * e8 + a.km[4] * m8 + a.ks[4] * (uy * Fz + uz * Fy);
    R q9 = a.ke[5] * e9 + a.km[5] * m9 + a.ks[5] * (uz * Fx + ux * Fz);
    R q10 = a.kg[0] * m10, q11 = a.kg[1] * m11, q12 = a.kg[2] * m12;
    R q13 = a.kg[3] * m13, q14 = a.kg[4] * m14, q15 = a.kg[5] * m15;
    R q16 = a.kg[6] * m16, q17 = a.kg[7] * m17, q18 = a.kg[8] * m18;

    if constexpr (NOISE) {
        static_assert(sizeof(R) == 8, "FP32 with noise: collide_mrt_f32");
        // 15 non-conserved modes, variance 3 rho kT b_k (1 - g_k^2); kn_k holds
        // c_k sqrt(3 kT b_k (1 - g_k^2)) sqrt(12). The
        // variates are 16-bit: two Philox calls give 16 half-words, mode 4 + j
        // takes half-word j (high half of word j/2 for even j, else the low
        // half), xi = sqrt(12) ((h + 1/2) 2^-16 - 1/2).
        const uint4 r0 = philox4x32_10(make_uint4(node, step, instance, 0u), key);
        const uint4 r1 = philox4x32_10(make_uint4(node, step, instance, 1u), key);
        const R sr = sqrt(rho);
        auto hi = [&](R &q, int k, uint32_t v) { q += (sr * a.kn[k]) * centred16_d(v >> 16); };
        auto lo = [&](R &q, int k, uint32_t v) { q += (sr * a.kn[k]) * centred16_d(v & 0xFFFFu); };
        hi(q4, 0, r0.x); lo(q5, 1, r0.x); hi(q6, 2, r0.y); lo(q7, 3, r0.y);
        hi(q8, 4, r0.z); lo(q9, 5, r0.z); hi(q10, 6, r0.w); lo(q11, 7, r0.w);
        hi(q12, 8, r1.x); lo(q13, 9, r1.x); hi(q14, 10, r1.y); lo(q15, 11, r1.y);
        hi(q16, 12, r1.z); lo(q17, 13, r1.z); hi(q18, 14, r1.w);
    }

    // back to populations: f*_i = w_i sum_k e_k(c_i) m*_k / b_k; with the
    // c_k folded in, diagonal links are E +- O, axis links 2 (E +- O), rest 12 E
    constexpr R c0 = R(1.0 / 36.0), c1 = R(1.0 / 12.0);
    const R q0 = c0 * m0;
    const R q1 = c1 * (jx + Fx), q2 = c1 * (jy + Fy), q3 = c1 * (jz + Fz);
    f[0] = R(12) * (q0 - q4 + q16);
    const R U = q0 - R(2) * q16, V = q17 - q5, Wv = q6 - q18;
    {
        const R E = U - R(2) * V, O = q1 - R(2) * q10;
        f[1] = R(2) * (E + O); f[2] = R(2) * (E - O);
    }
    {
        const R E = U + V + Wv, O = q2 - R(2) * q11;
        f[3] = R(2) * (E + O); f[4] = R(2) * (E - O);
    }
    {
        const R E = U + V - Wv, O = q3 - R(2) * q12;
        f[5] = R(2) * (E + O); f[6] = R(2) * (E - O);
    }
    const R Ed = q0 + q4 + q16;
    const R S5 = q5 + q17, S6 = q6 + q18;
    const R T1 = Ed + S5 + S6, T2 = Ed + S5 - S6, T3 = Ed - R(2) * S5;
    const R P = q1 + q10, Q = q2 + q11, Rr = q3 + q12;
    {
        const R O = P + Q + q13 - q14;
        f[7] = T1 + q7 + O; f[8] = T1 + q7 - O;
    }
    {
        const R O = P - Q + q13 + q14;
        f[9] = T1 - q7 + O; f[10] = T1 - q7 - O;
    }
    {
        const R O = P + Rr - q13 + q15;
        f[11] = T2 + q9 + O; f[12] = T2 + q9 - O;
    }
    {
        const R O = P - Rr - q13 - q15;
        f[13] = T2 - q9 + O; f[14] = T2 - q9 - O;
    }
    {
        const R O = Q + Rr + q14 - q15;
        f[15] = T3 + q8 + O; f[16] = T3 + q8 - O;
    }
    {
        const R O = Q - Rr + q14 + q15;
        f[17] = T3 - q8 + O; f[18] = T3 - q8 - O;
    }
}

// The MRT collision in FP32 on deviations, two values per instruction
// (fma.rn.f32x2 and its kin): the planes xy and xz, the axes y and z, and the
// modes they mix into share every formula but a sign, so links (7, 11), (9, 13),
// (3, 5) and (15, 17), components (y, z) and modes (5, 6), (7, 9), (11, 12),
// (14, -15), (17, 18) go in pairs: ~140 FP32 instructions instead of ~240, in a
// kernel that waits for memory at the occupancy its registers allow and, on a
// lattice that stays in L2, is bound by issue. Measured against the scalar
// form: 256^3 with noise 436.9 -> 427.5 us per launch, 64 batched boxes of 24^3
// with noise 30.9 -> 28.5, 256 uneven instances without 640 -> 629 (624 at 56
// registers); one lattice without noise 86.7 -> 88.0 (150 x 97 x 203: the pairs
// spill at the 64 registers that suit it), so that keeps the scalar form.
template <bool NOISE>
__device__ __forceinline__ void collide_mrt_f32(float (&f)[19], float Fx, float Fy, float Fz, const CollPairs &a,
                                                uint2 key, uint32_t instance, uint32_t node, uint32_t step) {
    auto add = [](float2 x, float2 y) { return __fadd2_rn(x, y); };
    auto mul = [](float2 x, float2 y) { return __fmul2_rn(x, y); };
    auto fma = [](float2 x, float2 y, float2 z) { return __ffma2_rn(x, y, z); };
    auto two = [](float x) { return make_float2(x, x); };
    auto sub = [](float2 x, float2 y) { return __ffma2_rn(y, make_float2(-1.f, -1.f), x); };
    auto pr = [](float x, float y) { return make_float2(x, y); };

    const float2 p1 = pr(f[7], f[11]), o1 = pr(f[8], f[12]), p2 = pr(f[9], f[13]), o2 = pr(f[10], f[14]);
    const float2 py = pr(f[3], f[5]), oy = pr(f[4], f[6]), pz = pr(f[15], f[17]), oz = pr(f[16], f[18]);
    const float2 s1 = add(p1, o1), d1 = sub(p1, o1), s2 = add(p2, o2), d2 = sub(p2, o2);
    const float2 sY = add(py, oy), dY = sub(py, oy), sZ = add(pz, oz), dZ = sub(pz, oz);
    const float sx = f[1] + f[2], dx = f[1] - f[2];
    const float2 Sp = add(s1, s2), m79 = sub(s1, s2);                     // (Sxy, Sxz), (m7, m9)
    const float2 dp = add(d1, d2), dm = sub(d1, d2);
    const float Syz = sZ.x + sZ.y, m8 = sZ.x - sZ.y;
    const float2 dz = pr(dZ.x + dZ.y, dZ.x - dZ.y);
    const float Sxx = Sp.x + Sp.y, Sd = Sxx + Syz, Sa = sY.x + sY.y, Sax = sx + Sa;
    const float m0 = f[0] + Sax + Sd;
    const float rho = a.rho0 + m0;
    const float tx = dp.x + dp.y, jx = dx + tx;
    const float2 tyz = add(dm, dz), jyz = add(dY, tyz);
    const float m10 = fmaf(-2.f, dx, tx), m13 = dp.x - dp.y;
    const float2 m1112 = fma(dY, two(-2.f), tyz), m1415 = sub(dz, dm);    // (m14, -m15)
    const float2 A = pr(fmaf(2.f, sx, -Sa), sY.x - sY.y), B = pr(fmaf(-2.f, Syz, Sxx), Sp.x - Sp.y);
    const float2 m56 = add(A, B), m1718 = sub(B, A);
    const float m4 = Sd - f[0], m16 = fmaf(-2.f, Sax, f[0] + Sd);

    const float ir = __fdividef(1.0f, rho);
    const float2 Fyz = pr(Fy, Fz);
    const float ux = fmaf(0.5f, Fx, jx) * ir;
    const float2 uyz = mul(fma(Fyz, two(0.5f), jyz), two(ir));
    // equilibrium stress rho u u and Guo source (uF + Fu; ks holds its 2)
    const float rux = rho * ux;
    const float2 ruyz = mul(two(rho), uyz), eyz = mul(ruyz, uyz);
    const float exx = rux * ux, et = eyz.x + eyz.y;
    const float2 e56 = pr(fmaf(2.f, exx, -et), eyz.x - eyz.y), e79 = mul(two(rux), uyz);
    const float e8 = ruyz.x * uyz.y;
    const float2 g = mul(uyz, Fyz);
    const float gx = ux * Fx, gt = g.x + g.y;
    const float2 g56 = pr(fmaf(2.f, gx, -gt), g.x - g.y), g79 = fma(two(ux), Fyz, mul(uyz, two(Fx)));
    const float g8 = fmaf(uyz.x, Fz, uyz.y * Fy);
    float q4 = fmaf(a.ke4, exx + et, fmaf(a.km4, m4, a.ks4 * (gx + gt)));
    float2 q56 = fma(a.ke56, e56, fma(a.km56, m56, mul(a.ks56, g56)));
    float2 q79 = fma(a.ke79, e79, fma(a.km79, m79, mul(a.ks79, g79)));
    float q8 = fmaf(a.ke8, e8, fmaf(a.km8, m8, a.ks8 * g8));
    float q10 = a.kg10 * m10, q13 = a.kg13 * m13, q16 = a.kg16 * m16;
    float2 q1112 = mul(a.kg1112, m1112), q1415 = mul(a.kg1415, m1415), q1718 = mul(a.kg1718, m1718);

    if (NOISE) {
        // 15 non-conserved modes, variance 3 rho kT b_k (1 - g_k^2); kn_k holds
        // c_k sqrt(3 kT b_k (1 - g_k^2)) sqrt(12) 2^-32. Mode 4 + j takes
        // half-word j of two Philox calls (high half of word j/2 for even j,
        // else the low half), xi = sqrt(12) ((h + 1/2) 2^-16 - 1/2): the
        // half-word and a 1/2 below it become the mantissa of y = 1 + (h + 1/2)
        // 2^-16 in [1, 2), and (y - 3/2) 2^32 is exact in one FMA (no
        // integer-to-float conversion).
        const uint4 r0 = philox4x32_10(make_uint4(node, step, instance, 0u), key);
        const uint4 r1 = philox4x32_10(make_uint4(node, step, instance, 1u), key);
        float sr;
        asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(sr) : "f"(rho));
        auto hi = [](uint32_t v) { return __uint_as_float(((v >> 9) & 0x7FFF80u) | 0x3F800040u); };
        auto lo = [](uint32_t v) { return __uint_as_float(((v << 7) & 0x7FFF80u) | 0x3F800040u); };
        auto n1 = [&](float &q, float k, float y) { q = fmaf(sr * k, fmaf(y, 0x1p32f, -0x1.8p32f), q); };
        auto n2 = [&](float2 &q, float2 k, float y, float z) {
            q = fma(mul(two(sr), k), fma(pr(y, z), two(0x1p32f), two(-0x1.8p32f)), q);
        };
        n1(q4, a.kn4, hi(r0.x));
        n2(q56, a.kn56, lo(r0.x), hi(r0.y));
        n2(q79, a.kn79, lo(r0.y), lo(r0.z));
        n1(q8, a.kn8, hi(r0.z));
        n1(q10, a.kn10, hi(r0.w));
        n2(q1112, a.kn1112, lo(r0.w), hi(r1.x));
        n1(q13, a.kn13, lo(r1.x));
        n2(q1415, a.kn1415, hi(r1.y), lo(r1.y));
        n1(q16, a.kn16, hi(r1.z));
        n2(q1718, a.kn1718, lo(r1.z), hi(r1.w));
    }

    // back to populations (as collide)
    constexpr float c0 = 1.0f / 36.0f, c1 = 1.0f / 12.0f;
    const float q0 = c0 * m0, q1 = c1 * (jx + Fx);
    const float2 q23 = mul(add(jyz, Fyz), two(c1));
    f[0] = 12.f * (q0 - q4 + q16);
    const float U = fmaf(-2.f, q16, q0);
    const float2 VW = sub(q1718, q56);                                    // (V, -W)
    {
        const float E = fmaf(-2.f, VW.x, U), O = fmaf(-2.f, q10, q1);
        f[1] = 2.f * (E + O);
        f[2] = 2.f * (E - O);
    }
    {
        const float UV = U + VW.x;
        const float2 E = pr(UV - VW.y, UV + VW.y), O = fma(q1112, two(-2.f), q23);
        const float2 u = mul(two(2.f), add(E, O)), v = mul(two(2.f), sub(E, O));
        f[3] = u.x; f[5] = u.y;
        f[4] = v.x; f[6] = v.y;
    }
    const float Ed = q0 + q4 + q16;
    const float2 S = add(q56, q1718);
    const float T = Ed + S.x, T3 = fmaf(-2.f, S.x, Ed);
    const float2 T12 = pr(T + S.y, T - S.y), Ep = add(T12, q79), Em = sub(T12, q79);
    const float P = q1 + q10;
    const float2 QR = add(q23, q1112), Pc = pr(P + q13, P - q13), G = sub(QR, q1415);
    const float2 O1 = add(Pc, G), O2 = sub(Pc, G);
    const float2 a7 = add(Ep, O1), a8 = sub(Ep, O1), a9 = add(Em, O2), a10 = sub(Em, O2);
    f[7] = a7.x; f[11] = a7.y;
    f[8] = a8.x; f[12] = a8.y;
    f[9] = a9.x; f[13] = a9.y;
    f[10] = a10.x; f[14] = a10.y;
    const float2 H = add(QR, q1415);                                      // (Q + q14, R - q15)
    const float2 O3 = pr(H.x + H.y, H.x - H.y), E3 = pr(T3 + q8, T3 - q8);
    const float2 a15 = add(E3, O3), a16 = sub(E3, O3);
    f[15] = a15.x; f[17] = a15.y;
    f[16] = a16.x; f[18] = a16.y;
}

// Fetches [p, p + bytes) into L2, without waiting (16-byte aligned, a multiple
// of 16 bytes).
__device__ __forceinline__ void fetch_l2(const void *p, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(__cvta_generic_to_global(p)), "r"(bytes) : "memory");
}

// Collision of one FP32 node: MRT in pairs (PAIRS, and always with noise), or
// as it stands.
template <int COLL, bool NOISE, bool PAIRS>
__device__ __forceinline__ void collide_f32(float (&f)[19], float Fx, float Fy, float Fz, const CollParams<float> &pf,
                                            const CollPairs &pk, uint2 key, uint32_t instance, uint32_t node,
                                            uint32_t step) {
    if constexpr (COLL == 1 && (PAIRS || NOISE)) collide_mrt_f32<NOISE>(f, Fx, Fy, Fz, pk, key, instance, node, step);
    else collide<float, true, COLL, false>(f, Fx, Fy, Fz, pf, key, instance, node, step);
}

}  // namespace lbk
