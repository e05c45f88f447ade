// The collision of two nodes at once in packed float32 pairs (sm_100+ f32x2
// instructions: one issue slot for two nodes' operation; the float32 pipe runs
// at the same rate either way, 36-37 T results/s measured for fma.rn.f32 and
// fma.rn.f32x2 on one GB300, so a pair saves issue slots, not pipe time).
//
// collide_pair gives, node by node, the bits of collide_node (lattice.cuh):
// the same operations in the same order, with the multiply-adds that the
// compiler contracts there written out. (Which products it contracts was
// found from collide_node's outputs on random nodes, and is held by the tests
// that compare this kernel's states with the scalar kernels' bit for bit.)
// Products by powers of two are exact, so their place does not matter.
#pragma once
#include <cuda_runtime.h>

#include <cstring>

#include "lattice.cuh"

namespace dmrt {

// Two floats, the first node's in the low half.
using F2 = unsigned long long;

__device__ __forceinline__ F2 f2_pack(float lo, float hi) {
    F2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}
__device__ __forceinline__ float f2_lo(F2 a) {
    float lo;
    asm("mov.b64 {%0, _}, %1;" : "=f"(lo) : "l"(a));
    return lo;
}
__device__ __forceinline__ float f2_hi(F2 a) {
    float hi;
    asm("mov.b64 {_, %0}, %1;" : "=f"(hi) : "l"(a));
    return hi;
}
__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {
    F2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ F2 f2_sub(F2 a, F2 b) {
    F2 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b) {
    F2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ F2 f2_fma(F2 a, F2 b, F2 c) {
    F2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ F2 f2_all(float v) { return f2_pack(v, v); }

// The constants of collide_pair as pairs (both halves equal), with the signs
// they are used in, so that a kernel takes them from its parameters as 64-bit
// operands: a cavity's relaxation rates, buoyancy and reference temperature,
// and the numbers of the transforms.
struct PairRates {
    F2 n_se36, snu4, sq12, n_seps36;
    F2 sk2, n_sk2, se20, snu4t, n_snu4t, n_a;
    F2 gbeta, theta_ref;
};
struct PairNumbers {
    F2 c2, m2, c3, m3, c4, m4, m1, c6, m6, m12, mh, q;  // 2, -2, 3, -3, 4, -4, -1, 1/6, -1/6, -1/12, -1/2, 1/4
};
struct PairConsts {
    PairRates r;
    PairNumbers n;
};

inline F2 pair_const(float v) {
    unsigned u;
    memcpy(&u, &v, sizeof u);
    return (F2)u | ((F2)u << 32);
}
inline PairRates make_pair_rates(const StepConsts& s) {
    PairRates p;
    p.n_se36 = pair_const(-s.se36);
    p.snu4 = pair_const(s.snu4);
    p.sq12 = pair_const(s.sq12);
    p.n_seps36 = pair_const(-s.seps36);
    p.sk2 = pair_const(s.sk2);
    p.n_sk2 = pair_const(-s.sk2);
    p.se20 = pair_const(s.se20);
    p.snu4t = pair_const(s.snu4t);
    p.n_snu4t = pair_const(-s.snu4t);
    p.n_a = pair_const(-s.a);
    p.gbeta = pair_const(s.gbeta);
    p.theta_ref = pair_const(s.theta_ref);
    return p;
}
inline PairNumbers make_pair_numbers() {
    PairNumbers p;
    p.c2 = pair_const(2.f);
    p.m2 = pair_const(-2.f);
    p.c3 = pair_const(3.f);
    p.m3 = pair_const(-3.f);
    p.c4 = pair_const(4.f);
    p.m4 = pair_const(-4.f);
    p.m1 = pair_const(-1.f);
    p.c6 = pair_const(1.f / 6.f);
    p.m6 = pair_const(-(1.f / 6.f));
    p.m12 = pair_const(-(1.f / 12.f));
    p.mh = pair_const(-0.5f);
    p.q = pair_const(0.25f);
    return p;
}
inline PairConsts make_pair_consts(const StepConsts& s) { return PairConsts{make_pair_rates(s), make_pair_numbers()}; }

// collide_node for a pair of nodes, in place (see there for the model; n_x is
// -x, used where it saves a negation).
__device__ __forceinline__ void collide_pair(F2 (&f)[9], F2 (&g)[5], const PairRates& K,
                                             const PairNumbers& C, F2& rho_out, F2& theta_out) {
    const F2 c2 = C.c2, m2 = C.m2, c3 = C.c3, m3 = C.m3, c4 = C.c4, m4 = C.m4;
    const F2 a13 = f2_sub(f[1], f[3]), a24 = f2_sub(f[2], f[4]);
    const F2 s13 = f2_add(f[1], f[3]), s24 = f2_add(f[2], f[4]);
    const F2 a56 = f2_sub(f[5], f[6]), a78 = f2_sub(f[7], f[8]);
    const F2 s56 = f2_add(f[5], f[6]), s78 = f2_add(f[7], f[8]);
    const F2 s1234 = f2_add(s13, s24), s5678 = f2_add(s56, s78);
    const F2 rho = f2_add(f2_add(f[0], s1234), s5678);
    const F2 ax = f2_add(a13, a56);
    const F2 u = f2_sub(ax, a78), n_u = f2_sub(a78, ax);
    const F2 v = f2_sub(f2_add(a24, s56), s78);
    const F2 n_e = f2_fma(m2, s5678, f2_fma(c4, f[0], s1234));
    const F2 pxx = f2_sub(s13, s24);
    const F2 pxy = f2_sub(f2_add(f[5], f[7]), f2_add(f[6], f[8]));
    const F2 qx = f2_sub(f2_fma(m2, a13, a56), a78);
    const F2 qy = f2_sub(f2_fma(m2, a24, s56), s78);
    const F2 eps = f2_fma(m2, f2_fma(m2, f[0], s1234), s5678);
    const F2 vv = f2_mul(v, v);
    const F2 uu = f2_fma(u, u, vv), n_uud = f2_fma(n_u, u, vv);
    const F2 theta = f2_add(f2_add(f2_add(f2_add(g[0], g[1]), g[2]), g[3]), g[4]);

    // Force terms of the moments, negated.
    const F2 Gy = f2_mul(K.gbeta, f2_sub(theta, K.theta_ref));
    const F2 n_g12 = f2_mul(Gy, C.m12);
    const F2 n_fe = f2_mul(f2_mul(n_g12, v), f2_fma(m3, uu, c2));
    const F2 n_fqx = f2_mul(f2_mul(f2_mul(C.mh, Gy), u), v);
    const F2 n_fqy = f2_mul(n_g12, f2_fma(f2_mul(c3, u), u, C.m1));
    const F2 g4 = f2_mul(C.q, Gy);
    const F2 n_fpxx = f2_mul(f2_mul(g4, v), f2_fma(m3, n_uud, c2));
    const F2 n_fpxy = f2_mul(f2_mul(g4, u), f2_fma(f2_mul(c3, v), v, C.m1));

    const F2 d3 = f2_fma(K.n_se36, f2_fma(c3, uu, f2_fma(m2, rho, n_e)), n_fe);
    const F2 d4 = f2_fma(K.snu4, f2_add(pxx, n_uud), n_fpxx);
    const F2 d5 = f2_fma(K.snu4, f2_fma(n_u, v, pxy), n_fpxy);
    const F2 d6 = f2_fma(K.sq12, f2_add(qx, u), n_fqx);
    const F2 d7 = f2_fma(K.sq12, f2_add(qy, v), n_fqy);
    const F2 n_d8 = f2_fma(K.n_seps36, f2_fma(c3, uu, f2_sub(eps, rho)), n_fe);

    const F2 c6 = C.c6, m6 = C.m6;
    f[0] = f2_fma(c4, n_d8, f2_fma(c4, d3, f[0]));
    f[1] = f2_fma(m2, n_d8, f2_fma(c2, d6, f2_sub(f2_add(f[1], d3), d4)));
    f[2] = f2_fma(Gy, c6, f2_fma(m2, n_d8, f2_fma(c2, d7, f2_add(f2_add(f[2], d3), d4))));
    f[3] = f2_fma(m2, n_d8, f2_fma(m2, d6, f2_sub(f2_add(f[3], d3), d4)));
    f[4] = f2_fma(Gy, m6, f2_fma(m2, n_d8, f2_fma(m2, d7, f2_add(f2_add(f[4], d3), d4))));
    f[5] = f2_fma(Gy, c6, f2_add(f2_sub(f2_sub(f2_sub(f2_fma(m2, d3, f[5]), d5), d6), d7), n_d8));
    f[6] = f2_fma(Gy, c6, f2_add(f2_sub(f2_add(f2_add(f2_fma(m2, d3, f[6]), d5), d6), d7), n_d8));
    f[7] = f2_fma(Gy, m6, f2_add(f2_add(f2_add(f2_sub(f2_fma(m2, d3, f[7]), d5), d6), d7), n_d8));
    f[8] = f2_fma(Gy, m6, f2_add(f2_add(f2_sub(f2_add(f2_fma(m2, d3, f[8]), d5), d6), d7), n_d8));

    const F2 n1 = f2_sub(g[1], g[3]), n_n2 = f2_sub(g[4], g[2]);
    const F2 n3 = f2_fma(m4, g[0], f2_add(f2_add(f2_add(g[1], g[2]), g[3]), g[4]));
    const F2 n4 = f2_sub(f2_add(g[1], g[3]), f2_add(g[2], g[4]));
    const F2 j1 = f2_fma(n_u, theta, n1), n_j2 = f2_fma(v, theta, n_n2);
    const F2 e3 = f2_mul(K.se20, f2_fma(K.n_a, theta, n3));
    g[0] = f2_fma(c4, e3, g[0]);
    g[1] = f2_fma(K.n_snu4t, n4, f2_sub(f2_fma(K.n_sk2, j1, g[1]), e3));
    g[2] = f2_fma(K.snu4t, n4, f2_sub(f2_fma(K.sk2, n_j2, g[2]), e3));
    g[3] = f2_fma(K.n_snu4t, n4, f2_sub(f2_fma(K.sk2, j1, g[3]), e3));
    g[4] = f2_fma(K.snu4t, n4, f2_sub(f2_fma(K.n_sk2, n_j2, g[4]), e3));

    rho_out = rho;
    theta_out = theta;
}

}  // namespace dmrt
