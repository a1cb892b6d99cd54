// pair_math.cuh - FP32 arithmetic on two values per register pair
// (add / mul / fma.rn.f32x2: one instruction issued for two nodes), and the
// collision of d3q19.cuh on two nodes at a time.
//
// Each lane of a packed operation rounds like the scalar one, and
// collide_pair() performs the operations of collide() in the same order and
// with the same fusions, so both give the same bits (pinned by the tests
// that compare the step kernels bit for bit). The collision is about 190 of
// the 280-330 instructions of a node update; two nodes at a time issue half.
#pragma once

#include "d3q19.cuh"

namespace lbm {

struct P2 {
  unsigned long long v;
};

__device__ __forceinline__ P2 pk(float a, float b) {
  P2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ P2 pk(float a) { return pk(a, a); }
__device__ __forceinline__ float2 unpk(P2 a) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a.v));
  return r;
}
__device__ __forceinline__ P2 operator+(P2 a, P2 b) {
  P2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ P2 operator*(P2 a, P2 b) {
  P2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ P2 fma2(P2 a, P2 b, P2 c) {
  P2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}

// Constants of collide_pair(), both halves alike: in a kernel parameter they
// are read from the constant bank as operands and take no registers.
struct PairConsts {
  P2 one, minus1, m15, k45;  // 1, -1, -3/2, 9/2
  P2 keep, cA, ncA, cB, ncB; // 1 - omega, +-omega/6, +-omega/12
  P2 ow0, owA, owB;          // omega w_i
  // body force (Guo): 1/2, -3, 9, 1 - omega/2, w_i, 3 w_i, -3 w_i
  P2 half, m3, nine, kf, w0, wA, wB, w3A, w3B, nw3A, nw3B;
};

__host__ __device__ inline PairConsts pair_consts(float omega, float kf) {
  auto both = [](float v) {
    union {
      float f[2];
      unsigned long long u;
    } x;
    x.f[0] = x.f[1] = v;
    return P2{x.u};
  };
  const float cB = omega * (1.0f / 12.0f), cA = 2.0f * cB;
  return {both(1.0f),          both(-1.0f), both(-1.5f), both(4.5f),
          both(1.0f - omega),  both(cA),    both(-cA),   both(cB),
          both(-cB),           both(omega * weight(0)), both(omega * weight(1)),
          both(omega * weight(7)),
          both(0.5f),          both(-3.0f), both(9.0f),  both(kf),
          both(weight(0)),     both(weight(1)),          both(weight(7)),
          both(3.0f * weight(1)),                        both(3.0f * weight(7)),
          both(-(3.0f * weight(1))),                     both(-(3.0f * weight(7)))};
}

// collide() on two nodes; F: the body force (FORCE).
template <bool FORCE>
__device__ __forceinline__ void collide_pair(P2 (&d)[Q], const PairConsts &c, const P2 (&F)[3],
                                             P2 &rho, P2 &ux, P2 &uy, P2 &uz) {
  // a - b: the product -b is exact, so one rounding
  auto sub = [&](P2 a, P2 b) { return fma2(b, c.minus1, a); };
  auto along = [&](P2 x, P2 y, P2 z, auto I) {  // e_i . (x, y, z)
    constexpr int i = decltype(I)::value, ex = kEx[i], ey = kEy[i], ez = kEz[i];
    if constexpr (ex != 0 && ey != 0)
      return ex * ey > 0 ? x + y : ex > 0 ? sub(x, y) : sub(y, x);
    else if constexpr (ex != 0 && ez != 0)
      return ex * ez > 0 ? x + z : ex > 0 ? sub(x, z) : sub(z, x);
    else if constexpr (ey != 0 && ez != 0)
      return ey * ez > 0 ? y + z : ey > 0 ? sub(y, z) : sub(z, y);
    else
      return ex != 0 ? x : ey != 0 ? y : z;
  };
  const P2 dr = ((d[0] + (d[1] + d[2])) + ((d[3] + d[4]) + (d[5] + d[6]))) +
                (((d[7] + d[8]) + (d[9] + d[10])) + ((d[11] + d[12]) + (d[13] + d[14]))) +
                ((d[15] + d[16]) + (d[17] + d[18]));
  const P2 d78 = sub(d[7], d[8]), d910 = sub(d[9], d[10]), d1516 = sub(d[15], d[16]);
  const P2 d1112 = sub(d[11], d[12]), d1314 = sub(d[13], d[14]), d1718 = sub(d[17], d[18]);
  // x + (b - a) is x - (a - b): negation is exact
  P2 jx = sub((sub(d[1], d[2]) + d78) + (d910 + d1516), d1718);
  P2 jy = (sub(d[3], d[4]) + d78) + sub(d1112, d910) + d1314;
  P2 jz = (sub(d[5], d[6]) + d1112) + sub(d1516, d1314) + d1718;
  rho = c.one + dr;
  const float2 r = unpk(rho);
  const P2 rinv = pk(__frcp_rn(r.x), __frcp_rn(r.y));
  if constexpr (FORCE) {
    jx = fma2(c.half, F[0], jx);
    jy = fma2(c.half, F[1], jy);
    jz = fma2(c.half, F[2], jz);
  }
  ux = jx * rinv;
  uy = jy * rinv;
  uz = jz * rinv;
  const P2 jsq = fma2(jx, jx, fma2(jy, jy, jz * jz));
  const P2 base = fma2(c.m15 * jsq, rinv, dr);
  const P2 k45 = c.k45 * rinv;
  const P2 bA = c.owA * base, bB = c.owB * base;
  const P2 kA = c.owA * k45, kB = c.owB * k45;
  P2 m3uF, k9;
  if constexpr (FORCE) {
    m3uF = c.m3 * fma2(ux, F[0], fma2(uy, F[1], uz * F[2]));
    k9 = c.nine * rinv;
  }
  d[0] = fma2(c.keep, d[0], c.ow0 * base);
  if constexpr (FORCE) d[0] = fma2(c.kf, c.w0 * m3uF, d[0]);
  static_for<0, 9>([&](auto P) {
    constexpr int i = 2 * decltype(P)::value + 1;
    constexpr int j = i + 1;
    const P2 b = i < 7 ? bA : bB, k = i < 7 ? kA : kB;
    const P2 es = along(jx, jy, jz, std::integral_constant<int, i>{});
    const P2 even = fma2(es * es, k, b);
    P2 vi = fma2(c.keep, d[i], fma2(i < 7 ? c.cA : c.cB, es, even));
    P2 vj = fma2(c.keep, d[j], fma2(i < 7 ? c.ncA : c.ncB, es, even));
    if constexpr (FORCE) {
      const P2 eF = along(F[0], F[1], F[2], std::integral_constant<int, i>{});
      const P2 s = fma2(k9 * es, eF, m3uF);  // 9 (e.u)(e.F) - 3 u.F
      const P2 ws = (i < 7 ? c.wA : c.wB) * s;
      vi = fma2(c.kf, fma2(i < 7 ? c.w3A : c.w3B, eF, ws), vi);
      vj = fma2(c.kf, fma2(i < 7 ? c.nw3A : c.nw3B, eF, ws), vj);
    }
    d[i] = vi;
    d[j] = vj;
  });
}

}  // namespace lbm
