// tri_vjp_laws.cuh -- the pair interactions of the acceleration + jerk evaluation and
// of the force VJPs for tri_kernel.cuh, in the form that tri_laws.cuh describes (each
// unordered pair once, two targets at a time). The terms and their order of evaluation
// are those of vjp_kernel.cuh; third particle array: velocities, or lambda.
#pragma once

#include "tri_laws.cuh"

namespace nbody {

// Words x, y, z, m of particle i and three more from its element of `p2`.
template <bool NC>
__device__ __forceinline__ void load_pos_and(const float4 *p0, const float4 *p2, int i, int n,
                                             float (&w)[7]) {
  const float4 p = i < n ? load4<NC>(p0 + i) : make_float4(1e18f, 1e18f, 1e18f, 0.0f);
  const float4 v = i < n ? load4<NC>(p2 + i) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  w[0] = p.x;
  w[1] = p.y;
  w[2] = p.z;
  w[3] = p.w;
  w[4] = v.x;
  w[5] = v.y;
  w[6] = v.z;
}

// Acceleration and jerk (Table 1 GAJ): d = x_j - x_k, u = v_j - v_k, y = 1/s,
// t = u - 3 y^2 (d.u) d; the target's sums are m_j y^3 d and m_j y^3 t, the source's
// -m_k y^3 d and -m_k y^3 t: 33 FP32 lane operations for both.
struct TriJerk {
  static constexpr int kWords = 7;
  static constexpr int kSums = 6;
  static constexpr unsigned kFlip = 0x3f;
  static constexpr bool kFine = false, kLow = false;
  static constexpr int kChunk = 16, kParts = 1;
  template <bool NC = false>
  static __device__ __forceinline__ void load(const float4 *p0, const float4 *, const float4 *p2,
                                              int i, int n, float (&w)[kWords]) {
    load_pos_and<NC>(p0, p2, i, n, w);
  }
  static __device__ __forceinline__ void as_target(float (&w)[kWords]) {
#pragma unroll
    for (int c = 0; c < kWords; ++c)
      if (c != 3) w[c] = -w[c];
  }
  template <bool MASK, bool SRC = true>
  static __device__ __forceinline__ void pair(const float (&S)[kWords], const float2 (&T)[kWords],
                                              float2 (&A)[kSums], float (&J)[2 * kSums],
                                              float2 e2, bool k0 = true, bool k1 = true) {
    const float2 dx = __fadd2_rn(bcast(S[0]), T[0]);
    const float2 dy = __fadd2_rn(bcast(S[1]), T[1]);
    const float2 dz = __fadd2_rn(bcast(S[2]), T[2]);
    const float2 ux = __fadd2_rn(bcast(S[4]), T[4]);
    const float2 uy = __fadd2_rn(bcast(S[5]), T[5]);
    const float2 uz = __fadd2_rn(bcast(S[6]), T[6]);
    float2 s2 = __ffma2_rn(dz, dz, e2);
    s2 = __ffma2_rn(dy, dy, s2);
    s2 = __ffma2_rn(dx, dx, s2);
    float2 y = rsqrt2(s2, false);
    if (MASK) {
      y.x = k0 ? y.x : 0.0f;
      y.y = k1 ? y.y : 0.0f;
    }
    const float2 y2 = __fmul2_rn(y, y);
    const float2 y3 = __fmul2_rn(y2, y);
    const float2 wi = __fmul2_rn(bcast(S[3]), y3);
    const float2 du = __ffma2_rn(dx, ux, __ffma2_rn(dy, uy, __fmul2_rn(dz, uz)));
    const float2 c = __fmul2_rn(du, __fmul2_rn(y2, bcast(-3.0f)));
    const float2 tx = __ffma2_rn(c, dx, ux);
    const float2 ty = __ffma2_rn(c, dy, uy);
    const float2 tz = __ffma2_rn(c, dz, uz);
    A[0] = __ffma2_rn(wi, dx, A[0]);
    A[1] = __ffma2_rn(wi, dy, A[1]);
    A[2] = __ffma2_rn(wi, dz, A[2]);
    A[3] = __ffma2_rn(wi, tx, A[3]);
    A[4] = __ffma2_rn(wi, ty, A[4]);
    A[5] = __ffma2_rn(wi, tz, A[5]);
    if (!SRC) return;
    float2 wj = __fmul2_rn(T[3], y3);
    jfma(J, wj, dx);
    jfma(J + 2, wj, dy);
    jfma(J + 4, wj, dz);
    jfma(J + 6, wj, tx);
    jfma(J + 8, wj, ty);
    jfma(J + 10, wj, tz);
  }
};

// Gravity VJP: w = m_k lam_j - m_j lam_k; the target's sums are
// y^3 (w - 3 y^2 (d.w) d) and (lam_j.d) y^3, the source's -y^3 (w - ...) and
// -(lam_k.d) y^3: 35 FP32 lane operations for both.
template <bool FINE>
struct TriGravVjp {
  static constexpr int kWords = 7;
  static constexpr int kSums = 4;
  static constexpr unsigned kFlip = 0xf;
  static constexpr bool kFine = FINE, kLow = false;
  static constexpr int kChunk = FINE ? 4 : 16, kParts = FINE ? 4 : 1;
  template <bool NC = false>
  static __device__ __forceinline__ void load(const float4 *p0, const float4 *, const float4 *p2,
                                              int i, int n, float (&w)[kWords]) {
    load_pos_and<NC>(p0, p2, i, n, w);
  }
  static __device__ __forceinline__ void as_target(float (&w)[kWords]) {
    w[0] = -w[0];
    w[1] = -w[1];
    w[2] = -w[2];
  }
  template <bool MASK, bool SRC = true>
  static __device__ __forceinline__ void pair(const float (&S)[kWords], const float2 (&T)[kWords],
                                              float2 (&A)[kSums], float (&J)[2 * kSums],
                                              float2 e2, bool k0 = true, bool k1 = true) {
    const float2 dx = __fadd2_rn(bcast(S[0]), T[0]);
    const float2 dy = __fadd2_rn(bcast(S[1]), T[1]);
    const float2 dz = __fadd2_rn(bcast(S[2]), T[2]);
    float2 s2 = __ffma2_rn(dz, dz, e2);
    s2 = __ffma2_rn(dy, dy, s2);
    s2 = __ffma2_rn(dx, dx, s2);
    float2 y = rsqrt2(s2, false);
    if (MASK) {
      y.x = k0 ? y.x : 0.0f;
      y.y = k1 ? y.y : 0.0f;
    }
    const float2 y2 = __fmul2_rn(y, y);
    const float2 y3 = __fmul2_rn(y2, y);
    const float2 nm = bcast(-S[3]);
    const float2 wx = __ffma2_rn(T[3], bcast(S[4]), __fmul2_rn(nm, T[4]));
    const float2 wy = __ffma2_rn(T[3], bcast(S[5]), __fmul2_rn(nm, T[5]));
    const float2 wz = __ffma2_rn(T[3], bcast(S[6]), __fmul2_rn(nm, T[6]));
    const float2 lj = __ffma2_rn(bcast(S[4]), dx,
                                 __ffma2_rn(bcast(S[5]), dy, __fmul2_rn(bcast(S[6]), dz)));
    const float2 lk = __ffma2_rn(T[4], dx, __ffma2_rn(T[5], dy, __fmul2_rn(T[6], dz)));
    const float2 dw = __ffma2_rn(T[3], lj, __fmul2_rn(nm, lk));
    const float2 c = __fmul2_rn(dw, __fmul2_rn(y2, bcast(-3.0f)));
    const float2 vx = __ffma2_rn(c, dx, wx);
    const float2 vy = __ffma2_rn(c, dy, wy);
    const float2 vz = __ffma2_rn(c, dz, wz);
    A[0] = __ffma2_rn(y3, vx, A[0]);
    A[1] = __ffma2_rn(y3, vy, A[1]);
    A[2] = __ffma2_rn(y3, vz, A[2]);
    A[3] = __ffma2_rn(lj, y3, A[3]);
    if (!SRC) return;
    const float2 yj = y3;
    jfma(J, yj, vx);
    jfma(J + 2, yj, vy);
    jfma(J + 4, yj, vz);
    jfma(J + 6, yj, lk);
  }
};

// LJ + Coulomb VJP (LIN: linear dielectric): words x, y, z, q~, s~, e~ and -u
// (u = lam / m); sums A (phi w + 2 phi' (d.w) d and the sigma term) and B (phi d and the
// epsilon term), as in vjp_kernel.cuh. The type terms are the same for both particles
// (d and w both change sign): 64 FP32 lane operations for both.
template <bool LIN>
struct TriLjcVjp {
  static constexpr int kWords = 9;
  static constexpr int kSums = 8;
  static constexpr unsigned kFlip = 0x77;
  static constexpr bool kFine = false, kLow = false;
  static constexpr int kChunk = 16, kParts = 1;
  template <bool NC = false>
  static __device__ __forceinline__ void load(const float4 *p0, const float4 *p1,
                                              const float4 *p2, int i, int n,
                                              float (&w)[kWords]) {
    const float4 p = i < n ? load4<NC>(p0 + i) : make_float4(1e18f, 1e18f, 1e18f, 0.0f);
    const float4 q = i < n ? __ldg(p1 + i) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    const float4 l = i < n ? load4<NC>(p2 + i) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    const float inv = i < n ? 1.0f / p.w : 0.0f;
    w[0] = p.x;
    w[1] = p.y;
    w[2] = p.z;
    w[3] = q.x;
    // pads and atoms without a radius: k2 below is 0, and 1 / s has to be finite (kept here,
    // once per load; a clamp in the pair function takes 1% of the kernel)
    w[4] = q.y == 0.0f ? 1e-30f : q.y;
    w[5] = q.z;
    w[6] = -(l.x * inv);
    w[7] = -(l.y * inv);
    w[8] = -(l.z * inv);
  }
  static __device__ __forceinline__ void as_target(float (&w)[kWords]) {
#pragma unroll
    for (int c = 0; c < kWords; ++c)
      if (c < 3 || c > 5) w[c] = -w[c];
  }
  template <bool MASK, bool SRC = true>
  static __device__ __forceinline__ void pair(const float (&S)[kWords], const float2 (&T)[kWords],
                                              float2 (&A)[kSums], float (&J)[2 * kSums], float2,
                                              bool k0 = true, bool k1 = true) {
    const float2 dx = __fadd2_rn(bcast(S[0]), T[0]);
    const float2 dy = __fadd2_rn(bcast(S[1]), T[1]);
    const float2 dz = __fadd2_rn(bcast(S[2]), T[2]);
    const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
    float2 y = rsqrt2(r2, false);
    if (MASK) {
      y.x = k0 ? y.x : 0.0f;
      y.y = k1 ? y.y : 0.0f;
    }
    const float2 y2 = __fmul2_rn(y, y);
    const float2 qq = __fmul2_rn(T[3], bcast(S[3]));
    const float2 s = __fadd2_rn(T[4], bcast(S[4]));
    const float2 ee = __fmul2_rn(T[5], bcast(S[5]));
    const float2 t = __fmul2_rn(__fmul2_rn(s, s), y2);
    const float2 u = __fmul2_rn(__fmul2_rn(t, t), t);
    const float2 qy3 = LIN ? __fmul2_rn(__fmul2_rn(qq, y2), __fadd2_rn(y2, y2))
                           : __fmul2_rn(qq, __fmul2_rn(y, y2));
    const float2 eey2 = __fmul2_rn(ee, y2);
    const float2 h = __fmul2_rn(__ffma2_rn(u, bcast(2.0f), bcast(-1.0f)), u);
    const float2 phi_lj = __fmul2_rn(eey2, h);
    const float2 phi = __fadd2_rn(phi_lj, qy3);
    const float2 k1v = __fmul2_rn(__ffma2_rn(u, bcast(-28.0f), bcast(8.0f)), u);
    const float2 tp = __fmul2_rn(
        y2, __ffma2_rn(eey2, k1v, __fmul2_rn(bcast(LIN ? -4.0f : -3.0f), qy3)));
    const float2 wx = __fadd2_rn(T[6], bcast(S[6]));
    const float2 wy = __fadd2_rn(T[7], bcast(S[7]));
    const float2 wz = __fadd2_rn(T[8], bcast(S[8]));
    const float2 dw = __ffma2_rn(dx, wx, __ffma2_rn(dy, wy, __fmul2_rn(dz, wz)));
    const float2 c = __fmul2_rn(tp, dw);
    const float2 k2 = __fmul2_rn(__ffma2_rn(u, bcast(4.0f), bcast(-1.0f)), u);
    float2 rs = make_float2(rcp_hw(s.x), rcp_hw(s.y));
    if (MASK) {
      rs.x = k0 ? rs.x : 0.0f;
      rs.y = k1 ? rs.y : 0.0f;
    }
    const float2 st = __fmul2_rn(__fmul2_rn(eey2, k2), rs);
    A[0] = __ffma2_rn(c, dx, __ffma2_rn(phi, wx, A[0]));
    A[1] = __ffma2_rn(c, dy, __ffma2_rn(phi, wy, A[1]));
    A[2] = __ffma2_rn(c, dz, __ffma2_rn(phi, wz, A[2]));
    A[3] = __ffma2_rn(dw, st, A[3]);
    A[4] = __ffma2_rn(phi, dx, A[4]);
    A[5] = __ffma2_rn(phi, dy, A[5]);
    A[6] = __ffma2_rn(phi, dz, A[6]);
    A[7] = __ffma2_rn(dw, phi_lj, A[7]);
    if (!SRC) return;
    const float2 cj = c, pj = phi;
    const float2 dj = dw;
    jfma(J, pj, wx);
    jfma(J, cj, dx);
    jfma(J + 2, pj, wy);
    jfma(J + 2, cj, dy);
    jfma(J + 4, pj, wz);
    jfma(J + 4, cj, dz);
    jfma(J + 6, dj, st);
    jfma(J + 8, pj, dx);
    jfma(J + 10, pj, dy);
    jfma(J + 12, pj, dz);
    jfma(J + 14, dj, phi_lj);
  }
};

}  // namespace nbody
