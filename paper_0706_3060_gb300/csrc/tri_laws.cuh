// tri_laws.cuh -- the pair interactions of tri_kernel.cuh: each unordered pair
// evaluated once for two targets at a time (the halves of the f32x2 values) against
// one source.
//
// A law gives the words of a particle (kWords: as a target two particles' words are
// packed in float2, as a source they are broadcast to both halves), the number of
// sums per particle (kSums) and the pair function
//   pair<MASK, SRC>(S, T, A, J, e2, k0, k1)
// which adds the target-side terms of both targets to A and the source-side terms to
// J (the even target's to J[2 c], the odd target's to J[2 c + 1]). MASK: a half counts
// only when its k0 / k1 is set. SRC false: the target side alone (a row's own groups,
// direct_kernel.cuh). kFlip bit c: the source-side term of sum c has the opposite sign
// (Newton's third law), applied when J is stored. kChunk, kParts: lengths of the plain sums;
// kFine, kLow: compensated sums and the potential's low parts (tri_kernel.cuh, Sums).
//
// The streamed kernels read the particles' words with ordinary loads: the finalize in front
// of them lets them be placed early (griddep_launch) and writes positions, velocities and
// lambda while they are, and only ordinary loads are ordered by griddep_start; the
// non-coherent ones (__ldg, NC) want memory that nobody writes as long as the kernel lives.
// The direct kernels, in front of which nothing triggers early, live only after the last
// write, and read through that path (Hermite steps of 1000 particles 7.2 us, with ordinary
// loads 7.7). Parameters are written by no kernel of a chain.
//
// The source-side sums are plain floats updated with scalar fused multiply-adds: they
// are added up and handed from lane to lane one word at a time (tri_kernel.cuh), and
// with three register operands the packed instruction loses time to register banks
// (measured, cycles per packed instruction: two operands 2.06, three 2.45; the scalar
// one 1.25 to 1.3 with three).
#pragma once

#include "device_common.cuh"

namespace nbody {

template <bool NC>
__device__ __forceinline__ float4 load4(const float4 *p) {
  return NC ? __ldg(p) : *p;
}

__device__ __forceinline__ float2 bcast(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 neg2(float2 v) { return make_float2(-v.x, -v.y); }

__device__ __forceinline__ float2 rsqrt2(float2 s, bool precise) {
  float2 y = make_float2(rsqrt_hw(s.x), rsqrt_hw(s.y));
  if (precise) {
    const float2 hs = __fmul2_rn(s, bcast(-0.5f));
    y = __fmul2_rn(y, __ffma2_rn(hs, __fmul2_rn(y, y), bcast(1.5f)));
  }
  return y;
}

// J[0], J[1] += w * d, half by half.
__device__ __forceinline__ void jfma(float *J, float2 w, float2 d) {
  J[0] = __fmaf_rn(w.x, d.x, J[0]);
  J[1] = __fmaf_rn(w.y, d.y, J[1]);
}
__device__ __forceinline__ void jadd(float *J, float2 v) {
  J[0] = __fadd_rn(J[0], v.x);
  J[1] = __fadd_rn(J[1], v.y);
}

// Softened gravity (Eq. 1): words x, y, z, m; sums m y^3 d (and m y with POT).
template <bool POT, bool PRECISE, bool FINE>
struct TriGrav {
  static constexpr int kWords = 4;
  static constexpr int kSums = POT ? 4 : 3;
  static constexpr unsigned kFlip = 0x7;
  static constexpr bool kFine = FINE, kLow = FINE && POT;
  static constexpr int kChunk = FINE ? 8 : 16, kParts = FINE ? 2 : 1;
  // words of particle i, or of the massless pad far away
  template <bool NC = false>
  static __device__ __forceinline__ void load(const float4 *p0, const float4 *, const float4 *,
                                              int i, int n, float (&w)[kWords]) {
    const float4 p = i < n ? load4<NC>(p0 + i) : make_float4(1e18f, 1e18f, 1e18f, 0.0f);
    w[0] = p.x;
    w[1] = p.y;
    w[2] = p.z;
    w[3] = p.w;
  }
  // target words as the pair function wants them (positions negated)
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
    float2 y = rsqrt2(s2, PRECISE);
    if (MASK) {
      y.x = k0 ? y.x : 0.0f;
      y.y = k1 ? y.y : 0.0f;
    }
    const float2 y3 = __fmul2_rn(__fmul2_rn(y, y), y);
    const float2 wi = __fmul2_rn(bcast(S[3]), y3);  // source mass: pull on the target
    A[0] = __ffma2_rn(wi, dx, A[0]);
    A[1] = __ffma2_rn(wi, dy, A[1]);
    A[2] = __ffma2_rn(wi, dz, A[2]);
    if (POT) A[kSums - 1] = __ffma2_rn(bcast(S[3]), y, A[kSums - 1]);
    if (!SRC) return;
    float2 wj = __fmul2_rn(T[3], y3);  // target mass: pull on the source
    jfma(J, wj, dx);
    jfma(J + 2, wj, dy);
    jfma(J + 4, wj, dz);
    if (POT) jfma(J + 2 * (kSums - 1), T[3], y);
  }
};

// Lennard-Jones + Coulomb (Table 1, constant or linear dielectric): words x, y, z,
// q~, s~, e~; sums f d (and the pair energy with POT), as in force_kernel.cuh.
template <bool LIN, bool POT, bool PRECISE>
struct TriLjc {
  static constexpr int kWords = 6;
  static constexpr int kSums = POT ? 4 : 3;
  static constexpr unsigned kFlip = 0x7;
  static constexpr bool kFine = false, kLow = false;
  static constexpr int kChunk = 16, kParts = 1;
  template <bool NC = false>
  static __device__ __forceinline__ void load(const float4 *p0, const float4 *p1, const float4 *,
                                              int i, int n, float (&w)[kWords]) {
    const float4 p = i < n ? load4<NC>(p0 + i) : make_float4(1e18f, 1e18f, 1e18f, 0.0f);
    const float4 q = i < n ? __ldg(p1 + i) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    w[0] = p.x;
    w[1] = p.y;
    w[2] = p.z;
    w[3] = q.x;
    w[4] = q.y;
    w[5] = q.z;
  }
  static __device__ __forceinline__ void as_target(float (&w)[kWords]) {
    w[0] = -w[0];
    w[1] = -w[1];
    w[2] = -w[2];
  }
  template <bool MASK, bool SRC = true>
  static __device__ __forceinline__ void pair(const float (&S)[kWords], const float2 (&T)[kWords],
                                              float2 (&A)[kSums], float (&J)[2 * kSums], float2,
                                              bool k0 = true, bool k1 = true) {
    const float2 dx = __fadd2_rn(bcast(S[0]), T[0]);
    const float2 dy = __fadd2_rn(bcast(S[1]), T[1]);
    const float2 dz = __fadd2_rn(bcast(S[2]), T[2]);
    float2 r2 = __fmul2_rn(dz, dz);
    r2 = __ffma2_rn(dy, dy, r2);
    r2 = __ffma2_rn(dx, dx, r2);
    float2 y = rsqrt2(r2, PRECISE);
    if (MASK) {
      y.x = k0 ? y.x : 0.0f;
      y.y = k1 ? y.y : 0.0f;
    }
    const float2 y2 = __fmul2_rn(y, y);
    const float2 qq = __fmul2_rn(bcast(S[3]), T[3]);
    const float2 s = __fadd2_rn(bcast(S[4]), T[4]);
    const float2 t = __fmul2_rn(__fmul2_rn(s, s), y2);
    const float2 u = __fmul2_rn(__fmul2_rn(t, t), t);
    const float2 ee = __fmul2_rn(bcast(S[5]), T[5]);
    const float2 fc = LIN ? __fmul2_rn(__fmul2_rn(qq, y2), __fadd2_rn(y2, y2))
                          : __fmul2_rn(__fmul2_rn(qq, y), y2);
    const float2 h = __fmul2_rn(__ffma2_rn(u, bcast(2.0f), bcast(-1.0f)), u);
    const float2 f = __ffma2_rn(__fmul2_rn(ee, y2), h, fc);
    A[0] = __ffma2_rn(f, dx, A[0]);
    A[1] = __ffma2_rn(f, dy, A[1]);
    A[2] = __ffma2_rn(f, dz, A[2]);
    if (SRC) {
      const float2 fj = f;
      jfma(J, fj, dx);
      jfma(J + 2, fj, dy);
      jfma(J + 4, fj, dz);
    }
    if (POT) {
      float2 e = __fmul2_rn(qq, LIN ? y2 : y);
      e = __ffma2_rn(__fmul2_rn(ee, bcast(1.0f / 6.0f)), __ffma2_rn(u, u, neg2(u)), e);
      A[kSums - 1] = __fadd2_rn(A[kSums - 1], e);
      if (SRC) jadd(J + 2 * (kSums - 1), e);
    }
  }
};

}  // namespace nbody
