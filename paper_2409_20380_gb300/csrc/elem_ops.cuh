// Element arithmetic shared by the element-by-element kernels: values of one case (float, double) or of a pair of
// adjacent cases of a node (float2, Blackwell's paired FP32 operations: one instruction, two cases; scalars are
// broadcast to both halves), and the products of the linear and the quadratic tet on them.
#pragma once

#include "fem_internal.cuh"

namespace fem {

__device__ __forceinline__ float2 bc2(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }

// Fixed-point sums: a bound below 2^E takes the scale 2^(30 - E) in and 2^(E - 30) back.  E is at least -96, so that both
// are normal FP32 numbers and their product is one (with each clamped by itself, sums of a bound below 2^-97 came back
// doubled); a smaller bound's sums are then exact to 2^-127, half of FP32's smallest normal number, below which FP32
// atomics flush to zero.  pow2 clamps to the normal range.
__device__ __forceinline__ float pow2(int e) { return __uint_as_float((uint32_t)min(max(e + 127, 1), 254) << 23); }
__device__ __forceinline__ int fixed_expo(float bound) {   // (bound < 2^(exponent field - 126))
  return max((int)((__float_as_uint(bound) >> 23) & 0xffu) - 126, -96);
}

template <typename V> struct ScalarOf { using type = V; };
template <> struct ScalarOf<float2> { using type = float; };
template <typename V> __device__ __forceinline__ V vzero() { return (V)0; }
template <> __device__ __forceinline__ float2 vzero<float2>() { return make_float2(0.f, 0.f); }
__device__ __forceinline__ float vneg(float a) { return -a; }
__device__ __forceinline__ double vneg(double a) { return -a; }
__device__ __forceinline__ float2 vneg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float vadd(float a, float b) { return a + b; }
__device__ __forceinline__ double vadd(double a, double b) { return a + b; }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return add2(a, b); }
__device__ __forceinline__ float vsub(float a, float b) { return a - b; }
__device__ __forceinline__ double vsub(double a, double b) { return a - b; }
__device__ __forceinline__ float2 vsub(float2 a, float2 b) { return sub2(a, b); }
__device__ __forceinline__ float vmul(float a, float b) { return a * b; }
__device__ __forceinline__ double vmul(double a, double b) { return a * b; }
__device__ __forceinline__ float2 vmul(float2 a, float b) { return mul2(a, bc2(b)); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double vfma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float2 vfma(float2 a, float b, float2 c) { return fma2(a, bc2(b), c); }
__device__ __forceinline__ float vfmv(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double vfmv(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float2 vfmv(float2 a, float2 b, float2 c) { return fma2(a, b, c); }

// sigma = lam tr(G) I + mu (G + G^T)
template <typename V, typename S>
__device__ __forceinline__ void stress(const V (&G)[3][3], S lam, S mu, V (&T)[3][3]) {
  const V ltr = vmul(vadd(vadd(G[0][0], G[1][1]), G[2][2]), lam);
  const S mu2 = mu + mu;
#pragma unroll
  for (int i = 0; i < 3; ++i) T[i][i] = vfma(G[i][i], mu2, ltr);
  T[0][1] = T[1][0] = vmul(vadd(G[0][1], G[1][0]), mu);
  T[0][2] = T[2][0] = vmul(vadd(G[0][2], G[2][0]), mu);
  T[1][2] = T[2][1] = vmul(vadd(G[1][2], G[2][1]), mu);
}

// Linear tet: ld(a, P) gives corner a's values, fl(a, Q) takes its sums; r the element record.  TWO: ld gives the
// values M acts on, ldk those K acts on.
template <bool DOT, bool TWO, typename V, typename S, typename LD, typename LDK, typename FL>
__device__ __forceinline__ void elem4(LD ld, LDK ldk, FL fl, const S (&r)[12], S aM, S aK, V& hd) {
  const S lam = aK * r[9], mu = aK * r[10], ms = aM * r[11];
  V P[4][3];
#pragma unroll
  for (int a = 0; a < 4; ++a) ld(a, P[a]);
  V U[4][3], G[3][3], T[3][3];
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    if (TWO) ldk(a, U[a]);
#pragma unroll
    for (int k = 0; k < 3; ++k)
      if (!TWO) U[a][k] = P[a][k];
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const V d1 = vsub(U[1][i], U[0][i]), d2 = vsub(U[2][i], U[0][i]), d3 = vsub(U[3][i], U[0][i]);
#pragma unroll
    for (int j = 0; j < 3; ++j) G[i][j] = vfma(d3, r[6 + j], vfma(d2, r[3 + j], vmul(d1, r[j])));
  }
  stress(G, lam, mu, T);
  V sum[3], fs[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    sum[k] = vadd(vadd(P[0][k], P[1][k]), vadd(P[2][k], P[3][k]));
  }
#pragma unroll
  for (int a = 1; a < 5; ++a) {
    V Q[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const V m = vadd(P[a & 3][k], sum[k]);
      if (a < 4) {
        const V F = vfma(T[k][2], r[3 * a - 1], vfma(T[k][1], r[3 * a - 2], vmul(T[k][0], r[3 * a - 3])));
        fs[k] = a == 1 ? F : vadd(fs[k], F);
        Q[k] = vfma(m, ms, F);
      } else {   // corner 0: minus the sum of the others' stiffness parts
        Q[k] = vfma(m, ms, vneg(fs[k]));
      }
      if (DOT) hd = vfmv(P[a & 3][k], Q[k], hd);
    }
    fl(a & 3, Q);
  }
}

// Quadratic tet (straight-sided, constant barycentric gradients g_a): the strain is linear over the element, so
// it is given by its values at the four corners, and with int L_c L_d dV = V (1 + delta_cd) / 20 the stiffness
// product is exact as
//   G_c = sum_a W_a^c (x) g_a,  W_c^c = 3 p_c,  W_a^c = 4 p_ca - p_a (a != c; p_ca the edge node),
//   S_c = sigma(G_c + sum_d G_d) V / 20,  T_a^c = S_c g_a,
//   f_c += 3 T_c^c,  f_a -= T_a^c,  f_ca += 4 T_a^c  (a != c),
// where sum_d G_d = 4 sum_a (sum of a's three edge nodes) (x) g_a needs no corner values.  About 610 operations
// with the mass against 820 for the sums over the four Gauss points (the same integral: the integrand is quadratic).
// Edges 4 .. 9: (0,1) (1,2) (0,2) (0,3) (1,3) (2,3).
__host__ __device__ constexpr int edge_node10(int a, int b) {   // (sum and product tell the six pairs apart)
  return a + b == 1 ? 4 : a + b == 2 ? 6 : a + b == 4 ? 8 : a + b == 5 ? 9 : a * b == 2 ? 5 : 7;
}
template <bool DOT, typename V, typename S, typename LD, typename FL>
__device__ __forceinline__ void elem10(LD ld, FL fl, const S (&r)[12], S aM, S aK, V& hd) {
  V P[10][3], Q[10][3], Gs[3][3];
#pragma unroll
  for (int i = 0; i < 10; ++i) ld(i, P[i]);
  // four times V / 20 (T below is four times T_a^c), rho V / 420
  const S lam = aK * r[9] * (S)0.2, mu = aK * r[10] * (S)0.2, rv = aM * r[11] * (S)(20.0 / 420.0);
  // consistent mass, 420 m_ij = 6 / 1 (corner diagonal / other corner), -4 / -6 (corner and an edge through it /
  // the others), 32 / 16 / 8 (edge diagonal / an edge sharing a corner / the opposite edge):
  //   corner a:      5 p_a + Sc - 6 Se + 2 Ea,   edge (a, b):  -6 Sc + 2 (p_a + p_b) + 16 Se + 16 p_ab - 8 p_opposite
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const V Sc = vadd(vadd(P[0][k], P[1][k]), vadd(P[2][k], P[3][k]));
    const V Se = vadd(vadd(vadd(P[4][k], P[5][k]), vadd(P[6][k], P[7][k])), vadd(P[8][k], P[9][k]));
    const V bc = vfma(Se, (S)-6, Sc), be = vfma(Sc, (S)-6, vmul(Se, (S)16));
    V Ea[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const int b0 = a == 0 ? 1 : 0, b1 = a <= 1 ? 2 : 1, b2 = a <= 2 ? 3 : 2;
      Ea[a] = vadd(vadd(P[edge_node10(a, b0)][k], P[edge_node10(a, b1)][k]), P[edge_node10(a, b2)][k]);
      Q[a][k] = vmul(vfma(P[a][k], (S)5, vfma(Ea[a], (S)2, bc)), rv);
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = a + 1; b < 4; ++b) {
        const int e = edge_node10(a, b), o = a == 0 ? (b == 1 ? 9 : b == 2 ? 8 : 5) : a == 1 ? (b == 2 ? 7 : 6) : 4;
        Q[e][k] = vmul(vfma(vadd(P[a][k], P[b][k]), (S)2, vfma(P[e][k], (S)16, vfma(P[o][k], (S)-8, be))), rv);
      }
    V D[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) D[a] = vmul(vsub(Ea[a + 1], Ea[0]), (S)4);
#pragma unroll
    for (int j = 0; j < 3; ++j) Gs[k][j] = vfma(D[2], r[6 + j], vfma(D[1], r[3 + j], vmul(D[0], r[j])));
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    V G[3][3], T[3][3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const V W0 = c == 0 ? vmul(P[0][k], (S)3) : vfma(P[edge_node10(c, c == 0 ? 1 : 0)][k], (S)4, vneg(P[0][k]));
      V D[3];
#pragma unroll
      for (int a = 1; a < 4; ++a)
        D[a - 1] = a == c ? vsub(vmul(P[a][k], (S)3), W0) : vsub(vfma(P[edge_node10(a, c == a ? 0 : c)][k], (S)4, vneg(P[a][k])), W0);
#pragma unroll
      for (int j = 0; j < 3; ++j) G[k][j] = vfma(D[2], r[6 + j], vfma(D[1], r[3 + j], vfma(D[0], r[j], Gs[k][j])));
    }
    stress(G, lam, mu, T);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      V F[4];
#pragma unroll
      for (int a = 1; a < 4; ++a)
        F[a] = vfma(T[k][2], r[3 * a - 1], vfma(T[k][1], r[3 * a - 2], vmul(T[k][0], r[3 * a - 3])));
      F[0] = vneg(vadd(vadd(F[1], F[2]), F[3]));
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        if (a == c) {
          Q[a][k] = vfma(F[a], (S)0.75, Q[a][k]);
        } else {
          Q[a][k] = vfma(F[a], (S)-0.25, Q[a][k]);
          const int e = edge_node10(a, c == a ? (a == 0 ? 1 : 0) : c);
          Q[e][k] = vadd(Q[e][k], F[a]);
        }
      }
    }
  }
#pragma unroll
  for (int i = 0; i < 10; ++i) {
    if (DOT)
#pragma unroll
      for (int k = 0; k < 3; ++k) hd = vfmv(P[i][k], Q[i][k], hd);
    fl(i, Q[i]);
  }
}

// The 12 values of an element record.
__device__ __forceinline__ void load_rec(const float* __restrict__ src, float (&r)[12]) {
  const float4* s4 = reinterpret_cast<const float4*>(src);
  const float4 a = __ldg(s4), b = __ldg(s4 + 1), c = __ldg(s4 + 2);
  r[0] = a.x; r[1] = a.y; r[2] = a.z; r[3] = a.w;
  r[4] = b.x; r[5] = b.y; r[6] = b.z; r[7] = b.w;
  r[8] = c.x; r[9] = c.y; r[10] = c.z; r[11] = c.w;
}
__device__ __forceinline__ void load_rec(const double* __restrict__ src, double (&r)[12]) {
  const double2* s2 = reinterpret_cast<const double2*>(src);
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const double2 v = __ldg(s2 + i);
    r[2 * i] = v.x;
    r[2 * i + 1] = v.y;
  }
}

}  // namespace fem
