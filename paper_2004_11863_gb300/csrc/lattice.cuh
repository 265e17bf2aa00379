// Velocity sets and the Hermite-equilibrium / collision arithmetic of the
// level update, evaluated in binary32 on shifted populations
// g_i = f_i - f0_i(rho0, U): deviations from the equilibrium of a reference
// state (rho0, U).  With U = 0 this is the rest-state shift f_i - w_i rho0;
// a reference velocity near the flow's mean velocity keeps the stored values
// (and every rounding of them) small where the flow is close to it.  All
// arithmetic below is written in the deviations drho = rho - rho0 and
// du = u - U, so that no large terms cancel.
//
// Lattices: D2Q9 in the velocity order of Sec. 3.1 (eqs. xi_i, w_i); D3Q19
// and D3Q27 built the same way (weights 1/3, 1/18, 1/36 and 8/27, 2/27, 1/54,
// 1/216).  c_s^2 = 1/3 on all three.
//
// Equilibrium (eq. fEqH truncated at third order, eq. fEqO3 in 2D):
//   f0_i = w_i rho [1 + 3 xi.u + 4.5 (xi.u)^2 - 1.5 u.u + T3_i(u u u)],
// where T3 is the lattice-supported third-order Hermite term set:
//   D2Q9:  H_xxy, H_xyy with 1/(2 cs^6);
//   D3Q27: the six H_aab with 1/(2 cs^6) and H_xyz with 1/cs^6;
//   D3Q19: for each odd axis b the orthogonal pair H_aab +- H_ccb, with
//          1/(2 cs^6) on the sum and 1/(6 cs^6) on the difference
//          (H_aab and H_ccb are not orthogonal on D3Q19 and H_xyz vanishes).
// Regularized collisions (eqs. reguProcedure, a1Proj, LBMscheme_reg, f1RR,
// a13RR): a1 = sum H2 (f - f0) is formed directly from the shifted second
// moment, a1_ab = sum xi_a xi_b g - rho u_a u_b - drho cs^2 delta_ab, and the
// post-collision state is f0 + (1 - 1/tau) f1 with
//   f1_i = w_i [4.5 H2_i : a1 + T3_i(a1^(3))],
//   a1^(3)_abc = u_a a1_bc + u_b a1_ac + u_c a1_ab   (RR; zero for REG).
#pragma once
#include <cuda_fp16.h>

#include <type_traits>
#include <utility>

namespace mlbm {

// ---------------------------------------------------------------- unrolling
template <class F, int... I>
__host__ __device__ __forceinline__ void sfor_impl(F&& f, std::integer_sequence<int, I...>) {
  (f(std::integral_constant<int, I>{}), ...);
}
template <int N, class F>
__host__ __device__ __forceinline__ void sfor(F&& f) {
  sfor_impl(f, std::make_integer_sequence<int, N>{});
}

// ------------------------------------------------------------------ lattices
struct D2Q9 {
  static constexpr int Q = 9, D = 2, ID = 0;
  __host__ __device__ static constexpr int c(int i, int a) {
    constexpr int t[9][3] = {{0, 0, 0},  {1, 0, 0},  {0, 1, 0},   {-1, 0, 0}, {0, -1, 0},
                             {1, 1, 0},  {-1, 1, 0}, {-1, -1, 0}, {1, -1, 0}};
    return t[i][a];
  }
  __host__ __device__ static constexpr double w(int i) {
    return i == 0 ? 4.0 / 9.0 : (i < 5 ? 1.0 / 9.0 : 1.0 / 36.0);
  }
};

// 3D sets: rest, then the 6 axis neighbours, then the 12 edge neighbours,
// then (D3Q27) the 8 corners; opposite pairs are adjacent (i, i+1) after 0.
struct D3Q19 {
  static constexpr int Q = 19, D = 3, ID = 1;
  __host__ __device__ static constexpr int c(int i, int a) {
    constexpr int t[19][3] = {{0, 0, 0},  {1, 0, 0},  {-1, 0, 0}, {0, 1, 0},   {0, -1, 0},
                              {0, 0, 1},  {0, 0, -1}, {1, 1, 0},  {-1, -1, 0}, {1, -1, 0},
                              {-1, 1, 0}, {1, 0, 1},  {-1, 0, -1}, {1, 0, -1}, {-1, 0, 1},
                              {0, 1, 1},  {0, -1, -1}, {0, 1, -1}, {0, -1, 1}};
    return t[i][a];
  }
  __host__ __device__ static constexpr double w(int i) {
    return i == 0 ? 1.0 / 3.0 : (i < 7 ? 1.0 / 18.0 : 1.0 / 36.0);
  }
};

struct D3Q27 {
  static constexpr int Q = 27, D = 3, ID = 2;
  __host__ __device__ static constexpr int c(int i, int a) {
    constexpr int t[27][3] = {
        {0, 0, 0},   {1, 0, 0},   {-1, 0, 0},  {0, 1, 0},   {0, -1, 0},  {0, 0, 1},  {0, 0, -1},
        {1, 1, 0},   {-1, -1, 0}, {1, -1, 0},  {-1, 1, 0},  {1, 0, 1},   {-1, 0, -1}, {1, 0, -1},
        {-1, 0, 1},  {0, 1, 1},   {0, -1, -1}, {0, 1, -1},  {0, -1, 1},  {1, 1, 1},  {-1, -1, -1},
        {1, 1, -1},  {-1, -1, 1}, {1, -1, 1},  {-1, 1, -1}, {-1, 1, 1},  {1, -1, -1}};
    return t[i][a];
  }
  __host__ __device__ static constexpr double w(int i) {
    return i == 0 ? 8.0 / 27.0 : (i < 7 ? 2.0 / 27.0 : (i < 19 ? 1.0 / 54.0 : 1.0 / 216.0));
  }
};

template <class L>
__host__ __device__ constexpr int opp(int i) {
  int k = 0;
  for (int j = 0; j < L::Q; ++j)
    if (L::c(j, 0) == -L::c(i, 0) && L::c(j, 1) == -L::c(i, 1) && L::c(j, 2) == -L::c(i, 2)) k = j;
  return k;
}

// Directions come in opposite pairs (i, opp(i)); pair_first<L>(p) is the
// lower index of the p-th pair, p = 0 .. (Q-1)/2 - 1.
template <class L>
__host__ __device__ constexpr int pair_first(int p) {
  int k = 0;
  for (int i = 1; i < L::Q; ++i)
    if (i < opp<L>(i)) {
      if (k == p) return i;
      ++k;
    }
  return -1;
}

// Third-order Hermite polynomial H_aab(xi_i) = xi_a^2 xi_b - cs^2 xi_b.
template <class L>
__host__ __device__ constexpr double h3(int i, int a, int b) {
  return double(L::c(i, a) * L::c(i, a) * L::c(i, b)) - double(L::c(i, b)) / 3.0;
}

// Third-order coefficient set, indexed [xxy, xxz, yyx, yyz, zzx, zzy, xyz].
enum { XXY = 0, XXZ, YYX, YYZ, ZZX, ZZY, XYZ };

// T3_i(A): the lattice-supported third-order term of the Hermite expansion
// for coefficients A (already including every factor except w_i).
template <class L, int I, class T>
__host__ __device__ __forceinline__ T third(const T (&A)[7]) {
  if constexpr (L::ID == 0) {
    constexpr T hxxy = T(13.5 * h3<L>(I, 0, 1)), hyyx = T(13.5 * h3<L>(I, 1, 0));
    return hxxy * A[XXY] + hyyx * A[YYX];
  } else if constexpr (L::ID == 2) {
    constexpr T k0 = T(13.5 * h3<L>(I, 0, 1)), k1 = T(13.5 * h3<L>(I, 0, 2)),
                k2 = T(13.5 * h3<L>(I, 1, 0)), k3 = T(13.5 * h3<L>(I, 1, 2)),
                k4 = T(13.5 * h3<L>(I, 2, 0)), k5 = T(13.5 * h3<L>(I, 2, 1)),
                k6 = T(27.0 * L::c(I, 0) * L::c(I, 1) * L::c(I, 2));
    return k0 * A[XXY] + k1 * A[XXZ] + k2 * A[YYX] + k3 * A[YYZ] + k4 * A[ZZX] + k5 * A[ZZY] +
           k6 * A[XYZ];
  } else {
    // odd axis y: (xxy, zzy); odd axis x: (yyx, zzx); odd axis z: (xxz, yyz)
    constexpr T py = T(13.5 * (h3<L>(I, 0, 1) + h3<L>(I, 2, 1))),
                my = T(4.5 * (h3<L>(I, 0, 1) - h3<L>(I, 2, 1)));
    constexpr T px = T(13.5 * (h3<L>(I, 1, 0) + h3<L>(I, 2, 0))),
                mx = T(4.5 * (h3<L>(I, 1, 0) - h3<L>(I, 2, 0)));
    constexpr T pz = T(13.5 * (h3<L>(I, 0, 2) + h3<L>(I, 1, 2))),
                mz = T(4.5 * (h3<L>(I, 0, 2) - h3<L>(I, 1, 2)));
    return py * (A[XXY] + A[ZZY]) + my * (A[XXY] - A[ZZY]) + px * (A[YYX] + A[ZZX]) +
           mx * (A[YYX] - A[ZZX]) + pz * (A[XXZ] + A[YYZ]) + mz * (A[XXZ] - A[YYZ]);
  }
}

// w_i * x without a systematic bias: binary32 cannot hold 1/9, 1/36, ...
// exactly, and a rounded weight would shift the equilibrium's mass and
// momentum by the same relative amount at every update (a drift that adds up
// over long runs).  The weight is split into a binary32 head and tail.
template <class L, int I, class T>
__host__ __device__ __forceinline__ T wmul(T x) {
  if constexpr (std::is_same<T, float>::value) {
    constexpr float hi = float(L::w(I));
    constexpr float lo = float(L::w(I) - double(hi));
    return fmaf(hi, x, lo * x);
  } else {
    return T(L::w(I)) * x;
  }
}

// xi_i . v with compile-time components.
template <class L, int I, class T>
__host__ __device__ __forceinline__ T cdot(T vx, T vy, T vz) {
  T s = T(0);
  if constexpr (L::c(I, 0) == 1) s += vx;
  if constexpr (L::c(I, 0) == -1) s -= vx;
  if constexpr (L::c(I, 1) == 1) s += vy;
  if constexpr (L::c(I, 1) == -1) s -= vy;
  if constexpr (L::D == 3) {
    if constexpr (L::c(I, 2) == 1) s += vz;
    if constexpr (L::c(I, 2) == -1) s -= vz;
  }
  return s;
}

// Macroscopic moments of shifted populations: drho = sum g, j = sum xi g.
template <class L, class T>
__host__ __device__ __forceinline__ void moments(const T (&g)[L::Q], T& drho, T& jx, T& jy,
                                                 T& jz) {
  drho = jx = jy = jz = T(0);
  sfor<L::Q>([&](auto I) {
    constexpr int i = decltype(I)::value;
    drho += g[i];
    if constexpr (L::c(i, 0) == 1) jx += g[i];
    if constexpr (L::c(i, 0) == -1) jx -= g[i];
    if constexpr (L::c(i, 1) == 1) jy += g[i];
    if constexpr (L::c(i, 1) == -1) jy -= g[i];
    if constexpr (L::c(i, 2) == 1) jz += g[i];
    if constexpr (L::c(i, 2) == -1) jz -= g[i];
  });
}

// Third-order coefficients of u (A) and their deviations from those of U
// (dA = A(u) - A(U)), in the order [xxy, xxz, yyx, yyz, zzx, zzy, xyz].
template <class T>
__host__ __device__ __forceinline__ void third_coeffs(T ux, T uy, T uz, T dux, T duy, T duz,
                                                      T Ux, T Uy, T Uz, T (&A)[7], T (&dA)[7]) {
  A[XXY] = ux * ux * uy;
  A[XXZ] = ux * ux * uz;
  A[YYX] = uy * uy * ux;
  A[YYZ] = uy * uy * uz;
  A[ZZX] = uz * uz * ux;
  A[ZZY] = uz * uz * uy;
  A[XYZ] = ux * uy * uz;
  // a^2 b - A^2 B = da (a + A) b + A^2 db
  dA[XXY] = dux * (ux + Ux) * uy + Ux * Ux * duy;
  dA[XXZ] = dux * (ux + Ux) * uz + Ux * Ux * duz;
  dA[YYX] = duy * (uy + Uy) * ux + Uy * Uy * dux;
  dA[YYZ] = duy * (uy + Uy) * uz + Uy * Uy * duz;
  dA[ZZX] = duz * (uz + Uz) * ux + Uz * Uz * dux;
  dA[ZZY] = duz * (uz + Uz) * uy + Uz * Uz * duy;
  dA[XYZ] = dux * uy * uz + Ux * (duy * uz + Uy * duz);
}

// Equilibrium deviation for direction I (FP64: the reference's own values in
// the population read-out; the steps use expand below):
//   g0_i = f0_i(rho0 + drho, U + du) - f0_i(rho0, U)
//        = w_i [ drho (1 + e_i(u)) + rho0 (e_i(u) - e_i(U)) ],
//   e_i(u) = 3 xi.u + 4.5 (xi.u)^2 - 1.5 u.u + T3_i(u u u),
//   e_i(u) - e_i(U) = 3 xi.du + 4.5 (xi.du)(xi.u + xi.U) - 1.5 du.(u + U) + T3_i(dA).
template <class L, int I, class T>
__host__ __device__ __forceinline__ T eq_dev_i(T drho, T rho0, T ux, T uy, T uz, T dux, T duy,
                                               T duz, T Ux, T Uy, T Uz, T usq, T dusq,
                                               const T (&A)[7], const T (&dA)[7]) {
  const T cu = cdot<L, I>(ux, uy, uz);
  const T cdu = cdot<L, I>(dux, duy, duz);
  const T cU = cdot<L, I>(Ux, Uy, Uz);
  const T e = T(3) * cu + T(4.5) * cu * cu - usq + third<L, I>(A);
  const T de = T(3) * cdu + T(4.5) * cdu * (cu + cU) - dusq + third<L, I>(dA);
  return wmul<L, I>(drho * (T(1) + e) + rho0 * de);
}

// All q equilibrium deviations at (rho0 + drho, U + du).
template <class L, class T>
__host__ __device__ __forceinline__ void equilibrium_dev(T drho, T dux, T duy, T duz, T rho0,
                                                         T Ux, T Uy, T Uz, T (&g0)[L::Q]) {
  if constexpr (L::D == 2) {
    duz = T(0);
    Uz = T(0);
  }
  const T ux = Ux + dux, uy = Uy + duy, uz = Uz + duz;
  T A[7], dA[7];
  third_coeffs(ux, uy, uz, dux, duy, duz, Ux, Uy, Uz, A, dA);
  const T usq = T(1.5) * (ux * ux + uy * uy + uz * uz);
  const T dusq = T(1.5) * (dux * (ux + Ux) + duy * (uy + Uy) + duz * (uz + Uz));
  sfor<L::Q>([&](auto I) {
    constexpr int i = decltype(I)::value;
    g0[i] = eq_dev_i<L, i>(drho, rho0, ux, uy, uz, dux, duy, duz, Ux, Uy, Uz, usq, dusq, A, dA);
  });
}

// ------------------------------------------------------- two-lane binary32
// Two independent binary32 values in the packed FP32 instructions (one issue
// slot for both lanes): two nodes, or the two runs of an interleaved pair.
// Each lane rounds like the scalar operation.
struct F2 {
  float2 v;
};

// The arithmetic below is written once over T = float or F2.
template <class T>
__device__ __forceinline__ T bc(float a) {
  if constexpr (std::is_same<T, F2>::value)
    return {make_float2(a, a)};
  else
    return T(a);
}
__device__ __forceinline__ float vfma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ F2 vfma(F2 a, F2 b, F2 c) { return {__ffma2_rn(a.v, b.v, c.v)}; }
__device__ __forceinline__ F2 operator+(F2 a, F2 b) { return {__fadd2_rn(a.v, b.v)}; }
__device__ __forceinline__ F2 operator*(F2 a, F2 b) { return {__fmul2_rn(a.v, b.v)}; }
// a - b, one instruction: b * (-1) is exact, the sum is rounded once
__device__ __forceinline__ F2 operator-(F2 a, F2 b) {
  return {__ffma2_rn(b.v, make_float2(-1.0f, -1.0f), a.v)};
}
// k x + y with a compile-time or warp-uniform binary32 factor
template <class T>
__device__ __forceinline__ T kfma(float k, T x, T y) { return vfma(bc<T>(k), x, y); }
template <class T>
__device__ __forceinline__ T kmul(float k, T x) { return bc<T>(k) * x; }

// 1 / x, correctly rounded: the bits of the IEEE division for every x, zero,
// infinity and subnormal numbers included (compared for every non-negative
// binary32 number).  The hardware's approximation r (one ulp) and one third-order
// Newton-Schulz step, r + r (e + e e) with e = 1 - x r exact; the second-order
// step misses a few subnormal quotients by their last bit.  Where r is zero or
// infinite e is no residual, and r itself is the quotient.  __frcp_rn gives the
// same bits and costs 1.6 % of a step in the mean of 37 kinds of run (4 to 7 %
// of the binary16 BGK ones); this form 0.1 % over the bare second-order step.
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float vrcp(float x) {
  const float r = rcp_approx(x), e = fmaf(-x, r, 1.0f);
  return fabsf(e) < 1.0f ? fmaf(r, fmaf(e, e, e), r) : r;
}
__device__ __forceinline__ F2 vrcp(F2 x) {
  const F2 r = {make_float2(rcp_approx(x.v.x), rcp_approx(x.v.y))};
  const F2 e = vfma(bc<F2>(-1.0f) * x, r, bc<F2>(1.0f));
  const F2 y = vfma(r, vfma(e, e, e), r);
  return {make_float2(fabsf(e.v.x) < 1.0f ? y.v.x : r.v.x, fabsf(e.v.y) < 1.0f ? y.v.y : r.v.y)};
}

// x / N without a systematic bias: 1 / N as a binary32 head and tail (a
// rounded constant would shift mass or momentum by the same relative amount
// at every update, a drift that adds up over long runs).
template <int N, class T>
__device__ __forceinline__ T over(T x) {
  constexpr float hi = float(1.0 / N);
  constexpr float lo = float(1.0 / N - double(hi));
  return vfma(bc<T>(hi), x, kmul(lo, x));
}

// Index of direction (x, y, z).
template <class L>
__host__ __device__ constexpr int dir(int x, int y, int z) {
  for (int i = 0; i < L::Q; ++i)
    if (L::c(i, 0) == x && L::c(i, 1) == y && L::c(i, 2) == z) return i;
  return -1;
}

// Second-order components, in this order.
enum { XX = 0, YY, ZZ, XY, XZ, YZ };

// Moments of a population set: d = sum g, j = sum xi g, P = sum xi xi g.
// Opposite directions enter only through their sum (even moments) and
// difference (odd ones).
template <class L, class T>
__device__ __forceinline__ void moments2(const T (&g)[L::Q], T& d, T (&j)[3],
                                                  T (&P)[6]) {
  auto even = [&](auto X, auto Y, auto Z) {
    constexpr int x = decltype(X)::value, y = decltype(Y)::value, z = decltype(Z)::value;
    return g[dir<L>(x, y, z)] + g[dir<L>(-x, -y, -z)];
  };
  auto odd = [&](auto X, auto Y, auto Z) {
    constexpr int x = decltype(X)::value, y = decltype(Y)::value, z = decltype(Z)::value;
    return g[dir<L>(x, y, z)] - g[dir<L>(-x, -y, -z)];
  };
  constexpr std::integral_constant<int, 0> o{};
  constexpr std::integral_constant<int, 1> p{};
  constexpr std::integral_constant<int, -1> m{};
  const T sx = even(p, o, o), dx = odd(p, o, o), sy = even(o, p, o), dy = odd(o, p, o);
  const T s1 = even(p, p, o), d1 = odd(p, p, o), s2 = even(p, m, o), d2 = odd(p, m, o);
  const T sxy = s1 + s2;
  if constexpr (L::D == 2) {
    P[XX] = sx + sxy;
    P[YY] = sy + sxy;
    P[XY] = s1 - s2;
    P[ZZ] = P[XZ] = P[YZ] = bc<T>(0.0f);
    d = (g[0] + sx) + P[YY];
    j[0] = dx + (d1 + d2);
    j[1] = dy + (d1 - d2);
    j[2] = bc<T>(0.0f);
  } else {
    const T sz = even(o, o, p), dz = odd(o, o, p);
    const T s3 = even(p, o, p), d3 = odd(p, o, p), s4 = even(p, o, m), d4 = odd(p, o, m);
    const T s5 = even(o, p, p), d5 = odd(o, p, p), s6 = even(o, p, m), d6 = odd(o, p, m);
    const T sxz = s3 + s4, syz = s5 + s6;
    T ax = sx, ay = sy, az = sz;
    P[XY] = s1 - s2;
    P[XZ] = s3 - s4;
    P[YZ] = s5 - s6;
    d = ((g[0] + sx) + (sy + sz)) + ((sxy + sxz) + syz);
    j[0] = (dx + (d1 + d2)) + (d3 + d4);
    j[1] = (dy + (d1 - d2)) + (d5 + d6);
    j[2] = (dz + (d3 - d4)) + (d5 - d6);
    if constexpr (L::Q == 27) {
      // corners (1,1,1), (1,1,-1), (1,-1,1), (-1,1,1) and their opposites
      const T c1 = even(p, p, p), e1 = odd(p, p, p), c2 = even(p, p, m), e2 = odd(p, p, m);
      const T c3 = even(p, m, p), e3 = odd(p, m, p), c4 = even(m, p, p), e4 = odd(m, p, p);
      const T c12 = c1 + c2, c34 = c3 + c4, b12 = c1 - c2, b34 = c3 - c4, c = c12 + c34;
      ax = ax + c;
      ay = ay + c;
      az = az + c;
      d = d + c;
      P[XY] = P[XY] + (c12 - c34);
      P[XZ] = P[XZ] + (b12 + b34);
      P[YZ] = P[YZ] + (b12 - b34);
      const T e12 = e1 + e2, e34 = e3 - e4;
      j[0] = j[0] + (e12 + e34);
      j[1] = j[1] + (e12 - e34);
      j[2] = j[2] + ((e1 - e2) + (e3 + e4));
    }
    P[XX] = ax + (sxy + sxz);
    P[YY] = ay + (sxy + syz);
    P[ZZ] = az + (sxz + syz);
  }
}

// Populations of a Hermite expansion (eq. fEqH to third order): direction i
// of  w_i [d + 3 xi.j + 4.5 H2_i:B + T3_i(A)],  each handed to
// emit(integral_constant<i>, value).  Takes C = A / 4 (order XXY .. XYZ).
// The coefficients are folded with the weights, which leaves powers of two
// and a few thirds (over<N>): a direction costs two to four operations
// instead of a polynomial of its own.
//   D2Q9, D3Q19: opposite directions share E +- O.  Along an axis
//     O = j_a / 6 ... - A_bba / 2 (- A_cca / 2), on an edge
//     (j_a / 3 + A_bba) / 4 +- (j_b / 3 + A_aab) / 4.
//   D3Q27: the raw moments M_pqr (p, q, r <= 2) of the expansion, halved
//     once per axis with a nonzero power, then one axis at a time
//     g_0 = M_0 - 2 M_2, g_+- = M_2 +- M_1.
template <class L, class T, class Emit>
__device__ __forceinline__ void expand(T d, const T (&j)[3], const T (&B)[6],
                                                const T (&C)[7], Emit&& emit) {
  // the pair (x, y, z) and its opposite from the even and the odd part, k O
  auto pair = [&](auto X, auto Y, auto Z, T even, float k, T odd) {
    constexpr int x = decltype(X)::value, y = decltype(Y)::value, z = decltype(Z)::value;
    emit(std::integral_constant<int, dir<L>(x, y, z)>{}, kfma(k, odd, even));
    emit(std::integral_constant<int, dir<L>(-x, -y, -z)>{}, kfma(-k, odd, even));
  };
  constexpr std::integral_constant<int, 0> o{};
  constexpr std::integral_constant<int, 1> p{};
  constexpr std::integral_constant<int, -1> m{};
  const T jx = over<12>(j[0]), jy = over<12>(j[1]);
  if constexpr (L::Q == 9) {
    const T d9 = over<9>(d), t3 = over<3>(B[XX] + B[YY]);
    emit(std::integral_constant<int, 0>{}, kfma(-2.0f, t3, kmul(4.0f, d9)));
    const T ax = kfma(-0.5f, t3, d9), c = kmul(0.25f, d9 + t3);
    pair(p, o, o, kfma(0.5f, B[XX], ax), 4.0f, kfma(-0.5f, C[YYX], jx));
    pair(o, p, o, kfma(0.5f, B[YY], ax), 4.0f, kfma(-0.5f, C[XXY], jy));
    const T X = jx + C[YYX], Y = jy + C[XXY];
    pair(p, p, o, kfma(0.25f, B[XY], c), 1.0f, X + Y);
    pair(p, m, o, kfma(-0.25f, B[XY], c), 1.0f, X - Y);
  } else if constexpr (L::Q == 19) {
    const T jz = over<12>(j[2]);
    const T s9 = over<9>(kfma(-1.5f, (B[XX] + B[YY]) + B[ZZ], d));
    emit(std::integral_constant<int, 0>{}, kmul(3.0f, s9));
    const T a = kmul(0.5f, s9), e = kmul(0.25f, s9);
    pair(p, o, o, kfma(0.25f, B[XX], a), 2.0f, jx - (C[YYX] + C[ZZX]));
    pair(o, p, o, kfma(0.25f, B[YY], a), 2.0f, jy - (C[XXY] + C[ZZY]));
    pair(o, o, p, kfma(0.25f, B[ZZ], a), 2.0f, jz - (C[XXZ] + C[YYZ]));
    auto edge = [&](auto X1, auto Y1, auto Z1, auto X2, auto Y2, auto Z2, T Baa, T Bbb, T Bab,
                    T X, T Y) {
      const T c = kfma(0.125f, Bbb, kfma(0.125f, Baa, e));
      pair(X1, Y1, Z1, kfma(0.25f, Bab, c), 1.0f, X + Y);
      pair(X2, Y2, Z2, kfma(-0.25f, Bab, c), 1.0f, X - Y);
    };
    edge(p, p, o, p, m, o, B[XX], B[YY], B[XY], jx + C[YYX], jy + C[XXY]);
    edge(p, o, p, p, o, m, B[XX], B[ZZ], B[XZ], jx + C[ZZX], jz + C[XXZ]);
    edge(o, p, p, o, p, m, B[YY], B[ZZ], B[YZ], jy + C[ZZY], jz + C[YYZ]);
  } else {
    const T jz = over<12>(j[2]);
    T M[3][3][3];  // [p][q][r]
    const T d3 = over<3>(d), d9 = over<9>(d);
    const T qx = over<3>(B[XX]), qy = over<3>(B[YY]), qz = over<3>(B[ZZ]);
    M[0][0][0] = d;
    M[1][0][0] = kmul(0.5f, j[0]);
    M[0][1][0] = kmul(0.5f, j[1]);
    M[0][0][1] = kmul(0.5f, j[2]);
    M[2][0][0] = kmul(0.5f, B[XX] + d3);
    M[0][2][0] = kmul(0.5f, B[YY] + d3);
    M[0][0][2] = kmul(0.5f, B[ZZ] + d3);
    M[1][1][0] = kmul(0.25f, B[XY]);
    M[1][0][1] = kmul(0.25f, B[XZ]);
    M[0][1][1] = kmul(0.25f, B[YZ]);
    const T qxy = (qx + qy) + d9;
    M[2][2][0] = kmul(0.25f, qxy);
    M[2][0][2] = kmul(0.25f, (qx + qz) + d9);
    M[0][2][2] = kmul(0.25f, (qy + qz) + d9);
    M[2][2][2] = over<24>(qxy + qz);
    M[2][1][0] = C[XXY] + jy;
    M[2][0][1] = C[XXZ] + jz;
    M[1][2][0] = C[YYX] + jx;
    M[0][2][1] = C[YYZ] + jz;
    M[1][0][2] = C[ZZX] + jx;
    M[0][1][2] = C[ZZY] + jy;
    M[1][1][1] = kmul(0.5f, C[XYZ]);
    M[2][2][1] = over<6>(M[2][0][1] + C[YYZ]);
    M[2][1][2] = over<6>(M[2][1][0] + C[ZZY]);
    M[1][2][2] = over<6>(M[1][2][0] + C[ZZX]);
    M[2][1][1] = over<24>(B[YZ]);
    M[1][2][1] = over<24>(B[XZ]);
    M[1][1][2] = over<24>(B[XY]);
    auto inv = [](T& a, T& b, T& c) {  // (M_0, M_1, M_2) -> (g_-, g_0, g_+)
      const T m1 = b, m2 = c;
      b = kfma(-2.0f, m2, a);
      a = m2 - m1;
      c = m2 + m1;
    };
#pragma unroll
    for (int q = 0; q < 3; ++q)
#pragma unroll
      for (int r = 0; r < 3; ++r) inv(M[0][q][r], M[1][q][r], M[2][q][r]);
#pragma unroll
    for (int x = 0; x < 3; ++x)
#pragma unroll
      for (int r = 0; r < 3; ++r) inv(M[x][0][r], M[x][1][r], M[x][2][r]);
    sfor<9>([&](auto K) {
      constexpr int x = decltype(K)::value / 3, y = decltype(K)::value % 3;
      inv(M[x][y][0], M[x][y][1], M[x][y][2]);
      emit(std::integral_constant<int, dir<L>(x - 1, y - 1, -1)>{}, M[x][y][0]);
      emit(std::integral_constant<int, dir<L>(x - 1, y - 1, 0)>{}, M[x][y][1]);
      emit(std::integral_constant<int, dir<L>(x - 1, y - 1, 1)>{}, M[x][y][2]);
    });
  }
}

// Reference state (rho0, U) of the shifted storage in binary32, with the
// products the deviations need, formed on the host in double precision.
struct RefF {
  float rho0;
  float U[3];
  float m[3];  // rho0 U_a
  float k[4];  // rho0 U_a U_a / 4, and rho0 U_x U_y / 4
};

// Second- and third-order deviations of the equilibrium from the reference,
//   dP_ab  = rho u_a u_b - rho0 U_a U_b = j_a u_b + rho0 U_a du_b,
//   dA_aab = rho u_a u_a u_b - rho0 U_a U_a U_b = dP_aa u_b + rho0 U_a U_a du_b,
// with j = rho u - rho0 U: no large terms cancel.  MOV = false: U = 0.
template <class L, bool MOV, class T>
__device__ __forceinline__ void second_dev(const T (&j)[3], const T (&u)[3],
                                                    const T (&du)[3], const RefF& R,
                                                    T (&dP)[6]) {
  auto prod = [&](int a, int b) {
    const T x = MOV ? kmul(R.m[a], du[b]) : bc<T>(0.0f);
    return MOV ? vfma(j[a], u[b], x) : j[a] * u[b];
  };
  dP[XX] = prod(0, 0);
  dP[YY] = prod(1, 1);
  dP[XY] = prod(0, 1);
  dP[ZZ] = dP[XZ] = dP[YZ] = bc<T>(0.0f);
  if constexpr (L::D == 3) {
    dP[ZZ] = prod(2, 2);
    dP[XZ] = prod(0, 2);
    dP[YZ] = prod(1, 2);
  }
}

// Third-order coefficients over four, C_aab = (V_aab + 2 u_a W_ab) / 4 with
// V_aab = Q_aa u_b + rho0 U_a U_a du_b (W_ab = 0: the equilibrium's own
// dA / 4 for Q = dP): with Q = dP + a1, W = a1 this is
// dA + a1^(3) of eq. a13RR, (a1^(3)_aab = 2 u_a a1_ab + u_b a1_aa).
template <class L, bool MOV, bool W1, class T>
__device__ __forceinline__ void third_dev(const T (&Q)[6], const T (&W)[6],
                                                   const T (&u)[3], const T (&du)[3],
                                                   const RefF& R, T (&C)[7]) {
  T uq[3], uh[3];
#pragma unroll
  for (int a = 0; a < L::D; ++a) {
    uq[a] = kmul(0.25f, u[a]);
    uh[a] = kmul(0.5f, u[a]);
  }
  auto aab = [&](int a, int b, int aa, int ab) {
    T c = bc<T>(0.0f);
    if constexpr (MOV) c = kmul(R.k[a], du[b]);
    if constexpr (W1) c = MOV ? vfma(uh[a], W[ab], c) : uh[a] * W[ab];
    return (MOV || W1) ? vfma(uq[b], Q[aa], c) : uq[b] * Q[aa];
  };
  C[XXY] = aab(0, 1, XX, XY);
  C[YYX] = aab(1, 0, YY, XY);
  if constexpr (L::D == 3) {
    C[XXZ] = aab(0, 2, XX, XZ);
    C[YYZ] = aab(1, 2, YY, YZ);
    C[ZZX] = aab(2, 0, ZZ, XZ);
    C[ZZY] = aab(2, 1, ZZ, YZ);
    if constexpr (L::Q == 27) {
      T c = bc<T>(0.0f);
      if constexpr (MOV) c = kmul(R.k[3], du[2]);
      if constexpr (W1) {
        c = MOV ? vfma(uq[0], W[YZ], c) : uq[0] * W[YZ];
        c = vfma(uq[1], W[XZ], c);
      }
      C[XYZ] = (MOV || W1) ? vfma(uq[2], Q[XY], c) : uq[2] * Q[XY];
    }
  }
}

// Equilibrium deviations f0(rho0 + drho, U + du) - f0(rho0, U), direction by
// direction to emit(integral_constant<i>, value).
template <class L, class Emit>
__device__ __forceinline__ void equilibrium_emit(float drho, float dux, float duy,
                                                          float duz, const RefF& R, Emit&& emit) {
  const float du[3] = {dux, duy, L::D == 3 ? duz : 0.0f};
  float u[3], j[3], dP[6], C[7];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    u[a] = R.U[a] + du[a];
    j[a] = fmaf(drho, u[a], R.rho0 * du[a]);
  }
  second_dev<L, true>(j, u, du, R, dP);
  third_dev<L, true, false>(dP, dP, u, du, R, C);
  expand<L>(drho, j, dP, C, emit);
}

// All q equilibrium deviations (binary32) at (rho0 + drho, U + du).
template <class L>
__device__ __forceinline__ void equilibrium_f(float drho, float dux, float duy, float duz,
                                                       const RefF& R, float (&g0)[L::Q]) {
  equilibrium_emit<L>(drho, dux, duy, duz, R,
                      [&](auto I, float v) { g0[decltype(I)::value] = v; });
}

// Density and velocity deviations of shifted populations:
// drho = sum g, du = (sum xi g - drho U) / (rho0 + drho).
template <class L>
__device__ __forceinline__ void deviations(const float (&g)[L::Q], const RefF& R, float& drho,
                                           float& dux, float& duy, float& duz) {
  float jx, jy, jz;
  moments<L>(g, drho, jx, jy, jz);
  const float inv = vrcp(R.rho0 + drho);
  dux = (jx - drho * R.U[0]) * inv;
  duy = (jy - drho * R.U[1]) * inv;
  duz = (L::D == 3) ? (jz - drho * R.U[2]) * inv : 0.0f;
}

// Strain-rate input of the hybrid collision (eq. a1ij_HRR):
// a1 <- sig a1 + ks rho S with ks = -2 tau cs^2 (1 - sig);
// s = (S_xx, S_yy, S_zz, S_xy, S_xz, S_yz).
template <class T>
struct HrrIn {
  float sig, ks;
  T s[6];
};

// Collision of shifted populations; the post-collision value of each
// direction is handed to emit(integral_constant<i>, value) as soon as it is
// formed, so no array of outputs (or of equilibria) stays live.
// COLL: 0 BGK (eq. BGKmodel), 1 REG (eq. LBMscheme_reg with H^(2) only),
// 2 RR (eqs. f1RR, a13RR), 3 H-RR (eq. a1ij_HRR, then the RR recursion;
// needs hy).  omega = 1 - 1/tau.
// MOV = false: the reference velocity is zero (rest-state shift) and every
// term in U is folded away at compile time.
// The regularized post-collision state f0 + omega f1 is one Hermite
// expansion in d, j (both conserved), B = dP + omega a1 and
// A = dA + omega a1^(3), so equilibrium and off-equilibrium parts are added
// as moments and expanded into populations once -- the updates in binary16
// storage are bound by these instructions, not by HBM (a polynomial per
// direction for each part, with the zero coefficients multiplied out, took
// 445 us for the fine update of a binary16 D3Q19 slab of 16.4 M nodes, this
// form 355; paired D2Q9 runs 80.6 -> 65.9 us for 33 x 513^2 nodes; in
// binary32 D3Q19 5.48 -> 5.77 TB/s, D2Q9 5.69 -> 5.88 TB/s).
template <class L, int COLL, bool MOV, class T, class Emit>
__device__ __forceinline__ void collide_emit(const T (&g)[L::Q], float omega,
                                                      const RefF& R, Emit&& emit,
                                                      const HrrIn<T>* hy = nullptr) {
  T d, j[3], P[6], dP[6], C[7], u[3], du[3];
  moments2<L>(g, d, j, P);
  const T rho = bc<T>(R.rho0) + d, inv = vrcp(rho);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (a >= L::D) {
      u[a] = du[a] = bc<T>(0.0f);
    } else if constexpr (MOV) {
      du[a] = kfma(-R.U[a], d, j[a]) * inv;
      u[a] = bc<T>(R.U[a]) + du[a];
    } else {
      u[a] = du[a] = j[a] * inv;
    }
  }
  second_dev<L, MOV>(j, u, du, R, dP);
  if constexpr (COLL == 0) {
    third_dev<L, MOV, false>(dP, dP, u, du, R, C);
    expand<L>(d, j, dP, C, [&](auto I, T v) {
      emit(I, kfma(omega, g[decltype(I)::value] - v, v));
    });
  } else {
    // omega a1, a1_ab = P_ab - d cs^2 delta_ab - dP_ab
    const T d3 = over<3>(d);
    T a1[6], B[6];
    auto fill = [&](int k) {
      T x = (k < 3 ? P[k] - d3 : P[k]) - dP[k];
      if constexpr (COLL == 3) x = vfma(kmul(hy->ks, rho), hy->s[k], kmul(hy->sig, x));
      a1[k] = kmul(omega, x);
      B[k] = dP[k] + a1[k];
    };
    fill(XX);
    fill(YY);
    fill(XY);
    a1[ZZ] = a1[XZ] = a1[YZ] = B[ZZ] = B[XZ] = B[YZ] = bc<T>(0.0f);
    if constexpr (L::D == 3) {
      fill(ZZ);
      fill(XZ);
      fill(YZ);
    }
    if constexpr (COLL == 1)
      third_dev<L, MOV, false>(dP, a1, u, du, R, C);
    else
      third_dev<L, MOV, true>(B, a1, u, du, R, C);
    expand<L>(d, j, B, C, emit);
  }
}

// ------------------------------------------------------------ storage types
template <class S>
struct Store;
template <>
struct Store<float> {
  __device__ __forceinline__ static float ld(const float* p) { return *p; }
  __device__ __forceinline__ static float ldg(const float* p) { return __ldg(p); }
  __device__ __forceinline__ static void st(float* p, float v) { *p = v; }
  __device__ __forceinline__ static void stcs(float* p, float v) { __stcs(p, v); }
};
template <>
struct Store<__half> {
  __device__ __forceinline__ static float ld(const __half* p) { return __half2float(*p); }
  __device__ __forceinline__ static float ldg(const __half* p) { return __half2float(__ldg(p)); }
  __device__ __forceinline__ static void st(__half* p, float v) { *p = __float2half_rn(v); }
  __device__ __forceinline__ static void stcs(__half* p, float v) { __stcs(p, __float2half_rn(v)); }
};

}  // namespace mlbm
