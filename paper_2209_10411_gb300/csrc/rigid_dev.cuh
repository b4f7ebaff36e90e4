// Rigid-body update of one particle for one DEM substep (Sec. 2.3.1), shared
// by the per-substep kernel and the fused DEM substep loop.
#pragma once

#include "mi_internal.cuh"

namespace mi {

// FP64: semi-implicit Euler for the velocity, Euler's equations in the body
// frame, exponential map for the orientation; buoyancy-corrected gravity
// (m - rho0 V) g.
//
// Bound by FP64 issue: a warp's FP64 instruction takes the pipe for about 64
// cycles on this part, for one lane as for 32, and the update is one dependent
// chain, so its time is its number of FP64 instructions.  Eight lanes of a warp
// share a particle (four particles to a warp) and every instruction does as
// many of its values as have the same form; values pass by shuffles, which
// cost next to nothing beside.  Lane c < 3 of either four owns component c of
// every 3-vector and of the quaternion's vector part, lane 3 its scalar; the
// first four rotate the angular velocity and sum the cosine's series while the
// second rotate the torque and sum the sine's.  The products of the
// quaternion's components serve the new rotation's rows (angular velocity to
// the world frame) and the next substep's columns.  47 FP64 instructions a
// substep: two particles' 100 substeps in one CTA take 227 us
// (367 with four lanes a particle, 100 instructions, no shared products).
//
// Rotations use R = 2 (v v^T + w [v]x + (w^2 - 1/2) I) of the unit quaternion
// (w, v); sin(a)/a and cos(a) of the half rotation angle a come from their
// Taylor series when a <= 1/64 (terms to a^8: the first omitted term is below
// 2^-53 relative there), from the library functions otherwise.  1/|q| of a
// quaternion whose squared norm n is within 2^-26 of 1 (every product made
// here) is 1.5 - n / 2, off by 3/8 (n - 1)^2 < 2^-53.  A quaternion made here has
// n within 6 ulps of 1 (the products' roundings and those of n itself), and one that is
// loaded is normalised when n is more than 8 off: a handed-in one is, and what a
// substep stored is taken as it is, as in the fused loop.
//
// Every operation is written out as a single rounding, so the substep kernel
// and the fused loop give the same bits whatever the compiler hoists.
__device__ __forceinline__ double pick3(int a, double x, double y, double z) { return a == 0 ? x : (a == 1 ? y : z); }

// One lane's part of a particle.
struct RigidLane {
  int c, a, a1, a2;          // lane of the four; its component and the two after it (cyclic; lane 3 repeats 2)
  bool second;               // of the second four
  double dt, hdt, acc, dtm;  // dt, dt / 2, (F + (m - rho0 V) g)_a, dt / m
  double T;                  // torque (world), component a
  double I[3], Ii[3];        // rows a of the inertia tensor and its inverse
  double pos, vel, om;       // component a
  double q;                  // component a of the quaternion's vector part, or its scalar (lane 3)
  double ca, cb, cc;         // half of R[a][a], R[a1][a], R[a2][a]
};

constexpr unsigned RIGID_FULL = 0xffffffffu;
constexpr int RIGID_LANES = 8;
__device__ __forceinline__ double quad(double v, int k) { return __shfl_sync(RIGID_FULL, v, k, 4); }
__device__ __forceinline__ double dot3(double a0, double b0, double a1, double b1, double a2, double b2) {
  return __fma_rn(a2, b2, __fma_rn(a1, b1, __dmul_rn(a0, b0)));
}
// the sum of the four lanes' squares, the same in each
__device__ __forceinline__ double quad_norm2(double v) {
  double s = __dmul_rn(v, v);
  s = __dadd_rn(s, __shfl_xor_sync(RIGID_FULL, s, 1));
  return __dadd_rn(s, __shfl_xor_sync(RIGID_FULL, s, 2));
}
// whether n lies within about `ulps` units in the last place of 1 (an integer comparison)
__device__ __forceinline__ bool near_one(double n, long long ulps) {
  const long long d = __double_as_longlong(n) - 0x3FF0000000000000LL;
  return d < ulps && d > -2 * ulps;
}

// The half entries of row a (ra, rb, rc along a, a1, a2) and of column a (in S) of the rotation of S.q.
__device__ __forceinline__ void rigid_rotation(RigidLane& S, double& rb, double& rc) {
  const double x = quad(S.q, 0), y = quad(S.q, 1), z = quad(S.q, 2), w = quad(S.q, 3);
  const double va = pick3(S.a, x, y, z), va1 = pick3(S.a1, x, y, z), va2 = pick3(S.a2, x, y, z);
  S.ca = __fma_rn(va, va, __fma_rn(w, w, -0.5));
  const double p1 = __dmul_rn(va, va1), p2 = __dmul_rn(w, va2), p3 = __dmul_rn(va, va2), p4 = __dmul_rn(w, va1);
  S.cb = __dadd_rn(p1, p2);
  S.cc = __dsub_rn(p3, p4);
  rb = __dsub_rn(p1, p2);
  rc = __dadd_rn(p3, p4);
}

// Particle p's lane (0..7).  The force sums were built with atomics by other
// threads: read past the L1.
__device__ __forceinline__ RigidLane rigid_load(const IntegrateLaunch& L, int p, int lane) {
  RigidLane S;
  const DevParticle& P = L.P[p];
  S.c = lane & 3;
  S.second = lane >= 4;
  S.a = S.c < 3 ? S.c : 2;
  S.a1 = S.a == 2 ? 0 : S.a + 1;
  S.a2 = S.a == 0 ? 2 : S.a - 1;
  double F = (double)__ldcg(L.facc + 6 * p + S.a) * FIX_INV;
  S.T = (double)__ldcg(L.facc + 6 * p + 3 + S.a) * FIX_INV;
  if (L.fc) {
    F = __dadd_rn(F, (double)__ldcg(L.fc + 6 * p + S.a) * FIX_INV);
    S.T = __dadd_rn(S.T, (double)__ldcg(L.fc + 6 * p + 3 + S.a) * FIX_INV);
  }
  const double m = P.mass;
  S.dt = L.dt;
  S.hdt = __dmul_rn(0.5, L.dt);
  S.dtm = __ddiv_rn(L.dt, m);
  S.acc = __fma_rn(__fma_rn(-L.rho0, P.volume, m), L.gravity[S.a], F);
  for (int k = 0; k < 3; ++k) {
    S.I[k] = P.inertia[3 * S.a + k];
    S.Ii[k] = P.inv_inertia[3 * S.a + k];
  }
  S.pos = P.pos[S.a];
  S.vel = P.vel[S.a];
  S.om = P.omega[S.a];
  S.q = P.quat[S.c < 3 ? S.c + 1 : 0];
  const double n = quad_norm2(S.q);
  if (!near_one(n, 8)) S.q = __dmul_rn(S.q, __ddiv_rn(1.0, __dsqrt_rn(n)));
  double rb, rc;
  rigid_rotation(S, rb, rc);
  return S;
}

__device__ __forceinline__ void rigid_store(const IntegrateLaunch& L, int p, const RigidLane& S) {
  if (S.second) return;
  DevParticle& P = L.P[p];
  P.quat[S.c < 3 ? S.c + 1 : 0] = S.q;
  if (S.c < 3) {
    P.pos[S.c] = S.pos;
    P.vel[S.c] = S.vel;
    P.omega[S.c] = S.om;
  }
}

// One substep; all 32 lanes of the warp take part (the shuffles).
__device__ __forceinline__ void rigid_substep(RigidLane& S) {
  const int a = S.a, a1 = S.a1, a2 = S.a2;
  S.vel = __fma_rn(S.dtm, S.acc, S.vel);
  S.pos = __fma_rn(S.dt, S.vel, S.pos);
  // body-frame angular velocity and torque: (R^T x)_a = R[a][a] x_a + R[a1][a] x_a1 + R[a2][a] x_a2
  const double v = S.second ? S.T : S.om;
  double b = dot3(S.ca, v, S.cb, quad(v, a1), S.cc, quad(v, a2));
  b = __dadd_rn(b, b);
  const double other = __shfl_xor_sync(RIGID_FULL, b, 4);
  const double wb = S.second ? other : b, Tb = S.second ? b : other;
  const double wb0 = quad(wb, 0), wb1 = quad(wb, 1), wb2 = quad(wb, 2);
  const double Iw = dot3(S.I[0], wb0, S.I[1], wb1, S.I[2], wb2);
  const double rhs = __fma_rn(pick3(a2, wb0, wb1, wb2), quad(Iw, a1), __fma_rn(-pick3(a1, wb0, wb1, wb2), quad(Iw, a2), Tb));
  const double wn = __fma_rn(S.dt, dot3(S.Ii[0], quad(rhs, 0), S.Ii[1], quad(rhs, 1), S.Ii[2], quad(rhs, 2)), wb);
  // q <- normalize(q (x) exp(u)): dq = (cos h, (sin h / h) u), u = wn dt / 2, h = |u|
  const double u = __dmul_rn(wn, S.hdt), u0 = quad(u, 0), u1 = quad(u, 1), u2 = quad(u, 2);
  const double h2 = dot3(u0, u0, u1, u1, u2, u2);
  double series;  // cos h (first four), sin(h) / h (second)
  if (h2 <= 1.0 / 4096.0) {
    series = __fma_rn(h2, S.second ? 1.0 / 362880 : 1.0 / 40320, S.second ? -1.0 / 5040 : -1.0 / 720);
    series = __fma_rn(h2, series, S.second ? 1.0 / 120 : 1.0 / 24);
    series = __fma_rn(h2, series, S.second ? -1.0 / 6 : -1.0 / 2);
    series = __fma_rn(h2, series, 1.0);
  } else {
    const double hn = __dsqrt_rn(h2);
    series = S.second ? __ddiv_rn(sin(hn), hn) : cos(hn);
  }
  __syncwarp();
  const double swap = __shfl_xor_sync(RIGID_FULL, series, 4);
  const double d0 = S.second ? swap : series, dv = __dmul_rn(S.second ? series : swap, u);
  const double d1 = quad(dv, 0), d2 = quad(dv, 1), d3 = quad(dv, 2);
  const double x = quad(S.q, 0), y = quad(S.q, 1), z = quad(S.q, 2), w = quad(S.q, 3);
  // this lane's component of q (x) dq
  const double e0 = S.c == 3 ? d0 : (S.c == 0 ? d1 : (S.c == 1 ? d2 : d3));    // with w
  const double e1 = S.c == 3 ? -d1 : (S.c == 0 ? d0 : (S.c == 1 ? -d3 : d2));  // with x
  const double e2 = S.c == 3 ? -d2 : (S.c == 0 ? d3 : (S.c == 1 ? d0 : -d1));  // with y
  const double e3 = S.c == 3 ? -d3 : (S.c == 0 ? -d2 : (S.c == 1 ? d1 : d0));  // with z
  const double r = __fma_rn(z, e3, dot3(w, e0, x, e1, y, e2));
  const double n = quad_norm2(r);
  S.q = __dmul_rn(r, near_one(n, 1LL << 26) ? __fma_rn(-0.5, n, 1.5) : __ddiv_rn(1.0, __dsqrt_rn(n)));
  // new angular velocity in the world frame: row a of the new rotation times wn
  double rb, rc;
  rigid_rotation(S, rb, rc);
  const double o = dot3(S.ca, wn, rb, quad(wn, a1), rc, quad(wn, a2));
  S.om = __dadd_rn(o, o);
}

// One substep of the particles [first, last) by the block's threads, four to a warp.
__device__ __forceinline__ void integrate_particles(const IntegrateLaunch& L, int first, int last) {
  const int lane = threadIdx.x & (RIGID_LANES - 1);
  for (int base = first + (int)(threadIdx.x >> 5) * 4; base < last; base += (int)blockDim.x / RIGID_LANES) {
    const int p = base + (int)((threadIdx.x & 31) / RIGID_LANES);
    const bool mine = p < last;
    RigidLane S = rigid_load(L, mine ? p : last - 1, lane);
    rigid_substep(S);
    __syncwarp();
    if (mine) rigid_store(L, p, S);
  }
}

}  // namespace mi
