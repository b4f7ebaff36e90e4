// Particle-side kernels: per-step prologue, solid flagging from the metaball
// field (Eq. 1), node classification with boundary/uncovered lists, the wall
// fraction q of every boundary link, the rigid-body update (Newton-Euler,
// Sec. 2.3.1) and mass-property quadrature.
//
// Flagging decides f >= 1 exactly as an FP64 evaluation would: an FP32 pass
// with the body-frame point formed in FP64 decides every node whose FP32 value
// is farther than GUARD from 1 (its error is below 3e-5 for control points at
// least 0.3 lu from the node), and the rare nodes inside the guard band are
// re-evaluated in FP64 with unfused operations in the order: x - X, R^T,
// ball by ball k / |x_b - c|^2 accumulated left to right.
#include <cfloat>
#include <climits>

#include "mi_internal.cuh"
#include "rigid_dev.cuh"

namespace mi {

namespace {
constexpr float GUARD = FIELD_GUARD;

// Entry k = lane of the body -> world rotation of the normalised quaternion q,
// unfused FP64 (lanes 9 and up repeat entry 8).  An FP64 instruction costs the
// same issue time for one lane as for 32 on this part, so the lanes share the
// work: lane l divides component l & 3 by the norm, and one sequence of
// products serves all nine entries, 1 - 2 (a^2 + c^2) or 2 (a b +- c d).
__device__ __forceinline__ double rotation_entry(const double q[4], int lane) {
  const double n = __dsqrt_rn(__dadd_rn(__dadd_rn(__dadd_rn(__dmul_rn(q[0], q[0]), __dmul_rn(q[1], q[1])),
                                                  __dmul_rn(q[2], q[2])),
                                        __dmul_rn(q[3], q[3])));
  const int c4 = lane & 3;
  const double v = __ddiv_rn(c4 == 0 ? q[0] : (c4 == 1 ? q[1] : (c4 == 2 ? q[2] : q[3])), n);
  // components (w, x, y, z) = 0..3 of the factors a b and c d of entry k, a hexadecimal digit each
  const int k = 4 * (lane < 8 ? lane : 8);
  const double a = __shfl_sync(0xffffffffu, v, (int)((0x121211112ull >> k) & 15ull)),
               b = __shfl_sync(0xffffffffu, v, (int)((0x133312322ull >> k) & 15ull)),
               c = __shfl_sync(0xffffffffu, v, (int)((0x200030003ull >> k) & 15ull)),
               d = __shfl_sync(0xffffffffu, v, (int)((0x212133233ull >> k) & 15ull));
  const bool minus = (0x62 >> (k / 4)) & 1, diag = (0x111 >> (k / 4)) & 1;
  const double p = __dmul_rn(c, d);
  const double t = __dmul_rn(2.0, __dadd_rn(__dmul_rn(a, b), minus ? -p : p));
  return diag ? __dsub_rn(1.0, t) : t;
}

// f(x) >= 1 in FP64, unfused, same operation order as the definition above,
// for the node (x, y, z) that every lane of the warp passes: the lanes form
// the terms of 32 balls at a time and the sum is taken in ball order, so the
// value is that of one thread summing ball after ball.
__device__ __noinline__ bool inside_exact_warp(const DevParticle& P, const double* balls_d, int x, int y, int z,
                                               unsigned lane) {
  const double d0 = __dsub_rn((double)x, P.pos[0]), d1 = __dsub_rn((double)y, P.pos[1]),
               d2 = __dsub_rn((double)z, P.pos[2]);
  const double* R = P.R;
  const double b0 = __dadd_rn(__dadd_rn(__dmul_rn(R[0], d0), __dmul_rn(R[3], d1)), __dmul_rn(R[6], d2));
  const double b1 = __dadd_rn(__dadd_rn(__dmul_rn(R[1], d0), __dmul_rn(R[4], d1)), __dmul_rn(R[7], d2));
  const double b2 = __dadd_rn(__dadd_rn(__dmul_rn(R[2], d0), __dmul_rn(R[5], d1)), __dmul_rn(R[8], d2));
  const int nb = P.n_balls;
  double f = 0.0;
  for (int base = 0; base < nb; base += 32) {
    double t = 0.0;
    const int i = base + (int)lane;
    if (i < nb) {
      const double* c = balls_d + 4 * (size_t)(P.ball_off + i);
      const double e0 = __dsub_rn(b0, c[0]), e1 = __dsub_rn(b1, c[1]), e2 = __dsub_rn(b2, c[2]);
      const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(e0, e0), __dmul_rn(e1, e1)), __dmul_rn(e2, e2));
      t = __ddiv_rn(c[3], r2);
    }
    const int m = nb - base < 32 ? nb - base : 32;
    for (int j = 0; j < m; ++j) f = __dadd_rn(f, __shfl_sync(0xffffffffu, t, j));
  }
  return f >= 1.0;
}

// Region of a box kernel: box [lo, lo + ext) widened by `pad`, clipped.
struct Region {
  int lo[3], n[3];
  unsigned total;
};
__device__ __forceinline__ Region clip_region(const int lo[3], const int ext[3], int pad, const LatticeGeom& g) {
  Region r;
  const int sz[3] = {g.nx, g.ny, g.nz};
  r.total = 1u;
  for (int a = 0; a < 3; ++a) {
    int l = lo[a] - pad, h = lo[a] + ext[a] + pad;
    l = l < 0 ? 0 : l;
    h = h > sz[a] ? sz[a] : h;
    r.lo[a] = l;
    r.n[a] = h > l ? h - l : 0;
    r.total *= (unsigned)r.n[a];
  }
  return r;
}

__device__ __forceinline__ long long lin(int x, int y, int z, const LatticeGeom& g) {
  return x + (long long)g.nx * (y + (long long)g.ny * z);
}

// Neighbour along direction d with periodic wrap; false if outside the domain.
__device__ __forceinline__ bool neighbour(int x, int y, int z, int dx, int dy, int dz, const LatticeGeom& g,
                                          long long& out) {
  // |dx|, |dy|, |dz| <= 1: one wrap at most
  int a = x + dx, b = y + dy, c = z + dz;
  if (a < 0 || a >= g.nx) {
    if (!g.periodic[0]) return false;
    a += a < 0 ? g.nx : -g.nx;
  }
  if (b < 0 || b >= g.ny) {
    if (!g.periodic[1]) return false;
    b += b < 0 ? g.ny : -g.ny;
  }
  if (c < 0 || c >= g.nz) {
    if (!g.periodic[2]) return false;
    c += c < 0 ? g.nz : -g.nz;
  }
  out = lin(a, b, c, g);
  return true;
}
}  // namespace

// The particle owning block b of a box kernel's 1D grid (off[p] <= b <
// off[p + 1], off[0] = 0) by binary search, its first block and block count.
struct BoxBlock {
  int p, b, nb;
};
__device__ __forceinline__ BoxBlock box_block(const int* __restrict__ off, int np, int b) {
  int lo = 0, hi = np;  // off[lo] <= b < off[hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (off[mid] <= b) lo = mid;
    else hi = mid;
  }
  const int o = off[lo];
  return {lo, b - o, off[lo + 1] - o};
}

// ---------------------------------------------------------------------------
// Prologue, one launch of two independent parts.  The first blocks, a warp
// per particle: bump the flag generation, zero counters and hydrodynamic
// force sums, rotation matrices and node boxes at the current pose.  The other
// blocks clear the owner buffer about to be rewritten over the boxes it was
// last written with (nothing the first part touches).
// ---------------------------------------------------------------------------
constexpr int PROLOGUE_THREADS = 256;
__global__ void __launch_bounds__(PROLOGUE_THREADS) k_prologue(ParticleLaunch L) {
  constexpr unsigned FULL = 0xffffffffu;
  const int nprol = (L.np + PROLOGUE_THREADS / 32 - 1) / (PROLOGUE_THREADS / 32);
  if ((int)blockIdx.x >= nprol) {
    const BoxBlock bb = box_block(L.flag_off, L.np, (int)blockIdx.x - nprol);
    const DevParticle& P = L.P[bb.p];
    const int* lo = P.lo_hist[L.cur_buf];
    if (lo[0] == BOX_NONE) return;
    const Region r = clip_region(lo, P.ext, 0, L.g);
    const unsigned n0 = (unsigned)r.n[0], n01 = n0 * (unsigned)r.n[1];
    for (unsigned i = bb.b * blockDim.x + threadIdx.x; i < r.total; i += bb.nb * blockDim.x) {
      const unsigned zi = i / n01, rem = i - zi * n01, yi = rem / n0;
      const int x = r.lo[0] + (int)(rem - yi * n0);
      const int y = r.lo[1] + (int)yi;
      const int z = r.lo[2] + (int)zi;
      L.owner_cur[lin(x, y, z, L.g)] = OWNER_NONE;
    }
    return;
  }
  const int p = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (p == 0 && lane == 0) {
    L.ctr->gen += 1u;
    L.ctr->n_bc = 0;
    L.ctr->n_links = 0;
    L.ctr->n_new = 0;
    L.ctr->n_cov = 0;
  }
  if (p >= L.np) return;
  DevParticle& P = L.P[p];
  const double r = rotation_entry(P.quat, lane);
  if (lane < 9) {
    const float rf = (float)r;
    P.R[lane] = r;
    P.Rf[lane] = rf;
  }
  if (L.balls_s) {
    // the body frame as float pairs (k_links_q16): R, R^T (X - floor X) by lanes
    // 0 to 2, R^T e_d by lane d
    double R[9], f[3];
#pragma unroll
    for (int k = 0; k < 9; ++k) R[k] = __shfl_sync(FULL, r, k);
    for (int k = 0; k < 3; ++k) f[k] = P.pos[k] - floor(P.pos[k]);
    if (lane < 9) {
      P.Rs[0][lane] = (float)r;
      P.Rs[1][lane] = (float)(r - (double)(float)r);
    }
    if (lane < 3) {
      const double t = pick3(lane, R[0], R[1], R[2]) * f[0] + pick3(lane, R[3], R[4], R[5]) * f[1] +
                       pick3(lane, R[6], R[7], R[8]) * f[2];
      P.Ts[0][lane] = (float)t;
      P.Ts[1][lane] = (float)(t - (double)(float)t);
    }
    if (lane < 19)
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const double e = R[k] * lex(lane) + R[3 + k] * ley(lane) + R[6 + k] * lez(lane);
        P.Es[lane][k] = (float)e;
        P.Es[lane][3 + k] = (float)(e - (double)(float)e);
      }
  }
  // axis a = lane of the box and of the position's split
  if (lane < 3) {
    const int a = lane;
    const double pos = P.pos[a], fl = floor(pos);
    const int lo = (int)floor(pos - P.Rt) - 1;
    P.lo[a] = lo;
    P.posf[a] = (float)pos;
    P.pos_i[a] = (int)fl;
    P.pos_fr[a] = (float)(pos - fl);
    P.velf[a] = (float)P.vel[a];
    P.omegaf[a] = (float)P.omega[a];
    P.sctr[L.cur_buf][a] = (float)pos;
    const int prev = P.lo_hist[L.prev_buf][a];
    if (prev != BOX_NONE && abs(lo - prev) > 2) atomicOr(&L.ctr->status, STATUS_MOVED_TOO_FAR);
  }
  if (lane == 0) P.srad2[L.cur_buf] = -1;  // the solid radius of this step, grown by k_flag
  if (lane < 6) L.facc[6 * p + lane] = 0;
}

cudaError_t launch_prologue(const ParticleLaunch& L, cudaStream_t s) {
  const int per = PROLOGUE_THREADS / 32, nprol = (L.np + per - 1) / per;
  k_prologue<<<nprol + (L.np > 0 ? L.flag_blocks : 1), PROLOGUE_THREADS, 0, s>>>(L);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// A ball in the lattice frame at the current pose, relative to floor X: its
// centre C = R c + (X - floor X) in FP64, as FP32 (with k), as its nearest
// multiple h of the particle's link_grid (with k's FP32 rounding) and as the
// FP32 remainder C - h (with k's).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void lattice_ball(const DevParticle& P, const double* __restrict__ c, float4* __restrict__ w) {
  const float k = (float)c[3], grid = P.link_grid, inv = 1.0f / grid;  // a power of two
  float C[3], h[3], l[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const double v = P.R[3 * a] * c[0] + P.R[3 * a + 1] * c[1] + P.R[3 * a + 2] * c[2] + (P.pos[a] - (double)P.pos_i[a]);
    C[a] = (float)v;
    h[a] = rintf(C[a] * inv) * grid;
    l[a] = (float)(v - (double)h[a]);
  }
  w[0] = make_float4(C[0], C[1], C[2], k);
  w[1] = make_float4(h[0], h[1], h[2], k);
  w[2] = make_float4(l[0], l[1], l[2], (float)(c[3] - (double)k));
}

// ---------------------------------------------------------------------------
// Solid flagging: node x of particle p's box is solid for p when
// f_p(R_p^T (x - X_p)) >= 1; the owner is the lowest such p (atomicMin).
//
// A lane takes the 2 x 2 x 2 nodes of a cube first, from f at their middle and
// the distance m to the nearest of the balls summed: a node is D = sqrt(3) / 2
// from the middle, so that each term k / r^2 of it, and with them their sum, lies
// between (m / (m + D))^2 and (m / (m - D))^2 times the middle's.  Cubes all
// inside (often from the first few balls, whose partial sum is a lower bound) or all
// outside are done; the nodes of the others (about 8 of 32, around the surface)
// are collected per warp and evaluated one by one, 32 at a time: that is most
// of the work left.  Before, a lane per box node: half the box's nodes are outside the
// bounding sphere, the solid ones leave the sum early, and their lanes
// waited (17 of 32 active).  Bound by FP32 issue and the reciprocal unit:
// 300 particles of 8 to 64 balls (18 M box nodes) 107 us, 283 before; three of 127 balls 19
// us, 34 before.
// ---------------------------------------------------------------------------
constexpr int FLAG_WARPS = 8;
__global__ void __launch_bounds__(32 * FLAG_WARPS, 3) k_flag(ParticleLaunch L) {
  constexpr unsigned FULL = 0xffffffffu;
  constexpr float D = 0.8661f;
  extern __shared__ float4 sb[];
  const BoxBlock bb = box_block(L.flag_off, L.np, blockIdx.x);
  const int p = bb.p;
  const DevParticle& P = L.P[p];
  const int nb = P.n_balls;
  const bool staged = nb <= L.max_balls_per_particle;
  __shared__ int rr_s;  // the block's largest squared solid distance (float bits)
  __shared__ unsigned open_s[FLAG_WARPS][35];  // the warp's undecided cubes
  volatile int* rr = &rr_s;
  unsigned* open = open_s[threadIdx.x >> 5];
  if (threadIdx.x == 0) rr_s = -1;
  if (staged)
    for (int i = threadIdx.x; i < nb; i += blockDim.x) sb[i] = L.balls[P.ball_off + i];
  // the ball table of FP32 storage's wall fractions (below), by the particle's first block
  if (bb.b == 0 && L.balls_w)
    for (int i = threadIdx.x; i < nb; i += blockDim.x)
      lattice_ball(P, L.balls_d + 4 * (size_t)(P.ball_off + i), L.balls_w + 3 * (size_t)(P.ball_off + i));
  __syncthreads();
  const float4* bl = staged ? sb : L.balls + P.ball_off;
  if (bb.b == 0 && threadIdx.x == 0)
    for (int a = 0; a < 3; ++a) L.P[p].lo_hist[L.cur_buf][a] = P.lo[a];
  const Region r = clip_region(P.lo, P.ext, 0, L.g);
  // x - X = (x - Xi) - Xf with Xi = floor(X): the integer part is exact in
  // FP32, the fraction carries one FP32 rounding (both set once per particle
  // by the prologue, with R in FP32: FP64 set-up in every thread would cost
  // more than the field evaluations on this part)
  const int o0 = r.lo[0] - P.pos_i[0], o1 = r.lo[1] - P.pos_i[1], o2 = r.lo[2] - P.pos_i[2];
  const float xf0 = P.pos_fr[0], xf1 = P.pos_fr[1], xf2 = P.pos_fr[2];
  float Rf[9];
  for (int k = 0; k < 9; ++k) Rf[k] = P.Rf[k];
  const float rt = (float)P.Rt * (1.0f + 1e-6f) + 1e-4f, rt2 = rt * rt;
  // cubes of the box: the last ones along an axis may be half outside
  const unsigned c0 = (unsigned)(r.n[0] + 1) >> 1, c1 = (unsigned)(r.n[1] + 1) >> 1, c2 = (unsigned)(r.n[2] + 1) >> 1;
  const unsigned c01 = c0 * c1, cubes = r.total ? c01 * c2 : 0u;
  const unsigned lane = threadIdx.x & 31u;
  // a warp's cubes at a time: 32, fewer where there are more warps than that
  // gives work to (4 make a full warp of nodes)
  const unsigned warps = bb.nb * FLAG_WARPS, warp = bb.b * FLAG_WARPS + (threadIdx.x >> 5);
  const unsigned each = min(32u, max(4u, (cubes + warps - 1u) / warps));
  // with warps for all nodes at once the cubes' sums would only lengthen the chain
  const bool probe = each > 4u;

  // the nodes of n (<= 4) collected cubes from `first`; whole warps step together
  // (the guard band's FP64 field is a warp collective)
  const auto nodes = [&](unsigned first, unsigned n) {
    int x = 0, y = 0, z = 0;
    bool inside = false, band = false;
    float d0 = 0.f, d1 = 0.f, d2 = 0.f;
    if ((lane >> 3) < n) {
      const unsigned cube = open[first + (lane >> 3)], zc = cube / c01, rem = cube - zc * c01, yc = rem / c0;
      x = (int)(2u * (rem - yc * c0) + (lane & 1u));
      y = (int)(2u * yc + ((lane >> 1) & 1u));
      z = (int)(2u * zc + ((lane >> 2) & 1u));
      d0 = (float)(x + o0) - xf0;
      d1 = (float)(y + o1) - xf1;
      d2 = (float)(z + o2) - xf2;
      // outside the box, or beyond the tight radius: fluid
      if (x < r.n[0] && y < r.n[1] && z < r.n[2] && d0 * d0 + d1 * d1 + d2 * d2 <= rt2) {
        const float b0 = Rf[0] * d0 + Rf[3] * d1 + Rf[6] * d2;
        const float b1 = Rf[1] * d0 + Rf[4] * d1 + Rf[7] * d2;
        const float b2 = Rf[2] * d0 + Rf[5] * d1 + Rf[8] * d2;
        // four independent partial sums (FP32 reordering moves the sum by far
        // less than GUARD, and sums within GUARD of 1 are redone in FP64)
        float f0 = 0.f, f1 = 0.f, f2 = 0.f, f3 = 0.f;
        int b = 0;
        for (; b + 4 <= nb; b += 4) {
          const float4 e0 = bl[b], e1 = bl[b + 1], e2 = bl[b + 2], e3 = bl[b + 3];
          f0 += __fdividef(e0.w, (b0 - e0.x) * (b0 - e0.x) + (b1 - e0.y) * (b1 - e0.y) + (b2 - e0.z) * (b2 - e0.z));
          f1 += __fdividef(e1.w, (b0 - e1.x) * (b0 - e1.x) + (b1 - e1.y) * (b1 - e1.y) + (b2 - e1.z) * (b2 - e1.z));
          f2 += __fdividef(e2.w, (b0 - e2.x) * (b0 - e2.x) + (b1 - e2.y) * (b1 - e2.y) + (b2 - e2.z) * (b2 - e2.z));
          f3 += __fdividef(e3.w, (b0 - e3.x) * (b0 - e3.x) + (b1 - e3.y) * (b1 - e3.y) + (b2 - e3.z) * (b2 - e3.z));
        }
        for (; b < nb; ++b) {
          const float4 c = bl[b];
          const float e0 = b0 - c.x, e1 = b1 - c.y, e2 = b2 - c.z;
          f0 += __fdividef(c.w, e0 * e0 + e1 * e1 + e2 * e2);
        }
        const float f = (f0 + f1) + (f2 + f3);
        if (f > 1.0f + GUARD) inside = true;
        else if (f < 1.0f - GUARD) inside = false;
        else band = true;  // within GUARD of 1 (or not a number): decided in FP64 below
      }
      x += r.lo[0];
      y += r.lo[1];
      z += r.lo[2];
    }
    // the nodes in the guard band, one at a time by the whole warp
    for (unsigned m = __ballot_sync(FULL, band); m; m &= m - 1u) {
      const int src = __ffs(m) - 1;
      const bool in = inside_exact_warp(P, L.balls_d, __shfl_sync(FULL, x, src), __shfl_sync(FULL, y, src),
                                        __shfl_sync(FULL, z, src), lane);
      if ((int)lane == src) inside = in;
    }
    if (inside) {
      atomicMin(L.owner_cur + lin(x, y, z, L.g), (uint32_t)p);
      // the block's solid radius in shared memory (non-negative floats
      // order as their bits): an atomic only where it grows
      const int dd = __float_as_int(d0 * d0 + d1 * d1 + d2 * d2);
      if (dd > *rr) atomicMax((int*)rr, dd);
    }
  };

  unsigned held = 0;  // collected cubes
  for (unsigned base = warp * each; base < cubes; base += warps * each) {
    const unsigned i = base + lane;
    bool undecided = false;
    if (lane < each && i < cubes) {
      const unsigned zc = i / c01, rem = i - zc * c01, yc = rem / c0;
      const int x = (int)(2u * (rem - yc * c0)), y = (int)(2u * yc), z = (int)(2u * zc);
      const float d0 = (float)(x + o0) - xf0, d1 = (float)(y + o1) - xf1, d2 = (float)(z + o2) - xf2;
      const float h0 = d0 + 0.5f, h1 = d1 + 0.5f, h2 = d2 + 0.5f;
      const float far = rt + D;
      if (h0 * h0 + h1 * h1 + h2 * h2 > far * far) {
        // all beyond the tight radius: fluid
      } else if (!probe) {
        undecided = true;
      } else {
        const float b0 = Rf[0] * h0 + Rf[3] * h1 + Rf[6] * h2;
        const float b1 = Rf[1] * h0 + Rf[4] * h1 + Rf[7] * h2;
        const float b2 = Rf[2] * h0 + Rf[5] * h1 + Rf[8] * h2;
        float f0 = 0.f, f1 = 0.f, m0 = INFINITY, m1 = INFINITY;
        bool inside = false;
        // all inside: f m^2 > (m + D)^2, for the balls summed so far
        const auto solid = [&]() {
          const float m2 = fminf(m0, m1), m = m2 * rsqrtf(m2) + D;
          return (f0 + f1) * m2 > (1.0f + GUARD) * m * m;
        };
        int b = 0;
        for (; b + 4 <= nb; b += 4) {
          const float4 e0 = bl[b], e1 = bl[b + 1], e2 = bl[b + 2], e3 = bl[b + 3];
          const float r0 = (b0 - e0.x) * (b0 - e0.x) + (b1 - e0.y) * (b1 - e0.y) + (b2 - e0.z) * (b2 - e0.z);
          const float r1 = (b0 - e1.x) * (b0 - e1.x) + (b1 - e1.y) * (b1 - e1.y) + (b2 - e1.z) * (b2 - e1.z);
          const float r2 = (b0 - e2.x) * (b0 - e2.x) + (b1 - e2.y) * (b1 - e2.y) + (b2 - e2.z) * (b2 - e2.z);
          const float r3 = (b0 - e3.x) * (b0 - e3.x) + (b1 - e3.y) * (b1 - e3.y) + (b2 - e3.z) * (b2 - e3.z);
          f0 += e0.w * rcp_start(r0) + e2.w * rcp_start(r2);
          f1 += e1.w * rcp_start(r1) + e3.w * rcp_start(r3);
          m0 = fminf(m0, fminf(r0, r2));
          m1 = fminf(m1, fminf(r1, r3));
          if ((b & 4) && solid()) {
            inside = true;
            break;
          }
        }
        if (!inside) {
          for (; b < nb; ++b) {
            const float4 c = bl[b];
            const float e0 = b0 - c.x, e1 = b1 - c.y, e2 = b2 - c.z, r0 = e0 * e0 + e1 * e1 + e2 * e2;
            f0 += c.w * rcp_start(r0);
            m0 = fminf(m0, r0);
          }
          inside = solid();
          const float m2 = fminf(m0, m1), m = m2 * rsqrtf(m2) - D;
          // all outside: f m^2 < (m - D)^2
          undecided = !inside && !(m > 0.f && (f0 + f1) * m2 < (1.0f - GUARD) * m * m);
        }
        if (inside) {
          // a cube half outside the box: its nodes one by one
          if (x + 1 < r.n[0] && y + 1 < r.n[1] && z + 1 < r.n[2]) {
            uint32_t* o = L.owner_cur + lin(x + r.lo[0], y + r.lo[1], z + r.lo[2], L.g);
#pragma unroll
            for (int k = 0; k < 8; ++k)
              atomicMin(o + (k & 1) + (long long)L.g.nx * ((k >> 1 & 1) + (long long)L.g.ny * (k >> 2)), (uint32_t)p);
            // its farthest node's distance, formed as for a node by itself
            const float g0 = (float)(x + 1 + o0) - xf0, g1 = (float)(y + 1 + o1) - xf1, g2 = (float)(z + 1 + o2) - xf2;
            const float a0 = fmaxf(fabsf(d0), fabsf(g0)), a1 = fmaxf(fabsf(d1), fabsf(g1)), a2 = fmaxf(fabsf(d2), fabsf(g2));
            const int dd = __float_as_int(a0 * a0 + a1 * a1 + a2 * a2);
            if (dd > *rr) atomicMax((int*)rr, dd);
          } else {
            undecided = true;
          }
        }
      }
    }
    const unsigned bits = __ballot_sync(FULL, undecided);
    if (undecided) open[held + __popc(bits & ((1u << lane) - 1u))] = i;  // held <= 3
    held += (unsigned)__popc(bits);
    __syncwarp();
    while (held >= 4) nodes(held -= 4, 4);
    __syncwarp();
  }
  if (held) nodes(0, held);
  __syncthreads();
  if (threadIdx.x == 0 && *rr >= 0) atomicMax(&L.P[p].srad2[L.cur_buf], *rr);
}

cudaError_t launch_flag(const ParticleLaunch& L, cudaStream_t s) {
  if (L.np == 0) return cudaSuccess;
  const size_t smem = sizeof(float4) * (size_t)L.max_balls_per_particle;
  k_flag<<<L.flag_blocks, 32 * FLAG_WARPS, smem, s>>>(L);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Classification over each particle's old and new boxes widened by 2: solid,
// boundary (fluid with a solid neighbour; 18-bit link mask), uncovered (fluid
// now, solid at the previous step), and with the cover/uncover rule covered
// (solid now, fluid at the previous step).  Boxes may overlap: every block
// writes the same class for a node, and a per-node generation stamp lets
// exactly one block append it to the boundary / uncovered / covered lists.
//
// One warp per R rows (y) at one z (four; one on small lattices, where there are
// warps for every row and the chain's length counts), 30 nodes of each at a time (lanes 1 to
// 30, lanes 0 and 31 their x neighbours): the owners of the rows and of those
// around them (18 for four) are one coalesced load each, a ballot turns each into a bit row,
// the boundary nodes come from the words shifted and merged, and only theirs
// are looked up bit by bit, a lane each, for the link masks (row by row, nine
// loads and 18 bits a node: twice the instructions).  A warp keeps its
// boundary nodes in shared memory and appends 32 at a time: all warps share
// the two list counters, and one same-address atomic per counter and chunk
// (about three boundary nodes) took most of the kernel's time on a lattice of
// 300 particles.  The 32 nodes' links are written by the whole warp, a lane
// per link.  Bound by latency (of the loads, and of the stamps' and counters'
// atomics): 300 particles (0.82 M boundary nodes) 264 us alone, 320 row by row,
// 588 with an append per chunk, 640 with a load per direction and node and links
// written node by node.
// ---------------------------------------------------------------------------
namespace {
constexpr int CLS_WARPS = 8, CLS_KEEP = 152;  // a chunk adds at most 4 x 30 nodes to at most 31 kept
struct BoundaryKeep {
  uint32_t x[CLS_KEEP], yz[CLS_KEEP], mask[CLS_KEEP];  // y in the low 16 bits, z in the high (both <= 65535)
};

// Append n (<= 32) kept nodes from `first` and their links to the lists.
__device__ __forceinline__ void append_boundary(const ParticleLaunch& L, const BoundaryKeep& K, int first, int n, int lane) {
  constexpr unsigned FULL = 0xffffffffu;
  const int at = first + lane;
  const uint32_t x = lane < n ? K.x[at] : 0u, yz = lane < n ? K.yz[at] : 0u, mask = lane < n ? K.mask[at] : 0u;
  const unsigned m = (unsigned)__popc(mask);
  unsigned incl = m;
#pragma unroll
  for (int k = 1; k < 32; k <<= 1) {
    const unsigned v = __shfl_up_sync(FULL, incl, k);
    if (lane >= k) incl += v;
  }
  const unsigned total = __shfl_sync(FULL, incl, 31);
  unsigned got = 0;
  if (lane == 0) got = atomicAdd(&L.ctr->n_bc, (unsigned)n);
  if (lane == 1) got = atomicAdd(&L.ctr->n_links, total);
  const unsigned bi = __shfl_sync(FULL, got, 0) + (unsigned)lane, base_l = __shfl_sync(FULL, got, 1);
  const unsigned lo_l = base_l + incl - m;
  bool fits = false;  // this node's links are written
  if (lane < n) {
    if (bi >= L.cap_bc) {
      atomicOr(&L.ctr->status, STATUS_BC_OVERFLOW);
    } else {
      L.bc_cell[bi] = (uint32_t)lin((int)x, (int)(yz & 0xffffu), (int)(yz >> 16), L.g);
      L.bc_mask[bi] = mask;
      L.bc_loff[bi] = lo_l;
      fits = lo_l + m <= L.cap_links;
      if (!fits) atomicOr(&L.ctr->status, STATUS_LINK_OVERFLOW);
    }
  }
  // the links, a lane each: the node (lane s) by binary search in the prefix
  // sums, the direction as the k-th set bit of its mask
  for (unsigned t0 = 0; t0 < total; t0 += 32) {
    const unsigned t = t0 + (unsigned)lane;
    int s = 0;
#pragma unroll
    for (int k = 16; k > 0; k >>= 1)
      if (__shfl_sync(FULL, incl, s + k - 1) <= t) s += k;
    const unsigned e = __shfl_sync(FULL, incl - m, s);
    unsigned ms = __shfl_sync(FULL, mask, s);
    const unsigned sbi = __shfl_sync(FULL, bi, s), sx = __shfl_sync(FULL, x, s), syz = __shfl_sync(FULL, yz, s);
    const bool ok = __shfl_sync(FULL, (int)fits, s) != 0;
    if (t < total && ok) {
      for (unsigned k = t - e; k > 0; --k) ms &= ms - 1u;
      const int d = __ffs(ms) - 1;
      long long nbr;
      neighbour((int)sx, (int)(syz & 0xffffu), (int)(syz >> 16), lex(d), ley(d), lez(d), L.g, nbr);
      L.link_bc[base_l + t] = sbi;
      L.link_dir[base_l + t] = (uint8_t)d;
      L.link_p[base_l + t] = L.owner_cur[nbr];
    }
  }
}
}  // namespace

template <bool COV, int R>
__global__ void __launch_bounds__(32 * CLS_WARPS, 3) k_classify(ParticleLaunch L) {
  constexpr unsigned FULL = 0xffffffffu;
  const BoxBlock bb = box_block(L.cls_off, L.np, blockIdx.x);
  const DevParticle& P = L.P[bb.p];
  int lo[3], ext[3];
  const int* lp = P.lo_hist[L.prev_buf];
  const bool had = lp[0] != BOX_NONE;
  for (int a = 0; a < 3; ++a) {
    if (!had) {
      lo[a] = P.lo[a];
      ext[a] = P.ext[a];
    } else {
      lo[a] = min(P.lo[a], lp[a]);
      ext[a] = max(P.lo[a], lp[a]) + P.ext[a] - lo[a];
    }
  }
  // nodes whose class can change: the solid nodes of this step and of the
  // previous one (within their solid radii of the positions they were
  // flagged at), the fluid nodes next to them (a link is at most sqrt 2
  // long), and the nodes uncovered at the previous step (solid two steps ago:
  // within a move of the previous solid, and a particle moves at most two
  // nodes per step): both spheres widened by 3
  const int sc = P.srad2[L.cur_buf], sp = had ? P.srad2[L.prev_buf] : -1;
  if (sc < 0 && sp < 0) return;
  const float rc = sc >= 0 ? sqrtf(__int_as_float(sc)) + 3.0f : -1.0f;
  const float rp = sp >= 0 ? sqrtf(__int_as_float(sp)) + 3.0f : -1.0f;
  const float rc2 = rc * rc, rp2 = rp * rp;
  const float cc0 = P.sctr[L.cur_buf][0], cc1 = P.sctr[L.cur_buf][1], cc2 = P.sctr[L.cur_buf][2];
  const float cp0 = P.sctr[L.prev_buf][0], cp1 = P.sctr[L.prev_buf][1], cp2 = P.sctr[L.prev_buf][2];
  const Region r = clip_region(lo, ext, 2, L.g);
  const unsigned gen = L.ctr->gen;
  const int lane = threadIdx.x & 31;
  __shared__ BoundaryKeep keep[CLS_WARPS];
  __shared__ unsigned words[CLS_WARPS][3 * (R + 2)];
  BoundaryKeep& K = keep[threadIdx.x >> 5];
  unsigned* W = words[threadIdx.x >> 5];  // the solid nodes of the rows around, a bit per lane
  int kept = 0;
  const LatticeGeom& g = L.g;
  // units of R rows (y) in tiles of 4 x 4 (y, z), which the warps take in
  // turn (parts of one when there are more warps): a warp's nodes then lie
  // together on the surface, and the gathers of the kernels that walk the lists
  // find each other's sectors in the caches
  const unsigned ty = ((unsigned)r.n[1] + 3u) / 4u, slots = (16u / R) * ty * (((unsigned)r.n[2] + 3u) / 4u);
  const unsigned wid = (bb.b * blockDim.x + threadIdx.x) >> 5, nw = (bb.nb * blockDim.x) >> 5;
  const unsigned each = min(16u / R, (slots + nw - 1u) / nw);
  for (unsigned n = 0, slot = wid * each; slot < slots;) {
    const unsigned at = slot;
    if (++n % each) ++slot;
    else slot += (nw - 1u) * each + 1u;
    const unsigned tile = at / (16u / R), part = at % (16u / R), tz = tile / ty;
    const int yi = (int)(4u * (tile - tz * ty) + R * (part % (4u / R))), zi = (int)(4u * tz + part / (4u / R));
    if (yi >= r.n[1] || zi >= r.n[2]) continue;
    const int y = r.lo[1] + yi, z = r.lo[2] + zi, rows = min(R, r.n[1] - yi);
    // the rows' x-interval inside either sphere, a lane per row
    int xa = INT_MAX, xb = INT_MIN;
    if (lane < rows) {
      const int yl = y + lane;
      const float hc = rc2 - ((yl - cc1) * (yl - cc1) + (z - cc2) * (z - cc2));
      if (rc >= 0.f && hc >= 0.f) {
        const float w = sqrtf(hc);
        xa = (int)ceilf(cc0 - w);
        xb = (int)floorf(cc0 + w);
      }
      const float hp = rp2 - ((yl - cp1) * (yl - cp1) + (z - cp2) * (z - cp2));
      if (rp >= 0.f && hp >= 0.f) {
        const float w = sqrtf(hp);
        xa = min(xa, (int)ceilf(cp0 - w));
        xb = max(xb, (int)floorf(cp0 + w));
      }
    }
    xa = max(__reduce_min_sync(FULL, xa), r.lo[0]);
    xb = min(__reduce_max_sync(FULL, xb), r.lo[0] + r.n[0] - 1);
    // rows outside both spheres (xa > xb) are skipped before any index is
    // formed: xa = INT_MAX + lane would overflow
    if (xa > xb) continue;
    // first nodes of the R + 2 by 3 rows around (32-bit: lists hold node indices),
    // and which of them are inside the domain
    unsigned yr[R + 2], zr[3], rin = 0;
#pragma unroll
    for (int k = 0; k < R + 2; ++k) {
      int b = y + k - 1;
      const bool out = b < 0 || b >= g.ny;
      if (out) b += b < 0 ? g.ny : -g.ny;
      yr[k] = (unsigned)b;
      if (k <= rows + 1 && (!out || g.periodic[1])) rin |= 1u << k;
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      int c = z + k - 1;
      const bool out = c < 0 || c >= g.nz;
      if (out) c += c < 0 ? g.nz : -g.nz;
      zr[k] = (unsigned)c * (unsigned)g.ny;
      if (!out || g.periodic[2]) rin |= 1u << (R + 2 + k);
    }
    const unsigned c0 = (zr[1] + (unsigned)y) * (unsigned)g.nx;
    for (int xs = xa - 1; xs < xb; xs += 30) {
      const int x = xs + lane;
      const bool node = lane >= 1 && lane <= 30 && x <= xb;
      int xw = x;
      if (x < 0 || x >= g.nx) xw = g.periodic[0] ? (x < 0 ? x + g.nx : x - g.nx) : -1;
      const bool load = x <= xb + 1 && xw >= 0;
      uint32_t o[3 * (R + 2)];
#pragma unroll
      for (int k = 0; k < 3 * (R + 2); ++k)
        o[k] = load && (rin >> (k % (R + 2)) & 1u) && (rin >> (R + 2 + k / (R + 2)) & 1u)
                   ? __ldg(L.owner_cur + ((zr[k / (R + 2)] + yr[k % (R + 2)]) * (unsigned)g.nx + (unsigned)xw))
                   : OWNER_NONE;
      bool was[R];
#pragma unroll
      for (int j = 0; j < R; ++j)
        was[j] = node && j < rows && L.owner_prev[c0 + (unsigned)(j * g.nx + x)] != OWNER_NONE;
      unsigned bits[3 * (R + 2)], word = 0;
#pragma unroll
      for (int k = 0; k < 3 * (R + 2); ++k) {
        bits[k] = __ballot_sync(FULL, o[k] != OWNER_NONE);
        if (lane == k) word = bits[k];
      }
      __syncwarp();
      if (lane < 3 * (R + 2)) W[lane] = word;
      bool bnd[R], isnew[R], iscov[R], list[R];
#pragma unroll
      for (int j = 0; j < R; ++j) {
        // the row's solid neighbours as a bit row: along x by the word beside
        const unsigned *zm = bits + j, *z0 = bits + (R + 2) + j, *zp = bits + 2 * (R + 2) + j;  // y - 1, y, y + 1 at z - 1, z, z + 1
        const unsigned S = z0[1], side = zm[1] | zp[1] | z0[0] | z0[2];
        const unsigned near = S << 1 | S >> 1 | side | side << 1 | side >> 1 | zm[0] | zm[2] | zp[0] | zp[2];
        const bool in = node && j < rows, solid = S >> lane & 1u;
        bnd[j] = in && !solid && (near >> lane & 1u);
        isnew[j] = in && !solid && was[j];
        // covered: listed for the cover/uncover rule only, and not in the step
        // that first flags the covering particle (it was not there before)
        iscov[j] = COV && in && solid && !was[j] && L.P[o[R + 3 + j]].lo_hist[L.prev_buf][0] != BOX_NONE;
        const unsigned c = c0 + (unsigned)(j * g.nx + x);
        if (in) L.cls[c] = (uint8_t)((solid ? CLS_SOLID : 0) | (bnd[j] ? CLS_BOUNDARY : 0) | (isnew[j] ? CLS_NEW : 0));
        list[j] = bnd[j] || isnew[j] || iscov[j];
        if (list[j]) list[j] = atomicExch(L.stamp + c, gen) != gen;  // else another block listed it
      }
      const int k0 = kept;
#pragma unroll
      for (int j = 0; j < R; ++j) {
        const unsigned c = c0 + (unsigned)(j * g.nx + x);
        const unsigned below = (1u << lane) - 1u;
        const unsigned newm = __ballot_sync(FULL, list[j] && isnew[j]), bcm = __ballot_sync(FULL, list[j] && bnd[j]);
        const unsigned covm = COV ? __ballot_sync(FULL, list[j] && iscov[j]) : 0u;
        if (newm | covm) {
          unsigned got = 0;
          if (lane == 0 && newm) got = atomicAdd(&L.ctr->n_new, (unsigned)__popc(newm));
          if (COV && lane == 1 && covm) got = atomicAdd(&L.ctr->n_cov, (unsigned)__popc(covm));
          const unsigned base_new = __shfl_sync(FULL, got, 0), base_cov = __shfl_sync(FULL, got, 1);
          if (list[j] && isnew[j]) {
            const unsigned k = base_new + __popc(newm & below);
            if (k < L.cap_new) L.new_cell[k] = c;
            else atomicOr(&L.ctr->status, STATUS_NEW_OVERFLOW);
          }
          if (COV && list[j] && iscov[j]) {
            const unsigned k = base_cov + __popc(covm & below);
            if (k < L.cap_new) L.cov_cell[k] = c;
            else atomicOr(&L.ctr->status, STATUS_NEW_OVERFLOW);
          }
        }
        if (list[j] && bnd[j]) {
          const int k = kept + __popc(bcm & below);
          K.x[k] = (uint32_t)x;
          K.yz[k] = (uint32_t)(y + j) | ((uint32_t)z << 16);
          K.mask[k] = (uint32_t)(lane | j << 5);  // where it is in the words, until its mask below
        }
        kept += __popc(bcm);
      }
      __syncwarp();
      // the link masks of the nodes just kept, a lane each
      for (int k = k0 + lane; k < kept; k += 32) {
        const int l = (int)(K.mask[k] & 31u), j = (int)(K.mask[k] >> 5);
        uint32_t mask = 0;
#pragma unroll
        for (int d = 1; d < 19; ++d) mask |= (W[(R + 2) * (cz(d) + 1) + cy(d) + 1 + j] >> (l + cx(d)) & 1u) << d;
        K.mask[k] = mask;
      }
      __syncwarp();
      while (kept >= 32) append_boundary(L, K, kept -= 32, 32, lane);
      __syncwarp();
    }
  }
  if (kept) append_boundary(L, K, 0, kept, lane);
}

cudaError_t launch_classify(const ParticleLaunch& L, cudaStream_t s) {
  if (L.np == 0) return cudaSuccess;
  const auto kernel = L.cls_unit == 1 ? (L.cover_uncover ? k_classify<true, 1> : k_classify<false, 1>)
                                      : (L.cover_uncover ? k_classify<true, 4> : k_classify<false, 4>);
  kernel<<<L.classify_blocks, 32 * CLS_WARPS, 0, s>>>(L);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Wall fraction of each link, FP32 storage (16 bits: k_links16.cu): root q in (0, 1]
// of g(q) = f_p(x_f + q e_d) - 1 (Sec. 2.3.2; reading A7: along the link that points
// into the solid, c0 = 1).
//
// In the lattice frame, with the balls' centres turned once per step (k_flag,
// FP64): a link point relative to floor X is n + q e with whole numbers n and e.
//
// Stage 1, FP32: Newton steps on h(q) = f^(-1/2) - 1, which has the same root
// and is close to linear along a link for fields of the form k / r^2 (the
// distance to a lone ball over its radius), kept inside a shrinking bracket
// [lo, hi] (bisection when a step leaves it), until a step is below 0.03.  The
// FP32 field's noise, divided by g'(q) = e . grad f (small on large smooth
// particles and on links that meet the surface at a grazing angle), leaves
// errors up to ~1e-4.
// Stage 2: Newton steps on the same h from an accurate residual g(q) (below),
// inside a bracket that starts at [0, 1] (the exact flags guarantee
// g(0) < 0 <= g(1)) and moves with the accurate signs.  A step ends it when it
// is below 2e-5 or when the error Newton's quadratic convergence leaves behind,
// |h'' / 2 h'| step^2, is below 1e-7 (usually the first step).  A link that
// grazes the surface takes more: with both roots of a sphere within 1e-3 of each other
// a step halves the error until it is as small as their distance, and one from
// between them leaves the bracket (bisection), so that up to 24 steps are
// allowed (four left 4e-4 at a depth of 1e-7 lu, 3e-5 at 1e-5).
//
// The residual: q = qh + ql with qh on the particle's grid, so that a link point
// less a ball's centre is u + m, u a multiple of the grid (exact) and m below
// about one grid spacing.  |u|^2 is exact in FP32 (link_grid_of), and
// r^2 = |u|^2 + m . (2 u + m), where the second term is 2^-10 of the first
// or less: its FP32 rounding is 2^-34 of r^2.  A quotient t = k / r^2 is split into
// a multiple of 2^-22, whose sum over the balls is exact near f = 1, and a
// remainder of FP32.  About 40 instructions a ball; float-float arithmetic
// throughout (TwoSum and products of pairs in the body frame) took over 100.
// Bound by FP32 issue: 3.35 M links on 300 particles of 8 to 64 balls 491 us, 842
// before; against FP64 the largest error of 2.3 M links is 1.3e-7 (before 6.9e-7).
// ---------------------------------------------------------------------------
namespace {
// g(q) = f(n + q e) - 1; g'(q) and g''(q) in FP32 (ee = e . e).  EXACT: |u|^2
// is exact (link_grid_of); otherwise its squares are summed as float pairs.
template <bool EXACT>
__device__ __forceinline__ float residual(const float4* __restrict__ bw, int nb, const float n[3], const float e[3],
                                          float q, float grid, float inv_grid, float ee, float& gp, float& gpp) {
  const float qh = rintf(q * inv_grid) * grid, ql = q - qh;
  float w[3], j[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    w[k] = __fmaf_rn(qh, e[k], n[k]);
    j[k] = ql * e[k];
  }
  float gh = 0.f, gl = 0.f, d1 = 0.f, d2 = 0.f, d3 = 0.f;
#pragma unroll 2
  for (int b = 0; b < nb; ++b) {
    const float4 h = __ldg(bw + 3 * b + 1), l = __ldg(bw + 3 * b + 2);
    const float u0 = w[0] - h.x, u1 = w[1] - h.y, u2 = w[2] - h.z;
    const float m0 = j[0] - l.x, m1 = j[1] - l.y, m2 = j[2] - l.z;
    const float y0 = u0 + m0, y1 = u1 + m1, y2 = u2 + m2;
    float A = __fmul_rn(u0, u0), D;
    if (EXACT) {
      A = __fmaf_rn(u2, u2, __fmaf_rn(u1, u1, A));
      D = m0 * (u0 + y0);
    } else {
      float lo = __fmaf_rn(u0, u0, -A);
#pragma unroll
      for (int k = 1; k < 3; ++k) {
        const float u = k == 1 ? u1 : u2, p = __fmul_rn(u, u), s = __fadd_rn(A, p), v = __fsub_rn(s, A);
        lo += __fmaf_rn(u, u, -p) + __fadd_rn(__fsub_rn(A, __fsub_rn(s, v)), __fsub_rn(p, v));
        A = s;
      }
      D = __fmaf_rn(m0, u0 + y0, lo);
    }
    D = __fmaf_rn(m2, u2 + y2, __fmaf_rn(m1, u1 + y1, D));
    const float s = __fadd_rn(A, D), r = __fadd_rn(__fsub_rn(A, s), D);  // r^2 = s + r
    const float ir = rcp_start(s);
    const float t = __fsub_rn(__fmaf_rn(h.w, ir, 3.0f), 3.0f);  // k / s to a multiple of 2^-22
    float res = __fmaf_rn(-t, s, h.w);
    res = __fmaf_rn(-t, r, res) + l.w;
    gh += t;
    gl = __fmaf_rn(res, ir, gl);
    // with v = y . e / r^2: g' = -2 sum t v, g'' = sum t (8 v^2 - 2 e.e / r^2)
    const float v = __fmaf_rn(y2, e[2], __fmaf_rn(y1, e[1], y0 * e[0])) * ir, tv = t * v;
    d1 += tv;
    d2 = __fmaf_rn(tv, v, d2);
    d3 = __fmaf_rn(t, ir, d3);
  }
  gp = -2.0f * d1;
  gpp = __fmaf_rn(8.0f, d2, -2.0f * ee * d3);
  return (gh - 1.0f) + gl;
}

// The root q of one link from its node n and direction e over the particle's nb balls bw.
template <bool EXACT>
__device__ __forceinline__ float link_root(const float4* __restrict__ bw, int nb, const float n[3], const float e[3],
                                           float grid) {
  // stage 1: FP32 Newton on h = f^(-1/2) - 1
  float lo = 0.f, hi = 1.f, q = 0.5f;
  for (int it = 0; it < 24; ++it) {
    float f0 = 0.f, f1 = 0.f, s0 = 0.f, s1 = 0.f, w[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) w[k] = __fmaf_rn(q, e[k], n[k]);
    int b = 0;
#pragma unroll 2
    for (; b + 2 <= nb; b += 2) {
      const float4 ca = __ldg(bw + 3 * b), cb = __ldg(bw + 3 * b + 3);
      const float u0 = w[0] - ca.x, u1 = w[1] - ca.y, u2 = w[2] - ca.z;
      const float v0 = w[0] - cb.x, v1 = w[1] - cb.y, v2 = w[2] - cb.z;
      const float iu = rcp_start(u0 * u0 + u1 * u1 + u2 * u2), iv = rcp_start(v0 * v0 + v1 * v1 + v2 * v2);
      const float tu = ca.w * iu, tv = cb.w * iv;
      f0 += tu;
      f1 += tv;
      // f' = -2 sum k (u . e) / r^4: the factor -2 is applied to the sums
      s0 = __fmaf_rn(tu * iu, u0 * e[0] + u1 * e[1] + u2 * e[2], s0);
      s1 = __fmaf_rn(tv * iv, v0 * e[0] + v1 * e[1] + v2 * e[2], s1);
    }
    if (b < nb) {
      const float4 ca = __ldg(bw + 3 * b);
      const float u0 = w[0] - ca.x, u1 = w[1] - ca.y, u2 = w[2] - ca.z;
      const float iu = rcp_start(u0 * u0 + u1 * u1 + u2 * u2);
      const float tu = ca.w * iu;
      f0 += tu;
      s0 = __fmaf_rn(tu * iu, u0 * e[0] + u1 * e[1] + u2 * e[2], s0);
    }
    const float f = f0 + f1, fp = -2.f * (s0 + s1);
    if (f >= 1.f) hi = q;
    else lo = q;
    // Newton on h: q + 2 f (1 - sqrt f) / f'
    const float step = 2.f * f * (1.f - f * rsqrtf(f)) / fp;
    float qn = q + step;
    // a step below 0.03 ends the stage (taken, clamped to the bracket): h is
    // close to linear, so the step leaves about the FP32 field's noise behind,
    // which the accurate stage removes
    if (fabsf(step) < 0.03f) {
      q = fminf(fmaxf(qn, lo), hi);
      break;
    }
    if (!(qn > lo && qn < hi)) qn = 0.5f * (lo + hi);
    q = qn;
    if (hi - lo < 1e-6f) break;
  }
  // stage 2: Newton on h from the accurate residual
  lo = 0.f;
  hi = 1.f;
  const float ee = e[0] * e[0] + e[1] * e[1] + e[2] * e[2], inv_grid = 1.0f / grid;
  for (int it = 0; it < 24; ++it) {
    float gp, gpp;
    const float g = residual<EXACT>(bw, nb, n, e, q, grid, inv_grid, ee, gp, gpp);
    if (g >= 0.f) hi = q;
    else lo = q;
    // 2 f (1 - sqrt f) / f' to second order in g = f - 1
    const float step = g / gp * __fmaf_rn(0.75f, g, 1.0f);
    float qn = q - step;
    // h'' / h' = g'' / g' - 1.5 g' / f
    const float bend = fabsf(__fmaf_rn(-1.5f * gp, gp, gpp));
    if (fabsf(step) < 2e-5f || (qn >= lo && qn <= hi && bend * step * step <= 2e-7f * fabsf(gp))) {
      q = fminf(fmaxf(qn, lo), hi);
      break;
    }
    if (!(qn > lo && qn < hi)) qn = 0.5f * (lo + hi);
    q = qn;
  }
  return q;
}
}  // namespace

__global__ void __launch_bounds__(256) k_links_q(ParticleLaunch L) {
  const unsigned nl = min(L.ctr->n_links, L.cap_links);
  const unsigned nbc = min(L.ctr->n_bc, L.cap_bc);
  for (unsigned l = blockIdx.x * blockDim.x + threadIdx.x; l < nl; l += gridDim.x * blockDim.x) {
    const unsigned bi = L.link_bc[l];
    if (bi >= nbc) continue;
    // an entry of this step: inside the range of the node it names, whose
    // links all fitted (entries of a node that overflowed were not written)
    const unsigned loff = L.bc_loff[bi], m = __popc(L.bc_mask[bi]);
    if (l < loff || l - loff >= m || (unsigned long long)loff + m > (unsigned long long)L.cap_links) continue;
    const int d = L.link_dir[l];
    const DevParticle& P = L.P[L.link_p[l]];
    // node indices of particle lists fit in 32 bits
    const unsigned cu = L.bc_cell[bi], row = cu / (unsigned)L.g.nx;
    const int x = (int)(cu - row * (unsigned)L.g.nx), z = (int)(row / (unsigned)L.g.ny), y = (int)(row - (unsigned)z * L.g.ny);
    const float n[3] = {(float)(x - P.pos_i[0]), (float)(y - P.pos_i[1]), (float)(z - P.pos_i[2])};
    const float e[3] = {(float)lex(d), (float)ley(d), (float)lez(d)};
    const float4* bw = L.balls_w + 3 * (size_t)P.ball_off;
    const float grid = P.link_grid;
    const float q = P.Rb_f < LINK_GRID_RB ? link_root<true>(bw, P.n_balls, n, e, grid)
                                          : link_root<false>(bw, P.n_balls, n, e, grid);
    L.link_q[l] = fminf(fmaxf(q, 1e-6f), 1.0f);
  }
}

cudaError_t launch_links_q(const ParticleLaunch& L, int grid, cudaStream_t s) {
  if (L.np == 0) return cudaSuccess;
  // no more blocks than the link list's capacity can use
  const unsigned long long need = ((unsigned long long)L.cap_links + 255ull) / 256ull;
  if (need < (unsigned long long)grid) grid = need < 1 ? 1 : (int)need;
  if (L.balls_s) return launch_links_q16(L, grid, s);
  k_links_q<<<grid, 256, 0, s>>>(L);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Rigid-body update, eight lanes of a warp per particle (rigid_dev.cuh).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(128) k_integrate(IntegrateLaunch L) {
  const int first = (int)blockIdx.x * (128 / RIGID_LANES);
  integrate_particles(L, first, min(L.np, first + 128 / RIGID_LANES));
}

cudaError_t launch_integrate(const IntegrateLaunch& L, cudaStream_t s) {
  if (L.np == 0) return cudaSuccess;
  const int per = 128 / RIGID_LANES;
  k_integrate<<<(L.np + per - 1) / per, 128, 0, s>>>(L);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Mass properties: midpoint quadrature of the indicator f >= 1 (FP32 with the
// FP64 guard band), FP64 moment sums per block.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_mass(const float4* balls, const double* balls_d, int nb, double Rb,
                                              double h, int n, double* partials) {
  __shared__ double red[10][256];
  double acc[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
  const long long total = (long long)n * n * n;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int ix = (int)(i % n), iy = (int)((i / n) % n), iz = (int)(i / ((long long)n * n));
    const double X = __dadd_rn(-Rb, __dmul_rn(ix + 0.5, h));
    const double Y = __dadd_rn(-Rb, __dmul_rn(iy + 0.5, h));
    const double Z = __dadd_rn(-Rb, __dmul_rn(iz + 0.5, h));
    if (mass_sample_inside(balls, balls_d, nb, X, Y, Z)) mass_sample_accumulate(acc, X, Y, Z);
  }
  for (int k = 0; k < 10; ++k) red[k][threadIdx.x] = acc[k];
  __syncthreads();
  for (int st = blockDim.x / 2; st > 0; st >>= 1) {
    if ((int)threadIdx.x < st)
      for (int k = 0; k < 10; ++k) red[k][threadIdx.x] += red[k][threadIdx.x + st];
    __syncthreads();
  }
  if (threadIdx.x == 0)
    for (int k = 0; k < 10; ++k) partials[10 * blockIdx.x + k] = red[k][0];
}

cudaError_t launch_mass_quadrature(const float4* balls, const double* balls_d, int n_balls, double Rb, double h,
                                   int n_side, double* partials, int blocks, cudaStream_t s) {
  k_mass<<<blocks, 256, 0, s>>>(balls, balls_d, n_balls, Rb, h, n_side, partials);
  return cudaGetLastError();
}

}  // namespace mi
