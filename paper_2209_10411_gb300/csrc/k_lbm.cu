// Lattice kernels: bulk pull stream-collide (D3Q19 BGK) and population
// packing.  The stream-collide follows the LBM basis of the paper's
// Sec. 2.3.2 (distributions G_i, weights omega_i, C = 1) with the D3Q19 BGK
// lattice; domain walls are halfway bounce-back with the moving-wall term
// 6 w_i rho0 (e_i . u_wall), the same form the paper gives for moving
// particle walls.
//
// Memory: populations are SoA, one plane of ncell elements per direction,
// x fastest.  One thread updates one node: 19 pulled loads (neighbour x - e_i,
// misaligned by one element for the 10 directions with e_x != 0; the L1/L2
// absorb the sector overlap so DRAM sees each element once), FP32 collision,
// 19 streaming stores.  Algorithmic traffic: 19 * 2 * sizeof(storage) bytes
// per node update.
#include <climits>
#include "mi_internal.cuh"

namespace mi {

// Division of a 32-bit index by a constant of the launch: q = floor(c / d) by
// a multiplication (Granlund and Montgomery 1994: with l = ceil(log2 d) and
// m = floor(2^32 (2^l - d) / d) + 1, t = floor(m c / 2^32),
// q = (t + (c - t) / 2) / 2^(l - 1)).
struct FastDiv {
  unsigned m, s1, s2;
  __device__ __forceinline__ unsigned div(unsigned c) const {
    const unsigned t = __umulhi(m, c);
    return (t + ((c - t) >> s1)) >> s2;
  }
};
static FastDiv fast_div(unsigned d) {
  unsigned l = 0;
  while (l < 32 && (1ull << l) < d) ++l;
  return {(unsigned)((((1ull << l) - d) << 32) / d + 1), l > 1 ? 1u : l, l > 1 ? l - 1 : 0u};
}

// BGK collision on deviations h_i = f_i - w_i.
//   rho = 1 + sum h_i, j = sum e_i h_i (sum w_i = 1, sum w_i e_i = 0)
//   f_eq,i - w_i = w_i (rho - 1) + w_i rho (3 e.u + 4.5 (e.u)^2 - 1.5 u.u)
//   h+_i = (1 - omega) h_i + omega (f_eq,i - w_i)   [+ Guo source]
// in two forms, by storage.  Every operation of either is written out as a single
// rounding, and a direction and its opposite (2k - 1, 2k) share what is the same
// or exactly the negative.

// 1 / rho, rounded to nearest (a start within an ulp and one Newton step in fused
// operations: Markstein 1990), without the range checks of the general division.
template <class V>
__device__ __forceinline__ V inverse(V rho) {
  const V r = rcp_start(rho);
  return vfma(r, vfma(vsub(vset(0.0f, r), rho), r, vset(1.0f, r)), r);
}

// FP32 storage: the moments from the sums and differences of opposite directions,
// the odd part of the equilibrium from the momentum, the even part from the odd
// one; about 150 operations a node.
//
// omega / 36 and omega / 12 are float pairs, and the weights 1, 2 and 12 times
// them: a rounded omega w_i is the same relative error at every node and step,
// a source of mass and momentum.  The states of the particles after 20 steps of
// a 64^3 box, against 64 bits: 1.2e-10 off with pairs, 5e-10 with rounded products.
// (1 - omega) h is h - omega h in one rounding: a rounded 1 - omega is off by up to
// 2^-25 whatever omega is, at tau = 100 1e-6 and at tau = 10,000 2e-4 of the viscosity
// (and the low half of a pair would be lost in the sum with the equilibrium).
template <bool FORCE>
__device__ __forceinline__ void collide_pairs(float (&h)[19], const CollideParams& P) {
  float s[10], d[10];  // pair k: h[2k - 1] + h[2k], h[2k - 1] - h[2k]
#pragma unroll
  for (int k = 1; k < 10; ++k) {
    s[k] = vadd(h[2 * k - 1], h[2 * k]);
    d[k] = vsub(h[2 * k - 1], h[2 * k]);
  }
  const float drho = vadd(vadd(vadd(h[0], vadd(s[1], s[2])), vadd(s[3], vadd(s[4], s[5]))),
                          vadd(vadd(s[6], s[7]), vadd(s[8], s[9])));
  float j[3], u[3];  // the momentum, 1.5 times the velocity
  j[0] = vadd(vadd(d[1], vadd(d[4], d[5])), vadd(d[6], d[7]));
  j[1] = vadd(vadd(d[2], vsub(d[4], d[5])), vadd(d[8], d[9]));
  j[2] = vadd(vadd(d[3], vsub(d[6], d[7])), vsub(d[8], d[9]));
  const float r15 = vmul(1.5f, inverse(vadd(1.0f, drho)));
  if (FORCE)
    for (int a = 0; a < 3; ++a) j[a] = vadd(j[a], 0.5f * P.force[a]);
  float v[3];  // omega / 12 times the momentum: odd part 3 omega w_i rho e.u, even part that times 1.5 e.u
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    u[a] = vmul(j[a], r15);
    v[a] = vfma(P.c12[0], j[a], vmul(P.c12[1], j[a]));
  }
  const float base = vsub(drho, vfma(j[0], u[0], vfma(j[1], u[1], vmul(j[2], u[2]))));  // drho - 1.5 rho u.u
  const float based = vfma(P.c36[0], base, vmul(P.c36[1], base)), basea = vadd(based, based);
  const float om = P.omega;
  float uF = 0.f;
  if (FORCE) uF = vfma(P.force[0], u[0], vfma(P.force[1], u[1], vmul(P.force[2], u[2])));
  const auto relax = [&](int i, float e) { h[i] = vadd(vfma(-om, h[i], h[i]), e); };
  {
    float e0 = vmul(12.0f, based);
    if (FORCE) e0 = vfma(-2.0f * (1.0f - 0.5f * om) * wq(0), uF, e0);
    relax(0, e0);
  }
#pragma unroll
  for (int k = 1; k < 10; ++k) {
    const int i = 2 * k - 1;
    // 1.5 e_i . u: the first non-zero component of every odd direction is +1
    const int a = cx(i) ? 0 : (cy(i) ? 1 : 2), b = cz(i) ? 2 : 1;
    const bool plus = (b == 1 ? cy(i) : cz(i)) > 0;
    const float eu = k <= 3 ? u[a] : (plus ? vadd(u[a], u[b]) : vsub(u[a], u[b]));
    float odd = k <= 3 ? vadd(v[a], v[a]) : (plus ? vadd(v[a], v[b]) : vsub(v[a], v[b]));
    float even = vfma(odd, eu, k <= 3 ? basea : based);
    if (FORCE) {
      const float g = (1.0f - 0.5f * om) * wq(i);
      const float eF = cx(i) * P.force[0] + cy(i) * P.force[1] + cz(i) * P.force[2];
      even = vadd(even, vfma(6.0f * g * eF, eu, vmul(-2.0f * g, uF)));
      odd = vadd(odd, 3.0f * g * eF);
    }
    relax(i, vadd(even, odd));
    relax(i + 1, vsub(even, odd));
  }
}

// The momentum of 16-bit storages: by the differences of opposite directions, or
// added direction by direction (SEQ: boundary nodes, links, covered nodes).
template <bool SEQ, class V>
__device__ __forceinline__ void momentum(const V (&h)[19], V (&j)[3]) {
  if (SEQ) {
    j[0] = vsub(h[1], h[2]);
    j[1] = vsub(h[3], h[4]);
    j[2] = vsub(h[5], h[6]);
#pragma unroll
    for (int i = 7; i < 19; ++i) {
      if (cx(i)) j[0] = cx(i) > 0 ? vadd(j[0], h[i]) : vsub(j[0], h[i]);
      if (cy(i)) j[1] = cy(i) > 0 ? vadd(j[1], h[i]) : vsub(j[1], h[i]);
      if (cz(i)) j[2] = cz(i) > 0 ? vadd(j[2], h[i]) : vsub(j[2], h[i]);
    }
  } else {
    V d[10];
#pragma unroll
    for (int k = 1; k < 10; ++k) d[k] = vsub(h[2 * k - 1], h[2 * k]);
    j[0] = vadd(vadd(vadd(vadd(d[1], d[4]), d[5]), d[6]), d[7]);
    j[1] = vadd(vadd(vsub(vadd(d[2], d[4]), d[5]), d[8]), d[9]);
    j[2] = vsub(vadd(vsub(vadd(d[3], d[6]), d[7]), d[8]), d[9]);
  }
}

// 16-bit storages, one node (V = float) or two (V = F32x2, packed FP32 pairs: one
// instruction for both; a node's result does not depend on which).  Here the order of
// the operations is part of the result: a value near the middle of two
// representable ones moves by a whole unit (2^-11 or 2^-8 of it) when its FP32 value
// moves by one ulp, the bounce-back hands such a unit on to the particles, and a
// light one's velocity then differs by 1e-7 after 20 steps.  So it is
// fixed, direction by direction,
//   fma(omega, fma(w_i, fma(rho, fma(-1.5, u.u, fma(3, e.u, 4.5 e.u e.u)), drho), -h_i), h_i)
// with omega = 1 / tau rounded once.  About 170 operations a node: 256 x 256 x 512 in
// FP16 takes 402 us with it, 397 with the form above.
template <bool FORCE, bool SEQ = false, class V>
__device__ __forceinline__ void collide_ordered(V (&h)[19], const CollideParams& P) {
  V drho = h[0];
#pragma unroll
  for (int i = 1; i < 19; ++i) drho = vadd(drho, h[i]);
  V u[3];
  momentum<SEQ>(h, u);
  const V rho = vadd(vset(1.0f, drho), drho), irho = inverse(rho);
#pragma unroll
  for (int a = 0; a < 3; ++a) u[a] = vmul(FORCE ? vadd(u[a], vset(0.5f * P.force[a], irho)) : u[a], irho);
  const V usq = vfma(u[2], u[2], vfma(u[0], u[0], vmul(u[1], u[1])));
  const V m15 = vset(-1.5f, rho), m_om = vset(-P.omega, rho), three = vset(3.0f, rho), m_three = vset(-3.0f, rho);
  V uF;
  if (FORCE) uF = vfma(u[2], vset(P.force[2], rho), vfma(u[0], vset(P.force[0], rho), vmul(u[1], vset(P.force[1], rho))));
  // h_i relaxed towards w_i (drho + rho n), n the bracket above; f: the source's bracket
  const auto relax = [&](int i, V n, V f) {
    const V x = vfma(vset(-wq(i), rho), vfma(rho, n, drho), h[i]);  // exactly the negative of f_eq - w - h
    h[i] = vfma(m_om, x, h[i]);
    if (FORCE) h[i] = vfma(vset((1.0f - 0.5f * P.omega) * wq(i), rho), f, h[i]);
  };
  relax(0, vmul(m15, usq), FORCE ? vmul(m_three, uF) : rho);
#pragma unroll
  for (int k = 1; k < 10; ++k) {
    const int i = 2 * k - 1;
    // e_i . u: the first non-zero component of every odd direction is +1
    const int a = cx(i) ? 0 : (cy(i) ? 1 : 2), b = cz(i) ? 2 : 1;
    const V eu = k <= 3 ? u[a] : ((b == 1 ? cy(i) : cz(i)) > 0 ? vadd(u[a], u[b]) : vsub(u[a], u[b]));
    const V sq = vmul(vmul(vset(4.5f, rho), eu), eu);
    const V np = vfma(m15, usq, vfma(three, eu, sq)), nm = vfma(m15, usq, vfma(m_three, eu, sq));
    V fp = rho, fm = rho;
    if (FORCE) {
      const V eF = vset(cx(i) * P.force[0] + cy(i) * P.force[1] + cz(i) * P.force[2], rho), n9 = vmul(vset(9.0f, rho), eu);
      fp = vfma(n9, eF, vmul(three, vsub(eF, uF)));
      fm = vfma(n9, eF, vmul(m_three, vadd(eF, uF)));
    }
    relax(i, np, fp);
    relax(i + 1, nm, fm);
  }
}

template <int ST, bool FORCE, bool SEQ = false>
__device__ __forceinline__ void collide(float (&h)[19], const CollideParams& P) {
  if constexpr (ST == MI_STORE_F32) collide_pairs<FORCE>(h, P);
  else collide_ordered<FORCE, SEQ>(h, P);
}

template <int ST, bool FORCE>
__device__ __forceinline__ void collide_store(float (&h)[19], typename Store<ST>::T* __restrict__ B,
                                              long long plane, long long c, const CollideParams& P) {
  collide<ST, FORCE>(h, P);
#pragma unroll
  for (int i = 0; i < 19; ++i) Store<ST>::put(B + i * plane + c, i, h[i]);
}

// Pull streaming (with halfway bounce-back at domain walls) of node (x, y, z),
// c its linear index: the 19 incoming deviations h_i = f_i - w_i.  At a face
// the source index is selected (the far end of a periodic axis, or the node's
// own opposite population at a wall) before one load per direction, so all 19
// loads are in flight together: with a branch per direction they were waited
// for one after another, and every warp that holds a row's end paid for it.
// Directions i with bit opp(i) of `own` set take the node's own opposite
// population too (links into a solid).
template <int ST>
__device__ __forceinline__ void pull_node(const typename Store<ST>::T* __restrict__ A, const LatticeGeom& g,
                                          const CollideParams& P, int x, int y, int z, long long c, float (&h)[19],
                                          uint32_t own = 0u) {
  const int nxy = g.nx * g.ny;
  // per axis: source offset and wall flag for e = +1 (source below) and e = -1
  const bool lo[3] = {x == 0, y == 0, z == 0}, hi[3] = {x == g.nx - 1, y == g.ny - 1, z == g.nz - 1};
  const int n[3] = {g.nx, g.ny, g.nz}, step[3] = {1, g.nx, nxy};
  int om[3], op[3];
  bool wm[3], wp[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    wm[a] = lo[a] && !g.periodic[a];
    wp[a] = hi[a] && !g.periodic[a];
    om[a] = lo[a] ? (n[a] - 1) * step[a] : -step[a];
    op[a] = hi[a] ? -(n[a] - 1) * step[a] : step[a];
  }
#pragma unroll
  for (int i = 0; i < 19; ++i) {
    const int e[3] = {cx(i), cy(i), cz(i)};
    const bool bx = e[0] == 1 ? wm[0] : (e[0] == -1 ? wp[0] : false);
    const bool by = e[1] == 1 ? wm[1] : (e[1] == -1 ? wp[1] : false);
    const bool bz = e[2] == 1 ? wm[2] : (e[2] == -1 ? wp[2] : false);
    const bool wall = bx | by | bz;
    int off = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) off += e[a] == 1 ? om[a] : (e[a] == -1 ? op[a] : 0);
    const long long at = wall || ((own >> opp(i)) & 1u) ? opp(i) * g.plane + c : i * g.plane + (c + off);
    h[i] = Store<ST>::dev(A + at, i);  // w_opp = w_i
    // halfway bounce-back: f_in,i(x) = f+_opp(i)(x) + 6 w_i rho0 e_i.u_wall; a
    // corner crossing is attributed to x, then y, then z
    if (i && wall)
      h[i] += bx ? P.bb_wall[e[0] == 1 ? 0 : 1][i] : (by ? P.bb_wall[e[1] == 1 ? 2 : 3][i] : P.bb_wall[e[2] == 1 ? 4 : 5][i]);
  }
}

// The same away from the faces: constant offsets.
template <int ST>
__device__ __forceinline__ void pull_interior(const typename Store<ST>::T* __restrict__ A, const LatticeGeom& g,
                                              long long c, float (&h)[19]) {
  const long long nxy = (long long)g.nx * g.ny;
#pragma unroll
  for (int i = 0; i < 19; ++i) {
    const long long off = cx(i) + (long long)g.nx * cy(i) + nxy * cz(i);
    h[i] = Store<ST>::dev(A + i * g.plane + (c - off), i);
  }
}

// Pull and collide one node.
template <int ST, bool FORCE>
__device__ __forceinline__ void update_node(const typename Store<ST>::T* __restrict__ A,
                                            typename Store<ST>::T* __restrict__ B, const LatticeGeom& g,
                                            const CollideParams& P, int x, int y, int z, long long c) {
  float h[19];
  pull_node<ST>(A, g, P, x, y, z, c, h);
  collide_store<ST, FORCE>(h, B, g.plane, c, P);
}

// Every node of the lattice, a thread per node, the blocks over the linear node
// index (x fastest): a warp's 32 nodes are one aligned stretch of every plane
// whatever nx is, and no lane idles at a row's end.  A warp that holds no face
// node takes the constant offsets, any other the selecting pull for all its
// lanes, so no warp runs both.  With particles this runs concurrently with
// the particle phases: boundary nodes are rewritten afterwards by k_boundary,
// solid nodes hold unspecified values, and the nodes next to a node uncovered
// this step (whose refilled populations this kernel may not have seen) are
// recomputed by k_near.  Nodes anywhere else have no solid or uncovered
// neighbour, so their update here is final.
//
// Bound by HBM: FP32 alone, 256 x 256 x 512 in 0.786 ms = 6.49 TB/s (0.955 of a
// copy), 512^3 in 3.05 ms = 6.68 TB/s (0.98), 141 x 83 x 119 in 37 us.  With
// rows as blocks, a branch per direction at the faces and the collision formed
// direction by direction these took 0.955 ms, 3.53 ms and 74 us.  Blocks of 64
// threads measured best from 64^3 to 512^3 (32: up to 3 % more, 128: 1 %).  The
// registers decide whether the 19 loads are issued together: 48 (40 with a body
// force, 0.787 ms), where the compiler's own choices of 42 and 48 took 0.799 and 0.801.
template <int ST, bool FORCE>
__global__ void __launch_bounds__(256, FORCE ? 6 : 5) k_bulk(const typename Store<ST>::T* __restrict__ A,
                                              typename Store<ST>::T* __restrict__ B, LatticeGeom g,
                                              CollideParams P, FastDiv by_nx, FastDiv by_ny, unsigned ncell) {
  const unsigned c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= ncell) return;
  const unsigned row = by_nx.div(c), zu = by_ny.div(row);
  const int x = (int)(c - row * (unsigned)g.nx), y = (int)(row - zu * (unsigned)g.ny), z = (int)zu;
  const bool interior = (x > 0) & (x < g.nx - 1) & (y > 0) & (y < g.ny - 1) & (z > 0) & (z < g.nz - 1);
  float h[19];
  if (__all_sync(__activemask(), interior)) pull_interior<ST>(A, g, c, h);
  else pull_node<ST>(A, g, P, x, y, z, c, h);
  collide_store<ST, FORCE>(h, B, g.plane, c, P);
}

template <int ST, bool FORCE>
static cudaError_t launch_bulk_t(const BulkLaunch& L, cudaStream_t s) {
  using T = typename Store<ST>::T;
  const unsigned n = (unsigned)((long long)L.g.nx * L.g.ny * L.g.nz), bx = (unsigned)L.block_x;
  k_bulk<ST, FORCE><<<n / bx + (n % bx ? 1u : 0u), bx, 0, s>>>(static_cast<const T*>(L.A), static_cast<T*>(L.B), L.g,
                                                               L.p, fast_div((unsigned)L.g.nx), fast_div((unsigned)L.g.ny), n);
  return cudaGetLastError();
}

// 16-bit storages: W = 2 or 4 x-adjacent nodes per thread (x0 .. x0 + W - 1, x0
// a multiple of W), the blocks over the linear groups of W nodes.  A direction
// with e_x = 0 is one aligned 32- or 64-bit load; for e_x = +1 (-1) the shifted
// elements are the thread's own aligned word plus the one element beside it,
// joined by shifts and a byte permute.  The values stay packed two to a
// register until the collision, which takes two nodes at a time in packed FP32
// pairs, and every direction is one aligned streaming store.  Groups at the x
// faces stay on this path (no warp mixes paths): the element beside them comes
// from the other end of the row when x is periodic, else the face node's
// pulled value is replaced after unpacking by its halfway bounce-back.  Rows
// on the y and z faces take the general per-node path.  The same concurrency
// contract as k_bulk.  Requires nx % W == 0.
//
// Bound by HBM: 256 x 256 x 512 FP16 in 0.402 ms = 6.34 TB/s (0.93 of a copy),
// 512^3 in 1.60 ms, four nodes per thread.  With unpacked FP32 arithmetic, rows
// as blocks and branches per direction at the faces these took 0.522 and 1.99
// ms: that kernel waited for instruction issue.  Two nodes per thread reach 0.430
// ms (more instructions a byte) but, with twice the threads, win on small
// lattices: 64^3 in 8 against 13 us; the one-node kernel takes 0.611 ms.  Five
// blocks of 128 threads per SM (96 registers, a few spilled) measured 4 % faster
// than four (128 registers), 5 % with a body force (0.425 ms).
template <int ST> __device__ __forceinline__ float2 unpack2(unsigned w);
template <> __device__ __forceinline__ float2 unpack2<MI_STORE_F16_DEV>(unsigned w) {
  return __half22float2(*reinterpret_cast<const __half2*>(&w));
}
template <> __device__ __forceinline__ float2 unpack2<MI_STORE_BF16_DEV>(unsigned w) {
  return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
}
template <int ST> __device__ __forceinline__ unsigned pack2(float a, float b);
template <> __device__ __forceinline__ unsigned pack2<MI_STORE_F16_DEV>(float a, float b) {
  const __half2 v = __floats2half2_rn(a, b);
  return *reinterpret_cast<const unsigned*>(&v);
}
template <> __device__ __forceinline__ unsigned pack2<MI_STORE_BF16_DEV>(float a, float b) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const unsigned*>(&v);
}

// W 16-bit elements in W / 2 words, one aligned access
template <int W> struct Words;
template <> struct Words<2> {
  unsigned w[1];
  __device__ __forceinline__ void load(const unsigned short* p) { w[0] = __ldg(reinterpret_cast<const unsigned*>(p)); }
  __device__ __forceinline__ void store(unsigned short* p) const { __stcs(reinterpret_cast<unsigned*>(p), w[0]); }
};
template <> struct Words<4> {
  unsigned w[2];
  __device__ __forceinline__ void load(const unsigned short* p) {
    const uint2 v = __ldg(reinterpret_cast<const uint2*>(p));
    w[0] = v.x;
    w[1] = v.y;
  }
  __device__ __forceinline__ void store(unsigned short* p) const {
    __stcs(reinterpret_cast<uint2*>(p), make_uint2(w[0], w[1]));
  }
};

template <int ST, bool FORCE, int W>
__global__ void __launch_bounds__(128, W == 4 ? 5 : (FORCE ? 7 : 8))
    k_bulk16(const typename Store<ST>::T* __restrict__ A, typename Store<ST>::T* __restrict__ B, LatticeGeom g,
             CollideParams P, FastDiv by_groups, FastDiv by_ny, unsigned ngroups) {
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= ngroups) return;
  const unsigned per_row = (unsigned)g.nx / W, row = by_groups.div(t), zu = by_ny.div(row);
  const int x0 = W * (int)(t - row * per_row), y = (int)(row - zu * (unsigned)g.ny), z = (int)zu;
  const long long c0 = (long long)W * t;
  if (!((y > 0) & (y < g.ny - 1) & (z > 0) & (z < g.nz - 1))) {
#pragma unroll 1
    for (int k = 0; k < W; ++k) update_node<ST, FORCE>(A, B, g, P, x0 + k, y, z, c0 + k);
    return;
  }
  const bool lo_edge = x0 == 0, hi_edge = x0 == g.nx - W, xper = g.periodic[0] != 0;
  const unsigned short* Au = reinterpret_cast<const unsigned short*>(A);
  const long long nxy = (long long)g.nx * g.ny;
  // the element before x0 and the one after x0 + W - 1 (at a wall any element
  // of the row: replaced below)
  const int before_at = lo_edge ? (xper ? g.nx - 1 : 0) : -1, after_at = hi_edge ? (xper ? W - g.nx : 0) : W;
  Words<W> in[19];
#pragma unroll
  for (int i = 0; i < 19; ++i) {
    // aligned position of node x0 in the source row of direction i
    const unsigned short* src = Au + i * g.plane + (c0 - ((long long)g.nx * cy(i) + nxy * cz(i)));
    in[i].load(src);
    if (cx(i) == 1) {  // elements x0 - 1 .. x0 + W - 2
      const unsigned before = __ldg(src + before_at), first = in[i].w[0];
      if (W == 4) in[i].w[W / 2 - 1] = __byte_perm(first, in[i].w[W / 2 - 1], 0x5432);
      in[i].w[0] = before | (first << 16);
    } else if (cx(i) == -1) {  // elements x0 + 1 .. x0 + W
      const unsigned after = __ldg(src + after_at);
      if (W == 4) in[i].w[0] = __byte_perm(in[i].w[0], in[i].w[W / 2 - 1], 0x5432);
      in[i].w[W / 2 - 1] = (in[i].w[W / 2 - 1] >> 16) | (after << 16);
    }
  }
#pragma unroll
  for (int k = 0; k < W / 2; ++k) {
    float2 v[19];
#pragma unroll
    for (int i = 0; i < 19; ++i) v[i] = unpack2<ST>(in[i].w[k]);
    if (!xper) {
      // halfway bounce-back at the x faces: f_in,i(x) = f+_opp(i)(x) + 6 w_i rho0 e_i.u_wall
      if (k == 0 && lo_edge) {
#pragma unroll
        for (int i = 0; i < 19; ++i)
          if (cx(i) == 1) v[i].x = dev16<ST>(__ldg(Au + opp(i) * g.plane + c0)) + P.bb_wall[0][i];
      }
      if (k == W / 2 - 1 && hi_edge) {
#pragma unroll
        for (int i = 0; i < 19; ++i)
          if (cx(i) == -1) v[i].y = dev16<ST>(__ldg(Au + opp(i) * g.plane + c0 + W - 1)) + P.bb_wall[1][i];
      }
    }
    F32x2 h[19];
#pragma unroll
    for (int i = 0; i < 19; ++i) h[i] = pack(v[i].x, v[i].y);
    collide_ordered<FORCE>(h, P);
#pragma unroll
    for (int i = 0; i < 19; ++i) {
      const float2 r = unpack(h[i]);
      in[i].w[k] = pack2<ST>(r.x, r.y);
    }
  }
  unsigned short* Bu = reinterpret_cast<unsigned short*>(B);
#pragma unroll
  for (int i = 0; i < 19; ++i) in[i].store(Bu + i * g.plane + c0);
}

template <int ST, bool FORCE, int W>
static cudaError_t launch_bulk16_t(const BulkLaunch& L, cudaStream_t s) {
  using T = typename Store<ST>::T;
  const unsigned n = (unsigned)((long long)L.g.nx / W * L.g.ny * L.g.nz), bx = (unsigned)L.block_x;
  k_bulk16<ST, FORCE, W><<<n / bx + (n % bx ? 1u : 0u), bx, 0, s>>>(
      static_cast<const T*>(L.A), static_cast<T*>(L.B), L.g, L.p, fast_div((unsigned)L.g.nx / W),
      fast_div((unsigned)L.g.ny), n);
  return cudaGetLastError();
}

template <int ST>
static cudaError_t launch_bulk_st(const BulkLaunch& L, cudaStream_t s) {
  if constexpr (ST != MI_STORE_F32) {
    if (L.nodes == 4 && L.g.nx % 4 == 0)
      return L.forcing ? launch_bulk16_t<ST, true, 4>(L, s) : launch_bulk16_t<ST, false, 4>(L, s);
    if (L.nodes == 2 && L.g.nx % 2 == 0)
      return L.forcing ? launch_bulk16_t<ST, true, 2>(L, s) : launch_bulk16_t<ST, false, 2>(L, s);
  }
  return L.forcing ? launch_bulk_t<ST, true>(L, s) : launch_bulk_t<ST, false>(L, s);
}

cudaError_t launch_bulk(const BulkLaunch& L, cudaStream_t s) {
  if (L.block_x <= 0 || L.block_x > 256 || (L.block_x % 32) != 0) return cudaErrorInvalidValue;
  if (L.nodes > 1 && L.block_x > 128) return cudaErrorInvalidValue;
  switch (L.storage) {
    case MI_STORE_F32: return launch_bulk_st<MI_STORE_F32>(L, s);
    case MI_STORE_F16_DEV: return launch_bulk_st<MI_STORE_F16_DEV>(L, s);
    case MI_STORE_BF16_DEV: return launch_bulk_st<MI_STORE_BF16_DEV>(L, s);
  }
  return cudaErrorInvalidValue;
}

// ---------------------------------------------------------------------------
// Refill of uncovered nodes (the paper's local bounce-back refill, Sec. 2.3.2),
// applied to the stored post-collision populations f+(t) before streaming:
//   f+_i(x_new) = f+_opp(i)(x_new + e_i) + 6 w_i rho0 (e_i . u_new)
// when x_new + e_i is a fluid node that was also fluid at the previous step,
// else f_eq,i(rho0, u_new); u_new is the rigid velocity at x_new of the
// particle that covered it.  One warp per uncovered node, a lane per direction:
// few nodes are uncovered in a step, and one thread per node waited for three
// dependent loads in each of its 19 directions (19 us for one node).  With the
// cover/uncover rule the same launch also moves node momenta: an uncovered
// node's refilled momentum is taken from its particle, a covered node's
// post-collision momentum is given to the particle that covers it.
// ---------------------------------------------------------------------------
namespace {
__device__ __forceinline__ bool nbr_wrap(int x, int y, int z, int dx, int dy, int dz, const LatticeGeom& g,
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
  out = a + (long long)g.nx * (b + (long long)g.ny * c);
  return true;
}

__device__ __forceinline__ void rigid_u(const DevParticle& P, double px, double py, double pz, float u[3]) {
  const float r0 = (float)(px - P.pos[0]), r1 = (float)(py - P.pos[1]), r2 = (float)(pz - P.pos[2]);
  u[0] = P.velf[0] + (P.omegaf[1] * r2 - P.omegaf[2] * r1);
  u[1] = P.velf[1] + (P.omegaf[2] * r0 - P.omegaf[0] * r2);
  u[2] = P.velf[2] + (P.omegaf[0] * r1 - P.omegaf[1] * r0);
}

// Node coordinates of a list entry (particle lists store node indices as
// uint32, so 32-bit divisions suffice).
__device__ __forceinline__ void coords(long long c, const LatticeGeom& g, int& x, int& y, int& z) {
  const unsigned cu = (unsigned)c, row = cu / (unsigned)g.nx;
  x = (int)(cu - row * (unsigned)g.nx);
  z = (int)(row / (unsigned)g.ny);
  y = (int)(row - (unsigned)z * (unsigned)g.ny);
}

template <int ST>
__device__ __forceinline__ void moments_at(const typename Store<ST>::T* __restrict__ A, long long plane,
                                           long long c, float& rho, float u[3]) {
  float h[19];
#pragma unroll
  for (int i = 0; i < 19; ++i) h[i] = Store<ST>::dev(A + i * plane + c, i);
  float dr = 0.f;
#pragma unroll
  for (int i = 0; i < 19; ++i) dr += h[i];
  rho = 1.0f + dr;
  const float jx = (h[1] - h[2]) + (h[7] - h[8]) + (h[9] - h[10]) + (h[11] - h[12]) + (h[13] - h[14]);
  const float jy = (h[3] - h[4]) + (h[7] - h[8]) + (h[10] - h[9]) + (h[15] - h[16]) + (h[17] - h[18]);
  const float jz = (h[5] - h[6]) + (h[11] - h[12]) + (h[14] - h[13]) + (h[15] - h[16]) + (h[18] - h[17]);
  u[0] = jx / rho;
  u[1] = jy / rho;
  u[2] = jz / rho;
}
}  // namespace

namespace {
// weight and opposite of a direction given at run time (lex, ley, lez: the
// shared header's packed direction tables)
__device__ __forceinline__ float lw(int j) { return j == 0 ? (1.0f / 3.0f) : (j <= 6 ? (1.0f / 18.0f) : (1.0f / 36.0f)); }
__device__ __forceinline__ int lopp(int j) { return j == 0 ? 0 : ((j & 1) ? j + 1 : j - 1); }

// Cover/uncover rule: a node's population momentum J = sum e_i h_i (FP32, lane i
// holds h_i, added direction by direction) and its torque about the particle's
// position, sign * (J, (x - X_p) x J), added to the particle's fixed-point
// hydrodynamic sums.
__device__ __forceinline__ void add_node_momentum(long long* facc, const DevParticle* Ps, uint32_t p, int x, int y,
                                                  int z, float h, float sign, unsigned lane) {
  float all[19], J[3];
#pragma unroll
  for (int i = 1; i < 19; ++i) all[i] = __shfl_sync(0xffffffffu, h, i);
  momentum<true>(all, J);
  const DevParticle& P = Ps[p];
  const float r0 = (float)(x - P.pos[0]), r1 = (float)(y - P.pos[1]), r2 = (float)(z - P.pos[2]);
  const float v[6] = {J[0], J[1], J[2], r1 * J[2] - r2 * J[1], r2 * J[0] - r0 * J[2], r0 * J[1] - r1 * J[0]};
#pragma unroll
  for (unsigned k = 0; k < 6; ++k)
    if (lane == k)
      atomicAdd(reinterpret_cast<unsigned long long*>(facc + 6 * (size_t)p + k),
                (unsigned long long)__float2ll_rn(sign * v[k] * 1099511627776.0f));
}
}  // namespace

template <int ST>
__global__ void __launch_bounds__(128) k_refill(BoundaryLaunch L) {
  using T = typename Store<ST>::T;
  T* A = static_cast<T*>(L.A);
  const LatticeGeom& g = L.pl.g;
  const unsigned nn = min(L.pl.ctr->n_new, L.pl.cap_new);
  const float rho0 = L.p.rho0;
  const unsigned lane = threadIdx.x & 31u, wid = (blockIdx.x * blockDim.x + threadIdx.x) >> 5,
                 nw = (gridDim.x * blockDim.x) >> 5;
  const int i = lane < 19u ? (int)lane : 0;
  const int ex = lex(i), ey = ley(i), ez = lez(i), oi = lopp(i);
  const float wi = lw(i);
  for (unsigned k = wid; k < nn; k += nw) {
    const long long c = L.pl.new_cell[k];
    int x, y, z;
    coords(c, g, x, y, z);
    const uint32_t pid = L.pl.owner_prev[c];
    const DevParticle& P = L.pl.P[pid];
    float u[3];
    rigid_u(P, x, y, z, u);
    const float usq15 = 1.5f * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
    const float eu = ex * u[0] + ey * u[1] + ez * u[2];
    long long nb = c;
    const bool from = i != 0 && nbr_wrap(x, y, z, ex, ey, ez, g, nb);
    const bool fluid = (L.pl.owner_cur[nb] == OWNER_NONE) & (L.pl.owner_prev[nb] == OWNER_NONE);
    const float there = Store<ST>::dev_at(A + oi * g.plane + nb, wi);
    const float h = from && fluid ? there + 6.0f * wi * rho0 * eu
                                  : wi * (rho0 - 1.0f) + wi * rho0 * (3.0f * eu + 4.5f * eu * eu - usq15);
    if (lane < 19u) Store<ST>::put_at(A + i * g.plane + c, wi, h);
    // cover/uncover rule: the particle that uncovered the node gives up the
    // momentum of the refilled populations, sum e_i (f_i - w_i)
    if (L.pl.cover_uncover) add_node_momentum(L.pl.facc, L.pl.P, pid, x, y, z, h, -1.0f, lane);
  }
  if (!L.pl.cover_uncover) return;
  // covered nodes: the momentum of their post-collision populations f+(t)
  // (still in A: they were fluid) goes to the particle that covered them
  const unsigned nc = min(L.pl.ctr->n_cov, L.pl.cap_new);
  for (unsigned k = wid; k < nc; k += nw) {
    const long long c = L.pl.cov_cell[k];
    int x, y, z;
    coords(c, g, x, y, z);
    const float h = Store<ST>::dev_at(A + i * g.plane + c, wi);
    add_node_momentum(L.pl.facc, L.pl.P, L.pl.owner_cur[c], x, y, z, h, 1.0f, lane);
  }
}

// ---------------------------------------------------------------------------
// An uncovered node and the nodes next to it: recomputed after the refill (the
// bulk kernel may have read its populations before they were refilled), solid
// ones too, whose values nothing uses but which would otherwise depend on
// which kernel came first.  One thread per (uncovered node, direction); a node
// reached twice is written twice with the same values.
// ---------------------------------------------------------------------------
template <int ST, bool FORCE>
__device__ __forceinline__ void near_nodes(const BoundaryLaunch& L, unsigned block, unsigned blocks) {
  using T = typename Store<ST>::T;
  const T* __restrict__ A = static_cast<const T*>(L.A);
  T* __restrict__ B = static_cast<T*>(L.B);
  const LatticeGeom& g = L.pl.g;
  const unsigned nn = min(L.pl.ctr->n_new, L.pl.cap_new);
  for (unsigned t = block * blockDim.x + threadIdx.x; t < nn * 19u; t += blocks * blockDim.x) {
    const unsigned k = t / 19u;
    const int d = (int)(t - 19u * k);
    int x, y, z;
    coords(L.pl.new_cell[k], g, x, y, z);
    long long nb;
    if (!nbr_wrap(x, y, z, lex(d), ley(d), lez(d), g, nb)) continue;
    if (L.pl.cls[nb] & CLS_BOUNDARY) continue;
    int a, b, c;
    coords(nb, g, a, b, c);
    update_node<ST, FORCE>(A, B, g, L.p, a, b, c, nb);
  }
}

template <int ST, bool FORCE>
__global__ void __launch_bounds__(128) k_near(BoundaryLaunch L) {
  near_nodes<ST, FORCE>(L, blockIdx.x, gridDim.x);
}

// ---------------------------------------------------------------------------
// Boundary nodes (Sec. 2.3.2), 128 to a block: a thread per node pulls its
// populations and forms its moments, a thread per link of the block's nodes the
// bounce-back population, a thread per node collides and stores into f+(t+1).
//
// A link (x_f, d) joins the node x_f to a solid node x_f + e_d of particle p at
// wall fraction q.  The population that would have streamed from the solid
// neighbour into x_f along j = opp(d) is the paper's interpolated bounce-back
// (Eqs. eqneq1, eqneq2, neqd):
//   G_j = f_eq,d(rho_f, u_d) + [f+_d(x_f) - f_eq,d(rho_f, u_f)] + 6 w_d rho0 (e_j . u_w)
//   u_d = u*/3 + 2 u**/3 (piecewise in q), u_w = v_p + omega_p x (x_w - X_p)
// (or the halfway rule f+_d + 6 w_d rho0 e_j.u_w in Ladd mode).  The Galilean-
// invariant momentum exchange of the link,
//   dP = (e_d - u_w) f+_d - (e_j - u_w) G_j = e_d (2 w_d + h_d + h_G) - u_w (h_d - h_G),
// and its torque about X_p are rounded to 2^-40 fixed point per link and
// summed in integers (over the warp, then by 64-bit atomics of whole warps): the
// sums do not depend on the order in which links are visited.
//
// Bound by the gathers: a link reads the 19 populations of the node behind its
// own, a 32-byte sector each.  One kernel per link (38 gathers: its own node's
// too) that kept G for a second kernel per node took 497 + 320 us for 0.82 M
// nodes and 3.35 M links in FP32 (300 particles, 512^3) and 27 + 22 us for
// three cobbles' 32 k nodes; together they take 467 us (408 in 16 bits) and 27
// us (569 and 474 before the list came nearly in particle order).  (A thread per node that goes through its links in turn, with atomics of
// its own where the particle changes, took 1200 us.)  The nodes around
// uncovered ones (k_near) are recomputed by the same launch.
//
// A link is used only when every link of its node fitted into the link list
// (an overflow, reported by the classification, leaves the node on halfway
// bounce-back without momentum exchange until the lists grow).
// ---------------------------------------------------------------------------
namespace {
constexpr unsigned FULLW = 0xffffffffu;

// Exact warp sum of 64-bit fixed-point values (|v| < 2^62): three 22-bit
// pieces, each summed by one integer warp reduction (at most 32 x 2^22 < 2^27,
// no overflow), recombined; the result is in every lane.
__device__ __forceinline__ long long warp_sum_fixed(long long v) {
  const unsigned c0 = (unsigned)(v & 0x3FFFFFLL);
  const unsigned c1 = (unsigned)((v >> 22) & 0x3FFFFFLL);
  const int c2 = (int)(v >> 44);
  const unsigned s0 = __reduce_add_sync(FULLW, c0);
  const unsigned s1 = __reduce_add_sync(FULLW, c1);
  const int s2 = __reduce_add_sync(FULLW, c2);
  return (long long)s0 + ((long long)s1 << 22) + ((long long)s2 << 44);
}

// v * 2^40 rounded to the nearest integer, ties to even: the same value as
// __float2ll_rn(v * 2^40) without a 64-bit conversion.  f = v 2^40 is exact;
// f = h 2^20 + r with h = rint(f 2^-20) (an integer-valued float) and the
// remainder r, |r| <= 2^19, exact in FP32; h 2^20 is an even integer, so the
// nearest-even integer to f is h 2^20 plus the nearest-even integer to r,
// which adding and removing 1.5 2^23 gives (|r| < 2^22).  |v| < 2^10.
__device__ __forceinline__ long long fixed_2m40(float v) {
  const float f = v * 1099511627776.0f;
  const float h = rintf(f * (1.0f / 1048576.0f));
  const float r = f - h * 1048576.0f;
  const int ir = __float_as_int(r + 12582912.0f) - 0x4B400000;
  return ((long long)__float2int_rn(h) << 20) + (long long)ir;
}

// The link entries of node bi fit into the list (its links were written by
// the classification of this step).
__device__ __forceinline__ bool links_fit(uint32_t loff, uint32_t mask, unsigned cap_links) {
  return (unsigned long long)loff + (unsigned)__popc(mask) <= (unsigned long long)cap_links;
}

__device__ __forceinline__ void add_force(long long* facc, int p, int k, long long v) {
  atomicAdd(reinterpret_cast<unsigned long long*>(facc + 6 * (size_t)p + k), (unsigned long long)v);
}
constexpr int BOUNDARY_THREADS = 128;
}  // namespace

template <int ST, bool FORCE, bool LADD>
__global__ void __launch_bounds__(BOUNDARY_THREADS) k_boundary(BoundaryLaunch L) {
  constexpr int N = BOUNDARY_THREADS;  // nodes of a block at a time
  __shared__ float s_g[18][N];         // the links' G by direction and node
  __shared__ float4 s_mom[N];          // rho_f, u_f
  __shared__ int3 s_xyz[N];
  __shared__ uint32_t s_mask[N], s_loff[N], s_cell[N];
  __shared__ int s_incl[N];            // links of the nodes up to this one
  __shared__ int s_warp[N / 32];
  using T = typename Store<ST>::T;
  const T* __restrict__ A = static_cast<const T*>(L.A);
  T* __restrict__ B = static_cast<T*>(L.B);
  const LatticeGeom& g = L.pl.g;
  const ParticleLaunch& pl = L.pl;
  const unsigned nbc = min(pl.ctr->n_bc, pl.cap_bc);
  const int t = (int)threadIdx.x, lane = t & 31, w = t >> 5;
  const float rho0 = L.p.rho0;
  // the last near_blocks blocks take the nodes around uncovered ones
  const unsigned blocks = gridDim.x - (unsigned)L.near_blocks;
  if (blockIdx.x >= blocks) {
    near_nodes<ST, FORCE>(L, blockIdx.x - blocks, (unsigned)L.near_blocks);
    return;
  }
  int pacc = -1;  // the particle of the warp's running fixed-point sums, component k in lane k
  long long acc = 0;
  for (unsigned first = blockIdx.x * N; first < nbc; first += blocks * N) {
    // ---- a thread per node: its pull and its moments ----
    const unsigned bi = first + (unsigned)t;
    const bool node = bi < nbc;
    long long c = 0;
    uint32_t mask = 0;
    int m = 0;
    float h[19];
    if (node) {
      c = pl.bc_cell[bi];
      mask = pl.bc_mask[bi];
      const uint32_t loff = pl.bc_loff[bi];
      m = links_fit(loff, mask, pl.cap_links) ? __popc(mask) : 0;
      int x, y, z;
      coords(c, g, x, y, z);
      pull_node<ST>(A, g, L.p, x, y, z, c, h, mask);
      if (!LADD) {
        float own[19], j[3];
#pragma unroll
        for (int i = 0; i < 19; ++i) own[i] = Store<ST>::dev(A + i * g.plane + c, i);
        float dr = 0.f;
#pragma unroll
        for (int i = 0; i < 19; ++i) dr += own[i];
        momentum<true>(own, j);
        const float rho = 1.0f + dr, irho = inverse(rho);
        s_mom[t] = make_float4(rho, j[0] * irho, j[1] * irho, j[2] * irho);
      }
      s_xyz[t] = make_int3(x, y, z);
      s_mask[t] = mask;
      s_loff[t] = loff;
      s_cell[t] = (uint32_t)c;
    }
    int incl = m;
#pragma unroll
    for (int k = 1; k < 32; k <<= 1) {
      const int v = __shfl_up_sync(FULLW, incl, k);
      if (lane >= k) incl += v;
    }
    if (lane == 31) s_warp[w] = incl;
    __syncthreads();
    int total = 0;
#pragma unroll
    for (int k = 0; k < N / 32; ++k) {
      if (k < w) incl += s_warp[k];
      total += s_warp[k];
    }
    s_incl[t] = incl;
    __syncthreads();
    // ---- a thread per link of the block's nodes ----
    for (int base = 32 * w; base < total; base += N) {
      const int i = base + lane;
      int p = -1;
      float v[6];
      if (i < total) {
        int s = 0;  // its node: the first with more than i links up to it
#pragma unroll
        for (int k = N / 2; k > 0; k >>= 1)
          if (s_incl[s + k - 1] <= i) s += k;
        const uint32_t ms = s_mask[s];
        const unsigned l = s_loff[s] + (unsigned)(i - (s_incl[s] - __popc(ms)));
        const long long cs = s_cell[s];
        const int3 at = s_xyz[s];
        const int d = pl.link_dir[l];
        p = (int)pl.link_p[l];
        const float q = LADD ? 0.5f : pl.link_q[l];
        const int ed[3] = {lex(d), ley(d), lez(d)};
        const float wd = lw(d);
        const float hopp = Store<ST>::dev_at(A + d * g.plane + cs, wd);  // f+_d(x_f) - w_d
        // u at the second fluid node x_f - e_d when it is fluid, else u_f
        float rho_f = 1.0f, uf[3] = {0.f, 0.f, 0.f}, uff[3] = {0.f, 0.f, 0.f};
        if (!LADD) {
          const float4 mom = s_mom[s];
          rho_f = mom.x;
          uff[0] = uf[0] = mom.y;
          uff[1] = uf[1] = mom.z;
          uff[2] = uf[2] = mom.w;
          long long ff;
          if (!((ms >> lopp(d)) & 1u) && nbr_wrap(at.x, at.y, at.z, -ed[0], -ed[1], -ed[2], g, ff)) {
            float rr;
            moments_at<ST>(A, g.plane, ff, rr, uff);
          }
        }
        // wall point relative to the particle position: x - X = (x - floor X) - frac X,
        // the integer part exact and the fraction rounded once to FP32
        const DevParticle& P = pl.P[p];
        const float r0 = ((float)(at.x - P.pos_i[0]) - P.pos_fr[0]) + q * ed[0];
        const float r1 = ((float)(at.y - P.pos_i[1]) - P.pos_fr[1]) + q * ed[1];
        const float r2 = ((float)(at.z - P.pos_i[2]) - P.pos_fr[2]) + q * ed[2];
        float uw[3];
        uw[0] = P.velf[0] + (P.omegaf[1] * r2 - P.omegaf[2] * r1);
        uw[1] = P.velf[1] + (P.omegaf[2] * r0 - P.omegaf[0] * r2);
        uw[2] = P.velf[2] + (P.omegaf[0] * r1 - P.omegaf[1] * r0);
        const float wall = 6.0f * wd * rho0 * (-ed[0] * uw[0] - ed[1] * uw[1] - ed[2] * uw[2]);
        float G;
        if (LADD) {
          G = hopp + wall;
        } else {
          float ud[3];
          const float i1q = 1.0f / (1.0f + q), iq = 1.0f / q;
          const float a1 = (1.0f - q) * i1q, a2 = 2.0f * q * i1q;
          const float b1 = (1.0f - q) * iq, b2 = (2.0f * q - 1.0f) * iq;
#pragma unroll
          for (int a = 0; a < 3; ++a) {
            const float us = q <= 0.5f ? 2.0f * q * uf[a] + (1.0f - 2.0f * q) * uff[a] : b1 * uf[a] + b2 * uw[a];
            ud[a] = us / 3.0f + 2.0f * (a1 * uff[a] + a2 * uw[a]) / 3.0f;
          }
          const float eud = ed[0] * ud[0] + ed[1] * ud[1] + ed[2] * ud[2];
          const float euf = ed[0] * uf[0] + ed[1] * uf[1] + ed[2] * uf[2];
          const float ud2 = ud[0] * ud[0] + ud[1] * ud[1] + ud[2] * ud[2];
          const float uf2 = uf[0] * uf[0] + uf[1] * uf[1] + uf[2] * uf[2];
          G = hopp + wd * rho_f * (3.0f * (eud - euf) + 4.5f * (eud * eud - euf * euf) - 1.5f * (ud2 - uf2)) + wall;
        }
        s_g[d - 1][s] = G;
        // momentum exchange, rounded per link (v * 2^40 is exact in FP32 and the
        // rounding is to nearest even: odd-symmetric, so opposite links of a
        // closed body cancel exactly)
        const float s2 = 2.0f * wd + hopp + G, dl = hopp - G;
        v[0] = ed[0] * s2 - uw[0] * dl;
        v[1] = ed[1] * s2 - uw[1] * dl;
        v[2] = ed[2] * s2 - uw[2] * dl;
        v[3] = r1 * v[2] - r2 * v[1];
        v[4] = r2 * v[0] - r0 * v[2];
        v[5] = r0 * v[1] - r1 * v[0];
      }
      // the links' sums over the warp, particle by particle (nearly always one)
      for (unsigned left = __ballot_sync(FULLW, p >= 0); left;) {
        const int ps = __shfl_sync(FULLW, p, __ffs(left) - 1);
        const bool mine = p == ps;
        left &= ~__ballot_sync(FULLW, mine);
        if (ps != pacc) {
          if (lane < 6 && pacc >= 0) add_force(pl.facc, pacc, lane, acc);
          pacc = ps;
          acc = 0;
        }
#pragma unroll
        for (int k = 0; k < 6; ++k) {
          const long long sum = warp_sum_fixed(mine ? fixed_2m40(v[k]) : 0);
          if (lane == k) acc += sum;
        }
      }
    }
    __syncthreads();
    // ---- a thread per node: collision and store ----
    if (node) {
      if (m)
#pragma unroll
        for (int j = 1; j < 19; ++j)
          if ((mask >> opp(j)) & 1u) h[j] = s_g[opp(j) - 1][t];
      collide<ST, FORCE, true>(h, L.p);
#pragma unroll
      for (int j = 0; j < 19; ++j) {
        if (L.tmp) Store<ST>::put(static_cast<T*>(L.tmp) + 19 * (size_t)bi + j, j, h[j]);
        else Store<ST>::put(B + j * g.plane + c, j, h[j]);
      }
    }
    __syncthreads();  // the shared arrays are free for the next nodes
  }
  if (lane < 6 && pacc >= 0) add_force(pl.facc, pacc, lane, acc);
}

// A list kernel's grid: the tuned block count, but no more blocks than the
// list's capacity (`items` work units at `threads` per block) can use, so
// that small lists do not dispatch thousands of empty blocks.
static inline int list_grid(int tuned, unsigned long long items, int threads) {
  const unsigned long long need = (items + (unsigned long long)threads - 1) / (unsigned long long)threads;
  return (int)(need < 1 ? 1 : (need < (unsigned long long)tuned ? need : (unsigned long long)tuned));
}

template <int ST>
static cudaError_t launch_refill_st(const BoundaryLaunch& L, cudaStream_t s) {
  // a warp per node; a step uncovers a small part of what the list can hold
  k_refill<ST><<<list_grid(L.grid, (L.pl.cap_new + 15ull) / 16ull, 4), 128, 0, s>>>(L);
  return cudaGetLastError();
}

cudaError_t launch_refill(const BoundaryLaunch& L, cudaStream_t s) {
  if (L.pl.np == 0) return cudaSuccess;
  switch (L.storage) {
    case MI_STORE_F32: return launch_refill_st<MI_STORE_F32>(L, s);
    case MI_STORE_F16_DEV: return launch_refill_st<MI_STORE_F16_DEV>(L, s);
    case MI_STORE_BF16_DEV: return launch_refill_st<MI_STORE_BF16_DEV>(L, s);
  }
  return cudaErrorInvalidValue;
}

// blocks of the nodes around uncovered ones: a step uncovers a small part of
// what the list can hold
static int near_grid(const BoundaryLaunch& L) {
  return list_grid(L.grid, 19ull * ((L.pl.cap_new + 15ull) / 16ull), BOUNDARY_THREADS);
}

template <int ST>
static cudaError_t launch_near_st(const BoundaryLaunch& L, cudaStream_t s) {
  const int grid = near_grid(L);
  if (L.forcing) k_near<ST, true><<<grid, 128, 0, s>>>(L);
  else k_near<ST, false><<<grid, 128, 0, s>>>(L);
  return cudaGetLastError();
}

cudaError_t launch_near(const BoundaryLaunch& L, cudaStream_t s) {
  if (L.pl.np == 0) return cudaSuccess;
  switch (L.storage) {
    case MI_STORE_F32: return launch_near_st<MI_STORE_F32>(L, s);
    case MI_STORE_F16_DEV: return launch_near_st<MI_STORE_F16_DEV>(L, s);
    case MI_STORE_BF16_DEV: return launch_near_st<MI_STORE_BF16_DEV>(L, s);
  }
  return cudaErrorInvalidValue;
}

template <int ST, bool FORCE>
static cudaError_t launch_boundary_st(const BoundaryLaunch& L, cudaStream_t s) {
  BoundaryLaunch M = L;
  M.near_blocks = L.near ? near_grid(L) : 0;
  const int grid = list_grid(L.grid, L.pl.cap_bc, BOUNDARY_THREADS) + M.near_blocks;
  if (L.bb_mode == MI_BB_LADD) k_boundary<ST, FORCE, true><<<grid, BOUNDARY_THREADS, 0, s>>>(M);
  else k_boundary<ST, FORCE, false><<<grid, BOUNDARY_THREADS, 0, s>>>(M);
  return cudaGetLastError();
}

template <typename T>
__global__ void __launch_bounds__(256) k_scatter_boundary(BoundaryLaunch L) {
  const unsigned nbc = min(L.pl.ctr->n_bc, L.pl.cap_bc);
  const T* __restrict__ tmp = static_cast<const T*>(L.tmp);
  T* __restrict__ B = static_cast<T*>(L.B);
  for (unsigned e = blockIdx.x * blockDim.x + threadIdx.x; e < 19u * nbc; e += gridDim.x * blockDim.x) {
    const unsigned k = e / 19u, j = e - 19u * k;
    B[j * L.pl.g.plane + L.pl.bc_cell[k]] = tmp[e];
  }
}

cudaError_t launch_scatter_boundary(const BoundaryLaunch& L, cudaStream_t s) {
  if (L.pl.np == 0 || !L.tmp) return cudaSuccess;
  const int grid = list_grid(L.grid, 19ull * L.pl.cap_bc, 256);
  if (L.storage == MI_STORE_F32) k_scatter_boundary<float><<<grid, 256, 0, s>>>(L);
  else k_scatter_boundary<unsigned short><<<grid, 256, 0, s>>>(L);
  return cudaGetLastError();
}

cudaError_t launch_boundary(const BoundaryLaunch& L, cudaStream_t s) {
  if (L.pl.np == 0) return cudaSuccess;
  switch (L.storage) {
    case MI_STORE_F32: return L.forcing ? launch_boundary_st<MI_STORE_F32, true>(L, s) : launch_boundary_st<MI_STORE_F32, false>(L, s);
    case MI_STORE_F16_DEV: return L.forcing ? launch_boundary_st<MI_STORE_F16_DEV, true>(L, s) : launch_boundary_st<MI_STORE_F16_DEV, false>(L, s);
    case MI_STORE_BF16_DEV: return L.forcing ? launch_boundary_st<MI_STORE_BF16_DEV, true>(L, s) : launch_boundary_st<MI_STORE_BF16_DEV, false>(L, s);
  }
  return cudaErrorInvalidValue;
}

// ---------------------------------------------------------------------------
// Fill / pack / unpack (set-up and inspection, not on the step path).
// ---------------------------------------------------------------------------
template <int ST>
__global__ void k_fill_rest(typename Store<ST>::T* pop, long long ncell, long long plane, float rho0) {
  const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= ncell) return;
#pragma unroll
  for (int i = 0; i < 19; ++i) Store<ST>::put(pop + i * plane + n, i, wq(i) * (rho0 - 1.0f));
}

template <int ST>
__global__ void k_pack(const float* __restrict__ src, typename Store<ST>::T* pop, long long ncell, long long plane) {
  const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= ncell) return;
#pragma unroll
  for (int i = 0; i < 19; ++i) Store<ST>::put(pop + i * plane + n, i, src[i * ncell + n] - wq(i));
}

// F32 storage keeps f itself: copy the bits so that a set/get round trip is exact.
__global__ void k_pack_f32(const float* __restrict__ src, float* pop, long long ncell, long long plane) {
  const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= ncell) return;
#pragma unroll
  for (int i = 0; i < 19; ++i) pop[i * plane + n] = src[i * ncell + n];
}
__global__ void k_unpack_f32(const float* pop, float* __restrict__ dst, long long ncell, long long plane) {
  const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= ncell) return;
#pragma unroll
  for (int i = 0; i < 19; ++i) dst[i * ncell + n] = pop[i * plane + n];
}

template <int ST>
__global__ void k_unpack(const typename Store<ST>::T* pop, float* __restrict__ dst, long long ncell, long long plane) {
  const long long n = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= ncell) return;
#pragma unroll
  for (int i = 0; i < 19; ++i) dst[i * ncell + n] = Store<ST>::dev(pop + i * plane + n, i) + wq(i);
}

static inline long long ncell_of(const LatticeGeom& g) { return (long long)g.nx * g.ny * g.nz; }

// Non-finite stored populations (NaN or infinite) at nodes that are not solid
// (owner NULL: every node): out[0] += their count, out[1] = the smallest
// such node index.  For 16-bit storages the test is on the bits (an all-ones
// exponent).
__device__ __forceinline__ bool bad_value(float v) { return !isfinite(v); }
__device__ __forceinline__ bool bad_value(__half v) { return (__half_as_ushort(v) & 0x7C00u) == 0x7C00u; }
__device__ __forceinline__ bool bad_value(__nv_bfloat16 v) { return (__bfloat16_as_ushort(v) & 0x7F80u) == 0x7F80u; }

template <int ST>
__global__ void __launch_bounds__(256) k_check(const typename Store<ST>::T* __restrict__ pop, long long ncell,
                                               long long plane, const uint32_t* __restrict__ owner,
                                               long long* __restrict__ out) {
  long long nbad = 0, first = LLONG_MAX;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < ncell; c += (long long)gridDim.x * blockDim.x) {
    if (owner && owner[c] != OWNER_NONE) continue;
    int k = 0;
#pragma unroll
    for (int i = 0; i < 19; ++i) k += bad_value(pop[i * plane + c]) ? 1 : 0;
    if (k) {
      nbad += k;
      first = c < first ? c : first;
    }
  }
  if (nbad) {
    atomicAdd(reinterpret_cast<unsigned long long*>(out), (unsigned long long)nbad);
    atomicMin(out + 1, first);
  }
}

cudaError_t launch_check(const void* pop, const LatticeGeom& g, int storage, const uint32_t* owner, long long* out,
                         int sm_count, cudaStream_t s) {
  const long long init[2] = {0, LLONG_MAX};
  cudaError_t e = cudaMemcpyAsync(out, init, sizeof(init), cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return e;
  const long long ncell = (long long)g.nx * g.ny * g.nz;
  const int grid = sm_count * 8;
  if (storage == MI_STORE_F16_DEV)
    k_check<MI_STORE_F16_DEV><<<grid, 256, 0, s>>>(static_cast<const __half*>(pop), ncell, g.plane, owner, out);
  else if (storage == MI_STORE_BF16_DEV)
    k_check<MI_STORE_BF16_DEV><<<grid, 256, 0, s>>>(static_cast<const __nv_bfloat16*>(pop), ncell, g.plane, owner, out);
  else
    k_check<MI_STORE_F32><<<grid, 256, 0, s>>>(static_cast<const float*>(pop), ncell, g.plane, owner, out);
  return cudaGetLastError();
}

cudaError_t launch_fill_rest(void* pop, const LatticeGeom& g, int storage, float rho0, cudaStream_t s) {
  const long long n = ncell_of(g);
  const unsigned blocks = (unsigned)((n + 255) / 256);
  switch (storage) {
    case MI_STORE_F32: k_fill_rest<MI_STORE_F32><<<blocks, 256, 0, s>>>((float*)pop, n, g.plane, rho0); break;
    case MI_STORE_F16_DEV: k_fill_rest<MI_STORE_F16_DEV><<<blocks, 256, 0, s>>>((__half*)pop, n, g.plane, rho0); break;
    case MI_STORE_BF16_DEV: k_fill_rest<MI_STORE_BF16_DEV><<<blocks, 256, 0, s>>>((__nv_bfloat16*)pop, n, g.plane, rho0); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_pack(const float* src, void* pop, const LatticeGeom& g, int storage, cudaStream_t s) {
  const long long n = ncell_of(g);
  const unsigned blocks = (unsigned)((n + 255) / 256);
  switch (storage) {
    case MI_STORE_F32: k_pack_f32<<<blocks, 256, 0, s>>>(src, (float*)pop, n, g.plane); break;
    case MI_STORE_F16_DEV: k_pack<MI_STORE_F16_DEV><<<blocks, 256, 0, s>>>(src, (__half*)pop, n, g.plane); break;
    case MI_STORE_BF16_DEV: k_pack<MI_STORE_BF16_DEV><<<blocks, 256, 0, s>>>(src, (__nv_bfloat16*)pop, n, g.plane); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_unpack(const void* pop, float* dst, const LatticeGeom& g, int storage, cudaStream_t s) {
  const long long n = ncell_of(g);
  const unsigned blocks = (unsigned)((n + 255) / 256);
  switch (storage) {
    case MI_STORE_F32: k_unpack_f32<<<blocks, 256, 0, s>>>((const float*)pop, dst, n, g.plane); break;
    case MI_STORE_F16_DEV: k_unpack<MI_STORE_F16_DEV><<<blocks, 256, 0, s>>>((const __half*)pop, dst, n, g.plane); break;
    case MI_STORE_BF16_DEV: k_unpack<MI_STORE_BF16_DEV><<<blocks, 256, 0, s>>>((const __nv_bfloat16*)pop, dst, n, g.plane); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace mi
