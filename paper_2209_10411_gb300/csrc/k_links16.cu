// Wall fraction of each link for the 16-bit storages: root q in (0, 1] of g(q) =
// f_p(x_f + q e_d) - 1 (Sec. 2.3.2; reading A7: along the link that points into
// the solid, c0 = 1), in the body frame and float-float arithmetic.
//
// Why these storages have a kernel of their own: q differs from that of k_links_q
// (lattice frame, k_particles.cu) by up to 7e-7, which moves a bounce-back population by
// an FP32 ulp or so.  An FP32 storage keeps it that way; a 16-bit one rounds to 2^-11
// or 2^-8, and where such a value lies near the middle of two it moves by a whole
// unit.  Each such unit is 2e-7 of a light particle's velocity (radius 3 lu,
// BF16), so the states after 20 steps would depend on which kernel formed q: 1e-7 apart.
// So 16-bit runs keep the arithmetic that they had: 300 particles, 3.35 M
// links of particles of 8 to 64 balls take 850 us, 494 with k_links_q.
//
// Inputs: the body-frame link origin p and direction e as float pairs hi + lo
// (the prologue forms the particle's frame in FP64 once per step; each link
// combines it in float-float arithmetic, without FP64, which runs at a small
// fraction of the FP32 rate on this part), and the ball table's split copy; origins
// and centres are split on the grid of 2^-12 when the particle's bounding
// radius is below 1000, so that p_hi - c_hi is exact in FP32 (otherwise the
// difference goes through TwoSum).
//
// Stage 1, FP32: Newton steps on h(q) = f^(-1/2) - 1, which has the same root
// and is close to linear along a link for fields of the form k / r^2 (the
// distance to a lone ball over its radius), kept inside a shrinking bracket
// [lo, hi] (bisection when a step leaves it), the field summed as two
// independent partial sums from the hi parts of the centres, until a step is
// below 1e-3.  The FP32 field's noise, divided by g'(q) = e . grad f, leaves
// errors up to ~1e-4.
// Stage 2, double-float: Newton steps whose residual g(q) is evaluated in
// float-float arithmetic (an unevaluated sum hi + lo of two floats, ~44
// significant bits; Knuth's TwoSum and the fused-multiply-add form of
// Dekker's product are exact), the derivative in FP32, inside a bracket that
// starts at [0, 1] (the exact flags guarantee g(0) < 0 <= g(1)) and moves with
// the accurate signs.  A step ends it when it is below 2e-5 or when the error
// Newton's quadratic convergence leaves behind, |g''/2g'| step^2 with g'' in
// FP32 from the same sums, is below 1e-7 (usually the first step); at most
// four steps.  The largest error of q over 2.3 M links is 6.9e-7; a link that grazes
// the surface (both roots within 1e-3 of each other) can need more than four.
#include "mi_internal.cuh"

namespace mi {

namespace {
struct F2 {
  float hi, lo;
};
__device__ __forceinline__ F2 two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bv = __fsub_rn(s, a);
  const float av = __fsub_rn(s, bv);
  return {s, __fadd_rn(__fsub_rn(a, av), __fsub_rn(b, bv))};
}
__device__ __forceinline__ F2 two_prod(float a, float b) {
  const float p = __fmul_rn(a, b);
  return {p, __fmaf_rn(a, b, -p)};
}
__device__ __forceinline__ F2 df_add(F2 a, F2 b) {
  const F2 s = two_sum(a.hi, b.hi);
  return two_sum(s.hi, s.lo + (a.lo + b.lo));
}
// a float pair re-split with hi on the grid of 2^-12 (|hi| < 2^11: exact)
__device__ __forceinline__ F2 to_grid(F2 v) {
  const float h = rintf(v.hi * 4096.0f) * (1.0f / 4096.0f);
  return {h, (v.hi - h) + v.lo};
}
// p_hi - c_hi as hi + lo (exact on the grid)
__device__ __forceinline__ F2 diff_hi(float p, float c, bool grid) {
  return grid ? F2{__fsub_rn(p, c), 0.f} : two_sum(p, -c);
}

// g(q) = f(p + q e) - 1 in float-float; g'(q) and g''(q) in FP32 (ee = e . e).
template <bool GRID>
__device__ __forceinline__ float residual_ff(const float4* __restrict__ bs, int nb, const F2 p[3], const F2 e[3],
                                             float q, float ee, float& gp, float& gpp) {
  float gh = 0.f, gl = 0.f, d1 = 0.f, d2 = 0.f;
  for (int b = 0; b < nb; ++b) {
    const float4 ch = __ldg(bs + 2 * b), cl = __ldg(bs + 2 * b + 1);
    const float c_hi[3] = {ch.x, ch.y, ch.z}, c_lo[3] = {cl.x, cl.y, cl.z};
    float r2h = 0.f, r2l = 0.f, ae = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      // a = (p - c) + q e as ah + al
      const F2 d = diff_hi(p[k].hi, c_hi[k], GRID);
      const float dl = GRID ? p[k].lo - c_lo[k] : d.lo + (p[k].lo - c_lo[k]);
      const F2 m = two_prod(q, e[k].hi);
      const float ml = __fmaf_rn(q, e[k].lo, m.lo);
      const F2 a = two_sum(d.hi, m.hi);
      const float al = a.lo + dl + ml;
      // a^2 = ah^2 + 2 ah al (al^2 is below the working precision)
      const F2 sq = two_prod(a.hi, a.hi);
      const float sql = __fmaf_rn(2.0f * a.hi, al, sq.lo);
      if (k == 0) {
        r2h = sq.hi;
        r2l = sql;
      } else {
        const F2 t = two_sum(r2h, sq.hi);
        r2h = t.hi;
        r2l += t.lo + sql;
      }
      ae = __fmaf_rn(a.hi, e[k].hi, ae);
    }
    const F2 r2 = two_sum(r2h, r2l);
    // k / r^2: a quotient of the hi parts (within 2 ulps), corrected by its
    // residual (formed by FMA, rounded at ~2^-46 of k)
    const float th = __fdividef(ch.w, r2.hi);
    float res = __fmaf_rn(-th, r2.hi, ch.w);
    res = __fmaf_rn(-th, r2.lo, res + cl.w);
    const float tl = __fdividef(res, r2.hi);
    const F2 s = two_sum(gh, th);
    gh = s.hi;
    gl += s.lo + tl;
    // k / r^2 along the link: r^2' = 2 a.e, r^2'' = 2 e.e, so
    // g' = -2 t (a.e) / r^2 and g'' = t / r^2 (8 (a.e)^2 / r^2 - 2 e.e), t = k / r^2
    const float ir2 = __fdividef(1.0f, r2.hi), u = ae * ir2;
    d1 = __fmaf_rn(-2.0f * th, u, d1);
    d2 = __fmaf_rn(th * ir2, __fmaf_rn(8.0f * ae, u, -2.0f * ee), d2);
  }
  gp = d1;
  gpp = d2;
  const F2 g = two_sum(gh, -1.0f);
  return g.hi + (g.lo + gl);
}
// The root q of one link from its body-frame origin ps and direction es
// (float pairs) over the particle's nb split balls bs; GRID: ps and the
// centres share the 2^-12 grid (hi parts subtract exactly).
template <bool GRID>
__device__ __forceinline__ float link_root(const float4* __restrict__ bs, int nb, const F2 ps[3], const F2 es[3]) {
  // stage 1: FP32 Newton on h = f^(-1/2) - 1
  float lo = 0.f, hi = 1.f, q = 0.5f;
  for (int it = 0; it < 24; ++it) {
    float f0 = 0.f, f1 = 0.f, s0 = 0.f, s1 = 0.f;
    // p_lo + q e, then + (p_hi - c_hi) per ball: the centres' lo parts (2^-24
    // of a centre) are left to the accurate stage
    float a[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) a[k] = __fmaf_rn(q, es[k].hi, ps[k].lo);
    int b = 0;
    for (; b + 2 <= nb; b += 2) {
      const float4 ha = __ldg(bs + 2 * b), hb = __ldg(bs + 2 * b + 2);
      const float u0 = diff_hi(ps[0].hi, ha.x, GRID).hi + a[0];
      const float u1 = diff_hi(ps[1].hi, ha.y, GRID).hi + a[1];
      const float u2 = diff_hi(ps[2].hi, ha.z, GRID).hi + a[2];
      const float v0 = diff_hi(ps[0].hi, hb.x, GRID).hi + a[0];
      const float v1 = diff_hi(ps[1].hi, hb.y, GRID).hi + a[1];
      const float v2 = diff_hi(ps[2].hi, hb.z, GRID).hi + a[2];
      const float iu = __fdividef(1.f, u0 * u0 + u1 * u1 + u2 * u2), iv = __fdividef(1.f, v0 * v0 + v1 * v1 + v2 * v2);
      const float tu = ha.w * iu, tv = hb.w * iv;
      f0 += tu;
      f1 += tv;
      // f' = -2 sum k (a . e) / r^4: the factor -2 is applied to the sums
      s0 = __fmaf_rn(tu * iu, u0 * es[0].hi + u1 * es[1].hi + u2 * es[2].hi, s0);
      s1 = __fmaf_rn(tv * iv, v0 * es[0].hi + v1 * es[1].hi + v2 * es[2].hi, s1);
    }
    if (b < nb) {
      const float4 ha = __ldg(bs + 2 * b);
      const float u0 = diff_hi(ps[0].hi, ha.x, GRID).hi + a[0];
      const float u1 = diff_hi(ps[1].hi, ha.y, GRID).hi + a[1];
      const float u2 = diff_hi(ps[2].hi, ha.z, GRID).hi + a[2];
      const float iu = __fdividef(1.f, u0 * u0 + u1 * u1 + u2 * u2);
      const float tu = ha.w * iu;
      f0 += tu;
      s0 = __fmaf_rn(tu * iu, u0 * es[0].hi + u1 * es[1].hi + u2 * es[2].hi, s0);
    }
    const float f = f0 + f1, fp = -2.f * (s0 + s1);
    if (f >= 1.f) hi = q;
    else lo = q;
    // Newton on h: q + 2 f (1 - sqrt f) / f'
    const float step = 2.f * f * (1.f - f * rsqrtf(f)) / fp;
    float qn = q + step;
    // a step below 1e-3 ends the stage (taken, clamped to the bracket): h is
    // close to linear, so the step leaves far less than the FP32 field's
    // noise behind, which the accurate stage removes
    if (fabsf(step) < 1e-3f) {
      q = fminf(fmaxf(qn, lo), hi);
      break;
    }
    if (!(qn > lo && qn < hi)) qn = 0.5f * (lo + hi);
    q = qn;
    if (hi - lo < 1e-6f) break;
  }
  // stage 2: double-float Newton
  lo = 0.f;
  hi = 1.f;
  const float ee = es[0].hi * es[0].hi + es[1].hi * es[1].hi + es[2].hi * es[2].hi;
  for (int it = 0; it < 4; ++it) {
    float gp, gpp;
    const float g = residual_ff<GRID>(bs, nb, ps, es, q, ee, gp, gpp);
    if (g >= 0.f) hi = q;
    else lo = q;
    const float step = g / gp;
    float qn = q - step;
    // the step ends the stage when it is below 2e-5, or when Newton's error
    // after it, |g'' / 2 g'| step^2, is below 1e-7 (and it stays in the bracket)
    if (fabsf(step) < 2e-5f || (qn >= lo && qn <= hi && fabsf(gpp) * step * step <= 2e-7f * fabsf(gp))) {
      q = fminf(fmaxf(qn, lo), hi);
      break;
    }
    if (!(qn > lo && qn < hi)) qn = 0.5f * (lo + hi);
    q = qn;
  }
  return q;
}

}  // namespace

__global__ void __launch_bounds__(256) k_links_q16(ParticleLaunch L) {
  const unsigned nl = min(L.ctr->n_links, L.cap_links);
  const unsigned nbc = min(L.ctr->n_bc, L.cap_bc);
  for (unsigned l = blockIdx.x * blockDim.x + threadIdx.x; l < nl; l += gridDim.x * blockDim.x) {
    const unsigned bi = L.link_bc[l];
    if (bi >= nbc) continue;
    // an entry of this step: inside the range of the node it names, whose
    // links all fitted (entries of a node that overflowed were not written)
    const unsigned loff = L.bc_loff[bi], m = __popc(L.bc_mask[bi]);
    if (l < loff || l - loff >= m || (unsigned long long)loff + m > (unsigned long long)L.cap_links) continue;
    const long long c = L.bc_cell[bi];
    const int d = L.link_dir[l];
    const DevParticle& P = L.P[L.link_p[l]];
    // node indices of particle lists fit in 32 bits (the lists store them as uint32)
    const unsigned cu = (unsigned)c, row = cu / (unsigned)L.g.nx;
    const int x = (int)(cu - row * (unsigned)L.g.nx), z = (int)(row / (unsigned)L.g.ny), y = (int)(row - (unsigned)z * L.g.ny);
    // body-frame link origin p = R^T (x - X) = R^T n - R^T (X - floor X), n = x - floor X
    // an exact small integer vector, in float-float arithmetic from the
    // prologue's float pairs (TwoProduct of R_hi n exact, R_lo n below it)
    const float n[3] = {(float)(x - P.pos_i[0]), (float)(y - P.pos_i[1]), (float)(z - P.pos_i[2])};
    F2 ps[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      F2 acc = {-P.Ts[0][k], -P.Ts[1][k]};
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        F2 t = two_prod(P.Rs[0][3 * a + k], n[a]);
        t.lo = __fmaf_rn(P.Rs[1][3 * a + k], n[a], t.lo);
        acc = df_add(acc, t);
      }
      ps[k] = acc;
    }
    // on the 2^-12 grid (|p|, |c| < 1024, split the same way by the host) the
    // hi parts subtract exactly; larger particles take TwoSum
    const bool grid = P.Rb_f < 1000.f;
    if (grid)
      for (int k = 0; k < 3; ++k) ps[k] = to_grid(ps[k]);
    const F2 es[3] = {{P.Es[d][0], P.Es[d][3]}, {P.Es[d][1], P.Es[d][4]}, {P.Es[d][2], P.Es[d][5]}};
    const float4* bs = L.balls_s + 2 * (size_t)P.ball_off;
    const int nb = P.n_balls;
    const float q = grid ? link_root<true>(bs, nb, ps, es) : link_root<false>(bs, nb, ps, es);
    L.link_q[l] = fminf(fmaxf(q, 1e-6f), 1.0f);
  }
}

cudaError_t launch_links_q16(const ParticleLaunch& L, int grid, cudaStream_t s) {
  k_links_q16<<<grid, 256, 0, s>>>(L);
  return cudaGetLastError();
}

}  // namespace mi
