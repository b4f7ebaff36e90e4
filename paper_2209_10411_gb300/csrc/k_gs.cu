// Gradient Search refinement of metaball models on point hulls (Sec. 2.2,
// Algorithm 2, Eq. GSloss), one fit at a time per CTA, the fits taken
// largest first by persistent CTAs.  The fit's hull points, model
// and gradients stay in shared memory for all epochs; an epoch is two passes:
// threads over pairs of hull points evaluate the field and dl/df (kept beside the
// points), then units of GS_BALLS control points and a chunk of the points are
// spread over the warps, each summing its gradient components with a fixed
// lane order, and one thread per control point adds its chunks in order.
// Everything is FP32; the reductions have a fixed order, so a fit's result
// does not depend on the other fits of the call.
//
// Bound by the FP32 and special-function (reciprocal) pipes.  Two points share
// every instruction (packed pairs), and a point read from shared memory serves
// GS_BALLS control points (one read per control point kept the shared memory busy
// for longer than the arithmetic took): 300 fits of 8-64 control points on 2048 points, 2 x 100
// epochs, in 4.7 ms; unpacked with a warp per control point 7.1 ms (four control
// points a unit spill at 1024 threads: 5.3 ms, at 512: 4.6 ms, both against 4.6
// with 1 / r^4 formed by itself).
#include <cmath>

#include "mi_gs.h"
#include "mi_internal.cuh"

namespace mi {
namespace {

constexpr int GS_THREADS = 512;  // one CTA per SM
constexpr int GS_CHUNKS = 8;  // most hull-point chunks per control point in the gradient pass
constexpr int GS_BALLS = 2;   // control points of a gradient unit
constexpr unsigned GS_FULL = 0xffffffffu;

// dl/df of Eq. GSloss: 2 (f - 1) on [2, inf), +1 on [1, 2), 2 (f - 1) - 1/f^2 below
__device__ __forceinline__ float gs_dl(float f) {
  return f >= 2.0f ? 2.0f * (f - 1.0f) : (f >= 1.0f ? 1.0f : 2.0f * (f - 1.0f) - 1.0f / (f * f));
}

// l(f) of Eq. GSloss
__device__ __forceinline__ float gs_l(float f) {
  return f >= 2.0f ? (f - 1.0f) * (f - 1.0f) : (f >= 1.0f ? f - 1.0f : (f - 1.0f) * (f - 1.0f) + 1.0f / f - 1.0f);
}

// f at (x, y, z): sum over the model's balls in order
__device__ __forceinline__ float gs_field(const float4* M, int n, float x, float y, float z) {
  float f = 0.f;
  for (int j = 0; j < n; ++j) {
    const float4 b = M[j];
    const float dx = x - b.x, dy = y - b.y, dz = z - b.z;
    f += b.w * __fdividef(1.0f, dx * dx + dy * dy + dz * dz);
  }
  return f;
}

// Sum of one value per thread in a fixed tree order; the result in every thread.
__device__ __forceinline__ float gs_block_sum(float v, float* red) {
  const int t = threadIdx.x;
  red[t] = v;
  __syncthreads();
  for (int s = GS_THREADS / 2; s > 0; s >>= 1) {
    if (t < s) red[t] += red[t + s];
    __syncthreads();
  }
  const float r = red[0];
  __syncthreads();
  return r;
}

struct GsLaunch {
  const int* hull_off;
  const float* hull;
  const int* ball_off;
  float* balls;
  const int* plane_off;
  const float* planes;
  int max_points, max_balls, epochs;
  float lr;
  int* active;
  float* loss;
};

// Chunks of the hull points in the gradient pass: the count (1 .. GS_CHUNKS)
// whose units take the warps the fewest turns, by instructions: about 34 per turn
// of a pair and lane for GS_BALLS control points, 60 per unit (its balls, the
// reduction).
__device__ __forceinline__ int gs_chunks(int n, int pairs) {
  const int groups = (n + GS_BALLS - 1) / GS_BALLS, warps = GS_THREADS / 32;
  int best = 1, cost = 0x7fffffff;
  for (int c = 1; c <= GS_CHUNKS; ++c) {
    const int turns = ((pairs + c - 1) / c + 31) / 32, rounds = (groups * c + warps - 1) / warps;
    const int t = rounds * (34 * turns + 60);
    if (t < cost) {
      cost = t;
      best = c;
    }
  }
  return best;
}

// Sums of 8 values per lane over the warp: lane l gets the sum of value l / 4
// (a transposed butterfly: half of the values change lanes in each step).
__device__ __forceinline__ float gs_sum8(float (&v)[8], int lane) {
#pragma unroll
  for (int o = 16, half = 4; half >= 1; o >>= 1, half >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < half; ++i) {
      const float send = up ? v[i] : v[i + half], keep = up ? v[i + half] : v[i];
      v[i] = keep + __shfl_xor_sync(GS_FULL, send, o);
    }
  }
  v[0] += __shfl_xor_sync(GS_FULL, v[0], 2);
  return v[0] + __shfl_xor_sync(GS_FULL, v[0], 1);
}

// One fit by the whole CTA (every thread calls it with the same fit).
__device__ __forceinline__ void gs_fit_one(const GsLaunch& G, int fit, float4* gsm, float* red) {
  // hull points by pairs: (x0 x1 y0 y1) and (z0 z1 w0 w1), w = dl/df of the last
  // field pass; the model (x, y, z, k), and every value twice, (x x y y) and (z z k k)
  const int max_pairs = (G.max_points + 1) / 2;
  float4 *HA = gsm, *HB = HA + max_pairs, *Ms = HB + max_pairs, *MA = Ms + G.max_balls, *MB = MA + G.max_balls + 1;
  float4* Ps = MB + G.max_balls + 1;  // gradient partial sums per (control point, chunk)
  int* act = reinterpret_cast<int*>(Ps + (size_t)(G.max_balls + GS_BALLS) * GS_CHUNKS);
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int h0 = G.hull_off[fit], m = G.hull_off[fit + 1] - h0;
  const int b0 = G.ball_off[fit], n = G.ball_off[fit + 1] - b0;
  const int p0 = G.plane_off[fit], np_ = G.plane_off[fit + 1] - p0;
  if (m <= 0 || n <= 0 || m > G.max_points || n > G.max_balls) {
    if (t == 0) G.loss[2 * fit] = G.loss[2 * fit + 1] = __int_as_float(0x7fc00000);
    return;
  }
  const int pairs = (m + 1) / 2;
  for (int i = t; i < pairs; i += GS_THREADS) {
    const float* a = G.hull + 3 * (size_t)(h0 + 2 * i);
    const float* b = 2 * i + 1 < m ? a + 3 : a;  // an odd last point twice, the copy without weight
    HA[i] = make_float4(a[0], b[0], a[1], b[1]);
    HB[i] = make_float4(a[2], b[2], 0.f, 0.f);
  }
  const auto put_ball = [&](int j, float4 v) {
    Ms[j] = v;
    MA[j] = make_float4(v.x, v.x, v.y, v.y);
    MB[j] = make_float4(v.z, v.z, v.w, v.w);
  };
  for (int j = t; j < n; j += GS_THREADS) {
    const float* b = G.balls + 4 * (b0 + j);
    put_ball(j, make_float4(b[0], b[1], b[2], b[3]));
    act[j] = 1;
  }
  __syncthreads();
  const int chunks = gs_chunks(n, pairs), csz = (pairs + chunks - 1) / chunks, groups = (n + GS_BALLS - 1) / GS_BALLS;
  float loss1 = 0.f;
  for (int round = 0; round < 2; ++round) {
    for (int e = 0; e < G.epochs; ++e) {
      // dl/df at every hull point, a pair per thread at a time
      for (int i = t; i < pairs; i += GS_THREADS) {
        const float4 ha = HA[i], hb = HB[i];
        const F32x2 x = pack(ha.x, ha.y), y = pack(ha.z, ha.w), z = pack(hb.x, hb.y);
        F32x2 f = pack(0.f, 0.f);
#pragma unroll 4
        for (int j = 0; j < n; ++j) {
          const float4 a = MA[j], b = MB[j];
          const F32x2 dx = vsub(x, pack(a.x, a.y)), dy = vsub(y, pack(a.z, a.w)), dz = vsub(z, pack(b.x, b.y));
          f = vfma(pack(b.z, b.w), rcp_start(vfma(dz, dz, vfma(dy, dy, vmul(dx, dx)))), f);
        }
        const float2 fv = unpack(f);
        HB[i].z = gs_dl(fv.x);
        HB[i].w = 2 * i + 1 < m ? gs_dl(fv.y) : 0.f;
      }
      __syncthreads();
      // gradient of every control point: dL/dk = sum w / r^2, dL/dc = sum w 2 k (H - c) / r^4,
      // as partial sums over contiguous chunks of the points
      for (int u = w; u < groups * chunks; u += GS_THREADS / 32) {
        const int gr = u / chunks, ch = u - gr * chunks, j0 = GS_BALLS * gr;
        const int i1 = min(pairs, (ch + 1) * csz);
        F32x2 bx[GS_BALLS], by[GS_BALLS], bz[GS_BALLS], k2[GS_BALLS];
        F32x2 gx[GS_BALLS], gy[GS_BALLS], gz[GS_BALLS], gk[GS_BALLS];
#pragma unroll
        for (int b = 0; b < GS_BALLS; ++b) {
          const int j = min(j0 + b, n - 1);  // past the last one: repeated, not stored
          const float4 a = MA[j], c = MB[j];
          bx[b] = pack(a.x, a.y);
          by[b] = pack(a.z, a.w);
          bz[b] = pack(c.x, c.y);
          k2[b] = vset(2.0f * c.z, bz[b]);
          gx[b] = gy[b] = gz[b] = gk[b] = pack(0.f, 0.f);
        }
        for (int i = ch * csz + lane; i < i1; i += 32) {
          const float4 ha = HA[i], hb = HB[i];
          const F32x2 x = pack(ha.x, ha.y), y = pack(ha.z, ha.w), z = pack(hb.x, hb.y), wt = pack(hb.z, hb.w);
#pragma unroll
          for (int b = 0; b < GS_BALLS; ++b) {
            const F32x2 dx = vsub(x, bx[b]), dy = vsub(y, by[b]), dz = vsub(z, bz[b]);
            const F32x2 inv = rcp_start(vfma(dz, dz, vfma(dy, dy, vmul(dx, dx))));
            // w 2 k / r^4 in this order: 1 / r^4 by itself leaves FP32 for distances
            // below 2e-10 or above 3e9 (2.5 % faster)
            const F32x2 wi = vmul(wt, inv), s = vmul(vmul(wi, k2[b]), inv);
            gk[b] = vadd(gk[b], wi);
            gx[b] = vfma(s, dx, gx[b]);
            gy[b] = vfma(s, dy, gy[b]);
            gz[b] = vfma(s, dz, gz[b]);
          }
        }
        float v[8];
#pragma unroll
        for (int b = 0; b < GS_BALLS; ++b) {
          const float2 a0 = unpack(gx[b]), a1 = unpack(gy[b]), a2 = unpack(gz[b]), a3 = unpack(gk[b]);
          v[4 * b] = a0.x + a0.y;
          v[4 * b + 1] = a1.x + a1.y;
          v[4 * b + 2] = a2.x + a2.y;
          v[4 * b + 3] = a3.x + a3.y;
        }
        const float sum = gs_sum8(v, lane);
        // lane 4 (4 b + component): partial sums by control point, then chunk
        if (!(lane & 3)) reinterpret_cast<float*>(Ps + (size_t)(j0 + (lane >> 4)) * chunks + ch)[(lane >> 2) & 3] = sum;
      }
      __syncthreads();
      for (int j = t; j < n; j += GS_THREADS)
        if (act[j]) {
          float4 g = Ps[j * chunks];
          for (int ch = 1; ch < chunks; ++ch) {
            const float4 q = Ps[j * chunks + ch];
            g.x += q.x;
            g.y += q.y;
            g.z += q.z;
            g.w += q.w;
          }
          float4 b = Ms[j];
          b.x -= G.lr * g.x;
          b.y -= G.lr * g.y;
          b.z -= G.lr * g.z;
          b.w -= G.lr * g.w;
          put_ball(j, b);
        }
      __syncthreads();
    }
    // the loss of the model after this descent
    float part = 0.f;
    for (int i = t; i < m; i += GS_THREADS) {
      const float4 ha = HA[i >> 1], hb = HB[i >> 1];
      part += (i & 1) ? gs_l(gs_field(Ms, n, ha.y, ha.w, hb.y)) : gs_l(gs_field(Ms, n, ha.x, ha.z, hb.x));
    }
    const float L = gs_block_sum(part, red);
    if (round == 0) {
      loss1 = L;
      // anomalies: k < 0, or outside a facet plane (FP32, single roundings, left to
      // right); a warp per control point, its lanes over the planes (one thread
      // per control point waited for some 4000 loads in turn: 0.4 ms a fit)
      for (int j = w; j < n; j += GS_THREADS / 32) {
        const float4 b = Ms[j];
        bool bad = b.w < 0.f;
        for (int p = lane; p < np_; p += 128) {
          float s[4], d[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float* P = G.planes + 4 * (size_t)(p0 + min(p + 32 * k, np_ - 1));
            s[k] = __fadd_rn(__fadd_rn(__fmul_rn(P[0], b.x), __fmul_rn(P[1], b.y)), __fmul_rn(P[2], b.z));
            d[k] = P[3];
          }
          bad = bad || s[0] > d[0] || s[1] > d[1] || s[2] > d[2] || s[3] > d[3];
        }
        bad = __any_sync(GS_FULL, bad);
        if (bad && lane == 0) {
          put_ball(j, make_float4(b.x, b.y, b.z, 0.f));
          act[j] = 0;
        }
      }
      __syncthreads();
    } else if (t == 0) {
      G.loss[2 * fit] = loss1;
      G.loss[2 * fit + 1] = L;
    }
  }
  for (int j = t; j < n; j += GS_THREADS) {
    float* b = G.balls + 4 * (b0 + j);
    const float4 v = Ms[j];
    b[0] = v.x;
    b[1] = v.y;
    b[2] = v.z;
    b[3] = v.w;
    G.active[b0 + j] = act[j];
  }
  __syncthreads();  // the shared buffers are free for the next fit
}

// Fits in decreasing order of work (hull points x control points, ties to the
// lower index): order[r] is the fit of rank r.
__global__ void k_gs_order(GsLaunch G, int n_fits, int* order) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n_fits) return;
  auto work = [&](int f) {
    return (long long)(G.hull_off[f + 1] - G.hull_off[f]) * (long long)(G.ball_off[f + 1] - G.ball_off[f]);
  };
  const long long wj = work(j);
  int r = 0;
  for (int i = 0; i < n_fits; ++i) {
    const long long wi = work(i);
    r += (wi > wj) || (wi == wj && i < j);
  }
  order[r] = j;
}

// Persistent CTAs, one per SM, take the fits largest first from a counter, so
// that the SMs' loads even out (longest-processing-time-first scheduling).
__global__ void __launch_bounds__(GS_THREADS, 1) k_gs_fit(GsLaunch G, int n_fits, const int* order, int* next) {
  extern __shared__ __align__(16) float4 gsm[];
  __shared__ float red[GS_THREADS];
  __shared__ int pick;
  for (;;) {
    if (threadIdx.x == 0) pick = atomicAdd(next, 1);
    __syncthreads();
    const int q = pick;
    __syncthreads();
    if (q >= n_fits) break;
    gs_fit_one(G, order[q], gsm, red);
  }
}

}  // namespace
}  // namespace mi

extern "C" mi_status mi_gs_fit(int n_fits, const int* hull_off, const float* hull, const int* ball_off, float* balls,
                               const int* plane_off, const float* planes, int max_points, int max_balls, int epochs,
                               float lr, int* active, float* loss, void* stream) {
  using namespace mi;
  if (n_fits < 0 || epochs < 0 || !std::isfinite(lr) || max_points < 1 || max_points > MI_GS_MAX_POINTS ||
      max_balls < 1 || max_balls > MI_GS_MAX_BALLS)
    return MI_EINVAL;
  if (n_fits == 0) return MI_OK;
  if (!hull_off || !hull || !ball_off || !balls || !plane_off || !planes || !active || !loss) return MI_EINVAL;
  GsLaunch G;
  G.hull_off = hull_off;
  G.hull = hull;
  G.ball_off = ball_off;
  G.balls = balls;
  G.plane_off = plane_off;
  G.planes = planes;
  G.max_points = max_points;
  G.max_balls = max_balls;
  G.epochs = epochs;
  G.lr = lr;
  G.active = active;
  G.loss = loss;
  // point pairs, the model thrice, the partial sums (whole units), the active flags
  const size_t smem = sizeof(float4) * (2 * (((size_t)max_points + 1) / 2) + 3 * (size_t)max_balls + 2 +
                                        (size_t)GS_CHUNKS * (max_balls + GS_BALLS)) + sizeof(int) * max_balls;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int dev = 0, sms = 0;
  if (cudaFuncSetAttribute(k_gs_fit, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
      cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return MI_ECUDA;
  // the fit order and the pick counter, stream-ordered scratch
  int* tmp = nullptr;
  if (cudaMallocAsync(reinterpret_cast<void**>(&tmp), sizeof(int) * ((size_t)n_fits + 1), s) != cudaSuccess)
    return MI_ECUDA;
  int* order = tmp + 1;
  cudaError_t e = cudaMemsetAsync(tmp, 0, sizeof(int), s);
  if (e == cudaSuccess) {
    k_gs_order<<<(n_fits + 255) / 256, 256, 0, s>>>(G, n_fits, order);
    const int grid = sms > 0 && sms < n_fits ? sms : n_fits;
    k_gs_fit<<<grid, GS_THREADS, smem, s>>>(G, n_fits, order, tmp);
    e = cudaGetLastError();
  }
  const cudaError_t ef = cudaFreeAsync(tmp, s);
  return e == cudaSuccess && ef == cudaSuccess ? MI_OK : MI_ECUDA;
}
