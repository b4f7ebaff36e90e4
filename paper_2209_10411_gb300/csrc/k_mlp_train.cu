// Training of the learned Newton guess's network (64 -> 256 -> 256 -> 4, ReLU):
// forward, MSE loss, backward and AdamW.  Every matrix product runs on the
// tensor cores as BF16 x BF16 -> FP32 (mma.sync m16n8k16); parameters,
// activations and gradients live in FP32 and are rounded to BF16 when a tile
// is staged in shared memory, so the network computes with BF16 operands and
// FP32 accumulation while the optimizer keeps FP32 master weights.
//
// A training step of a few thousand rows is 2 GFLOP: it is bound by latency and
// launches, not by the tensor cores.  So the whole forward is one kernel, the
// backpropagated deltas one, and the six gradients one.  A batch of 4096 with
// loss and update takes 49 us of GPU time in five launches; one
// generic product kernel per matrix, its inner dimension (the batch, for a
// weight gradient) on a single CTA per 64 x 64 tile, took 2556 us in 15.
#include <cooperative_groups.h>
#include <cstring>
#include <string>

#include "mi_internal.cuh"

namespace cg = cooperative_groups;

namespace mi {
void set_thread_error(const char* msg);  // engine.cu: message for mi_delbm_last_error(NULL)

namespace {

constexpr unsigned TR_FULL = 0xffffffffu;
constexpr int TR_ROWS = 32;                  // batch rows per CTA tile
constexpr int TR_LDH = 256 + 8, TR_LDX = 64 + 8, TR_LD16 = 16 + 8;  // padded row lengths (BF16)

__device__ __forceinline__ void mma_bf16(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldm4(unsigned (&r)[4], const __nv_bfloat16* p) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(s));
}
__device__ __forceinline__ void ldm4t(unsigned (&r)[4], const __nv_bfloat16* p) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(s));
}
// Fragments from shared tiles with row length LD.  A 16 x 16 (rows m, columns
// k) from a tile stored by m; B 16 x 16 (k by n: two 8-wide fragments, r[0],
// r[1] and r[2], r[3]) from a tile stored by n or by k.
template <int LD> __device__ __forceinline__ void frag_a(unsigned (&r)[4], const __nv_bfloat16* t, int m, int k, int lane) {
  ldm4(r, t + (m + ((lane >> 3) & 1) * 8 + (lane & 7)) * LD + k + (lane >> 4) * 8);
}
template <int LD> __device__ __forceinline__ void frag_b(unsigned (&r)[4], const __nv_bfloat16* t, int n, int k, int lane) {
  ldm4(r, t + (n + (lane >> 4) * 8 + (lane & 7)) * LD + k + ((lane >> 3) & 1) * 8);
}
template <int LD> __device__ __forceinline__ void frag_b_by_k(unsigned (&r)[4], const __nv_bfloat16* t, int n, int k, int lane) {
  ldm4t(r, t + (k + ((lane >> 3) & 1) * 8 + (lane & 7)) * LD + n + (lane >> 4) * 8);
}

// four consecutive floats; AL: the address is 16-byte aligned
template <bool AL> __device__ __forceinline__ float4 load4(const float* p) {
  if (AL) return __ldg(reinterpret_cast<const float4*>(p));
  return make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3));
}
template <bool AL> __device__ __forceinline__ void store2(float* p, float a, float b) {
  if (AL) *reinterpret_cast<float2*>(p) = make_float2(a, b);
  else {
    p[0] = a;
    p[1] = b;
  }
}
__device__ __forceinline__ void put4(__nv_bfloat16* p, float4 v) {  // p 8-byte aligned
  const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
  uint2 w;
  w.x = *reinterpret_cast<const unsigned*>(&lo);
  w.y = *reinterpret_cast<const unsigned*>(&hi);
  *reinterpret_cast<uint2*>(p) = w;
}
__device__ __forceinline__ void put2(__nv_bfloat16* p, float a, float b) {
  *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(a, b);
}

// rows x cols floats (row-major, cols a power of two times 4) into a BF16 tile of row length LD
template <bool AL, int ROWS, int COLS, int LD>
__device__ __forceinline__ void stage(__nv_bfloat16* t, const float* src, int tid, int threads) {
#pragma unroll 8
  for (int e = tid; e < ROWS * COLS / 4; e += threads) {
    const int r = e / (COLS / 4), c = 4 * (e % (COLS / 4));
    put4(t + r * LD + c, load4<AL>(src + r * COLS + c));
  }
}
// the same for the rows [r0, r0 + ROWS) of an n-row matrix, zero below
template <bool AL, int ROWS, int COLS, int LD>
__device__ __forceinline__ void stage_rows(__nv_bfloat16* t, const float* src, int r0, int n, int tid, int threads) {
  for (int e = tid; e < ROWS * COLS / 4; e += threads) {
    const int r = e / (COLS / 4), c = 4 * (e % (COLS / 4));
    const float4 v = r0 + r < n ? load4<AL>(src + (size_t)(r0 + r) * COLS + c) : make_float4(0.f, 0.f, 0.f, 0.f);
    put4(t + r * LD + c, v);
  }
}

struct Params {  // views of a parameter (or gradient) block
  float *W1, *b1, *W2, *b2, *W3, *b3;
};
Params views(const float* base) {
  float* p = const_cast<float*>(base);
  Params P;
  P.W1 = p;
  P.b1 = P.W1 + 64 * 256;
  P.W2 = P.b1 + 256;
  P.b2 = P.W2 + 256 * 256;
  P.W3 = P.b2 + 256;
  P.b3 = P.W3 + 256 * 4;
  return P;
}

// ---------------------------------------------------------------------------
// Forward: the weights in shared memory once per CTA (195 KB), 32 rows of the
// batch at a time; eight warps take 32 columns each of the hidden layers, two
// warps the output layer.
// ---------------------------------------------------------------------------
constexpr size_t FW_W1 = 0, FW_W2 = FW_W1 + 64 * TR_LDH, FW_W3 = FW_W2 + 256 * TR_LDH, FW_X = FW_W3 + 256 * 8,
                 FW_H1 = FW_X + TR_ROWS * TR_LDX, FW_H2 = FW_H1 + TR_ROWS * TR_LDH, FW_END = FW_H2 + TR_ROWS * TR_LDH;

// acc[i][j] += the 32 rows of A (by m) times the 32 columns from n0 of B, K deep in steps of 16
template <int K, int LDA, int LDB, bool B_BY_K>
__device__ __forceinline__ void product32(float (&acc)[2][4][4], const __nv_bfloat16* A, const __nv_bfloat16* Bt, int n0,
                                          int lane) {
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[i][j][c] = 0.f;
#pragma unroll 4
  for (int k = 0; k < K; k += 16) {
    unsigned a[2][4], b[2][4];
#pragma unroll
    for (int i = 0; i < 2; ++i) frag_a<LDA>(a[i], A, 16 * i, k, lane);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      if (B_BY_K) frag_b_by_k<LDB>(b[j], Bt, n0 + 16 * j, k, lane);
      else frag_b<LDB>(b[j], Bt, n0 + 16 * j, k, lane);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) mma_bf16(acc[i][j], a[i], b[j >> 1][2 * (j & 1)], b[j >> 1][2 * (j & 1) + 1]);
  }
}

// ReLU(acc + bias) to the FP32 activations and to the next layer's BF16 tile
template <bool AL>
__device__ __forceinline__ void hidden_out(const float (&acc)[2][4][4], const float* __restrict__ bias, float* H,
                                           __nv_bfloat16* t, int r0, int n, int n0, int lane) {
  const int gid = lane >> 2, tig = lane & 3;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int col = n0 + 8 * j + 2 * tig;
    const float b0 = __ldg(bias + col), b1 = __ldg(bias + col + 1);
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int row = 16 * i + gid + 8 * h;
        const float v0 = fmaxf(acc[i][j][2 * h] + b0, 0.f), v1 = fmaxf(acc[i][j][2 * h + 1] + b1, 0.f);
        put2(t + row * TR_LDH + col, v0, v1);
        if (r0 + row < n) store2<AL>(H + (size_t)(r0 + row) * 256 + col, v0, v1);
      }
  }
}

template <bool AL>
__global__ void __launch_bounds__(256, 1) k_mlp_forward(Params P, const float* __restrict__ X, int n, float* Y, float* H1,
                                                        float* H2) {
  extern __shared__ __align__(16) __nv_bfloat16 sm16[];
  __nv_bfloat16 *W1 = sm16 + FW_W1, *W2 = sm16 + FW_W2, *W3 = sm16 + FW_W3, *Xs = sm16 + FW_X, *H1s = sm16 + FW_H1,
                *H2s = sm16 + FW_H2;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n0 = 32 * warp;
  int r0 = blockIdx.x * TR_ROWS;
  stage_rows<AL, TR_ROWS, 64, TR_LDX>(Xs, X, r0, n, tid, 256);
  stage<AL, 64, 256, TR_LDH>(W1, P.W1, tid, 256);
  stage<AL, 256, 256, TR_LDH>(W2, P.W2, tid, 256);
  {
    const float4 w = load4<AL>(P.W3 + 4 * tid);
    put4(W3 + 8 * tid, w);
    put4(W3 + 8 * tid + 4, make_float4(0.f, 0.f, 0.f, 0.f));
  }
  for (;;) {
    __syncthreads();
    float acc[2][4][4];
    product32<64, TR_LDX, TR_LDH, true>(acc, Xs, W1, n0, lane);
    hidden_out<AL>(acc, P.b1, H1, H1s, r0, n, n0, lane);
    __syncthreads();
    product32<256, TR_LDH, TR_LDH, true>(acc, H1s, W2, n0, lane);
    hidden_out<AL>(acc, P.b2, H2, H2s, r0, n, n0, lane);
    // the next tile's rows: no warp reads Xs after the barrier above
    const int next = r0 + (int)gridDim.x * TR_ROWS;
    if (next < n) stage_rows<AL, TR_ROWS, 64, TR_LDX>(Xs, X, next, n, tid, 256);
    __syncthreads();
    if (warp < 2) {
      float y[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
      for (int k = 0; k < 256; k += 16) {
        unsigned a[4], b0, b1;
        frag_a<TR_LDH>(a, H2s, 16 * warp, k, lane);
        const unsigned s = (unsigned)__cvta_generic_to_shared(W3 + (k + (lane & 15)) * 8);
        asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];\n" : "=r"(b0), "=r"(b1) : "r"(s));
        mma_bf16(y, a, b0, b1);
      }
      const int gid = lane >> 2, tig = lane & 3;
      if (tig < 2)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int row = r0 + 16 * warp + gid + (c >= 2 ? 8 : 0), col = 2 * tig + (c & 1);
          if (row < n) Y[(size_t)row * 4 + col] = y[c] + __ldg(P.b3 + col);
        }
    }
    if (next >= n) break;
    r0 = next;
  }
}

// ---------------------------------------------------------------------------
// Deltas: dZ2 = (dY W3^T) where H2 > 0, dZ1 = (dZ2 W2^T) where H1 > 0 (relu(z)
// > 0 exactly where z > 0, so the saved activations give the masks); W2 in
// shared memory as it lies (by its input index, the product's column).
// ---------------------------------------------------------------------------
constexpr size_t DZ_W2 = 0, DZ_W3 = DZ_W2 + 256 * TR_LDH, DZ_Y = DZ_W3 + 256 * TR_LD16, DZ_Z2 = DZ_Y + TR_ROWS * TR_LD16,
                 DZ_END = DZ_Z2 + TR_ROWS * TR_LDH;

template <bool AL>
__device__ __forceinline__ void masked_out(const float (&acc)[2][4][4], const float* H, float* dZ, __nv_bfloat16* t, int r0,
                                           int n, int n0, int lane) {
  const int gid = lane >> 2, tig = lane & 3;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int row = 16 * i + gid + 8 * h;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int col = n0 + 8 * j + 2 * tig;
        float v0 = 0.f, v1 = 0.f;
        if (r0 + row < n) {
          const size_t at = (size_t)(r0 + row) * 256 + col;
          if (H[at] > 0.f) v0 = acc[i][j][2 * h];
          if (H[at + 1] > 0.f) v1 = acc[i][j][2 * h + 1];
          store2<AL>(dZ + at, v0, v1);
        }
        if (t) put2(t + row * TR_LDH + col, v0, v1);
      }
    }
}

template <bool AL>
__global__ void __launch_bounds__(256, 1) k_mlp_deltas(Params P, const float* __restrict__ dY, const float* __restrict__ H1,
                                                       const float* __restrict__ H2, int n, float* dZ1, float* dZ2) {
  extern __shared__ __align__(16) __nv_bfloat16 sm16[];
  __nv_bfloat16 *W2 = sm16 + DZ_W2, *W3 = sm16 + DZ_W3, *Ys = sm16 + DZ_Y, *Z2s = sm16 + DZ_Z2;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n0 = 32 * warp;
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  // the four outputs padded to the 16 of a product step
  put4(W3 + TR_LD16 * tid, load4<AL>(P.W3 + 4 * tid));
  for (int c = 4; c < 16; c += 4) put4(W3 + TR_LD16 * tid + c, zero);
  stage<AL, 256, 256, TR_LDH>(W2, P.W2, tid, 256);
  for (int r0 = blockIdx.x * TR_ROWS; r0 < n; r0 += (int)gridDim.x * TR_ROWS) {
    __syncthreads();
    if (tid < TR_ROWS) {
      put4(Ys + TR_LD16 * tid, r0 + tid < n ? load4<AL>(dY + 4 * (size_t)(r0 + tid)) : zero);
      for (int c = 4; c < 16; c += 4) put4(Ys + TR_LD16 * tid + c, zero);
    }
    __syncthreads();
    float acc[2][4][4];
    product32<16, TR_LD16, TR_LD16, false>(acc, Ys, W3, n0, lane);
    masked_out<AL>(acc, H2, dZ2, Z2s, r0, n, n0, lane);
    __syncthreads();
    product32<256, TR_LDH, TR_LDH, false>(acc, Z2s, W2, n0, lane);
    masked_out<AL>(acc, H1, dZ1, nullptr, r0, n, n0, lane);
  }
}

// ---------------------------------------------------------------------------
// Gradients: dW2 = H1^T dZ2, dW1 = X^T dZ1, dW3 = H2^T dY in 32 x 32 tiles (88
// CTAs), and the biases' column sums of the right factors (17 more).  The inner
// dimension is the batch, added by the tensor cores row after row in one chain
// per output (deterministic, no atomics, no workspace): a chain of 256
// products for 4096 rows takes 5 us, so it is the operands' way that has to be
// short.  A thread holds GW_AHEAD stages of 64 rows in registers on their way
// from memory (96 KB in flight per CTA) and rounds them to BF16 into shared
// memory, where the warps read fragments by transposing matrix loads.  4096
// rows in 24 us.  (Asynchronous copies of the FP32 rows, paired and
// rounded on the way into the fragments, took 31 us: 16 shared loads and 6
// conversions per product step and warp.  Eight CTAs of a cluster for a tile,
// an eighth of the rows each, took 20 us, but the other order of additions moved
// the gradients by 8e-6.)
// ---------------------------------------------------------------------------
constexpr int GW_THREADS = 256, GW_T = 32, GW_STEP = 64, GW_AHEAD = 6, GW_LD = GW_T + 8, GW_TILES = 88, GW_BIAS = 17;

template <int LD> __device__ __forceinline__ void frag_a_by_k(unsigned (&r)[4], const __nv_bfloat16* t, int m, int k, int lane) {
  ldm4t(r, t + (k + (lane >> 4) * 8 + (lane & 7)) * LD + m + ((lane >> 3) & 1) * 8);
}

// Column sums of 32 columns of D (ldd columns, n rows): eight row phases, each
// added in row order, then the phases in order.
__device__ __forceinline__ void column_sums(const float* __restrict__ D, int ldd, int c0, int n, float* out, float (*red)[32]) {
  const int lane = threadIdx.x & 31, y = threadIdx.x >> 5, c = c0 + lane;
  float s = 0.f;
  if (c < ldd) {
    const float* p = D + c;
    int r = y;
    for (; r + 8 * 15 < n; r += 8 * 16) {
      float v[16];
#pragma unroll
      for (int k = 0; k < 16; ++k) v[k] = __ldg(p + (size_t)(r + 8 * k) * ldd);
#pragma unroll
      for (int k = 0; k < 16; ++k) s += v[k];
    }
    for (; r < n; r += 8) s += __ldg(p + (size_t)r * ldd);
  }
  red[y][lane] = s;
  __syncthreads();
  if (y == 0 && c < ldd) {
    float t = red[0][lane];
    for (int k = 1; k < 8; ++k) t += red[k][lane];
    out[c] = t;
  }
}

template <bool AL>
__global__ void __launch_bounds__(GW_THREADS)
    k_mlp_grads(Params G, const float* __restrict__ X, const float* __restrict__ H1, const float* __restrict__ H2,
                const float* __restrict__ dY, const float* __restrict__ dZ1, const float* __restrict__ dZ2, int n) {
  __shared__ __align__(16) __nv_bfloat16 As[2][GW_STEP * GW_LD], Bs[2][GW_STEP * GW_LD];  // stored by batch row
  __shared__ float red[8][32];
  const int tile = (int)blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tile >= GW_TILES) {
    const int b = tile - GW_TILES;
    if (b < 8) column_sums(dZ2, 256, 32 * b, n, G.b2, red);
    else if (b < 16) column_sums(dZ1, 256, 32 * (b - 8), n, G.b1, red);
    else column_sums(dY, 4, 0, n, G.b3, red);
    return;
  }
  // the tile's product: left factor (lda columns, from m0), right factor (ldb columns, from n0)
  const float *A, *Bm;
  float* C;
  int lda, ldb, m0, n0;
  if (tile < 64) {
    A = H1; lda = 256; Bm = dZ2; ldb = 256; C = G.W2; m0 = GW_T * (tile >> 3); n0 = GW_T * (tile & 7);
  } else if (tile < 80) {
    A = X; lda = 64; Bm = dZ1; ldb = 256; C = G.W1; m0 = GW_T * ((tile - 64) >> 3); n0 = GW_T * (tile & 7);
  } else {
    A = H2; lda = 256; Bm = dY; ldb = 4; C = G.W3; m0 = GW_T * (tile - 80); n0 = 0;
  }
  const int width = ldb < GW_T ? ldb : GW_T;  // columns of the right factor in this tile
  const int steps = n / GW_STEP + (n % GW_STEP ? 1 : 0);
  const int c4 = 4 * (tid & 7), rr = tid >> 3;  // this thread's columns and first row of a stage
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  float4 a4[GW_AHEAD][2], b4[GW_AHEAD][2];
  const auto fetch = [&](int step, float4 (&av)[2], float4 (&bv)[2]) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const long long row = (long long)step * GW_STEP + rr + 32 * i;
      av[i] = row < n ? load4<AL>(A + (size_t)row * lda + m0 + c4) : zero;
      bv[i] = row < n && c4 < width ? load4<AL>(Bm + (size_t)row * ldb + n0 + c4) : zero;
    }
  };
#pragma unroll
  for (int k = 0; k < GW_AHEAD; ++k) fetch(k, a4[k], b4[k]);
  const int wm = (warp >> 2) * 16, wn = (warp & 3) * 8;
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
  for (int step0 = 0; step0 < steps; step0 += GW_AHEAD) {
#pragma unroll
    for (int d = 0; d < GW_AHEAD; ++d) {
      const int step = step0 + d;
      if (step >= steps) break;
      __nv_bfloat16 *sa = As[step & 1], *sb = Bs[step & 1];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        put4(sa + (rr + 32 * i) * GW_LD + c4, a4[d][i]);
        put4(sb + (rr + 32 * i) * GW_LD + c4, b4[d][i]);
      }
      fetch(step + GW_AHEAD, a4[d], b4[d]);
      __syncthreads();  // (the stage written next was last read before this barrier)
#pragma unroll
      for (int k = 0; k < GW_STEP; k += 16) {
        unsigned a[4], b0, b1;
        frag_a_by_k<GW_LD>(a, sa, wm, k, lane);
        const unsigned p = (unsigned)__cvta_generic_to_shared(sb + (k + (lane & 15)) * GW_LD + wn);
        asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];\n" : "=r"(b0), "=r"(b1) : "r"(p));
        mma_bf16(acc, a, b0, b1);
      }
    }
  }
  const int gid = lane >> 2, tig = lane & 3;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const int m = wm + gid + (c >= 2 ? 8 : 0), col = wn + 2 * tig + (c & 1);
    if (col < width) C[(size_t)(m0 + m) * ldb + n0 + col] = acc[c];
  }
}

// ---------------------------------------------------------------------------
// dY = 2 (Y - T) / n and the loss, the sum of (Y - T)^2 over n in FP64.  Up to
// MSE_CLUSTER_MAX values one cluster does both (one launch in place of two,
// the sums added in rank order); above, MSE_BLOCKS CTAs leave partial sums for
// a second launch.
// ---------------------------------------------------------------------------
constexpr int MSE_CLUSTER_MAX = 1 << 18, MSE_BLOCKS = 64;

// dY of this thread's elements and the block's sum of squares (in thread 0)
__device__ __forceinline__ double mse_block(const float* __restrict__ Y, const float* __restrict__ T, int count, float inv_n,
                                            float* __restrict__ dY) {
  __shared__ double red[8];
  double acc = 0.0;
#pragma unroll 8
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
    const float d = Y[i] - T[i];
    dY[i] = 2.0f * d * inv_n;
    acc += (double)d * d;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(TR_FULL, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  double s = red[0];
  if (threadIdx.x == 0)
    for (int k = 1; k < 8; ++k) s += red[k];
  return s;
}

__global__ void __cluster_dims__(8, 1, 1) __launch_bounds__(256)
    k_mse_cluster(const float* __restrict__ Y, const float* __restrict__ T, int count, float inv_n, double inv_nd,
                  float* __restrict__ dY, float* __restrict__ loss) {
  __shared__ double part;
  cg::cluster_group cluster = cg::this_cluster();
  const double s = mse_block(Y, T, count, inv_n, dY);
  if (threadIdx.x == 0) part = s;
  cluster.sync();
  if (cluster.block_rank() == 0 && threadIdx.x == 0) {
    double t = 0.0;
    for (int q = 0; q < 8; ++q) t += *cluster.map_shared_rank(&part, q);
    *loss = (float)(t * inv_nd);
  }
  cluster.sync();
}

__global__ void __launch_bounds__(256) k_mse(const float* __restrict__ Y, const float* __restrict__ T, int count, float inv_n,
                                             float* __restrict__ dY, double* __restrict__ partial) {
  const double s = mse_block(Y, T, count, inv_n, dY);
  if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

__global__ void k_loss_finish(const double* partial, int nb, double inv_n, float* loss) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  double s = 0.0;
  for (int b = 0; b < nb; ++b) s += partial[b];
  *loss = (float)(s * inv_n);
}

// AdamW (decoupled weight decay) on FP32 master parameters.
__global__ void k_adamw(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                        float* __restrict__ v, int n, float lr, float b1, float b2, float eps, float wd, float c1,
                        float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float mi = b1 * m[i] + (1.f - b1) * g[i];
  const float vi = b2 * v[i] + (1.f - b2) * g[i] * g[i];
  m[i] = mi;
  v[i] = vi;
  const float mh = mi / c1, vh = vi / c2;
  p[i] = p[i] - lr * (mh / (sqrtf(vh) + eps) + wd * p[i]);
}

// X[r][c] = (X[r][c] - shift[c]) * scale[c]: the training driver's feature
// standardisation and target weighting
__global__ void k_scale_columns(float* __restrict__ X, long long n, int cols, const float* __restrict__ shift,
                                const float* __restrict__ scale) {
  const long long total = n * cols;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(e % cols);
    X[e] = (X[e] - shift[c]) * scale[c];
  }
}

bool aligned16(std::initializer_list<const void*> ps) {
  for (const void* p : ps)
    if (reinterpret_cast<uintptr_t>(p) % 16 != 0) return false;
  return true;
}

// CTAs for n batch rows: a tile each, at most one CTA per SM
cudaError_t row_grid(int n, int& grid) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int tiles = n / TR_ROWS + (n % TR_ROWS ? 1 : 0);
  grid = tiles < sms ? tiles : sms;
  return e;
}

template <bool AL>
cudaError_t forward(const Params& P, const float* X, int n, float* Y, float* H1, float* H2, cudaStream_t s) {
  int grid = 0;
  cudaError_t e = row_grid(n, grid);
  const int smem = (int)(FW_END * sizeof(__nv_bfloat16));
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_mlp_forward<AL>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  k_mlp_forward<AL><<<grid, 256, smem, s>>>(P, X, n, Y, H1, H2);
  return cudaGetLastError();
}

template <bool AL>
cudaError_t backward(const Params& P, const Params& G, const float* X, const float* H1, const float* H2, const float* dY,
                     int n, float* dZ1, float* dZ2, cudaStream_t s) {
  int grid = 0;
  cudaError_t e = row_grid(n, grid);
  const int smem = (int)(DZ_END * sizeof(__nv_bfloat16));
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_mlp_deltas<AL>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  k_mlp_deltas<AL><<<grid, 256, smem, s>>>(P, dY, H1, H2, n, dZ1, dZ2);
  k_mlp_grads<AL><<<GW_TILES + GW_BIAS, GW_THREADS, 0, s>>>(G, X, H1, H2, dY, dZ1, dZ2, n);
  return cudaGetLastError();
}

}  // namespace
}  // namespace mi

using namespace mi;

extern "C" {

// Parameter block layout (floats): W1 64x256, b1 256, W2 256x256, b2 256, W3 256x4, b3 4.
size_t mi_mlp_param_count(void) { return 64 * 256 + 256 + 256 * 256 + 256 + 256 * 4 + 4; }

mi_status mi_mlp_forward(const float* params, const float* X, int n, float* Y, float* acts, void* stream) {
  if (n < 0 || (n > 0 && (!params || !X || !Y || !acts))) {
    set_thread_error("mi_mlp_forward: null pointer or negative batch");
    return MI_EINVAL;
  }
  if (n == 0) return MI_OK;
  const Params P = views(params);
  float* H1 = acts;                    // n x 256, relu(X W1 + b1)
  float* H2 = acts + (size_t)n * 256;  // n x 256, relu(H1 W2 + b2)
  cudaStream_t s = (cudaStream_t)stream;
  const cudaError_t e = aligned16({params, X, acts}) ? forward<true>(P, X, n, Y, H1, H2, s)
                                                     : forward<false>(P, X, n, Y, H1, H2, s);
  if (e != cudaSuccess) {
    set_thread_error("mi_mlp_forward: launch failed");
    return MI_ECUDA;
  }
  return MI_OK;
}

mi_status mi_mlp_mse(const float* Y, const float* T, int n, float* dY, float* loss, double* scratch, void* stream) {
  if (!Y || !T || !dY || !loss || !scratch || n <= 0) {
    set_thread_error("mi_mlp_mse: null pointer or empty batch");
    return MI_EINVAL;
  }
  cudaStream_t s = (cudaStream_t)stream;
  if (4 * (long long)n <= MSE_CLUSTER_MAX) {
    k_mse_cluster<<<8, 256, 0, s>>>(Y, T, 4 * n, 1.0f / n, 1.0 / n, dY, loss);
  } else {
    k_mse<<<MSE_BLOCKS, 256, 0, s>>>(Y, T, 4 * n, 1.0f / n, dY, scratch);
    k_loss_finish<<<1, 32, 0, s>>>(scratch, MSE_BLOCKS, 1.0 / n, loss);
  }
  if (cudaGetLastError() != cudaSuccess) {
    set_thread_error("mi_mlp_mse: launch failed");
    return MI_ECUDA;
  }
  return MI_OK;
}

mi_status mi_mlp_backward(const float* params, const float* X, const float* acts, const float* dY, int n,
                          float* grads, float* scratch, void* stream) {
  if (!params || !X || !acts || !dY || !grads || !scratch || n <= 0) {
    set_thread_error("mi_mlp_backward: null pointer or empty batch");
    return MI_EINVAL;
  }
  const Params P = views(params), G = views(grads);
  const float *H1 = acts, *H2 = acts + (size_t)n * 256;
  float *dZ2 = scratch, *dZ1 = scratch + (size_t)n * 256;  // n x 256 each
  cudaStream_t s = (cudaStream_t)stream;
  const cudaError_t e = aligned16({params, X, acts, dY, scratch})
                            ? backward<true>(P, G, X, H1, H2, dY, n, dZ1, dZ2, s)
                            : backward<false>(P, G, X, H1, H2, dY, n, dZ1, dZ2, s);
  if (e != cudaSuccess) {
    set_thread_error("mi_mlp_backward: launch failed");
    return MI_ECUDA;
  }
  return MI_OK;
}

mi_status mi_mlp_adamw(float* params, const float* grads, float* m, float* v, int step, float lr, float beta1,
                       float beta2, float eps, float weight_decay, void* stream) {
  if (!params || !grads || !m || !v || step < 1) {
    set_thread_error("mi_mlp_adamw: null pointer or step < 1");
    return MI_EINVAL;
  }
  const int n = (int)mi_mlp_param_count();
  const float c1 = 1.f - powf(beta1, (float)step), c2 = 1.f - powf(beta2, (float)step);
  k_adamw<<<(n + 255) / 256, 256, 0, (cudaStream_t)stream>>>(params, grads, m, v, n, lr, beta1, beta2, eps,
                                                             weight_decay, c1, c2);
  if (cudaGetLastError() != cudaSuccess) {
    set_thread_error("mi_mlp_adamw: launch failed");
    return MI_ECUDA;
  }
  return MI_OK;
}

mi_status mi_mlp_scale_columns(float* X, long long n, int cols, const float* shift, const float* scale, void* stream) {
  if (n < 0 || cols < 1 || (n > 0 && (!X || !shift || !scale))) {
    set_thread_error("mi_mlp_scale_columns: null pointer, n < 0 or cols < 1");
    return MI_EINVAL;
  }
  if (n == 0) return MI_OK;
  k_scale_columns<<<2048, 256, 0, (cudaStream_t)stream>>>(X, n, cols, shift, scale);
  if (cudaGetLastError() != cudaSuccess) {
    set_thread_error("mi_mlp_scale_columns: launch failed");
    return MI_ECUDA;
  }
  return MI_OK;
}

}  // extern "C"
