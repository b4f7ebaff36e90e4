// Genetic Algorithm capture of the principal outer contour (Sec. 2.2,
// Algorithm 1).  One generation is four launches: the draws (a thread per gene:
// its copy for the mutation, the mutating genes appended to a list, the pairing
// keys); the keys' ranks (the random pairing) and the new genes (a warp per
// listed gene: the convex-hull test of a candidate point spreads the facet planes
// over the lanes); the children and their fitness (a CTA per individual:
// crossover, then threads over hull points, fixed-order block sum); and the
// selection (a warp per candidate, its rank by counting over parents and
// children).  Random numbers come from a counter-based SplitMix64, so every
// draw is a function of (seed, generation, individual, gene, slot) and the
// run does not depend on the launch shapes.
//
// Bound by launches and latency up to a few hundred individuals, by the fitness'
// reciprocals above: 1200 individuals of 32 genes on 2048 points take 55 us a
// generation (137 in nine launches, with the planes read one after another and
// a single point per gene read).
#include <cmath>

#include "mi_ga.h"
#include "mi_internal.cuh"

namespace mi {
namespace {

constexpr unsigned GA_INIT_GEN = 0xFFFFFFFFu;
constexpr int GA_SLOT_MUTATE = 0, GA_SLOT_K = 1, GA_SLOT_KEY = 2;
constexpr int GA_TRIES_MUTATE = 8, GA_TRIES_INIT = 64;
constexpr int GA_FIT_THREADS = 256;

// SplitMix64 output for state x: the golden-gamma step, two xor-shift-multiply
// rounds and a final xor-shift (constants of the published generator).
__host__ __device__ __forceinline__ unsigned long long splitmix64(unsigned long long x) {
  unsigned long long z = x + 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

__device__ __forceinline__ unsigned long long ga_draw(unsigned long long seed, unsigned long long gen,
                                                      unsigned long long ind, int gene, int slot) {
  unsigned long long h = splitmix64(seed);
  h = splitmix64(h ^ gen);
  h = splitmix64(h ^ ind);
  return splitmix64(h ^ ((unsigned long long)gene * 256ull + (unsigned long long)slot));
}

// top 24 bits times 2^-24: exact in FP32
__device__ __forceinline__ float ga_uniform(unsigned long long seed, unsigned long long gen, unsigned long long ind,
                                            int gene, int slot) {
  return (float)(unsigned)(ga_draw(seed, gen, ind, gene, slot) >> 40) * 5.9604644775390625e-8f;
}

// lo + u (hi - lo), single FP32 roundings
__device__ __forceinline__ float ga_lerp(float lo, float hi, float u) {
  return __fadd_rn(lo, __fmul_rn(u, __fsub_rn(hi, lo)));
}

struct GaLaunch {
  int n_ind, n_genes, m, n_planes;
  const float* hull;
  const float* planes;
  float lo[3], hi[3], klo, khi;
  float c_m;
  int p;  // crossover point
  unsigned long long seed;
};

// outside the convex hull: n . p > d for some facet plane (FP32, single
// roundings, left to right), the planes spread over the lanes of a warp
// (every lane passes the same point), eight per lane in flight between votes:
// one after another, each waited for, an inside point took 128 turns for 4000
// planes, and an outside one as many in the lanes that see nothing of it
template <bool AL>  // AL: the planes are 16-byte aligned
__device__ __forceinline__ bool ga_outside_warp(const float* planes, int n_planes, float x, float y, float z,
                                                int lane) {
  for (int p0 = 0; p0 < n_planes; p0 += 256) {
    float4 P[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float* q = planes + 4 * (size_t)min(p0 + 32 * k + lane, n_planes - 1);
      P[k] = AL ? __ldg(reinterpret_cast<const float4*>(q)) : make_float4(__ldg(q), __ldg(q + 1), __ldg(q + 2), __ldg(q + 3));
    }
    bool out = false;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float s = __fadd_rn(__fadd_rn(__fmul_rn(P[k].x, x), __fmul_rn(P[k].y, y)), __fmul_rn(P[k].z, z));
      out = out || s > P[k].w;
    }
    if (__any_sync(0xffffffffu, out)) return true;
  }
  return false;
}

// a new gene inside the hull for (gen, ind, gene) by one warp; false after
// `tries` rejections
template <bool AL>
__device__ __forceinline__ bool ga_new_gene(const GaLaunch& G, unsigned long long gen, int ind, int gene, int tries,
                                            int lane, float4& out) {
  for (int t = 0; t < tries; ++t) {
    const float x = ga_lerp(G.lo[0], G.hi[0], ga_uniform(G.seed, gen, ind, gene, 3 + 3 * t));
    const float y = ga_lerp(G.lo[1], G.hi[1], ga_uniform(G.seed, gen, ind, gene, 3 + 3 * t + 1));
    const float z = ga_lerp(G.lo[2], G.hi[2], ga_uniform(G.seed, gen, ind, gene, 3 + 3 * t + 2));
    if (!ga_outside_warp<AL>(G.planes, G.n_planes, x, y, z, lane)) {
      out = make_float4(x, y, z, ga_lerp(G.klo, G.khi, ga_uniform(G.seed, gen, ind, gene, GA_SLOT_K)));
      return true;
    }
  }
  return false;
}

// one warp per gene of the initial population
template <bool AL>
__global__ void __launch_bounds__(256) k_ga_init(GaLaunch G, float4* pop) {
  const long long e = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (e >= (long long)G.n_ind * G.n_genes) return;
  const int ind = (int)(e / G.n_genes), gene = (int)(e - (long long)ind * G.n_genes);
  float4 v;
  if (!ga_new_gene<AL>(G, GA_INIT_GEN, ind, gene, GA_TRIES_INIT, lane, v)) {
    v = make_float4(__fmul_rn(0.5f, __fadd_rn(G.lo[0], G.hi[0])), __fmul_rn(0.5f, __fadd_rn(G.lo[1], G.hi[1])),
                    __fmul_rn(0.5f, __fadd_rn(G.lo[2], G.hi[2])),
                    ga_lerp(G.klo, G.khi, ga_uniform(G.seed, GA_INIT_GEN, ind, gene, GA_SLOT_K)));
  }
  if (lane == 0) pop[e] = v;
}

// F = sum_i (f_i - 1)^2 of the individual in shared memory: threads over the
// hull points (four at a time share a gene read), each thread's terms and the
// block's tree in a fixed order
__device__ __forceinline__ void ga_fitness(const GaLaunch& G, const float4* genes, float* fit) {
  __shared__ float red[GA_FIT_THREADS];
  const int t = threadIdx.x;
  float part = 0.f;
  for (int i0 = t; i0 < G.m; i0 += 4 * GA_FIT_THREADS) {
    float x[4], y[4], z[4], f[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int i = min(i0 + k * GA_FIT_THREADS, G.m - 1);
      x[k] = G.hull[3 * i];
      y[k] = G.hull[3 * i + 1];
      z[k] = G.hull[3 * i + 2];
      f[k] = 0.f;
    }
#pragma unroll 2
    for (int g = 0; g < G.n_genes; ++g) {
      const float4 b = genes[g];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float dx = x[k] - b.x, dy = y[k] - b.y, dz = z[k] - b.z;
        f[k] += b.w * rcp_start(dx * dx + dy * dy + dz * dz);
      }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (i0 + k * GA_FIT_THREADS < G.m) part += (f[k] - 1.0f) * (f[k] - 1.0f);
  }
  red[t] = part;
  __syncthreads();
#pragma unroll
  for (int s = GA_FIT_THREADS / 2; s > 16; s >>= 1) {
    if (t < s) red[t] += red[t + s];
    __syncthreads();
  }
  if (t < 32) {
    float v = red[t];
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) v += __shfl_down_sync(0xffffffffu, v, s);
    if (t == 0) *fit = v;
  }
}

// the fitness of every individual of a population, one per CTA
__global__ void __launch_bounds__(GA_FIT_THREADS) k_ga_fitness(GaLaunch G, const float4* pop, float* fit) {
  extern __shared__ float4 genes[];
  const int ind = blockIdx.x;
  for (int g = threadIdx.x; g < G.n_genes; g += GA_FIT_THREADS) genes[g] = pop[(long long)ind * G.n_genes + g];
  __syncthreads();
  ga_fitness(G, genes, fit + ind);
}

// The draws of a generation, a thread per gene: its copy for the mutation; the
// genes whose mutation draw falls below c_m, appended to a list (one append per
// warp; the list order does not matter); and the individuals' pairing keys.
__global__ void __launch_bounds__(256) k_ga_draws(GaLaunch G, unsigned gen, const float4* __restrict__ pop,
                                                  float4* __restrict__ mut, int* list, int* count,
                                                  unsigned long long* keys) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const bool there = e < (long long)G.n_ind * G.n_genes;
  bool listed = false;
  if (there) {
    const int ind = (int)(e / G.n_genes), gene = (int)(e - (long long)ind * G.n_genes);
    mut[e] = pop[e];
    listed = ga_uniform(G.seed, gen, ind, gene, GA_SLOT_MUTATE) < G.c_m;
    if (gene == 0) keys[ind] = ga_draw(G.seed, gen, (unsigned long long)ind, 0, GA_SLOT_KEY);
  }
  const unsigned m = __ballot_sync(0xffffffffu, listed), lane = threadIdx.x & 31u;
  int base = 0;
  if (lane == 0 && m) base = atomicAdd(count, __popc(m));
  base = __shfl_sync(0xffffffffu, base, 0);
  if (listed) list[base + __popc(m & ((1u << lane) - 1u))] = (int)e;
}

// Two independent parts of a launch.  The first perm_blocks blocks: perm[rank of
// key i] = i and rank[i], ranks ascending with ties to the lower index; a warp
// per key, its lanes counting over strided keys.  The others: a new gene for
// every listed gene, one warp each (every gene's draws are its own).
template <bool AL>
__global__ void __launch_bounds__(256) k_ga_pair_mutate(GaLaunch G, unsigned gen, const unsigned long long* __restrict__ keys,
                                                        int* perm, int* rank, const int* __restrict__ list,
                                                        const int* __restrict__ count, float4* mut, int perm_blocks) {
  const int lane = threadIdx.x & 31;
  if ((int)blockIdx.x < perm_blocks) {
    const int i = (int)(((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (i >= G.n_ind) return;
    const unsigned long long ki = keys[i];
    int r = 0;
#pragma unroll 4
    for (int j = lane; j < G.n_ind; j += 32) {
      const unsigned long long kj = keys[j];
      r += (kj < ki) || (kj == ki && j < i);
    }
    r = __reduce_add_sync(0xffffffffu, r);
    if (lane == 0) {
      perm[r] = i;
      rank[i] = r;
    }
    return;
  }
  const int n = *count;
  for (long long w = ((long long)(blockIdx.x - perm_blocks) * blockDim.x + threadIdx.x) >> 5; w < n;
       w += ((long long)(gridDim.x - perm_blocks) * blockDim.x) >> 5) {
    const int e = list[w];
    const int ind = e / G.n_genes, gene = e - ind * G.n_genes;
    float4 v;
    if (ga_new_gene<AL>(G, gen, ind, gene, GA_TRIES_MUTATE, lane, v) && lane == 0) mut[e] = v;
  }
}

// The children of the pairs (perm[2q], perm[2q+1]) of the mutated individuals
// and their fitness, one child per CTA: an individual's child has its own genes
// up to the crossover point and its partner's from there on (an odd last
// individual is copied).
__global__ void __launch_bounds__(GA_FIT_THREADS) k_ga_children(GaLaunch G, const float4* __restrict__ mut,
                                                                const int* __restrict__ perm, const int* __restrict__ rank,
                                                                float4* off, float* fit) {
  extern __shared__ float4 genes[];
  const int ind = blockIdx.x, q = rank[ind] ^ 1, mate = q < G.n_ind ? perm[q] : ind;
  for (int g = threadIdx.x; g < G.n_genes; g += GA_FIT_THREADS) {
    const float4 v = mut[(long long)(g < G.p ? ind : mate) * G.n_genes + g];
    genes[g] = v;
    off[(long long)ind * G.n_genes + g] = v;
  }
  __syncthreads();
  ga_fitness(G, genes, fit + ind);
}

// the n_ind fittest of parents (0..n_ind-1) and children (n_ind..), by
// counting: a warp per candidate, its lanes over strided candidates; the
// mutation list is emptied for the next generation.  Up to GA_STAGED individuals
// a block keeps the fitness values in shared memory.
constexpr int GA_STAGED = 4096;
template <bool STAGED>
__global__ void __launch_bounds__(256) k_ga_select(GaLaunch G, const float4* __restrict__ pop, const float* __restrict__ fit,
                                                   const float4* __restrict__ off, const float* __restrict__ fit_off,
                                                   float4* npop, float* nfit, int* count) {
  if (blockIdx.x == 0 && threadIdx.x == 0) *count = 0;
  extern __shared__ float vals[];  // all fitness values (STAGED), NaN as infinity
  const int n2 = 2 * G.n_ind;
  const int c = (int)(((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  auto val = [&](int d) {
    const float v = d < G.n_ind ? fit[d] : fit_off[d - G.n_ind];
    return isnan(v) ? INFINITY : v;
  };
  if (STAGED) {
#pragma unroll 4
    for (int d = threadIdx.x; d < n2; d += blockDim.x) vals[d] = val(d);
    __syncthreads();
  }
  if (c >= n2) return;
  const float fc = STAGED ? vals[c] : val(c);
  int r = 0;
#pragma unroll 8
  for (int d = lane; d < n2; d += 32) {
    const float fd = STAGED ? vals[d] : val(d);
    r += (fd < fc) || (fd == fc && d < c);
  }
  r = __reduce_add_sync(0xffffffffu, r);
  if (r >= G.n_ind) return;
  const float4* src = c < G.n_ind ? pop + (long long)c * G.n_genes : off + (long long)(c - G.n_ind) * G.n_genes;
  for (int g = lane; g < G.n_genes; g += 32) npop[(long long)r * G.n_genes + g] = src[g];
  if (lane == 0) nfit[r] = fc;
}

inline size_t align256(size_t b) { return (b + 255) / 256 * 256; }

}  // namespace
}  // namespace mi

extern "C" size_t mi_ga_scratch_bytes(int n_ind, int n_genes) {
  using namespace mi;
  if (n_ind < 1 || n_genes < 1) return 0;
  const size_t popb = align256(sizeof(float4) * (size_t)n_ind * n_genes);
  return 3 * popb + 3 * align256(sizeof(float) * n_ind) + align256(sizeof(unsigned long long) * n_ind) +
         align256(sizeof(int) * n_ind) + align256(sizeof(int) * (size_t)n_ind * n_genes) + 256;
}

extern "C" mi_status mi_ga_run(int n_ind, int n_genes, const float* hull, int m, const float* planes, int n_planes,
                               const float* bbox, const float* krange, float c_m, float c_c, unsigned long long seed,
                               int generations, int init, float* pop, float* fit, float* offspring,
                               float* fit_offspring, void* scratch, void* stream) {
  using namespace mi;
  if (n_ind < 2 || n_genes < 1 || m < 1 || n_planes < 1 || generations < 0 || !(c_m >= 0.f && c_m <= 1.f) ||
      !(c_c >= 0.f && c_c <= 1.f) || !hull || !planes || !bbox || !krange || !pop || !fit || !scratch)
    return MI_EINVAL;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  GaLaunch G;
  G.n_ind = n_ind;
  G.n_genes = n_genes;
  G.m = m;
  G.n_planes = n_planes;
  G.hull = hull;
  G.planes = planes;
  for (int a = 0; a < 3; ++a) {
    G.lo[a] = bbox[a];
    G.hi[a] = bbox[3 + a];
  }
  G.klo = krange[0];
  G.khi = krange[1];
  G.c_m = c_m;
  G.p = (int)std::floor((double)c_c * n_genes);
  G.seed = seed;
  // scratch: a second population, the children, two fitness arrays, ranks, keys,
  // the pairing, the mutated population, the mutation list and its count
  unsigned char* sp = static_cast<unsigned char*>(scratch);
  const size_t popb = align256(sizeof(float4) * (size_t)n_ind * n_genes);
  float4* popB = reinterpret_cast<float4*>(sp);
  float4* off = reinterpret_cast<float4*>(sp + popb);
  float* fitB = reinterpret_cast<float*>(sp + 2 * popb);
  float* fitO = reinterpret_cast<float*>(sp + 2 * popb + align256(sizeof(float) * n_ind));
  int* rank = reinterpret_cast<int*>(sp + 2 * popb + 2 * align256(sizeof(float) * n_ind));
  unsigned long long* keys =
      reinterpret_cast<unsigned long long*>(sp + 2 * popb + 3 * align256(sizeof(float) * n_ind));
  int* perm = reinterpret_cast<int*>(sp + 2 * popb + 3 * align256(sizeof(float) * n_ind) +
                                     align256(sizeof(unsigned long long) * n_ind));
  unsigned char* sp2 = reinterpret_cast<unsigned char*>(perm) + align256(sizeof(int) * n_ind);
  float4* mut = reinterpret_cast<float4*>(sp2);
  int* mlist = reinterpret_cast<int*>(sp2 + popb);
  int* mcount = reinterpret_cast<int*>(sp2 + popb + align256(sizeof(int) * (size_t)n_ind * n_genes));
  float4* cur = reinterpret_cast<float4*>(pop);
  float4* nxt = popB;
  float* fcur = fit;
  float* fnxt = fitB;
  const long long ng = (long long)n_ind * n_genes;
  const size_t gsm = sizeof(float4) * (size_t)n_genes;
  // with the reduction's static part: 48 KB is the limit of both together
  if (gsm + sizeof(float) * GA_FIT_THREADS > 48 * 1024 &&
      (cudaFuncSetAttribute(k_ga_fitness, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gsm) != cudaSuccess ||
       cudaFuncSetAttribute(k_ga_children, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gsm) != cudaSuccess))
    return MI_ECUDA;
  const bool al = reinterpret_cast<uintptr_t>(planes) % 16 == 0;
  if (init) {
    const unsigned blocks = (unsigned)((ng * 32 + 255) / 256);
    if (al) k_ga_init<true><<<blocks, 256, 0, s>>>(G, cur);
    else k_ga_init<false><<<blocks, 256, 0, s>>>(G, cur);
  }
  k_ga_fitness<<<n_ind, GA_FIT_THREADS, gsm, s>>>(G, cur, fcur);
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return MI_ECUDA;
  if (generations > 0 && cudaMemsetAsync(mcount, 0, sizeof(int), s) != cudaSuccess) return MI_ECUDA;
  const int perm_blocks = (int)(((long long)n_ind * 32 + 255) / 256);
  // 8 warps per block over the list, which holds at most every gene
  const long long most = (ng * 32 + 255) / 256;
  const int mut_blocks = (int)(most < 8LL * sms ? most : 8LL * sms);
  for (int gen = 0; gen < generations; ++gen) {
    k_ga_draws<<<(unsigned)((ng + 255) / 256), 256, 0, s>>>(G, (unsigned)gen, cur, mut, mlist, mcount, keys);
    if (al) k_ga_pair_mutate<true><<<perm_blocks + mut_blocks, 256, 0, s>>>(G, (unsigned)gen, keys, perm, rank, mlist, mcount, mut, perm_blocks);
    else k_ga_pair_mutate<false><<<perm_blocks + mut_blocks, 256, 0, s>>>(G, (unsigned)gen, keys, perm, rank, mlist, mcount, mut, perm_blocks);
    k_ga_children<<<n_ind, GA_FIT_THREADS, gsm, s>>>(G, mut, perm, rank, off, fitO);
    if (gen == generations - 1 && offspring) {
      if (cudaMemcpyAsync(offspring, off, sizeof(float4) * ng, cudaMemcpyDeviceToDevice, s) != cudaSuccess)
        return MI_ECUDA;
      if (fit_offspring &&
          cudaMemcpyAsync(fit_offspring, fitO, sizeof(float) * n_ind, cudaMemcpyDeviceToDevice, s) != cudaSuccess)
        return MI_ECUDA;
    }
    const unsigned sel = (unsigned)(((long long)2 * n_ind * 32 + 255) / 256);
    if (n_ind <= GA_STAGED) k_ga_select<true><<<sel, 256, 2 * sizeof(float) * n_ind, s>>>(G, cur, fcur, off, fitO, nxt, fnxt, mcount);
    else k_ga_select<false><<<sel, 256, 0, s>>>(G, cur, fcur, off, fitO, nxt, fnxt, mcount);
    float4* t4 = cur;
    cur = nxt;
    nxt = t4;
    float* tf = fcur;
    fcur = fnxt;
    fnxt = tf;
  }
  if (cur != reinterpret_cast<float4*>(pop)) {
    if (cudaMemcpyAsync(pop, cur, sizeof(float4) * ng, cudaMemcpyDeviceToDevice, s) != cudaSuccess ||
        cudaMemcpyAsync(fit, fcur, sizeof(float) * n_ind, cudaMemcpyDeviceToDevice, s) != cudaSuccess)
      return MI_ECUDA;
  }
  return cudaGetLastError() == cudaSuccess ? MI_OK : MI_ECUDA;
}
