// de.cu -- device-side DEOCT step (Algorithm 4; Eqs. mutation, crossover,
// selection; the fitness of Section 3.2) and tree decoding (Eq. aenc, Eq. benc).
//
// One CTA per subproblem.  A step kernel does, in order and as its flags ask:
//   DE_FIRST  fitness of the just-evaluated initial population, best;
//   DE_SELECT fitness of the just-evaluated trials, Eq. selection, best;
//   DE_TRIAL  trial vectors of generation g from (population, best), their
//             decoded nodes for the evaluator, and zeroed class counts.
// So one generation is two launches: evaluator, step(SELECT|TRIAL), the latter of up
// to 256 individuals on chip (de_step_chip_kernel); for one
// problem with more than 256 individuals the step(SELECT|TRIAL) is itself split
// over CTAs in two launches (de_select_wide_kernel, de_trial_wide_kernel).  Gene
// arithmetic is float32 with one rounding per operation (__fsub_rn, __fmul_rn,
// __fadd_rn); random numbers come from Philox4x64-10 keyed by (seed, stream).
#include "internal.cuh"

namespace deoct {

namespace {

__device__ __forceinline__ const DEProb& prob_of(const DEArgs& a) {
  return a.probs ? a.probs[blockIdx.x] : a.single;
}

// (double)e for 0 <= e < 2^53 (exact), built with integer operations only: the
// leading one sets the exponent, the bits below it the significand.
__device__ __forceinline__ double exact_double(int64_t e) {
  if (e <= 0) return 0.0;
  const int lz = __clzll(e);
  const uint64_t mant = ((uint64_t)e << (lz + 1)) >> 12;  // the 52 bits below the leading one
  return __longlong_as_double((long long)(((uint64_t)(1086 - lz) << 52) | mant));
}

// alpha = 0 and alpha >= 0 by its bits (alpha is not NaN): one FP64 comparison costs
// a warp tens of cycles on this GPU's FP64 pipe, and a step has 4 to 32 warps.
__device__ __forceinline__ bool is_zero(double x) { return (__double_as_longlong(x) << 1) == 0; }
__device__ __forceinline__ bool non_negative(double x) { return __double_as_longlong(x) >= 0 || is_zero(x); }

// Fitness order.  With alpha >= 0 every fitness is a non-negative double (not
// -0), whose bit pattern as a signed 64-bit integer orders exactly like the
// value, so comparisons need no FP64 arithmetic; a negative alpha compares the
// doubles.
__device__ __forceinline__ bool fit_le(double x, double y, bool bits) {
  return bits ? __double_as_longlong(x) <= __double_as_longlong(y) : x <= y;
}
__device__ __forceinline__ bool fit_lt(double x, double y, bool bits) {
  return bits ? __double_as_longlong(x) < __double_as_longlong(y) : x < y;
}

// Asynchronous copy of 16 bytes to shared memory (through L2 alone).
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ float clamp_gene(float v, float hi) {
  v = v < 0.0f ? 0.0f : v;
  return v > hi ? hi : v;
}

// block-wide argmin (lowest index among minimal values); result in *best_s.
// bits: compare in the order of fit_lt (see there)
__device__ void block_argmin(const double* __restrict__ fit, int P, int* best_s, double* red_f,
                             int* red_i, bool bits) {
  double bf = 0.0;
  int bi = -1;
  for (int r = threadIdx.x; r < P; r += blockDim.x) {
    double f = fit[r];
    if (bi < 0 || fit_lt(f, bf, bits)) {
      bf = f;
      bi = r;
    }
  }
  // warp reduce
  for (int off = 16; off > 0; off >>= 1) {
    double of = __shfl_down_sync(0xFFFFFFFFu, bf, off);
    int oi = __shfl_down_sync(0xFFFFFFFFu, bi, off);
    if (oi >= 0 && (bi < 0 || fit_lt(of, bf, bits) || (!fit_lt(bf, of, bits) && oi < bi))) {
      bf = of;
      bi = oi;
    }
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) {
    red_f[warp] = bf;
    red_i[warp] = bi;
  }
  __syncthreads();
  if (warp == 0) {  // the warps' winners, reduced by one warp in the same order
    const int nw = (blockDim.x + 31) >> 5;
    bf = lane < nw ? red_f[lane] : 0.0;
    bi = lane < nw ? red_i[lane] : -1;
    for (int off = 16; off > 0; off >>= 1) {
      double of = __shfl_down_sync(0xFFFFFFFFu, bf, off);
      int oi = __shfl_down_sync(0xFFFFFFFFu, bi, off);
      if (oi >= 0 && (bi < 0 || fit_lt(of, bf, bits) || (!fit_lt(bf, of, bits) && oi < bi))) {
        bf = of;
        bi = oi;
      }
    }
    if (lane == 0) *best_s = bi;
  }
  __syncthreads();
}

__global__ void __launch_bounds__(1024) de_init_kernel(const DEArgs a) {
  const DEProb& pb = prob_of(a);
  const int P = a.P, D = a.depth, B = (1 << D) - 1, m = 2 * B, L = 1 << D;
  const float ub_a = (float)(pb.F + 1);
  const float hi_a = below_bound(ub_a), hi_b = below_bound(1.0f);
  for (int r = threadIdx.x; r < P; r += blockDim.x) {
    float* g = pb.pop + (int64_t)r * m;
    if (r < pb.S) {
      for (int q = 0; q < m; ++q) g[q] = pb.seeds[(int64_t)r * m + q];
    } else {
      U64x4 blk;
      for (int q = 0; q < m; ++q) {
        if ((q & 7) == 0) blk = philox4x64_10(0ull, (uint64_t)r, (uint64_t)(q >> 3), 0ull, pb.seed,
                                              pb.stream_id);
        const float u = u01(draw_from_block(blk, (uint32_t)q));
        const bool is_a = q < B;
        g[q] = clamp_gene(__fmul_rn(u, is_a ? ub_a : 1.0f), is_a ? hi_a : hi_b);
      }
    }
    for (int t = 0; t < B; ++t) {
      int av;
      uint32_t th;
      decode_gene_pair(g[t], g[B + t], pb.F, pb.n_unique, &av, &th);
      pb.nodes[(int64_t)r * B + t] = pack_node(av, th);
    }
  }
  uint32_t* cnt = pb.counts;
  const int64_t total = (int64_t)P * L * pb.K;
  for (int64_t e = threadIdx.x; e < total; e += blockDim.x) cnt[e] = 0;
  if (threadIdx.x == 0 && pb.gen) *pb.gen = 1;
}

// (errors + V) + alpha splits.  A function of its own: inlined beside the integer
// form for alpha = 0, the compiler computes both and selects, and the FP64
// operations are most of a small step's selection.
__device__ __noinline__ double penalised(int64_t ev, double alpha, uint32_t splits) {
  return __dadd_rn((double)ev, __dmul_rn(alpha, (double)splits));
}

// The fitness of Section 3.2 of individual r from its class counts,
//   f = (errors + V) + alpha * splits, errors = n - sum_leaf max_k count,
//   V = #{leaf : 0 < n_leaf < n_min}, splits = #{t : a_t >= 1} (ahat_t >= 1),
// by its group of G lanes (G a power of two that divides 32; `sub` the lane's
// place in the group, `gm` the group's lane mask): each lane takes leaves sub,
// sub + G, ... and genes sub, sub + G, ..., and the integer partial sums meet
// by shuffles, so every lane returns the same value.
__device__ double group_fitness(const uint32_t* __restrict__ c, const float* __restrict__ genes,
                                int B, int L, int K, int64_t n_valid, int n_min, double alpha,
                                int sub, int G, uint32_t gm) {
  long long correct = 0;
  uint32_t v = 0, splits = 0;
  // the lane's counts (leaves sub, sub + G, ..., every class), sixteen loads in
  // flight at a time: one after another they were a chain of memory round trips
  const int nc = ((L - sub + G - 1) / G) * K;
  int li = sub, ki = 0;  // leaf and class of the next count loaded
  uint32_t mx = 0;
  int64_t nl = 0;
  int kr = 0;            // classes of the current leaf reduced so far
  for (int e0 = 0; e0 < nc; e0 += 16) {
    uint32_t x[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      x[j] = e0 + j < nc ? c[li * K + ki] : 0u;
      if (++ki == K) {
        ki = 0;
        li += G;
      }
    }
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      if (e0 + j < nc) {
        mx = x[j] > mx ? x[j] : mx;
        nl += x[j];
        if (++kr == K) {
          correct += mx;
          if (nl > 0 && nl < n_min) v += 1;
          mx = 0;
          nl = 0;
          kr = 0;
        }
      }
    }
  }
  for (int t = sub; t < B; t += G) splits += genes[t] >= 1.0f ? 1u : 0u;
  for (int o = G >> 1; o > 0; o >>= 1) {
    correct += __shfl_xor_sync(gm, correct, o);
    v += __shfl_xor_sync(gm, v, o);
    splits += __shfl_xor_sync(gm, splits, o);
  }
  const int64_t errors = n_valid - (int64_t)correct;
  // alpha = 0 (the default): the fitness is the integer errors + V, and
  // (errors + V) + 0 * splits is that integer exactly
  if (is_zero(alpha)) return exact_double(errors + (int64_t)v);
  return penalised(errors + (int64_t)v, alpha, splits);
}

// Eq. selection of individual r by its group of G lanes: the fitness of its
// just-evaluated trial from the class counts; the trial replaces the individual
// when it is no worse (ties go to the trial).
__device__ __forceinline__ void select_individual(const DEArgs& a, const DEProb& pb, int r, int B,
                                                  int L, int K, int sub, int G, uint32_t gm,
                                                  bool bits) {
  const int m = 2 * B;
  const float* genes = pb.trial + (int64_t)r * m;
  const double f = group_fitness(pb.counts + (int64_t)r * L * K, genes, B, L, K, pb.n_valid,
                                 a.n_min, a.alpha, sub, G, gm);
  const double fr = pb.fit[r];
  __syncwarp(gm);  // every lane has read fit[r] before it is rewritten
  if (sub == 0) pb.fit_trial[r] = f;
  if (fit_le(f, fr, bits)) {
    float* dst = pb.pop + (int64_t)r * m;
    for (int q = sub; q < m; q += G) dst[q] = genes[q];
    if (sub == 0) pb.fit[r] = f;
  }
}

// Generation g's trial vector of individual r (Eqs. mutation and crossover) from
// the population and its best individual, stored with its decoded nodes.  Lane
// `sub` of the group takes consecutive genes, which share Philox blocks.
__device__ __forceinline__ void trial_individual(const DEArgs& a, const DEProb& pb, int r, int g,
                                                 int best, int B, int sub, int G, uint32_t gm) {
  const int P = a.P, m = 2 * B;
  const float ub_a = (float)(pb.F + 1);
  const float hi_a = below_bound(ub_a), hi_b = below_bound(1.0f);
  const float* sb = pb.pop + (int64_t)best * m;
  const int per = (m + G - 1) / G;
  // draws 0..7 come from block 0: r1, r2, q_rand, M, genes 0..3
  const U64x4 blk0 = philox4x64_10((uint64_t)g, (uint64_t)r, 0ull, 0ull, pb.seed, pb.stream_id);
  const uint32_t x0 = draw_from_block(blk0, 0), x1 = draw_from_block(blk0, 1);
  const uint32_t x2 = draw_from_block(blk0, 2), x3 = draw_from_block(blk0, 3);
  int r1 = (int)below(x0, (uint32_t)(P - 1));
  if (r1 >= r) r1 += 1;
  int r2 = (int)below(x1, (uint32_t)(P - 2));
  const int lo = r < r1 ? r : r1, hi = r < r1 ? r1 : r;
  if (r2 >= lo) r2 += 1;
  if (r2 >= hi) r2 += 1;
  const int qrand = (int)below(x2, (uint32_t)m);
  const float M = a.dither ? u01(x3) : a.M;
  const float* s1 = pb.pop + (int64_t)r1 * m;
  const float* s2 = pb.pop + (int64_t)r2 * m;
  const float* sr = pb.pop + (int64_t)r * m;
  float* u = pb.trial + (int64_t)r * m;
  U64x4 blk = blk0;
  uint32_t cur = 0;  // block held in blk
  const int q0 = sub * per, q1 = min(m, q0 + per);
  for (int q = q0; q < q1; ++q) {
    const uint32_t s = 4u + (uint32_t)q;
    if ((s >> 3) != cur) {
      cur = s >> 3;
      blk = philox4x64_10((uint64_t)g, (uint64_t)r, (uint64_t)cur, 0ull, pb.seed, pb.stream_id);
    }
    const float v = __fadd_rn(sb[q], __fmul_rn(M, __fsub_rn(s1[q], s2[q])));
    const float vc = clamp_gene(v, q < B ? hi_a : hi_b);
    const float rq = u01(draw_from_block(blk, s));
    u[q] = (rq <= a.CR || q == qrand) ? vc : sr[q];
  }
  __syncwarp(gm);  // the group's genes are written before they are decoded
  for (int t = sub; t < B; t += G) {
    int av;
    uint32_t th;
    decode_gene_pair(u[t], u[B + t], pb.F, pb.n_unique, &av, &th);
    pb.nodes[(int64_t)r * B + t] = pack_node(av, th);
  }
}

// One CTA per subproblem; each individual is worked on by a group of `lanes`
// consecutive threads (lanes x P <= blockDim.x, lanes <= 4), which shortens the
// chain of dependent loads one thread would walk alone.  Every value is the one a
// single thread computes: integer sums, the draws of a (generation,
// individual, block) Philox key, one rounding per float operation.
__global__ void __launch_bounds__(1024) de_step_kernel(const DEArgs a, int g_arg, int flags,
                                                       int lanes) {
  __shared__ double red_f[32];
  __shared__ int red_i[32];
  __shared__ int best_s;
  __shared__ int g_s;
  const DEProb& pb = prob_of(a);
  const int P = a.P, D = a.depth, B = (1 << D) - 1, m = 2 * B, L = 1 << D, K = pb.K;
  const int G = lanes;
  const int sub = threadIdx.x & (G - 1);
  const uint32_t gm = (G == 32 ? 0xFFFFFFFFu : ((1u << G) - 1u)) << ((threadIdx.x & 31) & ~(G - 1));
  const int r0 = threadIdx.x / G, rstep = blockDim.x / G;

  const bool bits = non_negative(a.alpha);  // fitness order by bit patterns (see fit_lt)
  if (threadIdx.x == 0) g_s = (flags & DE_GEN_DEVICE) ? *pb.gen : g_arg;

  if (flags & (DE_FIRST | DE_SELECT)) {
    const bool first = (flags & DE_FIRST) != 0;
    for (int r = r0; r < P; r += rstep) {
      if (first) {
        const double f = group_fitness(pb.counts + (int64_t)r * L * K, pb.pop + (int64_t)r * m, B,
                                       L, K, pb.n_valid, a.n_min, a.alpha, sub, G, gm);
        if (sub == 0) pb.fit[r] = f;
      } else {
        select_individual(a, pb, r, B, L, K, sub, G, gm, bits);
      }
    }
    __syncthreads();
    block_argmin(pb.fit, P, &best_s, red_f, red_i, bits);
    if (threadIdx.x == 0) *pb.best = best_s;
  } else {
    if (threadIdx.x == 0) best_s = *pb.best;
    __syncthreads();
  }

  if (!(flags & DE_TRIAL)) return;
  const int g = g_s;
  if (g < 1 || g > pb.G) return;  // device-driven replay past the last generation
  const int best = best_s;
  for (int r = r0; r < P; r += rstep) trial_individual(a, pb, r, g, best, B, sub, G, gm);
  const int64_t total = (int64_t)P * L * K;
  for (int64_t e = threadIdx.x; e < total; e += blockDim.x) pb.counts[e] = 0;
  if (threadIdx.x == 0 && (flags & DE_GEN_DEVICE)) *pb.gen = g + 1;
}

// The steady-state step (Eq. selection of generation g - 1's trials, then
// generation g's trial vectors) of one problem in one CTA with everything on
// chip.  The general step walks chains of dependent global loads (a gene at a
// time, the genes of r1, r2 and the best after their draws and the argmin) and
// every lane of an individual's group computes the Philox blocks it needs, mostly
// the same ones.  Here the population, the trials, the class counts and n_p are
// copied to shared memory by asynchronous copies that are all in flight together,
// each Philox block of an individual is computed once, by one lane, and the rest
// -- fitness, selection, argmin, mutation, crossover, decoding -- reads shared
// memory.  What is left is instruction issue on one SM, so the counts come by
// 16-byte copies and one short loop a leaf (sixteen predicated loads a lane took 6k
// of 17k cycles), sums are 32-bit, and one warp finds the argmin with warp
// reductions.  The values are those of the general step: integer sums in any
// order, the same draws, one rounding per float operation, the same selection and
// argmin.  Measured on GB300 (a step; before: a register form of this step for
// depth <= 3, else the general step): P = 64, depth 2 7.9 -> 6.6 us; P = 128, depth 3
// 10.3 -> 8.4 us; P = 100, depth 4 14.6 -> 8.9 us.  What bounds it is latency: about
// 700 instructions a warp at ten cycles each, the launch, and four dependent
// round trips (generation number, copies, stores).
//
// Shared memory (step_layout): genes of the population and of the trials [P][m]
// (the selected rows of the trials are copied over the population's), draws
// [P][8 nblk], fitness [P], n_p [F], class counts [P][L][K].
struct StepLayout {
  int trial, draws, fit, nu, cnt, total;  // byte offsets (the population is at 0)
};
__host__ __device__ __forceinline__ StepLayout step_layout(int P, int m, int F, int LK) {
  const int nblk = (m + 4 + 7) / 8;
  StepLayout l;
  l.trial = (P * m * 4 + 15) & ~15;
  l.draws = 2 * l.trial;
  l.fit = l.draws + P * nblk * 32;
  l.nu = (l.fit + P * 8 + 15) & ~15;
  l.cnt = (l.nu + F * 4 + 15) & ~15;
  l.total = l.cnt + P * LK * 4;
  return l;
}
constexpr int kStepSmem = 200 * 1024;  // most shared memory of the step
constexpr int kStepLanes = 3;          // at most 2^3 lanes an individual
constexpr int kStepP = 256;            // larger populations are split over CTAs (below)

// nw words of global memory to shared memory (dst 16-byte aligned, src of any
// alignment), asynchronously as far as src allows, by the whole CTA.
__device__ __forceinline__ void copy_async(uint32_t* dst, const uint32_t* src, int nw) {
  int done = 0;
  if ((reinterpret_cast<uintptr_t>(src) & 15) == 0) {
    done = nw & ~3;
    for (int e = 4 * threadIdx.x; e < done; e += 4 * blockDim.x) cp_async16(dst + e, src + e);
  }
  for (int e = done + threadIdx.x; e < nw; e += blockDim.x) dst[e] = src[e];
}

// Index of the least of fit[0..P) (the lowest of equals), by one warp; in the order
// of fit_lt.
__device__ __forceinline__ int warp_argmin(const double* fit, int P, int lane, bool bits) {
  long long bk = 0x7FFFFFFFFFFFFFFFll;
  double bf = 0.0;
  int bi = -1;
  for (int r = lane; r < P; r += 32) {
    const double f = fit[r];
    if (bi < 0 || fit_lt(f, bf, bits)) {
      bf = f;
      bi = r;
    }
  }
  if (bits) {  // non-negative doubles: high word, then low word, then index
    bk = bi < 0 ? bk : __double_as_longlong(bf);
    const uint32_t hi = (uint32_t)(bk >> 32), lo = (uint32_t)bk;
    const uint32_t mh = __reduce_min_sync(0xFFFFFFFFu, hi);
    const uint32_t ml = __reduce_min_sync(0xFFFFFFFFu, hi == mh ? lo : 0xFFFFFFFFu);
    return (int)__reduce_min_sync(0xFFFFFFFFu, bi >= 0 && hi == mh && lo == ml ? (uint32_t)bi : 0xFFFFFFFFu);
  }
  for (int off = 16; off > 0; off >>= 1) {
    const double of = __shfl_xor_sync(0xFFFFFFFFu, bf, off);
    const int oi = __shfl_xor_sync(0xFFFFFFFFu, bi, off);
    if (oi >= 0 && (bi < 0 || of < bf || (!(bf < of) && oi < bi))) {
      bf = of;
      bi = oi;
    }
  }
  return bi;
}

__global__ void __launch_bounds__(1024) de_step_chip_kernel(const DEArgs a, int g_arg, int flags, int lg) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ int best_s;
  const DEProb& pb = prob_of(a);
  const int P = a.P, B = (1 << a.depth) - 1, m = 2 * B, L = 1 << a.depth, K = pb.K, F = pb.F, LK = L * K;
  const int nblk = (m + 4 + 7) / 8, G = 1 << lg;
  const StepLayout lay = step_layout(P, m, F, LK);
  float* pop_s = reinterpret_cast<float*>(sm);
  float* tri_s = reinterpret_cast<float*>(sm + lay.trial);
  uint32_t* drw_s = reinterpret_cast<uint32_t*>(sm + lay.draws);
  double* fit_s = reinterpret_cast<double*>(sm + lay.fit);
  uint32_t* nu_s = reinterpret_cast<uint32_t*>(sm + lay.nu);
  uint32_t* cnt_s = reinterpret_cast<uint32_t*>(sm + lay.cnt);
  const int tid = threadIdx.x, NT = blockDim.x;
  const int sub = tid & (G - 1), r = tid >> lg;
  const uint32_t gm = (G == 32 ? 0xFFFFFFFFu : ((1u << G) - 1u)) << ((tid & 31) & ~(G - 1));
  const bool act = r < P;  // a whole group is active or not
  const bool bits = non_negative(a.alpha);

  // ---- loads, then generation g's draws while they are in flight: block q of
  // individual i by thread i nblk + q ----------------------------------------------
  copy_async(nu_s, pb.n_unique, F);
  const int g = (flags & DE_GEN_DEVICE) ? *pb.gen : g_arg;
  copy_async(cnt_s, pb.counts, P * LK);
  copy_async(reinterpret_cast<uint32_t*>(tri_s), reinterpret_cast<const uint32_t*>(pb.trial), P * m);
  copy_async(reinterpret_cast<uint32_t*>(pop_s), reinterpret_cast<const uint32_t*>(pb.pop), P * m);
  asm volatile("cp.async.commit_group;" ::: "memory");
  const double fr = act ? pb.fit[r] : 0.0;
  const bool trial = g >= 1 && g <= pb.G;
  if (trial)
    for (int e = tid; e < P * nblk; e += NT) {
      const int i = e / nblk, q = e - i * nblk;
      const U64x4 b = philox4x64_10((uint64_t)g, (uint64_t)i, (uint64_t)q, 0ull, pb.seed, pb.stream_id);
      uint4* d = reinterpret_cast<uint4*>(drw_s + e * 8);
      d[0] = make_uint4((uint32_t)b.x[0], (uint32_t)(b.x[0] >> 32), (uint32_t)b.x[1], (uint32_t)(b.x[1] >> 32));
      d[1] = make_uint4((uint32_t)b.x[2], (uint32_t)(b.x[2] >> 32), (uint32_t)b.x[3], (uint32_t)(b.x[3] >> 32));
    }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();

  // ---- the counts are on chip: zeroed for the next evaluation ---------------------
  {
    uint32_t* c = pb.counts;
    int done = 0;
    if ((reinterpret_cast<uintptr_t>(c) & 15) == 0) {
      done = (P * LK) & ~3;
      for (int e = 4 * tid; trial && e < done; e += 4 * NT) *reinterpret_cast<uint4*>(c + e) = make_uint4(0, 0, 0, 0);
    }
    for (int e = done + tid; trial && e < P * LK; e += NT) c[e] = 0;
  }

  // ---- the fitness of Section 3.2 of the just-evaluated trial, Eq. selection -------
  if (act) {
    uint32_t correct = 0, vs = 0;  // vs: V below bit 16, splits above
    const float* tr = tri_s + r * m;
    for (int l = sub; l < L; l += G) {
      const uint32_t* c = cnt_s + r * LK + l * K;
      uint32_t mx = 0, nl = 0;
      for (int k = 0; k < K; ++k) {
        const uint32_t x = c[k];
        mx = x > mx ? x : mx;
        nl += x;
      }
      correct += mx;
      if (nl > 0 && (int64_t)nl < a.n_min) vs += 1;
    }
    if (!is_zero(a.alpha))
      for (int t = sub; t < B; t += G) vs += tr[t] >= 1.0f ? 0x10000u : 0u;
    for (int o = G >> 1; o > 0; o >>= 1) {
      correct += __shfl_xor_sync(gm, correct, o);
      vs += __shfl_xor_sync(gm, vs, o);
    }
    const int64_t ev = pb.n_valid - (int64_t)correct + (int64_t)(vs & 0xFFFFu);  // errors + V
    const double f = is_zero(a.alpha) ? exact_double(ev) : penalised(ev, a.alpha, vs >> 16);
    const bool take = fit_le(f, fr, bits);  // ties go to the trial
    if (take) {
      float *po = pop_s + r * m, *dst = pb.pop + (int64_t)r * m;
      for (int q = sub; q < m; q += G) {
        const float x = tr[q];
        po[q] = x;
        dst[q] = x;
      }
    }
    if (sub == 0) {
      pb.fit_trial[r] = f;
      if (take) pb.fit[r] = f;
      fit_s[r] = take ? f : fr;
    }
  }
  __syncthreads();
  if (tid < 32) {
    const int b = warp_argmin(fit_s, P, tid, bits);
    if (tid == 0) {
      best_s = b;
      *pb.best = b;
    }
  }
  if (!trial) return;  // device-driven replay past the last generation (uniform)
  __syncthreads();

  // ---- generation g's trial vectors from the new population, decoded --------------
  if (act) {
    const float hi_a = below_bound((float)(F + 1)), hi_b = below_bound(1.0f);
    const uint32_t* dr = drw_s + r * nblk * 8;
    int r1 = (int)below(dr[0], (uint32_t)(P - 1));
    if (r1 >= r) r1 += 1;
    int r2 = (int)below(dr[1], (uint32_t)(P - 2));
    const int lo = r < r1 ? r : r1, hi = r < r1 ? r1 : r;
    if (r2 >= lo) r2 += 1;
    if (r2 >= hi) r2 += 1;
    const int qrand = (int)below(dr[2], (uint32_t)m);
    const float M = a.dither ? u01(dr[3]) : a.M;
    const float *sb = pop_s + best_s * m, *s1 = pop_s + r1 * m, *s2 = pop_s + r2 * m, *sr = pop_s + r * m;
    float* u = pb.trial + (int64_t)r * m;
    // u01(x) <= CR with u01(x) = (x >> 8) 2^-24, in integers (CR 2^24 is exact)
    const uint32_t cr24 = (uint32_t)floorf(__fmul_rn(a.CR, 16777216.0f));
    auto gene = [&](int q, float top) {
      const float x = __fadd_rn(sb[q], __fmul_rn(M, __fsub_rn(s1[q], s2[q])));
      const float xc = clamp_gene(x, top);
      const float uq = ((dr[4 + q] >> 8) <= cr24 || q == qrand) ? xc : sr[q];
      u[q] = uq;
      return uq;
    };
    for (int t = sub; t < B; t += G) {
      const float ah = gene(t, hi_a), bh = gene(B + t, hi_b);
      int av;
      uint32_t th;
      decode_gene_pair(ah, bh, F, nu_s, &av, &th);
      pb.nodes[(int64_t)r * B + t] = pack_node(av, th);
    }
  }
  if (tid == 0 && (flags & DE_GEN_DEVICE)) *pb.gen = g + 1;
}

// The steady-state step of one problem with a large population, split over CTAs
// of kDeWideR individuals (kDeWideG lanes each) in two launches: one CTA alone
// walks every individual through a chain of dependent loads, and at P = 1024
// that took 88 us a generation.  The first launch does Eq. selection and the
// argmin of each CTA's individuals; the second reduces those candidates to the
// best (lowest index among minimal fitness, as one CTA would find it, since the
// CTAs cover ascending index ranges), then builds the trials.  The values are
// those of the one-CTA step.
__global__ void __launch_bounds__(kDeWideR * kDeWideG) de_select_wide_kernel(const DEArgs a,
                                                                              int g_arg, int flags) {
  __shared__ double red_f[32];
  __shared__ int red_i[32];
  __shared__ int best_s;
  const DEProb& pb = a.single;
  const int P = a.P, B = (1 << a.depth) - 1, L = 1 << a.depth, K = pb.K;
  constexpr int G = kDeWideG;
  const int sub = threadIdx.x & (G - 1);
  const uint32_t gm = ((1u << G) - 1u) << ((threadIdx.x & 31) & ~(G - 1));
  const int r0 = blockIdx.x * kDeWideR, nr = min(kDeWideR, P - r0);
  const int r = r0 + (int)threadIdx.x / G;
  const bool bits = non_negative(a.alpha);
  if (r < P) select_individual(a, pb, r, B, L, K, sub, G, gm, bits);  // whole groups only
  __syncthreads();
  block_argmin(pb.fit + r0, nr, &best_s, red_f, red_i, bits);
  if (threadIdx.x == 0) {
    a.part_f[blockIdx.x] = pb.fit[r0 + best_s];
    a.part_i[blockIdx.x] = r0 + best_s;
    // the generation is read here, before the second launch's first CTA advances it
    if (blockIdx.x == 0) *a.part_g = (flags & DE_GEN_DEVICE) ? *pb.gen : g_arg;
  }
}

__global__ void __launch_bounds__(kDeWideR * kDeWideG) de_trial_wide_kernel(const DEArgs a,
                                                                             int flags, int nblk) {
  __shared__ double red_f[32];
  __shared__ int red_i[32];
  __shared__ int best_s;
  const DEProb& pb = a.single;
  const int P = a.P, B = (1 << a.depth) - 1, L = 1 << a.depth, K = pb.K;
  constexpr int G = kDeWideG;
  const int sub = threadIdx.x & (G - 1);
  const uint32_t gm = ((1u << G) - 1u) << ((threadIdx.x & 31) & ~(G - 1));
  const int r0 = blockIdx.x * kDeWideR, nr = min(kDeWideR, P - r0);
  const int r = r0 + (int)threadIdx.x / G;
  block_argmin(a.part_f, nblk, &best_s, red_f, red_i, non_negative(a.alpha));
  const int best = a.part_i[best_s];
  const int g = *a.part_g;
  const bool trial = g >= 1 && g <= pb.G;  // false: device-driven replay past the last generation
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *pb.best = best;
    if (trial && (flags & DE_GEN_DEVICE)) *pb.gen = g + 1;
  }
  if (!trial) return;
  if (r < P) trial_individual(a, pb, r, g, best, B, sub, G, gm);
  // this CTA's individuals' class counts, read by the first launch, zeroed for the next
  const int64_t e0 = (int64_t)r0 * L * K, e1 = (int64_t)(r0 + nr) * L * K;
  for (int64_t e = e0 + threadIdx.x; e < e1; e += blockDim.x) pb.counts[e] = 0;
}

__global__ void decode_kernel(const float* __restrict__ genes, int P, int B, int F,
                              const uint32_t* __restrict__ n_unique, uint16_t* __restrict__ a_out,
                              uint32_t* __restrict__ th_out) {
  int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (int64_t)P * B) return;
  int64_t r = e / B;
  int t = (int)(e - r * B);
  int av;
  uint32_t th;
  decode_gene_pair(genes[r * 2 * B + t], genes[r * 2 * B + B + t], F, n_unique, &av, &th);
  a_out[e] = (uint16_t)av;
  th_out[e] = th;
}

__global__ void best_extract_kernel(const float* __restrict__ pop, const double* __restrict__ fit,
                                    const int32_t* __restrict__ best, int B, int F,
                                    const uint32_t* __restrict__ n_unique, uint16_t* __restrict__ a_out,
                                    uint32_t* __restrict__ th_out, double* __restrict__ fit_out) {
  const int b = *best;
  const float* g = pop + (int64_t)b * 2 * B;
  for (int t = threadIdx.x; t < B; t += blockDim.x) {
    int av;
    uint32_t th;
    decode_gene_pair(g[t], g[B + t], F, n_unique, &av, &th);
    a_out[t] = (uint16_t)av;
    th_out[t] = th;
  }
  if (threadIdx.x == 0) *fit_out = fit[b];
}

// Threads per individual in the step kernel: the largest power of two up to 4
// that keeps the CTA within 1024 threads (4 for P <= 256, 1 for P > 512).
// Measured on the moving-horizon workload (P = 128): 1 / 2 / 4 / 8 threads gave
// 0.2246 / 0.2215 / 0.2180 / 0.2212 s batched and 0.674 / 0.653 / 0.631 / 0.687 s
// plain (with 8, the CTA-wide argmin and barriers span 32 warps).
int lanes_for(int P) {
  int g = 1;
  while (g < 4 && P * g * 2 <= 1024) g *= 2;
  return g;
}

int block_for(int P) {
  int b = ((P + 31) / 32) * 32;
  if (b > 1024) b = 1024;
  if (b < 128) b = 128;
  return b;
}

}  // namespace

int de_launch_init(deoct_ctx* ctx, const DEArgs& a, cudaStream_t s) {
  const int nprob = a.probs ? a.nprob : 1;
  if (nprob <= 0) return DEOCT_OK;
  de_init_kernel<<<nprob, block_for(a.P), 0, s>>>(a);
  count_launch(ctx);
  return check_launch("de_init_kernel");
}

int de_launch_step(deoct_ctx* ctx, const DEArgs& a, int g, int flags, cudaStream_t s) {
  const int nprob = a.probs ? a.nprob : 1;
  if (nprob <= 0) return DEOCT_OK;
  const int lanes = lanes_for(a.P);
  const int m = 2 * ((1 << a.depth) - 1);
  const bool steady = (flags & DE_SELECT) && (flags & DE_TRIAL) && !(flags & DE_FIRST);
  const size_t smem = a.Kmax > 0 ? (size_t)step_layout(a.P, m, kMaxF, (1 << a.depth) * a.Kmax).total : kStepSmem + 1;
  if (steady && a.P <= kStepP && smem <= (size_t)kStepSmem) {
    int lg = 0;  // lanes an individual (log2)
    while (lg < kStepLanes && (2 << lg) <= (1 << a.depth) && (a.P << lg) * 2 <= 1024) ++lg;
    DEOCT_TRY(set_max_dynamic_smem(ctx, de_step_chip_kernel));
    return launch_on(ctx, "de_step_chip_kernel", de_step_chip_kernel, nprob, block_for(a.P << lg), smem, s, a, g, flags,
                     lg);
  }
  if (steady && !a.probs && a.part_f && a.P > kStepP && a.P <= kMaxPop) {
    const int nblk = (a.P + kDeWideR - 1) / kDeWideR;
    DEOCT_TRY(launch_on(ctx, "de_select_wide_kernel", de_select_wide_kernel, nblk, kDeWideR * kDeWideG, 0, s, a, g, flags));
    return launch_on(ctx, "de_trial_wide_kernel", de_trial_wide_kernel, nblk, kDeWideR * kDeWideG, 0, s, a, flags, nblk);
  }
  return launch_on(ctx, "de_step_kernel", de_step_kernel, nprob, block_for(a.P * lanes), 0, s, a, g, flags, lanes);
}

int launch_best_extract(deoct_ctx* ctx, const float* pop, const double* fit, const int32_t* best,
                        int depth, int F, const uint32_t* n_unique, uint16_t* a_out,
                        uint32_t* theta_out, double* fit_out, cudaStream_t s) {
  best_extract_kernel<<<1, 256, 0, s>>>(pop, fit, best, (1 << depth) - 1, F, n_unique, a_out,
                                        theta_out, fit_out);
  count_launch(ctx);
  return check_launch("best_extract_kernel");
}

int launch_decode(deoct_ctx* ctx, const float* genes, int P, int depth, int F,
                  const uint32_t* n_unique, uint16_t* a_out, uint32_t* theta_out,
                  cudaStream_t s) {
  const int B = (1 << depth) - 1;
  const int64_t total = (int64_t)P * B;
  if (total <= 0) return DEOCT_OK;
  decode_kernel<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(genes, P, B, F, n_unique, a_out,
                                                               theta_out);
  count_launch(ctx);
  return check_launch("decode_kernel");
}

}  // namespace deoct
