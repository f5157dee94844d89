// encode.cu -- rank encoder (the threshold sets of Section 3.1 as dense ranks).
//
// For every feature p the samples' float32 values are sorted (segmented LSD
// radix sort on order-preserving key bits, sample index as payload); a sample's
// rank is the number of distinct values before it in sorted order, i.e. an
// exclusive scan of "value differs from its predecessor" flags, scattered back
// to the sample's column.  n_p is the number of flags.  -0.0 is folded into
// +0.0 before sorting; NaN is reported.
#include "internal.cuh"

namespace deoct {

namespace {

constexpr int kThreads = 256;
constexpr int kItems = 8;
constexpr int kTile = kThreads * kItems;  // keys per tile

__device__ __forceinline__ uint32_t orderable(float v) {
  if (v == 0.0f) v = 0.0f;  // -0.0 and +0.0 are one value
  uint32_t b = __float_as_uint(v);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float from_orderable(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k);
}

// block-wide exclusive scan of one value per thread (blockDim.x == kThreads)
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t x, uint32_t* warp_tot,
                                                         uint32_t* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t incl = x;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, off);
    if (lane >= off) incl += y;
  }
  if (lane == 31) warp_tot[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    uint32_t w = lane < kThreads / 32 ? warp_tot[lane] : 0u;
    uint32_t wi = w;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      uint32_t y = __shfl_up_sync(0xFFFFFFFFu, wi, off);
      if (lane >= off) wi += y;
    }
    if (lane < kThreads / 32) warp_tot[lane] = wi - w;
    if (lane == kThreads / 32 - 1 && total) *total = wi;
  }
  __syncthreads();
  uint32_t r = warp_tot[warp] + incl - x;
  __syncthreads();
  return r;
}

// X [n][F] -> keys [F][n] (orderable bits), `S` samples a block through shared
// memory (rows of an odd number of words: no bank conflicts down a column).
__global__ void __launch_bounds__(kThreads) keys_kernel(const float* __restrict__ X, int64_t n, int F, int S,
                                                       uint32_t* __restrict__ keys, int* status) {
  extern __shared__ float xs[];  // [S][F | 1]
  const int64_t i0 = (int64_t)blockIdx.x * S;
  const int ns = n - i0 < S ? (int)(n - i0) : S;
  const int ld = F | 1;
  const int dl = kThreads / F, df = kThreads - dl * F;
  int l = threadIdx.x / F, f = threadIdx.x - l * F;
  bool nan = false;
  for (int e = threadIdx.x; e < ns * F; e += kThreads) {
    const float v = X[i0 * F + e];
    nan |= isnan(v);
    xs[l * ld + f] = v;
    l += dl;
    f += df;
    if (f >= F) {
      f -= F;
      ++l;
    }
  }
  if (nan) atomicOr(status, ST_NAN);
  __syncthreads();
  const int lane = threadIdx.x & 31;
  for (int g = threadIdx.x >> 5; g < F; g += kThreads / 32)
    for (int a = lane; a < ns; a += 32) keys[(int64_t)g * n + i0 + a] = orderable(xs[a * ld + g]);
}

// ---------------------------------------------------------------------------
// segmented LSD radix sort, one sweep a pass (the published one-sweep form: Adinets and
// Merrill, 2022, over Merrill and Garland's decoupled look-back, 2016)
// ---------------------------------------------------------------------------
// The digit counts of all passes come from one read of the keys (rs_hist_kernel).
// A pass then reads each key and value once and writes each once: a tile of 4096
// keys finds the positions of its digits by decoupled look-back (each tile
// publishes its digit counts, then, once the tiles before it are known, their
// prefix), orders its keys by digit in shared memory and writes the runs.  The
// former pass (a histogram read, a column scan and a scatter of single keys in
// three launches) took 197 + 49 + 823 us at n = 1e7, F = 10; a sweep takes 510 to 530
// (3.1 TB/s: ranking the keys, 50 instructions each, and the dependent phases of a
// tile bound it), the one histogram 205.  Look-backs that walked one word at a time
// over tiles of one segment at a time took 150 us more a sweep; 12 or 20 keys a
// thread were 1 to 5% slower.  The encoder as a whole: 5.83 -> 3.44 ms at n = 1e7, F = 10,
// 586 -> 353 us at n = 2e5, F = 33; its scatter of ranks (840 us, single words to random
// places) is the largest part left.
constexpr int kRsThreads = 256, kRsWarps = kRsThreads / 32;
constexpr int kRsItems = 16;
constexpr int kRsTile = kRsThreads * kRsItems;
constexpr int kRsHistTiles = 4;   // tiles a histogram block reads
// Tile status word: the count in the low 25 bits, above it 2 pass + 1 (the tile's
// own count) or 2 pass + 2 (with all tiles before it); any other value is not ready,
// so one clearing serves all passes of a sort.
constexpr uint32_t kRsCountMask = (1u << 25) - 1u;
constexpr int kRsPolls = 1 << 20;  // bound of a look-back wait
constexpr int kRsLook = 4;         // status words a look-back reads at once

// digit counts of up to four passes: tot[f][pass][digit] (zeroed before)
__global__ void __launch_bounds__(kRsThreads) rs_hist_kernel(const uint32_t* __restrict__ keys, int64_t n, int npass,
                                                            uint32_t* __restrict__ tot) {
  __shared__ uint32_t h[4][256];
  const int f = blockIdx.y;
  for (int p = 0; p < npass; ++p) h[p][threadIdx.x] = 0;
  __syncthreads();
  const uint32_t* k = keys + (int64_t)f * n;
  const int64_t base = (int64_t)blockIdx.x * kRsTile * kRsHistTiles;
#pragma unroll 4
  for (int it = 0; it < kRsItems * kRsHistTiles; ++it) {
    const int64_t j = base + it * kRsThreads + threadIdx.x;
    if (j < n) {
      const uint32_t x = k[j];
      for (int p = 0; p < npass; ++p) atomicAdd(&h[p][(x >> (8 * p)) & 255u], 1u);
    }
  }
  __syncthreads();
  for (int p = 0; p < npass; ++p) {
    const uint32_t c = h[p][threadIdx.x];
    if (c) atomicAdd(&tot[((int64_t)f * 4 + p) * 256 + threadIdx.x], c);
  }
}

// One pass over every segment.  FIRST: the values are the keys' places (vin unused).
template <bool FIRST>
__global__ void __launch_bounds__(kRsThreads, 4) rs_sweep_kernel(
    const uint32_t* __restrict__ kin, const uint32_t* __restrict__ vin, uint32_t* __restrict__ kout,
    uint32_t* __restrict__ vout, int64_t n, int F, int pass, int ntiles, const uint32_t* __restrict__ tot,
    uint32_t* __restrict__ state, uint32_t* __restrict__ ticket, int* status) {
  __shared__ uint32_t buf[kRsTile];            // keys, then values, in digit order
  __shared__ uint32_t wcnt[kRsWarps][256];     // digit counts of a warp, then of the warps before it
  __shared__ uint32_t gofs[256], wt[kRsThreads / 32];
  __shared__ uint32_t s_tile;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) s_tile = atomicAdd(ticket, 1u);  // tiles start in order: those before this one run or ran
#pragma unroll
  for (int w = 0; w < kRsWarps; ++w) wcnt[w][tid] = 0;
  __syncthreads();
  // the segments' tiles interleaved: fewer tiles of one segment in flight, shorter look-backs
  const int tile = (int)(s_tile / (uint32_t)F), f = (int)(s_tile - (uint32_t)tile * (uint32_t)F);
  const int shift = 8 * pass;
  const int64_t base = (int64_t)tile * kRsTile;
  const int nv = n - base < kRsTile ? (int)(n - base) : kRsTile;
  const uint32_t* k = kin + (int64_t)f * n + base;
  // a warp's keys are consecutive; past the end: the largest key, after every other
  const int j0 = warp * (32 * kRsItems) + lane;
  uint32_t key[kRsItems];
#pragma unroll
  for (int it = 0; it < kRsItems; ++it) key[it] = j0 + it * 32 < nv ? k[j0 + it * 32] : 0xFFFFFFFFu;
  uint32_t rank[kRsItems];  // place among the warp's keys of the same digit
  const uint32_t lt = (1u << lane) - 1u;
#pragma unroll
  for (int it = 0; it < kRsItems; ++it) {
    const uint32_t d = (key[it] >> shift) & 255u;
    // lanes of the same digit by its eight ballots (a match instruction was level at n =
    // 1e7 and 15% slower at n = 2e5)
    uint32_t peers = 0xFFFFFFFFu;
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      const bool on = (d >> b) & 1u;
      const uint32_t v = __ballot_sync(0xFFFFFFFFu, on);
      peers &= on ? v : ~v;
    }
    const uint32_t before = wcnt[warp][d];
    rank[it] = before + __popc(peers & lt);
    __syncwarp();
    if ((peers & lt) == 0) wcnt[warp][d] = before + __popc(peers);
    __syncwarp();
  }
  __syncthreads();
  {  // thread d: digit d
    uint32_t c = 0;
#pragma unroll
    for (int w = 0; w < kRsWarps; ++w) {
      const uint32_t x = wcnt[w][tid];
      wcnt[w][tid] = c;
      c += x;
    }
    uint32_t* st = state + ((int64_t)f * ntiles + tile) * 256 + tid;
    const uint32_t own = (uint32_t)(2 * pass + 1) << 25, all = (uint32_t)(2 * pass + 2) << 25;
    if (tile > 0) *reinterpret_cast<volatile uint32_t*>(st) = own | c;
    const uint32_t first = block_exclusive_scan(tot[((int64_t)f * 4 + pass) * 256 + tid], wt, nullptr);
    const uint32_t local = block_exclusive_scan(c, wt, nullptr);
    uint32_t prev = 0;  // keys of this digit in the tiles before
    for (int t = tile - 1, polls = 0; t >= 0;) {
      uint32_t x[kRsLook];  // four status words in flight
#pragma unroll
      for (int u = 0; u < kRsLook; ++u)
        x[u] = *reinterpret_cast<volatile uint32_t*>(st - (int64_t)(tile - max(t - u, 0)) * 256);
      bool done = false;
      int used = 0;
#pragma unroll
      for (int u = 0; u < kRsLook; ++u) {
        const uint32_t fl = x[u] & ~kRsCountMask;
        if (!done && used == u && t - u >= 0 && (fl == all || fl == own)) {
          prev += x[u] & kRsCountMask;
          used = u + 1;
          done = fl == all;
        }
      }
      t -= used;
      if (done) break;
      if (used) {
        polls = 0;
      } else if (++polls >= kRsPolls) {
        atomicOr(status, ST_TIMEOUT);
        break;
      }
    }
    *reinterpret_cast<volatile uint32_t*>(st) = all | (prev + c);
    gofs[tid] = first + prev - local;  // global place of a key = gofs[digit] + place in the tile
#pragma unroll
    for (int w = 0; w < kRsWarps; ++w) wcnt[w][tid] += local;
  }
  __syncthreads();
#pragma unroll
  for (int it = 0; it < kRsItems; ++it) {
    rank[it] += wcnt[warp][(key[it] >> shift) & 255u];
    buf[rank[it]] = key[it];
  }
  __syncthreads();
  uint32_t pos[kRsItems];
  uint32_t* ko = kout + (int64_t)f * n;
  uint32_t* vo = vout + (int64_t)f * n;
#pragma unroll
  for (int it = 0; it < kRsItems; ++it) {
    const int j = it * kRsThreads + tid;
    const uint32_t x = buf[j];
    pos[it] = gofs[(x >> shift) & 255u] + (uint32_t)j;
    if (j < nv && pos[it] < n) ko[pos[it]] = x;  // (pos < n unless a wait ran out)
  }
  __syncthreads();
  const uint32_t* v = vin + (int64_t)f * n + base;
#pragma unroll
  for (int it = 0; it < kRsItems; ++it) {
    const int j = j0 + it * 32;
    buf[rank[it]] = FIRST ? (uint32_t)(base + j) : (j < nv ? v[j] : 0u);
  }
  __syncthreads();
#pragma unroll
  for (int it = 0; it < kRsItems; ++it) {
    const int j = it * kRsThreads + tid;
    if (j < nv && pos[it] < n) vo[pos[it]] = buf[j];
  }
}

// "New value" flags of a warp's 256 consecutive sorted keys, 32 at a time: bit l of
// `flags` says that key j + l differs from the one before it (or is the first).
__device__ __forceinline__ uint32_t new_values(const uint32_t* k, int64_t j, int64_t n, int lane, uint32_t* key) {
  const bool in = j + lane < n;
  const uint32_t x = in ? k[j + lane] : 0u;
  uint32_t before = __shfl_up_sync(0xFFFFFFFFu, x, 1);
  if (lane == 0) before = j > 0 && in ? k[j - 1] : ~x;
  *key = x;
  return __ballot_sync(0xFFFFFFFFu, in && x != before);
}

// number of flags per tile of sorted keys
__global__ void __launch_bounds__(kThreads) rank_count_kernel(const uint32_t* __restrict__ keys,
                                                             int64_t n, int ntiles,
                                                             uint32_t* __restrict__ C) {
  __shared__ uint32_t total;
  const int f = blockIdx.y, tile = blockIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) total = 0;
  __syncthreads();
  const uint32_t* k = keys + (int64_t)f * n;
  const int64_t j0 = (int64_t)tile * kTile + warp * (32 * kItems);
  uint32_t cnt = 0;
#pragma unroll
  for (int it = 0; it < kItems; ++it) {
    uint32_t x;
    cnt += __popc(new_values(k, j0 + it * 32, n, lane, &x));
  }
  if (lane == 0) atomicAdd(&total, cnt);
  __syncthreads();
  if (threadIdx.x == 0) C[(int64_t)f * ntiles + tile] = total;
}

// exclusive scan of tile flag counts per feature; n_unique = total
__global__ void __launch_bounds__(kThreads) rank_scan_kernel(uint32_t* __restrict__ C, int ntiles,
                                                            uint32_t* __restrict__ n_unique) {
  __shared__ uint32_t wt[kThreads / 32];
  __shared__ uint32_t chunk_total;
  const int f = blockIdx.x;
  uint32_t* c = C + (int64_t)f * ntiles;
  uint32_t carry = 0;
  for (int c0 = 0; c0 < ntiles; c0 += kThreads) {
    int j = c0 + threadIdx.x;
    uint32_t x = j < ntiles ? c[j] : 0u;
    uint32_t ex = block_exclusive_scan(x, wt, &chunk_total);
    if (j < ntiles) c[j] = carry + ex;
    carry += chunk_total;
    __syncthreads();
  }
  if (threadIdx.x == 0) n_unique[f] = carry;
}

template <typename RT>
__global__ void __launch_bounds__(kThreads) rank_scatter_kernel(
    const uint32_t* __restrict__ keys, const uint32_t* __restrict__ vals, int64_t n, int ntiles,
    const uint32_t* __restrict__ C, RT* __restrict__ ranks, int64_t ld, float* __restrict__ uniq) {
  __shared__ uint32_t wt[kThreads / 32];
  const int f = blockIdx.y, tile = blockIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t* k = keys + (int64_t)f * n;
  const uint32_t* v = vals + (int64_t)f * n;
  const int64_t j0 = (int64_t)tile * kTile + warp * (32 * kItems);
  uint32_t flags[kItems], key[kItems], val[kItems], cnt = 0;
#pragma unroll
  for (int it = 0; it < kItems; ++it) {
    flags[it] = new_values(k, j0 + it * 32, n, lane, &key[it]);
    val[it] = j0 + it * 32 + lane < n ? v[j0 + it * 32 + lane] : 0u;
    cnt += __popc(flags[it]);
  }
  if (lane == 0) wt[warp] = cnt;
  __syncthreads();
  uint32_t r = C[(int64_t)f * ntiles + tile];  // values before the tile, then before the 32 keys
  for (int w = 0; w < warp; ++w) r += wt[w];
  RT* out = ranks + (int64_t)f * ld;
  const uint32_t le = 0xFFFFFFFFu >> (31 - lane);
#pragma unroll
  for (int it = 0; it < kItems; ++it) {
    const uint32_t mine = r + __popc(flags[it] & le) - 1u;
    if (j0 + it * 32 + lane < n) {
      if (val[it] < n) out[val[it]] = (RT)mine;  // (a place below n unless a wait of the sort ran out)
      if (uniq && ((flags[it] >> lane) & 1u)) uniq[(int64_t)f * ld + mine] = from_orderable(key[it]);
    }
    r += __popc(flags[it]);
  }
}

}  // namespace

// places: the values are the keys' places 0 .. n - 1 in their segment (v0 is then only
// the buffer of later passes)
static int sort_segments(deoct_ctx* ctx, uint32_t* k0, uint32_t* v0, bool places, uint32_t* k1, uint32_t* v1,
                         int64_t n, int F, int bits, uint32_t** keys_out, uint32_t** vals_out, cudaStream_t s) {
  const int ntiles = (int)((n + kRsTile - 1) / kRsTile);
  const int npass = (bits + 7) / 8;
  uint32_t *state = nullptr, *tot = nullptr;
  const size_t sbytes = sizeof(uint32_t) * (size_t)F * 256 * ntiles;
  const size_t tbytes = sizeof(uint32_t) * (size_t)F * 1024 + 64;
  DEOCT_TRY(scratch_get(ctx, SL_ENC_HIST, sbytes, (void**)&state));
  DEOCT_TRY(scratch_get(ctx, SL_ENC_TOT, tbytes, (void**)&tot));
  uint32_t* ticket = tot + (size_t)F * 1024;  // one per pass
  DEOCT_CUDA_TRY(cudaMemsetAsync(state, 0, sbytes, s));
  DEOCT_CUDA_TRY(cudaMemsetAsync(tot, 0, tbytes, s));
  const int64_t per = (int64_t)kRsTile * kRsHistTiles;
  rs_hist_kernel<<<dim3((unsigned)((n + per - 1) / per), F), kRsThreads, 0, s>>>(k0, n, npass, tot);
  count_launch(ctx);
  DEOCT_TRY(check_launch("rs_hist_kernel"));
  uint32_t *ki = k0, *vi = v0, *ko = k1, *vo = v1;
  for (int p = 0; p < npass; ++p) {
    const unsigned grid = (unsigned)ntiles * (unsigned)F;
    if (p == 0 && places)
      rs_sweep_kernel<true><<<grid, kRsThreads, 0, s>>>(ki, vi, ko, vo, n, F, p, ntiles, tot, state, ticket + p,
                                                       ctx->d_status);
    else
      rs_sweep_kernel<false><<<grid, kRsThreads, 0, s>>>(ki, vi, ko, vo, n, F, p, ntiles, tot, state, ticket + p,
                                                        ctx->d_status);
    count_launch(ctx);
    DEOCT_TRY(check_launch("rs_sweep_kernel"));
    uint32_t* t;
    t = ki; ki = ko; ko = t;
    t = vi; vi = vo; vo = t;
  }
  *keys_out = ki;
  *vals_out = vi;
  return DEOCT_OK;
}

int radix_sort_segments(deoct_ctx* ctx, uint32_t* k0, uint32_t* v0, uint32_t* k1, uint32_t* v1,
                        int64_t n, int F, int bits, uint32_t** keys_out, uint32_t** vals_out,
                        cudaStream_t s) {
  return sort_segments(ctx, k0, v0, false, k1, v1, n, F, bits, keys_out, vals_out, s);
}

int encode_run(deoct_ctx* ctx, const float* X, int64_t n, int F, int W, void* ranks_out,
               int64_t ld, uint32_t* n_unique_out, float* unique_out, cudaStream_t s, int* W_used) {
  const size_t elems = (size_t)n * F;
  uint32_t *k0, *k1, *v0, *v1, *C;
  DEOCT_TRY(scratch_get(ctx, SL_ENC_K0, elems * 4, (void**)&k0));
  DEOCT_TRY(scratch_get(ctx, SL_ENC_K1, elems * 4, (void**)&k1));
  DEOCT_TRY(scratch_get(ctx, SL_ENC_V0, elems * 4, (void**)&v0));
  DEOCT_TRY(scratch_get(ctx, SL_ENC_V1, elems * 4, (void**)&v1));
  const int ntiles = (int)((n + kTile - 1) / kTile);
  DEOCT_TRY(scratch_get(ctx, SL_ENC_TILE, sizeof(uint32_t) * (size_t)F * ntiles, (void**)&C));

  const int S = F <= 40 ? 256 : F <= 160 ? 64 : 32;  // at most 41 KB of shared memory
  keys_kernel<<<(unsigned)((n + S - 1) / S), kThreads, sizeof(float) * (size_t)S * (F | 1), s>>>(X, n, F, S, k0,
                                                                                                ctx->d_status);
  count_launch(ctx);
  DEOCT_TRY(check_launch("keys_kernel"));
  uint32_t *ks, *vs;
  DEOCT_TRY(sort_segments(ctx, k0, v0, true, k1, v1, n, F, 32, &ks, &vs, s));
  dim3 g(ntiles, F);
  rank_count_kernel<<<g, kThreads, 0, s>>>(ks, n, ntiles, C);
  rank_scan_kernel<<<F, kThreads, 0, s>>>(C, ntiles, n_unique_out);
  if (W == 0) {
    // automatic width: n_p is known once the flags are scanned, before any rank is written
    DEOCT_TRY(check_launch("rank count / scan kernels"));
    uint32_t* h = nullptr;
    DEOCT_TRY(pinned_get(ctx, sizeof(uint32_t) * F, (void**)&h));
    DEOCT_CUDA_TRY(cudaMemcpyAsync(h, n_unique_out, sizeof(uint32_t) * F, cudaMemcpyDeviceToHost, s));
    DEOCT_CUDA_TRY(cudaStreamSynchronize(s));
    uint32_t mx = 0;
    for (int f = 0; f < F; ++f) mx = h[f] > mx ? h[f] : mx;
    W = mx <= 65536u ? 2 : 4;
  }
  if (W_used) *W_used = W;
  if (W == 2)
    rank_scatter_kernel<uint16_t><<<g, kThreads, 0, s>>>(ks, vs, n, ntiles, C,
                                                        static_cast<uint16_t*>(ranks_out), ld,
                                                        unique_out);
  else
    rank_scatter_kernel<uint32_t><<<g, kThreads, 0, s>>>(ks, vs, n, ntiles, C,
                                                        static_cast<uint32_t*>(ranks_out), ld,
                                                        unique_out);
  count_launch(ctx, 3);
  return check_launch("rank kernels");
}

}  // namespace deoct
