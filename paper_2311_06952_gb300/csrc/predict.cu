// predict.cu -- a fitted tree applied to raw feature values (unseen samples).
//
// A rank threshold theta of feature p is the threshold set entry beta_{p,
// theta+1} of Section 3.1 in raw units: the midpoint of the theta-th and
// (theta+1)-th smallest distinct training values (1-based), computed in double
// (exact for float32 inputs); theta = 0 is beta_{p,1} = 0 after min-max
// scaling, i.e. the smallest training value.  On training samples "x < b"
// then routes exactly like "rank < theta".  Many rows of deep trees go through
// shared-memory tiles (predict_tile_kernel), others are walked a thread a row.
#include <algorithm>

#include "internal.cuh"

namespace deoct {
namespace {

__global__ void split_values_kernel(const float* __restrict__ unique, int64_t ld,
                                    const uint16_t* __restrict__ a, const uint32_t* __restrict__ theta,
                                    int B, double* __restrict__ b_out) {
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= B) return;
  const int av = a[t];
  if (av == 0) {
    b_out[t] = 0.0;  // unused: a_t = 0 sends every sample right
    return;
  }
  const float* u = unique + (int64_t)(av - 1) * ld;
  const uint32_t th = theta[t];
  b_out[t] = th == 0 ? (double)u[0] : __dmul_rn(__dadd_rn((double)u[th - 1], (double)u[th]), 0.5);
}

__global__ void predict_kernel(const float* __restrict__ X, int64_t m, int F,
                               const uint16_t* __restrict__ a, const double* __restrict__ b, int depth,
                               const uint8_t* __restrict__ leaf_class, const uint8_t* __restrict__ y,
                               uint8_t* __restrict__ pred, unsigned long long* __restrict__ correct) {
  extern __shared__ unsigned char sm[];
  const int B = (1 << depth) - 1, L = 1 << depth;
  double* bs = reinterpret_cast<double*>(sm);
  uint16_t* as = reinterpret_cast<uint16_t*>(bs + B);
  uint8_t* cs = reinterpret_cast<uint8_t*>(as + B);
  for (int t = threadIdx.x; t < B; t += blockDim.x) {
    bs[t] = b[t];
    as[t] = a[t];
  }
  for (int l = threadIdx.x; l < L; l += blockDim.x) cs[l] = leaf_class[l];
  __syncthreads();
  unsigned long long ok = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m;
       i += (int64_t)gridDim.x * blockDim.x) {
    int t = 1;
    while (t <= B) {
      const int p = as[t - 1];
      const bool left = p != 0 && p <= F && (double)X[i * F + (p - 1)] < bs[t - 1];
      t = left ? 2 * t : 2 * t + 1;
    }
    const uint8_t c = cs[t - L];
    if (pred) pred[i] = c;
    if (y) ok += (y[i] == c) ? 1ull : 0ull;
  }
  if (correct) {
    for (int off = 16; off > 0; off >>= 1) ok += __shfl_down_sync(0xFFFFFFFFu, ok, off);
    if ((threadIdx.x & 31) == 0 && ok) atomicAdd(correct, ok);
  }
}

// The same over tiles of S consecutive rows, which are one contiguous piece of X:
// bulk copies bring them into a ring of kTileStages zones in shared memory while
// earlier tiles are walked there.  In the kernel above a thread walks its row in
// global memory, `depth` dependent reads of which most miss (a row spans several
// sectors); here HBM sets the pace.  A threshold b becomes the least float not
// below it: x < b holds for a float x exactly when x is less than that float, so no
// FP64 comparison is left.
constexpr int kTileStages = 3, kTileThreads = 256;
constexpr int kTileBytes = 32 * 1024;  // most bytes of a zone

__global__ void __launch_bounds__(kTileThreads) predict_tile_kernel(
    const float* __restrict__ X, int64_t m, int F, int S, const uint16_t* __restrict__ a,
    const double* __restrict__ b, int depth, const uint8_t* __restrict__ leaf_class,
    const uint8_t* __restrict__ y, uint8_t* __restrict__ pred, unsigned long long* __restrict__ correct,
    int* status) {
  extern __shared__ __align__(128) unsigned char sm[];
  __shared__ __align__(8) uint64_t full[kTileStages];
  const int B = (1 << depth) - 1, L = 1 << depth;
  const uint32_t zone = (uint32_t)S * (uint32_t)F * 4u;  // a multiple of 16 (S of 32)
  uint2* nodes = reinterpret_cast<uint2*>(sm + (size_t)kTileStages * zone);  // {column, threshold}
  uint8_t* cs = reinterpret_cast<uint8_t*>(nodes + B);
  const int tid = threadIdx.x;
  const int64_t tiles = (m + S - 1) / S;
  auto issue = [&](int64_t t, int z) {  // thread 0: whole 16-byte pieces; the rest by plain loads
    const int64_t r0 = t * S;
    const int64_t left = (m - r0) * F * 4;
    const uint32_t bytes = (left < (int64_t)zone ? (uint32_t)left : zone) & ~15u;
    fence_proxy_async_smem();
    mbar_arrive_expect_tx(&full[z], bytes);
    if (bytes) bulk_g2s(sm + (size_t)z * zone, X + r0 * F, bytes, &full[z]);
  };
  if (tid == 0) {
    for (int z = 0; z < kTileStages; ++z) mbar_init(&full[z], 1);
    fence_mbar_init();
    for (int z = 0; z < kTileStages; ++z) {
      const int64_t t = blockIdx.x + (int64_t)z * gridDim.x;
      if (t < tiles) issue(t, z);
    }
  }
  for (int t = tid; t < B; t += kTileThreads) {
    const int p = a[t];
    // no split (or a feature past F): right, as nothing is below -inf
    nodes[t] = p != 0 && p <= F ? make_uint2((uint32_t)(p - 1), __float_as_uint(__double2float_ru(b[t])))
                                : make_uint2(0u, 0xFF800000u);
  }
  for (int l = tid; l < L; l += kTileThreads) cs[l] = leaf_class[l];
  __syncthreads();
  unsigned long long ok = 0;
  int z = 0;
  uint32_t ph = 0;
  for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
    // Ran out for a lane: recorded, one more bounded wait for copies in flight.  A warp
    // leaves as a whole: its lanes meet again in the sum below.
    if (__any_sync(0xFFFFFFFFu, !mbar_wait_bounded(&full[z], ph, status))) {
      mbar_wait_bounded(&full[z], ph, status);
      break;
    }
    const int64_t r0 = t * S;
    const int rows = m - r0 < S ? (int)(m - r0) : S;
    float* xt = reinterpret_cast<float*>(sm + (size_t)z * zone);
    const int have = rows == S ? S * F : rows * F & ~3;  // floats that landed (16-byte pieces)
    if (have < rows * F) {  // the last tile's tail
      for (int e = have + tid; e < rows * F; e += kTileThreads) xt[e] = X[r0 * F + e];
      __syncthreads();
    }
    for (int r = tid; r < rows; r += kTileThreads) {
      const float* x = xt + r * F;
      int n = 1;
      for (int d = 0; d < depth; ++d) {
        const uint2 nd = nodes[n - 1];
        n = 2 * n + (x[nd.x] < __uint_as_float(nd.y) ? 0 : 1);
      }
      const uint8_t c = cs[n - L];
      if (pred) pred[r0 + r] = c;
      if (y) ok += (y[r0 + r] == c) ? 1ull : 0ull;
    }
    __syncthreads();  // the zone is free
    if (tid == 0) {
      const int64_t nx = t + (int64_t)kTileStages * gridDim.x;
      if (nx < tiles) issue(nx, z);
    }
    if (++z == kTileStages) {
      z = 0;
      ph ^= 1u;
    }
  }
  if (correct) {
    for (int off = 16; off > 0; off >>= 1) ok += __shfl_down_sync(0xFFFFFFFFu, ok, off);
    if ((tid & 31) == 0 && ok) atomicAdd(correct, ok);
  }
}

}  // namespace

int launch_split_values(deoct_ctx* ctx, const float* unique, int64_t ld, const uint16_t* a,
                        const uint32_t* theta, int B, double* b_out, cudaStream_t s) {
  split_values_kernel<<<(B + 127) / 128, 128, 0, s>>>(unique, ld, a, theta, B, b_out);
  count_launch(ctx);
  return check_launch("split_values_kernel");
}

int launch_predict(deoct_ctx* ctx, const float* X, int64_t m, int F, const uint16_t* a,
                   const double* b, int depth, const uint8_t* leaf_class, const uint8_t* y,
                   uint8_t* pred_out, unsigned long long* correct_out, cudaStream_t s) {
  if (correct_out) DEOCT_CUDA_TRY(cudaMemsetAsync(correct_out, 0, sizeof(unsigned long long), s));
  if (m == 0) return DEOCT_OK;
  const int B = (1 << depth) - 1, L = 1 << depth;
  // The tiles read whole rows, the row walk only the sectors (8 floats) on its path:
  // tiles where a path touches most of a row.  GB300, device time in us with the walk /
  // with tiles, 5.3M rows: F = 16, depth 4 100 / 83; F = 28, depth 4 124 / 101, depth 8
  // 191 / 114; F = 33, depth 5 149 / 119, depth 6 160 / 123; F = 40, depth 5 165 / 144; F =
  // 48, depth 3 146 / 160, depth 6 198 / 180; 1.2M rows of 60, depth 8 67 / 59, depth 3 53 /
  // 53; 7e4 rows level.
  if (m >= 65536 && depth >= 4 && 8 * depth >= F && reinterpret_cast<uintptr_t>(X) % 16 == 0) {
    // a row per thread, or two: with powers of two (128 rows for F = 33 to 64) half the
    // threads had no row, and F = 33, depth 5 took 159 us against the walk's 149
    const int S = F <= 16 ? 512 : std::min(256, kTileBytes / (F * 4) / 32 * 32);
    const size_t smem = (size_t)kTileStages * S * F * 4 + (size_t)B * 8 + (size_t)L;
    DEOCT_TRY(set_max_dynamic_smem(ctx, predict_tile_kernel));
    const int grid = (int)std::min<int64_t>((m + S - 1) / S, (int64_t)ctx->num_sms * 2);
    predict_tile_kernel<<<grid, kTileThreads, smem, s>>>(X, m, F, S, a, b, depth, leaf_class, y, pred_out, correct_out,
                                                        ctx->d_status);
    count_launch(ctx);
    return check_launch("predict_tile_kernel");
  }
  const size_t smem = (size_t)B * 8 + (size_t)B * 2 + (size_t)L;
  DEOCT_TRY(set_max_dynamic_smem(ctx, predict_kernel));
  const int grid = (int)std::min<int64_t>((m + 255) / 256, (int64_t)ctx->num_sms * 8);
  predict_kernel<<<grid, 256, smem, s>>>(X, m, F, a, b, depth, leaf_class, y, pred_out, correct_out);
  count_launch(ctx);
  return check_launch("predict_kernel");
}

}  // namespace deoct
