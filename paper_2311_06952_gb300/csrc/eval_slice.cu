// eval_slice.cu -- the bit-sliced evaluator's host side (which launches it
// takes, their shapes) and planes_kernel, which writes the bit planes and class
// rows of a fit's samples to memory once (see eval_slice.cuh).
#include "eval_slice.cuh"

namespace deoct {
namespace slc {
namespace {

struct PlaneArgs {
  EvalProb single;
  const EvalProb* probs;  // nullptr: `single`
  int nprob;
  int Fmax;
  int64_t tiles;          // of all problems
  int* status;
};

// One warp per (tile, feature), and one per tile for the class rows.
template <int W>
__global__ void __launch_bounds__(256) planes_kernel(const PlaneArgs a) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t tasks = a.tiles * (a.Fmax + 1);
  for (int64_t task = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp; task < tasks;
       task += (int64_t)gridDim.x * (blockDim.x >> 5)) {
    const int64_t gt = task / (a.Fmax + 1);
    const int f = (int)(task - gt * (a.Fmax + 1));
    const EvalProb* pp = &a.single;
    if (a.probs) {
      int lo = 0, hi = a.nprob - 1;  // last problem with ptile0 <= gt
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (a.probs[mid].ptile0 <= gt) lo = mid; else hi = mid - 1;
      }
      pp = a.probs + lo;
    }
    const EvalProb& P = *pp;
    if (f > P.F) continue;
    const int64_t tile = gt - P.ptile0;
    const TileSpan t = tile_span(P, tile);
    uint32_t* blk = const_cast<uint32_t*>(P.planes) + (size_t)tile * slice_rows(P.F, P.K, P.nb) * 32;
    if (f == P.F) {  // class rows
      uint32_t* y = blk + (size_t)P.F * P.nb * 32;
      const uint32_t c = class_rows(P, t, lane, a.status, [&](int k, uint32_t v) { y[k * 32 + lane] = v; });
      if (lane == 0) y[(P.K + 1) * 32] = c;
      continue;
    }
    const int nb = P.nb;
    uint32_t x[16], h[16];
    RawWords<W> v;
    load_raw<W>(P, t, f, lane, a.status, v);
    raw_planes<W>(v, nb, x, h);
    uint32_t* out = blk + (size_t)f * P.nb * 32 + lane;
#pragma unroll
    for (int b = 0; b < 16; ++b)
      if (b < nb) out[b * 32] = x[b];
    if (W == 4) {
#pragma unroll
      for (int b = 0; b < 8; ++b)
        if (16 + b < nb) out[(16 + b) * 32] = h[b];
    } else if (nb > 16) {
      out[16 * 32] = 0u;
    }
  }
}

}  // namespace

int64_t slice_tiles(int64_t count) { return (count + kTile - 1) / kTile; }

size_t slice_plane_bytes(int64_t tiles, int F, int K, int nb) {
  return (size_t)tiles * slice_rows(F, K, nb) * 128;
}

// Rank bits that hold every theta < max_nu (the largest n_p).
int slice_bits(int W, uint32_t max_nu) {
  uint32_t mx = max_nu > 0 ? max_nu - 1 : 0;
  if (W == 2 && mx > kTheta16) mx = kTheta16;
  if (mx > kThetaMask) mx = kThetaMask;
  int b = 1;
  while (mx >> b) ++b;
  return b;
}

bool slice_choose(const deoct_ctx* ctx, int W, bool copied, int D, int F, int K, int P, int nb, int64_t tiles, int nprob,
                  SliceShape* out) {
  if (D < 1 || D > kMaxDepthSlice || P < 1 || tiles < 1) return false;
  if (ctx->force_S || ctx->force_TG || ctx->force_warps || ctx->force_grid || ctx->force_stream || ctx->force_slice < 0)
    return false;
  const size_t cap = (size_t)std::min(ctx->max_smem_optin, 227 * 1024) - 1024;  // room for static smem
  const int accw = count_words(D, K);
  const size_t ymask = (size_t)(K + 1) * 128;
  double best = -1.0;
  for (int groups = 1; groups <= 64 && groups <= (P + 3) / 4; ++groups) {
    int tg = (P + groups - 1) / groups;
    tg = (tg + 3) / 4 * 4;
    const int ng = (P + tg - 1) / tg;
    for (int rb : {16, 32, 48}) {
      const size_t rec = (size_t)warp_rec_bytes(D, rb);
      const size_t fixed = ymask + kWarps * rec + (size_t)tg * accw * 4 + 256;
      if (fixed + 4 * 128 > cap) continue;
      const int rows = (int)((cap - fixed) / 128);
      const int nd = pick_digits(nb, F, rows);
      if (nd == 0 || (nd + 3) / 4 * 16 > rb) continue;
      // Work of one (tile, group): expanding the rows, then the group's trees, in
      // cycles (weights estimated from phase timings, not fitted: they order the shapes;
      // the launch's time is modelled below); waves of them over the SMs (one CTA each).
      const double build = 900.0 + 1.3 * F * (digit_rows(nb, nd) + nb);
      const double wf = 4.0 * ((1 << D) - 1) * (2 * nd + 1) + 70.0 * std::max(1, (1 << D) / 8);
      const double quads = tg / 4.0;
      const double route = std::max(quads * wf, std::ceil(quads / kWarps) * 6.0 * wf);
      const int64_t items = tiles * ng;
      const double waves = (double)((items + ctx->num_sms - 1) / ctx->num_sms);
      const double cost = waves * (build + route);
      if (best < 0 || cost < best) {
        best = cost;
        out->TG = tg;
        out->nd = nd;
        out->rows = rows;
        out->rec_bytes = (int)rec;
      }
      break;
    }
  }
  if (best < 0) return false;
  // Time of a launch with planes, us, fitted to 725 random shapes (n = 100 to 1.5e6, F = 4
  // to 60, 6 to 20 bits, 16 to 1024 trees, depth 1 to 5, K = 2 to 9; standard deviation
  // 10%): the launch; the constant rows; per wave of items the table from the planes, the
  // trees' row loads (latency of a warp's quads, then the SM's rate), and the counts of
  // every class where tiles hold several.
  const int tg = out->TG, nd = out->nd, ng = (P + tg - 1) / tg, leaves8 = std::max(1, (1 << D) / 8);
  const double waves = (double)((tiles * ng + ctx->num_sms - 1) / ctx->num_sms);
  const double quads = tg / 4.0, rounds = std::ceil(quads / kWarps), loads = ((1 << D) - 1) * (2.0 * nd + 1);
  // classes of a tile: one where the samples are ordered by class, but for the tiles at the
  // K - 1 borders of a problem; all of them in a set too small to be ordered
  const int64_t borders = (int64_t)(K - 1) * nprob;
  const int classes = nprob == 0 ? (tiles >= 2 * K ? 1 : K) : tiles >= 2 * borders ? 1 : (int)std::min<int64_t>(K, 1 + (borders + tiles - 1) / tiles);
  out->us = 7.28 + 0.0038 * F * nd +
            waves * (0.595 + 8.2e-4 * F * (digit_rows(nb, nd) + nb) + loads * (0.00996 * rounds + 0.0015 * quads) +
                     0.2845 * rounds * leaves8 * classes);
  // The same without planes, fitted to 236 random shapes of 2^27 tree-samples and more
  // (192 to 4096 trees; standard deviation 12%): ranks and class rows are transposed in
  // the launch, and every tile holds every class.
  out->us_raw = 25.25 + waves * (loads * (0.0207 * rounds + 0.00107 * quads) + 0.161 * rounds * leaves8 * K +
                                 F * ((W == 2 ? 0.072 : 0.148) + (copied ? 0.0 : 0.49)) + 1.08 * K);
  return true;
}

// Taken wherever it could run, the bit-sliced evaluator was the slower one at 41% of those
// 725 shapes, and launches took 13% longer than the better one's on average; by the models
// 0.8%.  (5% in its favour: the average is the same from 1 to 1.05, and what is lost where
// the bit-sliced one is the better one falls from 0.5 to 0.2%.)  A generation on the ballot
// kernels / bit-sliced, us: n = 3e5, F = 38, 20 bits, 128 trees of depth 5 94 / 627 (the rows
// leave room for four trees a CTA); n = 1000, F = 30, 17 bits, 128 trees of depth 3 10.9 /
// 14.2; n = 1e5, F = 24, 16 bits, 128 trees of depth 3 25.4 / 18.4; n = 3e5, F = 10, 12 bits,
// 512 trees of depth 4 181 / 64.
bool slice_wins(const deoct_ctx* ctx, const SliceShape& s, const EvalConfig& ballot) {
  return ctx->force_slice > 0 || s.us < 1.05 * ballot.us;
}

// One evaluation on its own, whose tiles' ranks the kernel transposes itself.  Below 192
// trees or 2^27 tree-samples the ballot kernels were level or ahead (GB300: 100 to 128 trees
// 150 us bit-sliced against 145 at n = 1e6, F = 30, depth 3, 49 against 45 at n = 2e5, K = 10;
// 256 trees 39 against 35 at n = 1e5, F = 20, depth 3).  Above, by the models: of 236 random
// shapes the bit-sliced one was the slower at 53 (1201 trees of depth 5, n = 1.35e6, F = 30,
// uint32 7.16 ms against 3.10; 931, n = 1.5e5, K = 9 814 us against 381), taken by them 4,
// by 7% at most; 256 trees of depth 5 on 2e6 rows 500 us against 790, 1024 of depth 4 on 1e7
// 4.5 ms against 10.2.
bool slice_once(const deoct_ctx* ctx, int64_t n, int P) {
  return ctx->force_slice > 0 || (P >= 192 && n * P >= (int64_t(1) << 27));
}
bool slice_wins_once(const deoct_ctx* ctx, const SliceShape& s, const EvalConfig& ballot) {
  return ctx->force_slice > 0 || s.us_raw < 0.95 * ballot.us;
}

int slice_planes(deoct_ctx* ctx, int W, const EvalPlan& plan, const EvalProb* d_probs, int nprob, int64_t tiles,
                 cudaStream_t s) {
  PlaneArgs a;
  a.single = plan.single;
  a.probs = d_probs;
  a.nprob = nprob;
  a.Fmax = plan.Fmax;
  a.tiles = tiles;
  a.status = ctx->d_status;
  const int64_t blocks = (tiles * (plan.Fmax + 1) + 7) / 8;
  const int grid = (int)std::min<int64_t>(blocks, (int64_t)ctx->num_sms * 8);
  if (W == 2) planes_kernel<2><<<grid, 256, 0, s>>>(a);
  else planes_kernel<4><<<grid, 256, 0, s>>>(a);
  count_launch(ctx);
  return check_launch("planes_kernel");
}

int slice_launch(deoct_ctx* ctx, int D, const EvalPlan& plan, const SliceShape& shape, cudaStream_t s) {
  if (plan.total_tiles <= 0) return DEOCT_OK;
  SliceArgs sa;
  evk::EvalArgs& a = sa.e;
  memset(&a.tmap, 0, sizeof(a.tmap));
  a.tmap_box = 0;
  a.single = plan.single;
  a.probs = plan.d_probs;
  a.jobs = plan.d_jobs;
  a.njobs = plan.njobs;
  a.single_ntiles = plan.d_probs == nullptr ? (int)slice_tiles(plan.single.count) : 0;
  a.total_tiles = plan.total_tiles;
  a.S = kTile;
  a.TG = shape.TG;
  a.Fmax = plan.Fmax;
  a.Kmax = plan.Kmax;
  a.lab_stage = 0;
  a.nstage = 0;
  a.status = ctx->d_status;
  a.ticket = plan.d_probs == nullptr ? plan.ticket : nullptr;
  a.counts_out = plan.counts_out;
  a.errors_out = plan.errors_out;
  sa.rows = shape.rows;
  sa.ymask_off = shape.rows * 128;
  sa.rec_off = sa.ymask_off + (plan.Kmax + 1) * 128;
  sa.rec_bytes = shape.rec_bytes;
  sa.acc_off = sa.rec_off + kWarps * shape.rec_bytes;
  sa.smem_bytes = sa.acc_off + shape.TG * count_words(D, plan.Kmax) * 4;
  const int grid = (int)std::min<int64_t>(plan.total_tiles, ctx->num_sms);
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  DEOCT_CUDA_TRY(cudaStreamIsCapturing(s, &cs));
  const bool timed = ctx->timing && !ctx->building && cs == cudaStreamCaptureStatusNone;  // not inside graphs
  if (timed) {
    DEOCT_CUDA_TRY(cudaEventCreate(&e0));
    DEOCT_CUDA_TRY(cudaEventCreate(&e1));
    DEOCT_CUDA_TRY(cudaEventRecord(e0, s));
  }
  int rc = DEOCT_OK;
  switch (D) {
    case 1: rc = launch_slice_1(ctx, shape.nd, sa, shape.raw, grid, s); break;
    case 2: rc = launch_slice_2(ctx, shape.nd, sa, shape.raw, grid, s); break;
    case 3: rc = launch_slice_3(ctx, shape.nd, sa, shape.raw, grid, s); break;
    case 4: rc = launch_slice_4(ctx, shape.nd, sa, shape.raw, grid, s); break;
    case 5: rc = launch_slice_5(ctx, shape.nd, sa, shape.raw, grid, s); break;
    default: rc = set_error(DEOCT_ERR_INVALID, "bit-sliced evaluator: depth %d", D);
  }
  DEOCT_TRY(rc);
  ctx->eval_launches += 1;
  ctx->slice_launches += 1;
  ctx->slice_digits = shape.nd;
  if (timed) {
    DEOCT_CUDA_TRY(cudaEventRecord(e1, s));
    ctx->ev_pairs.push_back(e0);
    ctx->ev_pairs.push_back(e1);
  }
  return DEOCT_OK;
}

}  // namespace slc
}  // namespace deoct
