// Batched application of the Wilson-clover operator: many right-hand sides on one
// lattice, and several lattices of different sizes, in one persistent launch.
//
// A CTA works on tiles of 32 sites x RG right-hand sides (blockDim = (32, RG / NR)): warp y
// applies M to NR (1 or 2) right-hand sides from rg*RG + y*NR on the tile's 32 sites, so the
// links and the clover of those sites are fetched from DRAM once and served to the other
// warps from L1. Every output site runs the same stencil code as the single-RHS kernel, so
// results are bitwise identical. The tile shape (RG and the number of resident CTAs)
// is chosen per batch plan by timing the candidates once (the autotuner below), and a
// plan can record its launches in a CUDA graph for replay. With FP16 storage the plan
// also times the tensor-core kernel of mrhs_tc.cu (all right-hand sides of a site in
// one dense contraction) and keeps the faster of the two.
#include <algorithm>
#include <climits>
#include <cmath>
#include <string>
#include <vector>

#include "internal.h"
#include "mrhs_tc.h"
#include "wilson_ds.cuh"
#include "wilson.cuh"

namespace dirac {

static constexpr int kTileSites = 32;
static constexpr int kMaxRG = 16;
static constexpr int kMaxLat = 16;

// one lattice of a batch, as the kernel sees it
struct BatchLat {
  Geom g;
  const char* gauge;
  const char* clover;
  double kappa;
  const char* in;       // nrhs consecutive full fields
  char* out;
  size_t field_bytes;
  int nrhs;
  int tiles_site;       // 32-site groups (of one parity) of the lattice
  int tiles;            // tiles_site * ceil(nrhs / RG)
  int tile_begin;       // first tile of this lattice in the batch
  int rhs0;             // plan-wide index of this lattice's first right-hand side
  const double* mask;   // null, or mask[(rhs0 + r) * mstride] == 0: right-hand side r is skipped
  int mstride;
};

// output site idx of right-hand sides rhs .. rhs + N - 1
template <int PREC, int R, int N = 1>
__device__ __forceinline__ void batch_site(const BatchLat& L, int rhs, int idx, char* ring = nullptr) {
  WilsonArg a;
  a.g = L.g;
  a.gauge = L.gauge;
  a.clover = L.clover;
  a.kappa = L.kappa;
  a.dagger = 0;
  a.out_parity = 0;
  const size_t hb = L.field_bytes / 2;
  const char* in = L.in + (size_t)rhs * L.field_bytes;
  char* out = L.out + (size_t)rhs * L.field_bytes;
  a.in[0] = in;
  a.in[1] = in + hb;
  a.out[0] = out;
  a.out[1] = out + hb;
  wilson_site<PREC, R, true, N>(a, idx, L.field_bytes, ring);
}

// Tile t of lattice L: warp y of the CTA has right-hand sides y NR .. y NR + NR - 1 of the
// tile's RG (warp-uniform, so that the fields are uniform addresses). Where one of a pair
// is missing or masked out, the other runs alone.
template <int PREC, int R, int NR>
__device__ __forceinline__ void batch_tile(const BatchLat& L, int t, int RG) {
  const int rg = t / L.tiles_site, sg = t - rg * L.tiles_site;
  const int y = __shfl_sync(0xffffffffu, threadIdx.y, 0);
  int rhs = rg * RG + y * NR;
  const int idx = sg * kTileSites + threadIdx.x;
  auto on = [&](int r) { return r < L.nrhs && !(L.mask && L.mask[(size_t)(L.rhs0 + r) * L.mstride] == 0.0); };
  const bool first = on(rhs);
  if constexpr (NR == 2) {
    const bool second = on(rhs + 1);
    if (first && second) {
      batch_site<PREC, R, 2>(L, rhs, idx, ring_of_warp<PREC, R, 2>(y));
      return;
    }
    if (!first && !second) return;
    if (!first) ++rhs;
  } else {
    if (!first) return;
  }
  batch_site<PREC, R, 1>(L, rhs, idx);
}

// one lattice, descriptor by value
template <int PREC, int R, int NR>
__global__ void __launch_bounds__(kTileSites * kMaxRG, 1) mrhs_kernel(const __grid_constant__ BatchLat L, int RG) {
  pdl_begin();
  for (int t = blockIdx.x; t < L.tiles; t += gridDim.x) batch_tile<PREC, R, NR>(L, t, RG);
}

// several lattices: descriptor table in the parameter space (uniform loads), tiles numbered
// across lattices
struct LatTable { BatchLat v[kMaxLat]; };
template <int PREC, int R, int NR>
__global__ void __launch_bounds__(kTileSites * kMaxRG, 1)
    batch_kernel(const __grid_constant__ LatTable lats, int nlat, int ntiles, int RG) {
  pdl_begin();
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    int l = 0;
    while (l + 1 < nlat && t >= lats.v[l + 1].tile_begin) ++l;
    batch_tile<PREC, R, NR>(lats.v[l], t - lats.v[l].tile_begin, RG);
  }
}

// FP64 fields of a masked plan (the FP64 residuals of the batched solves): a warp per
// (right-hand side, 32-site group), over the right-hand sides that the masks leave. The FP64 pipe bounds this kernel (19 cycles per warp instruction and SM,
// four schedulers at 64), links and clover come from L2 at a tenth of its rate, so what
// counts is that every scheduler has the same number of warps with work: with warp y of a
// CTA tied to right-hand side 4 k + y, a reliable update of a few systems ran on one or two
// of the four schedulers. Without a mask the tuned shapes of batch_kernel are faster (us, that
// -> this): 8^3x16 x 1 43 -> 73, 12^3x20 x 1 80 -> 117, 10^2x14x18 x 3 158 -> 193, 16^4 x 3
// 408 -> 423.
static constexpr int kBatch64PerSM = 3;
static constexpr int kMaxBatch64Rhs = 1024;  // right-hand sides listed at a time
template <int R>
__global__ void __launch_bounds__(128, kBatch64PerSM)
    batch_kernel64(const BatchLat* __restrict__ lats, int nlat, int nrhs) {
  pdl_begin();
  __shared__ int first[kMaxBatch64Rhs + 1];  // first warp item of each listed right-hand side
  __shared__ int lat[kMaxBatch64Rhs], loc[kMaxBatch64Rhs];
  __shared__ int listed;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int r0 = 0; r0 < nrhs; r0 += kMaxBatch64Rhs) {
    const int r1 = min(nrhs, r0 + kMaxBatch64Rhs);
    __syncthreads();
    if (w == 0) {
      int n = 0, items = 0;
      for (int q0 = r0; q0 < r1; q0 += 32) {
        const int q = q0 + lane;
        int l = 0, cnt = 0;
        if (q < r1) {
          while (l + 1 < nlat && q >= lats[l + 1].rhs0) ++l;
          const BatchLat& L = lats[l];
          if (!L.mask || L.mask[(size_t)q * L.mstride] != 0.0) cnt = L.tiles_site;
        }
        const unsigned on = __ballot_sync(0xffffffffu, cnt > 0);
        int sum = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int t = __shfl_up_sync(0xffffffffu, sum, o);
          if (lane >= o) sum += t;
        }
        if (cnt > 0) {
          const int k = n + __popc(on & ((1u << lane) - 1));
          first[k] = items + sum - cnt;
          lat[k] = l;
          loc[k] = q - lats[l].rhs0;
        }
        n += __popc(on);
        items += __shfl_sync(0xffffffffu, sum, 31);
      }
      if (lane == 0) {
        listed = n;
        first[n] = items;
      }
    }
    __syncthreads();
    const int n = listed, items = first[n];
    for (int i = blockIdx.x * 4 + w; i < items; i += gridDim.x * 4) {
      int a = 0, b = n;  // first[a] <= i < first[b]
      while (b - a > 1) {
        const int m = (a + b) >> 1;
        if (first[m] <= i) a = m;
        else b = m;
      }
      batch_site<P64, R>(lats[lat[a]], loc[a], (i - first[a]) * kTileSites + lane);
    }
  }
}

// the double-single form (FP64 fields): 4 right-hand sides per CTA (the untimed default
// shape), so that a thread may hold the float-float values in up to 255 registers
__global__ void __launch_bounds__(kTileSites * 4, 1)
    batch_kernel_ds(const BatchLat* __restrict__ lats, int nlat, int ntiles) {
  pdl_begin();
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    int l = 0;
    while (l + 1 < nlat && t >= lats[l + 1].tile_begin) ++l;
    const BatchLat L = lats[l];
    batch_tile<P64DS, 18, 1>(L, t - L.tile_begin, 4);
  }
}

template <int PREC, int NR>
static void launch_mrhs_prec(int recon, const BatchLat& L, int RG, int grid, cudaStream_t st) {
  dim3 block(kTileSites, RG / NR);
  if (recon == 18) launch_pdl(mrhs_kernel<PREC, 18, NR>, grid, block, RG / NR * kRingWarp<PREC, 18, NR>, st, L, RG);
  else if (recon == 12) launch_pdl(mrhs_kernel<PREC, 12, NR>, grid, block, RG / NR * kRingWarp<PREC, 12, NR>, st, L, RG);
  else launch_pdl(mrhs_kernel<PREC, 8, NR>, grid, block, RG / NR * kRingWarp<PREC, 8, NR>, st, L, RG);
}
template <int PREC, int NR>
static void launch_batch_prec(int recon, const std::vector<BatchLat>& l, int ntiles, int RG, int grid, cudaStream_t st) {
  LatTable t;
  for (size_t k = 0; k < l.size(); ++k) t.v[k] = l[k];
  const int nlat = (int)l.size();
  dim3 block(kTileSites, RG / NR);
  if (recon == 18) launch_pdl(batch_kernel<PREC, 18, NR>, grid, block, RG / NR * kRingWarp<PREC, 18, NR>, st, t, nlat, ntiles, RG);
  else if (recon == 12) launch_pdl(batch_kernel<PREC, 12, NR>, grid, block, RG / NR * kRingWarp<PREC, 12, NR>, st, t, nlat, ntiles, RG);
  else launch_pdl(batch_kernel<PREC, 8, NR>, grid, block, RG / NR * kRingWarp<PREC, 8, NR>, st, t, nlat, ntiles, RG);
}

static void launch_batch64(int recon, const BatchLat* d, int nlat, int nrhs, int grid, cudaStream_t st) {
  if (recon == 18) launch_pdl(batch_kernel64<18>, grid, 128, 0, st, d, nlat, nrhs);
  else if (recon == 12) launch_pdl(batch_kernel64<12>, grid, 128, 0, st, d, nlat, nrhs);
  else launch_pdl(batch_kernel64<8>, grid, 128, 0, st, d, nlat, nrhs);
}

static BatchLat describe(const dirac_ctx* c, int prec, const void* in, void* out, int nrhs, int RG) {
  BatchLat L;
  L.g = c->g;
  L.gauge = c->gauge[prec];
  L.clover = c->p.csw != 0.0 ? c->clover[prec] : nullptr;
  L.kappa = c->p.kappa;
  L.in = (const char*)in;
  L.out = (char*)out;
  L.field_bytes = 2 * spinor_half_bytes(prec, 24, c->Vh);
  L.nrhs = nrhs;
  L.tiles_site = full_sites((int)c->Vh) / kTileSites;
  L.tiles = L.tiles_site * ((nrhs + RG - 1) / RG);
  L.tile_begin = 0;
  L.rhs0 = 0;
  L.mask = nullptr;
  L.mstride = 0;
  return L;
}

static int sm_count() {
  static int n = 0;
  if (!n) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (n <= 0) n = 1;
  }
  return n;
}

// CTAs for a shape: `per_sm` resident CTAs on every SM, no more than the tiles
static int grid_for(int per_sm, int tiles) {
  long g = (long)sm_count() * per_sm;
  return (int)(g < tiles ? g : tiles);
}

}  // namespace dirac

using namespace dirac;

struct dirac_batch {
  std::vector<dirac_ctx*> ctxs;
  std::vector<BatchLat> lats;    // host copy (RG-dependent fields refreshed by the tuner)
  BatchLat* d_lats = nullptr;    // device table
  int prec = 0, recon = 12, ntiles = 0, nrhs = 0;
  bool ds = false;               // FP64 fields: double-single arithmetic (18-real links)
  int RG = 1, NR = 1, per_sm = 1, grid = 1;
  int grid64 = 1;                // CTAs of the kernel for masked FP64 plans
  double tuned_ms = 0;
  std::vector<double> cand_ms;   // autotuner timings, candidate order
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  int graph_napply = 0;
  // tensor-core kernel (FP16 storage): its lattice table, grid and creation timing
  bool use_tc = false;
  TcLat* d_tc = nullptr;
  std::vector<int*> tc_nbr;      // per-lattice neighbour tables of the tensor-core kernel
  int tc_ntiles = 0, tc_grid = 0;
  double tc_ms = -1, cc_ms = -1;
  std::string err;
};

namespace dirac {

// the tile-shape candidates: (right-hand sides per CTA, CTAs per SM, right-hand sides per
// thread). 16 warps of the 128-register cap are resident per SM; the shapes with 32 hand the
// CTAs that do not fit to the SMs that finish first, which evens out ragged ends.
static const int kCand[][3] = {{1, 16, 1}, {2, 8, 1}, {4, 4, 1}, {2, 16, 1}, {4, 8, 1}, {2, 16, 2}, {4, 8, 2}, {8, 4, 2}};
static constexpr int kDefaultCand = 2, kDefaultPair = 6;

// Two right-hand sides per thread load and rebuild every link once for both, but a thread
// takes about 1.6 times as long and there are half as many: worth it from about two waves of
// resident warps on (16 per SM), most where links and clover come from DRAM. The rule of the
// calls that are not timed. Measured, one right-hand side per thread -> two, us: FP32 12^3x20 x
// 7 20.9 -> 20.1, 16^4 x 12 65 -> 66, 16^3x32 x 2 29.0 -> 26.5, x 12 148 -> 127, 24^3x32 x 12
// 510 -> 413; FP16 16^4 x 12 62.0 -> 61.3, 16^3x32 x 8 82.6 -> 76.4, 24^3x32 x 8 284 -> 252; below
// two waves 12^3x20 x 8 FP16 21.7 -> 22.6, 8^3x16 x 7 6.8 -> 7.9. With an odd count one thread of
// each group has a single right-hand side: FP32 still gains (16^4 x 3 18.0 -> 17.1, 24^3x32 x 3
// 154 -> 127, x 5 252 -> 206), FP16, which is compute-bound, does not (16^3x32 x 7 73.3 -> 79.2, x
// 15 162 -> 165).
static bool pair_rhs(int prec, long groups, int nrhs) {
  if (prec == P64 || groups * nrhs <= 32l * sm_count()) return false;
  return nrhs % 2 == 0 || (prec == P32 && nrhs >= 3);
}

// Warps per CTA for `items` warps on the same sites: the most (up to 4, they share the links
// through L1) of those that leave the fewest of an SM's 16 warps idle. (12 warps of 12 right-
// hand sides left a quarter of the SM empty: FP32 16^4 x 12 took 102.6 us against 51.6 x 7.)
static int group_warps(int items) {
  int best = 1, busy = 0;
  for (int w = 1; w <= 4; ++w) {
    const int b = 1000 * items / ((items + w - 1) / w * w) * (16 / w * w);
    if (b >= busy) busy = b, best = w;
  }
  return best;
}

static int batch_layout(dirac_batch* b, int RG, cudaStream_t st) {
  int begin = 0;
  for (size_t l = 0; l < b->lats.size(); ++l) {
    BatchLat& L = b->lats[l];
    L.tiles = L.tiles_site * ((L.nrhs + RG - 1) / RG);
    L.tile_begin = begin;
    begin += L.tiles;
  }
  b->ntiles = begin;
  // pageable source: the copy is staged before the call returns, so the host vector
  // may change afterwards
  if (cudaMemcpyAsync(b->d_lats, b->lats.data(), sizeof(BatchLat) * b->lats.size(), cudaMemcpyHostToDevice,
                      st) != cudaSuccess) {
    b->err = "descriptor copy failed";
    return DIRAC_ERR_CUDA;
  }
  return DIRAC_OK;
}

static void batch_launch_direct(dirac_batch* b, cudaStream_t st) {
  const int nlat = (int)b->lats.size();
  if (b->use_tc) {
    launch_mrhs_tc(b->recon, b->d_tc, nlat, b->tc_ntiles, b->tc_grid, st);
    return;
  }
  if (b->prec == P64 && b->ds)
    launch_pdl(batch_kernel_ds, b->grid, dim3(kTileSites, 4), 0, st, b->d_lats, nlat, b->ntiles);
  else if (b->prec == P64 && b->lats[0].mask) launch_batch64(b->recon, b->d_lats, nlat, b->nrhs, b->grid64, st);
  else if (b->prec == P64) launch_batch_prec<P64, 1>(b->recon, b->lats, b->ntiles, b->RG, b->grid, st);
  else if (b->prec == P32) (b->NR == 2 ? launch_batch_prec<P32, 2> : launch_batch_prec<P32, 1>)(b->recon, b->lats, b->ntiles, b->RG, b->grid, st);
  else (b->NR == 2 ? launch_batch_prec<P16, 2> : launch_batch_prec<P16, 1>)(b->recon, b->lats, b->ntiles, b->RG, b->grid, st);
}

}  // namespace dirac

extern "C" {

int dirac_apply_multi(dirac_ctx* c, void* out, const void* in, int nrhs, dirac_prec prec, void* stream) {
  int rc = check_op(c, prec, false);
  if (rc) return rc;
  if (c->p.kind != DIRAC_WILSON_CLOVER)
    return set_err(c, DIRAC_ERR_UNSUPPORTED, "multi-RHS apply is defined for Wilson-clover");
  if (!out || !in || nrhs < 1) return set_err(c, DIRAC_ERR_ARG, "bad multi-RHS arguments");
  const size_t fb = 2 * spinor_half_bytes(prec, 24, c->Vh);
  const char *i0 = (const char*)in, *o0 = (const char*)out;
  if (i0 < o0 + fb * nrhs && o0 < i0 + fb * nrhs) return set_err(c, DIRAC_ERR_ARG, "in and out overlap");
  const int NR = pair_rhs(prec, full_sites((int)c->Vh) / kTileSites, nrhs) ? 2 : 1;
  int warps = group_warps((nrhs + NR - 1) / NR);
  // an odd count leaves the last warp of its CTA a single right-hand side on every tile: with
  // two warps half of the chip's work is out of step (FP32 24^3x32 x 3 148 us against 127 with
  // one warp per CTA, 16^4 x 11 70 against 63)
  if (NR == 2 && nrhs % 2 && warps < 4) warps = 1;
  const int RG = warps * NR;
  const BatchLat L = describe(c, prec, in, out, nrhs, RG);
  const int grid = grid_for(16 / warps, L.tiles);
  cudaStream_t st = (cudaStream_t)stream;
  if ((int)prec == P64) launch_mrhs_prec<P64, 1>(c->p.recon[prec], L, RG, grid, st);
  else if ((int)prec == P32) (NR == 2 ? launch_mrhs_prec<P32, 2> : launch_mrhs_prec<P32, 1>)(c->p.recon[prec], L, RG, grid, st);
  else (NR == 2 ? launch_mrhs_prec<P16, 2> : launch_mrhs_prec<P16, 1>)(c->p.recon[prec], L, RG, grid, st);
  return cuda_check(c, "multi-RHS kernel");
}

int dirac_batch_create(dirac_ctx* const* ctxs, int nlat, void* const* out, const void* const* in,
                       const int* nrhs, dirac_prec prec, void* stream, dirac_batch** plan) {
  return dirac::batch_create(ctxs, nlat, out, in, nrhs, prec, (cudaStream_t)stream, plan, 2, false);
}

}  // extern "C"

namespace dirac {

int batch_create(dirac_ctx* const* ctxs, int nlat, void* const* out, const void* const* in, const int* nrhs,
                 int prec, cudaStream_t stream, dirac_batch** plan, int tune, bool ds) {
  if (!ctxs || !out || !in || !nrhs || !plan || nlat < 1 || nlat > kMaxLat) return DIRAC_ERR_ARG;
  *plan = nullptr;
  int recon = -1;
  for (int l = 0; l < nlat; ++l) {
    dirac_ctx* c = ctxs[l];
    if (!c || !out[l] || !in[l] || nrhs[l] < 1) return DIRAC_ERR_ARG;
    int rc = check_op(c, prec, false);
    if (rc) return rc;
    if (c->p.kind != DIRAC_WILSON_CLOVER) return set_err(c, DIRAC_ERR_UNSUPPORTED, "batch: Wilson-clover only");
    if (recon >= 0 && c->p.recon[prec] != recon)
      return set_err(c, DIRAC_ERR_ARG, "batch: every lattice needs the same link compression");
    recon = c->p.recon[prec];
  }
  if (ds && (prec != P64 || recon != 18 || tune != 0))
    return set_err(ctxs[0], DIRAC_ERR_UNSUPPORTED, "batch: double-single needs FP64 18-real links, untimed");
  dirac_batch* b = new dirac_batch();
  b->prec = prec;
  b->recon = recon;
  b->ds = ds;
  for (int l = 0, r0 = 0; l < nlat; ++l) {
    b->ctxs.push_back(ctxs[l]);
    b->lats.push_back(describe(ctxs[l], prec, in[l], out[l], nrhs[l], 1));
    b->lats.back().rhs0 = r0;
    r0 += nrhs[l];
    b->nrhs = r0;
  }
  long ctas64 = 0;
  for (const BatchLat& L : b->lats) ctas64 += (long)L.tiles_site * ((L.nrhs + 3) / 4);
  b->grid64 = grid_for(kBatch64PerSM, (int)std::min(ctas64, (long)INT_MAX));
  if (cudaMalloc(&b->d_lats, sizeof(BatchLat) * nlat) != cudaSuccess) {
    cudaGetLastError();
    delete b;
    return DIRAC_ERR_OOM;
  }
  // autotune: time every candidate shape once (after one warm-up launch) and keep the
  // fastest; the launches write the plan's outputs, which the caller owns anyway. One and two
  // right-hand sides per thread are both timed: which is faster turns on whether links and
  // clover come from L2 (FP16 12^3x20 x 8 24.7 us against 26.5, 10^2x14x18 x 10 22.5 against
  // 25.4) or from DRAM (FP32 24^3x32 x 9 409 against 354), and lattices of both kinds may share
  // a plan.
  cudaStream_t st = stream;
  int max_rhs = 1;
  for (int l = 0; l < nlat; ++l) max_rhs = nrhs[l] > max_rhs ? nrhs[l] : max_rhs;
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  double best = INFINITY;
  int bi = 0;
  // the untimed shape: pairs if they pay on every lattice
  bool pairs = true;
  for (int l = 0; l < nlat; ++l) pairs = pairs && pair_rhs(prec, b->lats[l].tiles_site, nrhs[l]);
  const int untimed = pairs ? kDefaultPair : kDefaultCand;
  const int ncand = (int)(sizeof(kCand) / sizeof(kCand[0]));
  for (int k = 0; k < ncand; ++k) {
    const int RG = kCand[k][0], per_sm = kCand[k][1];
    b->NR = kCand[k][2];
    // tune < 2: only the default shape (4 right-hand sides per CTA)
    // (the default shape also serves plans with fewer right-hand sides: idle warps exit)
    if (tune < 2 ? k != untimed : (RG > max_rhs && RG > 1) || (prec == P64 && b->NR > 1)) {
      b->cand_ms.push_back(-1);
      continue;
    }
    if (tune <= 0) {  // no timing at all
      best = 0;
      bi = k;
      b->cand_ms.push_back(-1);
      continue;
    }
    b->RG = RG;
    if (batch_layout(b, RG, st)) break;
    b->grid = grid_for(per_sm, b->ntiles);
    batch_launch_direct(b, st);
    // one launch, or the mean of three where one is short
    float ms = 0;
    for (int reps = 1; reps <= 3 && b->err.empty(); reps += 2) {
      cudaEventRecord(e0, st);
      for (int r = 0; r < reps; ++r) batch_launch_direct(b, st);
      cudaEventRecord(e1, st);
      if (cudaEventSynchronize(e1) != cudaSuccess || cudaGetLastError() != cudaSuccess) b->err = "autotune launch failed";
      cudaEventElapsedTime(&ms, e0, e1);
      ms /= reps;
      if (ms > 0.5f) break;
    }
    if (!b->err.empty()) break;
    b->cand_ms.push_back(ms);
    if (ms < best) { best = ms; bi = k; }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (!b->err.empty() || best == INFINITY) {
    cudaGetLastError();
    cudaFree(b->d_lats);
    delete b;
    return DIRAC_ERR_CUDA;
  }
  b->RG = kCand[bi][0];
  b->NR = kCand[bi][2];
  b->per_sm = kCand[bi][1];
  if (batch_layout(b, b->RG, st)) {
    cudaFree(b->d_lats);
    delete b;
    return DIRAC_ERR_CUDA;
  }
  b->grid = grid_for(b->per_sm, b->ntiles);
  b->tuned_ms = best;
  b->cc_ms = best;
  // the tensor-core kernel (FP16 storage, 12- or 18-real links): timed the same way; the
  // plan keeps whichever kernel is faster
  if (prec == DIRAC_PREC_F16 && (recon == 12 || recon == 18) && tune >= 0) {
    std::vector<TcLat> tl(nlat);
    int begin = 0;
    for (int l = 0; l < nlat; ++l) {
      const BatchLat& L = b->lats[l];
      TcLat& T = tl[l];
      T.g = L.g;
      T.gauge = L.gauge;
      T.clover = L.clover;
      T.kappa = (float)L.kappa;
      T.in = L.in;
      T.out = L.out;
      T.field_bytes = L.field_bytes;
      T.nrhs = L.nrhs;
      T.ctiles = tc_ctiles(L.g.Vh);
      T.tiles = tc_tiles(T);
      T.tile_begin = begin;
      int* nb = nullptr;
      if (tc_build_nbr(L.g, &nb, st) == DIRAC_OK) b->tc_nbr.push_back(nb);
      T.nbr = nb;
      begin += T.tiles;
    }
    b->tc_ntiles = begin;
    const long g = (long)sm_count() * tc_ctas_per_sm(recon);
    b->tc_grid = (int)(g < begin ? g : begin);
    bool tables = true;
    for (int l = 0; l < nlat; ++l) tables = tables && tl[l].nbr != nullptr;
    if (!tables || cudaMalloc(&b->d_tc, sizeof(TcLat) * nlat) != cudaSuccess ||
        cudaMemcpyAsync(b->d_tc, tl.data(), sizeof(TcLat) * nlat, cudaMemcpyHostToDevice, st) != cudaSuccess) {
      cudaGetLastError();
      if (b->d_tc) cudaFree(b->d_tc);
      b->d_tc = nullptr;
    } else if (tune == 0) {
      b->use_tc = true;  // untimed plans take the tensor-core kernel where there is one
    } else {
      cudaEvent_t f0, f1;
      cudaEventCreate(&f0);
      cudaEventCreate(&f1);
      b->use_tc = true;
      batch_launch_direct(b, st);
      cudaEventRecord(f0, st);
      for (int r = 0; r < 3; ++r) batch_launch_direct(b, st);
      cudaEventRecord(f1, st);
      float ms = 0;
      if (cudaEventSynchronize(f1) == cudaSuccess && cudaGetLastError() == cudaSuccess &&
          cudaEventElapsedTime(&ms, f0, f1) == cudaSuccess) {
        b->tc_ms = ms / 3;
        b->use_tc = b->tc_ms < best;
        if (b->use_tc) b->tuned_ms = b->tc_ms;
      } else {
        cudaGetLastError();
        b->use_tc = false;
      }
      cudaEventDestroy(f0);
      cudaEventDestroy(f1);
      if (b->tc_ms < 0) {
        // the tensor-core launch failed: the plan keeps the CUDA-core kernel
        cudaStreamSynchronize(st);
        cudaGetLastError();
      }
    }
  }
  *plan = b;
  return cudaStreamSynchronize(st) == cudaSuccess ? DIRAC_OK : DIRAC_ERR_CUDA;
}

// Right-hand sides whose mask entry is 0 are skipped by the CUDA-core kernels (their
// outputs are left as they are); a masked plan uses the CUDA-core kernel. The mask is
// read at every launch, so it may change between launches and inside captured graphs.
int batch_set_mask(dirac_batch* b, const double* mask, int stride, cudaStream_t st) {
  if (!b) return DIRAC_ERR_ARG;
  for (BatchLat& L : b->lats) {
    L.mask = mask;
    L.mstride = stride;
  }
  if (mask && b->use_tc) {
    b->use_tc = false;
    b->tuned_ms = b->cc_ms;
  }
  if (b->exec) { cudaGraphExecDestroy(b->exec); b->exec = nullptr; }
  if (b->graph) { cudaGraphDestroy(b->graph); b->graph = nullptr; }
  b->graph_napply = 0;
  return batch_layout(b, b->RG, st);
}

}  // namespace dirac

extern "C" {

int dirac_batch_apply(dirac_batch* b, void* stream) {
  if (!b) return DIRAC_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  if (b->exec) {
    if (cudaGraphLaunch(b->exec, st) != cudaSuccess) return DIRAC_ERR_CUDA;
    return DIRAC_OK;
  }
  batch_launch_direct(b, st);
  return cudaGetLastError() == cudaSuccess ? DIRAC_OK : DIRAC_ERR_CUDA;
}

int dirac_batch_capture(dirac_batch* b, int napply, void* stream) {
  if (!b || napply < 1) return DIRAC_ERR_ARG;
  if (b->exec) { cudaGraphExecDestroy(b->exec); b->exec = nullptr; }
  if (b->graph) { cudaGraphDestroy(b->graph); b->graph = nullptr; }
  cudaStream_t cap;
  if (cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking) != cudaSuccess) return DIRAC_ERR_CUDA;
  // the capture stream waits for the caller's stream so the descriptor table is in place
  cudaEvent_t ready;
  cudaEventCreateWithFlags(&ready, cudaEventDisableTiming);
  cudaEventRecord(ready, (cudaStream_t)stream);
  cudaStreamWaitEvent(cap, ready, 0);
  cudaStreamSynchronize(cap);
  cudaEventDestroy(ready);
  int rc = DIRAC_OK;
  if (cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal) != cudaSuccess) rc = DIRAC_ERR_CUDA;
  for (int k = 0; rc == DIRAC_OK && k < napply; ++k) batch_launch_direct(b, cap);
  if (rc == DIRAC_OK && cudaStreamEndCapture(cap, &b->graph) != cudaSuccess) rc = DIRAC_ERR_CUDA;
  if (rc == DIRAC_OK && cudaGraphInstantiate(&b->exec, b->graph, 0) != cudaSuccess) rc = DIRAC_ERR_CUDA;
  cudaStreamDestroy(cap);
  if (rc) {
    cudaGetLastError();
    if (b->graph) { cudaGraphDestroy(b->graph); b->graph = nullptr; }
    b->exec = nullptr;
    return rc;
  }
  b->graph_napply = napply;
  return DIRAC_OK;
}

int dirac_batch_info(const dirac_batch* b, int* rhs_per_cta, int* ctas_per_sm, int* grid, double* tuned_ms) {
  if (!b) return DIRAC_ERR_ARG;
  if (rhs_per_cta) *rhs_per_cta = b->RG;
  if (ctas_per_sm) *ctas_per_sm = b->per_sm;
  if (grid) *grid = b->grid;
  if (tuned_ms) *tuned_ms = b->tuned_ms;
  return DIRAC_OK;
}

int dirac_batch_set_tensor_cores(dirac_batch* b, int on) {
  if (!b) return DIRAC_ERR_ARG;
  if (on && !b->d_tc) return DIRAC_ERR_UNSUPPORTED;
  if (b->use_tc != (on != 0)) {
    // a captured graph holds the other kernel: drop it (capture again)
    if (b->exec) { cudaGraphExecDestroy(b->exec); b->exec = nullptr; }
    if (b->graph) { cudaGraphDestroy(b->graph); b->graph = nullptr; }
    b->graph_napply = 0;
  }
  b->use_tc = on != 0;
  b->tuned_ms = b->use_tc ? b->tc_ms : b->cc_ms;
  return DIRAC_OK;
}

int dirac_batch_rhs_per_thread(const dirac_batch* b) { return b ? b->NR : 0; }

int dirac_batch_set_rhs_per_thread(dirac_batch* b, int n, void* stream) {
  if (!b || n < 1 || n > 2) return DIRAC_ERR_ARG;
  if (n == 2 && b->prec == P64) return DIRAC_ERR_UNSUPPORTED;
  if (b->exec) { cudaGraphExecDestroy(b->exec); b->exec = nullptr; }
  if (b->graph) { cudaGraphDestroy(b->graph); b->graph = nullptr; }
  b->graph_napply = 0;
  const int* shape = kCand[n == 2 ? kDefaultPair : kDefaultCand];
  b->use_tc = false;
  b->RG = shape[0];
  b->per_sm = shape[1];
  b->NR = n;
  if (batch_layout(b, b->RG, (cudaStream_t)stream)) return DIRAC_ERR_CUDA;
  b->grid = grid_for(b->per_sm, b->ntiles);
  return DIRAC_OK;
}

int dirac_batch_kernel_info(const dirac_batch* b, int* tensor_cores, double* cuda_core_ms, double* tensor_core_ms) {
  if (!b) return DIRAC_ERR_ARG;
  if (tensor_cores) *tensor_cores = b->use_tc ? 1 : 0;
  if (cuda_core_ms) *cuda_core_ms = b->cc_ms;
  if (tensor_core_ms) *tensor_core_ms = b->tc_ms;
  return DIRAC_OK;
}

int dirac_batch_destroy(dirac_batch* b) {
  if (!b) return DIRAC_ERR_ARG;
  if (b->exec) cudaGraphExecDestroy(b->exec);
  if (b->graph) cudaGraphDestroy(b->graph);
  if (b->d_tc) cudaFree(b->d_tc);
  for (int* t : b->tc_nbr) cudaFree(t);
  if (b->d_lats) cudaFree(b->d_lats);
  delete b;
  cudaGetLastError();
  return DIRAC_OK;
}

}  // extern "C"
