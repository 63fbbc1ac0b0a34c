// The FP64 Wilson-clover stencil with one site's work split over 16 lanes, for lattices too
// small to fill the chip with one thread per site (wilson.cuh).
//
// The FP64 pipe of this part takes one warp instruction every 64 cycles per scheduler (19
// per SM with four schedulers busy), whatever the number of active lanes (measured), so a
// thread that walks all 8 hops of its site issues ~1150 FP64 instructions at 64 cycles each:
// 40 us for any lattice up to 10,000 sites, 0.5 us of which is arithmetic at 4^4. Here a
// warp takes 2 sites, 16 lanes each = 8 hops x 2 projected spins (the hop chosen by selects,
// not branches); the products U h go through shared memory and 12 of the 16 lanes then own
// one output component each, clover row included: ~85 FP64 instructions in a row. The sums
// run in the hop order and with the operations of wilson_site, so both forms give the same
// bits.
#pragma once
#include "wilson.cuh"

namespace dirac {

__device__ __forceinline__ double neg_if(double v, bool n) { return n ? -v : v; }

// Row i of block blk of M x for a clover-format FP64 matrix: the order of herm6_mv; x_k from
// global memory (chunks of a field at site cb, stride Vh) or a shared-memory vector.
template <class X>
__device__ __forceinline__ C<double> row64(const char* m, int Vh, int cb, int blk, int i, X&& x) {
  const double* dp = reinterpret_cast<const double*>(m + ((size_t)(18 * blk + (i >> 1)) * Vh + cb) * 16) + (i & 1);
  double2 l[5], t[5];
  const double d = __ldg(dp);
  const double2 xi = x(6 * blk + i);
#pragma unroll
  for (int kk = 0; kk < 5; ++kk) {
    const int k = kk + (kk >= i);
    const int o = k < i ? i * (i - 1) / 2 + k : k * (k - 1) / 2 + i;
    l[kk] = ldg_chunk<double2>(m + ((size_t)(18 * blk + 3 + o) * Vh + cb) * 16);
    l[kk].y = neg_if(l[kk].y, k > i);
    t[kk] = x(6 * blk + k);
  }
  C<double> y = {d * xi.x, d * xi.y};
#pragma unroll
  for (int kk = 0; kk < 5; ++kk) cmac(y, C<double>{l[kk].x, l[kk].y}, C<double>{t[kk].x, t[kk].y});
  return y;
}

template <int R, bool FULLM>
__global__ void __launch_bounds__(32) wilson_split64_kernel(const WilsonArg a) {
  pdl_begin();
  __shared__ double2 v[2][8][6];
  __shared__ double2 post[2][12];
  const Geom& g = a.g;
  const int Vh = g.Vh, n = FULLM ? 2 * Vh : Vh;
  const int st = threadIdx.x >> 4, l = threadIdx.x & 15;
  const int idx = blockIdx.x * 2 + st;
  const bool ok = idx < n;
  int par = a.out_parity, cb = ok ? idx : n - 1;
  if (FULLM) {
    par = cb >= Vh;
    cb -= par * Vh;
  }
  const char* src = par ? a.in[0] : a.in[1];
  const bool dagger = a.dagger != 0;
  {
    const int hop = l >> 1, spin = l & 1, mu = hop >> 1;
    const bool back = hop & 1;
    const bool plus = back != dagger;  // the projector's sign s
    int y[4], x[4];
    cb_coords(g, cb, par, x);
    bool neg = false;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      y[m] = x[m];
      if (m == mu) {
        const int L = g.L[m];
        y[m] += back ? -1 : 1;
        if (y[m] == L || y[m] < 0) {
          y[m] = back ? L - 1 : 0;
          neg = m == 3 && g.apbc;
        }
      }
    }
    const int ycb = cb_index(g, y);
    // the projected component h = u + phase l of this spin (wilson_project): the lower spin
    // that enters, whether it is multiplied by i, and its sign
    const int low = mu < 2 ? 1 - spin : spin;
    const bool im = mu == 0 || mu == 2;
    const bool minus = plus == ((mu == 1 && spin == 0) || (mu == 2 && spin == 1));
    double2 u[3], w[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      u[c] = ld_field<double2>(src + ((size_t)(3 * spin + c) * Vh + ycb) * 16);
      w[c] = ld_field<double2>(src + ((size_t)(6 + 3 * low + c) * Vh + ycb) * 16);
    }
    Link<double> U, W;
    LinkIO<P64, R>::load(a.gauge, Vh, mu, back ? 1 - par : par, back ? ycb : cb, U);
    C<double> h[3], p[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double lr = im ? -w[c].y : w[c].x, li = im ? w[c].x : w[c].y;
      h[c] = C<double>{u[c].x + neg_if(lr, minus), u[c].y + neg_if(li, minus)};
    }
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int c = 0; c < 3; ++c)
        W.m[r][c] = C<double>{back ? U.m[c][r].r : U.m[r][c].r, back ? -U.m[c][r].i : U.m[r][c].i};
    su3_mv(W, h, p);
    // the boundary sign is exact: it goes into the product
#pragma unroll
    for (int c = 0; c < 3; ++c) v[st][hop][3 * spin + c] = make_double2(neg_if(p[c].r, neg), neg_if(p[c].i, neg));
  }
  __syncwarp();
  const bool mine = l < 12;
  const int k = mine ? l : 0, s = k / 3, c = k - 3 * s;  // output component
  const size_t pb = CloverIO<P64>::parity_bytes(Vh);
  const char* self = FULLM ? (par ? a.in[1] : a.in[0]) : a.self;
  const char* cself = FULLM ? a.clover : a.c_self;
  C<double> acc = {0, 0}, av = {0, 0}, out;
  auto self_at = [&](int e) { return ld_field<double2>(self + ((size_t)e * Vh + cb) * 16); };
  if (self) {
    if (cself) {
      av = row64(cself + par * pb, Vh, cb, k >= 6, k >= 6 ? k - 6 : k, self_at);
    } else {
      const double2 t = self_at(k);
      av = C<double>{t.x, t.y};
    }
  }
  const bool low = s >= 2;
  const int q = s & 1;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int mu = j >> 1;
    const double2 t = v[st][j][3 * (low && mu < 2 ? 1 - q : q) + c];
    const bool plus = ((j & 1) != 0) != dagger;
    const bool im = low && (mu == 0 || mu == 2);
    const bool minus = low && (plus == ((mu == 1 || mu == 2) && q));
    // lower spins: s B^dagger v, with -i v = (v.i, -v.r) for mu = 0, 2
    const double tr = im ? t.y : t.x, ti = im ? -t.x : t.y;
    acc.r += neg_if(tr, minus);
    acc.i += neg_if(ti, minus);
  }
  if (FULLM) {
    const double mk = -a.kappa;
    out = C<double>{fma(mk, acc.r, av.r), fma(mk, acc.i, av.i)};
  } else {
    out = a.s * acc;
    if (self) out = out + av;
    if (a.c_post) {
      if (mine) post[st][k] = make_double2(out.r, out.i);
      __syncwarp();
      out = row64(a.c_post + par * pb, Vh, cb, k >= 6, k >= 6 ? k - 6 : k, [&](int e) { return post[st][e]; });
    }
  }
  if (ok && mine)
    *reinterpret_cast<double2*>((par ? a.out[1] : a.out[0]) + ((size_t)k * Vh + cb) * 16) = make_double2(out.r, out.i);
}

// Up to this many output sites the split form runs. Measured (us, one thread per site ->
// split): M 256 sites 39.7 -> 7.0, 4,096 39.7 -> 18.8, 8,192 39.7 -> 34.1, 12,288 39.9 -> 53.3; hop
// block 128 sites 31.0 -> 6.3, 4,096 31.0 -> 15.5, 8,192 31.0 -> 28.2, 10,368 31.2 -> 36.6: with the
// chip full, its 2 x larger integer and shared-memory work and the 4 idle lanes of the second
// phase cost more than the shorter chain saves.
constexpr int kSplitSites = 8192;

template <int R>
static void launch_split64(bool fullm, const WilsonArg& a, int n, cudaStream_t st) {
  if (fullm) launch_pdl(wilson_split64_kernel<R, true>, (n + 1) / 2, 32, 0, st, a);
  else launch_pdl(wilson_split64_kernel<R, false>, (n + 1) / 2, 32, 0, st, a);
}

// false: not launched (too many sites, or the hopping term is switched off)
inline bool launch_wilson_split64(int recon, bool fullm, const WilsonArg& a, cudaStream_t st) {
  const int n = fullm ? 2 * a.g.Vh : a.g.Vh;
  if (n > kSplitSites || (!fullm && a.s == 0.0)) return false;
  if (recon == 18) launch_split64<18>(fullm, a, n, st);
  else if (recon == 12) launch_split64<12>(fullm, a, n, st);
  else launch_split64<8>(fullm, a, n, st);
  return true;
}

}  // namespace dirac
