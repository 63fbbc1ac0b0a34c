// Improved staggered (asqtad) stencil (Eq. 3), one thread per output site of one
// parity. Read as the anti-Hermitian staggered operator with the phases
// eta_mu(x) = (-1)^(x_0 + ... + x_{mu-1}) applied in the kernel to phase-free links:
//
//   D psi(x) = sum_mu eta_mu(x) [ F_mu(x) psi(x+mu)  - F_mu(x-mu)^dagger  psi(x-mu)
//                                + L_mu(x) psi(x+3mu) - L_mu(x-3mu)^dagger psi(x-3mu) ]
//
// with F the fat links (18 reals, not unitary) and L the long links (18/12/8 reals).
// All hops are odd, so D maps one parity to the other. The kernel computes
//   out_p = a * x_p + b * D_{p,1-p} in_{1-p}
// which covers the hopping block (a = 0), M = m - D/2 per parity and the second half
// of the even-site normal operator m^2 - 1/4 D_eo D_oe.
#include "field.cuh"
#include "internal.h"

namespace dirac {

struct StagArg {
  char* out;             // half-field of parity out_parity
  const char* in;        // half-field of parity 1 - out_parity
  const char* x;         // half-field of parity out_parity for the a*x term, or null
  const char* fat;
  const char* lng;
  Geom g;
  int out_parity;
  double a, b;
};

__device__ __forceinline__ int stag_shift(int v, int n, int L, int& wraps) {
  v += n;
  wraps = 0;
  while (v >= L) { v -= L; ++wraps; }
  while (v < 0) { v += L; ++wraps; }
  return v;
}

// A neighbour spinor and the factor its link product is multiplied by: with FP16 storage
// the per-site norm is left out of the 6 values and folded into that factor.
template <int PREC, typename T>
__device__ __forceinline__ T load_stag_spinor(const char* src, int Vh, int cb, T v[6]) {
  if constexpr (PREC == P16) {
    return SpinorIO<P16, 6>::load_raw(src, Vh, cb, v);
  } else {
    SpinorIO<PREC, 6>::load(src, Vh, cb, v);
    return (T)1;
  }
}

// ---------------------------------------------------------------- 16-bit hops
// r = U chi (dag: U^dagger chi) from stored binary16 values: a link of R = 18 reals (all
// 9 entries, one complex per word, row-major) or R = 12 (rows 0 and 1; row 2 =
// conj(row0 x row1) is rebuilt in FP32) and a binary16 colour vector (3 words). Products
// of two binary16 values are exact, so each term is one fma.rn.f32.f16 into the FP32
// accumulator; only row 2 of a 12-real link needs the vector in FP32.
template <int R>
__device__ __forceinline__ void stag_mv_h(const uint32_t* uw, const uint32_t chi[3], bool dag, C<float> r[3]) {
  constexpr int NR = R / 6;  // rows stored
  uint32_t nchi[3];
#pragma unroll
  for (int b = 0; b < 3; ++b) nchi[b] = chi[b] ^ 0x80008000u;
#pragma unroll
  for (int a = 0; a < 3; ++a) r[a] = C<float>{0.f, 0.f};
  if (!dag) {
#pragma unroll
    for (int a = 0; a < NR; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const uint32_t u = uw[3 * a + b];
        r[a].r = fma_hh<1, 1>(u, nchi[b], fma_hh<0, 0>(u, chi[b], r[a].r));
        r[a].i = fma_hh<1, 0>(u, chi[b], fma_hh<0, 1>(u, chi[b], r[a].i));
      }
  } else {
#pragma unroll
    for (int b = 0; b < NR; ++b)
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const uint32_t u = uw[3 * b + a];
        r[a].r = fma_hh<1, 1>(u, chi[b], fma_hh<0, 0>(u, chi[b], r[a].r));
        r[a].i = fma_hh<1, 0>(u, nchi[b], fma_hh<0, 1>(u, chi[b], r[a].i));
      }
  }
  if constexpr (R == 12) {
    // row 2: c_j = conj(a_p b_q - a_q b_p), p = j + 1, q = j + 2 (mod 3), a / b rows 0 / 1
    C<float> c[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const int p = (j + 1) % 3, q = (j + 2) % 3;
      const uint32_t ap = uw[p], aq = uw[q], bp = uw[3 + p], bq = uw[3 + q];
      const uint32_t nap = ap ^ 0x80008000u, naq = aq ^ 0x80008000u;
      float cr = fma_hh<0, 0>(ap, bq, 0.f);
      cr = fma_hh<1, 1>(nap, bq, cr);
      cr = fma_hh<0, 0>(naq, bp, cr);
      cr = fma_hh<1, 1>(aq, bp, cr);
      float ci = fma_hh<0, 1>(ap, bq, 0.f);
      ci = fma_hh<1, 0>(ap, bq, ci);
      ci = fma_hh<0, 1>(naq, bp, ci);
      ci = fma_hh<1, 0>(naq, bp, ci);
      c[j] = C<float>{cr, -ci};
    }
    C<float> x[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&chi[b]));
      x[b] = C<float>{f.x, f.y};
    }
    if (!dag) {
#pragma unroll
      for (int b = 0; b < 3; ++b) cmac(r[2], c[b], x[b]);
    } else {
#pragma unroll
      for (int a = 0; a < 3; ++a) cmacc(r[a], c[a], x[2]);
    }
  }
}

// a 16-bit colour vector (3 binary16 words) and its norm
__device__ __forceinline__ float load_stag_h(const char* src, int Vh, int cb, uint32_t chi[3]) {
#pragma unroll
  for (int k = 0; k < 3; ++k) chi[k] = ld_field<uint32_t>(chunk_at<4>(src, k, Vh, cb));
  return ld_field<float>(chunk_at<4>(src, 3, Vh, cb));
}
// the stored words of a 16-bit link with R = 18 (9 words) or 12 (6 words) reals
template <int R>
__device__ __forceinline__ void load_link_h(const char* base, int Vh, int mu, int par, int cb, uint32_t uw[9]) {
  const char* plane = base + (size_t)(mu * 2 + par) * link_plane_bytes(R, 2, Vh);
  if constexpr (R == 18) {
#pragma unroll
    for (int k = 0; k < 9; ++k) uw[k] = __ldg(reinterpret_cast<const uint32_t*>(plane + ((size_t)k * Vh + cb) * 4));
  } else {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const uint2 q = __ldg(reinterpret_cast<const uint2*>(plane + ((size_t)k * Vh + cb) * 8));
      uw[2 * k] = q.x;
      uw[2 * k + 1] = q.y;
    }
  }
}

// One hop: acc += f r, with r the link product of the neighbour n mu (n = +-1: fat link,
// +-3: long link) and f its phase, boundary sign and (16-bit storage) norm.
template <int PREC, int RL, bool LONG, bool BACK, typename T>
__device__ __forceinline__ void stag_hop(const StagArg& a, const int x[4], int cb, int mu, T eta, C<T> r[3], T& f) {
  const Geom& g = a.g;
  const int Vh = g.Vh, par = a.out_parity;
  constexpr int n = (BACK ? -1 : 1) * (LONG ? 3 : 1);
  const char* links = LONG ? a.lng : a.fat;
  int v = 0, L = 1, stride = 1;  // selects: mu may differ from lane to lane
#pragma unroll
  for (int nu = 0, s = g.Lxh; nu < 4; ++nu) {
    if (nu == mu) {
      v = x[nu];
      L = g.L[nu];
      stride = s;
    }
    if (nu > 0) s *= g.L[nu];
  }
  int w;
  const int y = stag_shift(v, n, L, w);
  const int ycb = mu == 0 ? cb + (y >> 1) - (v >> 1) : cb + (y - v) * stride;
  const T bc = (mu == 3 && g.apbc && (w & 1)) ? (T)-1 : (T)1;
  // forward: link at x; backward: link (adjoint) at the neighbour
  const int lpar = BACK ? 1 - par : par, lcb = BACK ? ycb : cb;
  constexpr int RR = LONG ? RL : 18;
  T nrm;
  if constexpr (PREC == P16 && RL != 8) {
    uint32_t chi[3], uw[9];
    nrm = load_stag_h(a.in, Vh, ycb, chi);
    load_link_h<RR>(links, Vh, mu, lpar, lcb, uw);
    stag_mv_h<RR>(uw, chi, BACK, r);
  } else {
    T q[6];
    nrm = load_stag_spinor<PREC, T>(a.in, Vh, ycb, q);
    const C<T> h[3] = {{q[0], q[1]}, {q[2], q[3]}, {q[4], q[5]}};
    Link<T> U;
    LinkIO<PREC, RR>::load(links, Vh, mu, lpar, lcb, U);
    if (BACK) su3_mv_dag(U, h, r);
    else su3_mv(U, h, r);
  }
  f = (BACK ? -eta : eta) * bc * nrm;
}

// LANES = 1: a thread per output site. LANES = 4: the four directions of a site on four
// neighbouring lanes; the sum passes from lane to lane in the order of LANES = 1, so the
// results are the same bits. A small lattice is bound by the latency of a thread's 16 hops
// (2 to 3 of them in flight), which four lanes share.
// Nine CTAs per SM of the one-lane FP32 / FP16 form (56 registers; 18 reals spill two to
// four): the loads in flight are what the warps hold. Left to itself the compiler takes 64 to
// 72. Two launches, us, unset -> 9: 48^3x96 12-real FP32 1616 -> 1568 (10 CTAs 1555 to 1559),
// FP16 1009 -> 965 (10: 972); 24^4 18-real FP32 92 -> 63, FP16 47 -> 35 (10: 37).
template <int PREC, int LANES> constexpr int kStagCtas = PREC != P64 && LANES == 1 ? 9 : 0;
template <int PREC, int RL, int LANES>
__global__ void __launch_bounds__(128, (kStagCtas<PREC, LANES>)) staggered_kernel(const StagArg a) {
  pdl_begin();
  using T = typename Real<PREC>::T;
  const Geom& g = a.g;
  const int Vh = g.Vh;
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = LANES == 1 ? 0 : threadIdx.x % LANES;
  int cb = LANES == 1 ? idx : idx / LANES;
  const bool ok = cb < Vh;
  if (LANES == 1 && !ok) return;
  if (!ok) cb = Vh - 1;  // lanes past the end keep their warp's exchange whole
  const int par = a.out_parity;
  int x[4];
  cb_coords(g, cb, par, x);
  C<T> acc[3] = {{0, 0}, {0, 0}, {0, 0}};
  if constexpr (LANES == 1) {
    int esum = 0;
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
      const T eta = (esum & 1) ? (T)-1 : (T)1;
      esum += x[mu];
      C<T> r[3];
      T f;
      auto add = [&] {
#pragma unroll
        for (int c = 0; c < 3; ++c) acc[c] = C<T>{fma(f, r[c].r, acc[c].r), fma(f, r[c].i, acc[c].i)};
      };
      stag_hop<PREC, RL, false, false, T>(a, x, cb, mu, eta, r, f);
      add();
      stag_hop<PREC, RL, false, true, T>(a, x, cb, mu, eta, r, f);
      add();
      stag_hop<PREC, RL, true, false, T>(a, x, cb, mu, eta, r, f);
      add();
      stag_hop<PREC, RL, true, true, T>(a, x, cb, mu, eta, r, f);
      add();
    }
  } else {
    int esum = 0;
#pragma unroll
    for (int nu = 0; nu < 3; ++nu) esum += nu < lane ? x[nu] : 0;
    const T eta = (esum & 1) ? (T)-1 : (T)1;
    C<T> r[4][3];
    T f[4];
    stag_hop<PREC, RL, false, false, T>(a, x, cb, lane, eta, r[0], f[0]);
    stag_hop<PREC, RL, false, true, T>(a, x, cb, lane, eta, r[1], f[1]);
    stag_hop<PREC, RL, true, false, T>(a, x, cb, lane, eta, r[2], f[2]);
    stag_hop<PREC, RL, true, true, T>(a, x, cb, lane, eta, r[3], f[3]);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      if (lane == m) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
          for (int c = 0; c < 3; ++c)
            acc[c] = C<T>{fma(f[k], r[k][c].r, acc[c].r), fma(f[k], r[k][c].i, acc[c].i)};
      }
      if (m < 3) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const T pr = __shfl_up_sync(0xffffffffu, acc[c].r, 1, LANES);
          const T pi = __shfl_up_sync(0xffffffffu, acc[c].i, 1, LANES);
          if (lane == m + 1) acc[c] = C<T>{pr, pi};
        }
      }
    }
    if (lane != LANES - 1 || !ok) return;
  }
  T out[6];
  const T bb = (T)a.b;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    out[2 * c] = bb * acc[c].r;
    out[2 * c + 1] = bb * acc[c].i;
  }
  if (a.x) {
    T s[6];
    SpinorIO<PREC, 6>::load(a.x, Vh, cb, s);
    const T aa = (T)a.a;
#pragma unroll
    for (int k = 0; k < 6; ++k) out[k] = fma(aa, s[k], out[k]);
  }
  SpinorIO<PREC, 6>::store(a.out, Vh, cb, out);
}

template <int PREC, int LANES>
static void launch_stag_lanes(int recon, const StagArg& a, cudaStream_t st) {
  const int per = 128 / LANES;
  dim3 block(128), grid((a.g.Vh + per - 1) / per);
  if (recon == 18) launch_pdl(staggered_kernel<PREC, 18, LANES>, grid, block, 0, st, a);
  else if (recon == 12) launch_pdl(staggered_kernel<PREC, 12, LANES>, grid, block, 0, st, a);
  else launch_pdl(staggered_kernel<PREC, 8, LANES>, grid, block, 0, st, a);
}

// Up to this many output sites four lanes share a site. Measured (two launches, us, one lane
// -> four): FP32 4,096 sites 10.4 -> 8.1, 13,824 11.2 -> 8.3, 16,384 10.6 -> 9.7, 32,768 12.2 ->
// 18.3; FP16 13,824 11.7 -> 8.3, 32,768 12.6 -> 11.3; FP64 4,096 53 -> 21, 8,192 53 -> 39, 13,824
// 54.4 -> 55.3.
template <int PREC> constexpr int kStagSplitSites = PREC == P64 ? 8192 : 16384;

template <int PREC>
static void launch_stag_prec(int recon, const StagArg& a, cudaStream_t st) {
  if (a.g.Vh <= kStagSplitSites<PREC>) launch_stag_lanes<PREC, 4>(recon, a, st);
  else launch_stag_lanes<PREC, 1>(recon, a, st);
}

void launch_staggered(int prec, int recon, char* out, const char* in, const char* x,
                      const char* fat, const char* lng, const Geom& g, int out_parity, double a,
                      double b, cudaStream_t st) {
  StagArg arg{out, in, x, fat, lng, g, out_parity, a, b};
  if (prec == P64) launch_stag_prec<P64>(recon, arg, st);
  else if (prec == P32) launch_stag_prec<P32>(recon, arg, st);
  else launch_stag_prec<P16>(recon, arg, st);
}

}  // namespace dirac
