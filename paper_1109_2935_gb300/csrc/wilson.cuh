// Wilson-clover stencil (Eq. 2), one thread per output site.
//
//   hopping term  D psi(x) = sum_mu [ (1 - gamma_mu) U_mu(x) psi(x+mu)
//                                     + (1 + gamma_mu) U_mu(x-mu)^dagger psi(x-mu) ]
//   kappa form    M psi    = Ahat psi - kappa D psi,  Ahat = 1 + 2 kappa A  (stored)
//   adjoint       M^dagger = Ahat - kappa D^dagger, D^dagger swaps the projectors.
//
// Spin basis: chiral, gamma_mu = [[0, B_mu], [B_mu^dagger, 0]] with
//   B_x = [[0, i], [i, 0]], B_y = [[0, -1], [1, 0]], B_z = [[i, 0], [0, -i]], B_t = 1.
// For P = 1 + s gamma_mu (s = -1 forward, +1 backward; flipped for the adjoint):
//   P psi = [h ; s B^dagger h]  with  h = psi_up + s B psi_low,
// so every hop multiplies only the 2-spin half spinor h by the link (Sec. 5:
// "similarity transforms to increase the sparsity of the Dirac matrices").
#pragma once
#include "field.cuh"

namespace dirac {

struct WilsonArg {
  char* out[2];          // output half-field base for each parity
  const char* in[2];     // input half-field base for each parity
  const char* gauge;     // links of this precision, [mu][parity][chunk][Vh]
  const char* clover;    // Ahat of this precision, [parity][chunk][Vh]; null: Ahat = 1
  Geom g;
  double kappa;
  int dagger;            // 1: apply the adjoint
  int out_parity;        // hop mode: parity of the output half-field
  // hop mode: out_p = Cpost (Cself self_p + s D_{p,1-p} in_{1-p}); a null matrix is the
  // identity, a null self drops that term, s = 0 skips the hopping term. Cself / Cpost
  // are clover-format fields ([parity][chunk][Vh]: Ahat or Ahat^-1).
  const char* self = nullptr;
  const char* c_self = nullptr;
  const char* c_post = nullptr;
  double s = 1.0;
};

// A neighbour spinor for wilson_hop and the factor that multiplies its projection: with
// FP16 storage the per-site norm is left out of the 24 values and folded into that
// factor (one multiply per projected component instead of one per stored value).
template <int PREC, typename T>
__device__ __forceinline__ T load_hop_spinor(const char* src, int Vh, int cb, T psi[24], T bc) {
  if constexpr (PREC == P16) {
    return bc * SpinorIO<P16, 24>::load_raw(src, Vh, cb, psi);
  } else {
    SpinorIO<PREC, 24>::load(src, Vh, cb, psi);
    return bc;
  }
}

// The spin projection of one hop: h = psi_up + s B_mu psi_low (two spin components,
// 3 colours each). Shared by the stencil and by the face packing of the domain
// decomposition, so that a projected face equals the stencil's own projection bit for bit.
template <int MU, typename T>
__device__ __forceinline__ void wilson_project(const T* psi, T s, C<T> h0[3], C<T> h1[3]) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    C<T> u0 = {psi[2 * c], psi[2 * c + 1]};
    C<T> u1 = {psi[6 + 2 * c], psi[6 + 2 * c + 1]};
    C<T> l0 = {psi[12 + 2 * c], psi[12 + 2 * c + 1]};
    C<T> l1 = {psi[18 + 2 * c], psi[18 + 2 * c + 1]};
    if (MU == 0) {        // B l = (i l1, i l0)
      h0[c] = u0 + s * times_i(l1);
      h1[c] = u1 + s * times_i(l0);
    } else if (MU == 1) { // B l = (-l1, l0)
      h0[c] = u0 - s * l1;
      h1[c] = u1 + s * l0;
    } else if (MU == 2) { // B l = (i l0, -i l1)
      h0[c] = u0 + s * times_i(l0);
      h1[c] = u1 - s * times_i(l1);
    } else {              // B l = l
      h0[c] = u0 + s * l0;
      h1[c] = u1 + s * l1;
    }
  }
}

// wilson_hop_proj in FP32: the two spin components of the half spinor meet the same link,
// so they ride in the two lanes of packed instructions (the same roundings, fewer issue
// slots: FP16 M at 24^3x128 141 -> 137 us, FP32 M 192 -> 190 us).
template <int MU>
__device__ __forceinline__ void wilson_hop_pair(C<float> acc[4][3], const C<float> h0[3], const C<float> h1[3],
                                                const Link<float>& U, bool link_dag, float s, float bc) {
  C2 h[3], v[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) h[c] = pair2(h0[c], h1[c]);
  if (link_dag) su3_mv2<true>(U, h, v);
  else su3_mv2<false>(U, h, v);
  const float ks = s * bc;
  const float2 b2 = dup2(bc), k2 = dup2(ks), x2 = make_float2(ks, -ks), y2 = make_float2(-ks, ks);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    C2 up = pair2(acc[0][c], acc[1][c]);
    up.r = __ffma2_rn(b2, v[c].r, up.r);
    up.i = __ffma2_rn(b2, v[c].i, up.i);
    acc[0][c] = C<float>{up.r.x, up.i.x};
    acc[1][c] = C<float>{up.r.y, up.i.y};
    if (MU == 0) {        // B^dagger v = (-i v1, -i v0)
      acc[2][c] = C<float>{fmaf(ks, v[c].i.y, acc[2][c].r), fmaf(-ks, v[c].r.y, acc[2][c].i)};
      acc[3][c] = C<float>{fmaf(ks, v[c].i.x, acc[3][c].r), fmaf(-ks, v[c].r.x, acc[3][c].i)};
    } else if (MU == 1) { // B^dagger v = (v1, -v0)
      acc[2][c] = C<float>{fmaf(ks, v[c].r.y, acc[2][c].r), fmaf(ks, v[c].i.y, acc[2][c].i)};
      acc[3][c] = C<float>{fmaf(-ks, v[c].r.x, acc[3][c].r), fmaf(-ks, v[c].i.x, acc[3][c].i)};
    } else {
      C2 lo = pair2(acc[2][c], acc[3][c]);
      if (MU == 2) {      // B^dagger v = (-i v0, i v1)
        lo.r = __ffma2_rn(x2, v[c].i, lo.r);
        lo.i = __ffma2_rn(y2, v[c].r, lo.i);
      } else {
        lo.r = __ffma2_rn(k2, v[c].r, lo.r);
        lo.i = __ffma2_rn(k2, v[c].i, lo.i);
      }
      acc[2][c] = C<float>{lo.r.x, lo.i.x};
      acc[3][c] = C<float>{lo.r.y, lo.i.y};
    }
  }
}

// The rest of a hop after the projection: v = U h (U^dagger h for a backward hop), then
// acc += bc P-reconstruction of v.
template <int MU, typename T>
__device__ __forceinline__ void wilson_hop_proj(C<T> acc[4][3], const C<T> h0[3], const C<T> h1[3],
                                                const Link<T>& U, bool link_dag, T s, T bc) {
  C<T> v0[3], v1[3];
  if constexpr (std::is_same<T, float>::value) {
    wilson_hop_pair<MU>(acc, h0, h1, U, link_dag, s, bc);
    return;
  }
  if (link_dag) {
    su3_mv_dag(U, h0, v0);
    su3_mv_dag(U, h1, v1);
  } else {
    su3_mv(U, h0, v0);
    su3_mv(U, h1, v1);
  }
  // the hop's factor bc multiplies the accumulation (one fused multiply-add per real);
  // with bc = +-1 (FP32 / FP64 storage) this is exactly acc +- v
  const T ks = s * bc;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    acc[0][c] = C<T>{fma(bc, v0[c].r, acc[0][c].r), fma(bc, v0[c].i, acc[0][c].i)};
    acc[1][c] = C<T>{fma(bc, v1[c].r, acc[1][c].r), fma(bc, v1[c].i, acc[1][c].i)};
    if (MU == 0) {        // B^dagger v = (-i v1, -i v0)
      acc[2][c] = C<T>{fma(ks, v1[c].i, acc[2][c].r), fma(-ks, v1[c].r, acc[2][c].i)};
      acc[3][c] = C<T>{fma(ks, v0[c].i, acc[3][c].r), fma(-ks, v0[c].r, acc[3][c].i)};
    } else if (MU == 1) { // B^dagger v = (v1, -v0)
      acc[2][c] = C<T>{fma(ks, v1[c].r, acc[2][c].r), fma(ks, v1[c].i, acc[2][c].i)};
      acc[3][c] = C<T>{fma(-ks, v0[c].r, acc[3][c].r), fma(-ks, v0[c].i, acc[3][c].i)};
    } else if (MU == 2) { // B^dagger v = (-i v0, i v1)
      acc[2][c] = C<T>{fma(ks, v0[c].i, acc[2][c].r), fma(-ks, v0[c].r, acc[2][c].i)};
      acc[3][c] = C<T>{fma(-ks, v1[c].i, acc[3][c].r), fma(ks, v1[c].r, acc[3][c].i)};
    } else {
      acc[2][c] = C<T>{fma(ks, v0[c].r, acc[2][c].r), fma(ks, v0[c].i, acc[2][c].i)};
      acc[3][c] = C<T>{fma(ks, v1[c].r, acc[3][c].r), fma(ks, v1[c].i, acc[3][c].i)};
    }
  }
}

template <int MU, typename T>
__device__ __forceinline__ void wilson_hop(C<T> acc[4][3], const T* psi, const Link<T>& U,
                                           bool link_dag, T s, T bc) {
  C<T> h0[3], h1[3];
  wilson_project<MU, T>(psi, s, h0, h1);
  wilson_hop_proj<MU, T>(acc, h0, h1, U, link_dag, s, bc);
}

// out[12] = Ahat(x) in[12] for the clover of precision PREC (block by block to bound
// register use).
template <int PREC, typename T>
__device__ __forceinline__ void apply_clover_site(const char* b, int Vh, int cb, const C<T> in[12],
                                                  C<T> out[12]) {
  if constexpr (PREC == P64 || PREC == P64DS) {
#pragma unroll
    for (int blk = 0; blk < 2; ++blk) {
      T v[36];
#pragma unroll
      for (int k = 0; k < 18; ++k) {
        double2 q = ldg_chunk<double2>(chunk_at<16>(b, (18 * blk + k), Vh, cb));
        v[2 * k] = T(q.x); v[2 * k + 1] = T(q.y);
      }
      herm6_mv<T>(v, in + 6 * blk, out + 6 * blk);
    }
  } else if constexpr (PREC == P32) {
#pragma unroll
    for (int blk = 0; blk < 2; ++blk) {
      float v[36];
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        float4 q = ldg_chunk<float4>(chunk_at<16>(b, (9 * blk + k), Vh, cb));
        v[4 * k] = q.x; v[4 * k + 1] = q.y; v[4 * k + 2] = q.z; v[4 * k + 3] = q.w;
      }
      herm6_mv<T>(v, in + 6 * blk, out + 6 * blk);
    }
  } else {
    // 16-bit clover: the stored values times the per-site norm, which scales the 12
    // input components instead of the 72 entries
    float v[72];
    const float n = CloverIO<P16>::load_raw(b, Vh, cb, v);
    C<T> x[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) x[k] = n * in[k];
    herm6_mv<T>(v, x, out);
    herm6_mv<T>(v + 36, x + 6, out + 6);
  }
}

// ---------------------------------------------------------------- 16-bit Ahat x self
// y = A x for one chirality block with the stored binary16 values of both: blk = the
// block's 18 half2 words (6 real diagonal entries in words 0..2, then L_ij, i > j, one
// complex per word), x = 6 complex binary16 words (re low, im high).
__device__ __forceinline__ void herm6_hh(const uint32_t blk[18], const uint32_t x[6], C<float> y[6]) {
  uint32_t nx[6];  // (-re, -im)
#pragma unroll
  for (int i = 0; i < 6; ++i) nx[i] = x[i] ^ 0x80008000u;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const uint32_t d = blk[i >> 1];
    if (i & 1) y[i] = C<float>{fma_hh<1, 0>(d, x[i], 0.f), fma_hh<1, 1>(d, x[i], 0.f)};
    else y[i] = C<float>{fma_hh<0, 0>(d, x[i], 0.f), fma_hh<0, 1>(d, x[i], 0.f)};
  }
  int w = 3;
#pragma unroll
  for (int i = 1; i < 6; ++i) {
#pragma unroll
    for (int j = 0; j < i; ++j) {
      const uint32_t l = blk[w++];
      // y_i += L x_j
      y[i].r = fma_hh<1, 1>(l, nx[j], fma_hh<0, 0>(l, x[j], y[i].r));
      y[i].i = fma_hh<1, 0>(l, x[j], fma_hh<0, 1>(l, x[j], y[i].i));
      // y_j += conj(L) x_i
      y[j].r = fma_hh<1, 1>(l, x[i], fma_hh<0, 0>(l, x[i], y[j].r));
      y[j].i = fma_hh<1, 0>(l, nx[i], fma_hh<0, 1>(l, x[i], y[j].i));
    }
  }
}

// av = Ahat self for 16-bit storage, from the stored binary16 values of the clover and of
// the site's own spinor; their two per-site norms scale the 12 results once.
__device__ __forceinline__ void clover_self_h(const char* clov, const char* self, int Vh, int cb, C<float> av[12]) {
  const float nc = __ldg(reinterpret_cast<const float*>(clov + (size_t)144 * Vh) + cb);
  const float ns = ld_field<float>(chunk_at<4>(self, 12, Vh, cb));
  uint32_t x[12];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int4 q = ld_field<int4>(chunk_at<16>(self, k, Vh, cb));
    x[4 * k] = (uint32_t)q.x; x[4 * k + 1] = (uint32_t)q.y; x[4 * k + 2] = (uint32_t)q.z; x[4 * k + 3] = (uint32_t)q.w;
  }
  // block 0: words 0..17 (chunks 0..3 and half of chunk 4); block 1: words 18..35
  uint32_t c[20];
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const int4 q = ldg_chunk<int4>(chunk_at<16>(clov, k, Vh, cb));
    c[4 * k] = (uint32_t)q.x; c[4 * k + 1] = (uint32_t)q.y; c[4 * k + 2] = (uint32_t)q.z; c[4 * k + 3] = (uint32_t)q.w;
  }
  herm6_hh(c, x, av);
  c[0] = c[18];
  c[1] = c[19];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int4 q = ldg_chunk<int4>(chunk_at<16>(clov, (5 + k), Vh, cb));
    c[2 + 4 * k] = (uint32_t)q.x; c[3 + 4 * k] = (uint32_t)q.y; c[4 + 4 * k] = (uint32_t)q.z; c[5 + 4 * k] = (uint32_t)q.w;
  }
  herm6_hh(c, x + 6, av + 6);
  const float n = nc * ns;
#pragma unroll
  for (int k = 0; k < 12; ++k) av[k] = n * av[k];
}

// ---------------------------------------------------------------- 16-bit neighbours
// A 16-bit neighbour spinor for a hop: the upper two spin components converted (u, 12
// reals), the lower two kept as binary16 pairs (l, 6 words: spin 2 colours 0..2, spin 3
// colours 0..2, re low / im high); returns bc times the site norm, the hop's factor.
__device__ __forceinline__ float load_hop_h(const char* src, int Vh, int cb, float u[12], uint32_t l[6], float bc) {
  const float n = ld_field<float>(chunk_at<4>(src, 12, Vh, cb));
  uint32_t w[12];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int4 q = ld_field<int4>(chunk_at<16>(src, k, Vh, cb));
    w[4 * k] = (uint32_t)q.x; w[4 * k + 1] = (uint32_t)q.y; w[4 * k + 2] = (uint32_t)q.z; w[4 * k + 3] = (uint32_t)q.w;
  }
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[k]));
    u[2 * k] = f.x;
    u[2 * k + 1] = f.y;
    l[k] = w[6 + k];
  }
  return bc * n;
}

// The projection of wilson_project with binary16 lower components: each real is one
// fma of (s or -s) times a binary16 value into the FP32 upper value (sw: s in the low
// half, -s in the high half). s = +-1, so the result is round(u +- l), as in FP32.
template <int MU>
__device__ __forceinline__ void wilson_project_h(const float u[12], const uint32_t l[6], uint32_t sw,
                                                 C<float> h0[3], C<float> h1[3]) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float u0r = u[2 * c], u0i = u[2 * c + 1], u1r = u[6 + 2 * c], u1i = u[7 + 2 * c];
    const uint32_t l0 = l[c], l1 = l[3 + c];
    if (MU == 0) {        // h = u + s (i l1, i l0)
      h0[c] = C<float>{fma_hh<1, 1>(sw, l1, u0r), fma_hh<0, 0>(sw, l1, u0i)};
      h1[c] = C<float>{fma_hh<1, 1>(sw, l0, u1r), fma_hh<0, 0>(sw, l0, u1i)};
    } else if (MU == 1) { // h = u + s (-l1, l0)
      h0[c] = C<float>{fma_hh<1, 0>(sw, l1, u0r), fma_hh<1, 1>(sw, l1, u0i)};
      h1[c] = C<float>{fma_hh<0, 0>(sw, l0, u1r), fma_hh<0, 1>(sw, l0, u1i)};
    } else if (MU == 2) { // h = u + s (i l0, -i l1)
      h0[c] = C<float>{fma_hh<1, 1>(sw, l0, u0r), fma_hh<0, 0>(sw, l0, u0i)};
      h1[c] = C<float>{fma_hh<0, 1>(sw, l1, u1r), fma_hh<1, 0>(sw, l1, u1i)};
    } else {              // h = u + s l
      h0[c] = C<float>{fma_hh<0, 0>(sw, l0, u0r), fma_hh<0, 1>(sw, l0, u0i)};
      h1[c] = C<float>{fma_hh<0, 0>(sw, l1, u1r), fma_hh<0, 1>(sw, l1, u1i)};
    }
  }
}
__device__ __forceinline__ uint32_t signs_h(float s) { return s > 0.f ? 0xBC003C00u : 0x3C00BC00u; }

template <int MU>
__device__ __forceinline__ void wilson_hop_h(C<float> acc[4][3], const float u[12], const uint32_t l[6],
                                             const Link<float>& U, bool link_dag, float s, float bc) {
  C<float> h0[3], h1[3];
  wilson_project_h<MU>(u, l, signs_h(s), h0, h1);
  wilson_hop_proj<MU, float>(acc, h0, h1, U, link_dag, s, bc);
}

// Launch shape per storage precision (threads per CTA, minimum resident CTAs per SM,
// which caps registers). FP32/FP16 are memory-latency bound and want many warps in
// flight, each with as many loads in flight as its registers hold; FP64 is FP64-ALU bound on
// this part. Measured on GB300 at 24^3x128 (clover M): FP16 64 x 8 (128-register cap)
// 135.2 us, 64 x 10 139.3, 64 x 12 138.6; FP32 64 x 8 190.6 us, before the packed arithmetic
// 199 us against 288 us for 128 x 1 (up to 255 registers).
template <int PREC> struct WilsonShape { static constexpr int threads = 64, minb = 8; };
template <> struct WilsonShape<P64> { static constexpr int threads = 128, minb = 1; };
template <> struct WilsonShape<P64DS> { static constexpr int threads = 128, minb = 2; };

// Output site idx of the full operator. The two parities alternate every 32 threads (a
// warp): the forward link U_mu(x) read by site x is read again as a backward link by the
// neighbour x + mu of the other parity close in time, so it comes from cache instead of a
// second DRAM pass over all links. The parity is made warp-uniform (all lanes enter), so
// that the field and link planes of a thread are uniform addresses. full_sites: the number
// of idx values, idle ones of a ragged last warp (cb >= Vh) included.
__host__ __device__ __forceinline__ int full_sites(int Vh) { return (Vh + 31) / 32 * 64; }
__device__ __forceinline__ void full_site(int idx, int& par, int& cb) {
  const int w = __shfl_sync(0xffffffffu, idx >> 5, 0);
  par = w & 1;
  cb = (w >> 1) * 32 + (idx & 31);
}

// out = Ahat self - kappa acc for N right-hand sides of one site, chirality block by block:
// a block's clover is loaded once for all of them. acc is overwritten with the result.
template <int PREC, int N>
__device__ __forceinline__ void clover_site_n(const char* clov, const char* self, size_t stride, int Vh, int cb,
                                              float mk, C<float> acc[N][4][3]) {
#pragma unroll
  for (int blk = 0; blk < 2; ++blk) {
    if constexpr (PREC == P16) {
      uint32_t c[20];
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        const int4 q = ldg_chunk<int4>(chunk_at<16>(clov, 4 * blk + k, Vh, cb));
        c[4 * k] = (uint32_t)q.x; c[4 * k + 1] = (uint32_t)q.y; c[4 * k + 2] = (uint32_t)q.z; c[4 * k + 3] = (uint32_t)q.w;
      }
      const float nc = __ldg(reinterpret_cast<const float*>(chunk_at<4>(clov, 36, Vh, cb)));
#pragma unroll
      for (int r = 0; r < N; ++r) {
        const char* s = self + r * stride;
        uint32_t x[8];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const int4 q = ld_field<int4>(chunk_at<16>(s, blk + k, Vh, cb));
          x[4 * k] = (uint32_t)q.x; x[4 * k + 1] = (uint32_t)q.y; x[4 * k + 2] = (uint32_t)q.z; x[4 * k + 3] = (uint32_t)q.w;
        }
        const float n = nc * ld_field<float>(chunk_at<4>(s, 12, Vh, cb));
        C<float> y[6];
        herm6_hh(c + 2 * blk, x + 2 * blk, y);
#pragma unroll
        for (int k = 0; k < 6; ++k) {
          C<float>& o = acc[r][2 * blk + k / 3][k % 3];
          o = C<float>{fmaf(mk, o.r, n * y[k].r), fmaf(mk, o.i, n * y[k].i)};
        }
      }
    } else {
      float v[36];
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        const float4 q = ldg_chunk<float4>(chunk_at<16>(clov, 9 * blk + k, Vh, cb));
        v[4 * k] = q.x; v[4 * k + 1] = q.y; v[4 * k + 2] = q.z; v[4 * k + 3] = q.w;
      }
#pragma unroll
      for (int r = 0; r < N; ++r) {
        C<float> x[6], y[6];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const float4 q = ld_field<float4>(chunk_at<16>(self + r * stride, 3 * blk + k, Vh, cb));
          x[2 * k] = C<float>{q.x, q.y};
          x[2 * k + 1] = C<float>{q.z, q.w};
        }
        herm6_mv<float>(v, x, y);
#pragma unroll
        for (int k = 0; k < 6; ++k) {
          C<float>& o = acc[r][2 * blk + k / 3][k % 3];
          o = C<float>{fmaf(mk, o.r, y[k].r), fmaf(mk, o.i, y[k].i)};
        }
      }
    }
  }
}

// One hop for N right-hand sides: the link is loaded and rebuilt once.
template <int PREC, int R, int N, int MU, typename T>
__device__ __forceinline__ void wilson_hop_n(C<T> acc[N][4][3], const char* src, size_t stride, const char* gauge,
                                             int Vh, int ycb, int lpar, int lcb, bool dag, T s, T bc) {
  if constexpr (PREC == P16) {
    float u[N][12], n[N];
    uint32_t l[N][6];
#pragma unroll
    for (int r = 0; r < N; ++r) n[r] = load_hop_h(src + r * stride, Vh, ycb, u[r], l[r], bc);
    Link<T> U;
    LinkIO<PREC, R>::load(gauge, Vh, MU, lpar, lcb, U);
#pragma unroll
    for (int r = 0; r < N; ++r) wilson_hop_h<MU>(acc[r], u[r], l[r], U, dag, s, n[r]);
  } else {
    T psi[N][24], n[N];
#pragma unroll
    for (int r = 0; r < N; ++r) n[r] = load_hop_spinor<PREC, T>(src + r * stride, Vh, ycb, psi[r], bc);
    Link<T> U;
    LinkIO<PREC, R>::load(gauge, Vh, MU, lpar, lcb, U);
#pragma unroll
    for (int r = 0; r < N; ++r) wilson_hop<MU>(acc[r], psi[r], U, dag, s, n[r]);
  }
}

// FP16 storage, two right-hand sides per thread: the registers of a hop in flight are what
// limits the loads in flight, so the next kRing hops (spinors and link, as stored) travel into
// shared memory by asynchronous copies instead, a ring of slots per warp, each laid out like a
// field of 32 sites. A thread reads only what it copied itself: its own wait is the only
// synchronisation. 3 lattices x 12 right-hand sides 3.01 -> 2.87 ms with 2 slots; 3 and 4 take
// the L1 (3.17, 4.27 ms), and one right-hand side per thread gains nothing (133 us: 143 / 133 /
// 130 with 2 / 3 / 4, small lattices slower).
constexpr int kRing = 2;
template <int R, int N> constexpr int kRingSlot = 32 * (N * 52 + LinkIO<P16, R>::kChunks * LinkIO<P16, R>::kChunkBytes);
// bytes of dynamic shared memory per warp of a kernel with up to N right-hand sides a thread
// (at most 8960: the 4 warps of a CTA stay below the default limit of 48 KB)
template <int PREC, int R, int N> constexpr int kRingWarp = PREC == P16 && N == 2 ? kRing * kRingSlot<R, N> : 0;
template <int PREC, int R, int N> __device__ __forceinline__ char* ring_of_warp(int w) {
  extern __shared__ __align__(16) char ring_smem[];
  return ring_smem + w * kRingWarp<PREC, R, N>;
}
template <int B> __device__ __forceinline__ void copy_async(char* dst, const char* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src), "n"(B) : "memory");
}
template <int R, int N>
__device__ __forceinline__ void ring_request(char* slot, int t, const char* src, size_t stride, const char* plane,
                                             int Vh, int ycb, int lcb) {
  using LIO = LinkIO<P16, R>;
  constexpr int T = 32;
#pragma unroll
  for (int r = 0; r < N; ++r) {
    char* f = slot + r * 52 * T;
#pragma unroll
    for (int k = 0; k < 3; ++k)
      copy_async<16>(const_cast<char*>(chunk_at<16>(f, k, T, t)), chunk_at<16>(src + r * stride, k, Vh, ycb));
    copy_async<4>(const_cast<char*>(chunk_at<4>(f, 12, T, t)), chunk_at<4>(src + r * stride, 12, Vh, ycb));
  }
  char* l = slot + N * 52 * T;
#pragma unroll
  for (int k = 0; k < LIO::kChunks; ++k)
    copy_async<LIO::kChunkBytes>(const_cast<char*>(chunk_at<LIO::kChunkBytes>(l, k, T, t)),
                                 chunk_at<LIO::kChunkBytes>(plane, k, Vh, lcb));
}
template <int R, int N, int MU>
__device__ __forceinline__ void ring_hop(C<float> acc[N][4][3], const char* slot, int t, bool dag, float s, float bc) {
  constexpr int T = 32;
  Link<float> U;
  LinkIO<P16, R>::template load_plane<false>(slot + N * 52 * T, T, t, U);
#pragma unroll
  for (int r = 0; r < N; ++r) {
    float u[12];
    uint32_t l[6];
    const float n = load_hop_h(slot + r * 52 * T, T, t, u, l, bc);
    wilson_hop_h<MU>(acc[r], u, l, U, dag, s, n);
  }
}

// One output site of the stencil: thread index idx over the Vh (hop mode) or full_sites
// (full operator) indices. Shared by the single-RHS, multi-RHS and batched kernels. N > 1
// (FP32 / FP16 full operator): N right-hand sides, `stride` bytes apart, with one load and
// rebuild of every link and one load of the clover; each gets the bits of N = 1.
template <int PREC, int R, bool FULLM, int N = 1>
__device__ __forceinline__ void wilson_site(const WilsonArg& a, int idx, size_t stride = 0, char* ring = nullptr) {
  using T = typename Real<PREC>::T;
  static_assert(N == 1 || (FULLM && (PREC == P32 || PREC == P16)), "");
  const Geom& g = a.g;
  const int Vh = g.Vh;
  int par, cb;
  if (FULLM) {
    full_site(idx, par, cb);
  } else {
    par = a.out_parity;
    cb = idx;
  }
  if (cb >= Vh) return;
  int x[4];
  cb_coords(g, cb, par, x);
  // selects, not a runtime index into the parameter arrays (which would copy them
  // to local memory)
  const char* src = par ? a.in[0] : a.in[1];
  const char* self_in = par ? a.in[1] : a.in[0];
  char* dst = par ? a.out[1] : a.out[0];
  const T sf = a.dagger ? (T)1 : (T)-1;  // forward projector 1 - gamma (adjoint: 1 + gamma)
  const T sb = -sf;

  C<T> acc[N][4][3];
#pragma unroll
  for (int r = 0; r < N; ++r)
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int c = 0; c < 3; ++c) acc[r][s][c] = C<T>{0, 0};

  if constexpr (PREC == P16 && N == 2) {
    const int t = threadIdx.x & 31;
    constexpr int slot_bytes = kRingSlot<R, N>;
    float bc3[2] = {1.f, 1.f};  // the signs of the two t hops
    auto request = [&](int j) {
      const int mu = j >> 1;
      const bool back = j & 1;
      bool edge;
      const int ycb = hop_index(g, x, cb, mu, !back, edge);
      if (mu == 3 && edge && g.apbc) bc3[j & 1] = -1.f;
      const char* plane = a.gauge + (size_t)(mu * 2 + (back ? 1 - par : par)) * link_plane_bytes(R, 2, Vh);
      ring_request<R, N>(ring + (j % kRing) * slot_bytes, t, src, stride, plane, Vh, ycb, back ? ycb : cb);
    };
    {
#pragma unroll
      for (int j = 0; j < kRing; ++j) {
        request(j);
        asm volatile("cp.async.commit_group;" ::: "memory");
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kRing - 1) : "memory");
        const char* slot = ring + (j % kRing) * slot_bytes;
        const T s = (j & 1) ? sb : sf;
        const bool back = j & 1;
        if (j < 2) ring_hop<R, N, 0>(acc, slot, t, back, s, 1.f);
        else if (j < 4) ring_hop<R, N, 1>(acc, slot, t, back, s, 1.f);
        else if (j < 6) ring_hop<R, N, 2>(acc, slot, t, back, s, 1.f);
        else ring_hop<R, N, 3>(acc, slot, t, back, s, bc3[j & 1]);
        if (j + kRing < 8) request(j + kRing);
        asm volatile("cp.async.commit_group;" ::: "memory");
      }
    }
  } else {
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
      if (!FULLM && a.s == 0.0) break;  // hop mode without the hopping term
#pragma unroll
      for (int dir = 0; dir < 2; ++dir) {
        // forward neighbour x + mu with link U_mu(x), stored at (mu, par, cb); backward
        // neighbour x - mu with U_mu(x - mu)^dagger, stored at (mu, 1 - par, cb(x - mu))
        bool edge;
        const int ycb = hop_index(g, x, cb, mu, dir == 0, edge);
        const T bc = (mu == 3 && edge && g.apbc) ? (T)-1 : (T)1;
        const int lpar = dir ? 1 - par : par, lcb = dir ? ycb : cb;
        const T s = dir ? sb : sf;
        if (mu == 0) wilson_hop_n<PREC, R, N, 0, T>(acc, src, stride, a.gauge, Vh, ycb, lpar, lcb, dir == 1, s, bc);
        if (mu == 1) wilson_hop_n<PREC, R, N, 1, T>(acc, src, stride, a.gauge, Vh, ycb, lpar, lcb, dir == 1, s, bc);
        if (mu == 2) wilson_hop_n<PREC, R, N, 2, T>(acc, src, stride, a.gauge, Vh, ycb, lpar, lcb, dir == 1, s, bc);
        if (mu == 3) wilson_hop_n<PREC, R, N, 3, T>(acc, src, stride, a.gauge, Vh, ycb, lpar, lcb, dir == 1, s, bc);
      }
    }
  }

  T out[24];
  if constexpr (FULLM && (PREC == P32 || PREC == P16)) {
    const float mk = -(float)a.kappa;
    if (a.clover)
      clover_site_n<PREC, N>(a.clover + (size_t)par * CloverIO<PREC>::parity_bytes(Vh), self_in, stride, Vh, cb, mk, acc);
#pragma unroll
    for (int r = 0; r < N; ++r) {
      if (!a.clover) {
        float self[24];
        SpinorIO<PREC, 24>::load(self_in + r * stride, Vh, cb, self);
#pragma unroll
        for (int k = 0; k < 12; ++k) {
          C<float>& o = acc[r][k / 3][k % 3];
          o = C<float>{fmaf(mk, o.r, self[2 * k]), fmaf(mk, o.i, self[2 * k + 1])};
        }
      }
#pragma unroll
      for (int k = 0; k < 12; ++k) {
        out[2 * k] = acc[r][k / 3][k % 3].r;
        out[2 * k + 1] = acc[r][k / 3][k % 3].i;
      }
      SpinorIO<PREC, 24>::store(dst + r * stride, Vh, cb, out);
    }
    return;
  } else if constexpr (FULLM) {
    T self[24];
    C<T> sv[12], av[12];
    SpinorIO<PREC, 24>::load(self_in, Vh, cb, self);
#pragma unroll
    for (int k = 0; k < 12; ++k) sv[k] = C<T>{self[2 * k], self[2 * k + 1]};
    if (a.clover) {
      apply_clover_site<PREC, T>(a.clover + (size_t)par * CloverIO<PREC>::parity_bytes(Vh), Vh, cb, sv, av);
    } else {
#pragma unroll
      for (int k = 0; k < 12; ++k) av[k] = sv[k];
    }
    const T mk = -(T)a.kappa;
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        out[6 * s + 2 * c] = fma(mk, acc[0][s][c].r, av[3 * s + c].r);
        out[6 * s + 2 * c + 1] = fma(mk, acc[0][s][c].i, av[3 * s + c].i);
      }
  } else {
    const T sc = (T)a.s;
    C<T> v[12];
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int c = 0; c < 3; ++c) v[3 * s + c] = sc * acc[0][s][c];
    const size_t pb = CloverIO<PREC>::parity_bytes(Vh);
    if (a.self) {
      C<T> cv[12];
      bool done = false;
      if constexpr (PREC == P16) {
        if (a.c_self) {  // Cself self from the stored binary16 values
          clover_self_h(a.c_self + par * pb, a.self, Vh, cb, cv);
          done = true;
        }
      }
      if (!done) {
        T sl[24];
        SpinorIO<PREC, 24>::load(a.self, Vh, cb, sl);
        C<T> sv[12];
#pragma unroll
        for (int k = 0; k < 12; ++k) sv[k] = C<T>{sl[2 * k], sl[2 * k + 1]};
        if (a.c_self) {
          apply_clover_site<PREC, T>(a.c_self + par * pb, Vh, cb, sv, cv);
        } else {
#pragma unroll
          for (int k = 0; k < 12; ++k) cv[k] = sv[k];
        }
      }
#pragma unroll
      for (int k = 0; k < 12; ++k) v[k] = v[k] + cv[k];
    }
    if (a.c_post) {
      C<T> w[12];
      apply_clover_site<PREC, T>(a.c_post + par * pb, Vh, cb, v, w);
#pragma unroll
      for (int k = 0; k < 12; ++k) v[k] = w[k];
    }
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      out[2 * k] = v[k].r;
      out[2 * k + 1] = v[k].i;
    }
  }
  SpinorIO<PREC, 24>::store(dst, Vh, cb, out);
}

template <int PREC, int R, bool FULLM>
__global__ void __launch_bounds__(WilsonShape<PREC>::threads, WilsonShape<PREC>::minb)
    wilson_kernel(const WilsonArg a) {
  pdl_begin();
  wilson_site<PREC, R, FULLM>(a, blockIdx.x * blockDim.x + threadIdx.x);
}

template <int PREC>
void launch_wilson_prec(int recon, bool fullm, const WilsonArg& a, cudaStream_t st) {
  const int n = fullm ? full_sites(a.g.Vh) : a.g.Vh;
  constexpr int T = WilsonShape<PREC>::threads;
  dim3 block(T), grid((n + T - 1) / T);
  if (recon == 18) {
    if (fullm) launch_pdl(wilson_kernel<PREC, 18, true>, grid, block, 0, st, a);
    else launch_pdl(wilson_kernel<PREC, 18, false>, grid, block, 0, st, a);
  } else if (recon == 12) {
    if (fullm) launch_pdl(wilson_kernel<PREC, 12, true>, grid, block, 0, st, a);
    else launch_pdl(wilson_kernel<PREC, 12, false>, grid, block, 0, st, a);
  } else {
    if (fullm) launch_pdl(wilson_kernel<PREC, 8, true>, grid, block, 0, st, a);
    else launch_pdl(wilson_kernel<PREC, 8, false>, grid, block, 0, st, a);
  }
}

}  // namespace dirac
