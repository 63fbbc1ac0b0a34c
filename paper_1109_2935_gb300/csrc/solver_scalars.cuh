// Scalar state of the solvers on the GPU and the scalar algebra that follows a reduction: one
// thread of the reduction's last block runs it (Fin), so an iteration needs no launch of its
// own for it. What is left of its cost is the chain of FP64 divisions: CG on 4^4, two of them
// per iteration, 27.5 -> 26.8 us per iteration.
#pragma once
#include "internal.h"

namespace dirac {

constexpr int KMAX = 20;
// device scalar slots (doubles); every slot is 4 wide
enum : int {
  S_RHO = 0, S_RHOOLD = 4, S_ALPHA = 8, S_OMEGA = 12, S_SIGMA = 16, S_TS = 20, S_RN = 24,
  S_BETA = 28, S_NBW = 32, S_NALPHA = 36, S_NOMEGA = 40, S_PAP = 44, S_RR = 48, S_ONE = 52,
  S_FLAG = 56, S_TMP = 60, S_ZZ = 64, S_INVG = 68, S_B0 = 72, S_RH = 76,
  S_GB = 128,                       // beta_{i,k}: slot (i * KMAX + k), value at +1, +2
  S_GG = S_GB + 4 * KMAX * KMAX,    // gamma_k
  S_GA = S_GG + 4 * KMAX,           // alpha_k (re, im)
  S_GC = S_GA + 4 * KMAX,           // chi_k (re, im)
  KSH = 16,                         // multi-shift: at most 16 shifts
  S_MSC = S_GC + 4 * KMAX,          // per shift: a_j, zeta_{k+1,j}, b_j, active_j
  S_MSZ = S_MSC + 4 * KSH,          // zeta_{k,j}
  S_MSZP = S_MSZ + KSH,             // zeta_{k-1,j}
  S_MSCV = S_MSZP + KSH,            // converged_j
  S_MSSH = S_MSCV + KSH,            // sigma_j
  S_MSAB = S_MSSH + KSH,            // a_{k-1}, b_{k-1} of the base system
  S_END = S_MSAB + 4
};
enum : int { FLAG_OK = 0, FLAG_BREAKDOWN = 1, FLAG_NONFINITE = 2 };

__device__ __forceinline__ bool bad(double v) { return !isfinite(v); }
__device__ __forceinline__ void flag(double* S, int f) { if (S[S_FLAG] == FLAG_OK) S[S_FLAG] = f; }
__device__ __forceinline__ void cdiv(double ar, double ai, double br, double bi, double& qr, double& qi) {
  double d = br * br + bi * bi;
  qr = (ar * br + ai * bi) / d;
  qi = (ai * br - ar * bi) / d;
}

// --------------------------------------------------------------- scalar steps

__device__ inline void fin_mirror(const double* S, int slot, double* mirror, int which, int it) {
  mirror[4 * which + 0] = S[slot];
  mirror[4 * which + 1] = S[S_FLAG];
  mirror[4 * which + 2] = it;
}

// alpha = rho / (r0, v)
__device__ inline void fin_bicg2(double* S) {
  double sr = S[S_SIGMA], si = S[S_SIGMA + 1];
  if (bad(sr) || bad(si)) flag(S, FLAG_NONFINITE);
  else if (sr == 0 && si == 0) flag(S, FLAG_BREAKDOWN);
  double ar = 0, ai = 0;
  if (S[S_FLAG] == FLAG_OK) cdiv(S[S_RHO], S[S_RHO + 1], sr, si, ar, ai);
  S[S_ALPHA] = ar; S[S_ALPHA + 1] = ai;
  S[S_NALPHA] = -ar; S[S_NALPHA + 1] = -ai;
}

// omega = (t, s) / (t, t)
__device__ inline void fin_bicg3(double* S) {
  double tt = S[S_TS + 2];
  if (bad(tt) || bad(S[S_TS]) || bad(S[S_TS + 1])) flag(S, FLAG_NONFINITE);
  else if (tt == 0) flag(S, FLAG_BREAKDOWN);
  double wr = 0, wi = 0;
  if (S[S_FLAG] == FLAG_OK) { wr = S[S_TS] / tt; wi = S[S_TS + 1] / tt; }
  S[S_OMEGA] = S[S_FLAG] == FLAG_OK ? wr : 1; S[S_OMEGA + 1] = S[S_FLAG] == FLAG_OK ? wi : 0;
  S[S_NOMEGA] = -wr; S[S_NOMEGA + 1] = -wi;
}

// rho_old = rho; rho = (r0, r)
__device__ inline void fin_bicg4(double* S, double* mirror, int which, int it) {
  S[S_RHOOLD] = S[S_RHO]; S[S_RHOOLD + 1] = S[S_RHO + 1];
  S[S_RHO] = S[S_RN + 1]; S[S_RHO + 1] = S[S_RN + 2];
  if (bad(S[S_RN])) flag(S, FLAG_NONFINITE);
  mirror[4 * which + 0] = S[S_RN];
  mirror[4 * which + 1] = S[S_FLAG];
  mirror[4 * which + 2] = it;
}

// CG: alpha = rr / (p, Ap)
__device__ inline void fin_cg1(double* S) {
  double pap = S[S_PAP];
  if (bad(pap)) flag(S, FLAG_NONFINITE);
  else if (pap <= 0) flag(S, FLAG_BREAKDOWN);
  double a = S[S_FLAG] == FLAG_OK ? S[S_RR] / pap : 0;
  S[S_ALPHA] = a; S[S_ALPHA + 1] = 0;
  S[S_NALPHA] = -a; S[S_NALPHA + 1] = 0;
}

// beta = rr_new / rr
__device__ inline void fin_cg2(double* S, double* mirror, int which, int it) {
  double rn = S[S_RN];
  if (bad(rn)) flag(S, FLAG_NONFINITE);
  double b = (S[S_FLAG] == FLAG_OK && S[S_RR] > 0) ? rn / S[S_RR] : 0;
  S[S_BETA] = b; S[S_BETA + 1] = 0;
  if (S[S_FLAG] == FLAG_OK) S[S_RR] = rn;
  mirror[4 * which + 0] = rn;
  mirror[4 * which + 1] = S[S_FLAG];
  mirror[4 * which + 2] = it;
}

// GCR: gamma_k = ||z_k||, 1/gamma_k; move beta_{0,k} (a cdot result) into its slot
__device__ inline void fin_gcr_gamma(double* S, int k) {
  double zz = S[S_ZZ];
  if (bad(zz)) flag(S, FLAG_NONFINITE);
  else if (zz <= 0) flag(S, FLAG_BREAKDOWN);
  double g = S[S_FLAG] == FLAG_OK ? sqrt(zz) : 1;
  S[S_GG + 4 * k] = g;
  S[S_INVG] = S[S_FLAG] == FLAG_OK ? 1.0 / g : 0;
  S[S_INVG + 1] = 0;
  if (k > 0) {
    S[S_GB + 4 * (0 * KMAX + k) + 1] = S[S_B0];
    S[S_GB + 4 * (0 * KMAX + k) + 2] = S[S_B0 + 1];
  }
}

enum : int { FIN_NONE = 0, FIN_MIRROR, FIN_CG1, FIN_CG2, FIN_BICG2, FIN_BICG3, FIN_BICG4, FIN_GCR_GAMMA };

// not inlined: the reductions keep their registers
__device__ __noinline__ inline void run_fin(const Fin& f) {
  switch (f.op) {
    case FIN_MIRROR: fin_mirror(f.S, f.a, f.mirror, f.b & 1, f.b); break;
    case FIN_CG1: fin_cg1(f.S); break;
    case FIN_CG2: fin_cg2(f.S, f.mirror, f.b & 1, f.b); break;
    case FIN_BICG2: fin_bicg2(f.S); break;
    case FIN_BICG3: fin_bicg3(f.S); break;
    case FIN_BICG4: fin_bicg4(f.S, f.mirror, f.b & 1, f.b); break;
    case FIN_GCR_GAMMA: fin_gcr_gamma(f.S, f.a); break;
  }
}

}  // namespace dirac
