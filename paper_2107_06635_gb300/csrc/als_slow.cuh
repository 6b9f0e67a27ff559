// The ALS solves that the Gershgorin discs do not decide (metrics of states
// part-way into a quench or thermal run, whose spectrum spans many decades):
// the selection by triangular factorisations, and through the spectrum of the
// tridiagonal form, on the FP64 contexts (a mixed context's cell step turns a
// change of the last bit here into one of 1e-6 of its result, through the
// roundings of the next bond's environment, and keeps its solves).  Included
// by als_kernel.cuh.
//
// One CTA works on one n x n Hermitian matrix, n = n_A <= 256.  An SM retires
// two FP64 FMAs per cycle, i.e. one FP64 instruction of a warp holds the pipe
// of its quarter of the SM for 64 cycles whatever its active lanes, so both
// are bound by that pipe (n^3/6 complex multiply-adds for the factor, 2 n^3/3
// for the tridiagonal form): lanes are packed, no quantity is computed by
// every warp, and nothing long runs on one thread.  Up to n = LOW_SH_MAX the working
// matrix is the packed lower triangle in the SVD work arrays, which are free
// during a solve; above it stays in global memory.
#pragma once
#include "als_types.cuh"

namespace ntu {

// Candidate relative tolerances 1e-k of the pseudo-inverse (Eq. 4), as
// correctly rounded decimal literals.
__device__ __forceinline__ double als_tau(int k) {
  switch (k) {
    case 0: return 1e0;   case 1: return 1e-1;  case 2: return 1e-2;  case 3: return 1e-3;
    case 4: return 1e-4;  case 5: return 1e-5;  case 6: return 1e-6;  case 7: return 1e-7;
    case 8: return 1e-8;  case 9: return 1e-9;  case 10: return 1e-10; case 11: return 1e-11;
    case 12: return 1e-12; case 13: return 1e-13; case 14: return 1e-14; case 15: return 1e-15;
    case 16: return 1e-16; case 17: return 1e-17; case 18: return 1e-18; case 19: return 1e-19;
    default: return 1e-20;
  }
}

static_assert(offsetof(AlsShared, p) == offsetof(AlsShared, y2) + 256 * sizeof(double2),
              "y2 and p are contiguous (the factor of T)");
constexpr int LOW_SH_MAX = 77;               // n (n + 1) / 2 <= 3 * 32 * 32
static_assert(offsetof(SvdSmem, V) == sizeof(double2) * 1024 &&
              offsetof(SvdSmem, W) == sizeof(double2) * 2048 &&
              LOW_SH_MAX * (LOW_SH_MAX + 1) / 2 <= 3 * 1024,
              "the packed triangle fits in the contiguous SVD work arrays");

// Lower triangle of an n x n matrix: element (i, k), i >= k, at off(k) + i;
// packed columns in shared memory (SH) or a full column-major array.
template <bool SH>
struct LowTri {
  double2* a;
  int n;
  __device__ __forceinline__ int off(int k) const { return SH ? k * n - k * (k + 1) / 2 : k * n; }
  __device__ __forceinline__ double2& at(int i, int k) const { return a[off(k) + i]; }
};

// 2^e as a double, -1022 <= e <= 1023.
__device__ __forceinline__ double pow2i(int e) { return __hiloint2double((e + 1023) << 20, 0); }

// Element pos of the pair of rows (q, m-1-q) of a lower triangle of m rows,
// which hold m + 1 elements together (q + 1 when the rows coincide): a thread
// per pair and part has the same work wherever its rows lie.
__device__ __forceinline__ bool low_pair(int m, int q, int pos, int& i, int& k) {
  const int i2 = m - 1 - q;
  const bool first = pos <= q;
  i = first ? q : i2;
  k = first ? pos : pos - q - 1;
  return first || (i2 != q && k <= i2);
}

// Whether sg (gX - shift I), sg = 1 or -1, is positive definite: an L D L^H
// factorisation of it minus a margin I in double-FP32 arithmetic succeeds.  Every
// entry is renormalised after each update (|lo| <= 2^-24 |hi|: a pivot that has
// cancelled to the size of its low part would otherwise be tested by a high
// part without meaning), so an update of a_ik errs by at most 2^-46 of
// 5 |c_i c_k| / d + sqrt(a_ii a_kk), and n of them perturb a positive definite
// matrix by a matrix of norm below 4 (n + 2) 2^-46 tr.  That is the margin, with
// the trace bounded by tr gX (sg = 1) or n shift (sg = -1): success proves
// it, and a matrix that is definite by less goes to the spectrum.  A warp's
// double-FP32 complex multiply-add takes 60 issue slots where the FP64 one
// holds its pipe for 256 cycles; one barrier per step, the reciprocal pivot
// from FP32 and one double-FP32 correction by every thread.
template <bool SH>
static __device__ int low_certify(AlsShared& sm, int n, const double2* gX, void* buf, double shift,
                                  double tr, int e, double sg) {
  const int tid = threadIdx.x;
  float4* A = reinterpret_cast<float4*>(buf);
  const LowTri<SH> L = {nullptr, n};
  const double f = sg * pow2i(-e);                          // entries of about 1 at most
  const double sh = shift + sg * 4.0 * (n + 2) * 0x1p-46 * (sg > 0.0 ? tr : n * shift);
  for (int idx = tid; idx < n * n; idx += NTU_CTA) {
    const int i = idx % n, k = idx / n;
    if (i < k) continue;
    double2 v = gX[idx];
    if (i == k) v = make_double2(v.x - sh, 0.0);
    A[L.off(k) + i] = df_split(cscale(v, f));
  }
  __syncthreads();
  for (int j = 0; j < n; ++j) {
    const float4* c = A + L.off(j);
    const float4 dj = c[j];
    if (!(dj.x > 0.f) || !isfinite(dj.x)) return 0;         // the same in every thread
    const int m = n - 1 - j;
    if (m == 0) break;
    // 1 / d: r + r (1 - d r)
    const float r = 1.0f / dj.x;
    const float h = fmaf(-dj.x, r, 1.0f) - dj.z * r;
    const float4 rd = make_float4(r, 0.f, r * h, 0.f);
    const int half = (m + 1) >> 1, parts = NTU_CTA / half, q = tid % half, pt = tid / half;
    if (pt < parts) {
      const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
      float4 v1 = z, v2 = z;                                // -c_i / d
      auto scaled = [&](float4 x) {
        float4 o = z;
        df_mac1(o.x, o.z, -x.x, -x.z, rd.x, rd.z);
        df_mac1(o.y, o.w, -x.y, -x.w, rd.x, rd.z);
        return o;
      };
      v1 = scaled(c[j + 1 + q]);
      v2 = scaled(c[n - 1 - q]);
      int i, k;
      for (int pos = pt; low_pair(m, q, pos, i, k); pos += parts) {
        float4* x = A + L.off(j + 1 + k) + j + 1 + i;
        float4 acc = *x;
        df_cmac<true>(acc, c[j + 1 + k], i == q ? v1 : v2); // a -= (c_i / d) conj(c_k)
        df_renorm(acc.x, acc.z);
        df_renorm(acc.y, acc.w);
        *x = acc;
      }
    }
    __syncthreads();
  }
  __syncthreads();
  return 1;
}

// L D L^H of the Hermitian A in FP64 (in place; A holds gX's lower triangle):
// column j becomes the unit-lower L's, the diagonal (d_j, 1 / d_j).  One
// barrier per step: the update takes the column unscaled, a -= (c_i / d)
// conj(c_k), and warp 7 meanwhile forms the next pivot's reciprocal (an FP64
// instruction holds a warp's pipe for 64 cycles, a division ten of them).
template <bool SH>
static __device__ int low_ldl(AlsShared& sm, const LowTri<SH>& A) {
  const int tid = threadIdx.x, wid = tid >> 5, n = A.n;
  constexpr int UPD = NTU_CTA - 32;
  if (tid == 0) A.at(0, 0).y = 1.0 / A.at(0, 0).x;
  __syncthreads();
  for (int j = 0; j < n; ++j) {
    const double2* c = A.a + A.off(j);
    const double dj = c[j].x, rj = c[j].y;
    if (!(dj > 0.0) || !isfinite(dj)) return 0;             // the same in every thread
    const int m = n - 1 - j;
    if (m == 0) break;
    if (wid < NTU_WARPS - 1) {
      const int half = (m + 1) >> 1, parts = UPD / half, q = tid % half, pt = tid / half;
      if (pt < parts) {
        const double2 v1 = cscale(c[j + 1 + q], rj), v2 = cscale(c[n - 1 - q], rj);
        int i, k;
        for (int pos = pt; low_pair(m, q, pos, i, k); pos += parts) {
          double2& x = A.at(j + 1 + i, j + 1 + k);
          const double2 o = cfmsc(i == q ? v1 : v2, c[j + 1 + k], x);
          if (i + k > 0) x = o;                             // the next pivot is warp 7's
        }
      }
    } else {
      const double2 l = c[j + 1], o = cfmsc(cscale(l, rj), l, A.at(j + 1, j + 1));
      const double r = 1.0 / o.x;
      __syncwarp();
      if (tid == NTU_CTA - 32) A.at(j + 1, j + 1) = make_double2(o.x, r);
    }
    __syncthreads();
  }
  __syncthreads();
  for (int idx = tid; idx < n * n; idx += NTU_CTA) {
    const int i = idx % n, k = idx / n;
    if (i > k) A.at(i, k) = cscale(A.at(i, k), A.at(k, k).y);
  }
  __syncthreads();
  return 1;
}

// b <- (L D L^H)^{-1} b, b in shared memory, a thread per real component.
template <bool SH>
static __device__ void low_solve(const LowTri<SH>& L, double2* b) {
  const int tid = threadIdx.x, n = L.n, im = tid & 1;
  double* bc = reinterpret_cast<double*>(b) + im;
  const double sg = im ? 1.0 : -1.0;
  for (int j = 0; j < n - 1; ++j) {                         // b_i -= l_ij b_j
    for (int i = tid >> 1; i < n; i += NTU_CTA / 2)
      if (i > j) {
        const double2 l = L.at(i, j), y = b[j];
        bc[2 * i] = fma(-l.x, im ? y.y : y.x, fma(-sg * l.y, im ? y.x : y.y, bc[2 * i]));
      }
    __syncthreads();
  }
  for (int i = tid >> 1; i < n; i += NTU_CTA / 2) bc[2 * i] *= L.at(i, i).y;
  __syncthreads();
  for (int j = n - 1; j > 0; --j) {                         // b_i -= conj(l_ji) b_j
    for (int i = tid >> 1; i < j; i += NTU_CTA / 2) {
      const double2 l = L.at(j, i), x = b[j];
      bc[2 * i] = fma(-l.x, im ? x.y : x.x, fma(sg * l.y, im ? x.x : x.y, bc[2 * i]));
    }
    __syncthreads();
  }
}

static __device__ void als_matvec(AlsShared& sm, const double2* A, const float4* Adf, const double2* v,
                                  double2* out, int nA, bool df, float* rsum);

// v <- v / |v| (n entries in shared memory).
static __device__ void low_normalise(AlsShared& sm, double2* v, int n) {
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += NTU_CTA) s += cabs2(v[i]);
  s = block_sum<true>(s, sm.red);
  const double f = s > 0.0 ? rsqrt(s) : 0.0;
  for (int i = threadIdx.x; i < n; i += NTU_CTA) v[i] = cscale(v[i], f);
  __syncthreads();
}

// Tier 2: the selection by factorisations.  B >= lambda_max is the smallest of
// the Gershgorin bound, the Frobenius bound and, where the first test fails
// with those, 1.01 times a Rayleigh quotient once 1.01 of it minus gX is shown
// to be positive definite.  Where gX - (tau + 1e-12) B I is
// positive definite at the largest tolerance, every candidate keeps every
// eigenpair and M = x = gX^{-1} J.  Otherwise let tau_k be the largest
// tolerance that passes this test: it keeps all, as do the smaller ones, so
// the rule chooses it unless tau_{k-1} comes within 1e-14 eps0 of the
// minimum, i.e. unless the pairs below thr = tau_{k-1} lambda_max carry less
// than that of eps.  With y = W^H J and thr taken from a Rayleigh quotient of
// gX (thr <= tau_{k-1} lambda_max), the sums
//   F_p = sum_i |y_i|^2 / lambda_i (thr / lambda_i)^p
// come from repeated solves (F_0 = x^H J).  The terms above thr never grow with
// p and one below it grows at most by (thr / lambda_min)^2 a step p -> p + 2, so
// with b thr < lambda_min (certified like the first test, at tau_k B or at 0.6
// of the Rayleigh quotient rho of u) the pairs below thr carry at least
//   (F_{p+2} - F_p) / (b^-2 - 1) b^p
// of eps; tau_k is chosen when this exceeds 2e-14 eps0 for some p.  Anything
// else goes to the spectrum.  Returns 0 (undecided), 1
// (by the first test) or 2; M in sm.MA or sm.MB, tolerance in sm.tau_sel.  Measured (one
// CTA): 0.12, 0.19 and 2.2 ms at n = 50, 64 and 128 where the first test holds
// (the fixed-point iteration on the shifted factor took 5 ms at n = 64), 0.2 to
// 0.5 ms at n = 50 to 72 where the sums decide (11 ms through the eigenpairs).
template <bool SH>
static __device__ __noinline__ int als_solve_certified(AlsShared& sm, const AlsArgs& a, int side,
                                                       const double2* gX, double2* gC,
                                                       const double2* jv, double bmax) {
  const int tid = threadIdx.x, n = a.nA;
  const LowTri<SH> L = {SH ? sm.S.A : gC, n};
  void* buf = SH ? (void*)sm.S.A : (void*)gC;
  const int kmin = a.kmin < 0 ? 0 : a.kmin, kmax = a.kmax > 20 ? 20 : a.kmax;
  double fs = 0.0, low = 0.0, tr = 0.0;
  for (int idx = tid; idx < n * n; idx += NTU_CTA) fs += cabs2(gX[idx]);
  for (int i = tid; i < n; i += NTU_CTA) {
    low = fmax(low, gX[(size_t)i * n + i].x);
    tr += gX[(size_t)i * n + i].x;
  }
  fs = sqrt(block_sum<true>(fs, sm.red)) * (1.0 + 1e-12);
  low = block_max<true>(low, sm.red);
  tr = block_sum<true>(tr, sm.red);
  double B = fs < bmax ? fs : bmax;
  if (!(B > 0x1p-900) || !(B < 0x1p900)) return 0;
  const int e = ilogb(B);
  const int all = low_certify<SH>(sm, n, gX, buf, (als_tau(kmin) + 1e-12) * B, tr, e, 1.0);
  if (!all) {
    // lambda_max from below by eight steps of the power iteration on J, and
    // from above, where it holds, by 1.01 times that
    for (int i = tid; i < n; i += NTU_CTA) sm.p[i] = jv[i];
    __syncthreads();
    for (int it = 0; it < 8; ++it) {
      low_normalise(sm, sm.p, n);
      als_matvec(sm, gX, nullptr, sm.p, sm.ap, n, false, nullptr);
      double s = 0.0;
      for (int i = tid; i < n; i += NTU_CTA) {
        s += cmulc(sm.p[i], sm.ap[i]).x;
        sm.p[i] = sm.ap[i];
      }
      low = fmax(low, block_sum<true>(s, sm.red));
    }
    for (int t = 0; t < 2; ++t) {
      const double b = (t ? 1.08 : 1.01) * low;
      if (b < B && low_certify<SH>(sm, n, gX, buf, b, tr, e, -1.0)) { B = b; break; }
      __syncthreads();
    }
  }
  __syncthreads();
  for (int idx = tid; idx < n * n; idx += NTU_CTA) {
    const int i = idx % n, k = idx / n;
    if (i >= k) L.at(i, k) = gX[idx];
  }
  __syncthreads();
  if (!low_ldl<SH>(sm, L)) return 0;
  for (int i = tid; i < n; i += NTU_CTA) sm.y[i] = jv[i];
  __syncthreads();
  low_solve<SH>(L, sm.y);
  int k = kmin;
  if (!all) {
    double f0 = 0.0;
    for (int i = tid; i < n; i += NTU_CTA) {
      sm.p[i] = sm.y[i];
      f0 += cmulc(sm.y[i], jv[i]).x;
    }
    f0 = block_sum<true>(f0, sm.red);
    // u_q = (thr / gX)^q x and F_2q = thr u_q^H u_{q-1}, with thr at k = kmin + 1;
    // a larger k rescales F_p by 10^-p per step (F in units of that thr)
    const double thr1 = als_tau(kmin) * low * (1.0 - 1e-9);
    double F[9], rho = INFINITY, rp = INFINITY, sig = 0.0;  // sig: the bound to certify
    F[0] = f0;
    bool done = false;
#pragma unroll
    for (int q = 1; q < 9; ++q) {
      if (!done) {
        for (int i = tid; i < n; i += NTU_CTA) sm.y2[i] = sm.p[i];
        __syncthreads();
        low_solve<SH>(L, sm.p);
        double s = 0.0, uu = 0.0;
        for (int i = tid; i < n; i += NTU_CTA) {
          const double2 u = cscale(sm.p[i], thr1);
          sm.p[i] = u;
          s += cmulc(u, sm.y2[i]).x;
          uu += cabs2(u);
        }
        F[q] = thr1 * block_sum<true>(s, sm.red);
        uu = block_sum<true>(uu, sm.red);
        rp = rho;
        rho = F[q] / uu;                                    // >= lambda_min
        if (!(F[q] > 0.0) || !isfinite(uu)) return 0;
        while (k <= kmax && !(rho > (als_tau(k) + 1e-12) * B)) ++k;
        if (k > kmax || als_tau(k) < 1e-11) return 0;
        if (k == kmin) {                                    // the tighter B may keep all after all
          done = q > 3 && rho > 0.98 * rp;
          sig = (als_tau(k) + 1e-12) * B;
        } else {
          const double sc = als_tau(k - 1) / als_tau(kmin), sc2 = sc * sc;
          const double thr = thr1 * sc;
          double f = 1.0;                                   // sc^(2 (q - 1))
          for (int t = 1; t < q; ++t) f *= sc2;
          const double rise = F[q] * (f * sc2) - F[q - 1] * f;
          if (rho < thr && rise > 1e-6 * F[q - 1] * f) {
            // with lambda_min > tau_k B or, once rho has settled, > 0.6 rho
            for (int t = 0; t < 2 && !done; ++t) {
              sig = (als_tau(k) + 1e-12) * B;
              if (t == 1) {
                if (!(q > 3 && 0.6 * rho > sig)) break;
                sig = 0.6 * rho;
              }
              const double lb = sig / thr, lb2 = lb * lb;
              double g = rise * lb2 / (1.0 - lb2);
              for (int p = 1; p < q; ++p) g *= lb2;
              done = lb2 < 0.99 && g > 2e-14 * sm.eps0;
            }
          }
        }
      }
    }
    if (!done) return 0;
    __syncthreads();
    if (!low_certify<SH>(sm, n, gX, buf, sig, tr, e, 1.0)) return 0;
  }
  double2* M = side == 0 ? sm.MA : sm.MB;
  for (int i = tid; i < n; i += NTU_CTA) M[i] = sm.y[i];
  if (tid == 0) sm.tau_sel = als_tau(k);
  __syncthreads();
  return all ? 1 : 2;
}

// Tier 2 of the mixed contexts: Cholesky factor L L^H of gX - sigma I, then the
// fixed-point iteration (L L^H) v_{k+1} = J - sigma v_k.  A mixed cell step
// feeds its result into the FP32 and BF16 roundings of the next bond's
// environment, where a change of the last bit becomes one of up to 1e-6, so
// every entry sees the operations of the plain right-looking factorisation
// and of the column-by-column substitutions in their order; only who carries
// them out differs: rows in pairs (low_pair), the next pivot's square root and
// reciprocal on a warp of their own, a thread per real component and one
// barrier per substitution step where one warp took n serial steps with a
// division each.  Measured at n = 64 (K = 16, D = 4), some 60 iterations: 1.7
// against 3.5 ms a solve; what is left is the chain of a multiplication and two
// FMAs a step.
// Returns 1 when solved (v in sm.y).
template <bool SH>
static __device__ __noinline__ int als_solve_fixpoint(AlsShared& sm, int n, const double2* M,
                                                      const double2* gX, double2* gC,
                                                      const double2* jv, double sigma) {
  const int tid = threadIdx.x, wid = tid >> 5;
  const LowTri<SH> L = {SH ? sm.S.A : gC, n};
  for (int idx = tid; idx < n * n; idx += NTU_CTA) {
    const int i = idx % n, k = idx / n;
    if (i >= k) L.at(i, k) = gX[idx];
  }
  for (int i = tid; i < n; i += NTU_CTA) sm.y[i] = M[i];    // warm start
  if (tid == 0) {
    const double piv = gX[0].x - sigma;
    sm.red[0] = piv;
    sm.red[1] = sqrt(piv);
    sm.red[2] = 1.0 / sm.red[1];
  }
  __syncthreads();
  constexpr int UPD = NTU_CTA - 32;
  for (int j = 0; j < n; ++j) {
    const double* pv = sm.red + 4 * (j & 1);
    const double piv = pv[0], sp = pv[1], rp = pv[2];
    if (!(piv > 0.0) || !isfinite(piv)) return 0;           // the same in every thread
    double2* c = L.a + L.off(j);
    const int m = n - 1 - j;
    if (tid == 0) c[j] = make_double2(sp, rp);
    for (int i = j + 1 + tid; i < n; i += NTU_CTA) c[i] = cscale(c[i], rp);
    __syncthreads();
    if (m == 0) break;
    if (wid < NTU_WARPS - 1) {
      const int half = (m + 1) >> 1, parts = UPD / half, q = tid % half, pt = tid / half;
      if (pt < parts) {
        const double2 v1 = c[j + 1 + q], v2 = c[n - 1 - q];
        int i, k;
        for (int pos = pt; low_pair(m, q, pos, i, k); pos += parts) {
          double2& x = L.at(j + 1 + i, j + 1 + k);
          const double2 o = cfmsc(i == q ? v1 : v2, c[j + 1 + k], x);
          if (i + k > 0) x = o;                             // the next pivot is warp 7's
        }
      }
    } else {
      const double2 l = c[j + 1], o = cfmsc(l, l, L.at(j + 1, j + 1));
      const double p = o.x - sigma, s = sqrt(p), r = 1.0 / s;
      if (tid == UPD) {
        double* nx = sm.red + 4 * ((j + 1) & 1);
        nx[0] = p; nx[1] = s; nx[2] = r;
      }
    }
    __syncthreads();
  }
  const int im = tid & 1;
  double prev = INFINITY;
  for (int it = 0; it < 60; ++it) {
    double *b = reinterpret_cast<double*>(sm.y2), *w = reinterpret_cast<double*>(sm.p),
           *x = reinterpret_cast<double*>(sm.ap);
    for (int i = tid; i < n; i += NTU_CTA) {
      const double2 v = sm.y[i], j = jv[i];
      sm.y2[i] = make_double2(fma(-sigma, v.x, j.x), fma(-sigma, v.y, j.y));
    }
    __syncthreads();
    for (int j = 0; j < n; ++j) {                           // w = L^-1 b
      const double r = L.at(j, j).y, y0 = b[2 * j] * r, y1 = b[2 * j + 1] * r;
      for (int i = tid >> 1; i < n; i += NTU_CTA / 2) {
        if (i > j) {
          const double2 l = L.at(i, j);
          double t = b[2 * i + im];
          t = fma(-l.x, im ? y1 : y0, t);
          t = fma(im ? -l.y : l.y, im ? y0 : y1, t);
          b[2 * i + im] = t;
        } else if (i == j) {
          w[2 * j + im] = im ? y1 : y0;
        }
      }
      __syncthreads();
    }
    for (int j = n - 1; j >= 0; --j) {                      // x = L^-H w
      const double r = L.at(j, j).y, x0 = w[2 * j] * r, x1 = w[2 * j + 1] * r;
      for (int i = tid >> 1; i <= j; i += NTU_CTA / 2) {
        if (i < j) {
          const double2 l = L.at(j, i);
          double t = w[2 * i + im];
          t = fma(im ? x0 : -x0, im ? l.y : l.x, t);
          t = fma(-x1, im ? l.x : l.y, t);
          w[2 * i + im] = t;
        } else {
          x[2 * j + im] = im ? x1 : x0;
        }
      }
      __syncthreads();
    }
    double diff = 0.0, vmax = 0.0;
    for (int i = tid; i < n; i += NTU_CTA) {
      const double2 nw = sm.ap[i], o = sm.y[i];
      diff = fmax(diff, fabs(nw.x - o.x) + fabs(nw.y - o.y));
      vmax = fmax(vmax, fabs(nw.x) + fabs(nw.y));
      sm.y[i] = nw;
    }
    diff = block_max(diff, sm.red);
    vmax = block_max(vmax, sm.red);
    if (diff <= 1e-15 * vmax) return 1;                     // converged
    if (it >= 3 && diff >= 0.5 * prev && diff <= 1e-13 * vmax) return 1;   // rounding floor
    prev = diff;
  }
  return 0;
}

// ------------------------------------------------ tridiagonal form
// Householder reduction of the Hermitian A (lower triangle) to tridiagonal
// form with diagonal d (real) and subdiagonal e (complex), Q = H_0 H_1 ...,
// H_j = I - c_j v_j v_j^H = H_j^H on rows j + 1.., v_j left in column j below
// the diagonal, and y <- Q^H y (y = sm.y).  Warp 0 forms each reflector (of the
// column scaled by an exact power of two, so that entries far below the
// square root of the smallest normal number neither vanish from nor zero out
// the norm) and w; one part of the threads per row forms A v; the rank-2
// update takes rows q and m-1-q together, so every thread has the same
// number of elements.  Four barriers per step.
template <bool SH>
static __device__ void low_tridiag(AlsShared& sm, const LowTri<SH>& A, double* d, double2* e,
                                   double* c) {
  const int tid = threadIdx.x, wid = tid >> 5, lid = tid & 31, n = A.n;
  double2 *v = sm.y2, *w = sm.p, *part = sm.ap;
  for (int j = 0; j + 2 < n; ++j) {
    const int m = n - 1 - j, b = j + 1;
    double2* col = A.a + A.off(j) + b;                      // x_i = col[i], i < m
    if (wid == 0) {
      unsigned mx = 0;
      for (int i = lid; i < m; i += 32) {
        const double2 x = col[i];
        mx = max(mx, max((unsigned)__double2hiint(x.x) & 0x7fffffffu,
                         (unsigned)__double2hiint(x.y) & 0x7fffffffu));
      }
      mx = __reduce_max_sync(0xffffffffu, mx);
      int ex = (int)(mx >> 20) - 1023;
      ex = ex < -1000 ? -1000 : (ex > 1000 ? 1000 : ex);
      const double down = pow2i(-ex);
      double s2 = 0.0, t2 = 0.0;
      for (int i = lid; i < m; i += 32) {
        const double q = cabs2(cscale(col[i], down));
        s2 += q;
        if (i > 0) t2 += q;
      }
      s2 = warp_sum(s2);
      t2 = warp_sum(t2);
      const double2 al = cscale(col[0], down);
      const double nx = sqrt(s2), aa = sqrt(cabs2(al));
      const double2 ph = aa > 0.0 ? cscale(al, 1.0 / aa) : make_double2(1.0, 0.0);
      const double cj = t2 != 0.0 ? 1.0 / (nx * (nx + aa)) : 0.0;
      const double2 x0 = col[0];
      __syncwarp();
      if (cj != 0.0)
        for (int i = lid; i < m; i += 32) {
          const double2 vi = i == 0 ? cscale(ph, aa + nx) : cscale(col[i], down);
          v[i] = vi;
          col[i] = vi;
        }
      if (lid == 0) {
        d[j] = A.at(j, j).x;
        e[j] = cj != 0.0 ? cscale(ph, -nx * pow2i(ex)) : x0;
        c[j] = cj;
        sm.red[j & 1] = cj;
      }
    }
    __syncthreads();
    const double cj = sm.red[j & 1];
    if (cj == 0.0) continue;
    const int parts = NTU_CTA / m;                          // m <= 255
    {
      const int i = tid % m, pt = tid / m;
      if (pt < parts) {
        double2 acc = cz();
        for (int k = pt; k < m; k += parts) {               // A_ik = conj(A_ki) above the diagonal
          double2 x = k <= i ? A.at(b + i, b + k) : A.at(b + k, b + i);
          if (k > i) x.y = -x.y;
          acc = cfma(x, v[k], acc);
        }
        part[pt * m + i] = acc;
      }
    }
    __syncthreads();
    if (wid == 0) {
      double vp = 0.0;
      for (int i = lid; i < m; i += 32) {
        double2 s = part[i];
        for (int q = 1; q < parts; ++q) s = cadd(s, part[q * m + i]);
        s = cscale(s, cj);
        w[i] = s;
        vp += cmulc(v[i], s).x;
      }
      const double kk = 0.5 * cj * warp_sum(vp);
      for (int i = lid; i < m; i += 32)
        w[i] = make_double2(fma(-kk, v[i].x, w[i].x), fma(-kk, v[i].y, w[i].y));
    } else if (wid == 1) {
      double2 s = cz();
      for (int i = lid; i < m; i += 32) s = cfmac(v[i], sm.y[b + i], s);
      s = cscale(warp_sum2(s), cj);
      for (int i = lid; i < m; i += 32) sm.y[b + i] = cfms(s, v[i], sm.y[b + i]);
    }
    __syncthreads();
    const int half = (m + 1) >> 1, parts2 = NTU_CTA / half;
    {
      const int q = tid % half, pt = tid / half;
      if (pt < parts2) {
        const double2 v1 = v[q], w1 = w[q], v2 = v[m - 1 - q], w2 = w[m - 1 - q];
        int i, k;
        for (int pos = pt; low_pair(m, q, pos, i, k); pos += parts2) {
          double2& x = A.at(b + i, b + k);
          x = cfmsc(i == q ? w1 : w2, v[k], cfmsc(i == q ? v1 : v2, w[k], x));
        }
      }
    }
    __syncthreads();
  }
  if (tid == 0) {
    if (n >= 2) {
      d[n - 2] = A.at(n - 2, n - 2).x;
      e[n - 2] = A.at(n - 1, n - 2);
    }
    d[n - 1] = A.at(n - 1, n - 1).x;
  }
  __syncthreads();
}

// Number of eigenvalues below x of the tridiagonal (d, e) of norm about 1,
// e2 = e^2, from the signs of the leading principal minors of T - x (three
// FP64 operations a step where the quotient form takes a division), which
// are rescaled by an exact power of two every fourth step.
static __device__ int sturm_count(const double* d, const double* e2, int n, double x) {
  double p0 = 1.0, p1 = d[0] - x;
  if (p1 == 0.0) p1 = -0x1p-100;
  int cnt = (unsigned)__double2hiint(p1) >> 31;
  for (int i = 1; i < n; ++i) {
    double t = fma(d[i] - x, p1, -(e2[i - 1] * p0));
    if (t == 0.0) t = p1 * -0x1p-100;
    cnt += (unsigned)(__double2hiint(t) ^ __double2hiint(p1)) >> 31;
    p0 = p1;
    p1 = t;
    if ((i & 3) == 3) {
      const int h0 = __double2hiint(p0) & 0x7ff00000, h1 = __double2hiint(p1) & 0x7ff00000;
      const int h = max(h0, h1);
      const double f = __hiloint2double((h > 0 && h < 0x7ff00000 ? 0x7fe00000 - h : 0x3ff00000), 0);
      p0 *= f;
      p1 *= f;
    }
  }
  return cnt;
}

// Factor of T - x with partial pivoting (T tridiagonal, (d, e)): rows of U
// (1 / u0, u1, u2), multipliers l, interchange flags sw, all at stride st;
// pivots below 2^-53 are raised to it.
static __device__ void tri_factor(const double* d, const double* e, int n, double x, double* u0,
                                  double* u1, double* u2, double* l, int* sw, int st) {
  double a = d[0] - x, b = n > 1 ? e[0] : 0.0;
  for (int k = 0; k + 1 < n; ++k) {
    const double sub = e[k], nd = d[k + 1] - x, ns = k + 2 < n ? e[k + 1] : 0.0;
    if (fabs(a) >= fabs(sub)) {
      if (fabs(a) < 0x1p-53) a = copysign(0x1p-53, a);
      const double r = 1.0 / a, f = sub * r;
      u0[k * st] = r; u1[k * st] = b; u2[k * st] = 0.0; l[k * st] = f; sw[k * st] = 0;
      a = fma(-f, b, nd);
      b = ns;
    } else {
      const double s = fabs(sub) < 0x1p-53 ? copysign(0x1p-53, sub) : sub;
      const double r = 1.0 / s, f = a * r;
      u0[k * st] = r; u1[k * st] = nd; u2[k * st] = ns; l[k * st] = f; sw[k * st] = 1;
      a = fma(-f, nd, b);
      b = -f * ns;
    }
  }
  if (!(fabs(a) >= 0x1p-53)) a = copysign(0x1p-53, a);
  u0[(n - 1) * st] = 1.0 / a;
}

// b <- (T - x)^{-1} b with the factor of tri_factor; b has stride sb.
static __device__ void tri_solve(int n, const double* u0, const double* u1, const double* u2,
                                 const double* l, const int* sw, int st, double* b, int sb) {
  double cur = b[0];
  for (int k = 0; k + 1 < n; ++k) {
    const double nx = b[(k + 1) * sb], f = l[k * st];
    if (sw[k * st]) {
      b[k * sb] = nx;
      cur = fma(-f, nx, cur);
    } else {
      b[k * sb] = cur;
      cur = fma(-f, cur, nx);
    }
  }
  double x1 = cur * u0[(n - 1) * st], x2 = 0.0;
  b[(n - 1) * sb] = x1;
  for (int k = n - 2; k >= 0; --k) {
    const double t = (b[k * sb] - u1[k * st] * x1 - u2[k * st] * x2) * u0[k * st];
    b[k * sb] = t;
    x2 = x1;
    x1 = t;
  }
}

// Orthonormalises the rows W[j * n ..], j < m (twice-applied classical
// Gram-Schmidt in order, warps sharing the inner products).
static __device__ void tri_orthonormalise(AlsShared& sm, double* W, int n, int m, double* cf) {
  const int tid = threadIdx.x, wid = tid >> 5, lid = tid & 31;
  for (int j = 0; j < m; ++j) {
    double* wj = W + (size_t)j * n;
    for (int pass = 0; pass < 3; ++pass) {                  // scale, then project and scale twice
      if (pass > 0) {
        if (j == 0) break;
        for (int i = wid; i < j; i += NTU_WARPS) {
          double s = 0.0;
          for (int k = lid; k < n; k += 32) s = fma(W[(size_t)i * n + k], wj[k], s);
          s = warp_sum(s);
          if (lid == 0) cf[i] = s;
        }
        __syncthreads();
        if (tid < n) {
          double x = wj[tid];
          for (int i = 0; i < j; ++i) x = fma(-cf[i], W[(size_t)i * n + tid], x);
          wj[tid] = x;
        }
        __syncthreads();
      }
      double mx = tid < n ? fabs(wj[tid]) : 0.0;
      mx = block_max<true>(mx, sm.red);
      const double f = mx > 0.0 && isfinite(mx) ? 1.0 / mx : 0.0;
      const double x = tid < n ? wj[tid] * f : 0.0;
      const double s = block_sum<true>(x * x, sm.red);
      if (tid < n) wj[tid] = s > 0.0 ? x * rsqrt(s) : 0.0;
      __syncthreads();
    }
  }
}

// y <- y - sum_{i < m} w_i (w_i^T y), y complex in shared memory, n <= CTA.
static __device__ void tri_project(const double* W, int n, int m, double2* y, double2* cf) {
  const int tid = threadIdx.x, wid = tid >> 5, lid = tid & 31;
  if (m == 0) return;
  for (int i = wid; i < m; i += NTU_WARPS) {
    double2 s = cz();
    for (int k = lid; k < n; k += 32) {
      const double w = W[(size_t)i * n + k];
      s.x = fma(w, y[k].x, s.x); s.y = fma(w, y[k].y, s.y);
    }
    s = warp_sum2(s);
    if (lid == 0) cf[i] = s;
  }
  __syncthreads();
  if (tid < n) {
    double2 v = y[tid];
    for (int i = 0; i < m; ++i) {
      const double w = W[(size_t)i * n + tid];
      v.x = fma(-w, cf[i].x, v.x); v.y = fma(-w, cf[i].y, v.y);
    }
    y[tid] = v;
  }
  __syncthreads();
}

// The same selection through a serial QR iteration of the tridiagonal by one
// thread (d, e unscaled in global memory, y = sm.y): the fallback for a
// spectrum whose eigenvectors the inverse iteration does not resolve.
static __device__ void tri_select_serial(AlsShared& sm, const AlsArgs& a, double* d, double* e, int n,
                                         RotLog log) {
  if (threadIdx.x == 0) {
    const int st = tridiag_qr(d, e, n, log, sm.y);
    if (st) sm.err |= WHY_ALS_QR;
    double lmax = d[0];
    for (int i = 1; i < n; ++i) lmax = fmax(lmax, d[i]);
    const int kmin = a.kmin < 0 ? 0 : a.kmin, kmax = a.kmax > 20 ? 20 : a.kmax;
    double tsel = als_tau(kmin);
    if (lmax > 0.0 && !st) {
      double emin = INFINITY;
      for (int pass = 0; pass < 2; ++pass)
        for (int k = kmin; k <= kmax; ++k) {
          const double thr = als_tau(k) * lmax;
          double s = 0.0;
          for (int i = 0; i < n; ++i)
            if (d[i] > thr) s += cabs2(sm.y[i]) / d[i];
          if (pass == 0) emin = fmin(emin, sm.eps0 - s);
          else if (sm.eps0 - s <= emin + 1e-14 * sm.eps0) { tsel = als_tau(k); break; }
        }
      const double thr = tsel * lmax;
      for (int i = 0; i < n; ++i) sm.y[i] = d[i] > thr ? cscale(sm.y[i], 1.0 / d[i]) : cz();
      rotlog_apply_z(log, sm.y);
    } else {
      for (int i = 0; i < n; ++i) sm.y[i] = cz();
    }
    sm.tau_sel = tsel;
  }
  __syncthreads();
}

// Tier 3: M = pinv_tau(gX) J with the tolerance of the grid that minimises
// eps(tau) = eps0 - sum_{lambda_i > tau lambda_max} |y_i|^2 / lambda_i,
// y = W^H J (Eq. 4 inserted in Eq. 3); ties within 1e-14 eps0 go to the larger
// tau.  Only the eigenpairs below tau_max lambda_max take part in the
// selection: gX is reduced to a real tridiagonal T, sign counts give
// lambda_max and the number of eigenvalues below every threshold, bisection
// those below the largest one, inverse iteration with orthogonalisation their
// vectors.  The kept part of T is inverted by a pivoted solve of T v = y on the
// complement of the dropped vectors, refined once (or by the sum over all
// eigenpairs where all were found).  gX is overwritten for n > LOW_SH_MAX.
// Measured (one CTA, 11 of n = 72 eigenvalues below the threshold): 2.1 ms,
// 0.76 ms of it the reduction, where the implicit QR of T by one thread with
// its rotation log took 11 ms.
template <bool SH>
static __device__ __noinline__ void als_solve_spectrum(AlsShared& sm, const AlsArgs& a, int side,
                                                       double2* gX, const double2* jv, double2* pv,
                                                       double2* tauv, double* dv, double* ev,
                                                       double2* Tm, RotLog log) {
  const int tid = threadIdx.x, wid = tid >> 5, lid = tid & 31, n = a.nA;
  const LowTri<SH> A = {SH ? sm.S.A : gX, n};
  double* cfac = reinterpret_cast<double*>(tauv);           // c_j
  double2* ph = pv;                                         // first e_j, then the phases
  double* W = reinterpret_cast<double*>(Tm);                // n x m vectors
  double2* coef = Tm + (size_t)a.ng * n - n;                // past W: n^2 / 2 + n <= n_g n for n >= 2
  if (SH)
    for (int idx = tid; idx < n * n; idx += NTU_CTA) {
      const int i = idx % n, k = idx / n;
      if (i >= k) A.at(i, k) = gX[idx];
    }
  for (int i = tid; i < n; i += NTU_CTA) sm.y[i] = jv[i];
  __syncthreads();
  low_tridiag<SH>(sm, A, dv, ph, cfac);
  // T real: T <- D^H T D with phases D, y <- D^H y; scaled by an exact power
  // of two to norm about 1
  double *d = reinterpret_cast<double*>(sm.ap), *e = d + 256;
  double *e2 = reinterpret_cast<double*>(sm.y2);            // e^2, later the factor of T
  double mxe = 0.0;
  for (int i = tid; i < n; i += NTU_CTA) {
    const double2 z = i + 1 < n ? ph[i] : cz();
    const double r = hypot(z.x, z.y);
    d[i] = dv[i];
    e[i] = r;
    sm.p[i] = r > 0.0 ? make_double2(z.x / r, z.y / r) : make_double2(1.0, 0.0);
    mxe = fmax(mxe, fmax(fabs(dv[i]), r));
  }
  mxe = block_max<true>(mxe, sm.red);
  const bool finite = isfinite(mxe) && mxe > 0.0;
  int se = finite ? ilogb(mxe) : 0;
  se = se < -1000 ? -1000 : (se > 1000 ? 1000 : se);
  const double up = pow2i(se), down = pow2i(-se);
  if (tid == 0) {
    double2 f = make_double2(1.0, 0.0);
    for (int i = 0; i < n; ++i) {
      const double2 u = sm.p[i];
      sm.p[i] = f;
      f = cmul(f, u);
    }
  }
  __syncthreads();
  if (tid < n) {
    const double2 f = sm.p[tid];
    ph[tid] = f;
    sm.y[tid] = cmulc(f, sm.y[tid]);
    d[tid] *= down;
    e[tid] *= down;
    e2[tid] = e[tid] * e[tid];
  }
  if (tid == 0) { sm.n_eig += 1; sm.flag = 1; }
  __syncthreads();
  const int kmin = a.kmin < 0 ? 0 : a.kmin, kmax = a.kmax > 20 ? 20 : a.kmax, nk = kmax - kmin + 1;
  int* cnt = reinterpret_cast<int*>(sm.ph);                 // eigenvalues below tau_k lambda_max
  int* ndrop = cnt + 32;                                    // pairs dropped (a word of its own: every
                                                            // warp still reads sm.flag then)
  double* lim = reinterpret_cast<double*>(sm.ph + 16);      // [lower bound, lambda_max]
  if (wid == 0) {
    double lo = INFINITY, hi = -INFINITY;
    for (int i = lid; i < n; i += 32) {
      const double s = e[i] + (i > 0 ? e[i - 1] : 0.0);
      lo = fmin(lo, d[i] - s);
      hi = fmax(hi, d[i] + s);
    }
    lo = -warp_max(-lo) - 1e-14;
    hi = warp_max(hi) + 1e-14;
    const double low = lo;
    if (finite)
      for (int round = 0; round < 11; ++round) {            // 33 sections a round
        const double x = lo + (hi - lo) * ((lid + 1) * (1.0 / 33.0));
        const unsigned all = __ballot_sync(0xffffffffu, sturm_count(d, e2, n, x) == n);
        const int f = all ? __ffs(all) - 1 : 32;
        const double h2 = __shfl_sync(0xffffffffu, x, f & 31), l2 = __shfl_sync(0xffffffffu, x, (f + 31) & 31);
        if (f < 32) hi = h2;
        if (f > 0) lo = l2;
      }
    if (lid == 0) { lim[0] = low; lim[1] = hi; }
    if (lid < nk) cnt[lid] = finite ? sturm_count(d, e2, n, als_tau(kmin + lid) * hi) : n;
  }
  __syncthreads();
  const double lmax = lim[1];
  double2* M = side == 0 ? sm.MA : sm.MB;
  if (!finite || !(lmax > 0.0)) {
    if (!finite && tid == 0 && !isfinite(mxe)) sm.err |= WHY_ALS_QR;
    for (int i = tid; i < n; i += NTU_CTA) M[i] = cz();
    if (tid == 0) sm.tau_sel = als_tau(kmin);
    __syncthreads();
    return;
  }
  const int m = n > 1 ? cnt[0] : 0;                         // those the selection may drop
  if (n == 1 && tid == 0) sm.flag = 0;                      // a single eigenvalue: the plain rule
  __syncthreads();
  if (m > 0) {
    // eigenvalues 0 .. m-1 by bisection, 32 / 2^ceil(log2 m) sections each
    int lanes = 32;
    while (lanes > 1 && lanes * m > 32) lanes >>= 1;
    const int per = 32 / lanes, i = wid * per + lid / lanes, s = lid % lanes;
    if (wid * per < m) {
      const int want = i < m ? i : m - 1;
      double lo = lim[0], hi = als_tau(kmin) * lmax;
      const unsigned grp = (lanes == 32 ? 0xffffffffu : ((1u << lanes) - 1u)) << (lid - s);
      for (int it = 0; it < 60 && __any_sync(0xffffffffu, hi - lo > 0x1p-55); ++it) {
        const double h = hi - lo, x = lo + h * ((s + 1) / (double)(lanes + 1));
        const unsigned above =
            __ballot_sync(0xffffffffu, sturm_count(d, e2, n, x) > want) & grp;
        const int f = above ? __ffs(above) - 1 : lid - s + lanes;   // first lane at or above
        const double h2 = __shfl_sync(0xffffffffu, x, f & 31), l2 = __shfl_sync(0xffffffffu, x, (f + 31) & 31);
        if (f < lid - s + lanes) hi = h2;
        if (f > lid - s) lo = l2;
      }
      if (s == 0 && i < m) dv[i] = 0.5 * (lo + hi);
    }
    __syncthreads();
    // their vectors: inverse iteration, a thread per vector, three rounds
    double *u0 = log.c, *u1 = u0 + (size_t)n * m, *u2 = u1 + (size_t)n * m, *ll = u2 + (size_t)n * m;
    if (tid < m) {
      tri_factor(d, e, n, dv[tid], u0 + tid, u1 + tid, u2 + tid, ll + tid, log.k + tid, m);
      unsigned r = 0x9e3779b9u * (tid + 1);
      for (int k = 0; k < n; ++k) {
        r ^= r << 13; r ^= r >> 17; r ^= r << 5;
        W[(size_t)tid * n + k] = (int)r * 0x1p-31;
      }
    }
    for (int round = 0; round < 3; ++round) {
      if (tid < m)
        tri_solve(n, u0 + tid, u1 + tid, u2 + tid, ll + tid, log.k + tid, m, W + (size_t)tid * n, 1);
      __syncthreads();
      tri_orthonormalise(sm, W, n, m, reinterpret_cast<double*>(coef));
    }
    // every pair has to satisfy T w = lambda w; y_i = w_i^T y
    for (int q = wid; q < m; q += NTU_WARPS) {
      const double* w = W + (size_t)q * n;
      const double lam = dv[q];
      double rs = 0.0, ws = 0.0;
      double2 yw = cz();
      for (int k = lid; k < n; k += 32) {
        double t = (d[k] - lam) * w[k];
        if (k > 0) t = fma(e[k - 1], w[k - 1], t);
        if (k + 1 < n) t = fma(e[k], w[k + 1], t);
        rs = fma(t, t, rs);
        ws = fma(w[k], w[k], ws);
        yw.x = fma(w[k], sm.y[k].x, yw.x); yw.y = fma(w[k], sm.y[k].y, yw.y);
      }
      rs = warp_sum(rs);
      ws = warp_sum(ws);
      yw = warp_sum2(yw);
      if (lid == 0) {
        coef[q] = yw;
        if (!(rs <= 1e-26) || !(fabs(ws - 1.0) <= 1e-12)) sm.flag = 0;
      }
    }
    __syncthreads();
  }
  if (!sm.flag) {
    for (int i = tid; i < n; i += NTU_CTA) { dv[i] = d[i] * up; ev[i] = e[i] * up; }
    __syncthreads();
    tri_select_serial(sm, a, dv, ev, n, log);
  } else {
    // selection: |y_i|^2 / lambda_i gained by keeping the pairs below the
    // largest threshold; the first pair kept at tolerance k is cnt[k]
    if (tid == 0) {
      double all = 0.0, part = 0.0;
      for (int q = cnt[nk - 1]; q < m; ++q) all += cabs2(coef[q]) / (dv[q] * up);
      int k = 0;
      for (; k < nk - 1; ++k) {
        part = 0.0;
        for (int q = cnt[nk - 1]; q < cnt[k]; ++q) part += cabs2(coef[q]) / (dv[q] * up);
        if (sm.eps0 - (all - part) <= sm.eps0 - all + 1e-14 * sm.eps0) break;
      }
      sm.tau_sel = als_tau(kmin + k);
      *ndrop = cnt[k];
    }
    __syncthreads();
    const int drop = *ndrop;
    if (m == n) {
      double2 v = cz();
      if (tid < n)
        for (int q = drop; q < n; ++q) {
          const double f = W[(size_t)q * n + tid] / dv[q];
          v.x = fma(f, coef[q].x, v.x); v.y = fma(f, coef[q].y, v.y);
        }
      __syncthreads();
      if (tid < n) sm.y[tid] = cscale(v, down);
      __syncthreads();
    } else {
      tri_project(W, n, drop, sm.y, coef);
      double *u0 = e2, *u1 = u0 + 256, *u2 = u1 + 256, *ll = u2 + 256;    // y2 and p
      double2* rhs = reinterpret_cast<double2*>(log.s);
      if (tid == 0) tri_factor(d, e, n, 0.0, u0, u1, u2, ll, log.k, 1);
      if (tid < n) rhs[tid] = sm.y[tid];
      __syncthreads();
      double2 x = cz();
      for (int pass = 0; pass < 2; ++pass) {                // solve, then one refinement
        // the real and the imaginary part by one thread each
        if (tid < 2) tri_solve(n, u0, u1, u2, ll, log.k, 1, reinterpret_cast<double*>(sm.y) + tid, 2);
        __syncthreads();
        tri_project(W, n, drop, sm.y, coef);
        if (tid < n) x = cadd(x, sm.y[tid]);
        __syncthreads();
        if (pass == 0) {
          if (tid < n) {
            double2 t = make_double2(fma(-d[tid], x.x, rhs[tid].x), fma(-d[tid], x.y, rhs[tid].y));
            if (tid > 0) t = make_double2(fma(-e[tid - 1], sm.y[tid - 1].x, t.x), fma(-e[tid - 1], sm.y[tid - 1].y, t.y));
            if (tid + 1 < n) t = make_double2(fma(-e[tid], sm.y[tid + 1].x, t.x), fma(-e[tid], sm.y[tid + 1].y, t.y));
            coef[tid] = t;
          }
          __syncthreads();
          if (tid < n) sm.y[tid] = coef[tid];
          __syncthreads();
          tri_project(W, n, drop, sm.y, coef);
        }
      }
      if (tid < n) sm.y[tid] = cscale(x, down);
      __syncthreads();
    }
  }
  // back: M = Q D v
  if (tid < n) sm.y[tid] = cmul(ph[tid], sm.y[tid]);
  __syncthreads();
  if (wid == 0)
    for (int j = n - 3; j >= 0; --j) {
      const double c = cfac[j];
      if (c == 0.0) continue;
      const int mm = n - 1 - j, b = j + 1;
      const double2* v = A.a + A.off(j) + b;
      double2 s = cz();
      for (int i = lid; i < mm; i += 32) s = cfmac(v[i], sm.y[b + i], s);
      s = cscale(warp_sum2(s), c);
      for (int i = lid; i < mm; i += 32) sm.y[b + i] = cfms(s, v[i], sm.y[b + i]);
      __syncwarp();
    }
  __syncthreads();
  for (int i = tid; i < n; i += NTU_CTA) M[i] = sm.y[i];
  __syncthreads();
}

}  // namespace ntu
