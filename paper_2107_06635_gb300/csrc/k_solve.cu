// FP64 solvers of the bond update: Hermitisation and non-negativity repair
// of the metric g (Sec. II), the slicing of g for the tensor-core build of
// the ALS reduced metric, and the host side of the ALS truncation of Fig. 5
// (argument set-up and the choice of instantiation; the kernel is in
// als_kernel.cuh).  One CTA per bond update.
#include <cuda_runtime.h>
#include <math.h>

#include <type_traits>

#include "ntu_dev.cuh"
#include "ntu_impl.h"
#include "als_types.cuh"
#include "oz_build.cuh"

namespace ntu {

__device__ __forceinline__ double2 ld2(const double2* p) { return *p; }
__device__ __forceinline__ double2 ld2(const float2* p) {
  float2 v = *p;
  return make_double2((double)v.x, (double)v.y);
}

// ------------------------------------------------------------- repair
// g <- (g + g^H)/2.  g is positive definite, and clipping its negative
// eigenvalues would change nothing, when the Gershgorin discs of the rows
// lie right of zero (min_i d_i - s_i > 0, s_i = sum_{j != i} |Re| + |Im| >=
// sum_{j != i} |g_ij|) or, failing that, when a triangular factorisation of g
// succeeds; otherwise g = W diag(max(lambda, 0)) W^H from a full
// eigendecomposition.  Finally g /= trace(g).
// diag = [||g - g^H|| / ||g||, lambda_min / lambda_max (NaN on the two
// certified paths), log(trace)].
//
// The discs decide almost every metric of a batch, so they are taken grid-wide
// in three streaming kernels: row statistics (a block per 32 rows; the entries
// (c, r) come in 32 x 32 tiles turned in shared memory), the decision (a block
// per item) and the scaled result (a block per pair of mirrored tiles).  One
// block per item with strided reads of the mirrored entries held a K = 32
// metric for 4 ms on one SM; now 45 of them take 0.65 ms, 912 at K = 16 0.90
// against 1.24 ms.  k_repair then runs for the undecided items only.
struct RowStat {
  double d, lo;                 // diagonal entry, disc's left end
};
// Shift of the FP32 certificate (k_herm_certify), and the multiple of it below
// which a diagonal entry says that the attempt would hardly pass.
__device__ __forceinline__ double cert_shift(int n, double tr) { return 6.0 * (n + 3) * 0x1p-24 * tr; }
constexpr double CERT_DIAG = 3.0;

template <typename C2in>
__global__ void __launch_bounds__(256) k_herm_stats(int ng, const C2in* __restrict__ graw,
                                                    RowStat* __restrict__ rows,
                                                    double2* __restrict__ part) {
  constexpr bool F32 = std::is_same<C2in, float2>::value;
  typedef typename std::conditional<F32, float, double>::type R;
  __shared__ C2in tb[32][33];
  __shared__ double red[2 * NTU_WARPS];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, r0 = blockIdx.x * 32;
  const long long item = blockIdx.y;
  const C2in* gr = graw + item * (long long)ng * ng;
  C2in zero;
  zero.x = 0; zero.y = 0;
  R sr[4] = {0, 0, 0, 0}, n2 = 0, h2 = 0;
  double dr[4] = {0.0, 0.0, 0.0, 0.0};
  for (int c0 = 0; c0 < ng; c0 += 32) {
    C2in a[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = r0 + w + 8 * i, c = c0 + w + 8 * i;
      a[i] = r < ng && c0 + lane < ng ? gr[(size_t)r * ng + c0 + lane] : zero;
      tb[w + 8 * i][lane] = c < ng && r0 + lane < ng ? gr[(size_t)c * ng + r0 + lane] : zero;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const C2in b = tb[lane][w + 8 * i];                   // entry (c, r)
      const R dx = a[i].x - b.x, dy = a[i].y + b.y;
      n2 = fma(a[i].x, a[i].x, fma(a[i].y, a[i].y, n2));
      h2 = fma(dx, dx, fma(dy, dy, h2));
      if (r0 + w + 8 * i == c0 + lane) dr[i] = (double)a[i].x;
      else sr[i] += (R)0.5 * (fabs(a[i].x + b.x) + fabs(a[i].y - b.y));
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = r0 + w + 8 * i;
    const double d = warp_sum(dr[i]);                       // one lane holds it
    // relative rounding of the radius below 2e-5 in FP32 (n_g <= 1024 terms)
    const double s = F32 ? (double)warp_sum_f((float)sr[i]) * (1.0 + 1e-4)
                         : warp_sum((double)sr[i]) * (1.0 + 1e-12);
    if (lane == 0 && r < ng) rows[item * ng + r] = RowStat{d, d - s};
  }
  const double2 t = block_sum2(make_double2((double)n2, (double)h2), red);
  if (threadIdx.x == 0) part[item * ng + blockIdx.x] = t;
}

// scale[item] = 1 / (2 tr) where the discs decide, else 0.  The trace is
// summed as k_repair sums it (rows r, r + 8, ... by warp, then the warps).
__global__ void __launch_bounds__(NTU_CTA) k_herm_decide(int ng, const RowStat* __restrict__ rows,
                                                         const double2* __restrict__ part,
                                                         double* __restrict__ scale,
                                                         double* __restrict__ trace,
                                                         double* __restrict__ diag, int* __restrict__ cert,
                                                         int* paths) {
  __shared__ double red[2 * NTU_WARPS], tw[NTU_WARPS];
  const int tid = threadIdx.x, wid = tid >> 5, lid = tid & 31;
  const long long item = blockIdx.x;
  const RowStat* rs = rows + item * ng;
  double lo = INFINITY, dmin = INFINITY;
  for (int r = tid; r < ng; r += NTU_CTA) {
    lo = fmin(lo, rs[r].lo);
    dmin = fmin(dmin, rs[r].d);
  }
  lo = block_min(lo, red);
  dmin = block_min(dmin, red);
  if (lid == 0) {
    double t = 0.0;
    for (int r = wid; r < ng; r += NTU_WARPS) t += rs[r].d;
    tw[wid] = t;
  }
  __syncthreads();
  if (tid == 0) {
    double tr = 0.0, n2 = 0.0, h2 = 0.0;
    for (int w = 0; w < NTU_WARPS; ++w) tr += tw[w];
    for (int b = 0; b < (ng + 31) / 32; ++b) { n2 += part[item * ng + b].x; h2 += part[item * ng + b].y; }
    const bool ok = lo > 0.0 && isfinite(lo) && tr > 0.0 && isfinite(tr);
    scale[item] = ok ? 0.5 / tr : 0.0;
    trace[item] = tr;
    cert[item] = ok || dmin > CERT_DIAG * cert_shift(ng, tr) ? 0 : -1;
    diag[item * 3 + 0] = n2 > 0.0 ? sqrt(h2 / n2) : 0.0;
    if (ok) {
      if (paths) atomicAdd(paths + 3, 1);
      diag[item * 3 + 1] = __longlong_as_double(0x7ff8000000000000ULL);   // NaN
      diag[item * 3 + 2] = log(tr);
    }
  }
}

// The decided items: g = (graw + graw^H) / (2 tr), tile (I, J), I >= J, and its
// mirror image, turned in shared memory: each pair of entries is converted and
// scaled once (FP64 operations and conversions bound this kernel).
template <typename C2in>
__global__ void __launch_bounds__(256) k_herm_write(int ng, const C2in* __restrict__ graw,
                                                    const double* __restrict__ scale,
                                                    double2* __restrict__ g) {
  __shared__ double2 t[32][33];
  const long long item = blockIdx.y;
  const double hinv = scale[item];
  if (hinv == 0.0) return;
  int I = (int)((sqrtf(8.0f * (float)blockIdx.x + 1.0f) - 1.0f) * 0.5f);
  while ((I + 1) * (I + 2) / 2 <= (int)blockIdx.x) ++I;
  while (I > 0 && I * (I + 1) / 2 > (int)blockIdx.x) --I;
  const int J = (int)blockIdx.x - I * (I + 1) / 2;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, r0 = I * 32, c0 = J * 32;
  const C2in* gr = graw + item * (long long)ng * ng;
  double2* gi = g + item * (long long)ng * ng;
  C2in* tb = reinterpret_cast<C2in*>(&t[0][0]);             // [32][33] of the raw type first
  C2in a[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int k = w + 8 * i;
    if (r0 + k < ng && c0 + lane < ng) a[i] = gr[(size_t)(r0 + k) * ng + c0 + lane];
    if (c0 + k < ng && r0 + lane < ng) tb[k * 33 + lane] = gr[(size_t)(c0 + k) * ng + r0 + lane];
  }
  __syncthreads();
  double2 h[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int k = w + 8 * i;
    if (r0 + k < ng && c0 + lane < ng) {
      const double2 u = ld2(&a[i]), v = ld2(&tb[lane * 33 + k]);
      h[i] = make_double2((u.x + v.x) * hinv, (u.y - v.y) * hinv);
      gi[(size_t)(r0 + k) * ng + c0 + lane] = h[i];
    }
  }
  if (I == J) return;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 4; ++i) t[w + 8 * i][lane] = h[i];
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int k = w + 8 * i;
    if (c0 + k < ng && r0 + lane < ng) gi[(size_t)(c0 + k) * ng + r0 + lane] = cconj(t[lane][k]);
  }
}

// The three in one, a block per item with a warp per row, for metrics whose
// mirrored entries lie in L1: up to n_g = 64 the launches cost more than the
// strided reads (n_g = 16, 48 metrics: 20 us a repair, 33 with three launches).
constexpr int HERM_SMALL = 64;
template <typename C2in>
__global__ void __launch_bounds__(NTU_CTA) k_herm_small(int ng, const C2in* __restrict__ graw,
                                                        double2* __restrict__ g, double* __restrict__ scale,
                                                        double* __restrict__ trace, double* __restrict__ diag,
                                                        int* __restrict__ cert, int* paths) {
  constexpr bool F32 = std::is_same<C2in, float2>::value;
  typedef typename std::conditional<F32, float, double>::type R;
  __shared__ double red[2 * NTU_WARPS], tw[NTU_WARPS];
  const int tid = threadIdx.x, wid = tid >> 5, lid = tid & 31;
  const long long item = blockIdx.x;
  const C2in* gr = graw + item * (long long)ng * ng;
  double2* gi = g + item * (long long)ng * ng;
  R n2 = 0, h2 = 0;
  double lo = INFINITY, dmin = INFINITY, t = 0.0;
  for (int r = wid; r < ng; r += NTU_WARPS) {
    R sr = 0;
    double dr = 0.0;
    for (int c = lid; c < ng; c += 32) {
      const C2in a = gr[r * ng + c], b = gr[c * ng + r];
      const R dx = a.x - b.x, dy = a.y + b.y;
      n2 = fma(a.x, a.x, fma(a.y, a.y, n2));
      h2 = fma(dx, dx, fma(dy, dy, h2));
      if (c == r) dr = (double)a.x;
      else sr += (R)0.5 * (fabs(a.x + b.x) + fabs(a.y - b.y));
    }
    const double d = warp_sum(dr);
    const double s = F32 ? (double)warp_sum_f((float)sr) * (1.0 + 1e-4)
                         : warp_sum((double)sr) * (1.0 + 1e-12);
    lo = fmin(lo, d - s);
    dmin = fmin(dmin, d);
    t += d;
  }
  lo = block_min(lo, red);
  dmin = block_min(dmin, red);
  const double2 def = block_sum2(make_double2((double)n2, (double)h2), red);
  if (lid == 0) tw[wid] = t;
  __syncthreads();
  double tr = 0.0;
  for (int w = 0; w < NTU_WARPS; ++w) tr += tw[w];
  const bool ok = lo > 0.0 && isfinite(lo) && tr > 0.0 && isfinite(tr);
  const double hinv = 0.5 / tr;
  if (ok)
    for (int idx = tid; idx < ng * ng; idx += NTU_CTA) {
      const double2 u = ld2(gr + idx), v = ld2(gr + (idx % ng) * ng + idx / ng);
      gi[idx] = make_double2((u.x + v.x) * hinv, (u.y - v.y) * hinv);
    }
  if (tid == 0) {
    scale[item] = ok ? hinv : 0.0;
    trace[item] = tr;
    cert[item] = ok || dmin > CERT_DIAG * cert_shift(ng, tr) ? 0 : -1;
    diag[item * 3 + 0] = def.x > 0.0 ? sqrt(def.y / def.x) : 0.0;
    if (ok) {
      if (paths) atomicAdd(paths + 3, 1);
      diag[item * 3 + 1] = __longlong_as_double(0x7ff8000000000000ULL);   // NaN
      diag[item * 3 + 2] = log(tr);
    }
  }
}

// Whether H - delta I (H row-major, Hermitian) has an L D L^H
// factorisation in FP32, delta = 6 (n + 3) 2^-24 tr H: the rounding of the
// factorisation is a perturbation of at most 4 (n + 2) 2^-24 |L| |D| |L|^H,
// whose norm is below 4 (n + 2) 2^-24 tr H for a positive definite matrix, and
// that of the entries below 2^-24 tr H, so success proves H positive definite.
// It decides metrics with lambda_min above some 1e-4 tr H at 64 times the FP64
// rate (n = 400: 3.1 ms, bound by the trailing columns' traffic to L2, where the
// FP64 Cholesky held the SM's FP64 pipe for 21 ms and the double-FP32 one 10 ms); a
// warp per column, four rows a lane in flight.  A metric with a diagonal entry
// below the shift cannot pass, and one below three times it hardly does: such a
// metric (of a state part-way into a run, graded) is left alone, and where all
// items run at once (n <= lone) so is the whole batch, which lasts as long as its
// longest item: there the attempt had made the repair up to 31% longer (24 items at
// D = 6: 1.12 ms, 0.87 now; one at D = 2, r = 16: 150, 124).
// cert[item] = 1 where it succeeds (0 before; -1: left alone); a block of
// CERT_THREADS per item.
constexpr int CERT_THREADS = 1024;
template <typename C2in>
__global__ void __launch_bounds__(CERT_THREADS) k_herm_certify(int n, const C2in* __restrict__ graw,
                                                               const double* __restrict__ scale,
                                                               const double* __restrict__ traces,
                                                               double2* __restrict__ scr, int lone,
                                                               int* __restrict__ cert) {
  __shared__ float2 col[1024];                              // n_g <= 1024
  const long long item = blockIdx.x;
  const int tid = threadIdx.x, wid = tid >> 5, lid = tid & 31;
  if (scale[item] != 0.0 || cert[item] < 0) return;         // decided by the discs; left alone
  if ((int)gridDim.x <= lone && __syncthreads_or(tid < (int)gridDim.x && cert[tid] < 0)) return;
  const double trace = traces[item];
  if (!(trace > 0x1p-900) || !(trace < 0x1p900)) return;
  const double f = scalbn(1.0, -ilogb(trace)), delta = cert_shift(n, trace);
  const C2in* gr = graw + item * (long long)n * n;
  float2* A = reinterpret_cast<float2*>(scr + item * (long long)n * n);
  for (int idx = tid; idx < n * n; idx += CERT_THREADS) {
    const int k = idx / n, i = idx % n;                     // column k, row i: conj of (k, i)
    if (i < k) continue;
    const double2 a = ld2(gr + idx), b = ld2(gr + (size_t)i * n + k);
    double hx = 0.5 * (a.x + b.x);
    if (i == k) hx -= delta;
    A[idx] = make_float2((float)(hx * f), (float)(-0.5 * (a.y - b.y) * f));
  }
  __syncthreads();
  for (int j = 0; j < n; ++j) {
    const float2* c = A + (size_t)j * n;
    const float d = c[j].x;
    if (!(d > 0.f) || !isfinite(d)) return;                 // the same in every thread
    const float r = 1.0f / d;
    for (int i = j + 1 + tid; i < n; i += CERT_THREADS) col[i] = c[i];
    __syncthreads();
    for (int k = j + 1 + wid; k < n; k += CERT_THREADS / 32) {   // a_ik -= c_i conj(c_k) / d
      const float2 ck = col[k];
      const float lx = ck.x * r, ly = ck.y * r;
      float2* ak = A + (size_t)k * n;
      for (int i0 = k + lid; i0 < n; i0 += 128) {
        float2 x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (i0 + 32 * u < n) x[u] = ak[i0 + 32 * u];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int i = i0 + 32 * u;
          if (i < n) {
            const float2 ci = col[i];
            x[u].x = fmaf(-ci.x, lx, fmaf(-ci.y, ly, x[u].x));
            x[u].y = fmaf(-ci.y, lx, fmaf(ci.x, ly, x[u].y));
            ak[i] = x[u];
          }
        }
      }
    }
    __syncthreads();
  }
  if (tid == 0) cert[item] = 1;
}

template <typename C2in>
__global__ void __launch_bounds__(NTU_CTA) k_repair(int ng, const C2in* __restrict__ graw,
                                                    double2* __restrict__ g,
                                                    double2* __restrict__ scr,
                                                    double2* __restrict__ Wv,
                                                    double* __restrict__ Z,
                                                    double* __restrict__ de,
                                                    double2* __restrict__ tau,
                                                    double2* __restrict__ pv,
                                                    double* __restrict__ diag, int* status,
                                                    int* paths,
                                                    const double* __restrict__ scale,
                                                    const int* __restrict__ cert) {
  if (scale[blockIdx.x] != 0.0) return;             // decided by the discs
  extern __shared__ __align__(16) double chain[];   // 2 * ng (also n_g float4 for the Cholesky)
  __shared__ double sred[2 * NTU_WARPS];
  __shared__ int sh[4];
  __shared__ int okflag;
  const int tid = threadIdx.x;
  const long long item = blockIdx.x;
  const size_t nn = (size_t)ng * ng;
  const C2in* gr = graw + item * nn;
  double2* gi = g + item * nn;
  double2* sc = scr + item * nn;
  for (size_t idx = tid; idx < nn; idx += NTU_CTA) {
    int r = idx / ng, c = idx % ng;
    double2 a = ld2(gr + idx), b = ld2(gr + (size_t)c * ng + r);
    gi[idx] = make_double2(0.5 * (a.x + b.x), 0.5 * (a.y - b.y));
  }
  __syncthreads();
  // 1. a triangular factorisation certifies positive definiteness: in FP32
  // with room for its rounding (k_herm_certify), else in double-FP32 for an FP32 raw metric
  // (mixed contexts; it resolves it far below its own rounding), in FP64
  // otherwise
  constexpr bool kDf = std::is_same<C2in, float2>::value;
  int ok = cert[item] > 0;
  if (!ok) {
    for (size_t idx = tid; idx < nn; idx += NTU_CTA) {      // column-major copy
      const size_t t = (idx % ng) * ng + idx / ng;
      if (kDf) reinterpret_cast<float4*>(sc)[t] = df_split(gi[idx]);
      else sc[t] = gi[idx];
    }
    __syncthreads();
    ok = kDf ? cta_cholesky_df(reinterpret_cast<float4*>(sc), ng, &okflag,
                               reinterpret_cast<float4*>(chain))
             : cta_cholesky(sc, ng, 0.0, &okflag);
  }
  if (tid == 0 && paths) atomicAdd(paths + (ok ? 4 : 5), 1);
  double ratio = __longlong_as_double(0x7ff8000000000000ULL);   // NaN
  if (!ok) {
    // 2. full eigendecomposition and clipping of negative eigenvalues
    double2* ta = tau + item * ng;
    double2* pp = pv + item * ng;
    double* dd = de + item * 2 * ng;
    double* ee = dd + ng;
    double* Zi = Z + item * nn;
    double2* Wi = Wv + item * nn;
    for (size_t idx = tid; idx < nn; idx += NTU_CTA) {
      int r = idx / ng, c = idx % ng;
      sc[(size_t)c * ng + r] = gi[idx];
    }
    __syncthreads();
    cta_hetrd(sc, ng, dd, ee, ta, pp, sred);
    int st = cta_tridiag_qr_z(dd, ee, ng, Zi, chain, sh);
    if (st && tid == 0) raise_status(status, st, WHY_REPAIR_QR);
    // W = Q Z, one column per thread
    for (int k = tid; k < ng; k += NTU_CTA) {
      double2* col = Wi + (size_t)k * ng;
      for (int i = 0; i < ng; ++i) col[i] = make_double2(Zi[(size_t)i * ng + k], 0.0);
      for (int j = ng - 2; j >= 0; --j) {
        double2 t = ta[j];
        if (t.x == 0.0 && t.y == 0.0) continue;
        const double2* v = sc + (size_t)j * ng + j + 1;
        int m = ng - j - 1;
        double2 s = cz();
        for (int i = 0; i < m; ++i) s = cfmac(i == 0 ? make_double2(1.0, 0.0) : v[i], col[j + 1 + i], s);
        double2 f = cmul(t, s);
        for (int i = 0; i < m; ++i)
          col[j + 1 + i] = csub(col[j + 1 + i], cmul(f, i == 0 ? make_double2(1.0, 0.0) : v[i]));
      }
    }
    __syncthreads();
    double lmin = dd[0], lmax = dd[0];
    for (int i = 1; i < ng; ++i) { lmin = fmin(lmin, dd[i]); lmax = fmax(lmax, dd[i]); }
    ratio = lmax > 0.0 ? lmin / lmax : 0.0;
    for (size_t idx = tid; idx < nn; idx += NTU_CTA) {
      int r = idx / ng, c = idx % ng;
      double2 acc = cz();
      for (int k = 0; k < ng; ++k) {
        double lk = dd[k];
        if (lk <= 0.0) continue;
        acc = cfma(cscale(Wi[(size_t)k * ng + r], lk), cconj(Wi[(size_t)k * ng + c]), acc);
      }
      gi[idx] = acc;
    }
    __syncthreads();
  }
  // 3. unit trace
  double tr = 0.0;
  for (int i = tid; i < ng; i += NTU_CTA) tr += gi[(size_t)i * ng + i].x;
  tr = block_sum(tr, sred);
  if (!(tr > 0.0) || !isfinite(tr)) {
    if (tid == 0) raise_status(status, ST_NUMERIC, WHY_REPAIR_TRACE);
    tr = 1.0;
  }
  const double inv = 1.0 / tr;
  for (size_t idx = tid; idx < nn; idx += NTU_CTA) gi[idx] = cscale(gi[idx], inv);
  if (tid == 0) {
    diag[item * 3 + 1] = ratio;
    diag[item * 3 + 2] = log(tr);
  }
}

// ------------------------------------------- double-FP32 copy of g
// The mixed contexts' ALS reads g as double-FP32 pairs gdf = g 2^-e.  e = 0
// while max |Re|, |Im| lies in [2^-60, 2^60] (products and sums of the
// build then stay far inside the FP32 range); otherwise 2^e is the power of
// two just above the maximum, an exact scaling.  Two streaming passes over
// the batch, spread over every SM: the largest |Re|, |Im| of each item, then
// the split; for the lane build of the reduced metric also the copy
// gdfT[(kB',kA'),(kB,kA)] = gdf[(kA',kB'),(kA,kB)], which lets the B step
// read its blocks along rows as the A step does.  The maximum is taken on
// the bit patterns, whose order is that of the non-negative values; NaN
// entries are skipped.
__global__ void __launch_bounds__(NTU_CTA) k_gmax(long long nn, const double2* __restrict__ g,
                                                  unsigned long long* __restrict__ gmax) {
  __shared__ unsigned long long red[NTU_WARPS];
  const long long item = blockIdx.y;
  const double2* gi = g + item * nn;
  unsigned long long m = 0;
  for (long long i = blockIdx.x * (long long)NTU_CTA + threadIdx.x; i < nn;
       i += (long long)gridDim.x * NTU_CTA) {
    const double2 v = gi[i];
    unsigned long long a = dfb_bits(v.x) & 0x7fffffffffffffffull;
    unsigned long long b = dfb_bits(v.y) & 0x7fffffffffffffffull;
    if (a > 0x7ff0000000000000ull) a = 0;
    if (b > 0x7ff0000000000000ull) b = 0;
    m = max(m, max(a, b));
  }
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < NTU_WARPS; ++w) m = max(m, red[w]);
    atomicMax(gmax + item, m);
  }
}

__device__ __forceinline__ int gscale_exp(unsigned long long mb) {
  const double mx = dfb_double(mb);
  return (mx > 0.0 && isfinite(mx) && (mx > 0x1p60 || mx < 0x1p-60)) ? ilogb(mx) + 1 : 0;
}

// Without the swapped copy a thread loads four entries of the item before
// it splits and stores them (one load at a time left the kernel latency-
// bound at a sixth of the HBM rate, measured); with it, one row of g per
// block iteration: row r of gdf is written in place, and row
// r' = (r mod K) K + r / K of gdfT, whose entry (c mod K) K + c / K is entry
// c of row r, from a copy staged in shared memory, so that both writes are
// contiguous, while the next row's entries are already being loaded.
constexpr int GSPLIT_BATCH = 4;
__global__ void __launch_bounds__(NTU_CTA) k_gsplit(int ng, int K, const double2* __restrict__ g,
                                                    const unsigned long long* __restrict__ gmax,
                                                    int* __restrict__ gscale,
                                                    float4* __restrict__ gdf,
                                                    float4* __restrict__ gdfT) {
  __shared__ float4 row[1024];                          // ng <= 1024
  const long long item = blockIdx.y, nn = (long long)ng * ng;
  const int e = gscale_exp(gmax[item]);
  if (blockIdx.x == 0 && threadIdx.x == 0) gscale[item] = e;
  const double2* gi = g + item * nn;
  float4* di = gdf + item * nn;
  if (!gdfT) {
    const long long step = (long long)gridDim.x * NTU_CTA;
    for (long long i0 = blockIdx.x * (long long)NTU_CTA + threadIdx.x; i0 < nn;
         i0 += GSPLIT_BATCH * step) {
      double2 v[GSPLIT_BATCH];
#pragma unroll
      for (int u = 0; u < GSPLIT_BATCH; ++u) {
        const long long i = i0 + u * step;
        v[u] = i < nn ? gi[i] : make_double2(0.0, 0.0);
      }
#pragma unroll
      for (int u = 0; u < GSPLIT_BATCH; ++u) {
        const long long i = i0 + u * step;
        if (i < nn) {
          if (e != 0) v[u] = make_double2(scalbn(v[u].x, -e), scalbn(v[u].y, -e));
          di[i] = df_split_bits(v[u]);
        }
      }
    }
    return;
  }
  float4* ti = gdfT + item * nn;
  constexpr int PER = 1024 / NTU_CTA;                   // entries of a row per thread, at most
  double2 cur[PER], nxt[PER];
  auto load_row = [&](int r, double2* dst) {
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      const int c = threadIdx.x + u * NTU_CTA;
      dst[u] = (r < ng && c < ng) ? gi[(size_t)r * ng + c] : make_double2(0.0, 0.0);
    }
  };
  load_row(blockIdx.x, cur);
  for (int r = blockIdx.x; r < ng; r += gridDim.x) {
    load_row(r + gridDim.x, nxt);
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      const int c = threadIdx.x + u * NTU_CTA;
      if (c < ng) {
        double2 v = cur[u];
        if (e != 0) v = make_double2(scalbn(v.x, -e), scalbn(v.y, -e));
        const float4 d = df_split_bits(v);
        di[(size_t)r * ng + c] = d;
        row[(c % K) * K + c / K] = d;
      }
    }
    __syncthreads();
    float4* tr = ti + (size_t)((r % K) * K + r / K) * ng;
    for (int c = threadIdx.x; c < ng; c += NTU_CTA) tr[c] = row[c];
    __syncthreads();
#pragma unroll
    for (int u = 0; u < PER; ++u) cur[u] = nxt[u];
  }
}

size_t als_smem_bytes() { return sizeof(AlsShared); }

long long oz_rows_side(int K) { return oz_supported(K) ? oz_geo(K).rows_side : 0; }

template <typename C2in>
static cudaError_t run_repair(ntu_ctx* c, int n, const C2in* graw, double2* g, double* diag) {
  const Plan& P = c->plan;
  Work& W = c->w;
  RowStat* rows = reinterpret_cast<RowStat*>(W.gtau);       // n_g entries of 16 bytes per item
  double* scale = reinterpret_cast<double*>(W.x0);          // ALS scratch, free here
  double* trace = scale + n;
  int* cert = reinterpret_cast<int*>(W.gx0);                // ALS scratch, free here
  cudaError_t e;
  if (P.ng <= HERM_SMALL) {
    k_herm_small<C2in><<<n, NTU_CTA, 0, c->stream>>>(P.ng, graw, g, scale, trace, diag, cert,
                                                          c->d_paths);
    e = after_launch(c, "k_herm_small");
    if (e != cudaSuccess) return e;
  } else {
    const int nb = (P.ng + 31) / 32;
    k_herm_stats<C2in><<<dim3((unsigned)nb, (unsigned)n), 256, 0, c->stream>>>(P.ng, graw, rows, W.gp);
    e = after_launch(c, "k_herm_stats");
    if (e != cudaSuccess) return e;
    k_herm_decide<<<n, NTU_CTA, 0, c->stream>>>(P.ng, rows, W.gp, scale, trace, diag, cert, c->d_paths);
    e = after_launch(c, "k_herm_decide");
    if (e != cudaSuccess) return e;
    k_herm_write<C2in><<<dim3((unsigned)(nb * (nb + 1) / 2), (unsigned)n), 256, 0, c->stream>>>(
        P.ng, graw, scale, g);
    e = after_launch(c, "k_herm_write");
    if (e != cudaSuccess) return e;
  }
  // the FP32 certificate: from n_g = 33 on, below which the exact factorisation
  // takes no longer than its launch
  if (P.ng > 32) {
    const int lone = c->sms < CERT_THREADS ? c->sms : CERT_THREADS;
    k_herm_certify<C2in><<<n, CERT_THREADS, 0, c->stream>>>(P.ng, graw, scale, trace, W.gscr, lone, cert);
    e = after_launch(c, "k_herm_certify");
    if (e != cudaSuccess) return e;
  }
  const size_t sm = 2 * sizeof(double) * P.ng;             // at most 16 KB: no limit to set
  k_repair<C2in><<<n, NTU_CTA, sm, c->stream>>>(P.ng, graw, g, W.gscr, W.gw, W.gz, W.geig, W.gtau,
                                                W.gp, diag, c->d_status, c->d_paths, scale, cert);
  return after_launch(c, "k_repair");
}

cudaError_t launch_repair(ntu_ctx* c, int n, const void* graw, int raw_is_f32, double2* g,
                          double* diag) {
  return raw_is_f32 ? run_repair(c, n, (const float2*)graw, g, diag)
                    : run_repair(c, n, (const double2*)graw, g, diag);
}

cudaError_t launch_als(ntu_ctx* c, int n, const double2* g, const double2* RA,
                       const double2* RB, double2* MA, double2* MB, double* info, int sweeps) {
  const Plan& P = c->plan;
  Work& W = c->w;
  AlsArgs a;
  a.D = P.D; a.K = P.K; a.ng = P.ng; a.nA = P.nA;
  a.sweeps = sweeps < 0 ? c->cfg.als_sweeps : sweeps;
  a.kmin = c->cfg.tau_kmin; a.kmax = c->cfg.tau_kmax;
  a.g = g; a.RA = RA; a.RB = RB; a.MA = MA; a.MB = MB; a.info = info;
  a.x0 = W.x0; a.gx0 = W.gx0; a.Tm = W.Tm; a.gA = W.gA; a.gC = W.gC; a.jv = W.jv; a.pv = W.pv;
  a.path_counts = c->d_paths;
  a.tauv = W.tauv; a.dv = W.dv; a.ev = W.ev; a.rc = W.rc; a.rs = W.rs; a.rk = W.rk;
  a.rotcap = W.rotcap; a.status = c->d_status;
  a.df = c->cfg.precision != NTU_FP64;
  a.gdf = reinterpret_cast<float4*>(W.gscr);
  a.gdfT = reinterpret_cast<float4*>(W.gw);     // the repair's eigenvector scratch, free here
  size_t sm = sizeof(AlsShared);
  const int sms = c->sms;
  // a batch that leaves SMs idle gives each item 2 or 4 CTAs (one cluster),
  // as many as keep about one CTA per SM: co-resident CTAs of a cluster
  // mostly share the SM for the work they duplicate.  Measured on GB300:
  // at D = 8 up to one CTA per SM pays, at D <= 4 (a quarter of the solve
  // work per CTA) up to 1.5
  int split = a.df ? W.als_split : 1;
  const long long cap = P.D <= 4 ? 3LL * sms / 2 : (long long)sms;
  if (c->tune.als_split > 0) split = c->tune.als_split;   // ntu_set_tuning (<= W.als_split)
  else
    while (split > 1 && (long long)n * split > cap) split >>= 1;
  a.split = split;
  a.sync = W.als_sync;
  a.wait_polls = c->wait_polls;
  a.sync_extra = c->inject_timeout;
  // the tensor-core build of the reduced metric (K = 16 or 32, on one CTA
  // or a cluster) unless the tuning asks for the lane build.  Measured on
  // GB300 it takes 17-30 % off the ALS at K = 32 and up to 5 % at K = 16,
  // where a few cluster launches favour the lanes by as much
  a.oz = (c->plan.oz_ok && c->tune.als_build != 1) ? 1 : 0;
  a.gsl = reinterpret_cast<__nv_bfloat16*>(W.gsl);
  a.gexp = W.gexp;
  a.gmap = W.gmap;
  a.gscale = W.gscale;
  if (a.df) {
    // the double-FP32 copies of g, on every SM: blocks per item enough for
    // about eight per SM in all
    const long long nn = (long long)P.ng * P.ng;
    long long bx = (8LL * sms + n - 1) / n;
    const long long most = (nn + 4LL * NTU_CTA - 1) / (4LL * NTU_CTA);
    if (bx > most) bx = most;
    if (bx < 1) bx = 1;
    cudaError_t e = cudaMemsetAsync(W.gmaxb, 0, sizeof(unsigned long long) * (size_t)n, c->stream);
    if (e != cudaSuccess) return e;
    k_gmax<<<dim3((unsigned)bx, (unsigned)n), NTU_CTA, 0, c->stream>>>(nn, g, W.gmaxb);
    e = after_launch(c, "k_gmax");
    if (e != cudaSuccess) return e;
    long long bs = (8LL * sms + n - 1) / n;              // blocks per item
    if (bs > P.ng) bs = P.ng;
    k_gsplit<<<dim3((unsigned)bs, (unsigned)n), NTU_CTA, 0, c->stream>>>(
        P.ng, P.K, g, W.gmaxb, W.gscale, a.gdf, a.oz ? nullptr : a.gdfT);
    e = after_launch(c, "k_gsplit");
    if (e != cudaSuccess) return e;
  }
  if (a.oz) {
    // slices of every item's g for the tensor-core build
    const long long tasks = (long long)n * 2 * P.K * P.ng * (P.K / 4);
    long long blocks = (tasks + NTU_CTA - 1) / NTU_CTA;
    if (blocks > 16LL * sms) blocks = 16LL * sms;
    void (*sk)(int, const double2*, __nv_bfloat16*, short*) =
        P.K == 16 ? k_oz_slice<16> : k_oz_slice<32>;
    sk<<<(int)blocks, NTU_CTA, 0, c->stream>>>(n, g, reinterpret_cast<__nv_bfloat16*>(W.gsl),
                                               W.gexp);
    cudaError_t e = after_launch(c, "k_oz_slice");
    if (e != cudaSuccess) return e;
  }
  const size_t smk = sm + (a.oz ? ALS_OZ_SLACK : 0);
  if (split > 1) {
    cudaError_t e = cudaMemsetAsync(W.als_sync, 0, sizeof(int) * (size_t)n, c->stream);
    if (e != cudaSuccess) return e;
  }
  const bool three =
      split == 1 && (c->tune.als_ctas_per_sm ? c->tune.als_ctas_per_sm == 3 : n > 2 * sms);
  cudaError_t e = !a.df ? als_launch_fp64(a, n, split, three, smk, c->stream)
                  : !a.oz ? als_launch_lanes(a, n, split, three, smk, c->stream)
                  : P.K == 16 ? als_launch_tc16(a, n, split, three, smk, c->stream)
                              : als_launch_tc32(a, n, split, three, smk, c->stream);
  if (e != cudaSuccess) return e;
  return after_launch(c, split > 1 ? (a.oz ? "k_als (cluster, tensor-core build)" : "k_als (cluster)")
                                   : (a.oz ? "k_als (tensor-core build)" : "k_als"));
}

}  // namespace ntu
