// FP64 complex GEMMs of the environment contraction (Fig. 4) on the tensor
// cores of the FP64 contexts, by error-free slicing (in the manner of Ozaki,
// Ogita, Oishi and Rump's exact matrix products).
//
// An SM retires two FP64 FMAs per cycle (1.25 TFLOP/s in all), so the FP64
// SIMT environment, at 98% of that, took 92% of a D = 8 bond update; the
// BF16 tensor cores do 1.9 PFLOP/s.  Each row of an operand is scaled by a
// power of two into (-1, 1), rounded to 2^-54 and written as seven signed
// digits of eight bits (|d| <= 128, exact in BF16):
//   x = 2^(e-6) sum_i d_i 2^(-8 i),  i = 0 .. 6.
// A product of two digits is an integer of at most 2^14 (2^13 with a leading
// digit, |d_0| <= 64), so the sums over up to 256 terms of the at most five
// pairs (i, j) of one level l = i + j <= 4 stay within 2^24: their FP32
// accumulators in tensor memory are exact.  Every 256 terms they are drained
// into integer registers; levels 5 to 7 accumulate over all terms, and the
// levels above 7 (below 2^-64) are left out (without level 7 the sums of 12 to
// 32 terms were up to 1.7 times less accurate than the FP64 chain).  Those are
// exact too up to 170 terms; beyond, digits of one sign (equal entries) can
// bring level 5 to 2^16.4 a term, rounded to 24 bits at each of its 6 N / 16
// accumulations: at the N = 8192 of the D = 8 join at most 2^17.6 units of
// 2^-40, i.e. 2^-45 of a sum of equal terms.  With level 4 left to accumulate
// as well the metric of equal entries was off by up to 2.7e-13 at D = 8, where
// the FP64 chain is by 1.1e-13; now by 1.1e-14.  Digits without a pattern
// stay exact at every level.
// The epilogue joins the levels as integers and rounds once to FP64, without
// FP64 instructions (one holds the pipe of a quarter of the SM for 64 cycles).
// What is left is the operands' rounding to 2^-55 of their row's largest entry.
// A floating-point sum does not care how its index is scaled (a bond whose leg
// grows on one site as its partner falls on the other), a rounding relative to
// a row does, so the terms are balanced first: with a_k and b_k the exponents of
// the largest entries of term k on either side, the left operand is taken times
// 2^((b_k - a_k) / 2) and the right one divided by it, in the exponents alone.
// (Scales 1 .. 1e-8 on a leg and their inverses on its partner cost the metric
// all its digits without.)  The edges are Gram products: a_k = b_k.
// With that, relative to 113-bit sums the metric at D = 2 to 4 is off by 1e-16 to
// 1e-15 where the FP64 chain was off by 3e-16 to 2.3e-15, of its norm; an entry far
// below the norm keeps less relative accuracy than the chain gave it.
//
// Measured, environment of 48 bond updates at D = 8, r = 2: 14.2 ms against
// 196.6 ms on the FP64 pipe; of one at D = 3: 0.50 against 1.2 ms (a 64 x 64
// FP64 tile of the SIMT product holds one SM for 0.3 ms whatever its padding),
// so the sliced products run at every size.  Of the 14.2 ms the GEMMs take 7.4
// (the join at 40% of the BF16 peak, t1 to h bound by their epilogues), the
// slices 3.5, the exponents of rows and terms 1.4, the side edges and Y 1.4.
//
// Complex products are one real GEMM: rows of B hold [Re | Im] along K, a
// complex row of A the two real rows [Re | -Im] and [Im | Re].  They lie 16
// rows apart, so that lanes l and l + 16 of an epilogue warp hold the real and
// the imaginary part of one entry and exchange columns to store 16 bytes each.
//
// One persistent CTA per SM: warp 0 fetches stages of 32 real terms of all
// seven slices (TMA boxes 32 x rows x 7, 64-byte swizzle), warp 1 issues the
// MMAs (A slice i against B slices 0 .. 7-i, which are contiguous rows of
// shared memory: accumulator columns 64 l .. hold level l; 13 instructions and
// 34 digit products per 16 terms), sixteen warps drain.  The 64 x 64 complex tile (all 512 TMEM
// columns) is single-buffered: the drain costs about a tenth of the products
// of 256 terms.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>
#include <string.h>

#include "ntu_dev.cuh"
#include "ntu_impl.h"
#include "tc_sm103.cuh"

namespace ntu {

namespace {
constexpr int ZS = OZ64_SLICES;                       // 7
constexpr int ZK = 32;                                // real terms of a stage
constexpr int ZN = 64;                                // complex columns of a tile
constexpr int ZA_SLICE = 128 * ZK * 2, ZB_SLICE = ZN * ZK * 2;
constexpr int ZSTAGE = ZS * (ZA_SLICE + ZB_SLICE), ZSTAGES = 2;
constexpr int ZCHUNK = 8;                             // stages between drains (256 terms)
constexpr int ZEPI = 16, ZTHREADS = 64 + 32 * ZEPI;
constexpr size_t ZSMEM = (size_t)ZSTAGES * ZSTAGE + 1024 + 256;
constexpr long long ZWAIT = 1ll << 28;
constexpr int ZNAN = 20000;                           // exponent of a row with a non-finite entry
constexpr int ZNONE = -(1 << 24), ZINF = 1 << 24;     // exponent of 0, of a non-finite entry
static_assert(ZSMEM <= 227 * 1024, "shared memory budget");

// K-major tile whose rows are 64 bytes, written by TMA with the 64-byte
// swizzle; 8-row groups are 512 bytes apart (layout type 4).
__device__ __forceinline__ uint64_t sdesc_k64(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFF) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(512 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)4 << 61;
  return d;
}

__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* map, uint64_t* bar, int x,
                                            int y, int z, int w) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%3, %4, %5, %6}], [%2];" ::"r"(tc::smem_u32(dst)),
      "l"(map), "r"(tc::smem_u32(bar)), "r"(x), "r"(y), "r"(z), "r"(w)
      : "memory");
}

// Real row of complex row c in a doubled operand (+ 16: the imaginary row).
__host__ __device__ __forceinline__ int oz64_row(int c) {
  return (c >> 6) * 128 + ((c & 63) >> 4) * 32 + (c & 15);
}

// (hi 2^32 + lo) 2^ex rounded to the nearest double.
__device__ __forceinline__ double oz64_join(long long hi, long long lo, int ex) {
  long long h = hi + (lo >> 32);
  unsigned long long l = (unsigned)lo;
  const bool neg = h < 0;
  if (neg) {
    h = -h - (l != 0 ? 1 : 0);
    l = (0ull - l) & 0xffffffffull;
  }
  unsigned long long m = (unsigned long long)h;
  int s = m ? __clzll((long long)m) : 32;
  s = s < 32 ? s : 32;
  const bool sticky = (l & ((1ull << (32 - s)) - 1ull)) != 0;
  m = (m << s) | (l >> (32 - s));
  if (m == 0) return 0.0;
  const int z = __clzll((long long)m);
  m <<= z;
  unsigned long long q = m >> 11;
  const unsigned r = (unsigned)(m & 0x7ff);
  q += r > 0x400u || (r == 0x400u && (sticky || (q & 1)));
  const int e = ex + 32 - s + 63 - z + 1023;             // biased exponent of the leading bit
  if (e <= 0) return 0.0;
  unsigned long long b = ((unsigned long long)(e - 1) << 52) + q;
  if (e >= 2047) b = 0x7ff0000000000000ull;
  return __longlong_as_double((long long)(b | (neg ? 0x8000000000000000ull : 0ull)));
}
}  // namespace

struct Oz64Args {
  int M, N, mtiles, ntiles, stages;
  const int *rowC, *colC, *eA, *eB;      // eA: 64 mtiles, eB: 64 ntiles per item
  double2* C;
  long long sC;
  int* err;
};

__global__ void __launch_bounds__(ZTHREADS, 1) k_oz64_gemm(const __grid_constant__ CUtensorMap tmA,
                                                           const __grid_constant__ CUtensorMap tmB,
                                                           Oz64Args a, int items) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(smem + (size_t)ZSTAGES * ZSTAGE);
  uint64_t* empty = full + ZSTAGES;
  uint64_t* accf = empty + ZSTAGES;                        // a chunk's accumulators are complete
  uint64_t* acce = accf + 1;                               // and have been read
  uint64_t* done = acce + 1;
  uint32_t* slot = (uint32_t*)(done + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int per_item = a.mtiles * a.ntiles;
  const long long total = (long long)per_item * items;
  if (tid == 0) {
    for (int s = 0; s < ZSTAGES; ++s) { tc::mbar_init(&full[s], 1); tc::mbar_init(&empty[s], 1); }
    tc::mbar_init(accf, 1);
    tc::mbar_init(acce, ZEPI);
    tc::mbar_init(done, 1);
    tc::fence_barrier_init();
  }
  if (warp == 0) tc::tmem_alloc(slot, 512);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = *slot;
  if (warp == 0) {
    if (lane == 0) {
      long long g = 0;
      bool ok = true;
      for (long long t = blockIdx.x; t < total && ok; t += gridDim.x) {
        const int z = (int)(t / per_item), rem = (int)(t % per_item);
        const int mt = rem / a.ntiles, nt = rem % a.ntiles;
        for (int it = 0; it < a.stages; ++it, ++g) {
          const int s = (int)(g % ZSTAGES);
          if (g >= ZSTAGES && !tc::mbar_wait(&empty[s], (uint32_t)((g / ZSTAGES - 1) & 1), ZWAIT)) {
            raise_status(a.err, ST_TIMEOUT, WHY_TC_WAIT);
            ok = false;
            break;
          }
          tc::mbar_expect_tx(&full[s], ZSTAGE);
          tma_load_4d(smem + (size_t)s * ZSTAGE, &tmA, &full[s], it * ZK, mt * 128, 0, z);
          tma_load_4d(smem + (size_t)s * ZSTAGE + ZS * ZA_SLICE, &tmB, &full[s], it * ZK, nt * ZN,
                      0, z);
        }
      }
      for (long long q = g < ZSTAGES ? 0 : g - ZSTAGES; q < g; ++q)   // no copy in flight at exit
        if (!tc::mbar_wait(&full[q % ZSTAGES], (uint32_t)((q / ZSTAGES) & 1), ZWAIT))
          raise_status(a.err, ST_TIMEOUT, WHY_TC_WAIT);
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0) {
      long long g = 0, chunk = 0;
      bool ok = true;
      for (long long t = blockIdx.x; t < total && ok; t += gridDim.x) {
        for (int it = 0; it < a.stages && ok; ++it, ++g) {
          const bool first = it % ZCHUNK == 0;
          if (first && chunk > 0 && !tc::mbar_wait(acce, (uint32_t)((chunk - 1) & 1), ZWAIT)) ok = false;
          const int s = (int)(g % ZSTAGES);
          if (ok && !tc::mbar_wait(&full[s], (uint32_t)((g / ZSTAGES) & 1), ZWAIT)) ok = false;
          if (!ok) {
            raise_status(a.err, ST_TIMEOUT, WHY_TC_WAIT);
            break;
          }
          tc::fence_after_sync();
          const uint64_t da = sdesc_k64(tc::smem_u32(smem + (size_t)s * ZSTAGE));
          const uint64_t db = sdesc_k64(tc::smem_u32(smem + (size_t)s * ZSTAGE + ZS * ZA_SLICE));
#pragma unroll
          for (int kk = 0; kk < ZK / 16; ++kk)
#pragma unroll
            for (int i = 0; i < ZS; ++i) {
              const uint64_t ai = da + (uint64_t)(i * (ZA_SLICE >> 4) + 2 * kk);
              const uint64_t b0 = db + (uint64_t)(2 * kk);
              // levels l .. l + n - 1: slices l - i .. of B
              auto levels = [&](int l, int n, uint32_t add) {
                tc::mma_bf16(tmem + 64 * l, ai, b0 + (uint64_t)((l - i) * (ZB_SLICE >> 4)),
                             tc::idesc_bf16_f32(128, n * 64), add);
              };
              // the drained levels i .. 4 (256 columns at most), begun by i = 0
              const uint32_t add = !(first && kk == 0 && i == 0);
              if (i < 5) levels(i, i == 0 ? 4 : 5 - i, add);
              if (i == 0) levels(4, 1, add);
              // the levels to 7 (there is no slice 7 for i = 0: i = 1 begins level 7)
              const int l0 = i < 5 ? 5 : i;
              const bool split = i == 1 && it == 0 && kk == 0;
              levels(l0, (i == 0 || split ? 7 : 8) - l0, !(it == 0 && kk == 0 && i == 0));
              if (split) levels(7, 1, 0);
            }
          tc::mma_commit(&empty[s]);
          if (it % ZCHUNK == ZCHUNK - 1 || it == a.stages - 1) {
            tc::mma_commit(accf);
            ++chunk;
          }
        }
      }
      tc::mma_commit(done);                                  // every MMA has retired before TMEM goes
      if (!tc::mbar_wait(done, 0, ZWAIT)) raise_status(a.err, ST_TIMEOUT, WHY_TC_WAIT);
    }
    __syncwarp();
  } else {
    const int quarter = warp & 3, cs = ((warp - 2) >> 2) * 16;   // TMEM lanes, columns cs .. cs + 15
    const uint32_t tb = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)cs;
    const int ethreads = 32 * ZEPI;
    long long chunk = 0;
    bool ok = true;
    for (long long t = blockIdx.x; t < total && ok; t += gridDim.x) {
      const int z = (int)(t / per_item), rem = (int)(t % per_item);
      const int mt = rem / a.ntiles, nt = rem % a.ntiles;
      long long hi[16];                                      // levels 0 .. 3
      int l4[16];
#pragma unroll
      for (int q = 0; q < 16; ++q) { hi[q] = 0; l4[q] = 0; }
      for (int it = 0; it < a.stages; it += ZCHUNK, ++chunk) {
        const bool got = tc::mbar_wait(accf, (uint32_t)(chunk & 1), ZWAIT);
        if (!tc::bar_and(1, ethreads, got)) {
          if (tid == 64) raise_status(a.err, ST_TIMEOUT, WHY_TC_WAIT);
          ok = false;
          break;
        }
        tc::fence_after_sync();
#pragma unroll 1
        for (int l = 0; l < 4; ++l) {
          float v[16];
          tc::tmem_ld16(tb + 64 * l, v);
#pragma unroll
          for (int q = 0; q < 16; ++q) hi[q] += (long long)__float2int_rn(v[q]) << (24 - 8 * l);
        }
        float v[16];
        tc::tmem_ld16(tb + 64 * 4, v);
#pragma unroll
        for (int q = 0; q < 16; ++q) l4[q] += __float2int_rn(v[q]);
        if (it + ZCHUNK < a.stages) {
          tc::fence_before_sync();
          __syncwarp();
          if (lane == 0) tc::mbar_arrive(acce);
        }
      }
      if (!ok) break;
      long long lo[16];
#pragma unroll
      for (int q = 0; q < 16; ++q) lo[q] = l4[q];
#pragma unroll
      for (int l = 5; l < 8; ++l) {
        float v[16];
        tc::tmem_ld16(tb + 64 * l, v);
#pragma unroll
        for (int q = 0; q < 16; ++q) lo[q] = (lo[q] << 8) + __float2int_rn(v[q]);
      }
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(acce);
      // ++chunk happened in the loop; lane < 16: Re, lane >= 16: Im of row m
      const int m = mt * 64 + quarter * 16 + (lane & 15), n0 = nt * ZN + cs;
      const int em = a.eA[(long long)z * a.mtiles * 64 + m] - 68;
      const int* eb = a.eB + (long long)z * a.ntiles * ZN + n0;
      double2* C = a.C + (long long)z * a.sC + (m < a.M ? a.rowC[m] : 0);
      const bool im = lane >= 16;
#pragma unroll
      for (int q = 0; q < 16; q += 2) {
        double o[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int e = em + eb[q + u];
          o[u] = e > ZNAN / 2 ? __longlong_as_double(0x7ff8000000000000ll)
                              : oz64_join(hi[q + u], lo[q + u], e);
        }
        // lane l keeps column q, lane l + 16 column q + 1
        const double give = im ? o[0] : o[1];
        const double take = __shfl_xor_sync(0xffffffffu, give, 16);
        const int n = n0 + q + (im ? 1 : 0);
        if (m < a.M && n < a.N)
          C[a.colC[n]] = im ? make_double2(take, o[1]) : make_double2(o[0], take);
      }
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if (warp == 0) tc::tmem_dealloc(tmem, 512);
}

// ------------------------------------------------------------ slicing
struct Oz64Slice {
  const double2* src;
  long long s_src;                       // per item
  const int *row, *kk;                   // element offsets row[r] + kk[k]
  int rows, K, Kh, rowsP, conj, doubled; // Kh: padded terms of a half; rowsP: rows of a slice
  __nv_bfloat16* out;                    // [item][7][rowsP][2 Kh]
  int* ex;                               // [item][epitch] row exponents
  int epitch;
  int* mx;                               // [item][epitch] exponents of the largest entries
  int* cm;                               // [item][2][kpitch] exponents of the terms, left and
  int kpitch;                            // right (NULL: not balanced)
};

// Biased exponent of the leading bit of the larger part of v (below 1 for
// subnormals).
__device__ __forceinline__ int oz64_exp(double2 v) {
  const unsigned h = max((unsigned)__double2hiint(v.x) & 0x7fffffffu, (unsigned)__double2hiint(v.y) & 0x7fffffffu);
  const int e = (int)(h >> 20);
  if (e == 0) {
    const long long m = 0xfffffffffffffll;
    const long long b = max(__double_as_longlong(v.x) & m, __double_as_longlong(v.y) & m);
    return b ? 12 - __clzll(b) : ZNONE;
  }
  return e == 0x7ff ? ZINF : e;
}

// Exponent of the factor of term k: (b_k - a_k) / 2 on the left operand, its
// negative on the right one; 0 where a side has no finite non-zero entry.
__device__ __forceinline__ int oz64_factor(const Oz64Slice& s, long long z, int k) {
  if (!s.cm || k >= s.K) return 0;
  const int* c = s.cm + z * 2 * s.kpitch + k;
  const int a = c[0], b = c[s.kpitch];
  if (a < -4096 || b < -4096 || a > 4096 || b > 4096) return 0;
  const int f = (b - a) >> 1;
  return s.doubled ? f : -f;
}

// Exponents of the largest entries of every term of both operands: a warp
// takes eight terms of 128 rows, coalesced along the rows.
__global__ void __launch_bounds__(256) k_oz64_terms(Oz64Slice left, Oz64Slice right, int lblocks) {
  const bool lt = (int)blockIdx.x < lblocks;
  const Oz64Slice& s = lt ? left : right;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int r0 = ((int)blockIdx.x - (lt ? 0 : lblocks)) * 128 + lane, k0 = blockIdx.y * 64 + w;
  const double2* p = s.src + (long long)blockIdx.z * s.s_src;
  int* c = s.cm + ((long long)blockIdx.z * 2 + (lt ? 0 : 1)) * s.kpitch;
  int off[4];
#pragma unroll
  for (int t = 0; t < 4; ++t) off[t] = r0 + 32 * t < s.rows ? s.row[r0 + 32 * t] : -1;
#pragma unroll 2
  for (int i = 0; i < 8; ++i) {
    const int k = k0 + 8 * i;
    if (k >= s.K) break;
    const int kk = s.kk[k];
    int e = ZNONE;
#pragma unroll
    for (int t = 0; t < 4; ++t)
      if (off[t] >= 0) e = max(e, oz64_exp(p[off[t] + kk]));
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) atomicMax(c + k, e);
  }
}

// Exponent of the largest entry of every row, for rows of more than 64 terms;
// 32 rows x 8 terms per pass, coalesced along the rows.
__global__ void __launch_bounds__(256) k_oz64_max(Oz64Slice s) {
  __shared__ int red[8][32], fac[256];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int r = blockIdx.x * 32 + lane, k0 = blockIdx.y * 256;
  fac[threadIdx.x] = oz64_factor(s, blockIdx.z, k0 + (int)threadIdx.x);
  __syncthreads();
  int m = ZNONE;
  if (r < s.rows) {
    const double2* p = s.src + (long long)blockIdx.z * s.s_src + s.row[r];
    const int k1 = k0 + 256 < s.K ? k0 + 256 : s.K;
#pragma unroll 4
    for (int k = k0 + w; k < k1; k += 8) m = max(m, oz64_exp(p[s.kk[k]]) + fac[k - k0]);
  }
  red[w][lane] = m;
  __syncthreads();
  if (w == 0 && r < s.rows) {
    for (int i = 1; i < 8; ++i) m = max(m, red[i][lane]);
    atomicMax(s.mx + (long long)blockIdx.z * s.epitch + r, m);
  }
}

// x 2^(f + 54 - e) rounded to the nearest integer, e = em - 1022 (em the biased
// exponent of the row's largest entry times its factor), from the bits.
__device__ __forceinline__ long long oz64_fix(double x, int em, int f) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  int ex = (int)(b >> 52) & 0x7ff;
  unsigned long long m = b & 0xfffffffffffffull;
  if (ex) {
    m |= 0x10000000000000ull;
  } else {                                                // subnormal (or 0, which stays 0)
    const int z = __clzll((long long)m) - 11;
    m <<= z;
    ex = 1 - z;
  }
  const int sh = em - 1 - ex - f;                         // >= -1
  const long long v = sh < 0 ? (long long)(m << 1)
                             : (sh == 0 ? (long long)m
                                        : (sh < 56 ? (long long)((m + (1ull << (sh - 1))) >> sh) : 0ll));
  return (long long)b < 0 ? -v : v;
}

// One block: 32 rows x 64 terms, read along the rows, turned in shared memory,
// written as 16-byte runs of eight terms of every slice.
__global__ void __launch_bounds__(256) k_oz64_slice(Oz64Slice s) {
  __shared__ double2 tile[64 * 33];
  __shared__ int red[8][32], em[32], fac[64];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int r0 = blockIdx.x * 32, k0 = blockIdx.y * 64;
  const long long z = blockIdx.z;
  {
    const int r = r0 + lane;
    int m = ZNONE;
    const double2* p = s.src + z * s.s_src + (r < s.rows ? s.row[r] : 0);
    double2 v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int k = k0 + w + 8 * i;
      v[i] = make_double2(0.0, 0.0);
      if (r < s.rows && k < s.K) v[i] = p[s.kk[k]];
    }
    if (threadIdx.x < 64) fac[threadIdx.x] = oz64_factor(s, z, k0 + (int)threadIdx.x);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int k = w + 8 * i;
      if (s.conj) v[i].y = -v[i].y;
      tile[k * 33 + lane] = v[i];
      m = max(m, oz64_exp(v[i]) + fac[k]);
    }
    red[w][lane] = m;
    __syncthreads();
    if (w == 0) {
      if (s.mx) {
        m = r < s.rows ? s.mx[z * s.epitch + r] : ZNONE;
      } else {
        for (int i = 1; i < 8; ++i) m = max(m, red[i][lane]);
      }
      const int e = m < -8192 ? 1 : m;                      // a row of zeros
      em[lane] = e;
      if (blockIdx.y == 0 && r < s.epitch) s.ex[z * s.epitch + r] = e > 8192 ? ZNAN : e - 1022;
    }
    __syncthreads();
  }
  const int rl = threadIdx.x >> 3, kg = (threadIdx.x & 7) * 8, r = r0 + rl;
  if (r >= s.rows || k0 + kg >= s.Kh) return;              // Kh is a multiple of 16
  const int e = em[rl];
  const long long pitch = 2LL * s.Kh, slice = pitch * s.rowsP;
  __nv_bfloat16* o = s.out + z * ZS * slice + k0 + kg;
  const int rr = s.doubled ? oz64_row(r) : r;
#pragma unroll 1
  for (int c = 0; c < 2; ++c) {                            // Re, Im
    uint32_t dg[ZS][4];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      uint32_t two[2][ZS];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const double2 v = tile[(kg + 2 * p + u) * 33 + rl];
        long long x = e > 8192 ? 0 : oz64_fix(c ? v.y : v.x, e, fac[kg + 2 * p + u]);
#pragma unroll
        for (int i = ZS - 1; i >= 0; --i) {
          const int d = i ? (int)((unsigned)(x + 128) & 255u) - 128 : (int)x;
          x = (x - d) >> 8;
          // the float of a small integer, whose upper half is its BF16
          two[u][i] = __float_as_uint(__int_as_float(0x4b400000 + d) - 12582912.0f);
        }
      }
#pragma unroll
      for (int i = 0; i < ZS; ++i) dg[i][p] = __byte_perm(two[0][i], two[1][i], 0x7632);
    }
#pragma unroll
    for (int i = 0; i < ZS; ++i) {
      const uint4 v = make_uint4(dg[i][0], dg[i][1], dg[i][2], dg[i][3]);
      const uint4 n = make_uint4(v.x ^ 0x80008000u, v.y ^ 0x80008000u, v.z ^ 0x80008000u,
                                 v.w ^ 0x80008000u);
      __nv_bfloat16* oi = o + i * slice + (long long)rr * pitch;
      if (!s.doubled) {
        *reinterpret_cast<uint4*>(oi + c * s.Kh) = v;
      } else {
        // real row [Re | -Im], imaginary row [Im | Re]
        *reinterpret_cast<uint4*>(oi + c * s.Kh) = c ? n : v;
        *reinterpret_cast<uint4*>(oi + 16 * pitch + (1 - c) * s.Kh) = v;
      }
    }
  }
}

// ---------------------------------------------------------- host side
static int oz64_map(CUtensorMap* map, void* base, long long cols, long long rows, long long items,
                    int box_rows) {
  static PFN_cuTensorMapEncodeTiled_v12000 enc = nullptr;
  if (!enc) {
    cudaDriverEntryPointQueryResult q;
    void* fn = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      enc = (PFN_cuTensorMapEncodeTiled_v12000)fn;
  }
  if (!enc) return NTU_EUNSUPPORTED;
  cuuint64_t dims[4] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)ZS, (cuuint64_t)items};
  cuuint64_t strides[3] = {(cuuint64_t)cols * 2, (cuuint64_t)(cols * rows * 2),
                           (cuuint64_t)(cols * rows * 2 * ZS)};
  cuuint32_t box[4] = {ZK, (cuuint32_t)box_rows, ZS, 1}, es[4] = {1, 1, 1, 1};
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, base, dims, strides, box, es,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? NTU_OK : NTU_ECUDA;
}

static void oz64_geometry(Oz64Geo& g, const GemmOp& op) {
  g.Kh = (op.Kd + 15) / 16 * 16;
  g.rowsA = (op.M + 63) / 64 * 128;
  g.rowsB = (op.N + 63) / 64 * 64;
}

// Geometry, chunk of items and scratch of the sliced GEMMs; leaves oz64.items
// at 0 (the SIMT path then runs) on a device without tcgen05 or where the
// scratch cannot be had.
void oz64_init(ntu_ctx* c) {
  Plan& P = c->plan;
  Oz64& z = P.oz64;
  memset(&z, 0, sizeof(z));
  if (c->cfg.precision != NTU_FP64) return;
  int dev = 0, major = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess ||
      major != 10)
    return;
  if (cudaFuncSetAttribute(k_oz64_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ZSMEM) !=
      cudaSuccess) {
    cudaGetLastError();
    return;
  }
  const GemmOp* ops[4] = {&P.eTL, &P.t1, &P.t2, &P.join};
  long long a = 0, b = 0;
  int ra = 0, rb = 0;
  for (int i = 0; i < 4; ++i) {
    Oz64Geo& g = z.geo[i];
    oz64_geometry(g, *ops[i]);
    const long long sa = (long long)g.rowsA * 2 * g.Kh * ZS * 2, sb = (long long)g.rowsB * 2 * g.Kh * ZS * 2;
    a = sa > a ? sa : a;
    b = sb > b ? sb : b;
    ra = g.rowsA / 2 > ra ? g.rowsA / 2 : ra;
    rb = g.rowsB > rb ? g.rowsB : rb;
  }
  z.kpitch = 1;
  for (const GemmOp* o : ops) z.kpitch = o->Kd > z.kpitch ? o->Kd : z.kpitch;
  a = (a + 1023) / 1024 * 1024;
  b = (b + 1023) / 1024 * 1024;
  // items at a time: enough to fill the SMs, within about 2 GB.  Rows beyond
  // an operand's own stay as they are: they enter only results that are not
  // stored
  long long items = (2ll << 30) / (a + b);
  if (items < 1) items = 1;
  if (items > c->cfg.max_batch) items = c->cfg.max_batch;
  const long long tbytes = items * OZ64_BALANCED * 2LL * z.kpitch * 4;
  const long long ebytes = items * (ra + 2LL * rb + ra) * 4 + tbytes;
  void* base = nullptr;
  if (cudaMalloc(&base, items * (a + b) + ebytes) != cudaSuccess) {
    cudaGetLastError();                                    // no room: the SIMT path
    return;
  }
  z.base = base;
  z.SA = (char*)base;
  z.SB = z.SA + items * a;
  z.eA = (int*)(z.SB + items * b);
  z.eB = z.eA + items * ra;
  z.cm = z.eB + items * rb;
  z.mx = z.cm + tbytes / 4;
  int st = NTU_OK;
  for (int i = 0; i < 4 && st == NTU_OK; ++i) {
    Oz64Geo& g = z.geo[i];
    st = oz64_map(&g.mapA, z.SA, 2 * g.Kh, g.rowsA, items, 128);
    if (st == NTU_OK) st = oz64_map(&g.mapB, z.SB, 2 * g.Kh, g.rowsB, items, ZN);
  }
  if (st == NTU_OK) z.items = (int)items;
}

void oz64_free(ntu_ctx* c) {
  if (c->plan.oz64.base) cudaFree(c->plan.oz64.base);
  c->plan.oz64.base = nullptr;
}

// Empties the term exponents of a pass's balanced products.
cudaError_t oz64_begin(ntu_ctx* c) {
  const Oz64& z = c->plan.oz64;
  return cudaMemsetAsync(z.cm, 0x80, sizeof(int) * (size_t)z.items * OZ64_BALANCED * 2 * z.kpitch, c->stream);
}

static Oz64Slice oz64_operand(ntu_ctx* c, const GemmOp& op, const Oz64Geo& g, int slot, bool left,
                              const double2* src) {
  const Oz64& z = c->plan.oz64;
  const int* t = c->plan.d_tab;
  Oz64Slice s;
  s.src = src;
  s.s_src = left ? op.sA : op.sB;
  s.row = t + (left ? op.rowA : op.colB);
  s.kk = t + (left ? op.kA : op.kB);
  s.rows = left ? op.M : op.N;
  s.K = op.Kd;
  s.Kh = g.Kh;
  s.rowsP = left ? g.rowsA : g.rowsB;
  s.conj = left ? op.conjA : op.conjB;
  s.doubled = left ? 1 : 0;
  s.out = reinterpret_cast<__nv_bfloat16*>(left ? z.SA : z.SB);
  s.ex = left ? z.eA : z.eB;
  s.epitch = left ? g.rowsA / 2 : g.rowsB;
  s.mx = g.Kh > 64 ? z.mx : nullptr;
  s.cm = slot < 0 ? nullptr : z.cm + (size_t)slot * z.items * 2 * z.kpitch;
  s.kpitch = z.kpitch;
  return s;
}

static cudaError_t oz64_slice(ntu_ctx* c, const Oz64Slice& s, int n) {
  const unsigned bx = (unsigned)((s.rows + 31) / 32);
  if (s.mx) {
    cudaError_t e = cudaMemsetAsync(s.mx, 0x80, sizeof(int) * (size_t)n * s.epitch, c->stream);
    if (e != cudaSuccess) return e;
    k_oz64_max<<<dim3(bx, (unsigned)((s.K + 255) / 256), (unsigned)n), 256, 0, c->stream>>>(s);
    e = after_launch(c, "k_oz64_max");
    if (e != cudaSuccess) return e;
  }
  k_oz64_slice<<<dim3(bx, (unsigned)((s.Kh + 63) / 64), (unsigned)n), 256, 0, c->stream>>>(s);
  return after_launch(c, "k_oz64_slice");
}

// C = A B of one plan GEMM for n <= oz64.items items (geometry index gi; slot:
// that of its term exponents among the pass's balanced products, -1 for a Gram
// product).
cudaError_t launch_oz64(ntu_ctx* c, const GemmOp& op, int gi, int slot, int n, const double2* A,
                        const double2* B, double2* C) {
  Oz64& z = c->plan.oz64;
  const Oz64Geo& g = z.geo[gi];
  const Oz64Slice sa = oz64_operand(c, op, g, slot, true, A), sb = oz64_operand(c, op, g, slot, false, B);
  cudaError_t e = cudaSuccess;
  if (slot >= 0) {
    const int la = (sa.rows + 127) / 128, lb = (sb.rows + 127) / 128;
    k_oz64_terms<<<dim3((unsigned)(la + lb), (unsigned)((op.Kd + 63) / 64), (unsigned)n), 256, 0, c->stream>>>(
        sa, sb, la);
    e = after_launch(c, "k_oz64_terms");
  }
  if (e == cudaSuccess) e = oz64_slice(c, sa, n);
  if (e == cudaSuccess) e = oz64_slice(c, sb, n);
  if (e != cudaSuccess) return e;
  Oz64Args a;
  const int* t = c->plan.d_tab;
  a.M = op.M; a.N = op.N;
  a.mtiles = g.rowsA / 128; a.ntiles = g.rowsB / ZN;
  a.stages = 2 * g.Kh / ZK;
  a.rowC = t + op.rowC; a.colC = t + op.colC;
  a.eA = z.eA; a.eB = z.eB;
  a.C = C; a.sC = op.sC;
  a.err = c->d_status;
  const long long tiles = (long long)a.mtiles * a.ntiles * n;
  k_oz64_gemm<<<(int)(tiles < c->sms ? tiles : c->sms), ZTHREADS, ZSMEM, c->stream>>>(g.mapA, g.mapB, a, n);
  return after_launch(c, "k_oz64_gemm");
}

}  // namespace ntu
